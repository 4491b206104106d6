// Host side of the tensor path: tile planner, tensor maps, single, repacked and shared launches.  The kernel and what it
// does are in conv_tc_kernel.cuh.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <cstring>
#include <mutex>
#include <utility>

#include "conv_tc_kernel.cuh"

namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }();
    return fn;
}

// Held while a tensor map is looked up, encoded or copied out.  The maps lie in the context (activations) and in the handle
// (weights), and both may be in use by several threads at once, a handle by several contexts too: one lock for all.  (An
// uncontended lock costs some 20 ns of a call's 3 us of host time.)
std::mutex g_maps;

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Which operand the positions are.  A tcgen05.mma costs about the same whatever its N, so the wide operand should be
// N: with the filters as M and up to 256 positions as N a layer of 128 filters per tile runs near the tensor peak.
// A narrow layer wastes most of M that way and, worse, leaves three of four epilogue warps without TMEM lanes to
// read; with the positions as M every lane carries an output and a thread's filters are contiguous in NHWC.  The
// price is one instruction per 128 positions instead of per 256: taken where few instructions are needed anyway.
bool use_pxm(const rtoss_packed* p) { return p->Cout <= kPxmMaxCout && p->ksize == 1 && p->dtype != RTOSS_F32; }

// fp32 layers whose small products are bf16 ones
bool has_corr16(const rtoss_packed* p) { return p->dtype == RTOSS_F32 && rtoss_f32_corr16(p->Cin, p->ksize); }

// Bytes of a staged row: 16-bit layers of at most 32 input channels stage 64-byte rows (64-byte swizzle) instead of
// 128-byte rows half of which would be zero fill.
int row_bytes_of(const rtoss_packed* p) { return (p->dtype != RTOSS_F32 && p->Cin <= 32) ? 64 : kRowBytes; }
// channel blocks (staged rows' worth of channels) of a layer
int ncb_of(const rtoss_packed* p) {
    const int cb_ch = row_bytes_of(p) / (p->dtype == RTOSS_F32 ? 4 : 2);
    return (p->Cin + cb_ch - 1) / cb_ch;
}

struct TcPlan {
    int TH, TW, Wq, N_px, NA, NB, G, n_sub, sub_rows, rows_staged, tiles_x, smem;
    int KS, cb_per;      // CTAs that share a tile's channel blocks (a cluster), blocks per share
    long tiles;          // tiles of the layer (not counting shares)
    int half;            // 3x3 stride 2: a channel block in two activation stages (TcArgs::half)
    double us;           // what the model below expects of a launch of its own (half: of one with a channel block in one stage)
    double tile_us, epi_us;   // and of one tile: operands and instructions, epilogue
};

// What a plan depends on; plain values, so that equal calls have equal plans whatever tensors they bring.
struct PlanKey {
    int N, Ho, Wo, ksize, S, Cin, Cout, dtype;
    int resid;       // a residual operand (its staging takes shared memory)
    int sms, dev;    // SMs to fill; device whose cluster limits hold (-1: the built-in ones)
    int shared;      // a problem of a shared launch, which never splits; 1: beside others, tiles are judged by the work they
                     // do per cycle; 2: with nothing beside it
    int max_px;      // most positions per tile
    int force_G, n_tabs;
    int may_half;    // 3x3 stride 2: its channel blocks may come in two activation stages (see single_plan_key)
    int half;        // and do (a search's, see plan_tc)
    int three;       // fp32: the cost of three tf32 products a tap, whatever the layer's kernel forms (see plan_tc)
};

// Most thread-block clusters of `ks` CTAs (one CTA per SM) a device holds at once.  Clusters live inside a GPC and the
// GPCs of a B200 differ in size, so 148 SMs hold 32 clusters of four and 15 of eight, not 37 and 18: a launch of one more
// takes twice the time (measured: 32 x 4 CTAs 11 us, 36 x 4 CTAs 19 us).  Asked of the device once; -1 or a device that
// cannot be asked: the figures of this one.
std::atomic<int> g_max_clusters[64][9];
int max_clusters(int dev, int ks, int sms) {
    static const int kDefault[9] = {0, 148, 74, 40, 32, 20, 20, 15, 15};
    if (ks <= 1) return sms;
    int have = dev >= 0 && dev < 64 ? g_max_clusters[dev][ks].load(std::memory_order_relaxed) : 0;
    if (have <= 0) have = kDefault[ks];
    return have * sms / 148 < have ? have * sms / 148 : have;
}

// Expected time of a launch, in microseconds, for one way of cutting a layer.  16-bit data: the constants are a fit to 6 500
// measured (layer, tile, split) combinations of the two detectors' layers at eleven sizes, batch 1 to 16, launches back to
// back (programmatic dependent launch); typical error 7 %, and the plan it picks is on average 1.9 % from the best measured
// one (4 % with the constants of the kernel before it was compiled in forms).  fp32 keeps the fit made then, when one warp split
// the activation blocks: layers of three tf32 products take 0.47 to 1.35 of what it expects of them, 0.78 in the geometric mean
// of 54 random ones.  What it knows:
//   - an instruction takes N / 2 cycles for N positions, but never less than 47; per weight stage 0.13 us of barrier
//     round trip;
//   - a CTA is fed at most 118 KB per us (tiles of stride 2, whose boxes overlap, count 0.56);
//   - the epilogue's sixteen warps take the accumulator in chunks of 32 columns, four warps a chunk: up to 128 positions
//     cost what 32 cost, 0.57 us; positions on M: filters in groups of 16 instead;
//   - a launch costs 1.9 us whatever it does, 0.9 more when it leaves no SM for the next one to start on, and 0.5 us until
//     its first operands are there;
//   - sharing a tile's channel blocks: 0.39 us + 0.27 per CTA of the cluster + 0.37 per chunk exchanged.
struct PlanFit {
    double cycles, stage, block, feed, lone, epi_pxm, epi_split, epi, launch, busy, first, tail, split, split_cta, split_chunk, strided;
};
constexpr PlanFit kFit16 = {46.7, 0.13, 0.027, 118, 1.05, 0.473, 0.116, 0.573, 1.93, 0.905, 0.50, 0.297, 0.39, 0.273, 0.369, 0.563};
constexpr PlanFit kFit32 = {79.0, 0.205, 0.09, 87, 0.0, 0.46, 0.26, 0.52, 1.92, 0.59, 0.51, 0.61, 0.13, 0.34, 0.33, 1.0};
struct PlanCost {
    double us, tile_us, epi_us;
};
PlanCost plan_cost(const PlanKey& k, bool pxm, int w_rows, int row_bytes, int R, int n_px, int halves, int a_bytes, int G, int na,
                   long tiles, int KS, int cb_per) {
    const bool f32 = k.dtype == RTOSS_F32;
    const int taps = k.ksize == 3 ? 9 : 1;
    const int slab_ch = f32 ? 8 : 16, cb_ch = row_bytes / (f32 ? 4 : 2);
    const bool corr16 = f32 && rtoss_f32_corr16(k.Cin, k.ksize) && !k.three;
    const double slabs = (double)(k.Cin < cb_ch ? k.Cin : cb_ch) / slab_ch * (corr16 ? 2 : f32 ? 3 : 1);
    const int wstages = f32 ? 2 * taps / G : taps / G;
    const PlanFit& f = f32 ? kFit32 : kFit16;
    const double instr = (pxm ? f.cycles * halves : n_px / 2.0 > f.cycles ? n_px / 2.0 : f.cycles) / 1900.0;
    double mma = taps * slabs * instr + f.stage * wstages + f.block;
    if (corr16) {
        // fp32 3x3 layers whose small products are bf16 ones, 256->256 @80x80 x32 cut in eight ways, 96 to 240 positions a tile: a
        // weight stage of one tap takes its four instructions + 0.1 us, at least 0.28; one of three taps its twelve + 0.27.  66
        // other layers (32 to 512 channels, both strides, 16 to 256 positions, cut and uncut) take 0.67 to 1.15 of the model's
        // time, 0.83 in the geometric mean: too dear throughout, by about the same, so that it still orders the ways to cut one
        const double s = G * 4 * (n_px / 2.0 > 47.0 ? n_px / 2.0 : 47.0) / 1900.0 + (G == 3 ? 0.27 : 0.10);
        mma = wstages * (s > 0.28 ? s : 0.28) + f.block;
    }
    const double kb_b = (double)taps * w_rows * row_bytes * (f32 ? 2 : 1) / 1024.0, kb_a = a_bytes / 1024.0;
    const bool half = k.half != 0;
    const double kb_fed = kb_a * (k.S == 2 ? f.strided : 1.0) * (half ? 2 : 1);
    const double feed = (kb_fed + kb_b) / (corr16 ? 110 : f.feed);
    double blk = mma > feed ? mma : feed;
    if (half) {
        // a stage is asked for when the one it takes the place of has been read (half_order): what of its way the instructions
        // from there to its own do not cover
        const double way = 0.5 + 0.5 * kb_fed / f.feed, one = mma / 3, two = 2 * mma / 3;
        const double odd = way - (na == 2 ? one : mma), even = way - (na == 2 ? one : na == 3 ? two : mma);
        const double late = mma + (odd > 0 ? odd : 0) + (even > 0 ? even : 0);
        blk = late > blk ? late : blk;
        na = 2;
    }
    // one activation stage: loads and instructions take turns (fp32: and the split of the block between them, as long as one warp
    // took for it; four warps do it now, and layers planned with one stage take 0.52 to 0.83 of the model's time, seven of them)
    if (na == 1) blk = mma + (f32 ? 0.045 * kb_a : f.lone * kb_fed / 87.0);
    if (f32 && !corr16 && G == 3) blk += 2.0;   // (then only two weight stages fit: the ring's round trip shows)
    const int chunks = (n_px + 31) / 32;
    double epi;
    if (pxm) epi = f.epi_pxm * ((halves * ((k.Cout + 15) / 16) + 3) / 4);
    else if (KS > 1) epi = f.epi_split * ((2 * ((chunks + KS - 1) / KS) + 3) / 4);
    else epi = f.epi * ((chunks + 4 * R - 1) / (4 * R));
    if (f32) epi *= 12.9;   // element stores
    const double first_kb = kb_a + kb_b / taps * G;
    PlanCost c;
    c.tile_us = cb_per * blk;
    c.epi_us = epi;
    const long ctas = tiles * KS < k.sms ? tiles * KS : k.sms;
    const long waves = (tiles * KS + k.sms - 1) / k.sms;
    double us = f.launch + (ctas > k.sms / 2 ? f.busy * (ctas - k.sms / 2) / (k.sms / 2.0) : 0.0) + f.first + first_kb / f.feed + c.tile_us + epi;
    if (waves > 1) us += (waves - 1) * (c.tile_us > epi ? c.tile_us : epi) + f.tail * tiles / k.sms;
    if (KS > 1) us += f.split + f.split_cta * KS + f.split_chunk * chunks;
    c.us = us;
    return c;
}

// Geometry of a tile.  Positions of a tile run over TH rows of pitch Wq = TW + (columns of halo the
// staged rows carry); every tap reads the staged list from a shifted start row.
//   3x3 stride 1: one staged tile, TH+2 rows of TW+2 pixels, tap (r,c) at shift r*Wq + c.
//   1x1:          one staged tile, TH rows of TW pixels (stride 2: every second pixel and row, picked by
//                 the TMA element strides), shift 0.
//   3x3 stride 2: four staged tiles, one per (row parity, column parity) of the input, each TH+1 rows of
//                 TW+1 pixels fetched with element strides 2; tap r reads the odd rows for r = 0, 2 and
//                 the even rows for r = 1, one staged row further down for r = 1, 2; columns alike.
// The plan picks TH, the column segment TW (images wider than a TMA box are cut into segments), the
// ring depths, how many taps share a weight stage, and over how many CTAs of a cluster the channel blocks of a tile are
// spread (split K: a tile's MMAs are one serial chain; at most 8 CTAs, all of a launch's clusters on the device at once).
// only_ks: 0 = any split, else that one.
bool plan_search(const PlanKey& k, bool resid, int only_ks, TcPlan* out) {
    const bool f32 = k.dtype == RTOSS_F32;
    const bool pxm = k.ksize == 1 && k.Cout <= kPxmMaxCout && !f32;
    const int w_rows = pxm ? round_up(k.Cout, 16) : kMTile;
    const int row_bytes = (!f32 && k.Cin <= 32) ? 64 : kRowBytes;
    const int cb_ch = row_bytes / (f32 ? 4 : 2), ncb = (k.Cin + cb_ch - 1) / cb_ch;
    const int co_tiles = pxm ? 1 : (k.Cout + kMTile - 1) / kMTile;
    const int R = rtoss_wtc_layout_of(k.Cout, k.Cin, k.ksize, (rtoss_dtype)k.dtype).copies;
    const int S = k.S, Ho = k.Ho, Wo = k.Wo, ksize = k.ksize;
    const int halo = ksize == 3 ? (S == 1 ? 2 : 1) : 0;
    const bool half = k.half != 0;   // (then three taps a weight stage, and a_bytes is one of the block's two stages)
    const int n_sub = half ? 2 : (ksize == 3 && S == 2) ? 4 : 1;
    const int max_pitch = S == 1 ? 256 : 128;  // TMA box: at most 256 elements traversed per dimension
    const int fixed = 1024 /*alignment slack*/ + 512 /*barriers*/ + kEpiWarps * kPatchBytes /*epilogue patches*/ +
                      k.n_tabs * kMaxPx * 8 /*position tables*/ + (resid ? kEpiWarps * kResStage : 0) /*staging of the residual operand*/;
    const int cap = 227 * 1024 - 64;
    double best = 0;
    bool found = false;
    // One row of pixels (1x1, see row_form): tiles of any multiple of 16 of them.
    const bool one_row = ksize == 1 && S == 1 && k.N == 1 && Ho == 1;
    for (int seg = 1; seg <= 16; ++seg) {
        const int tw = one_row ? (16 * seg < Wo ? 16 * seg : Wo) : (Wo + seg - 1) / seg, nseg = one_row ? (Wo + tw - 1) / tw : seg;
        const int wq = tw + halo;
        if (wq > max_pitch || wq > 256) continue;
        if (one_row && 16 * (seg - 1) >= Wo) break;
        if (!one_row && nseg > 1 && (tw < 4 || (Wo + nseg - 2) / (nseg - 1) == tw) && found) continue;   // (the same columns as with fewer segments)
        for (int th = 1; th <= Ho; ++th) {
            const int rows_staged = th + halo;
            if (th * wq > 256 || rows_staged * S > 256) break;
            const int ty = (Ho + th - 1) / th;
            if (th > 1 && (Ho + ty - 1) / ty != th) continue;   // (the same bands with fewer rows)
            const int n_px = round_up(th * wq, 16);
            if (n_px > k.max_px && found) break;
            const int max_shift = ksize == 3 ? (S == 1 ? 2 * wq + 2 : wq + 1) : 0;
            int need_rows = n_px + max_shift > rows_staged * wq ? n_px + max_shift : rows_staged * wq;
            // positions as the M operand: every instruction reads 128 rows, also where the tile's list ends earlier
            const int halves = n_px > 128 ? 2 : 1;
            if (pxm && max_shift + 128 * halves > need_rows) need_rows = max_shift + 128 * halves;
            const int sub_rows = round_up(need_rows, 8);
            const int a_bytes = n_sub * sub_rows * row_bytes * (f32 ? 2 : 1);   // (fp32: heads and remainders)
            const long tiles = (long)k.N * ty * nseg * co_tiles;
            for (int G = (ksize == 3 ? 3 : 1); G >= (half ? 3 : 1); G -= 2) {
                if (k.force_G && G != k.force_G) continue;   // (the problems of one launch share the weight ring: one G for all)
                const int b_bytes = G * w_rows * row_bytes;
                int na = (cap - fixed - 2 * b_bytes) / a_bytes;
                if (na < (half ? 2 : 1)) continue;
                if (na > kMaxA) na = kMaxA;
                // A channel block feeds nine taps: with several blocks per tile two stages cover the load.  A layer of
                // one block per tile (at most 64 channels; 32 with 64-byte rows) has the next TILE's block as its next
                // stage, and its instructions (18 or 36 of at most 128 cycles) are over before a fetch from L2 returns:
                // it keeps as many stages as fit.
                if (na > 2 && ksize == 3 && ncb > 1 && !half) na = 2;
                int nb = (cap - fixed - na * a_bytes) / b_bytes;
                if (nb > kMaxB) nb = kMaxB;
                if (nb < 2) continue;
                const int rings = na * a_bytes + nb * b_bytes;
                for (int ks = 1; ks <= 8; ++ks) {
                    if (only_ks && ks != only_ks) continue;
                    int cb_per = ncb;
                    if (ks > 1) {
                        if (k.shared || pxm || R != 1 || tiles * ks > k.sms || ks > ncb) break;
                        if (tiles > max_clusters(k.dev, ks, k.sms)) continue;
                        cb_per = (ncb + ks - 1) / ks;
                        if ((ncb + cb_per - 1) / cb_per != ks) continue;   // (a share would be empty)
                        // the owners' buffers for the partial sums lie in the rings
                        const int n_lc = ((n_px + 31) / 32 + ks - 1) / ks;
                        if (ks * n_lc > 16 || ks * n_lc * 16384 > rings) continue;
                    }
                    const PlanCost c = plan_cost(k, pxm, w_rows, row_bytes, R, n_px, halves, a_bytes, G, na, tiles, ks, cb_per);
                    double cost = c.us;
                    if (k.shared == 1) {
                        // One of several problems that run side by side and together fill the SMs: what counts is the work
                        // a tile does for the time it keeps a CTA (3x3 stride 1: bound by its instructions, N / 2 cycles but
                        // never less than 76; other tiles by what surrounds the instructions: as many positions as fit).  The 76
                        // and the factors below are of the kernel whose issuing thread was alone in its warp; the single
                        // launches' model has 47 since (kFit16), these tiles have not been measured again.
                        const bool by_cycles = ksize == 3 && S == 1 && n_px / 2.0 < 128.0;
                        const double cyc = by_cycles ? (n_px / 2.0 > 76.0 ? n_px / 2.0 : 76.0) : 128.0;
                        const double eff = (double)(th * tw) / (2.0 * cyc) * Ho / (double)(ty * th) * Wo / (double)(tw * nseg);
                        const double halo_cost = (double)(th * tw) / (double)(rows_staged * wq);  // staged pixels that are outputs
                        cost = -(eff * (G == 3 || ksize == 1 ? 1.0 : (f32 ? 0.95 : 0.8)) * (na >= 2 ? 1.0 : (f32 ? 0.7 : 0.8)) *
                                     (0.8 + 0.2 * halo_cost) + 1e-4 * th);
                    }
                    if (!found || cost < best) {
                        found = true;
                        best = cost;
                        out->TH = th;
                        out->TW = tw;
                        out->Wq = wq;
                        out->N_px = n_px;
                        out->NA = na;
                        out->NB = nb;
                        out->G = G;
                        out->n_sub = n_sub;
                        out->sub_rows = sub_rows;
                        out->rows_staged = rows_staged;
                        out->tiles_x = nseg;
                        out->smem = rings + fixed;
                        out->KS = ks;
                        out->cb_per = cb_per;
                        out->half = k.half;
                        out->tiles = tiles;
                        out->us = c.us;
                        out->tile_us = c.tile_us;
                        out->epi_us = c.epi_us;
                    }
                }
                if (!f32) break;  // 16-bit data: the largest G that fits is taken for this (th, tw); fp32 weighs both
            }
        }
    }
    return found;
}

// The plan of a call.  The split is decided as if the call had a residual operand, whether it has one or not: a call with
// a residual then adds up its products in the order of the same call without one (same bits).
// Searching takes tens of microseconds of host time, more than a launch: every thread remembers the plans of its last
// few hundred kinds of call.  A single call looks up one key, a grouped one some fifty (ten convolutions at seven tile sizes):
// eight ways a set, the least recently used one given up, so that a call does not drive out its own plans.  (With one way it
// nearly always did: ten 3x3 layers on five levels took 13 to 60 us to issue, by the chance of the hash, 14 now; finding a plan
// among eight ways takes such a call 1 us more than among one.)  A plan is a function of its key and of the device's cluster
// limits, which whoever plans for a device has had asked first (ensure_device): it does not matter which thread or context asks.
bool plan_tc(const PlanKey& k, TcPlan* out) {
    struct Memo {
        PlanKey key;
        TcPlan plan;
        unsigned hash;
        bool ok;
        unsigned long long used;   // when it was last asked for (0: empty)
    };
    constexpr int kSets = 64, kWays = 8;   // (fifty keys over the sets: nine in one are as good as never)
    static thread_local Memo memo[kSets][kWays];
    static thread_local unsigned long long asked = 0;
    unsigned h = 2166136261u;
    const int* w = reinterpret_cast<const int*>(&k);
    for (size_t i = 0; i < sizeof(PlanKey) / sizeof(int); ++i) h = (h ^ (unsigned)w[i]) * 16777619u;
    h ^= h >> 15;
    h *= 0x9E3779B1u;   // (sizes are multiples of something: the low bits alone repeat)
    Memo* set = memo[h >> 26];
    static_assert(kSets == 1 << (32 - 26), "the hash's upper bits name a set");
    int way = 0;
    while (way < kWays && !(set[way].used && set[way].hash == h && memcmp(&set[way].key, &k, sizeof(k)) == 0)) ++way;
    const bool known = way < kWays;
    for (int i = way = known ? way : 0; !known && i < kWays; ++i)
        if (set[i].used < set[way].used) way = i;
    Memo& m = set[way];
    if (!known) {
        m.used = 0;
        const bool pxm = k.ksize == 1 && k.Cout <= kPxmMaxCout && k.dtype != RTOSS_F32;
        if (k.shared || pxm) {
            m.ok = plan_search(k, k.resid != 0, 1, &m.plan);
        } else {
            int ks = 1;
            PlanKey q = k;
            // The tensor core cuts off at every accumulation, so the longer a sum, the larger its error.  fp32 layers whose small
            // products are bf16 ones are cut along K where three tf32 products would be: every sum then has two thirds of the
            // accumulations that those take, which is what makes up for the rounded factors.  Cut by the cost of the cheaper
            // instructions a layer is left in longer pieces: 96->360 @42x33 x3 in two shares instead of three errs by 3.6e-6
            // instead of the 3.3e-6 of three products, 128->128 @60x60 s2 x2 in two instead of four by 3.0e-6 instead of 2.7e-6.
            if (k.dtype == RTOSS_F32 && rtoss_f32_corr16(k.Cin, k.ksize)) q.three = 1;
            if (plan_search(q, true, 0, &m.plan)) ks = m.plan.KS;
            m.ok = plan_search(k, k.resid != 0, ks, &m.plan);
            if (m.ok && k.may_half) {
                // In two activation stages, cut along K as in one (the same sums): a second barrier round trip a block, which
                // launches of a few microseconds feel (2 to 6 % where every layer took it), against fetching under the
                // instructions.  The model has to expect 7 % and half a microsecond of it, which is about its own error; the
                // layers that gain are then those of several tiles a CTA (20 % and more; 60 layers of 16 to 512 channels, batch
                // 1 to 32, take 0.935 of the time in one stage in the geometric mean, the slowest 1.016).
                TcPlan two;
                q = k;
                q.half = 1;
                if (plan_search(q, k.resid != 0, ks, &two) && two.us < 0.93 * m.plan.us && two.us < m.plan.us - 0.5) {
                    two.us = m.plan.us;   // (by which calls are grouped, and that decides where sums are cut)
                    m.plan = two;
                }
            }
        }
        m.key = k;
        m.hash = h;
    }
    m.used = ++asked;
    *out = m.plan;
    return m.ok;
}

PlanKey plan_key(const rtoss_packed* p, const rtoss_conv_desc* d, int sms, int dev) {
    PlanKey k;
    memset(&k, 0, sizeof(k));
    k.N = d->N;
    k.Ho = (d->H - 1) / d->stride + 1;
    k.Wo = (d->W - 1) / d->stride + 1;
    k.ksize = p->ksize;
    k.S = d->stride;
    k.Cin = p->Cin;
    k.Cout = p->Cout;
    k.dtype = (int)p->dtype;
    k.resid = d->residual_dev ? 1 : 0;
    k.sms = sms;
    k.dev = dev;
    k.max_px = kMaxPx;
    k.n_tabs = 1;
    return k;
}

// A 1x1 convolution of stride 1 over channels-last images is one over a single row of N*H*W pixels, which can be cut into
// tiles of exactly as many positions as a tile takes: rows of 68, 80 or 272 pixels fill 204, 240 and 136 of 256 (bf16
// 256->1024 @50x68 x4 11.3 us instead of 11.7, the 38 such layers of the large detector at batch 4 11 us less; no layer slower).
rtoss_conv_desc row_form(const rtoss_packed* p, const rtoss_conv_desc* d) {
    rtoss_conv_desc dd = *d;
    if (p->ksize == 1 && d->stride == 1 && d->layout == RTOSS_NHWC && (long long)d->N * d->H * d->W <= 1ll << 30) {
        dd.W = d->N * d->H * d->W;
        dd.N = dd.H = 1;
    }
    return dd;
}

// Can the layer be cut at all?  Its smallest tile is one row of the narrowest segment, with a weight stage per tap.
bool plan_exists(const rtoss_packed* p, const rtoss_conv_desc* d) {
    const int S = d->stride, Wo = p->ksize == 1 && S == 1 && row_form(p, d).H == 1 ? 16 : (d->W - 1) / S + 1;
    const bool f32 = p->dtype == RTOSS_F32, k3 = p->ksize == 3;
    const int wq = (Wo + 15) / 16 + (k3 ? (S == 1 ? 2 : 1) : 0);
    if (wq > (S == 1 ? 256 : 128)) return false;
    const int rows = (k3 ? (S == 1 ? 3 : 2) : 1) * wq, shift = k3 ? (S == 1 ? 2 * wq + 2 : wq + 1) : 0;
    const int list = round_up(wq, 16) + shift > rows ? round_up(wq, 16) + shift : rows;
    const int need = use_pxm(p) ? shift + 256 : list;
    const int a_bytes = (k3 && S == 2 ? 4 : 1) * round_up(need, 8) * row_bytes_of(p) * (f32 ? 2 : 1);
    const int fixed = 1024 + 512 + kEpiWarps * kPatchBytes + kMaxPx * 8 + (d->residual_dev ? kEpiWarps * kResStage : 0);
    return a_bytes + 2 * kMTile * kRowBytes + fixed <= 227 * 1024 - 64;
}

// What one problem adds to a launch besides its TcArgs.
struct ProbPlan {
    TcPlan plan;
    int a_stage_bytes, b_stage_bytes, acc_cols;
};

// Geometry, operand roles and TMA descriptors of one convolution.  The rings' depths and the split along K are the
// launch's business (the caller's).  Returns a cudaError_t as int.
int build_problem(const rtoss_ctx* ctx, const rtoss_packed* p, const void* x, void* y, const rtoss_conv_desc* d, const PlanKey& plan_k,
                  TcArgs* out, ProbPlan* pp, CUtensorMap* tmA_out, CUtensorMap* tmB_out) {
    const int taps = p->ksize == 3 ? 9 : 1;
    const int S = d->stride;
    const int Ho = (d->H - 1) / S + 1, Wo = (d->W - 1) / S + 1;
    const int N_T = kMTile;
    TcPlan& plan = pp->plan;
    // narrow layers put the positions on the M operand (all 128 TMEM lanes carry outputs whatever Cout is)
    const bool pxm = use_pxm(p);
    const int w_rows = pxm ? round_up(p->Cout, 16) : kMTile;
    const bool f32 = p->dtype == RTOSS_F32;
    const int esize = f32 ? 4 : 2;
    const int row_bytes = row_bytes_of(p);
    if (!plan_tc(plan_k, &plan))
        return (int)cudaErrorInvalidConfiguration;

    TcArgs& a = *out;
    memset(&a, 0, sizeof(a));
    a.y = y;
    a.resid = d->residual_dev;
    a.resid_post = (d->residual_dev && d->residual_after_act) ? 1 : 0;
    a.bias = d->bias_dev;
    a.issue = p->ksize == 3 ? p->issue : nullptr;
    a.N = d->N;
    a.Ho = Ho;
    a.Wo = Wo;
    a.S = S;
    a.Cin = p->Cin;
    a.Cout = p->Cout;
    a.Wq = plan.Wq;
    a.TH = plan.TH;
    a.TW = plan.TW;
    a.taps = taps * (f32 ? 2 : 1);   // weight tiles per channel block: fp32 has the heads, then the remainders
    a.taps_real = taps;
    a.row_bytes = row_bytes;
    a.desc_hi = (unsigned)(make_sw_desc(0, row_bytes) >> 32);
    a.cb_ch = row_bytes / esize;
    a.tiles_x = plan.tiles_x;
    a.n_sub = plan.n_sub;
    if (plan.half) a.half = 1;   // (the launch writes the order here)
    a.sub_bytes = plan.sub_rows * row_bytes;
    if (p->ksize == 3 && S == 1) {
        a.x_add[0] = a.y_add[0] = -1;
        for (int t = 0; t < 9; ++t) a.tap_shift[t] = (t / 3) * plan.Wq + (t % 3);
    } else if (p->ksize == 3) {
        // sub-tile index = 2*(row parity) + (column parity); parity 0 = even input rows / columns
        for (int sub = 0; sub < 4; ++sub) {
            a.y_add[sub] = (sub >> 1) ? -1 : -2;
            a.x_add[sub] = (sub & 1) ? -1 : -2;
        }
        for (int t = 0; t < 9; ++t) {
            const int r = t / 3, c = t % 3;
            a.tap_sub[t] = (a.half ? 0 : 2 * (r == 1 ? 0 : 1)) + (c == 1 ? 0 : 1);   // (inside its stage)
            a.tap_shift[t] = (r == 0 ? 0 : 1) * plan.Wq + (c == 0 ? 0 : 1);
        }
    }
    a.N_px = plan.N_px;
    a.ncb = (p->Cin + a.cb_ch - 1) / a.cb_ch;
    a.tiles_y = (Ho + plan.TH - 1) / plan.TH;
    a.co_tiles = (p->Cout + N_T - 1) / N_T;
    a.lo_off = f32 ? plan.n_sub * plan.sub_rows * row_bytes : 0;
    pp->a_stage_bytes = plan.n_sub * plan.sub_rows * row_bytes * (f32 ? 2 : 1);
    a.w_rows = w_rows;
    // narrow 3x3 layers keep the filters on M and repeat them down the 128 rows of the tile
    const rtoss_wtc_layout lay = rtoss_wtc_layout_of(p->Cout, p->Cin, p->ksize, p->dtype);  // how rtoss_pack laid the weights out
    a.rep_rows = lay.copies > 1 ? lay.rep_rows : 128;
    a.R = lay.copies;
    a.rep_shift = a.rep_rows == 32 ? 5 : a.rep_rows == 64 ? 6 : 7;
    pp->b_stage_bytes = plan.G * w_rows * row_bytes;
    a.G = plan.G;
    pp->acc_cols = round_up(plan.N_px, 32);  // the epilogue reads 32 columns at a time
    a.a_tx_bytes = (unsigned)(row_bytes * plan.Wq * plan.rows_staged);  // per sub-tile
    a.b_tx_bytes = (unsigned)(row_bytes * w_rows);
    a.act = (int)d->act;
    a.y_c_off = d->y_channel_offset;
    const int cs = d->y_channel_stride ? d->y_channel_stride : p->Cout;   // channels of the output tensor
    a.nchw = d->layout == RTOSS_NCHW ? 1 : 0;   // (of the output: x is channels last here, see rtoss_launch_conv_tc_repacked)
    a.y_c_stride = a.nchw ? 1 : cs;
    a.y_co = a.nchw ? Ho * Wo : 1;
    a.y_img = (long long)cs * Ho * Wo;
    a.is_bf16 = p->dtype == RTOSS_BF16;
    // instruction descriptor: fp32 accumulate, A and B of the io type (f16 0, bf16 1; kind::tf32: tf32 2), both K-major,
    // N/8 and M/16
    const unsigned fmt = f32 ? 2u : a.is_bf16 ? 1u : 0u;
    a.idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((unsigned)(plan.N_px >> 3) << 17) | ((unsigned)(kMTile >> 4) << 24);
    if (has_corr16(p)) a.idesc16 = (a.idesc & ~((7u << 7) | (7u << 10))) | (1u << 7) | (1u << 10);   // (bf16)
    a.pxm = pxm ? 1 : 0;
    a.MH = plan.N_px > 128 ? 2 : 1;
    a.n_cols = round_up(p->Cout, 16);
    if (pxm) {
        pp->acc_cols = round_up(a.MH * a.n_cols, 32);
        a.idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((unsigned)(a.n_cols >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
    }
    a.KS = 1;
    a.cb_per = a.ncb;
    magic_of(a.KS, a.div_ks);
    magic_of(pxm ? 1 : a.co_tiles, a.div_co);   // (positions on M: one filter tile covers the layer)
    magic_of(a.tiles_x, a.div_tx);
    magic_of(a.tiles_y, a.div_ty);

    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return (int)cudaErrorNotSupported;
    // The driver encodes for the thread's current context, and a thread that has made no runtime call yet has none.
    auto bind_context = [&] { return (int)cudaSetDevice(ctx->device); };
    const CUtensorMapDataType dt = f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : a.is_bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    std::lock_guard<std::mutex> hold(g_maps);
    // activations: descriptor cached per (pointer, shape, box)
    const int key[7] = {d->N, d->H, d->W, p->Cin, plan.rows_staged * 8 + S, plan.Wq * 4 + (int)p->dtype, d->x_channel_stride};   // (row size: a function of Cin and dtype)
    rtoss_tmap_entry* ea = nullptr;
    for (rtoss_tmap_entry& e : ctx->tmap_cache)
        if (e.valid && e.base == x && memcmp(e.dims, key, sizeof(key)) == 0) ea = &e;
    if (!ea) {
        ea = &ctx->tmap_cache[ctx->tmap_next];
        ctx->tmap_next = (ctx->tmap_next + 1) % 32;
        const cuuint64_t cin_p = (cuuint64_t)lay.cin_p;   // (the caller's tensor: cin_p == Cin)
        const cuuint64_t cp = d->x_channel_stride ? (cuuint64_t)d->x_channel_stride : cin_p;   // pixels are cp channels apart
        cuuint64_t dims[4] = {cin_p, (cuuint64_t)d->W, (cuuint64_t)d->H, (cuuint64_t)d->N};
        cuuint64_t strides[3] = {cp * esize, (cuuint64_t)d->W * cp * esize, (cuuint64_t)d->H * d->W * cp * esize};
        // with element strides the box is counted in traversed elements: S*n covers n fetched pixels
        cuuint32_t box[4] = {(cuuint32_t)a.cb_ch, (cuuint32_t)(plan.Wq * S), (cuuint32_t)(plan.rows_staged * S), 1};
        cuuint32_t es[4] = {1, (cuuint32_t)S, (cuuint32_t)S, 1};
        ea->valid = 0;
        if (const int e = bind_context()) return e;
        CUresult r = enc(reinterpret_cast<CUtensorMap*>(ea->map), dt, 4, const_cast<void*>(x), dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return (int)cudaErrorInvalidValue;
        ea->base = x;
        memcpy(ea->dims, key, sizeof(key));
        ea->valid = 1;
    }
    // weights: one descriptor per handle
    rtoss_tmap_entry* eb = &p->wtc_map;
    if (!eb->valid || eb->base != p->wtc || eb->dims[0] != w_rows || eb->dims[1] != plan.G) {
        cuuint64_t dims[3] = {(cuuint64_t)lay.cin_p, (cuuint64_t)lay.rows, (cuuint64_t)a.taps};
        cuuint64_t strides[2] = {(cuuint64_t)lay.cin_p * esize, (cuuint64_t)lay.rows * lay.cin_p * esize};
        cuuint32_t box[3] = {(cuuint32_t)a.cb_ch, (cuuint32_t)w_rows, (cuuint32_t)plan.G};  // a weight stage is one copy
        cuuint32_t es[3] = {1, 1, 1};
        eb->valid = 0;
        if (const int e = bind_context()) return e;
        CUresult r = enc(reinterpret_cast<CUtensorMap*>(eb->map), dt, 3, p->wtc, dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return (int)cudaErrorInvalidValue;
        eb->base = p->wtc;
        eb->dims[0] = w_rows;
        eb->dims[1] = plan.G;
        eb->valid = 1;
    }
    memcpy(tmA_out, ea->map, sizeof(CUtensorMap));
    memcpy(tmB_out, eb->map, sizeof(CUtensorMap));
    return 0;
}

typedef void (*SingleKernel)(const TcLaunch1);
void* form_kernel(const rtoss_ctx*, bool bf16, bool shared, int form) { return bf16 ? rtoss_tc_form_bf16(form, shared) : rtoss_tc_form_f16(form, shared); }
int rtoss_tc_prepare_forms(bool bf16) { return bf16 ? rtoss_tc_prepare_forms_bf16() : rtoss_tc_prepare_forms_f16(); }
int ctx_sms(const rtoss_ctx* ctx) { return ctx->sm_count > 0 ? ctx->sm_count : 148; }
int ctx_dev(const rtoss_ctx* ctx) { return ctx->device >= 0 && ctx->device < 64 ? ctx->device : -1; }
// Once per device: every instantiation may use up to the whole shared memory of an SM (the attribute belongs to the
// (function, device) pair), and the planner learns how many clusters fit.
int ensure_device(const rtoss_ctx* ctx) {
    static std::atomic<bool> attr_set[64];
    const int dev_slot = ctx_dev(ctx);
    if (dev_slot < 0 || !attr_set[dev_slot].load(std::memory_order_acquire)) {
        cudaError_t e = cudaFuncSetAttribute(conv_tc_kernel<__nv_bfloat16, TcLaunch1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<__half, TcLaunch1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<__nv_bfloat16, TcLaunchN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<__half, TcLaunchN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<float, TcLaunch1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<float, TcLaunch1, false, kFormCorr>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<float, TcLaunchN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<__nv_bfloat16, TcLaunch1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<__half, TcLaunch1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return (int)e;
        for (int i = 0; i < 2; ++i) {
            e = (cudaError_t)rtoss_tc_prepare_forms(i == 0);
            if (e != cudaSuccess) return (int)e;
        }
        // how many clusters of each size the device holds at once (one CTA of this kernel per SM)
        for (int ks = 2; ks <= 8 && dev_slot >= 0; ++ks) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(ctx_sms(ctx) / ks * ks));
            cfg.blockDim = dim3(kTcThreads);
            cfg.dynamicSmemBytes = 116 * 1024;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)ks;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, conv_tc_kernel<__nv_bfloat16, TcLaunch1>, &cfg) == cudaSuccess && n > 0)
                g_max_clusters[dev_slot][ks].store(n, std::memory_order_relaxed);
            else
                cudaGetLastError();
        }
        if (dev_slot >= 0) attr_set[dev_slot].store(true, std::memory_order_release);
    }
    return 0;
}

template <typename G>
void launch_common(const rtoss_ctx* ctx, G* g) {
    g->status = ctx->dev_status;
    g->wait_cycles = ctx->wait_cycles > 0 ? ctx->wait_cycles : kWaitCycles;
    g->inject = 0;
    g->AS = 2;
    int alloc = 32;
    while (alloc < g->AS * g->acc_stride) alloc <<= 1;
    g->tmem_cols = alloc;
}

}  // namespace

// Handles that get weights for the tensor path: 16-bit ones (rows padded to 16 bytes), fp32 ones whose rows are multiples
// of 16 bytes as they are.
bool rtoss_tc_weights_eligible(const rtoss_packed* p) { return p->dtype != RTOSS_F32 || p->Cin % 4 == 0; }
// Layers whose channels-last activations TMA can read where they lie.
static bool rows_fit_tma(const rtoss_packed* p) { return p->Cin % (p->dtype == RTOSS_F32 ? 4 : 8) == 0; }

// Can this call run on the tensor path?  (rtoss_tc_takes: by its sizes, types and alignment; no device is asked.)
bool rtoss_tc_takes(const rtoss_packed* p, const rtoss_conv_desc* d, const void* x, const void* y) {
    if (!p->wtc || !rows_fit_tma(p)) return false;
    if (d->layout != RTOSS_NHWC || (int)d->io_dtype != (int)p->dtype) return false;
    if ((reinterpret_cast<uintptr_t>(x) & 15) || (reinterpret_cast<uintptr_t>(y) & 15)) return false;
    if (d->x_channel_stride % (p->dtype == RTOSS_F32 ? 4 : 8) != 0) return false;   // a slice: the pitch as TMA wants it
    // a residual operand: 16-byte aligned, and not for the positions-as-M form (narrow 1x1 layers)
    if (d->residual_dev && (use_pxm(p) || (reinterpret_cast<uintptr_t>(d->residual_dev) & 15))) return false;
    return plan_exists(p, d);
}
bool rtoss_tc_eligible(const rtoss_packed* p, const rtoss_conv_desc* d, const void* x, const void* y) {
    return rtoss_tc_takes(p, d, x, y) && encode_fn();
}

// May this call be one of several in a launch?  (Tensor path with the filters on M.)
bool rtoss_tc_groupable(const rtoss_packed* p, const rtoss_conv_desc* d, const void* x, const void* y) {
    return !use_pxm(p) && rtoss_tc_eligible(p, d, x, y);
}

// What one shared launch is expected to take for these independent calls, and the most positions a tile should have: many
// small tiles where the set would leave SMs idle, 256 positions where it fills them for several rounds.
static double shared_cost(const rtoss_ctx* ctx, int n, const rtoss_packed* const* ps, const rtoss_conv_desc* const* ds, bool three, int* px_out) {
    static const int kPx[] = {256, 192, 128, 96, 64, 48, 32};
    const int sms = ctx_sms(ctx);
    double best = 1e30;
    for (int px : kPx) {
        double work = 0, longest = 0, epi = 0;
        long tiles = 0;
        bool ok = true;
        for (int i = 0; i < n && ok; ++i) {
            const rtoss_conv_desc dd = row_form(ps[i], ds[i]);
            PlanKey key = plan_key(ps[i], &dd, sms, ctx_dev(ctx));
            key.shared = n > 1 ? 1 : 2;
            key.max_px = px;
            key.three = three && has_corr16(ps[i]) ? 1 : 0;
            TcPlan plan;
            ok = plan_tc(key, &plan);
            if (!ok) break;
            const double t = plan.tile_us > plan.epi_us ? plan.tile_us : plan.epi_us;
            work += (double)plan.tiles * t;
            tiles += plan.tiles;
            if (t > longest) longest = t;
            if (plan.epi_us > epi) epi = plan.epi_us;
        }
        if (!ok) continue;
        // (3.4 us: launch, parameters of many problems, first operands; past one round a CTA may draw half a tile more than its share)
        const double us = 3.4 + epi + (tiles <= sms ? longest : work / sms + 0.5 * longest);
        if (us < 0.97 * best) {
            best = us;
            if (px_out) *px_out = px;
        }
    }
    return best;
}
// (Whether calls share a launch decides where sums are cut: fp32 by the cost of three tf32 products, see plan_tc.)
double rtoss_tc_shared_cost(const rtoss_ctx* ctx, int n, const rtoss_packed* const* ps, const rtoss_conv_desc* const* ds) {
    if (ensure_device(ctx)) return 1e30;   // (the launch that follows reports the error)
    return shared_cost(ctx, n, ps, ds, true, nullptr);
}

// The plan key of a launch of one convolution: 16-bit 3x3 layers of stride 2 may have their channel blocks in two activation
// stages.  Only where there is a form for it: whole 16-byte pieces out, no residual operand.
static PlanKey single_plan_key(const rtoss_packed* p, const rtoss_conv_desc* d, int sms, int dev) {
    PlanKey k = plan_key(p, d, sms, dev);
    const int cs = d->y_channel_stride ? d->y_channel_stride : p->Cout;
    const bool pieces = d->layout == RTOSS_NCHW || (p->Cout % 8 == 0 && cs % 8 == 0 && d->y_channel_offset % 8 == 0);
    k.may_half = p->ksize == 3 && d->stride == 2 && p->dtype != RTOSS_F32 && pieces && !d->residual_dev ? 1 : 0;
    return k;
}
// TcArgs::half for NA stages: a block's odd rows are read until its end, its even rows for two thirds of it, and a stage is
// filled again by whatever comes next once it is free.  With two stages the odd and the even rows change places from block
// to block; with three the even rows keep theirs; with four a block has a pair.
static unsigned half_order(int NA) { return NA == 2 ? 0u | 1u << 2 | 1u << 4 | 0u << 6 : NA == 3 ? 0u | 1u << 2 | 2u << 4 | 1u << 6 : 0u | 1u << 2 | 2u << 4 | 3u << 6; }

// What a launch of its own is expected to take for this call (the planner's model), over how many CTAs it spreads a tile's
// channel blocks, and how many tiles it has.  (Shared launches never split.)
bool rtoss_tc_single_cost(const rtoss_ctx* ctx, const rtoss_packed* p, const rtoss_conv_desc* d, double* us, int* ks, long* tiles) {
    TcPlan plan;
    const rtoss_conv_desc dd = row_form(p, d);
    if (ensure_device(ctx)) return false;
    PlanKey k = single_plan_key(p, &dd, ctx_sms(ctx), ctx_dev(ctx));
    k.three = has_corr16(p) ? 1 : 0;
    if (!plan_tc(k, &plan)) return false;
    *us = plan.us;
    *ks = plan.KS;
    *tiles = plan.tiles;
    return true;
}

// Weights that fit beside three activation stages (or the plan's own number) stay in shared memory while a CTA walks its tiles:
// bf16 1x1 64->64 @160x160 x16 24.7 -> 23.7 us, 128->512 @100x136 x4 16.2 -> 15.9, 3x3 24->24 @100x100 x16 (rows of 48 bytes, which
// weight copies take slowly) 30.2 -> 15.9; with two stages 512->256 @100x136 x4 16.4 -> 22.4.
// stages: weight stages of a tile; ct: filter tiles.  Gives the activation stages and the CTAs (a multiple of ct: each keeps its
// filter tile from tile to tile).
static bool resident_rings(const TcPlan& plan, int a_stage, int b_stage, int stages, int ct, size_t units, int sms, int* na, unsigned* ctas) {
    const int fixed = plan.smem - plan.NA * a_stage - plan.NB * b_stage, room = (227 * 1024 - 64 - fixed - stages * b_stage) / a_stage;
    const unsigned grid = (unsigned)(units < (size_t)sms ? units : (size_t)sms), even = grid - grid % (unsigned)ct;
    *na = room < kMaxA ? room : kMaxA;
    *ctas = even;
    return stages <= kMaxB && *na >= 2 && (*na >= 3 || *na >= plan.NA) && even > 0 && units > (size_t)even && (units + even - 1) / even == (units + grid - 1) / grid;
}

extern "C" rtoss_status rtoss_tensor_plan_of(const rtoss_conv_desc* d, int ksize, int Cin, int Cout, rtoss_dtype dtype, int sm_count,
                                            rtoss_tensor_plan* out) {
    if (!d || !out || (ksize != 1 && ksize != 3) || Cin < 1 || Cout < 1 || (int)dtype < 0 || (int)dtype > 2 || d->N < 1 || d->H < 1 ||
        d->W < 1 || (d->stride != 1 && d->stride != 2))
        return RTOSS_ERR_INVALID_ARG;
    memset(out, 0, sizeof(*out));
    rtoss_packed fake;
    memset(&fake, 0, sizeof(fake));
    fake.Cin = Cin, fake.Cout = Cout, fake.ksize = ksize, fake.dtype = dtype;
    const rtoss_packed* p = &fake;
    if (!rows_fit_tma(p) || d->layout != RTOSS_NHWC) return RTOSS_OK;   // (eligible stays 0)
    const int sms = sm_count > 0 ? sm_count : 148;
    const bool pxm = use_pxm(p), f32 = dtype == RTOSS_F32;
    const int w_rows = pxm ? round_up(Cout, 16) : kMTile;
    const int row_bytes = row_bytes_of(p);
    TcPlan plan;
    const rtoss_conv_desc row = row_form(p, d);
    if (!plan_tc(single_plan_key(p, &row, sms, -1), &plan)) return RTOSS_OK;
    out->eligible = 1;
    out->rows_per_tile = plan.TH, out->cols_per_tile = plan.TW, out->pitch = plan.Wq, out->positions = plan.N_px;
    out->act_stages = plan.NA, out->weight_stages = plan.NB, out->taps_per_weight_stage = plan.G;
    out->row_bytes = row_bytes;
    out->act_stage_bytes = plan.n_sub * plan.sub_rows * row_bytes * (f32 ? 2 : 1);
    out->weight_stage_bytes = plan.G * w_rows * row_bytes;
    out->staged_rows = plan.rows_staged, out->sub_tiles = ksize == 3 && d->stride == 2 ? 4 : 1;
    out->shared_bytes = plan.smem;
    out->positions_on_m = pxm ? 1 : 0;
    out->tiles = (int)(plan.tiles > 0x7FFFFFFF ? 0x7FFFFFFF : plan.tiles);
    out->split_k = plan.KS;
    if (plan.KS == 1) {
        const int stages = ncb_of(p) * ((ksize == 3 ? 9 : 1) * (f32 ? 2 : 1) / plan.G);
        int na;
        unsigned ctas;
        if (resident_rings(plan, out->act_stage_bytes, out->weight_stage_bytes, stages, pxm ? 1 : (Cout + kMTile - 1) / kMTile, (size_t)plan.tiles, sms, &na, &ctas)) {
            out->shared_bytes += (na - plan.NA) * out->act_stage_bytes + (stages - plan.NB) * out->weight_stage_bytes;
            out->act_stages = na, out->weight_stages = stages;
        }
    }
    return RTOSS_OK;
}

static int threads_of(bool f32) { return f32 ? kThreadsOf<float> : kThreadsOf<__half>; }

// The kernel a launch of one convolution runs: a form where there is one for it, else the general one.
static SingleKernel single_kernel(const rtoss_ctx* ctx, bool f32, bool repacked, const TcArgs& a) {
    if (!f32 && (a.taps == 1 || a.G == 3)) {
        const bool pieces = a.pxm || a.nchw || (a.y_c_stride % 8 == 0 && a.y_c_off % 8 == 0 && a.Cout % 8 == 0);
        const int form = (pieces ? 0 : kFormElem) | (a.half ? kFormHalf : 0) | form_of(a.taps == 9 ? 3 : a.pxm ? 2 : 1, a.act, a.KS > 1, a.resid ? 1 + a.resid_post : 0, a.nchw != 0);
        if (void* k = form_kernel(ctx, a.is_bf16, false, form)) return reinterpret_cast<SingleKernel>(k);
    }
    if (!f32 && a.half) return nullptr;   // (forms only; single_plan_key asks for what they cover)
    if (f32) return a.idesc16 ? conv_tc_kernel<float, TcLaunch1, false, kFormCorr> : conv_tc_kernel<float, TcLaunch1>;
    if (repacked) return a.is_bf16 ? conv_tc_kernel<__nv_bfloat16, TcLaunch1, true> : conv_tc_kernel<__half, TcLaunch1, true>;
    return a.is_bf16 ? conv_tc_kernel<__nv_bfloat16, TcLaunch1> : conv_tc_kernel<__half, TcLaunch1>;
}

// The kernel of a shared launch: a form where its members agree on what they are.
typedef void (*SharedKernel)(const TcLaunchN);
static SharedKernel shared_kernel(const rtoss_ctx* ctx, bool f32, const TcLaunchN& g) {
    if (!f32) {
        int kind = 0, act = -2, res = -2;
        bool one = true;
        for (int i = 0; i < g.n_prob && one; ++i) {
            const TcArgs& a = g.prob[i];
            const int k = a.taps == 9 ? (a.G == 3 ? 3 : 0) : a.pxm ? 0 : 1, r = a.resid ? 1 + a.resid_post : 0;
            one = k != 0 && (i == 0 || k == kind) && !a.nchw && a.y_c_stride % 8 == 0 && a.y_c_off % 8 == 0 && a.Cout % 8 == 0;
            kind = k;
            act = i == 0 || act == a.act ? a.act : -1;
            res = i == 0 || res == r ? r : 3;
        }
        // (a residual is a run-time choice of the members: the form for it takes any)
        if (one && res != 0) act = -1, res = 3;
        if (one && res != 3)
            if (void* k = form_kernel(ctx, g.prob[0].is_bf16, true, form_of(kind, act, false, res, false))) return reinterpret_cast<SharedKernel>(k);
        return g.prob[0].is_bf16 ? conv_tc_kernel<__nv_bfloat16, TcLaunchN> : conv_tc_kernel<__half, TcLaunchN>;
    }
    return conv_tc_kernel<float, TcLaunchN>;
}

// Filter tiles of a problem (the positions on M: one covers the layer).
static int pxm_tiles(const TcArgs& a) { return a.pxm ? 1 : a.co_tiles; }

// One convolution, channels last in x.  repacked: x is the copy of rtoss_launch_conv_tc_repacked.
static int launch_single(const rtoss_ctx* ctx, const rtoss_packed* p, const void* x, void* y, const rtoss_conv_desc* call, bool repacked,
                         void* stream) {
    const rtoss_conv_desc row = row_form(p, call);
    const rtoss_conv_desc* d = &row;
    const int sms = ctx_sms(ctx);
    int e = ensure_device(ctx);
    if (e) return e;
    static thread_local TcLaunch1 g;   // several KB: kept off the stack
    ProbPlan pp;
    g.n_prob = 1;
    PlanKey key = single_plan_key(p, d, sms, ctx_dev(ctx));
    if (ctx->inject_next) key.sms = 1;   // (failure-detection hook: as few CTAs as the layer allows)
    e = build_problem(ctx, p, x, y, d, key, &g.prob[0], &pp, &g.tmA[0], &g.tmB[0]);
    if (e) return e;
    TcArgs& a = g.prob[0];
    if (repacked && a.act == RTOSS_ACT_SILU) a.act = kActSiluX;
    const TcPlan& plan = pp.plan;
    const bool f32 = p->dtype == RTOSS_F32;
    a.NA = plan.NA;
    a.NB = plan.NB;
    a.a_stage = (unsigned)pp.a_stage_bytes;
    a.b_stage = (unsigned)pp.b_stage_bytes;
    a.sB_off = (unsigned)plan.NA * a.a_stage;
    const int rings = (int)(a.sB_off + (unsigned)plan.NB * a.b_stage);
    g.res_off = rings;   // the staging of a residual operand lies behind the rings
    g.ring_bytes = rings + (d->residual_dev ? kEpiWarps * kResStage : 0);
    g.max_na = plan.NA;
    g.max_nb = plan.NB;
    g.n_tabs = 1;
    g.done = nullptr;
    g.acc_stride = pp.acc_cols;
    launch_common(ctx, &g);
    a.KS = plan.KS;
    a.cb_per = plan.cb_per;
    magic_of(a.KS, a.div_ks);
    size_t n_units = (size_t)d->N * a.tiles_y * a.tiles_x * a.co_tiles * a.KS;
    if (ctx->inject_next) {
        // failure-detection hook: honoured by a launch of one CTA only (every role of that CTA then runs into its
        // bounded wait and leaves through the normal exit)
        ctx->inject_next = 0;
        if (n_units != 1) return (int)cudaErrorNotSupported;
        g.inject = 1;
    }
    g.unit_end[0] = (int)n_units;
    dim3 grid((unsigned)(n_units < (size_t)sms ? n_units : (size_t)sms));
    int smem_need = plan.smem;
    if (a.KS == 1) {
        const int stages = a.ncb * (a.taps / a.G);
        int na;
        unsigned even;
        if (resident_rings(plan, (int)a.a_stage, (int)a.b_stage, stages, pxm_tiles(a), n_units, sms, &na, &even)) {
            a.resident = 1;
            grid.x = even;
            smem_need = plan.smem + (na - plan.NA) * (int)a.a_stage + (stages - plan.NB) * (int)a.b_stage;
            a.NA = na;
            a.NB = stages;
            a.sB_off = (unsigned)a.NA * a.a_stage;
            const int rings = (int)(a.sB_off + (unsigned)a.NB * a.b_stage);
            g.res_off = rings;
            g.ring_bytes = rings + (d->residual_dev ? kEpiWarps * kResStage : 0);
            g.max_na = a.NA;
            g.max_nb = a.NB;
        }
    }
    if (!f32 && a.half) a.half = half_order(a.NA);
    SingleKernel kernel = single_kernel(ctx, f32, repacked, a);
    if (!kernel) return (int)cudaErrorInvalidDeviceFunction;
    // at least half an SM's shared memory, so that a second CTA (which would wait for TMEM) never shares the SM
    const size_t smem = (size_t)(smem_need > 116 * 1024 ? smem_need : 116 * 1024);
    cudaError_t le;
    if (a.KS > 1) {
        // one cluster per tile; if the device cannot place the clusters the layer runs uncut
        le = rtoss_dev::launch_pdl(kernel, grid, threads_of(f32), smem, (cudaStream_t)stream, a.KS, g);
        if (le == cudaSuccess) return 0;
        cudaGetLastError();
        a.KS = 1;
        magic_of(a.KS, a.div_ks);
        a.cb_per = a.ncb;
        n_units = (size_t)d->N * a.tiles_y * a.tiles_x * a.co_tiles;
        g.unit_end[0] = (int)n_units;
        grid = dim3((unsigned)(n_units < (size_t)sms ? n_units : (size_t)sms));
        kernel = single_kernel(ctx, f32, repacked, a);   // (uncut: another form)
        if (!kernel) return (int)cudaErrorInvalidDeviceFunction;
    }
    le = rtoss_dev::launch_pdl(kernel, grid, threads_of(f32), smem, (cudaStream_t)stream, 1, g);
    return (int)le;
}

int rtoss_launch_conv_tc(const rtoss_ctx* ctx, const rtoss_packed* p, const void* x, void* y, const rtoss_conv_desc* d,
                         void* stream) {
    return launch_single(ctx, p, x, y, d, false, stream);
}

// The calls the tensor path takes behind a pass that lays x out for it (repack.cu): 16-bit data in NCHW, or channels last
// with pixels of no multiple of 16 bytes.  What then runs: 1x1 layers of stride 2 keep only the pixels they read and
// become layers of stride 1.  Three-channel stems stay with their own kernel (conv3x3_small_cin_kernel), which reads the
// image once and has next to nothing to contract.
static rtoss_conv_desc repacked_desc(const rtoss_packed* p, const rtoss_conv_desc* d) {
    rtoss_conv_desc dd = *d;
    dd.x_channel_stride = 0;   // (of the copy)
    if (p->ksize == 1 && d->stride == 2) {
        dd.H = (d->H - 1) / 2 + 1;
        dd.W = (d->W - 1) / 2 + 1;
        dd.stride = 1;
    }
    return dd;
}
static bool x_is_slice(const rtoss_packed* p, const rtoss_conv_desc* d) { return d->x_channel_stride && d->x_channel_stride != p->Cin; }
bool rtoss_tc_takes_repacked(const rtoss_packed* p, const rtoss_conv_desc* d) {
    if (d->path != RTOSS_PATH_AUTO || d->residual_dev || x_is_slice(p, d) || !p->wtc || p->dtype == RTOSS_F32 || (int)d->io_dtype != (int)p->dtype) return false;
    if (d->layout == RTOSS_NHWC && rows_fit_tma(p)) return false;   // (native, or declined for another reason)
    if (p->ksize == 3 && p->Cin <= 4) return false;
    const rtoss_conv_desc dd = repacked_desc(p, d);
    // (the pass counts its pieces, and its blocks, with 31 bits: copies of up to 32 GiB)
    if ((long long)dd.N * dd.H * dd.W > 0x7FFFFFFFLL / (rtoss_cin_pitch(p->Cin, p->dtype) / 8)) return false;
    return plan_exists(p, &dd);
}
bool rtoss_tc_repack_eligible(const rtoss_packed* p, const rtoss_conv_desc* d) { return rtoss_tc_takes_repacked(p, d) && encode_fn(); }
// Returns a cudaError_t, or -1 when there was no memory for the channels-last copy (nothing was launched).  The copy
// lives from here to the end of the convolution in the stream's order, in the context's pool: any number of streams and
// threads may be in such a call.  Inside a stream capture the copy belongs to the graph (rtoss_copy_get).
int rtoss_launch_conv_tc_repacked(const rtoss_ctx* ctx, const rtoss_packed* p, const void* x, void* y, const rtoss_conv_desc* d,
                                  void* stream) {
    const rtoss_conv_desc dd = repacked_desc(p, d);
    const int cp = rtoss_cin_pitch(p->Cin, p->dtype), S = dd.stride == d->stride ? 1 : 2;
    bool of_graph = false;
    size_t bytes = (size_t)dd.N * dd.H * dd.W * cp * 2;
    void* ws = rtoss_copy_get(ctx, &bytes, stream, &of_graph);
    if (!ws) return -1;
    int e = rtoss_launch_repack16(x, ws, dd.N, p->Cin, cp, d->H, d->W, S, d->layout, stream);
    if (!e) e = launch_single(ctx, p, ws, y, &dd, true, stream);
    if (of_graph) {
        if (!e) rtoss_copy_read(ws, bytes, stream);
        return e;
    }
    const cudaError_t fe = cudaFreeAsync(ws, (cudaStream_t)stream);
    return e ? e : (int)fe;
}

// Several convolutions in ONE launch: independent ones side by side, dependent ones one behind the other.
//
// after[i] (null: none depends on another) has bit j set when convolution i must see convolution j (j < i) complete:
// it reads what j writes, or overwrites what j reads or writes.  The kernel then keeps the CTAs that reach a tile of
// i waiting until every CTA has reported its tiles of j done (a counter per problem in device memory; the waits are
// bounded like all others).  That is only sound when all CTAs of the launch are on the device together: the grid is at
// most one CTA per SM, and nothing else may hold SMs forever while such a launch runs.
//
// All convolutions must qualify for the tensor path with the filters on M and share the data type; at most kMaxProb.
// They are sorted into levels (a convolution's level is one more than the highest level it waits for); the
// convolutions of a level with the same kernel size (and stride class, for 3x3) share one ring layout, planned as the
// grouped launches always were; a CTA that passes from one layout to another lets its rings run empty in between.
// Returns 0 after a launch, -1 when the set cannot share a launch (nothing was launched: the caller runs the calls
// one by one, in order), or a cudaError_t.
int rtoss_launch_conv_tc_chain(const rtoss_ctx* ctx, int n, const rtoss_packed* const* ps, const void* const* xs, void* const* ys,
                               const rtoss_conv_desc* const* ds, const uint32_t* after, void* stream) {
    if (n < 2 || n > kMaxProb || ctx->inject_next) return -1;
    const int sms = ctx_sms(ctx);
    const int e0 = ensure_device(ctx);
    if (e0) return e0;
    bool resid = false, chained = false;
    int level[kMaxProb], cls[kMaxProb];
    for (int i = 0; i < n; ++i) {
        if (use_pxm(ps[i]) || ps[i]->dtype != ps[0]->dtype) return -1;
        if (!rtoss_tc_eligible(ps[i], ds[i], xs[i], ys[i])) return -1;
        resid = resid || ds[i]->residual_dev != nullptr;
        level[i] = 0;
        if (after && after[i]) {
            if (i == 0 || (after[i] >> i)) return (int)cudaErrorInvalidValue;   // only earlier convolutions may be named
            chained = true;
            for (int j = 0; j < i; ++j)
                if ((after[i] >> j) & 1u) level[i] = level[j] + 1 > level[i] ? level[j] + 1 : level[i];
        }
        cls[i] = ps[i]->ksize == 3 ? 3 + ds[i]->stride : 1;   // 1x1 (any stride), 3x3 stride 1, 3x3 stride 2
    }
    if (chained && !ctx->chain_done) return -1;
    static thread_local TcLaunchN g;
    static thread_local TcArgs args[kMaxProb];
    static thread_local CUtensorMap mapA[kMaxProb], mapB[kMaxProb];
    ProbPlan pp[kMaxProb];
    long n_tiles[kMaxProb];
    int geo_of[kMaxProb];
    struct Geo {
        int a, b, na, nb;
        bool under;   // planned below the staging area of residual operands
    } geos[kMaxProb];
    int n_geo = 0, acc_max = 0, n_tabs_planned = 0;
    const int cap = 227 * 1024 - 64;
    const int res_bytes = resid ? kEpiWarps * kResStage : 0;
    // Shared memory outside the rings: alignment slack, barriers, epilogue patches, the position tables.  How many
    // tables the launch needs is known once every problem is planned: planned with four first, with kMaxTabs if that
    // was too few.
    for (int tabs_try = 4; tabs_try <= kMaxTabs; tabs_try += kMaxTabs - 4) {
        const int fixed = 1024 + 512 + kEpiWarps * kPatchBytes + tabs_try * kMaxPx * 8;
        bool seen[kMaxProb] = {};
        n_geo = acc_max = 0;
        for (int i0 = 0; i0 < n; ++i0) {
            if (seen[i0]) continue;
            // the set of this convolution: same level, same class
            int set[kMaxProb], m = 0;
            bool set_res = false;
            for (int j = i0; j < n; ++j)
                if (!seen[j] && level[j] == level[i0] && cls[j] == cls[i0]) set[m++] = j, seen[j] = true, set_res = set_res || ds[j]->residual_dev;
            // The staging area of residual operands is the top end of the ring area.  A set of 3x3 convolutions none of
            // which has a residual operand may lay its rings over it (the kernel then lets the epilogues that use the
            // area finish first); every other set stays below it.
            const bool under = resid && (set_res || ps[i0]->ksize != 3);
            // every problem is planned on its own first; where they disagree on the taps per weight stage, all are
            // planned again with the smallest (a stage per tap fits whatever fits three)
            int force_G = 0, a_max = 0, b_bytes = 0, set_px = kMaxPx;
            if (m > 1) {
                const rtoss_packed* sp[kMaxProb];
                const rtoss_conv_desc* sd[kMaxProb];
                for (int q = 0; q < m; ++q) sp[q] = ps[set[q]], sd[q] = ds[set[q]];
                shared_cost(ctx, m, sp, sd, false, &set_px);
            }
            for (int pass = 0; pass < 2; ++pass) {
                bool agree = true;
                int g_min = 9;
                a_max = 0;
                for (int q = 0; q < m; ++q) {
                    const int i = set[q];
                    rtoss_conv_desc dd = row_form(ps[i], ds[i]);
                    static const int dummy = 0;
                    dd.residual_dev = under ? &dummy : nullptr;   // (only the plan's memory budget looks at it here)
                    PlanKey key = plan_key(ps[i], &dd, sms, ctx_dev(ctx));
                    key.shared = m > 1 ? 1 : 2;
                    key.max_px = set_px;
                    key.force_G = force_G;
                    key.n_tabs = tabs_try;
                    int e = build_problem(ctx, ps[i], xs[i], ys[i], &dd, key, &args[i], &pp[i], &mapA[i], &mapB[i]);
                    if (e == (int)cudaErrorInvalidConfiguration) return -1;
                    if (e) return e;
                    args[i].resid = ds[i]->residual_dev;
                    args[i].resid_post = (ds[i]->residual_dev && ds[i]->residual_after_act) ? 1 : 0;
                    if (q == 0) b_bytes = pp[i].b_stage_bytes;
                    if (pp[i].b_stage_bytes != b_bytes || args[i].G != args[set[0]].G) agree = false;
                    if (args[i].G < g_min) g_min = args[i].G;
                    if (pp[i].a_stage_bytes > a_max) a_max = pp[i].a_stage_bytes;
                    if (pp[i].acc_cols > acc_max) acc_max = pp[i].acc_cols;
                    n_tiles[i] = (long)args[i].N * args[i].tiles_y * args[i].tiles_x * args[i].co_tiles;
                }
                if (agree) break;
                if (pass == 1) return -1;
                force_G = g_min;
            }
            // the rings every problem of the set fits into
            const int room = cap - fixed - (under ? res_bytes : 0);
            int na = (room - 2 * b_bytes) / a_max;
            if (na > kMaxA) na = kMaxA;
            bool one_block = true;   // (see plan_tc: layers of one channel block per tile keep more activation stages)
            for (int q = 0; q < m; ++q) one_block = one_block && ncb_of(ps[set[q]]) == 1;
            if (na > 2 && ps[i0]->ksize == 3 && !one_block) na = 2;
            if (na < 1) return -1;
            int nb = (room - na * a_max) / b_bytes;
            if (nb > kMaxB) nb = kMaxB;
            if (nb < 2) return -1;
            int gi = 0;
            while (gi < n_geo && !(geos[gi].a == a_max && geos[gi].b == b_bytes && geos[gi].na == na && geos[gi].nb == nb && geos[gi].under == under)) ++gi;
            if (gi == n_geo) geos[n_geo++] = Geo{a_max, b_bytes, na, nb, under};
            for (int q = 0; q < m; ++q) geo_of[set[q]] = gi;
        }
        // distinct position tables
        int n_distinct = 0;
        for (int i = 0; i < n; ++i) {
            bool fresh = true;
            for (int j = 0; j < i && fresh; ++j)
                fresh = !(args[j].Wq == args[i].Wq && args[j].TH == args[i].TH && args[j].TW == args[i].TW && args[j].N_px == args[i].N_px &&
                          args[j].Wo == args[i].Wo && args[j].y_c_stride == args[i].y_c_stride);
            n_distinct += fresh ? 1 : 0;
        }
        n_tabs_planned = tabs_try;
        if (n_distinct <= tabs_try) break;
        if (tabs_try == kMaxTabs) return -1;
    }
    const int fixed = 1024 + 512 + kEpiWarps * kPatchBytes + n_tabs_planned * kMaxPx * 8;
    // the launch's order: by level, inside a level by ring layout, then by falling tile count (stable)
    int order[kMaxProb];
    for (int i = 0; i < n; ++i) order[i] = i;
    for (int i = 1; i < n; ++i)
        for (int j = i; j > 0; --j) {
            const int u = order[j], v = order[j - 1];
            const bool before = level[u] != level[v] ? level[u] < level[v] : geo_of[u] != geo_of[v] ? geo_of[u] < geo_of[v] : n_tiles[u] > n_tiles[v];
            if (!before) break;
            std::swap(order[j], order[j - 1]);
        }
    int where[kMaxProb];   // position of convolution i in the launch
    for (int k = 0; k < n; ++k) where[order[k]] = k;
    g.n_prob = n;
    g.n_tabs = 0;
    g.ring_bytes = res_bytes;
    g.max_na = g.max_nb = 1;
    long units = 0;
    for (int k = 0; k < n; ++k) {
        const int i = order[k];
        TcArgs& a = g.prob[k];
        a = args[i];
        g.tmA[k] = mapA[i];
        g.tmB[k] = mapB[i];
        const Geo& ge = geos[geo_of[i]];
        a.NA = ge.na;
        a.NB = ge.nb;
        a.a_stage = (unsigned)ge.a;
        a.b_stage = (unsigned)ge.b;
        a.sB_off = (unsigned)ge.na * (unsigned)ge.a;
        a.geo = geo_of[i];
        const int ring = ge.na * ge.a + ge.nb * ge.b + (ge.under ? res_bytes : 0);
        if (ring > g.ring_bytes) g.ring_bytes = ring;
        if (ge.na > g.max_na) g.max_na = ge.na;
        if (ge.nb > g.max_nb) g.max_nb = ge.nb;
        // position table: shared with an earlier problem of the same tile geometry and output pitch
        a.tab = -1;
        for (int q = 0; q < k && a.tab < 0; ++q) {
            const TcArgs& b = g.prob[q];
            if (b.Wq == a.Wq && b.TH == a.TH && b.TW == a.TW && b.N_px == a.N_px && b.Wo == a.Wo && b.y_c_stride == a.y_c_stride) a.tab = b.tab;
        }
        if (a.tab < 0) {
            if (g.n_tabs == n_tabs_planned) return -1;
            a.tab = g.n_tabs++;
        }
        a.dep_mask = 0;
        if (after)
            for (int j = 0; j < i; ++j)
                if ((after[i] >> j) & 1u) a.dep_mask |= 1u << where[j];
        units += n_tiles[i];
        if (units > 0x3FFFFFFF) return -1;
        g.unit_end[k] = (int)units;
    }
    const int grid_n = (int)(units < sms ? units : sms);
    g.res_off = g.ring_bytes - res_bytes;
    for (int k = 0; k < n; ++k) {
        const long mine = n_tiles[order[k]];
        TcArgs& a = g.prob[k];
        a.done_target = (unsigned)((mine < grid_n ? mine : grid_n) * kEpiWarps);
        a.over_res = (resid && (int)(a.sB_off + (unsigned)a.NB * a.b_stage) > g.res_off) ? 1 : 0;
    }
    g.done = nullptr;
    if (chained) {
        // a block of counters of the context, taken in turn (launches that share a block must follow one another in a stream)
        g.done = ctx->chain_done + (size_t)(ctx->chain_next % RTOSS_CHAIN_SLOTS) * RTOSS_CHAIN_SLOT_WORDS;
        ctx->chain_next = (ctx->chain_next + 1) % RTOSS_CHAIN_SLOTS;
    }
    g.acc_stride = acc_max;
    launch_common(ctx, &g);
    if (g.tmem_cols > 512) return -1;
    const size_t smem_need = (size_t)fixed + (size_t)g.ring_bytes;
    if (smem_need > (size_t)cap) return -1;
    const size_t smem = smem_need > 116 * 1024 ? smem_need : 116 * 1024;
    dim3 grid((unsigned)grid_n);
    const cudaError_t le = rtoss_dev::launch_pdl(shared_kernel(ctx, ps[0]->dtype == RTOSS_F32, g), grid, threads_of(ps[0]->dtype == RTOSS_F32), smem, (cudaStream_t)stream, 1, g);
    return (int)le;
}

// Several independent convolutions of one class (kernel size, stride class, data type) in one launch.
int rtoss_launch_conv_tc_group(const rtoss_ctx* ctx, int n, const rtoss_packed* const* ps, const void* const* xs, void* const* ys,
                               const rtoss_conv_desc* const* ds, void* stream) {
    for (int i = 1; i < n; ++i) {
        if (ps[i]->ksize != ps[0]->ksize) return -1;
        if (ps[i]->ksize == 3 && ds[i]->stride != ds[0]->stride) return -1;   // (3x3: stride 2 stages four sub-tiles per block)
    }
    return rtoss_launch_conv_tc_chain(ctx, n, ps, xs, ys, ds, nullptr, stream);
}

int rtoss_tc_max_problems() { return kMaxProb; }
