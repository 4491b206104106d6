// Tensor-core path of the pattern convolutions (bf16 / fp16 / fp32, NHWC, stride 1 or 2).
//
// Per-kernel patterns cannot be compacted into a dense contraction (every
// filter keeps different (channel, tap) positions), so this path evaluates the
// convolution of Section II.B of arXiv 2303.02191 as a masked dense implicit
// GEMM on the 5th-generation tensor cores: the pruned taps are multiplied as
// zeros.  It performs 9/k times the non-zero FLOPs and is still several times
// faster than the FMA pipes; the FMA path stays the one for shapes and layouts
// this kernel does not take.
//
// GEMM view:  D[co, position] = sum over taps t and channels ci of
//                               Wt[t][co][ci] * X[position shifted by t, ci]
//   * A CTA tile is TH output rows of one image (all columns) times 128 output
//     channels.  The input rows it needs (with the one-pixel halo, zero-filled
//     by TMA outside the image) are staged once per block of 64 channels as a
//     flat list of "padded pixels", 128 bytes (64 channels) each, row pitch
//     Wp = W + 2 pixels.  In that list the input pixel of tap (r, c) for output
//     position p is at p + r*Wp + c: the activation operand of every tap is
//     the SAME shared-memory tile read from a different start row, so the halo
//     tile is loaded once and used by all nine taps.  Output positions run over
//     the padded pitch too; the two junk positions per row are computed and
//     dropped.
//   * Operand roles: the weights are the M operand (128 filters = the 128 TMEM
//     lanes), the positions are the N operand (up to 256 per instruction), K =
//     16 channels per instruction.  One instruction takes N / 2 cycles, but
//     never less than about 47, and with M = 64 as long as with M = 128
//     (measured), so N must be wide.
//   * Weights are the dense-expanded form Wt[t][co][ci] that rtoss_pack builds
//     next to the packed arrays; one TMA box per (kernel row of three taps,
//     channel block); filters
//     beyond Cout are zero-filled by TMA.
//   * Persistent CTAs, one per SM, each walking a strided list of tiles.  Warp
//     roles: warp 0 issues the TMA copies of the activations, warp 1 issues
//     tcgen05.mma and owns the TMEM allocation, warps 2..17 run the epilogue
//     (tcgen05.ld, bias, activation, rounding, a transpose through shared memory,
//     16-byte NHWC stores), warp 18 issues the TMA copies of the weights (a stage
//     of three taps is one copy: issuing a copy occupies its thread for hundreds
//     of cycles whatever the size); fp32 data has four more, which split the
//     activation blocks (see below).  Activation and weight stages form rings
//     that run on across tiles; two accumulator stages in TMEM let the epilogue
//     of a tile run under the MMAs of the next.
//   * Layers with few tiles and long channel loops are cut along the channel
//     blocks: the CTAs that share a tile form a thread-block cluster and exchange
//     their partial sums through distributed shared memory (split K).
//   * Launched with programmatic stream serialization: barrier set-up, TMEM allocation and descriptor
//     prefetch run before griddepcontrol.wait, i.e. possibly under the tail of the previous kernel.
//   * Every mbarrier wait is bounded; a wait that runs out records a code in
//     the context's status word and the CTA leaves through the normal exit
//     (TMEM is always released).
//   * A 3x3 layer's handle says, per (tile of 128 filters, 16-channel slab, tap), whether any kept weight lies there
//     (rtoss_pack gathers that from the pattern ids).  Where none does, the instruction would multiply zeros only and
//     is not issued.  With per-kernel patterns on dense random weights every such block holds kept weights; when a
//     block of kernels shares one pattern (rtoss_select_patterns_shared) only k of the 9 taps of a slab are issued:
//     the contraction is then compacted to the non-zero work.
//   * fp32 data runs on the same pipeline with kind::tf32 instructions and three products per tap in place of one:
//     every value is split into a tf32 head (19 leading bits) and the remainder, x = xh + xl, w = wh + wl, and
//     wh*xh + wh*xl + wl*xh is accumulated in fp32 (the dropped wl*xl is below 2^-21 of the product).  The weights are
//     split when they are packed; an activation block is split in shared memory by four warps (head in place, remainder
//     into the second half of the stage) before the MMA thread may read it.  (One warp, the one that fetches, took 48 clocks
//     a row, 14 000 for 288 rows, and the copy of the next block waited for it.)
//     3x3 layers of whole blocks of 32 channels form the two small products from bf16 numbers, at twice the tf32 rate and
//     in two instructions of 16 channels instead of four of eight: bf16(w) * bf16(xl) + bf16(wl) * bf16(x), heads rounded to
//     nearest.  Eight instructions a tap and block instead of twelve; bf16 has fp32's range.  The rounded factors cost 6.5e-7 of
//     the sum where three tf32 products cost 3.5e-7, but what decides is the tensor core's own accumulation, which cuts off
//     and loses in proportion to the instructions of a sum.  Relative error against 64-bit sums, three products -> now, by
//     the blocks of 32 channels that one CTA adds up (four kept taps a kernel): one 2.7e-6 -> 1.8e-6, two 4.6 -> 3.0, four
//     8.3 -> 5.4, eight 15.6 -> 10.4, sixteen 30 -> 20; block patterns of two taps 1.06 -> 0.80, 1.54 -> 1.00, 2.48 -> 1.50,
//     4.3 -> 2.6, 8.0 -> 5.0.  158 random calls: 0.60 to 0.85 of the error of three products (the cut along K is theirs, see
//     plan_tc).  1x1 layers, with a ninth of the instructions, keep three tf32 products (eight blocks 2.3e-6).
//     256->256 @80x80 x32 1084 -> 755 us, the split by four warps and the corrections together; the four units of tensor time
//     it takes instead of six are 593 us at the bf16 peak.
//   * One launch may carry several independent convolutions ("problems": the pyramid levels of a detection tower,
//     the two branches of a block): the tile list runs over all of them, every role looks its tile's problem up.
//     Small problems then fill the tail of the large ones' waves instead of paying a launch each.
//
// This header holds the kernel; conv_tc.cu plans and launches it, conv_tc_bf16.cu and conv_tc_f16.cu hold its forms.
#ifndef RTOSS_CONV_TC_KERNEL_CUH
#define RTOSS_CONV_TC_KERNEL_CUH

#include <cuda.h>

#include <cstddef>

#include "conv_common.cuh"
#include "select_core.cuh"


namespace {

using namespace rtoss_dev;

constexpr int kEpiWarps = 16;
constexpr int kTcThreads = (3 + kEpiWarps) * 32;  // activation TMA warp, MMA warp, sixteen epilogue warps, weight TMA warp
constexpr int kWeightWarp = 2 + kEpiWarps;        // this warp loads the weights; it is the last one but for fp32 data
constexpr int kSplitWarps = 4;                    // fp32: behind it, the warps that split the activation blocks
template <typename T> constexpr int kThreadsOf = kTcThreads + (sizeof(T) == 4 ? kSplitWarps * 32 : 0);
constexpr int kPatchRows = 16;       // positions an epilogue warp turns at a time
constexpr int kMaxA = 4, kMaxB = 8;  // most activation stages / weight slots
constexpr int kMTile = 128;          // filters per tile = TMEM lanes
constexpr int kPxmMaxCout = 64;      // layers this narrow run with positions as the M operand
constexpr int kMaxPx = 256;          // most positions in a tile's list
constexpr int kPairPitch = 144;      // bytes per row (a pair of positions x 32 filters, + 16 pad) of the packed patch
constexpr int kResStage = 2048;   // per epilogue warp: two buffers of 2 x 32 residual pieces of 16 bytes
constexpr int kPatchBytes = kPatchRows / 2 * kPairPitch;  // an epilogue warp's transpose patch
constexpr int kKBlock = 64;       // channels per staged block: 128 bytes of bf16 / fp16
constexpr int kRowBytes = 128;    // one padded pixel, one channel block
constexpr long long kWaitCycles = 2000000000LL;  // about one second

constexpr int kMaxProb = 20;      // convolutions one launch may carry
constexpr int kMaxTabs = 8;       // distinct position tables of a launch (problems of equal tile geometry share one)

// One convolution of a launch.
struct TcArgs {
    void* y;
    const void* resid;   // residual operand laid out like y, or null
    int resid_post;      // 1: the residual is added behind the activation (y = act(conv) + residual), 0: in front of it
    // (Between two pointers, where the struct had four bytes to spare.  A launch reads it cold: with the fields that follow moved by
    // four bytes, and no other change, the 55 launches of the small detector took 2.5 us more, 244.5 -> 247.)
    union {
        // 16-bit 3x3 of stride 2, where the planner says so and there is a form for it (0: not): a channel block comes as two
        // activation stages, the odd input rows (two column phases, read by the first and the last row of taps) and the even ones
        // (read by the middle row).  The even rows are done with first, so the stages are taken in the order in which they come
        // free, which this word lists: the stage of the odd and the even rows of a block, then of the next, two bits each
        // (half_order).  The taps go out in their own order, so that a layer adds up here as it does in one stage.  As one stage,
        // of which only one fits beside the weights at 100 positions and more, fetching and multiplying take turns: 240->112
        // @132x66 x18 34.5 -> 26.9 us, 144->240 @134x71 x9 24.3 -> 19.5, 48->304 @110x115 x31 62.4 -> 50.6.
        unsigned half;
        // fp32: the instruction descriptor of the two small products of a tap where they are bf16 ones (0: they are not; see the
        // head of the file)
        unsigned idesc16;
    };
    const float* bias;
    const unsigned long long* issue;   // 3x3: which (tap, slab) pairs of (filter tile, channel block) to multiply; null = all
    int N, Ho, Wo, Cin, Cout;    // output image size
    int S;                       // stride
    int Wq, TH, TW, taps;        // position pitch, output rows and columns per tile, 9 or 1
    int N_px, ncb;               // positions per tile (the MMA's N, multiple of 16), channel blocks
    int tiles_y, tiles_x, co_tiles;
    // A unit's index is taken apart into (share of the channel blocks, filter tile, column segment, row band, image) by
    // every role for every tile: the four divisors as multiply-and-shift pairs (see tile_of), set by the host.
    unsigned div_ks[2], div_co[2], div_tx[2], div_ty[2];
    int n_sub, sub_bytes;        // sub-tiles of an activation stage (3x3 stride 2: the 4 input phases, or 2 of them) and their size
    int x_add[4], y_add[4];      // TMA start coordinate of sub-tile s: x = x0*S + x_add[s], y = y0*S + y_add[s]
    int tap_sub[9], tap_shift[9];  // which sub-tile tap t reads, and from which start row
    int G;                                     // taps per weight stage (one barrier round trip per G taps)
    unsigned a_tx_bytes, b_tx_bytes;
    // Output element (n, oy, ox, co) lies at n * y_img + (oy * Wo + ox) * y_c_stride + (y_c_off + co) * y_co:
    // channels last y_co = 1; NCHW (nchw = 1) y_co = the plane, y_c_stride = 1.
    int act, y_c_off, y_c_stride, is_bf16;
    int nchw, y_co;
    long long y_img;
    unsigned idesc;
    int w_rows;           // filter rows per staged weight tile (128; fewer with positions as the M operand)
    int rep_rows, R;      // filters as M, narrow layer: the tile holds R copies of rep_rows filter rows (else 128, 1)
    int rep_shift;        // log2(rep_rows)
    int pxm, MH, n_cols;  // positions as the M operand: M halves of 128 positions per tile, filters per tile (the MMA's N)
    // Split K: a tile's channel blocks are shared out to the KS CTAs of a thread-block cluster, cb_per blocks each;
    // the partial sums are exchanged through distributed shared memory and every CTA finishes a part of the tile.
    int KS, cb_per;
    int cb_ch;            // channels per staged block (128 bytes): 64 for 16-bit data, 32 for fp32
    // Bytes of a staged row (one padded pixel resp. one filter, one channel block): 128 with the 128-byte swizzle, or 64
    // with the 64-byte swizzle for 16-bit layers of at most 32 input channels (half of a 128-byte row would be zero fill,
    // and it is the traffic from L2 to shared memory that bounds such layers).  desc_hi: the matching upper word of the
    // shared-memory matrix descriptors.
    int row_bytes;
    unsigned desc_hi;
    int taps_real;        // 9 or 1; `taps` counts weight tiles per channel block: twice that for fp32 (heads, then remainders)
    int lo_off;           // fp32: byte offset of the second half of an activation stage (remainders, or what idesc16 says)
    // The operand rings this problem runs with: NA activation stages of a_stage bytes from the start of the ring area, NB
    // weight stages of b_stage bytes from sB_off.  Problems of one launch with the same `geo` share all five; where a
    // CTA passes to a problem of another geometry its rings run empty first (see bar_switch in the kernel).
    int NA, NB;
    unsigned a_stage, b_stage, sB_off;
    int resident;         // NB is a tile's number of weight stages and all tiles of a CTA have the same filters: the stages are
                          // filled once and serve every tile (launches of one problem)
    int geo;
    int tab;              // which of the launch's position tables
    // over_res: this problem's rings reach into the launch's residual staging area (only problems without a residual
    // operand may): a CTA that comes to it from a problem with one waits for that problem's epilogues first.
    int over_res;
    // Dependent problems of one launch: bit j of dep_mask = problem j (earlier in the launch's order) must be complete
    // -- all its outputs written -- before this one reads an activation or writes an output; done_target = arrivals
    // on this problem's counter that make it complete (epilogue warps x CTAs that hold units of it).
    unsigned dep_mask, done_target;
};
static_assert(offsetof(TcArgs, bias) == 3 * sizeof(void*), "half and idesc16 take the four bytes behind resid_post");

// A launch: up to NP convolutions sharing the CTA's rings (stage sizes are the largest any of them needs).  The struct
// travels as the kernel's parameter: a launch of one convolution carries the small instantiation (a large parameter
// block costs launch time).
template <int NP>
struct TcLaunchT {
    int n_prob;
    int unit_end[NP];   // units (tile x share of the channel blocks) of problems 0..i
    int* status;
    long long wait_cycles;    // limit of every wait
    int inject;               // test hook: 1 = the first weight copy of the launch is withheld (the wait for it must run out)
    int ring_bytes;           // the ring area: the most any problem's activation + weight stages take
    int max_na, max_nb;       // most activation / weight stages any problem uses (barriers to set up)
    int n_tabs;               // position tables
    int res_off;              // where in the ring area the staging of residual operands lies (its top end), when a problem has one
    unsigned* done;           // dependent problems: kMaxProb completion counters + one exit counter, all zero between launches; else null
    int AS, acc_stride;                        // accumulator stages in TMEM and columns per stage
    int tmem_cols;
    TcArgs prob[NP];
    CUtensorMap tmA[NP], tmB[NP];
};
using TcLaunch1 = TcLaunchT<1>;
using TcLaunchN = TcLaunchT<kMaxProb>;
static_assert(sizeof(TcLaunchN) <= 16384, "kernel parameters: well inside the 32 KB a launch may carry");
static_assert(kMaxProb <= 32, "dependencies are a 32-bit mask");

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bounded wait on a phase parity; false when the limit ran out.
__device__ __forceinline__ unsigned mbar_try(unsigned bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done;
}
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, long long limit) {
    if (mbar_try(bar, parity)) return true;  // the common case costs one instruction, no clock read
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try(bar, parity)) return true;
        if (clock64() - t0 > limit) return false;
    }
}

// Thread-block cluster primitives (split K): rank of this CTA, the address of a peer's shared memory, a store to it,
// and the cluster-wide barrier (release / acquire: stores to peers before it are visible after it).
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned peer_smem(unsigned local_addr, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_peer_f32(unsigned addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* map, int c0, int c1, int c2, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor, K-major operand with 128-byte swizzle: rows of 128 bytes, groups
// of 8 rows 1024 bytes apart.  The start may be any 16-byte aligned address inside a tile whose base
// is 1024-byte aligned: the swizzle is a function of the absolute shared-memory address, the same
// function TMA applied when it wrote the tile, so a start in the middle of an 8-row group (a tap
// shift) or 32 bytes into a row (a K step) needs no correction (base-offset field 0).
// With rows of 64 bytes and the 64-byte swizzle the same holds for groups of 8 rows 512 bytes apart.
__host__ __device__ __forceinline__ unsigned long long make_sw_desc(unsigned addr, int row_bytes) {
    unsigned long long d = 0;
    d |= (unsigned long long)((addr & 0x3FFFFu) >> 4);        // start address
    d |= (unsigned long long)1 << 16;                          // leading byte offset (unused for swizzled K-major)
    d |= (unsigned long long)((8 * row_bytes) >> 4) << 32;     // stride byte offset: 8 rows
    d |= (unsigned long long)1 << 46;                          // descriptor version of this architecture
    d |= (unsigned long long)(row_bytes == 64 ? 4 : 2) << 61;  // 64-byte resp. 128-byte swizzle
    return d;
}

// The MMA warp runs its loop as one, every value in it the same for all lanes, and only the elected lane (leader != 0)
// issues: descriptors and addresses then live in uniform registers, which is where tcgen05.mma takes them from.  (With the
// loop inside "if (lane == 0)" a 1x1 layer's thread took 870 cycles for the four instructions of a channel block, 660 in
// this form: 1x1 128->128 @40x40 3.3 -> 2.9 us, 256->1024 @50x68 batch 4 13.3 -> 11.8, 3x3 32->32 @160x160 batch 16 31.3 ->
// 24.7.  The producers' loops, which issue few copies, were 1 to 3 % slower this way and stay with one lane.)
__device__ __forceinline__ unsigned elect_one() {
    unsigned e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}
template <bool TF32>
__device__ __forceinline__ void umma_f16(unsigned leader, unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc,
                                         unsigned idesc, unsigned accumulate) {
    if (TF32)
        asm volatile(
            "{\n\t.reg .pred p, pe;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "setp.ne.b32 pe, %5, 0;\n\t"
            "@pe tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(leader)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p, pe;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "setp.ne.b32 pe, %5, 0;\n\t"
            "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(leader)
            : "memory");
}
// The MMAs of one tap of one channel block (filters on M) for the 16-channel slabs named by the mask m4 (bit s = slab
// s), with a look at the "full" barriers of the NEXT activation and weight stage started in front of them
// (mbarrier.test_wait: the answer comes back while the MMAs are being issued).  A wait costs the issuing thread a
// round trip of a few hundred cycles through a memory pipe the epilogue warps keep busy, and with four MMAs per wait
// nothing hides two of those per channel block; the stages ahead are normally full already, so the look usually
// replaces both waits of the next block.  The first instruction issued takes `accumulate` as its accumulate flag,
// the later ones add.  Returns bit 0: next activation stage full, bit 1: next weight stage full.
#define RTOSS_DEFINE_PEEK(NAME, KIND)                                                                                   \
    __device__ __forceinline__ unsigned NAME(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc,     \
                                             unsigned idesc, unsigned accumulate, unsigned m4, unsigned barA,          \
                                             unsigned parA, unsigned barB, unsigned parB) {                            \
        unsigned res;                                                                                                  \
        asm volatile(                                                                                                  \
            "{\n\t.reg .pred pa, pb, q, p0, p1, p2, p3;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t.reg .b32 ta, tb, tm;\n\t"     \
            "mbarrier.test_wait.parity.shared::cta.b64 pa, [%7], %8;\n\t"                                              \
            "mbarrier.test_wait.parity.shared::cta.b64 pb, [%9], %10;\n\t"                                             \
            "setp.ne.b32 q, %5, 0;\n\t"                                                                                \
            "and.b32 tm, %6, 1;\n\tsetp.ne.b32 p0, tm, 0;\n\t"                                                        \
            "and.b32 tm, %6, 2;\n\tsetp.ne.b32 p1, tm, 0;\n\t"                                                        \
            "and.b32 tm, %6, 4;\n\tsetp.ne.b32 p2, tm, 0;\n\t"                                                        \
            "and.b32 tm, %6, 8;\n\tsetp.ne.b32 p3, tm, 0;\n\t"                                                        \
            "add.u64 a1, %2, 2;\n\tadd.u64 a2, %2, 4;\n\tadd.u64 a3, %2, 6;\n\t"                                      \
            "add.u64 b1, %3, 2;\n\tadd.u64 b2, %3, 4;\n\tadd.u64 b3, %3, 6;\n\t"                                      \
            "@p0 tcgen05.mma.cta_group::1.kind::" KIND " [%1], %2, %3, %4, q;\n\t"                                     \
            "or.pred q, q, p0;\n\t"                                                                                    \
            "@p1 tcgen05.mma.cta_group::1.kind::" KIND " [%1], a1, b1, %4, q;\n\t"                                     \
            "or.pred q, q, p1;\n\t"                                                                                    \
            "@p2 tcgen05.mma.cta_group::1.kind::" KIND " [%1], a2, b2, %4, q;\n\t"                                     \
            "or.pred q, q, p2;\n\t"                                                                                    \
            "@p3 tcgen05.mma.cta_group::1.kind::" KIND " [%1], a3, b3, %4, q;\n\t"                                     \
            "selp.u32 ta, 1, 0, pa;\n\t"                                                                               \
            "selp.u32 tb, 2, 0, pb;\n\t"                                                                               \
            "or.b32 %0, ta, tb;\n\t}"                                                                                  \
            : "=r"(res)                                                                                                \
            : "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(m4), "r"(barA), "r"(parA), "r"(barB), \
              "r"(parB)                                                                                                \
            : "memory");                                                                                               \
        return res;                                                                                                    \
    }
RTOSS_DEFINE_PEEK(umma_block_peek_f16, "f16")
RTOSS_DEFINE_PEEK(umma_block_peek_tf32, "tf32")
#undef RTOSS_DEFINE_PEEK
template <bool TF32>
__device__ __forceinline__ unsigned umma_block_peek(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc,
                                                    unsigned idesc, unsigned accumulate, unsigned m4, unsigned barA,
                                                    unsigned parA, unsigned barB, unsigned parB) {
    return TF32 ? umma_block_peek_tf32(d_tmem, adesc, bdesc, idesc, accumulate, m4, barA, parA, barB, parB)
                : umma_block_peek_f16(d_tmem, adesc, bdesc, idesc, accumulate, m4, barA, parA, barB, parB);
}
// Arrive on an mbarrier once all tcgen05.mma issued so far by this thread have completed.
__device__ __forceinline__ void umma_commit(unsigned leader, unsigned bar) {
    asm volatile(
        "{\n\t.reg .pred pe;\n\tsetp.ne.b32 pe, %1, 0;\n\t"
        "@pe tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(leader)
        : "memory");
}

__device__ __forceinline__ void tmem_ld32(unsigned taddr, unsigned (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

template <typename T>
__device__ __forceinline__ unsigned pack2(float a, float b);
template <>
__device__ __forceinline__ unsigned pack2<__nv_bfloat16>(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<unsigned*>(&v);
}
template <>
__device__ __forceinline__ unsigned pack2<__half>(float a, float b) {
    __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned*>(&v);
}

__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// Internal activation code: SiLU in the exponential form of the FMA path for 16-bit outputs too (calls that path used
// to take keep its precision: the tanh form's 2^-11 is as coarse as half a unit in the last place of fp16).
constexpr int kActSiluX = 3;
__device__ __forceinline__ float silu_exp(float v) { return __fdividef(v, 1.f + __expf(-v)); }

// Sixteen consecutive filters of one position (positions as the M operand): bias, activation, rounding, packed
// two to a register in memory order.
template <typename T, int ACT>
__device__ __forceinline__ void act_pack16(const unsigned (&r)[16], const float* bias16, unsigned (&o)[8]) {
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        float v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            v[e] = __uint_as_float(r[j + e]) + bias16[j + e];
            if (ACT == RTOSS_ACT_RELU) v[e] = fmaxf(v[e], 0.f);
            if (ACT == RTOSS_ACT_SILU) {
                float th;
                asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(0.5f * v[e]));
                v[e] = v[e] * fmaf(0.5f, th, 0.5f);
            }
            if (ACT == kActSiluX) v[e] = silu_exp(v[e]);
        }
        o[j >> 1] = pack2<T>(v[0], v[1]);
    }
}

// Two fp32 values rounded to the 16-bit output type and packed (lo in the low half), with the ReLU folded into
// the conversion where asked for.
template <typename T, bool RELU>
__device__ __forceinline__ unsigned round_pack(float lo, float hi);
template <>
__device__ __forceinline__ unsigned round_pack<__nv_bfloat16, false>(float lo, float hi) {
    return pack2<__nv_bfloat16>(lo, hi);
}
template <>
__device__ __forceinline__ unsigned round_pack<__half, false>(float lo, float hi) {
    return pack2<__half>(lo, hi);
}
template <>
__device__ __forceinline__ unsigned round_pack<__nv_bfloat16, true>(float lo, float hi) {
    unsigned d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
template <>
__device__ __forceinline__ unsigned round_pack<__half, true>(float lo, float hi) {
    unsigned d;
    asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// SiLU of an fp32 output: v / (1 + e^-v) with the fast exponential (a few ulp: the tanh form below is good to 2^-11
// only, enough for 16-bit outputs, not for the 1e-4 bound of fp32 ones).
__device__ __forceinline__ float silu_f32(float v) { return v / (1.f + __expf(-v)); }

// Bias and activation of one accumulator value.  bs is the bias, for SiLU half the bias:
//   v * sigmoid(v) = h + h * tanh(h) with h = v / 2 = fma(acc, 0.5, b / 2): two fused multiply-adds around one
//   special-function op (tanh.approx, relative error about 2^-11: below half an ulp of bf16, about one ulp of
//   fp16).  ReLU is left to the conversion.
template <int ACT>
__device__ __forceinline__ float bias_act(unsigned acc_bits, float bs) {
    const float acc = __uint_as_float(acc_bits);
    if (ACT == RTOSS_ACT_SILU) {
        const float h = fmaf(acc, 0.5f, bs);
        float th;
        asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(h));
        return fmaf(h, th, h);
    }
    if (ACT == kActSiluX) return silu_exp(acc + bs);   // (bs is the plain bias)
    return acc + bs;
}

// Eight outputs of one position (four words of two 16-bit values, already rounded without activation) plus the eight
// residual values at the same place: sum in fp32, activation, one more rounding -- what a convolution without
// activation followed by an element-wise add + activation gives, bit for bit (act none and ReLU; SiLU here is the
// tanh form of the epilogue).
template <typename T, int ACT>
__device__ __forceinline__ uint4 add_residual8(uint4 o, const uint4 rv) {
    const T* oe = reinterpret_cast<const T*>(&o);
    const T* re = reinterpret_cast<const T*>(&rv);
    unsigned w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            v[e] = to_f32<T>(oe[2 * i + e]) + to_f32<T>(re[2 * i + e]);
            if (ACT == RTOSS_ACT_SILU) {
                const float h = 0.5f * v[e];
                float th;
                asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(h));
                v[e] = fmaf(h, th, h);
            }
        }
        w[i] = round_pack<T, ACT == RTOSS_ACT_RELU>(v[0], v[1]);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Sixteen positions of one filter per lane (a half chunk of split K, whose sums come from shared memory that way): round,
// transpose through the patch, store.  A lane rounds two neighbouring positions of its filter into one word and stores it
// to row (position pair), column (filter); lane (pair lane / 4, filter group lane % 4) reads its group's eight words, splits
// low and high halves and writes each as one 16-byte store.
// With a residual operand (rbv, laid out like the output) the activation moves behind the residual add.
template <typename T, int ACT>
__device__ __forceinline__ void epilogue_half(const unsigned (&r)[16], float bs, unsigned wr, unsigned rd, unsigned tab_at,
                                              T* ybv, unsigned ry, unsigned rx, const T* rbv = nullptr, bool post = false) {
    const bool res = rbv != nullptr;   // then (unless post) bs is the plain bias and nothing is activated before the add
#pragma unroll
    for (int jp = 0; jp < kPatchRows / 2; ++jp) {
        const unsigned w = (res && !post) ? round_pack<T, false>(__uint_as_float(r[2 * jp]) + bs, __uint_as_float(r[2 * jp + 1]) + bs)
                               : round_pack<T, ACT == RTOSS_ACT_RELU>(bias_act<ACT>(r[2 * jp], bs), bias_act<ACT>(r[2 * jp + 1], bs));
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(wr + jp * kPairPitch), "r"(w) : "memory");
    }
    __syncwarp();
    unsigned w[8], e[4];
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(rd));
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "r"(rd + 16));
    // table entries of positions 2 jp and 2 jp + 1 (an even position: 16-byte aligned)
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(e[0]), "=r"(e[1]), "=r"(e[2]), "=r"(e[3]) : "r"(tab_at));
    if ((e[1] >> 16) < ry && (e[1] & 0xFFFFu) < rx) {
        uint4 o = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410), __byte_perm(w[4], w[5], 0x5410),
                             __byte_perm(w[6], w[7], 0x5410));
        if (res) {
            const uint4 rv = *reinterpret_cast<const uint4*>(rbv + e[0]);
            o = post ? add_residual8<T, RTOSS_ACT_NONE>(o, rv) : add_residual8<T, ACT>(o, rv);
        }
        *reinterpret_cast<uint4*>(ybv + e[0]) = o;
    }
    if ((e[3] >> 16) < ry && (e[3] & 0xFFFFu) < rx) {
        uint4 o = make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632), __byte_perm(w[4], w[5], 0x7632),
                             __byte_perm(w[6], w[7], 0x7632));
        if (res) {
            const uint4 rv = *reinterpret_cast<const uint4*>(rbv + e[2]);
            o = post ? add_residual8<T, RTOSS_ACT_NONE>(o, rv) : add_residual8<T, ACT>(o, rv);
        }
        *reinterpret_cast<uint4*>(ybv + e[2]) = o;
    }
    __syncwarp();
}

// ---- the filters-as-M epilogue of 16-bit layers ------------------------------------------------------------------
// A warp owns 32 filters (its TMEM lane quarter) and takes the positions sixteen at a time (a half chunk); NHWC wants the
// filters of one position side by side.  The accumulator is read as matrix fragments (tcgen05.ld 16x256b: a thread gets
// two neighbouring positions of one filter per register pair, four filters in all), so that after bias, activation and
// rounding a packed register is exactly what stmatrix takes, and two transposing stmatrix.x4 lay the half chunk down as
// sixteen rows of 64 bytes, one per position.  The 16-byte piece g of row p sits at piece g ^ ((p / 2) mod 4): the eight
// rows stmatrix writes at once and the two rows eight lanes read at once both fall on 32 different banks.  A lane then
// reads the piece (position lane / 4 resp. + 8, filters 8 (lane mod 4) ...) and stores its 16 bytes: four lanes cover the
// 64 contiguous bytes of a position.
// Where a position goes comes from the table built in the prologue: tab[p] = {element offset inside the tile, row << 16 |
// column}.  Two register sets: the next half chunk's loads are in flight while the current one is worked on.
// (The form before this read a filter per lane, stored eight words, read three vectors and split them with eight byte
// permutes per half chunk: 171 warp instructions all told, a third of its shared-memory wavefronts bank conflicts.)
__device__ __forceinline__ void tmem_ld_frag(unsigned taddr, unsigned (&lo)[8], unsigned (&hi)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(lo[0]), "=r"(lo[1]), "=r"(lo[2]), "=r"(lo[3]), "=r"(lo[4]), "=r"(lo[5]), "=r"(lo[6]), "=r"(lo[7])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(hi[0]), "=r"(hi[1]), "=r"(hi[2]), "=r"(hi[3]), "=r"(hi[4]), "=r"(hi[5]), "=r"(hi[6]), "=r"(hi[7])
                 : "r"(taddr + (16u << 16))
                 : "memory");
}

// What a lane needs for every half chunk of a tile.
struct FragLane {
    float b[4];      // bias of filters lane / 4 + 0, 8, 16, 24 (as bias_act expects it)
    unsigned st;     // stmatrix row address of this lane (position lane mod 8, piece lane / 8)
    unsigned rd;     // this lane's piece of position lane / 4
    unsigned tab;    // table entry of position lane / 4 of the tile
};
__device__ __forceinline__ FragLane frag_lane(float bs, unsigned patch, unsigned tab, int lane) {
    FragLane f;
#pragma unroll
    for (int q = 0; q < 4; ++q) f.b[q] = __shfl_sync(0xFFFFFFFFu, bs, 8 * q + (lane >> 2));
    const unsigned p = (unsigned)lane & 7u, g = (unsigned)lane >> 3;
    f.st = patch + p * 64u + ((g ^ ((p >> 1) & 3u)) << 4);
    const unsigned q = (unsigned)lane >> 2, h = (unsigned)lane & 3u;
    f.rd = patch + q * 64u + ((h ^ ((q >> 1) & 3u)) << 4);
    f.tab = tab + q * 8u;
    return f;
}

// Half chunk -> patch.  ACT = none and RELU false: the plain rounded sum.
template <typename T, int ACT>
__device__ __forceinline__ void frag_to_patch(const unsigned (&lo)[8], const unsigned (&hi)[8], const FragLane& f) {
    constexpr bool kRelu = ACT == RTOSS_ACT_RELU;
#pragma unroll
    for (int po = 0; po < 2; ++po) {   // positions 8 po ... 8 po + 7
        const unsigned w0 = round_pack<T, kRelu>(bias_act<ACT>(lo[4 * po], f.b[0]), bias_act<ACT>(lo[4 * po + 1], f.b[0]));
        const unsigned w1 = round_pack<T, kRelu>(bias_act<ACT>(lo[4 * po + 2], f.b[1]), bias_act<ACT>(lo[4 * po + 3], f.b[1]));
        const unsigned w2 = round_pack<T, kRelu>(bias_act<ACT>(hi[4 * po], f.b[2]), bias_act<ACT>(hi[4 * po + 1], f.b[2]));
        const unsigned w3 = round_pack<T, kRelu>(bias_act<ACT>(hi[4 * po + 2], f.b[3]), bias_act<ACT>(hi[4 * po + 3], f.b[3]));
        asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(f.st + 512u * po), "r"(w0), "r"(w1),
                     "r"(w2), "r"(w3)
                     : "memory");
    }
    __syncwarp();
}
__device__ __forceinline__ uint4 lds128(unsigned at) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at));
    return v;
}
__device__ __forceinline__ uint2 lds64(unsigned at) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at));
    return v;
}
__device__ __forceinline__ bool inside(const uint2& e, unsigned ry, unsigned rx) { return (e.y >> 16) < ry && (e.y & 0xFFFFu) < rx; }

template <typename T, int ACT>
__device__ __forceinline__ void frag_half(const unsigned (&lo)[8], const unsigned (&hi)[8], const FragLane& f, unsigned c0, T* ybv, unsigned ry,
                                          unsigned rx) {
    const uint2 e0 = lds64(f.tab + c0 * 8u), e1 = lds64(f.tab + c0 * 8u + 64u);
    frag_to_patch<T, ACT>(lo, hi, f);
    const uint4 o0 = lds128(f.rd), o1 = lds128(f.rd + 512u);
    if (inside(e0, ry, rx)) *reinterpret_cast<uint4*>(ybv + e0.x) = o0;
    if (inside(e1, ry, rx)) *reinterpret_cast<uint4*>(ybv + e1.x) = o1;
    __syncwarp();
}

// One tile for one warp: its lane quarter of the accumulator stage at d_base, the 32-column chunks c0, c0 + c_step, ...
template <typename T, int ACT>
__device__ __forceinline__ void epilogue_chunks(unsigned d_base, int c0, int c_step, int n_px, float bs,
                                                unsigned patch, unsigned tab, T* yb, unsigned ry, unsigned rx, int lane) {
    const FragLane f = frag_lane(bs, patch, tab, lane);
    T* ybv = yb + (lane & 3) * 8;
    if (c0 >= n_px) return;
    unsigned la[8], ha[8], lb[8], hb[8];
    tmem_ld_frag(d_base + (unsigned)c0, la, ha);
    for (; c0 < n_px; c0 += c_step) {
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        tmem_ld_frag(d_base + (unsigned)(c0 + kPatchRows), lb, hb);
        frag_half<T, ACT>(la, ha, f, (unsigned)c0, ybv, ry, rx);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c0 + c_step < n_px) tmem_ld_frag(d_base + (unsigned)(c0 + c_step), la, ha);
        frag_half<T, ACT>(lb, hb, f, (unsigned)(c0 + kPatchRows), ybv, ry, rx);
    }
}

// The same with a residual operand.  Its values arrive by asynchronous 16-byte copies (global -> shared, no
// registers held while they fly): every lane fetches the two pieces it will add (positions lane / 4 and + 8, its
// eight filters) into its own slots of the warp's staging area, one half chunk ahead of the one being finished, so a
// load from memory has a whole half chunk of work to hide behind.  A lane reads back only what it fetched itself:
// cp.async.wait_group is all the ordering needed.  stage: shared address of the warp's kResStage bytes, two buffers
// of [2 pieces][32 lanes] x 16 bytes.
template <typename T>
__device__ __forceinline__ void fetch_residual(unsigned tab_at, const T* rbv, unsigned ry, unsigned rx, unsigned slot) {
    const uint2 e0 = lds64(tab_at), e1 = lds64(tab_at + 64u);
    if (inside(e0, ry, rx)) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot), "l"(rbv + e0.x) : "memory");
    if (inside(e1, ry, rx)) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot + 512u), "l"(rbv + e1.x) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// POST: activated and rounded as without a residual (the bias is then what bias_act expects); else the plain sum first.
template <typename T, int ACT, bool POST>
__device__ __forceinline__ void frag_half_res(const unsigned (&lo)[8], const unsigned (&hi)[8], const FragLane& f, unsigned c0, T* ybv,
                                              unsigned ry, unsigned rx, unsigned slot) {
    const uint2 e0 = lds64(f.tab + c0 * 8u), e1 = lds64(f.tab + c0 * 8u + 64u);
    frag_to_patch<T, POST ? ACT : RTOSS_ACT_NONE>(lo, hi, f);
    const uint4 o0 = lds128(f.rd), o1 = lds128(f.rd + 512u);
    if (inside(e0, ry, rx)) *reinterpret_cast<uint4*>(ybv + e0.x) = add_residual8<T, POST ? RTOSS_ACT_NONE : ACT>(o0, lds128(slot));
    if (inside(e1, ry, rx)) *reinterpret_cast<uint4*>(ybv + e1.x) = add_residual8<T, POST ? RTOSS_ACT_NONE : ACT>(o1, lds128(slot + 512u));
    __syncwarp();
}

template <typename T, int ACT, bool POST>
__device__ __forceinline__ void epilogue_chunks_res(unsigned d_base, int c0, int c_step, int n_px, float bias,
                                                    unsigned patch, unsigned tab, T* yb, unsigned ry, unsigned rx,
                                                    int lane, const T* rb, unsigned stage) {
    const FragLane f = frag_lane(bias, patch, tab, lane);
    T* ybv = yb + (lane & 3) * 8;
    const T* rbv = rb + (lane & 3) * 8;
    if (c0 >= n_px) return;
    const unsigned slot0 = stage + (unsigned)lane * 16, slot1 = slot0 + 1024u;
    unsigned la[8], ha[8], lb[8], hb[8];
    fetch_residual<T>(f.tab + (unsigned)c0 * 8, rbv, ry, rx, slot0);
    tmem_ld_frag(d_base + (unsigned)c0, la, ha);
    for (; c0 < n_px; c0 += c_step) {
        fetch_residual<T>(f.tab + (unsigned)(c0 + kPatchRows) * 8, rbv, ry, rx, slot1);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        tmem_ld_frag(d_base + (unsigned)(c0 + kPatchRows), lb, hb);
        asm volatile("cp.async.wait_group 1;" ::: "memory");   // the pieces of this half are in
        frag_half_res<T, ACT, POST>(la, ha, f, (unsigned)c0, ybv, ry, rx, slot0);
        const bool more = c0 + c_step < n_px;
        if (more)
            fetch_residual<T>(f.tab + (unsigned)(c0 + c_step) * 8, rbv, ry, rx, slot0);
        else
            asm volatile("cp.async.commit_group;" ::: "memory");   // keeps the group count in step
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (more) tmem_ld_frag(d_base + (unsigned)(c0 + c_step), la, ha);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        frag_half_res<T, ACT, POST>(lb, hb, f, (unsigned)(c0 + kPatchRows), ybv, ry, rx, slot1);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// NCHW outputs: sixteen positions of 32 filters (a half chunk).  NCHW wants the positions of one filter side by side,
// which is what a lane holds, but a store wants its 32 lanes to be neighbours: the half chunk goes through the warp's
// patch (32 rows of eight words, word j of filter f at column j ^ (f / 4): both the stores, all filters of one position
// pair, and the loads, eight pairs of four filters, touch 32 different banks) and leaves as 32-byte runs, one word of
// two positions per lane where the pair is one aligned word, else one element at a time.  pair_ok: planes of an even
// number of elements, so that one look at the offsets holds for every filter.
template <typename T, int ACT>
__device__ __forceinline__ void epilogue_half_nchw(const unsigned (&r)[16], float bs, unsigned patch, unsigned tab_at, T* yb,
                                                   unsigned ry, unsigned rx, int lane, int n_co, int plane, bool pair_ok) {
    const unsigned wr = patch + (unsigned)lane * 32u;
    const unsigned sw = (unsigned)(lane >> 2) & 7u;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const unsigned w = round_pack<T, ACT == RTOSS_ACT_RELU>(bias_act<ACT>(r[2 * j], bs), bias_act<ACT>(r[2 * j + 1], bs));
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(wr + ((j ^ sw) << 2)), "r"(w) : "memory");
    }
    __syncwarp();
    const int jj = lane & 7, f0 = lane >> 3;
    unsigned e[4];   // table entries of positions 2 jj and 2 jj + 1
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(e[0]), "=r"(e[1]), "=r"(e[2]), "=r"(e[3]) : "r"(tab_at + (unsigned)jj * 16u));
    const bool ok0 = (e[1] >> 16) < ry && (e[1] & 0xFFFFu) < rx, ok1 = (e[3] >> 16) < ry && (e[3] & 0xFFFFu) < rx;
    const bool pair = pair_ok && ok0 && ok1 && e[2] == e[0] + 1 && !(reinterpret_cast<uintptr_t>(yb + e[0]) & 3);
    T* d = yb + (size_t)f0 * plane;
#pragma unroll
    for (int i = 0; i < 8; ++i, d += (size_t)4 * plane) {
        const int f = 4 * i + f0;
        unsigned w;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w) : "r"(patch + (unsigned)f * 32u + ((jj ^ i) << 2)));   // (f / 4 = i)
        if (f < n_co) {
            if (pair) {
                *reinterpret_cast<unsigned*>(d + e[0]) = w;
            } else {
                const T* h = reinterpret_cast<const T*>(&w);
                if (ok0) d[e[0]] = h[0];
                if (ok1) d[e[2]] = h[1];
            }
        }
    }
    __syncwarp();
}
template <typename T, int ACT>
__device__ __forceinline__ void epilogue_chunks_nchw(unsigned d_base, int c0, int c_step, int n_px, float bs, unsigned patch, unsigned tab,
                                                     T* yb, unsigned ry, unsigned rx, int lane, int n_co, int plane, bool pair_ok) {
    if (c0 >= n_px) return;
    unsigned ra[16], rb[16];
    tmem_ld16(d_base + (unsigned)c0, ra);
    for (; c0 < n_px; c0 += c_step) {
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        tmem_ld16(d_base + (unsigned)(c0 + kPatchRows), rb);
        epilogue_half_nchw<T, ACT>(ra, bs, patch, tab + (unsigned)c0 * 8, yb, ry, rx, lane, n_co, plane, pair_ok);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c0 + c_step < n_px) tmem_ld16(d_base + (unsigned)(c0 + c_step), ra);
        epilogue_half_nchw<T, ACT>(rb, bs, patch, tab + (unsigned)(c0 + kPatchRows) * 8, yb, ry, rx, lane, n_co, plane, pair_ok);
    }
}

// Split K, second half.  Every CTA of the cluster owns the 32-column chunks c of the tile with c % KS == its rank
// (its local chunk lc = c / KS) and holds, in its own shared memory at `buf`, what each of the KS shares summed
// for them: share i, local chunk lc, column col, accumulator lane row at ((i * n_lc + lc) * 32 + col) * 128 + row
// floats.  The owned chunks are finished as half chunks of 16 columns dealt to the four warps of a lane quarter.
template <typename T, int ACT, bool VEC>   // VEC: whole 16-byte pieces only (vec_ok: this quarter holds filters at all)
__device__ __forceinline__ void epilogue_from_shares(unsigned buf, int KS, int rank, int n_lc, int sub, int row, int n_px, float bs,
                                                     bool vec_ok, bool co_ok, unsigned patch, unsigned tab, const uint2* pos_tab,
                                                     T* yb, unsigned ry, unsigned rx, int lane, const T* rb, bool post, bool nchw,
                                                     int n_co, int y_co) {
    const unsigned wr = patch + lane * 4;
    const unsigned rd = patch + (lane >> 2) * kPairPitch + (lane & 3) * 32;
    const unsigned tab_l = tab + (unsigned)(2 * (lane >> 2)) * 8;
    T* ybv = yb + (lane & 3) * 8;
    const T* rbv = rb ? rb + (lane & 3) * 8 : nullptr;
    for (int t = sub; t < 2 * n_lc; t += 4) {
        const int lc = t >> 1, c0 = (lc * KS + rank) * 32 + (t & 1) * kPatchRows;   // first column of the half chunk
        if (c0 >= n_px) continue;
        float sum[kPatchRows];
#pragma unroll
        for (int j = 0; j < kPatchRows; ++j) sum[j] = 0.f;
        for (int i = 0; i < KS; ++i) {
            const unsigned q = buf + (unsigned)((((i * n_lc + lc) * 32 + (t & 1) * kPatchRows) * 128 + row) * 4);
#pragma unroll
            for (int j = 0; j < kPatchRows; ++j) {
                float v;
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(q + j * 512));
                sum[j] += v;
            }
        }
        unsigned r[16];
#pragma unroll
        for (int j = 0; j < kPatchRows; ++j) r[j] = __float_as_uint(sum[j]);
        bool done = false;
        if constexpr (sizeof(T) == 2) {
            if (vec_ok) {
                epilogue_half<T, ACT>(r, bs, wr, rd, tab_l + (unsigned)c0 * 8, ybv, ry, rx, rbv, post);
                done = true;
            } else if (nchw) {
                epilogue_half_nchw<T, ACT>(r, bs, patch, tab + (unsigned)c0 * 8, yb, ry, rx, lane, n_co, y_co, (y_co & 1) == 0);
                done = true;
            }
        }
        if (!VEC && !done) {
            constexpr bool f32 = sizeof(T) == 4;   // (fp32: bs is the plain bias and SiLU the exponential form)
#pragma unroll
            for (int j = 0; j < kPatchRows; ++j) {
                const uint2 e = pos_tab[c0 + j];
                if (co_ok && (e.y >> 16) < ry && (e.y & 0xFFFFu) < rx) {
                    float v;
                    if (rb && post) {   // activate, round, add the residual, round
                        v = f32 ? (ACT == RTOSS_ACT_SILU ? silu_f32(__uint_as_float(r[j]) + bs) : __uint_as_float(r[j]) + bs) : bias_act<ACT>(r[j], bs);
                        if (ACT == RTOSS_ACT_RELU) v = fmaxf(v, 0.f);
                        v = to_f32<T>(from_f32<T>(v)) + to_f32<T>(rb[e.x + lane]);
                    } else if (rb) {   // round, add the residual, activate, round
                        v = to_f32<T>(from_f32<T>(__uint_as_float(r[j]) + bs)) + to_f32<T>(rb[e.x + lane]);
                        if (ACT == RTOSS_ACT_RELU) v = fmaxf(v, 0.f);
                        if (ACT == RTOSS_ACT_SILU) {
                            if (f32) {
                                v = silu_f32(v);
                            } else {
                                float th;
                                asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(0.5f * v));
                                v = fmaf(0.5f * v, th, 0.5f * v);
                            }
                        }
                    } else {
                        v = f32 ? (ACT == RTOSS_ACT_SILU ? silu_f32(__uint_as_float(r[j]) + bs) : __uint_as_float(r[j]) + bs) : bias_act<ACT>(r[j], bs);
                        if (ACT == RTOSS_ACT_RELU) v = fmaxf(v, 0.f);
                    }
                    yb[e.x + lane] = from_f32<T>(v);
                }
            }
        }
    }
}

// Which problem a unit of the launch's list belongs to, and its index inside that problem.  A CTA's units ascend, so
// the search goes on from the problem of its previous unit (`from`).
template <bool kMulti, typename G>
__device__ __forceinline__ int find_problem(const G& g, int unit, int& local, int from = 0) {
    if (!kMulti) {   // a launch of one problem: the index is a compile-time constant
        local = unit;
        return 0;
    }
    int pi = from;
    while (pi + 1 < g.n_prob && unit >= g.unit_end[pi]) ++pi;
    local = unit - (pi ? g.unit_end[pi - 1] : 0);
    return pi;
}

// n / d for n < 2^31 by a multiplication: md = {ceil(2^(31 + l) / d), l - 1} with l = ceil(log2 d), or {0, 0} for d = 1
// (exact: the multiplier's error, below 2^l / d <= 2 parts in 2^(31 + l), cannot carry a quotient of n < 2^31 over).
__host__ __device__ __forceinline__ void magic_of(int d, unsigned (&md)[2]) {
    md[0] = md[1] = 0;
    if (d <= 1) return;
    int l = 0;
    while ((1ll << l) < d) ++l;
    md[0] = (unsigned)((((unsigned long long)1 << (31 + l)) + (unsigned)d - 1) / (unsigned)d);
    md[1] = (unsigned)(l - 1);
}
__device__ __forceinline__ int fdiv(int n, const unsigned (&md)[2]) {
    return md[0] ? (int)(__umulhi((unsigned)n, md[0]) >> md[1]) : n;
}
// A unit of problem a taken apart.
struct TileIdx {
    int ks, cot, tx, ty, n;
};
__device__ __forceinline__ TileIdx tile_of(const TcArgs& a, int local) {
    TileIdx t;
    int rest = fdiv(local, a.div_ks);
    t.ks = local - rest * a.KS;
    int q = fdiv(rest, a.div_co);
    t.cot = rest - q * a.co_tiles;
    rest = q;
    q = fdiv(rest, a.div_tx);
    t.tx = rest - q * a.tiles_x;
    rest = q;
    t.n = fdiv(rest, a.div_ty);
    t.ty = rest - t.n * a.tiles_y;
    return t;
}

// A ring of stages with one "full" and one "empty" mbarrier per stage: position s and, per stage, the parity of the
// phase its next use belongs to (bit i of par = stage i).  The parities are kept per stage because the problems of a
// launch may run with different ring depths: the stages then do not all have the same number of uses behind them.
struct Ring {
    int s = 0;
    unsigned par = 0;
    __device__ __forceinline__ unsigned parity() const { return (par >> s) & 1u; }
    __device__ __forceinline__ void advance(int n, unsigned flip = 1u) {   // flip 0: the stages are filled once and stay
        par ^= flip << s;
        if (++s == n) s = 0;
    }
};

// Dependent problems of one launch: waits (bounded) until every problem named in dep_mask has all its outputs written,
// then orders this thread's coming bulk copies behind what it has seen.  The writers' side is at the end of the
// epilogue's tile loop.
template <typename G>
__device__ __forceinline__ bool wait_deps(const G& g, unsigned dep_mask) {
    const long long t0 = clock64();
    while (dep_mask) {
        const int j = __ffs((int)dep_mask) - 1;
        dep_mask &= dep_mask - 1;
        const unsigned target = g.prob[j].done_target;
        for (;;) {
            unsigned seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(g.done + j) : "memory");
            if (seen >= target) break;
            if (clock64() - t0 > g.wait_cycles) return false;
            __nanosleep(100);
        }
    }
    // the outputs were written with ordinary stores; the copies that fetch them go through the asynchronous proxy
    asm volatile("fence.proxy.async;" ::: "memory");
    return true;
}

// fp32 activation blocks in shared memory (see the head of the file): n16 pieces of 16 bytes at src, split by kSplitWarps warps.
// Heads in place, fp32 remainders at dst.
__device__ __forceinline__ void split_block32(unsigned src, unsigned dst, int n16, int first) {
#pragma unroll 4
    for (int i = first; i < n16; i += kSplitWarps * 32) {
        const uint4 u = lds128(src + 16u * i);
        const float v[4] = {__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z), __uint_as_float(u.w)};
        float h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) h[e] = tf32_head(v[e]), l[e] = __fsub_rn(v[e], h[e]);
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(src + 16u * i), "f"(h[0]), "f"(h[1]), "f"(h[2]), "f"(h[3]) : "memory");
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + 16u * i), "f"(l[0]), "f"(l[1]), "f"(l[2]), "f"(l[3]) : "memory");
    }
}
// Heads (nearest) in place; at dst per pixel 32 channels in bf16, then their 32 remainders, in the swizzle TMA would have used
// (16-byte piece j of row r lies at j ^ (r mod 8)).  A lane takes two neighbouring pieces of a row, eight channels; lanes of odd
// rows store the two results the other way round, which keeps eight lanes on 32 different banks.
__device__ __forceinline__ void split_block16(unsigned src, unsigned dst, int n16, int first) {
#pragma unroll 2
    for (int i = first; i < n16 >> 1; i += kSplitWarps * 32) {
        const unsigned r = (unsigned)i >> 2, m = (unsigned)i & 3u, x7 = r & 7u;
        const unsigned row = src + (r << 7), p0 = row + (((2 * m) ^ x7) << 4), p1 = row + (((2 * m + 1) ^ x7) << 4);
        const uint4 u0 = lds128(p0), u1 = lds128(p1);
        const float v[8] = {__uint_as_float(u0.x), __uint_as_float(u0.y), __uint_as_float(u0.z), __uint_as_float(u0.w),
                            __uint_as_float(u1.x), __uint_as_float(u1.y), __uint_as_float(u1.z), __uint_as_float(u1.w)};
        float h[8];
        unsigned w16[4], l16[4];
#pragma unroll
        for (int e = 0; e < 8; ++e) h[e] = tf32_near(v[e]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            w16[e] = bf16x2_sat(v[2 * e], v[2 * e + 1]);
            l16[e] = bf16x2_sat(__fsub_rn(v[2 * e], h[2 * e]), __fsub_rn(v[2 * e + 1], h[2 * e + 1]));
        }
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p0), "f"(h[0]), "f"(h[1]), "f"(h[2]), "f"(h[3]) : "memory");
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p1), "f"(h[4]), "f"(h[5]), "f"(h[6]), "f"(h[7]) : "memory");
        const unsigned at = dst + (r << 7) + ((m ^ x7) << 4);   // (the remainders: the same with bit 6 flipped)
        const bool odd = (r & 1u) != 0;
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(odd ? at ^ 64u : at), "r"(odd ? l16[0] : w16[0]),
                     "r"(odd ? l16[1] : w16[1]), "r"(odd ? l16[2] : w16[2]), "r"(odd ? l16[3] : w16[3])
                     : "memory");
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(odd ? at : at ^ 64u), "r"(odd ? w16[0] : l16[0]),
                     "r"(odd ? w16[1] : l16[1]), "r"(odd ? w16[2] : l16[2]), "r"(odd ? w16[3] : l16[3])
                     : "memory");
    }
}

// What a launch is known to be when its kernel is compiled (0: anything).  Every launch starts on cold instruction caches,
// and a layer of the small networks is over after three microseconds: the general kernel is 220 KB of code of which a
// launch runs a tenth, in pieces all over it.  A form has nothing in it but what its launches run (25 to 50 KB).  Measured,
// launches back to back: 1x1 128->128 @40x40 batch 1 3.97 -> 3.3 us, 3x3 128->128 @40x40 7.0 -> 6.2, and large layers gain
// too: 3x3 32->32 @160x160 batch 16 36.9 -> 31.3, 1x1 256->1024 @50x68 batch 4 14.9 -> 13.3.
//   bits 0-1  1 = 1x1, filters on M; 2 = 1x1, positions on M; 3 = 3x3 with three taps per weight stage
//   bits 2-4  activation + 1 (0: from the arguments; 4: SiLU in the exponential form)
//   bit 5     cut along K
//   bits 6-7  residual operand: 0 none, 1 in front of the activation, 2 behind it, 3 from the arguments
//   bit 8     the output is NCHW
//   bit 9     element stores (no residual): filter counts of no multiple of eight, unaligned channel slices
// Forms are for 16-bit data; but for bit 9, channels-last outputs leave in whole 16-byte pieces.
//   bit 10    fp32 with bf16 corrections (the only form of fp32 data; as a run-time branch it cost narrow layers without them 4 %)
//   bit 11    3x3 of stride 2 in two activation stages a channel block (TcArgs::half)
constexpr int kFormElem = 512, kFormCorr = 1024, kFormHalf = 2048;
constexpr int form_of(int kind, int act, bool split, int res, bool nchw) { return kind | (act + 1) << 2 | (split ? 32 : 0) | res << 6 | (nchw ? 256 : 0); }

// kRep: the launch follows a layout pass (rtoss_launch_conv_tc_repacked): 16-bit outputs may be NCHW and SiLU takes its
// exponential form.  An instantiation of its own: carried as run-time branches the two cost every other launch 0.5-1 %.
template <typename T, typename G, bool kRep = false, int kForm = 0>
__global__ void __launch_bounds__(kThreadsOf<T>, 1)
conv_tc_kernel(const __grid_constant__ G g) {
    constexpr bool kMulti = sizeof(G) > sizeof(TcLaunch1);
    constexpr bool kF32 = sizeof(T) == 4;   // fp32 data: tf32 instructions, three products per tap (see the head of the file)
    constexpr bool kAny = (kForm & ~kFormCorr) == 0;
    constexpr bool kCorr1 = (kForm & kFormCorr) != 0;   // (fp32, one convolution: whether a.idesc16; several: as it says)
    constexpr int kKind = kForm & 3, kAct = ((kForm >> 2) & 7) - 1;   // (kAny: both from the arguments)
    constexpr bool kSplitF = (kForm & 32) != 0, kNchw = (kForm & 256) != 0;
    constexpr int kRes = (kForm >> 6) & 3;
    constexpr bool kHalf = (kForm & kFormHalf) != 0;   // (forms only: as a run-time branch it costs the launches without it)
    constexpr bool kElem = (kForm & kFormElem) != 0;
    constexpr bool kActKnown = kAct >= 0;
    constexpr int kActC = kActKnown ? kAct : 0;
    extern __shared__ unsigned char smem_dyn[];
    // tiles need 1024-byte alignment for the 128-byte swizzle pattern
    const unsigned base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const unsigned sA = base;                                        // the ring area: a problem's [NA][a_stage], then its [NB][b_stage]
    const unsigned sBar = sA + (unsigned)g.ring_bytes;               // barriers, 8 bytes each
    const unsigned bar_fullA = sBar, bar_emptyA = sBar + 8 * kMaxA;
    const unsigned bar_fullB = bar_emptyA + 8 * kMaxA, bar_emptyB = bar_fullB + 8 * kMaxB;
    const unsigned bar_accFull = bar_emptyB + 8 * kMaxB, bar_accEmpty = bar_accFull + 16;
    const unsigned bar_loFull = bar_accEmpty + 16;   // fp32: activation stage split into heads and remainders
    // A CTA passing from a problem to one of another ring geometry: the MMA thread commits here once everything it
    // issued for the old problem has completed, i.e. has read its operands; both producers wait for that before they
    // write the first stage of the new layout over the old one.
    const unsigned bar_switch = bar_loFull + 8 * kMaxA;
    const unsigned s_tmem_ptr = bar_switch + 16;   // (what follows needs 16-byte alignment)
    volatile unsigned* tmem_ptr_gen = reinterpret_cast<volatile unsigned*>(smem_dyn + (s_tmem_ptr - smem_u32(smem_dyn)));
    unsigned char* epi_patch = smem_dyn + (s_tmem_ptr + 16 - smem_u32(smem_dyn));  // [kEpiWarps][kPatchBytes], 16-byte aligned
    uint2* pos_tab_all = reinterpret_cast<uint2*>(epi_patch + kEpiWarps * kPatchBytes);  // [n_tabs][kMaxPx]
    const unsigned s_tab_all = s_tmem_ptr + 16 + kEpiWarps * kPatchBytes;                // the same, as a shared address
    const unsigned s_res = sA + (unsigned)g.res_off;   // [kEpiWarps][kResStage], present when a call has a residual operand

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles = g.unit_end[g.n_prob - 1];  // units of work over all problems: (tile, share of the channel blocks)
    // Programmatic dependent launch: the next kernel of the stream may start its own prologue now (on SMs this
    // grid leaves free); before its own griddepcontrol.wait it reads nothing but handles (see conv_common.cuh).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (threadIdx.x == 0) {
        for (int i = 0; i < g.max_na; ++i) {
            mbar_init(bar_fullA + 8 * i, 1);
            mbar_init(bar_emptyA + 8 * i, 1);
            mbar_init(bar_loFull + 8 * i, kSplitWarps);
        }
        for (int i = 0; i < g.max_nb; ++i) {
            mbar_init(bar_fullB + 8 * i, 1);
            mbar_init(bar_emptyB + 8 * i, 1);
        }
        mbar_init(bar_switch, 1);
        for (int i = 0; i < g.AS; ++i) {
            mbar_init(bar_accFull + 8 * i, 1);
            mbar_init(bar_accEmpty + 8 * i, kEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int i = 0; i < g.n_prob; ++i) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&g.tmA[i]) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&g.tmB[i]) : "memory");
        }
    }
    // Where position p of a tile's list lies: the same for every tile (the tile's origin and the image's edges
    // come in per tile), so the epilogue looks it up instead of dividing.  {element offset from the tile's first
    // output, row << 16 | column}; positions that are no output (pitch padding, the list's tail) get 0xFFFFFFFF.
    for (int q = threadIdx.x; q < g.n_tabs * kMaxPx; q += kThreadsOf<T>) {
        int owner = 0;   // (any problem that uses the table describes it)
        while (owner + 1 < g.n_prob && g.prob[owner].tab != q / kMaxPx) ++owner;
        const TcArgs& a = g.prob[owner];
        const int p = q % kMaxPx;
        const int oyl = p / a.Wq, oxl = p - oyl * a.Wq;
        const bool is_out = p < a.N_px && oyl < a.TH && oxl < a.TW;
        pos_tab_all[q] = make_uint2((unsigned)((oyl * a.Wo + oxl) * a.y_c_stride), is_out ? (unsigned)(oyl << 16 | oxl) : 0xFFFFFFFFu);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_tmem_ptr), "r"(g.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem_base = *tmem_ptr_gen;
    // Everything above (barriers, TMEM, descriptor prefetch) touched no tensor.  What depends on the kernels before this
    // one in the stream -- the activations, the bias, the residual operand, and y, which they may still read -- is only
    // touched behind a griddepcontrol.wait, which the activation producer and the epilogue warps execute at the top of
    // their roles.  The weights and the issue words are not: they are constant while a network runs, and the kernels
    // that write them (packing) never let a successor start early, so the weight producer and the MMA thread begin at
    // once and the weight ring is full by the time the activations may be fetched.

    // Every role walks the same list of tiles: tile = blockIdx.x, + gridDim.x, ...  A tile is (image,
    // row band, filter tile) with the filter tile fastest, so CTAs working side by side read the same
    // activations from L2.  Stage counters run on across tiles, which lets the producer fetch the next
    // tile's operands while the current one is still being multiplied, and the two accumulator stages
    // let the epilogue of one tile run under the MMAs of the next.
    if (warp == 0) {
        // ---------------- TMA producer of the activations.  Issuing a bulk copy keeps its thread busy for some
        // hundred cycles whatever the size, so the activations and the weights have a producer thread each, and a
        // weight stage (G taps) is ONE copy.
        asm volatile("griddepcontrol.wait;" ::: "memory");   // the activations come from the kernels before this one
        if (lane == 0) {
            bool ok = true;
            Ring ra;
            int hq = 0;          // TcArgs::half: 0 or 2, which half of the order the coming block takes
            int pi = 0, cur_pi = -1;
            unsigned n_sw = 0;   // geometry changes so far
            for (int unit = blockIdx.x; unit < n_tiles && ok; unit += gridDim.x) {
                int local;
                pi = find_problem<kMulti>(g, unit, local, pi);
                const TcArgs& a = g.prob[pi];
                if (kMulti && pi != cur_pi) {
                    // another problem: if its rings are laid out differently, the old ones must have run empty; if it
                    // depends on problems of this launch, they must be complete
                    const bool regeo = cur_pi >= 0 && a.geo != g.prob[cur_pi].geo;
                    if (regeo) ok = mbar_wait(bar_switch, n_sw & 1u, g.wait_cycles);
                    if (ok && a.dep_mask) ok = wait_deps(g, a.dep_mask);
                    if (regeo) {
                        ++n_sw;
                        ra.s = 0;
                    }
                    cur_pi = pi;
                }
                const TileIdx ti = tile_of(a, local);
                const int ks = ti.ks, n = ti.n;
                const int y0 = ti.ty * a.TH, x0 = ti.tx * a.TW;
                const int cb_end = min(a.ncb, (ks + 1) * a.cb_per);
                for (int cb = ks * a.cb_per; cb < cb_end; ++cb) {
                    const int n_sub = (kKind == 1 || kKind == 2) ? 1 : kHalf ? 2 : a.n_sub;
                    auto fill = [&](int sub0) {   // one stage, sub-tiles sub0 and up
                        const int sa = ra.s;
                        ok = ok && mbar_wait(bar_emptyA + 8 * sa, ra.parity() ^ 1, g.wait_cycles);
                        if (!ok) return;
                        mbar_expect_tx(bar_fullA + 8 * sa, a.a_tx_bytes * n_sub);
                        for (int sub = 0; sub < n_sub; ++sub)
                            tma_load_4d(sA + sa * a.a_stage + sub * a.sub_bytes, &g.tmA[pi], cb * a.cb_ch, x0 * a.S + a.x_add[sub0 + sub],
                                        y0 * a.S + a.y_add[sub0 + sub], n, bar_fullA + 8 * sa);
                        ra.advance(a.NA);
                    };
                    if constexpr (kHalf) {   // the odd rows, then the even ones
                        ra.s = (int)(a.half >> (2 * hq)) & 3;
                        fill(2);
                        ra.s = (int)(a.half >> (2 * hq + 2)) & 3;
                        hq ^= 2;
                    }
                    fill(0);
                    if (!ok) break;
                }
            }
            if (!ok) atomicExch(g.status, 1);
        }
        __syncwarp();  // lanes 1..31 wait here for lane 0: the warp reaches the final barrier as one
    } else if (warp == kWeightWarp) {
        // ---------------- TMA producer of the weights: per tile and channel block, taps / G stages of G taps each
        if (lane == 0) {
            bool ok = true;
            Ring rb;
            int pi = 0, cur_pi = -1;
            unsigned n_sw = 0;
            for (int unit = blockIdx.x; unit < n_tiles && ok; unit += gridDim.x) {
                int local;
                pi = find_problem<kMulti>(g, unit, local, pi);
                const TcArgs& a = g.prob[pi];
                if (kMulti && pi != cur_pi) {
                    if (cur_pi >= 0 && a.geo != g.prob[cur_pi].geo) {   // the old rings must have run empty
                        ok = mbar_wait(bar_switch, n_sw & 1u, g.wait_cycles);
                        if (!ok) break;
                        ++n_sw;
                        rb.s = 0;
                    }
                    cur_pi = pi;
                }
                const unsigned sB = sA + a.sB_off;
                const TileIdx ti = tile_of(a, local);
                const int ks = ti.ks, cot = ti.cot;
                const int co0 = cot * ((kAny ? a.pxm != 0 : kKind == 2) ? a.n_cols : kMTile);
                const int w_taps = kAny ? a.taps : kKind == 3 ? 9 : 1, w_G = kAny ? a.G : kKind == 3 ? 3 : 1;
                const int cb_end = min(a.ncb, (ks + 1) * a.cb_per);
                for (int cb = ks * a.cb_per; cb < cb_end && ok; ++cb) {
                    for (int t0 = 0; t0 < w_taps; t0 += w_G) {
                        const int sb = rb.s;
                        ok = mbar_wait(bar_emptyB + 8 * sb, rb.parity() ^ 1u, g.wait_cycles);
                        if (!ok) break;
                        // (failure-detection hook: the launch's very first weight copy is withheld, so the wait for it runs out)
                        if (!(g.inject == 1 && unit == (int)blockIdx.x && cb == ks * a.cb_per && t0 == 0)) {
                            mbar_expect_tx(bar_fullB + 8 * sb, a.b_tx_bytes * w_G);
                            tma_load_3d(sB + sb * a.b_stage, &g.tmB[pi], cb * a.cb_ch, co0, t0, bar_fullB + 8 * sb);
                        }
                        rb.advance(a.NB);
                    }
                }
                if (!kMulti && a.resident) break;
            }
            if (!ok) atomicExch(g.status, 4);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer (the whole warp, see umma_f16)
        {
            const unsigned leader = elect_one();
            // One thread issues every tcgen05.mma, so the instructions between two of them are the budget: with one or
            // two instructions per tap (few channels, or few filters with the positions as M) the tensor pipe waits
            // for this thread.  Hence: ring positions and phases are carried as counters (no division), a descriptor
            // is a constant high word plus address / 16 in the low word (addresses stay below 2^18: adding never
            // carries out of the field), a tap's offset is a register picked by a compile-time index (the taps of
            // a 3x3 layer are unrolled), and K steps (+2 = 32 bytes = 16 channels) or the second half of the
            // positions (+1024 = 128 rows) are additions.
            bool ok = true;
            const unsigned desc_lo0 = (unsigned)make_sw_desc(0, 128);   // (the lower word does not depend on the row size)
            // per problem (recomputed when a tile belongs to another problem than the one before)
            unsigned tap16[9], wtile16 = 0, idesc = 0, hi_cols = 0, astage16 = 0, bstage16 = 0, sB = 0, desc_hi = 0, half16 = 0;
            int NA = 1, NB = 1;
            bool pxm = false, two = false, unrolled9 = false;
            int cur_pi = -1, pi = 0;
            const unsigned bar_rdyA = kF32 ? bar_loFull : bar_fullA;   // the barrier that says an activation stage may be read
            Ring ra, rb;
            int hq = 0;                         // (as the activation producer's)
            int as = 0, n_done = 0;
            unsigned pacc = 0;                  // phase parity of the accumulator ring
            const unsigned flip_b = !kMulti && g.prob[0].resident ? 0u : 1u;   // (see TcArgs::resident)
            unsigned peek = 0;                  // what umma_block_peek saw of the stages now current
            int since_res = 1 << 20;            // tiles issued since this CTA's last tile with a residual operand
            auto mk = [&desc_hi](unsigned lo) { return ((unsigned long long)desc_hi << 32) | lo; };
            // all instructions of one tap: the K slabs named by m4 (times two halves of positions with the positions as M)
            auto issue_tap = [&](unsigned d_base, unsigned wl, unsigned xl, unsigned m4, unsigned& acc) {
                if (kAny && pxm) {
#pragma unroll
                    for (int k4 = 0; k4 < kKBlock / 16; ++k4) {
                        if (m4 & (1u << k4)) {
                            umma_f16<kF32>(leader, d_base, mk(xl + 2 * k4), mk(wl + 2 * k4), idesc, acc);
                            if (two) umma_f16<kF32>(leader, d_base + hi_cols, mk(xl + half16 + 2 * k4), mk(wl + 2 * k4), idesc, acc);
                            acc = 1;
                        }
                    }
                } else {
#pragma unroll
                    for (int k4 = 0; k4 < kKBlock / 16; ++k4) {
                        if (m4 & (1u << k4)) {
                            umma_f16<kF32>(leader, d_base, mk(wl + 2 * k4), mk(xl + 2 * k4), idesc, acc);
                            acc = 1;
                        }
                    }
                }
            };
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++n_done) {
                int local;
                pi = find_problem<kMulti>(g, tile, local, pi);
                const TcArgs& a = g.prob[pi];
                if (pi != cur_pi) {
                    if (kMulti && cur_pi >= 0 && a.geo != g.prob[cur_pi].geo) {
                        if (a.over_res) {
                            // The new rings cover the staging area of residual operands.  An epilogue that may still use it
                            // belongs to one of this CTA's last AS tiles (the accumulator stage of an older one has been
                            // waited for since), and only if that tile had a residual operand: `since_res` tiles ago or earlier.
                            int as_b = as;
                            unsigned pacc_b = pacc;
                            for (int i = 0; i < g.AS && i < n_done && ok; ++i) {
                                if (--as_b < 0) {
                                    as_b = g.AS - 1;
                                    pacc_b ^= 1;
                                }
                                if (i >= since_res) ok = mbar_wait(bar_accEmpty + 8 * as_b, pacc_b, g.wait_cycles);
                            }
                            if (!ok) break;
                        }
                        // rings of another layout: the producers may write them once everything issued so far has read its operands
                        umma_commit(leader, bar_switch);
                        ra.s = rb.s = 0;
                        peek = 0;
                    }
                    cur_pi = pi;
                    astage16 = a.a_stage >> 4;
                    bstage16 = a.b_stage >> 4;
                    sB = sA + a.sB_off;
                    NA = a.NA;
                    NB = a.NB;
#pragma unroll
                    for (int t = 0; t < 9; ++t) tap16[t] = (unsigned)(a.tap_sub[t] * a.sub_bytes + a.tap_shift[t] * a.row_bytes) >> 4;
                    wtile16 = (unsigned)(a.w_rows * a.row_bytes) >> 4;
                    desc_hi = a.desc_hi;
                    half16 = (unsigned)(128 * a.row_bytes) >> 4;   // the second 128 positions of a tile
                    idesc = a.idesc;
                    hi_cols = (unsigned)a.n_cols;
                    pxm = kAny ? a.pxm != 0 : kKind == 2;
                    two = a.MH == 2;
                    unrolled9 = kAny ? !kF32 && a.taps == 9 && a.G == 3 : kKind == 3;
                }
                const TileIdx ti = tile_of(a, local);
                const int ks = ti.ks, cb_end = min(a.ncb, (ks + 1) * a.cb_per);
                // which (tap, slab) pairs of this filter tile hold kept weights: one word per channel block, the next
                // block's word asked for while this block's instructions go out
                const unsigned long long* iss = a.issue ? a.issue + (size_t)ti.cot * a.ncb : nullptr;
                unsigned long long bits = iss ? __ldcg(iss + ks * a.cb_per) : ~0ull;
                ok = mbar_wait(bar_accEmpty + 8 * as, pacc ^ 1, g.wait_cycles);  // epilogue has drained this stage
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const unsigned d_base = tmem_base + (unsigned)(as * g.acc_stride);
                unsigned acc = 0;  // the first instruction of a tile overwrites the accumulator
                int left = a.Cin - ks * a.cb_per * a.cb_ch;
                for (int cb = ks * a.cb_per; cb < cb_end && ok; ++cb, left -= a.cb_ch) {
                    // 32-byte slabs of this block that hold channels (the rest of the row is TMA zero fill)
                    constexpr int kSlab = kF32 ? 8 : 16;
                    const int nk4 = (min(left, a.cb_ch) + kSlab - 1) / kSlab;
                    const unsigned nkmask = (1u << nk4) - 1u;
                    if (kHalf) ra.s = (int)(a.half >> (2 * hq)) & 3;
                    const int sa = ra.s;
                    if (kAny ? a.taps == 1 : kKind != 3) {
                        const int sb = rb.s;
                        if (!(peek & 1u)) ok = mbar_wait(bar_rdyA + 8 * sa, ra.parity(), g.wait_cycles);
                        if (ok && !(peek & 2u)) ok = mbar_wait(bar_fullB + 8 * sb, rb.parity(), g.wait_cycles);
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        ra.advance(NA);   // now at the next stages, which the instruction below looks at
                        rb.advance(NB, flip_b);
                        const int sa_n = ra.s, sb_n = rb.s;
                        const unsigned pa_n = ra.parity(), pb_n = rb.parity();
                        const unsigned wl0 = desc_lo0 + (sB >> 4) + (unsigned)sb * bstage16;
                        const unsigned xl0 = desc_lo0 + (sA >> 4) + (unsigned)sa * astage16;
                        if (kAny ? !pxm : kKind != 2) {
                            peek = umma_block_peek<kF32>(d_base, mk(wl0), mk(xl0), idesc, acc, leader ? nkmask : 0u, bar_rdyA + 8 * sa_n, pa_n,
                                                   bar_fullB + 8 * sb_n, pb_n);
                        } else {
                            // positions on M: the first 128 positions with the look ahead, then the second 128
                            peek = umma_block_peek<kF32>(d_base, mk(xl0), mk(wl0), idesc, acc, leader ? nkmask : 0u, bar_rdyA + 8 * sa_n, pa_n,
                                                   bar_fullB + 8 * sb_n, pb_n);
                            if (two) {
                                unsigned acc2 = acc;
#pragma unroll
                                for (int k4 = 0; k4 < kKBlock / 16; ++k4) {
                                    if (k4 < nk4) {
                                        umma_f16<kF32>(leader, d_base + hi_cols, mk(xl0 + half16 + 2 * k4), mk(wl0 + 2 * k4), idesc, acc2);
                                        acc2 = 1;
                                    }
                                }
                            }
                        }
                        acc = 1;
                        umma_commit(kMulti || flip_b ? leader : 0u, bar_emptyB + 8 * sb);
                        umma_commit(leader, bar_emptyA + 8 * sa);
                        continue;
                    }
                    const unsigned long long bits_n = (iss && cb + 1 < cb_end) ? __ldcg(iss + cb + 1) : ~0ull;
                    if (!(peek & 1u)) ok = mbar_wait(bar_rdyA + 8 * sa, ra.parity(), g.wait_cycles);   // (peek stays 0 on the paths that do not look ahead)
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const unsigned xl0 = desc_lo0 + (sA >> 4) + (unsigned)sa * astage16;
                    ra.advance(NA);   // (sa stays this block's stage; ra is at the next one, which the look ahead reads)
                    if (kAny ? unrolled9 : kKind == 3) {
                        if (kHalf) ra.s = (int)(a.half >> (2 * hq + 2)) & 3;
                        const int sa_e = ra.s;   // (half: the stage of the even rows)
                        int sa_n = ra.s;
                        unsigned pa_n = ra.parity();
#pragma unroll
                        for (int s3 = 0; s3 < 3; ++s3) {
                            if (s3 == 1 && kHalf) {   // the even rows; the look ahead is for the next block from here on
                                if (!(peek & 1u)) ok = ok && mbar_wait(bar_rdyA + 8 * sa_e, ra.parity(), g.wait_cycles);
                                ra.advance(NA);
                                hq ^= 2;
                                ra.s = sa_n = (int)(a.half >> (2 * hq)) & 3;
                                pa_n = ra.parity();
                            }
                            if (s3 == 2 && kHalf && ok) umma_commit(leader, bar_emptyA + 8 * sa_e);
                            const unsigned xl = s3 == 1 && kHalf ? desc_lo0 + (sA >> 4) + (unsigned)sa_e * astage16 : xl0;
                            const int sb = rb.s;
                            if (!(peek & 2u)) ok = ok && mbar_wait(bar_fullB + 8 * sb, rb.parity(), g.wait_cycles);
                            if (ok) {
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                                const unsigned wl0 = desc_lo0 + (sB >> 4) + (unsigned)sb * bstage16;
                                const unsigned m_first = (unsigned)(bits >> (12 * s3)) & nkmask;
                                rb.advance(NB, flip_b);
                                if (kAny ? !pxm : true) {
                                    // the first tap of the stage goes out together with a look at the next stages
                                    peek = umma_block_peek<kF32>(d_base, mk(wl0), mk(xl + tap16[s3 * 3]), idesc, acc, leader ? m_first : 0u,
                                                           bar_rdyA + 8 * sa_n, pa_n, bar_fullB + 8 * rb.s, rb.parity());
                                    if (m_first) acc = 1;
#pragma unroll
                                    for (int i = 1; i < 3; ++i)
                                        issue_tap(d_base, wl0 + i * wtile16, xl + tap16[s3 * 3 + i],
                                                  (unsigned)(bits >> (12 * s3 + 4 * i)) & nkmask, acc);
                                } else {
#pragma unroll
                                    for (int i = 0; i < 3; ++i)
                                        issue_tap(d_base, wl0 + i * wtile16, xl + tap16[s3 * 3 + i],
                                                  (unsigned)(bits >> (12 * s3 + 4 * i)) & nkmask, acc);
                                }
                                umma_commit(kMulti || flip_b ? leader : 0u, bar_emptyB + 8 * sb);  // this weight stage may be refilled once the MMAs have read it
                            }
                        }
                    } else if constexpr (kAny) {
                        for (int t0 = 0; t0 < a.taps && ok; t0 += a.G) {
                            const int sb = rb.s;
                            ok = mbar_wait(bar_fullB + 8 * sb, rb.parity(), g.wait_cycles);
                            if (!ok) break;
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const unsigned wl0 = desc_lo0 + (sB >> 4) + (unsigned)sb * bstage16;
                            // weight tile v of the block: tap v (16-bit data); fp32: the heads of tap v, then (v >= 9 resp. 1) what
                            // corrects tap v - 9.  Heads meet the activations' heads and remainders, remainders the heads
                            // only; with bf16 corrections heads meet heads, and the rest is in the second arrays.
                            if (kF32 && (kMulti ? a.idesc16 != 0 : kCorr1)) {
                                const unsigned xr0 = xl0 + ((unsigned)a.lo_off >> 4);
                                for (int i = 0; i < a.G; ++i) {
                                    const int v = t0 + i, t = v >= 9 ? v - 9 : v;
                                    const unsigned off = (unsigned)(a.tap_sub[t] * a.sub_bytes + a.tap_shift[t] * a.row_bytes) >> 4;
                                    const unsigned m4 = (unsigned)(bits >> (4 * t)) & nkmask;
                                    if (v < 9) {
                                        issue_tap(d_base, wl0 + i * wtile16, xl0 + off, m4, acc);
                                        continue;
                                    }
                                    const unsigned wr = wl0 + i * wtile16, xr = xr0 + off;
#pragma unroll
                                    for (int h = 0; h < 2; ++h) {   // sixteen channels (a tap's heads came first: the accumulator holds something)
                                        if ((m4 >> (2 * h)) & 3u) {
                                            umma_f16<false>(leader, d_base, mk(wr + 2 * h), mk(xr + 4 + 2 * h), a.idesc16, 1u);
                                            umma_f16<false>(leader, d_base, mk(wr + 4 + 2 * h), mk(xr + 2 * h), a.idesc16, 1u);
                                        }
                                    }
                                }
                            } else {
                                for (int i = 0; i < a.G; ++i) {
                                    const int v = t0 + i, t = v >= a.taps_real ? v - a.taps_real : v;
                                    const unsigned off = (unsigned)(a.tap_sub[t] * a.sub_bytes + a.tap_shift[t] * a.row_bytes) >> 4;
                                    const unsigned m4 = (unsigned)(bits >> (4 * t)) & nkmask;
                                    issue_tap(d_base, wl0 + i * wtile16, xl0 + off, m4, acc);
                                    if (kF32 && v < a.taps_real) issue_tap(d_base, wl0 + i * wtile16, xl0 + off + ((unsigned)a.lo_off >> 4), m4, acc);
                                }
                            }
                            umma_commit(kMulti || flip_b ? leader : 0u, bar_emptyB + 8 * sb);
                            rb.advance(NB, flip_b);
                        }
                    }
                    if (ok) umma_commit(leader, bar_emptyA + 8 * sa);
                    bits = bits_n;
                }
                if (ok) umma_commit(leader, bar_accFull + 8 * as);
                since_res = a.resid ? 0 : since_res + 1;
                if (++as == g.AS) {
                    as = 0;
                    pacc ^= 1;
                }
            }
            // TMEM may only be released after the epilogue has drained the last tiles: the last min(AS, tiles done)
            // stages used, walking backwards from the ring position
            for (int i = 0; i < g.AS && i < n_done && ok && (kAny ? g.prob[0].KS == 1 : !kSplitF); ++i) {   // (split K: the cluster barriers below order it)
                if (--as < 0) {
                    as = g.AS - 1;
                    pacc ^= 1;
                }
                ok = mbar_wait(bar_accEmpty + 8 * as, pacc, g.wait_cycles);
            }
            if (!ok && leader) atomicExch(g.status, 2);
        }
        __syncwarp();
    } else if (kF32 && warp > kWeightWarp) {
        // ---------------- fp32: the warps that split the activation blocks.  x = head + remainder; the head takes the value's
        // place, the second half of the stage receives what the small products need.  Plain loads and stores; the fence hands
        // them to the proxy the tensor core reads through; then the stage is announced to the MMA thread.  Any word may be
        // split: rows the copy did not write are never outputs.
        bool ok = true;
        Ring ra;
        int pi = 0, cur_pi = -1;
        for (int unit = blockIdx.x; unit < n_tiles && ok; unit += gridDim.x) {
            int local;
            pi = find_problem<kMulti>(g, unit, local, pi);
            const TcArgs& a = g.prob[pi];
            if (kMulti && pi != cur_pi) {
                if (cur_pi >= 0 && a.geo != g.prob[cur_pi].geo) ra.s = 0;   // (a new layout's first stage is full only behind the switch)
                cur_pi = pi;
            }
            const int ks = tile_of(a, local).ks, cb_end = min(a.ncb, (ks + 1) * a.cb_per);
            for (int cb = ks * a.cb_per; cb < cb_end; ++cb, ra.advance(a.NA)) {
                if (lane == 0) ok = mbar_wait(bar_fullA + 8 * ra.s, ra.parity(), g.wait_cycles);
                ok = __shfl_sync(0xFFFFFFFFu, (int)ok, 0) != 0;
                if (!ok) break;
                __syncwarp();   // (lane 0 has seen the copy; a shuffle orders no memory, and all lanes read the block)
                const unsigned src = sA + ra.s * a.a_stage, dst = src + (unsigned)a.lo_off;
                const int n16 = (a.n_sub * a.sub_bytes) >> 4, first = (warp - kWeightWarp - 1) * 32 + lane;
                if (kMulti ? a.idesc16 != 0 : kCorr1) split_block16(src, dst, n16, first);
                else split_block32(src, dst, n16, first);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_loFull + 8 * ra.s) : "memory");
            }
        }
        if (!ok && lane == 0) atomicExch(g.status, 1);
        __syncwarp();
    } else {
        // ---------------- epilogue: TMEM -> registers -> bias / activation -> NHWC global
        asm volatile("griddepcontrol.wait;" ::: "memory");   // bias, residual and y belong to the stream's order
        const int quarter = warp & 3;      // TMEM lanes a warp may read: 32 * (warp id mod 4)
        const int sub = (warp - 2) >> 2;   // four warps share a lane quarter and take every fourth 32-column chunk
        bool ok = true;
        int gt = 0;
        if constexpr (!kF32 && (kAny || kKind == 2)) if (!kAny || g.prob[0].pxm) {
            // (a launch with the positions as M carries one problem; 16-bit data only)
            const TcArgs& a = g.prob[0];
            T* __restrict__ yg = reinterpret_cast<T*>(a.y);
            const uint2* pos_tab = pos_tab_all;
            // Positions are the TMEM lanes: a thread owns one position and reads its filters sixteen at a time, which
            // are contiguous in NHWC -- no transpose.  One filter tile covers the layer, so the bias is staged once.
            float* bias_s = reinterpret_cast<float*>(epi_patch);
            for (int i = threadIdx.x - 64; i < a.n_cols; i += kEpiWarps * 32)
                bias_s[i] = (a.bias && i < a.Cout) ? __ldg(a.bias + i) : 0.f;
            asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
            const int n_chunks = a.n_cols >> 4, items = a.MH * n_chunks;
            const bool vec_ok = (a.y_c_stride % 8 == 0) && (a.y_c_off % 8 == 0);
            int as = 0;
            unsigned pfull = 0;   // accumulator stage of this tile and the parity of its "full" phase
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++gt, pfull ^= (as + 1 == g.AS), as = as + 1 == g.AS ? 0 : as + 1) {
                const TileIdx ti = tile_of(a, tile);
                const int n = ti.n;
                const int y0 = ti.ty * a.TH, x0 = ti.tx * a.TW;
                ok = mbar_wait(bar_accFull + 8 * as, pfull, g.wait_cycles);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const unsigned d_base = tmem_base + (unsigned)(as * g.acc_stride) + ((unsigned)(quarter * 32) << 16);
                T* yb = (kRep || kNchw) ? yg + (size_t)n * a.y_img + ((size_t)y0 * a.Wo + x0) * a.y_c_stride + (size_t)a.y_c_off * a.y_co
                             : yg + (((size_t)n * a.Ho + y0) * a.Wo + x0) * a.y_c_stride + a.y_c_off;
                const unsigned ry = (unsigned)min(a.TH, a.Ho - y0), rx = (unsigned)min(a.TW, a.Wo - x0);
                for (int item = sub; item < items; item += 4) {
                    const int h = item / n_chunks, c = item - h * n_chunks;
                    unsigned r[16];
                    tmem_ld16(d_base + (unsigned)(h * a.n_cols + c * 16), r);
                    const uint2 e = pos_tab[h * 128 + quarter * 32 + lane];
                    const bool px_ok = (e.y >> 16) < ry && (e.y & 0xFFFFu) < rx;
                    const float* b16 = bias_s + c * 16;
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    unsigned o[8];
                    if constexpr (kActKnown) act_pack16<T, kActC>(r, b16, o);
                    else if (a.act == RTOSS_ACT_SILU) act_pack16<T, RTOSS_ACT_SILU>(r, b16, o);
                    else if (a.act == RTOSS_ACT_RELU) act_pack16<T, RTOSS_ACT_RELU>(r, b16, o);
                    else if (kRep && a.act == kActSiluX) act_pack16<T, kActSiluX>(r, b16, o);
                    else act_pack16<T, RTOSS_ACT_NONE>(r, b16, o);
                    if (px_ok) {
                        T* dst = yb + e.x + (kRep || kNchw ? (size_t)(c * 16) * a.y_co : (size_t)(c * 16));   // (NCHW: a store covers 32 neighbouring positions of a filter)
                        if (!kNchw && vec_ok && c * 16 + 16 <= a.Cout) {
                            reinterpret_cast<uint4*>(dst)[0] = make_uint4(o[0], o[1], o[2], o[3]);
                            reinterpret_cast<uint4*>(dst)[1] = make_uint4(o[4], o[5], o[6], o[7]);
                        } else {
                            // NCHW, ragged filter count or unaligned channel slice: element stores
                            const T* ov = reinterpret_cast<const T*>(o);
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (c * 16 + j < a.Cout) dst[kRep || kNchw ? (size_t)j * a.y_co : (size_t)j] = ov[j];
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_accEmpty + 8 * as) : "memory");
            }
            gt = -1;   // (done: the loop below does not run)
        }
        int pi = 0, as = 0;
        unsigned pfull = 0;   // accumulator stage of this tile and the parity of its "full" phase
        if constexpr (kAny || kKind != 2) for (int tile = blockIdx.x; gt >= 0 && tile < n_tiles && ok; tile += gridDim.x, ++gt, pfull ^= (as + 1 == g.AS), as = as + 1 == g.AS ? 0 : as + 1) {
            int local;
            pi = find_problem<kMulti>(g, tile, local, pi);
            const TcArgs& a = g.prob[pi];
            T* __restrict__ yg = reinterpret_cast<T*>(a.y);
            const uint2* pos_tab = pos_tab_all + a.tab * kMaxPx;
            const unsigned s_tab = s_tab_all + (unsigned)a.tab * kMaxPx * 8;
            const TileIdx ti = tile_of(a, local);   // a unit is (tile proper, share of the channel blocks)
            const int n = ti.n;
            const int y0 = ti.ty * a.TH, x0 = ti.tx * a.TW, co0 = ti.cot * kMTile;
            // Everything that does not need the accumulator comes before the wait for it: the bias is a global load
            // (a cold one costs more than a thousand cycles) and would otherwise sit on the path of every tile.
            // TMEM lane = filter.  A narrow layer's filters are repeated down the lanes (R copies): every lane quarter
            // then holds outputs, and the copies share the tile's columns between them.
            const int copy = (quarter * 32) >> a.rep_shift, row0 = quarter * 32 - (copy << a.rep_shift);   // (rep_rows is 32, 64 or 128)
            const int co = co0 + row0 + lane;
            const bool co_ok = co < a.Cout;
            const float bv = (a.bias && co_ok) ? __ldg(a.bias + co) : 0.f;
            const unsigned patch = s_tmem_ptr + 16 + (unsigned)(warp - 2) * kPatchBytes;  // shared address
            // (fp32 outputs leave through the element stores below: a warp's 32 filters of one position are 128 contiguous bytes)
            const bool vec_ok = !kAny ? !kNchw && !kElem && co0 + row0 < a.Cout : !kF32 && (a.y_c_stride % 8 == 0) && ((a.y_c_off + co0) % 8 == 0) && (co0 + row0 + 32 <= a.Cout);
            T* yb = (kRep || kNchw) ? yg + (size_t)n * a.y_img + ((size_t)y0 * a.Wo + x0) * a.y_c_stride + (size_t)(a.y_c_off + co0 + row0) * a.y_co
                         : yg + (((size_t)n * a.Ho + y0) * a.Wo + x0) * a.y_c_stride + a.y_c_off + co0 + row0;
            const int n_co = a.Cout - co0 - row0;   // this quarter's filters inside the layer (at most 32 count)
            unsigned ry = (unsigned)min(a.TH, a.Ho - y0);   // rows / columns inside the image
            const unsigned rx = (unsigned)min(a.TW, a.Wo - x0);
            if (!kAny && !kNchw && !kElem && co0 + row0 + 8 * (lane & 3) >= a.Cout) ry = 0;   // this lane's eight filters are beyond the layer
            const int c_first = (sub + 4 * copy) * 32, c_step = 128 * a.R;
            const T* rb = (kAny ? a.resid != nullptr : kRes != 0) ? reinterpret_cast<const T*>(a.resid) + (yb - yg) : nullptr;   // laid out like y
            const bool post = (kAny || kRes == 3) ? a.resid_post != 0 : kRes == 2;
            const float bs = (!kF32 && (kActKnown ? kAct : a.act) == RTOSS_ACT_SILU && (!rb || post)) ? 0.5f * bv : bv;   // (a residual in front of the activation, or fp32 data: plain bias)
            ok = mbar_wait(bar_accFull + 8 * as, pfull, g.wait_cycles);
            if (!ok && (kAny ? a.KS == 1 : !kSplitF)) break;   // (split K: the cluster barriers below must still be passed)
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned d_base = tmem_base + (unsigned)(as * g.acc_stride) + ((unsigned)(quarter * 32) << 16);
            if (kAny ? a.KS > 1 : kSplitF) {
                // ---- split K.  The KS CTAs of the cluster hold the partial sums of one tile.  Barrier 1: every CTA's
                // MMAs have completed, so the operand rings of all of them are free; each CTA then stores its partial
                // sums of chunk c into the shared memory of the chunk's owner (rank c % KS); barrier 2: all stores have
                // landed; every CTA adds up and finishes the chunks it owns.  Every thread of the cluster passes both
                // barriers, whatever happened to its waits (the other roles pass them at the end of the kernel).
                const int rank = (int)cluster_rank(), n_chunks = (a.N_px + 31) >> 5, n_lc = (n_chunks + a.KS - 1) / a.KS;
                cluster_sync_all();
                if (ok) {
                    for (int c0 = c_first; c0 < a.N_px; c0 += c_step) {
                        unsigned r[32];
                        tmem_ld32(d_base + (unsigned)c0, r);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        const int c = c0 >> 5;
                        const unsigned dst = peer_smem(sA + (unsigned)((((rank * n_lc + c / a.KS) * 32) * 128 + quarter * 32 + lane) * 4),
                                                       (unsigned)(c % a.KS));
#pragma unroll
                        for (int j = 0; j < 32; ++j) st_peer_f32(dst + j * 512, __uint_as_float(r[j]));   // 128 contiguous bytes per warp
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                cluster_sync_all();
                if (ok) {
                    const int row = quarter * 32 + lane;
#define RTOSS_SHARES(ACT_) \
        epilogue_from_shares<T, ACT_, !kAny && !kElem>(sA, a.KS, rank, n_lc, sub, row, a.N_px, bs, vec_ok, co_ok, patch, s_tab, pos_tab, yb, ry, rx, lane, rb, post, kNchw || (kRep && a.nchw), n_co, a.y_co)
                    if constexpr (kActKnown) RTOSS_SHARES(kActC);
                    else if (a.act == RTOSS_ACT_SILU) RTOSS_SHARES(RTOSS_ACT_SILU);
                    else if (a.act == RTOSS_ACT_RELU) RTOSS_SHARES(RTOSS_ACT_RELU);
                    else if (kRep && a.act == kActSiluX) RTOSS_SHARES(kActSiluX);
                    else RTOSS_SHARES(RTOSS_ACT_NONE);
#undef RTOSS_SHARES
                }
                continue;
            }
            bool stored = !kAny && !kElem;
            if constexpr (!kF32) {
                if (vec_ok) {
                    stored = true;
                    if (kAny ? rb != nullptr : kRes != 0) {
                        const unsigned stage = s_res + (unsigned)(warp - 2) * kResStage;
#define RTOSS_RES_CALL(ACT_, POST_) \
        epilogue_chunks_res<T, ACT_, POST_>(d_base, c_first, c_step, a.N_px, bs, patch, s_tab, yb, ry, rx, lane, rb, stage)
                        if constexpr (kActKnown && (kRes == 1 || kRes == 2)) {
                            RTOSS_RES_CALL(kActC, (kRes == 2 && kActC != RTOSS_ACT_NONE));
                        } else if (post) {
                            if (a.act == RTOSS_ACT_SILU) RTOSS_RES_CALL(RTOSS_ACT_SILU, true);
                            else if (a.act == RTOSS_ACT_RELU) RTOSS_RES_CALL(RTOSS_ACT_RELU, true);
                            else RTOSS_RES_CALL(RTOSS_ACT_NONE, false);   // no activation: both orders are the same sum
                        } else {
                            if (a.act == RTOSS_ACT_SILU) RTOSS_RES_CALL(RTOSS_ACT_SILU, false);
                            else if (a.act == RTOSS_ACT_RELU) RTOSS_RES_CALL(RTOSS_ACT_RELU, false);
                            else RTOSS_RES_CALL(RTOSS_ACT_NONE, false);
                        }
#undef RTOSS_RES_CALL
                    } else {
#define RTOSS_CHUNKS(ACT_) epilogue_chunks<T, ACT_>(d_base, c_first, c_step, a.N_px, bs, patch, s_tab, yb, ry, rx, lane)
                        if constexpr (kActKnown) RTOSS_CHUNKS(kActC);
                        else if (a.act == RTOSS_ACT_SILU) RTOSS_CHUNKS(RTOSS_ACT_SILU);
                        else if (a.act == RTOSS_ACT_RELU) RTOSS_CHUNKS(RTOSS_ACT_RELU);
                        else if (kRep && a.act == kActSiluX) RTOSS_CHUNKS(kActSiluX);
                        else RTOSS_CHUNKS(RTOSS_ACT_NONE);
#undef RTOSS_CHUNKS
                    }
                } else if (kNchw || (kRep && a.nchw)) {
                    stored = true;
                    const bool pair_ok = (a.y_co & 1) == 0;
#define RTOSS_NCHW(ACT_) epilogue_chunks_nchw<T, ACT_>(d_base, c_first, c_step, a.N_px, bs, patch, s_tab, yb, ry, rx, lane, n_co, a.y_co, pair_ok)
                    if constexpr (kActKnown) RTOSS_NCHW(kActC);
                    else if (a.act == kActSiluX) RTOSS_NCHW(kActSiluX);
                    else if (a.act == RTOSS_ACT_RELU) RTOSS_NCHW(RTOSS_ACT_RELU);
                    else RTOSS_NCHW(RTOSS_ACT_NONE);
#undef RTOSS_NCHW
                }
            }
            if ((kAny || kElem) && !stored) {
                // ragged filter counts, unaligned channel slices, fp32 data: element stores, lane = filter
                const int act = kActKnown ? kActC : a.act;
                for (int c0 = c_first; c0 < a.N_px; c0 += c_step) {
                    unsigned r[32];
                    tmem_ld32(d_base + (unsigned)c0, r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const uint2 e = pos_tab[c0 + j];
                        const bool in_img = co_ok && (e.y >> 16) < ry && (e.y & 0xFFFFu) < rx;
                        float v = __uint_as_float(r[j]) + bv;
                        if (rb && in_img && !post) v = to_f32<T>(from_f32<T>(v)) + to_f32<T>(__ldcg(rb + e.x + lane));   // round, then add the residual
                        if (act == RTOSS_ACT_RELU) v = fmaxf(v, 0.f);
                        if (act == RTOSS_ACT_SILU) {
                            if (kF32) {
                                v = silu_f32(v);
                            } else {
                                float th;
                                asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(0.5f * v));
                                v = v * fmaf(0.5f, th, 0.5f);
                            }
                        }
                        if ((kRep || kElem) && act == kActSiluX) v = silu_exp(v);
                        if (rb && in_img && post) v = to_f32<T>(from_f32<T>(v)) + to_f32<T>(__ldcg(rb + e.x + lane));   // behind the activation
                        if (co_ok && (e.y >> 16) < ry && (e.y & 0xFFFFu) < rx) yb[e.x + lane] = from_f32<T>(v);
                    }
                }
            }
            // this warp has read everything it needs from the accumulator stage
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_accEmpty + 8 * as) : "memory");
            if (kMulti && g.done && tile + (int)gridDim.x >= g.unit_end[pi]) {
                // This was the CTA's last tile of the problem: the warp reports its share of the outputs written.  The
                // lanes' stores are ordered before lane 0's fence by the __syncwarp above, the fence before the count.
                if (lane == 0) {
                    __threadfence();
                    atomicAdd(g.done + pi, 1u);
                }
            }
        }
        if (!ok && lane == 0) atomicExch(g.status, 3);
    }

    if ((kAny ? g.prob[0].KS > 1 : kSplitF) && (warp < 2 || warp >= kWeightWarp)) {   // (a launch cut along K carries one problem)   // split K: the barriers the epilogue warps pass around the exchange
        cluster_sync_all();
        cluster_sync_all();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(g.tmem_cols) : "memory");
    }
    if (kMulti && g.done && threadIdx.x == 0) {
        // The completion counters go back to zero for the next launch: by the last CTA to get here, when no CTA of this
        // launch reads them any more.
        __threadfence();
        if (atomicAdd(g.done + kMaxProb, 1u) == gridDim.x - 1) {
            for (int i = 0; i <= kMaxProb; ++i) g.done[i] = 0u;
        }
    }
}

}  // namespace

#endif
