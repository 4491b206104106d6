// Per-kernel arithmetic of pattern selection and packing (Algorithm 2; Algorithm 3 after regrouping), shared by
// the single-layer kernels and the whole-model batch so that both give the same bits.
#ifndef RTOSS_SELECT_CORE_CUH
#define RTOSS_SELECT_CORE_CUH

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

namespace rtoss_dev {

// Squares in fp32, pattern sums in fp32 over ascending taps, first strictly larger sum wins (ties -> lowest id,
// a NaN sum never wins).  __fmul_rn / __fadd_rn keep the compiler from contracting or reordering the arithmetic.
// `tab[p]` is the 9-bit mask of pattern p.
template <typename Tab>
__device__ __forceinline__ int select_best(const float (&w)[9], const Tab& tab, int P) {
    float q[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) q[t] = __fmul_rn(w[t], w[t]);
    int best = 0;
    float best_s = 0.f;
    for (int p = 0; p < P; ++p) {
        const unsigned m = tab[p];
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < 9; ++t)
            if (m & (1u << t)) s = __fadd_rn(s, q[t]);
        if (p == 0) {
            best_s = s;
        } else if (s > best_s || (best_s != best_s && s == s)) {
            best = p;
            best_s = s;
        }
    }
    return best;
}

// An fp32 value's tf32 head: the 19 leading bits; or the nearest value of 19 bits (a value that would round to infinity is cut
// off instead), whose remainder is half as large.
__device__ __forceinline__ float tf32_head(float f) { return __uint_as_float(__float_as_uint(f) & 0xFFFFE000u); }
__device__ __forceinline__ float tf32_near(float f) {
    const unsigned u = __float_as_uint(f);
    return __uint_as_float(((u << 1) >= 0xFEFFE000u ? u : u + 0x1000u) & 0xFFFFE000u);
}
// Two floats rounded to bf16, a in the low half; finite values stay finite.
__device__ __forceinline__ unsigned bf16x2_sat(float a, float b) {
    unsigned d;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}
// The second array of rtoss_f32_corr16 layers: weight and remainder of flat position f (rows are whole blocks of 32 channels)
// into its block; two neighbouring positions, the first even.
__device__ __forceinline__ uint16_t* corr16_at(float* lo, int64_t f) { return reinterpret_cast<uint16_t*>(lo) + 2 * (f & ~(int64_t)31) + (f & 31); }
__device__ __forceinline__ void put_corr16_one(uint16_t* at, float w, float rest) {
    const unsigned u = bf16x2_sat(w, rest);
    at[0] = (uint16_t)u;
    at[32] = (uint16_t)(u >> 16);
}
__device__ __forceinline__ void put_corr16_two(uint16_t* at, float w0, float w1, float rest0, float rest1) {
    *reinterpret_cast<unsigned*>(at) = bf16x2_sat(w0, w1);
    *reinterpret_cast<unsigned*>(at + 32) = bf16x2_sat(rest0, rest1);
}
template <typename V> __device__ __forceinline__ V narrow_to(float v);
template <> __device__ __forceinline__ float narrow_to<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 narrow_to<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ __half narrow_to<__half>(float v) { return __float2half_rn(v); }

// The dense expansion of one kernel (see pack_one).  fp32: the tensor path multiplies tf32 operands, so every weight is stored as its
// tf32 head and, in a second copy of the array behind the first, what corrects it: the remainder (exact in fp32), or two bf16
// numbers (rtoss_f32_corr16).  (A loop of its own for those: as a choice per tap it cost every fp32 layer, re-packing 64x36
// 6.5 -> 7.2 us.)
template <typename V>
__device__ __forceinline__ void expand_one(const float* w, unsigned m, int64_t i, V* __restrict__ wtc, int ksize, int Cin, int rows,
                                           int rep_rows, int copies, int cin_p) {
    const int64_t tap_step = (int64_t)rows * cin_p, copy_step = (int64_t)rep_rows * cin_p, lo_at = (ksize == 3 ? 9 : 1) * tap_step;
    auto put = [&](int64_t at, float f) {
        if constexpr (sizeof(V) == 4) {
            wtc[at] = tf32_head(f);
            wtc[lo_at + at] = __fsub_rn(f, tf32_head(f));
        } else {
            wtc[at] = narrow_to<V>(f);
        }
    };
    if (ksize != 3) {
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t at = i * 9 + t;   // flat position; rows are cin_p apart where they are padded
            if (cin_p != Cin) at += (int64_t)((unsigned)at / (unsigned)Cin) * (cin_p - Cin);
            put(at, (m & (1u << t)) ? w[t] : 0.f);
        }
        return;
    }
    // (layers hold fewer than 2^31 kernels: 32-bit division, several times cheaper than the 64-bit one)
    const int64_t co = (int64_t)((unsigned)i / (unsigned)Cin), p = co * cin_p + (i - co * Cin);   // copy 0 of tap 0; copy c lies c * rep_rows rows further down
    if constexpr (sizeof(V) == 4) {
        if (rtoss_f32_corr16(Cin, 3)) {
            V* at = wtc + p;
            uint16_t* lo = corr16_at(wtc + lo_at, p);   // (taps and copies lie whole blocks apart)
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const float f = (m & (1u << t)) ? w[t] : 0.f, h = tf32_near(f), rest = __fsub_rn(f, h);
                for (int c = 0; c < copies; ++c) {
                    at[t * tap_step + c * copy_step] = h;
                    put_corr16_one(lo + 2 * (t * tap_step + c * copy_step), f, rest);
                }
            }
            return;
        }
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        const float f = (m & (1u << t)) ? w[t] : 0.f;
        for (int c = 0; c < copies; ++c) put(p + t * tap_step + c * copy_step, f);
    }
}

// Writes of one kernel (3x3) or run of nine (1x1) with mask m: its k kept values, ascending taps, rounded to V, to
// val[i*k ...]; and, where the handle carries dense-expanded weights for the tensor path (wtc != nullptr), all nine
// taps, pruned ones as +0:  3x3 -> wtc[t][row][ci] with `rows` rows of cin_p channels per tap, filter co = i / Cin at rows
// c*rep_rows + co for c < copies (one copy at row co in the plain layout);  1x1 -> position 9*i + t of the flat matrix.  fp32 handles hold
// two such arrays back to back: tf32 heads, then what corrects them (expand_one).
template <typename V>
__device__ __forceinline__ void pack_one(const float (&w)[9], unsigned m, int64_t i, int k, V* __restrict__ val,
                                         V* __restrict__ wtc, int ksize, int Cin, int rows, int rep_rows, int copies, int cin_p) {
    V* out = val + i * k;
    if (k * (int)sizeof(V) == 8) {
        // the k kept values of a kernel are 8 aligned bytes (four 16-bit or two 32-bit values): pushed into a 64-bit word
        // from the top, tap by tap in ascending order, so that after k pushes the first kept value sits in the lowest
        // bits (a valid mask has exactly k bits); written with one store
        unsigned long long word = 0;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            if (m & (1u << t)) {
                const V v = narrow_to<V>(w[t]);
                unsigned long long bits;
                if constexpr (sizeof(V) == 4) {
                    bits = (unsigned long long)__float_as_uint(v);
                } else {
                    bits = (unsigned long long)*reinterpret_cast<const unsigned short*>(&v);
                }
                word = (word >> (8 * sizeof(V))) | (bits << (64 - 8 * sizeof(V)));
            }
        }
        *reinterpret_cast<unsigned long long*>(out) = word;
    } else {
        int j = 0;
#pragma unroll
        for (int t = 0; t < 9; ++t)
            if (m & (1u << t)) out[j++] = narrow_to<V>(w[t]);
    }
    if (wtc) expand_one<V>(w, m, i, wtc, ksize, Cin, rows, rep_rows, copies, cin_p);
}

// ---- two kernels per thread --------------------------------------------------------------------------------------
// The whole-model pass gives a thread two consecutive kernels: the pattern table's words and the tests of their bits are
// shared by two sums.

constexpr int kPair = 2;

// fp32 pairs in one register pair: one instruction rounds both halves as two single ones would (add.rn / mul.rn).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack_f32x2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack_f32x2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 mul_f32x2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// The thread's two kernels, tap t of both in q[t].
// fp32: nine 8-byte loads 72 bytes apart; 16 bits: nine 4-byte loads 36 apart (both free of bank conflicts).
template <typename T> __device__ __forceinline__ void load_pair(const unsigned char* raw, int pair, f32x2 (&q)[9]) {
    float w[18];
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        if constexpr (sizeof(T) == 4) {
            const float2 v = reinterpret_cast<const float2*>(raw)[pair * 9 + j];
            w[2 * j] = v.x, w[2 * j + 1] = v.y;
        } else {
            const unsigned v = reinterpret_cast<const unsigned*>(raw)[pair * 9 + j];
            if constexpr (std::is_same<T, __half>::value) {
                w[2 * j] = __half2float(__ushort_as_half((unsigned short)(v & 0xFFFFu)));
                w[2 * j + 1] = __half2float(__ushort_as_half((unsigned short)(v >> 16)));
            } else {
                w[2 * j] = __uint_as_float(v << 16);
                w[2 * j + 1] = __uint_as_float(v & 0xFFFF0000u);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) q[t] = pack_f32x2(w[t], w[9 + t]);
}

__device__ __forceinline__ f32x2 fma_f32x2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// A pattern as factors: 1 for a kept tap, 0 for a pruned one, each twice (one per kernel of the pair), padded to ten taps.
constexpr int kFactorPatterns = 64;
struct __align__(16) PatternFactors {
    f32x2 f[10];
};

// select_best for two kernels: the same sums in the same order.  q comes in as the weights and is squared here.  (Sums are
// never negative: starting from -1, the first sum that is a number wins, as in select_best.)
// A sum is nine fused multiply-adds with the pattern's factors: fma(1, q, s) is q + s rounded once and fma(0, q, s) is s,
// as long as no square is infinite or not a number -- such a pair takes the loop of predicated additions, and so do
// tables of more than kFactorPatterns patterns.  (Testing nine mask bits per pattern took 47 instructions per pattern and pair.)
template <int kUnroll, typename Tab>
__device__ __forceinline__ void select_best2(f32x2 (&q)[9], const Tab& tab, const PatternFactors* factors, int P, int (&best)[kPair]) {
    float best_s[kPair] = {-1.f, -1.f};
    best[0] = best[1] = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) q[t] = mul_f32x2(q[t], q[t]);
    f32x2 all = q[0];
#pragma unroll
    for (int t = 1; t < 9; ++t) all = fma_f32x2(q[t], pack_f32x2(1.f, 1.f), all);
    float a, b;
    unpack_f32x2(all, a, b);
    const float inf = __int_as_float(0x7F800000);
    if (P <= kFactorPatterns && a < inf && b < inf) {
#pragma unroll kUnroll
        for (int p = 0; p < P; ++p) {
            const ulonglong2* f = reinterpret_cast<const ulonglong2*>(factors[p].f);
            f32x2 s = 0;
#pragma unroll
            for (int h = 0; h < 5; ++h) {
                const ulonglong2 c = f[h];
                s = fma_f32x2(q[2 * h], c.x, s);
                if (h < 4) s = fma_f32x2(q[2 * h + 1], c.y, s);
            }
            unpack_f32x2(s, a, b);
            if (a > best_s[0]) best_s[0] = a, best[0] = p;
            if (b > best_s[1]) best_s[1] = b, best[1] = p;
        }
    } else {
#pragma unroll 1
        for (int p = 0; p < P; ++p) {
            const unsigned m = tab[p];
            f32x2 s = 0;
#pragma unroll
            for (int t = 0; t < 9; ++t)
                asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\t@p add.rn.f32x2 %0, %0, %2;\n\t}" : "+l"(s) : "r"(m & (1u << t)), "l"(q[t]));
            unpack_f32x2(s, a, b);
            if (a > best_s[0]) best_s[0] = a, best[0] = p;
            if (b > best_s[1]) best_s[1] = b, best[1] = p;
        }
    }
}

// Stable counting sort of the Cout filters of input channel ci by pattern id, by one warp: perm[ci*Cout + j] lists
// the filters by ascending id (ties by ascending filter), bucket_off[ci*(P+1) + p] is where pattern p starts.
// Ranks inside a group of 32 filters come from __match_any_sync.
// Ids must be < P; a filter whose id is not is left out of perm (the channel's list is then short by it, the last
// bucket ends before bucket_off's closing entry Cout) rather than written past the channel's slice.
//
// On the way the warp also records which taps the tensor path has to multiply at all: `issue` (nullable) holds one
// 64-bit word per (tile of 128 filters, block of 2^cb_log2 input channels: 64 for 16-bit handles, 32 for fp32 ones --
// 128 bytes of a row), bit 4 t + s set when some kernel of the tile with its channel in slab s (a quarter) of the
// block keeps tap t (the union of the kept taps over the tile, from
// `masks`, the table as the device sees it).  The words must be zero before the pass; channels add their bits with
// atomicOr.  A (tile, slab, tap) whose bit stays clear holds only pruned weights: its matrix instruction is skipped.
// The warp's shared memory: `fill`, 256 words (a pattern's count, later its next position), and `smask`, 256 half words.
constexpr int kOrderKeys = 16;
__device__ __forceinline__ void order_channel(const uint8_t* __restrict__ pid, int Cout, int Cin, int P, int ci,
                                              uint32_t* __restrict__ perm, uint32_t* __restrict__ bucket_off,
                                              uint32_t* fill, uint16_t* smask, int lane, const uint16_t* __restrict__ masks,
                                              unsigned long long* __restrict__ issue, int cb_log2) {
    // The ids of a channel lie Cin bytes apart: every load is a line of its own.  Up to kOrderKeys loads per lane (512
    // filters) are put in flight together; more filters take further rounds.
    unsigned keys[kOrderKeys];
    const bool kept = Cout <= 32 * kOrderKeys;   // one round: the second pass uses the same registers
    auto fetch = [&](int base0) {
#pragma unroll
        for (int r = 0; r < kOrderKeys; ++r) {
            const int co = base0 + 32 * r + lane;
            keys[r] = co < Cout ? pid[(size_t)co * Cin + ci] : 0xFFFFu;
            if (keys[r] >= (unsigned)P) keys[r] = 0xFFFFu;   // an id outside the table is not placed (nothing is written for it)
        }
    };
    if (kept) fetch(0);
    for (int p = lane; p < 256; p += 32) {
        fill[p] = 0;
        if (issue) smask[p] = p < P ? masks[p] : (uint16_t)0;
    }
    __syncwarp();
    // pass 1: histogram
    unsigned used = 0;   // taps kept by any filter of the current tile of 128
    const int cb_mask = (1 << cb_log2) - 1, ncb = (Cin + cb_mask) >> cb_log2;
    for (int base0 = 0; base0 < Cout; base0 += 32 * kOrderKeys) {
        if (!kept) fetch(base0);
#pragma unroll
        for (int r = 0; r < kOrderKeys; ++r) {
            const int base = base0 + 32 * r;
            if (base >= Cout) break;
            const unsigned key = keys[r];
            const unsigned peers = __match_any_sync(0xFFFFFFFFu, key);
            if (key != 0xFFFFu && lane == __ffs(peers) - 1) fill[key] += __popc(peers);
            if (issue) {
                used |= __reduce_or_sync(0xFFFFFFFFu, key != 0xFFFFu ? (unsigned)smask[key] : 0u);
                if (((base + 32) & 127) == 0 || base + 32 >= Cout) {
                    if (lane == 0 && used) {
                        unsigned long long bits = 0;
#pragma unroll
                        for (int t = 0; t < 9; ++t)
                            if (used & (1u << t)) bits |= 1ull << (4 * t + ((ci & cb_mask) >> (cb_log2 - 2)));
                        atomicOr(issue + (size_t)(base >> 7) * ncb + (ci >> cb_log2), bits);
                    }
                    used = 0;
                }
            }
            __syncwarp();
        }
    }
    // exclusive scan over the P buckets (P <= 255: eight per lane, then a warp scan of lane totals)
    uint32_t local[8];
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int p = lane * 8 + j;
        local[j] = sum;
        sum += (p < P) ? fill[p] : 0;
    }
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += o;
    }
    const uint32_t excl = incl - sum;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int p = lane * 8 + j;
        if (p < P) {
            fill[p] = excl + local[j];
            bucket_off[(size_t)ci * (P + 1) + p] = excl + local[j];
        }
    }
    if (lane == 0) bucket_off[(size_t)ci * (P + 1) + P] = (uint32_t)Cout;
    __syncwarp();
    // pass 2: placement, filters in ascending order inside each bucket
    for (int base0 = 0; base0 < Cout; base0 += 32 * kOrderKeys) {
        if (!kept) fetch(base0);
#pragma unroll
        for (int r = 0; r < kOrderKeys; ++r) {
            const int co = base0 + 32 * r + lane;
            if (base0 + 32 * r >= Cout) break;
            const unsigned key = keys[r];
            const unsigned peers = __match_any_sync(0xFFFFFFFFu, key);
            const unsigned before = peers & ((1u << lane) - 1u);
            if (key != 0xFFFFu) perm[(size_t)ci * Cout + fill[key] + __popc(before)] = (uint32_t)co;
            __syncwarp();
            if (key != 0xFFFFu && before == 0) fill[key] += __popc(peers);
            __syncwarp();
        }
    }
}

// The same for layers of at most 512 filters and 36 patterns (every layer of the two detectors but the widest, the preset
// tables of up to four taps), sixteen neighbouring channels to a block of 256 threads.  A thread is (segment of up to 32
// filters, channel): it counts its segment's patterns one filter after the other into a column of its own, a scan over segments and
// patterns turns counts into first positions, a second walk places the filters in shared memory, and the lists leave in
// whole lines.  Sixteen channels ride along in every instruction, where the form above spends 75 instructions on every
// 32 filters of every channel (33 us for the 7 000 channels of the larger detector; both its id loads, a line per filter,
// and its instructions were in the way; 15 us now).
constexpr int kFewFilters = 512, kFewPatterns = 36, kOrderThreads = 256;
constexpr int kOrderChannels = 16, kOrderSegs = kOrderThreads / kOrderChannels, kIdPitch = kOrderChannels + 4;
static_assert(kOrderSegs * 32 == kFewFilters, "a segment is at most 32 filters");
struct OrderFew {
    uint8_t ids[kFewFilters * kIdPitch];
    uint16_t cnt[kOrderSegs][kFewPatterns][kOrderChannels];
    uint16_t start[kFewPatterns + 1][kOrderChannels];
    uint16_t list[kOrderChannels][kFewFilters + 2];
    uint16_t masks[kFewPatterns];
};
// Which form: kernels = how many the launch orders in all.  Barriers and walks of the form of sixteens take 7 us however little
// there is to sort (ordering kernel alone; a warp for each channel 4.5 us at 64 filters, 18 at 600): it is for layers of more
// than 128 filters and for launches whose instructions count.  Whole pass, sixteens / warps: 50 layers of 16x32 (25 600 kernels) 8.8 / 7.3 us,
// 5 of 40x300 (60 000) 10.3 / 9.4, 20 of 64x64 (81 920) 8.9 / 9.0, 12 of 100x200 (240 000) 11.5 / 15.3.  Layers that fit neither limit: a warp each
// (600x64: 28.7 us with two channels to each of eight warps of a block, 14.6 with one to each of four).
constexpr int kManyKernels = 80000;
inline __host__ __device__ bool order_in_sixteens(int Cout, int P, long long kernels) {
    return Cout <= kFewFilters && P <= kFewPatterns && (Cout > 128 || kernels > kManyKernels);
}
// Channels to a block: sixteen, or one to each of four warps.
constexpr int kOrderWarps = 4;
inline __host__ __device__ int order_channels_of(bool sixteens) { return sixteens ? kOrderChannels : kOrderWarps; }

// All threads of the block; `masks` as the device sees the table (global or shared).
__device__ __forceinline__ void order_channels_few(const uint8_t* __restrict__ pid, int Cout, int Cin, int P, int ci0,
                                                   uint32_t* __restrict__ perm, uint32_t* __restrict__ bucket_off, OrderFew& sh,
                                                   const uint16_t* __restrict__ masks, unsigned long long* __restrict__ issue, int cb_log2) {
    const int tid = (int)threadIdx.x;
    if (tid < P) sh.masks[tid] = masks[tid];
    if ((Cin & 15) == 0) {
        // rows of sixteen ids, one load each; all of a thread's loads in flight together
        uint4 v[kFewFilters / kOrderThreads];
#pragma unroll
        for (int q = 0; q < kFewFilters / kOrderThreads; ++q) {
            const int co = tid + q * kOrderThreads;
            if (co < Cout) v[q] = __ldcg(reinterpret_cast<const uint4*>(pid + (size_t)co * Cin + ci0));
        }
#pragma unroll
        for (int q = 0; q < kFewFilters / kOrderThreads; ++q) {
            const int co = tid + q * kOrderThreads;
            unsigned* to = reinterpret_cast<unsigned*>(sh.ids + co * kIdPitch);
            if (co < Cout) to[0] = v[q].x, to[1] = v[q].y, to[2] = v[q].z, to[3] = v[q].w;
        }
    } else if ((Cin & 3) == 0) {
        // aligned words of four ids, eight of a thread's loads in flight (88 channels, 400 filters, byte by byte: 8 000 cycles)
        constexpr int kQ = 8;
        for (int i0 = tid; i0 < Cout * (kOrderChannels / 4); i0 += kQ * kOrderThreads) {
            unsigned v[kQ];
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                const int i = i0 + q * kOrderThreads, co = i >> 2, c = (i & 3) * 4;
                v[q] = ~0u;
                if (co < Cout && ci0 + c < Cin) v[q] = __ldcg(reinterpret_cast<const unsigned*>(pid + (size_t)co * Cin + ci0 + c));
            }
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                const int i = i0 + q * kOrderThreads, co = i >> 2;
                if (co < Cout) *reinterpret_cast<unsigned*>(sh.ids + co * kIdPitch + (i & 3) * 4) = v[q];
            }
        }
    } else {
        constexpr int kQ = 8;
        for (int i0 = tid; i0 < Cout * kOrderChannels; i0 += kQ * kOrderThreads) {
            uint8_t v[kQ];
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                const int i = i0 + q * kOrderThreads, co = i / kOrderChannels, c = i % kOrderChannels;
                v[q] = co < Cout && ci0 + c < Cin ? __ldcg(pid + (size_t)co * Cin + ci0 + c) : (uint8_t)255;
            }
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                const int i = i0 + q * kOrderThreads, co = i / kOrderChannels;
                if (co < Cout) sh.ids[co * kIdPitch + i % kOrderChannels] = v[q];
            }
        }
    }
    // Filters of a segment: as few as the sixteen segments allow, a power of two so that none crosses a tile of 128.  (Always
    // 32: 3 000 cycles per walk for layers of 64 filters, of which two threads in sixteen did the work; 900 and 2 100 now.)
    int seg = 32;
    while (seg > 1 && (seg / 2) * kOrderSegs >= Cout) seg >>= 1;
    const int c = tid % kOrderChannels, s = tid / kOrderChannels, co0 = min(seg * s, Cout), co1 = min(co0 + seg, Cout);
    const bool real = ci0 + c < Cin;
    for (int p = 0; p < P; ++p) sh.cnt[s][p][c] = 0;
    __syncthreads();
    unsigned used = 0;   // taps kept by any filter of the segment
    constexpr int kWalk = 8;   // ids read ahead of the counts, which the compiler takes for the same memory
    for (int f0 = co0; f0 < co1; f0 += kWalk) {
        unsigned id[kWalk];
#pragma unroll
        for (int j = 0; j < kWalk; ++j) id[j] = sh.ids[min(f0 + j, co1 - 1) * kIdPitch + c];
#pragma unroll
        for (int j = 0; j < kWalk; ++j) {
            if (f0 + j < co1 && id[j] < (unsigned)P) {   // (an id outside the table is not placed)
                used |= sh.masks[id[j]];
                sh.cnt[s][id[j]][c] = (uint16_t)(sh.cnt[s][id[j]][c] + 1);
            }
        }
    }
    if (issue) {
        // a slab is a quarter of a block of 2^cb_log2 channels: sixteen or eight neighbouring ones
        if (!real) used = 0;
        used |= __shfl_xor_sync(0xFFFFFFFFu, used, 1);
        used |= __shfl_xor_sync(0xFFFFFFFFu, used, 2);
        used |= __shfl_xor_sync(0xFFFFFFFFu, used, 4);
        if (cb_log2 == 6) used |= __shfl_xor_sync(0xFFFFFFFFu, used, 8);
        const int slab_mask = (1 << (cb_log2 - 2)) - 1;
        if ((c & slab_mask) == 0 && used) {
            const int ci = ci0 + c, ncb = (Cin + (1 << cb_log2) - 1) >> cb_log2;
            unsigned long long bits = 0;
#pragma unroll
            for (int t = 0; t < 9; ++t)
                if (used & (1u << t)) bits |= 1ull << (4 * t + ((ci & ((1 << cb_log2) - 1)) >> (cb_log2 - 2)));
            atomicOr(issue + (size_t)(co0 >> 7) * ncb + (ci >> cb_log2), bits);
        }
    }
    __syncthreads();
    // counts -> exclusive prefix over the segments; totals per pattern
    for (int i = tid; i < P * kOrderChannels; i += kOrderThreads) {
        const int p = i / kOrderChannels, ch = i % kOrderChannels;
        unsigned sum = 0;
#pragma unroll
        for (int g = 0; g < kOrderSegs; ++g) {
            const unsigned n = sh.cnt[g][p][ch];
            sh.cnt[g][p][ch] = (uint16_t)sum;
            sum += n;
        }
        sh.start[p][ch] = (uint16_t)sum;
    }
    __syncthreads();
    if (tid < kOrderChannels) {
        unsigned sum = 0;
        for (int p = 0; p < P; ++p) {
            const unsigned n = sh.start[p][tid];
            sh.start[p][tid] = (uint16_t)sum;
            sum += n;
        }
        sh.start[P][tid] = (uint16_t)sum;   // filters placed (fewer than Cout only where ids lie outside the table)
    }
    __syncthreads();
    for (int f0 = co0; f0 < co1; f0 += kWalk) {
        unsigned id[kWalk], at[kWalk];
#pragma unroll
        for (int j = 0; j < kWalk; ++j) id[j] = sh.ids[min(f0 + j, co1 - 1) * kIdPitch + c];
#pragma unroll
        for (int j = 0; j < kWalk; ++j) at[j] = id[j] < (unsigned)P ? sh.start[id[j]][c] : 0u;
#pragma unroll
        for (int j = 0; j < kWalk; ++j) {
            if (f0 + j < co1 && id[j] < (unsigned)P) {
                const unsigned n = sh.cnt[s][id[j]][c];
                sh.cnt[s][id[j]][c] = (uint16_t)(n + 1);
                sh.list[c][at[j] + n] = (uint16_t)(f0 + j);
            }
        }
    }
    const int off_n = P + 1;
    for (int i = tid; i < off_n * kOrderChannels; i += kOrderThreads) {
        const int ch = i / off_n, p = i - ch * off_n;
        if (ci0 + ch < Cin) bucket_off[(size_t)(ci0 + ch) * off_n + p] = p == P ? (uint32_t)Cout : sh.start[p][ch];
    }
    __syncthreads();
    const int warp = tid >> 5, lane = tid & 31;
    for (int ch = warp; ch < kOrderChannels && ci0 + ch < Cin; ch += kOrderThreads / 32) {
        const int n = sh.start[P][ch];
        uint32_t* to = perm + (size_t)(ci0 + ch) * Cout;
        for (int i = lane; i < n; i += 32) to[i] = sh.list[ch][i];
    }
}

}  // namespace rtoss_dev

#endif
