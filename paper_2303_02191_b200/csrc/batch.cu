// Whole-model pruning pass: pattern selection (Algorithm 2; Algorithm 3 for 1x1 layers) and packing of EVERY layer
// of a model in two launches instead of three per layer.  The per-kernel arithmetic is the one of the single-layer
// calls (select_core.cuh), so the results are the same bits.
//
//   batch_select_pack_kernel : two kernels / runs of nine per thread, 512 or 128 per block step; a block step ("chunk")
//                              belongs to one layer and is described by a table built at plan time.
//                              Writes the pattern id (caller's array and the handle's), the k kept values and the
//                              tensor path's dense-expanded weights.
//   batch_order_kernel       : per (3x3 layer, input channel) the stable order of filters by pattern id, sixteen
//                              channels to a block or one to a warp, through a task -> layer table.
//
// A layer that inherits its parent's patterns (Section IV.A: children of a group share the parent's kernel
// patterns) evaluates the selection on the PARENT's weights and packs its own with the result; it reads no other
// layer's output, so all layers run in the same launch.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "conv_common.cuh"
#include "rtoss_internal.h"
#include "select_core.cuh"

namespace {

// Threads of a block, kPair kernels to a thread; a block step ("chunk") is that many kernels.  Models of at most two blocks of
// 256 threads an SM are cut into blocks of 64: more SMs take part in the stores, and registers are left for four patterns in
// flight.  Whole pass, blocks of 256 / of 64: 32x16 3x3 in fp32 13.2 / 7.8 us, 64x64 3x3 with 49 patterns 12.9 / 8.8, 512x256 1x1
// 4.2 / 3.4, 256x256 3x3 with 49 patterns 16.5 / 14.3, 20 layers of 64x64 in fp32 (160 blocks of 256) 11.6 / 10.2.
constexpr int kBatchThreads = 256, kSmallThreads = 64;
__host__ __device__ constexpr int chunk_of(int threads) { return threads * rtoss_dev::kPair; }

struct alignas(16) BatchLayer {
    const void* w;      // weights to pack
    const void* w_sel;  // weights the selection reads: w, or the group parent's
    int pid_out_vec;    // the caller's id array takes 2-byte stores
    uint8_t* pid_out;   // caller's id array (nullable)
    uint8_t* pid;       // the handle's arrays
    void* val;
    void* wtc;
    uint32_t* perm;
    uint32_t* bucket_off;
    unsigned long long* issue;  // the handle's issue words (tensor path, 3x3), or null
    int issue_n;
    long long n_kernels;
    rtoss_wtc_layout lay;  // layout of wtc
    int Cout, Cin, ksize, P, k;
    unsigned k_magic;   // ceil(2^16 / k): o / k = o * k_magic >> 16 for o below 2^13
    int w_dtype, sel_dtype, v_dtype;
    unsigned chunk0;  // first chunk of this layer
    unsigned task0;   // first ordering task (3x3 layers)
    int sixteens;     // how its channels are ordered (order_in_sixteens)
    uint16_t masks[256];
};

// A block step: where its weights (those the selection reads) lie, how many bytes, whose they are.
struct BatchChunk {
    const unsigned char* src;
    unsigned bytes, layer;
};

// 9*count weights of `count` consecutive kernels starting at kernel `first`, as raw bytes, coalesced; 16 bytes per
// thread where the chunk is whole (a whole chunk is a multiple of 16 bytes and the base is 16-byte aligned).
template <int T>
__device__ __forceinline__ void stage_raw(const void* w, long long first, int count, int esize, unsigned char* smem) {
    const unsigned char* src = reinterpret_cast<const unsigned char*>(w) + (size_t)first * 9 * esize;
    const int bytes = count * 9 * esize;
    if (count == chunk_of(T)) {
        const uint4* s4 = reinterpret_cast<const uint4*>(src);
        uint4* d4 = reinterpret_cast<uint4*>(smem);
        for (int i = threadIdx.x; i < bytes / 16; i += T) d4[i] = __ldg(s4 + i);
    } else if (esize == 4) {
        const uint32_t* s1 = reinterpret_cast<const uint32_t*>(src);
        uint32_t* d1 = reinterpret_cast<uint32_t*>(smem);
        for (int i = threadIdx.x; i < bytes / 4; i += T) d1[i] = s1[i];
    } else {
        const uint16_t* s1 = reinterpret_cast<const uint16_t*>(src);
        uint16_t* d1 = reinterpret_cast<uint16_t*>(smem);
        for (int i = threadIdx.x; i < bytes / 2; i += T) d1[i] = s1[i];
    }
}

__device__ __forceinline__ void cp_async16(void* smem, const void* g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(g) : "memory");
}

// Starts fetching a chunk: the layer's record (unless it is there already) and the weights its selection reads.  A ragged chunk's last bytes are plain
// loads (16-bit weights: 2-byte pieces).
template <int T>
__device__ __forceinline__ void fetch_chunk(const BatchLayer* layers, const BatchChunk& c, BatchLayer* s_layer, unsigned char* raw) {
    const unsigned char* rec = reinterpret_cast<const unsigned char*>(layers + c.layer);
    if (s_layer)
        for (int o = (int)threadIdx.x * 16; o < (int)sizeof(BatchLayer); o += T * 16) 
            cp_async16(reinterpret_cast<unsigned char*>(s_layer) + o, rec + o);
    const int whole = (int)(c.bytes & ~15u);
    for (int o = (int)threadIdx.x * 16; o < whole; o += T * 16) cp_async16(raw + o, c.src + o);
    const int o = whole + (int)threadIdx.x * 2;
    if (o < (int)c.bytes) *reinterpret_cast<uint16_t*>(raw + o) = *reinterpret_cast<const uint16_t*>(c.src + o);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// ---- one chunk ----------------------------------------------------------------------------------------------------
// The chunk's weights lie in shared memory as they are in memory.  Phase 1: a thread selects for two neighbouring kernels
// and leaves their pattern ids and masks in shared memory.  Phase 2: the outputs are written the way memory wants them,
// whatever kernel an element belongs to: kept values and the flat 1x1 expansion as consecutive words, the 3x3 expansion tap
// by tap (consecutive kernels are consecutive channels).  Nothing per kernel is held in registers between the phases.

template <typename T> __device__ __forceinline__ float raw_at(const unsigned char* raw, int e) {
    if constexpr (sizeof(T) == 4) return reinterpret_cast<const float*>(raw)[e];
    else return rtoss_dev::to_f32<T>(reinterpret_cast<const T*>(raw)[e]);
}

template <int kUnroll, typename T>
__device__ __forceinline__ void select_chunk(const BatchLayer& L, long long first, int count, const unsigned char* raw, const rtoss_dev::PatternFactors* factors,
                                             uint8_t* s_pid, uint16_t* s_mask) {
    using namespace rtoss_dev;
    const int base = (int)threadIdx.x * kPair;
    if (base >= count) return;
    f32x2 q[9];
    int best[kPair];
    load_pair<T>(raw, (int)threadIdx.x, q);
    select_best2<kUnroll>(q, L.masks, factors, L.P, best);
    const long long i = first + base;
    const unsigned ids = (unsigned)best[0] | (unsigned)best[1] << 8;
    *reinterpret_cast<uint16_t*>(s_pid + base) = (uint16_t)ids;
    *reinterpret_cast<unsigned*>(s_mask + base) = (unsigned)L.masks[best[0]] | (unsigned)L.masks[best[1]] << 16;
    if (base + 1 < count) {
        *reinterpret_cast<uint16_t*>(L.pid + i) = (uint16_t)ids;
        if (L.pid_out && L.pid_out_vec) {
            *reinterpret_cast<uint16_t*>(L.pid_out + i) = (uint16_t)ids;
        } else if (L.pid_out) {
            L.pid_out[i] = (uint8_t)best[0];
            L.pid_out[i + 1] = (uint8_t)best[1];
        }
    } else {
        L.pid[i] = (uint8_t)best[0];
        if (L.pid_out) L.pid_out[i] = (uint8_t)best[0];
    }
}

template <typename V> __device__ __forceinline__ unsigned round2(float a, float b) {
    if constexpr (std::is_same<V, __half>::value) {
        const __half2 u = __floats2half2_rn(a, b);
        return *reinterpret_cast<const unsigned*>(&u);
    } else {
        const __nv_bfloat162 u = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<const unsigned*>(&u);
    }
}
// Two neighbouring positions as one aligned word; fp32: tf32 heads, and at lo what corrects them (see expand_one).
template <typename V, bool kCorr16> __device__ __forceinline__ void put_pair(V* at, V* lo, float a, float b) {
    using namespace rtoss_dev;
    if constexpr (sizeof(V) == 2) {
        *reinterpret_cast<unsigned*>(at) = round2<V>(a, b);
    } else if constexpr (kCorr16) {
        const float ha = tf32_near(a), hb = tf32_near(b);
        *reinterpret_cast<float2*>(at) = make_float2(ha, hb);
        put_corr16_two(reinterpret_cast<uint16_t*>(lo), a, b, __fsub_rn(a, ha), __fsub_rn(b, hb));
    } else {
        *reinterpret_cast<float2*>(at) = make_float2(tf32_head(a), tf32_head(b));
        *reinterpret_cast<float2*>(lo) = make_float2(__fsub_rn(a, tf32_head(a)), __fsub_rn(b, tf32_head(b)));
    }
}
template <typename V> __device__ __forceinline__ void put_one(V* at, V* lo, bool corr16, float a) {
    using namespace rtoss_dev;
    if constexpr (sizeof(V) == 2) {
        *at = narrow_to<V>(a);
    } else if (corr16) {
        const float h = tf32_near(a);
        *at = h;
        put_corr16_one(reinterpret_cast<uint16_t*>(lo), a, __fsub_rn(a, h));
    } else {
        *at = tf32_head(a);
        *lo = __fsub_rn(a, tf32_head(a));
    }
}

template <int kThreads, typename T, typename V>
__device__ __forceinline__ void pack_chunk(const BatchLayer& L, long long first, int count, const unsigned char* raw, const uint8_t* s_pid,
                                           const uint16_t* s_mask, const unsigned long long* s_taps) {
    using namespace rtoss_dev;
    V* val = reinterpret_cast<V*>(L.val) + first * L.k;   // (a chunk's first value is at a multiple of 512 k)
    if (sizeof(V) == 2 && L.k == 4) {
        // the usual case: a kernel's four values are one aligned 8-byte word
        for (int g = (int)threadIdx.x; g < count; g += kThreads) {
            const unsigned taps = (unsigned)s_taps[s_pid[g]];
            const unsigned char* w = raw + (size_t)g * 9 * sizeof(T);
            uint2 u;
            u.x = round2<V>(raw_at<T>(w, taps & 15), raw_at<T>(w, (taps >> 4) & 15));
            u.y = round2<V>(raw_at<T>(w, (taps >> 8) & 15), raw_at<T>(w, (taps >> 12) & 15));
            *reinterpret_cast<uint2*>(val + 4 * g) = u;
        }
    } else {
        // value o of the chunk is the (o mod k)-th kept tap of kernel o / k; two to a thread
        const int n = count * L.k, k = L.k;
        auto value = [&](int o) {
            const int g = (int)(((unsigned)o * L.k_magic) >> 16);   // o / k
            const int tap = (int)(s_taps[s_pid[g]] >> (4 * (o - g * k))) & 15;
            return raw_at<T>(raw, g * 9 + tap);
        };
        for (int o = 2 * (int)threadIdx.x; o < n; o += 2 * kThreads) {
            const float a = value(o);
            if (o + 1 < n) {
                const float b = value(o + 1);
                if constexpr (sizeof(V) == 4) *reinterpret_cast<float2*>(val + o) = make_float2(a, b);
                else *reinterpret_cast<unsigned*>(val + o) = round2<V>(a, b);
            } else {
                val[o] = narrow_to<V>(a);
            }
        }
    }
    if (!L.wtc) return;
    V* wtc = reinterpret_cast<V*>(L.wtc);
    const int Cin = L.Cin, cin_p = L.lay.cin_p;
    const int64_t tap_step = (int64_t)L.lay.rows * cin_p;
    if (L.ksize == 3) {
        const int64_t lo_at = 9 * tap_step, copy_step = (int64_t)L.lay.rep_rows * cin_p;
        const int base = (int)threadIdx.x * kPair;
        if (base >= count) return;
        const unsigned mm = *reinterpret_cast<const unsigned*>(s_mask + base);
        const bool two = base + 1 < count;
        // kernel i lies at flat position i of a tap's matrix; where the stored rows are longer than the layer's, further on
        int64_t p0 = first + base, p1 = p0 + 1;
        if (cin_p != Cin) {
            p0 += (int64_t)((unsigned)p0 / (unsigned)Cin) * (cin_p - Cin);
            p1 += (int64_t)((unsigned)p1 / (unsigned)Cin) * (cin_p - Cin);
        }
        const bool word = two && p1 == p0 + 1 && (p0 & 1) == 0 && (tap_step & 1) == 0 && (copy_step & 1) == 0;
        V* at = wtc + p0;
        const int64_t d1 = p1 - p0;
        // fp32: where what corrects position p lies; a tap or a copy further down is as far as in the first array (with bf16
        // corrections both steps are whole blocks of 32 channels)
        const bool corr16 = sizeof(V) == 4 && rtoss_f32_corr16(Cin, 3);
        auto lo_of = [&](int64_t p) -> V* {
            if constexpr (sizeof(V) == 4) return corr16 ? reinterpret_cast<V*>(corr16_at(wtc + lo_at, p)) : wtc + lo_at + p;
            else return nullptr;
        };
        V* lo = lo_of(p0);
        if (word && L.lay.copies == 1) {
            if constexpr (sizeof(V) == 4) {
                if (corr16) {
                    const int64_t to_lo = lo - at;
#pragma unroll
                    for (int t = 0; t < 9; ++t, at += tap_step) {
                        const float a = (mm >> t) & 1u ? raw_at<T>(raw, base * 9 + t) : 0.f;
                        const float b = (mm >> (16 + t)) & 1u ? raw_at<T>(raw, base * 9 + 9 + t) : 0.f;
                        put_pair<V, true>(at, at + to_lo, a, b);
                    }
                    return;
                }
            }
#pragma unroll
            for (int t = 0; t < 9; ++t, at += tap_step) {
                const float a = (mm >> t) & 1u ? raw_at<T>(raw, base * 9 + t) : 0.f;
                const float b = (mm >> (16 + t)) & 1u ? raw_at<T>(raw, base * 9 + 9 + t) : 0.f;
                put_pair<V, false>(at, at + lo_at, a, b);
            }
            return;
        }
        // Narrow layers (repeated filters) and odd rows: the nine taps in registers, then copy by copy, nine independent
        // stores at a time.  (Tap by tap with the copies inside, a value was read, rounded and stored 36 times one after the
        // other: 9 600 cycles for 18 filters, of a launch that holds four blocks; 4 200 now.)
        if constexpr (sizeof(V) == 2) {
            unsigned u[9];
#pragma unroll
            for (int t = 0; t < 9; ++t)
                u[t] = round2<V>((mm >> t) & 1u ? raw_at<T>(raw, base * 9 + t) : 0.f, (mm >> (16 + t)) & 1u ? raw_at<T>(raw, base * 9 + 9 + t) : 0.f);
#pragma unroll 1
            for (int c = 0; c < L.lay.copies; ++c, at += copy_step) {
                V* to = at;
                if (word) {
#pragma unroll
                    for (int t = 0; t < 9; ++t, to += tap_step) *reinterpret_cast<unsigned*>(to) = u[t];
                } else {
#pragma unroll
                    for (int t = 0; t < 9; ++t, to += tap_step) {
                        *reinterpret_cast<uint16_t*>(to) = (uint16_t)u[t];
                        if (two) *reinterpret_cast<uint16_t*>(to + d1) = (uint16_t)(u[t] >> 16);
                    }
                }
            }
        } else {
            const int64_t to_lo = lo - at, to_lo1 = lo_of(p1) - at;
#pragma unroll 1
            for (int c = 0; c < L.lay.copies; ++c, at += copy_step) {
                V* to = at;
#pragma unroll 3
                for (int t = 0; t < 9; ++t, to += tap_step) {
                    const float a = (mm >> t) & 1u ? raw_at<T>(raw, base * 9 + t) : 0.f;
                    const float b = (mm >> (16 + t)) & 1u ? raw_at<T>(raw, base * 9 + 9 + t) : 0.f;
                    if (word && corr16) {
                        put_pair<V, true>(to, to + to_lo, a, b);
                    } else if (word) {
                        put_pair<V, false>(to, to + to_lo, a, b);
                    } else {
                        put_one<V>(to, to + to_lo, corr16, a);
                        if (two) put_one<V>(to + d1, to + to_lo1, corr16, b);
                    }
                }
            }
        }
    } else {
        // the flat matrix: four positions to a thread (a multiple of four: at most two kernels, one aligned word)
        const int n = count * 9;
        const bool words = cin_p == Cin && (tap_step & 3) == 0;   // (rows as long as the layer's; fp32 remainders aligned alike)
        for (int e = 4 * (int)threadIdx.x; e < n; e += 4 * kThreads) {
            const int g = (int)(((unsigned)e * 7282u) >> 16);   // e / 9 (e is below 2^13)
            const unsigned mm = ((unsigned)s_mask[g] | (unsigned)s_mask[min(g + 1, chunk_of(kThreads) - 1)] << 9) >> (e - 9 * g);   // bit j: position e + j is kept
            const int64_t f = first * 9 + e;
            float v[4];
            if constexpr (sizeof(T) == 4) {
                const float4 x = *reinterpret_cast<const float4*>(raw + (size_t)e * 4);
                v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
            } else {
                const uint2 x = *reinterpret_cast<const uint2*>(raw + (size_t)e * 2);
                const T* h = reinterpret_cast<const T*>(&x);
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = to_f32<T>(h[j]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = (mm >> j) & 1u ? v[j] : 0.f;
            if (words && e + 4 <= n) {
                if constexpr (sizeof(V) == 4) {
                    *reinterpret_cast<float4*>(wtc + f) = make_float4(tf32_head(v[0]), tf32_head(v[1]), tf32_head(v[2]), tf32_head(v[3]));
                    *reinterpret_cast<float4*>(wtc + f + tap_step) =
                        make_float4(__fsub_rn(v[0], tf32_head(v[0])), __fsub_rn(v[1], tf32_head(v[1])), __fsub_rn(v[2], tf32_head(v[2])), __fsub_rn(v[3], tf32_head(v[3])));
                } else {
                    *reinterpret_cast<uint2*>(wtc + f) = make_uint2(round2<V>(v[0], v[1]), round2<V>(v[2], v[3]));
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (e + j < n) {
                        V* at = wtc + f + j + (cin_p != Cin ? (int64_t)((unsigned)(f + j) / (unsigned)Cin) * (cin_p - Cin) : 0);
                        put_one<V>(at, at + tap_step, false, v[j]);
                    }
            }
        }
    }
}

// Bound by instructions (0.75 a cycle and scheduler; 35 % of the copy rate).  fp32 handles with bf16 corrections have a loop of
// their own over the taps, which keeps two addresses: with the choice and the second address made per tap the kernel of 40
// registers spilled, and 32 M bf16 weights took 107 us instead of 89 (7 M fp32 ones 41 instead of 33).  32 M weights, 8 patterns of four taps: 131 us
// with one kernel per thread that held its weights in registers through all outputs, 65 us in this form; 20 us instead of
// 31 for 7 M.  (Prefetching the next chunk with a second buffer cost occupancy and was slower: 142 us on the older form.)
template <int T>
__global__ void __launch_bounds__(T, T == kBatchThreads ? 6 : 8) batch_select_pack_kernel(const BatchLayer* __restrict__ layers,
                                                                          const BatchChunk* __restrict__ chunks,
                                                                          unsigned n_chunks, int order_follows) {
    // The ordering kernel behind this one waits for the end of this grid and does not let its own successors start before
    // its end, so it may be set up meanwhile; no other kernel may be (a reader of handles does not wait).
    if (order_follows) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    rtoss_dev::pdl_enter_handle_writer();
    constexpr int kStep = chunk_of(T), kUnroll = T == kBatchThreads ? 2 : 4;   // (patterns in flight: few warps have only themselves to overlap)
    __shared__ __align__(16) unsigned char raw[kStep * 9 * 4];
    __shared__ BatchLayer s_layer;
    __shared__ __align__(16) uint16_t s_mask[kStep];
    __shared__ __align__(16) uint8_t s_pid[kStep];
    __shared__ rtoss_dev::PatternFactors s_factors[rtoss_dev::kFactorPatterns];
    __shared__ unsigned long long s_taps[256];   // a pattern's taps in ascending order, four bits each
    const unsigned per = n_chunks / gridDim.x, extra = n_chunks % gridDim.x;
    const unsigned begin = blockIdx.x * per + min(blockIdx.x, extra), end = begin + per + (blockIdx.x < extra ? 1u : 0u);
    if (begin >= end) return;
    BatchChunk c = chunks[begin];
    uint32_t have = 0xFFFFFFFFu;   // which layer s_layer is
    for (unsigned chunk = begin; chunk < end; ++chunk) {
        const bool fresh = c.layer != have;
        fetch_chunk<T>(layers, c, fresh ? &s_layer : nullptr, raw);
        have = c.layer;
        c = chunks[min(chunk + 1, end - 1)];
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const BatchLayer& L = s_layer;
        const long long first = (long long)(chunk - L.chunk0) * kStep;
        const int count = (int)(L.n_kernels - first < kStep ? L.n_kernels - first : kStep);
        // the layer's first chunk clears its issue words: the ordering kernel (next launch) ORs the bits in
        if (chunk == L.chunk0 && L.issue)
            for (int i = threadIdx.x; i < L.issue_n; i += T) L.issue[i] = 0ull;
#pragma unroll 1
        for (int p0 = 0; p0 < 256; p0 += T) {
            const int p = p0 + (int)threadIdx.x;
            if (!fresh || p >= L.P) break;
            const unsigned m = L.masks[p];
            unsigned long long taps = 0;
            int j = 0;
#pragma unroll
            for (int t = 0; t < 9; ++t)
                if (m & (1u << t)) taps |= (unsigned long long)t << (4 * j++);
            s_taps[p] = taps;
            if (p < rtoss_dev::kFactorPatterns) {
#pragma unroll
                for (int t = 0; t < 10; ++t) {
                    const float f = (m >> t) & 1u ? 1.f : 0.f;   // (bit 9 is never set)
                    s_factors[p].f[t] = rtoss_dev::pack_f32x2(f, f);
                }
            }
        }
        if (fresh) __syncthreads();
        if (L.sel_dtype == RTOSS_F32) select_chunk<kUnroll, float>(L, first, count, raw, s_factors, s_pid, s_mask);
        else if (L.sel_dtype == RTOSS_BF16) select_chunk<kUnroll, __nv_bfloat16>(L, first, count, raw, s_factors, s_pid, s_mask);
        else select_chunk<kUnroll, __half>(L, first, count, raw, s_factors, s_pid, s_mask);
        __syncthreads();
        if (L.w_sel != L.w) {   // the patterns are inherited: this layer's own weights take the buffer
            stage_raw<T>(L.w, first, count, L.w_dtype == RTOSS_F32 ? 4 : 2, raw);
            __syncthreads();
        }
#define RTOSS_PACK(T_, V_) pack_chunk<T, T_, V_>(L, first, count, raw, s_pid, s_mask, s_taps)
#define RTOSS_PACK_TO(V_)                                       \
    if (L.w_dtype == RTOSS_F32) RTOSS_PACK(float, V_);          \
    else if (L.w_dtype == RTOSS_BF16) RTOSS_PACK(__nv_bfloat16, V_); \
    else RTOSS_PACK(__half, V_)
        if (L.v_dtype == RTOSS_F32) { RTOSS_PACK_TO(float); }
        else if (L.v_dtype == RTOSS_BF16) { RTOSS_PACK_TO(__nv_bfloat16); }
        else { RTOSS_PACK_TO(__half); }
#undef RTOSS_PACK_TO
#undef RTOSS_PACK
        __syncthreads();   // the buffer and the record are free
    }
    rtoss_dev::handle_writer_done();
}

// kSixteens: some layer is ordered sixteen channels to a block; else all go a channel to a warp, in blocks half the size.
template <bool kSixteens>
__global__ void __launch_bounds__(kSixteens ? rtoss_dev::kOrderThreads : rtoss_dev::kOrderWarps * 32, kSixteens ? 4 : 1)
    batch_order_kernel(const BatchLayer* __restrict__ layers, const uint32_t* __restrict__ task_layer, unsigned n_tasks) {
    using namespace rtoss_dev;
    struct Many {
        uint32_t fill[kOrderWarps][256];
        uint16_t mask[kOrderWarps][256];
    };
    union Shared {
        Many many;
        typename std::conditional<kSixteens, OrderFew, Many>::type few;
    };
    __shared__ Shared sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the first task's record is the plan's, which no kernel writes: it comes in ahead of the wait for the pattern ids
    uint32_t layer = blockIdx.x < n_tasks ? __ldcg(task_layer + blockIdx.x) : 0u;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(layers + layer));
    pdl_enter_handle_writer();
    for (unsigned task = blockIdx.x; task < n_tasks; task += gridDim.x) {
        if (task != blockIdx.x) layer = task_layer[task];
        const BatchLayer& L = layers[layer];
        const int ci0 = (int)(task - L.task0) * order_channels_of(L.sixteens != 0), cb_log2 = L.v_dtype == RTOSS_F32 ? 5 : 6;
        if (kSixteens && L.sixteens) {
            if constexpr (kSixteens) order_channels_few(L.pid, L.Cout, L.Cin, L.P, ci0, L.perm, L.bucket_off, sh.few, L.masks, L.issue, cb_log2);
        } else if (warp < kOrderWarps && ci0 + warp < L.Cin) {
            order_channel(L.pid, L.Cout, L.Cin, L.P, ci0 + warp, L.perm, L.bucket_off, sh.many.fill[warp], sh.many.mask[warp], lane, L.masks, L.issue, cb_log2);
        }
        __syncthreads();   // the shared arrays are free
    }
    handle_writer_done();
}

void set_err(rtoss_ctx* ctx, const char* what) {
    if (!ctx) return;
    snprintf(ctx->err, sizeof(ctx->err), "batch: %s", what);
}

}  // namespace

struct rtoss_batch {
    int device;
    int L;
    BatchLayer* layers_dev;
    BatchChunk* chunks_dev;
    uint32_t* task_layer_dev;
    unsigned n_chunks, n_tasks;
    int threads;     // of a block of the first kernel
    bool sixteens;   // some layer's channels are ordered sixteen to a block
};

extern "C" {

rtoss_status rtoss_batch_create(rtoss_ctx* ctx, const rtoss_batch_item* items, int L, rtoss_batch** out) {
    if (!ctx) return RTOSS_ERR_INVALID_ARG;
    if (!items || L < 1 || !out) {
        set_err(ctx, "null argument or no layers");
        return RTOSS_ERR_INVALID_ARG;
    }
    *out = nullptr;
    std::vector<BatchLayer> layers((size_t)L);
    std::vector<BatchChunk> chunks;
    std::vector<uint32_t> task_layer;
    long long kernels = 0, steps = 0;   // 3x3 kernels, which the ordering kernel sees; block steps of the first kernel, in large ones
    bool sixteens = false;
    for (int i = 0; i < L; ++i) {
        const long long n = (long long)items[i].Cout * items[i].Cin / (items[i].ksize == 3 ? 1 : 9);   // (checked below)
        kernels += items[i].ksize == 3 ? n : 0;
        steps += (n + chunk_of(kBatchThreads) - 1) / chunk_of(kBatchThreads);
    }
    const int threads = steps <= 2 * ctx->sm_count ? kSmallThreads : kBatchThreads;
    const long long chunk = chunk_of(threads);
    for (int i = 0; i < L; ++i) {
        const rtoss_batch_item& it = items[i];
        rtoss_packed* p = it.packed;
        if (!it.w_dev || !p || !it.masks_host || (int)it.w_dtype < 0 || (int)it.w_dtype > 2) {
            set_err(ctx, "item with a null pointer or bad dtype");
            return RTOSS_ERR_INVALID_ARG;
        }
        if (p->device != ctx->device || p->Cout != it.Cout || p->Cin != it.Cin || p->ksize != it.ksize || p->P != it.P ||
            p->k != it.k) {
            set_err(ctx, "item's packed handle describes another layer, table size or device");
            return RTOSS_ERR_INVALID_ARG;
        }
        if (!rtoss_table_ok(it.masks_host, it.P, it.k)) {
            set_err(ctx, "pattern table invalid");
            return RTOSS_ERR_BAD_PATTERN_TABLE;
        }
        if (reinterpret_cast<uintptr_t>(it.w_dev) & 15) {
            set_err(ctx, "weights must be 16-byte aligned");
            return RTOSS_ERR_ALIGNMENT;
        }
        for (int j = 0; j < i; ++j)
            if (items[j].packed == p) {
                set_err(ctx, "two items share one packed handle");
                return RTOSS_ERR_INVALID_ARG;
            }
        BatchLayer& B = layers[(size_t)i];
        memset(&B, 0, sizeof(B));
        B.w = it.w_dev;
        B.w_sel = it.w_dev;
        B.sel_dtype = B.w_dtype = (int)it.w_dtype;
        if (it.pid_from >= 0) {
            // inherit the patterns of an earlier item: same shape and the same table, so that ids mean the same masks
            if (it.pid_from >= i) {
                set_err(ctx, "pid_from must name an earlier item");
                return RTOSS_ERR_INVALID_ARG;
            }
            const rtoss_batch_item& par = items[it.pid_from];
            if (par.Cout != it.Cout || par.Cin != it.Cin || par.ksize != it.ksize || par.P != it.P || par.k != it.k ||
                memcmp(par.masks_host, it.masks_host, sizeof(uint16_t) * (size_t)it.P) != 0) {
                set_err(ctx, "pid_from names a layer of another shape or pattern table");
                return RTOSS_ERR_INVALID_ARG;
            }
            B.w_sel = layers[(size_t)it.pid_from].w_sel;  // the root of the chain
            B.sel_dtype = layers[(size_t)it.pid_from].sel_dtype;
        } else if (it.pid_from != -1) {
            set_err(ctx, "pid_from must be -1 or the index of an earlier item");
            return RTOSS_ERR_INVALID_ARG;
        }
        B.pid_out = it.pid_dev;
        B.pid_out_vec = (reinterpret_cast<uintptr_t>(it.pid_dev) & 1) == 0;
        B.pid = p->pid;
        B.val = p->val;
        B.wtc = p->wtc;
        B.perm = p->perm;
        B.bucket_off = p->bucket_off;
        B.issue = p->issue;
        B.issue_n = p->issue_n;
        B.n_kernels = p->n_kernels;
        B.lay = rtoss_wtc_layout_of(it.Cout, it.Cin, it.ksize, p->dtype);
        B.Cout = it.Cout;
        B.Cin = it.Cin;
        B.ksize = it.ksize;
        B.P = it.P;
        B.k = it.k;
        B.k_magic = (65536u + (unsigned)it.k - 1u) / (unsigned)it.k;
        B.v_dtype = (int)p->dtype;
        memcpy(B.masks, it.masks_host, sizeof(uint16_t) * (size_t)it.P);
        B.chunk0 = (unsigned)chunks.size();
        const long long nc = (p->n_kernels + chunk - 1) / chunk;
        if ((long long)chunks.size() + nc > 0x7FFFFFFFLL) {
            set_err(ctx, "model too large for one batch");
            return RTOSS_ERR_UNSUPPORTED;
        }
        const size_t kernel_bytes = 9 * (B.sel_dtype == RTOSS_F32 ? 4 : 2);
        for (long long c = 0; c < nc; ++c) {
            const long long left = p->n_kernels - c * chunk;
            chunks.push_back(BatchChunk{static_cast<const unsigned char*>(B.w_sel) + (size_t)c * chunk * kernel_bytes,
                                        (unsigned)((left < chunk ? left : chunk) * (long long)kernel_bytes), (unsigned)i});
        }
        B.sixteens = rtoss_dev::order_in_sixteens(it.Cout, it.P, kernels) ? 1 : 0;
        const int per = rtoss_dev::order_channels_of(B.sixteens != 0);
        sixteens = sixteens || (it.ksize == 3 && B.sixteens);
        B.task0 = (unsigned)task_layer.size();
        if (it.ksize == 3) task_layer.insert(task_layer.end(), (size_t)((it.Cin + per - 1) / per), (uint32_t)i);
    }
    rtoss_batch* b = new (std::nothrow) rtoss_batch();
    if (!b) return RTOSS_ERR_ALLOC;
    memset(b, 0, sizeof(*b));
    b->device = ctx->device;
    b->L = L;
    b->n_chunks = (unsigned)chunks.size();
    b->n_tasks = (unsigned)task_layer.size();
    b->sixteens = sixteens;
    b->threads = threads;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ctx->device);
    if (threads == kSmallThreads) rtoss_dev::writers_carveout<batch_select_pack_kernel<kSmallThreads>>();
    else rtoss_dev::writers_carveout<batch_select_pack_kernel<kBatchThreads>>();
    if (sixteens) rtoss_dev::writers_carveout<batch_order_kernel<true>>();
    else rtoss_dev::writers_carveout<batch_order_kernel<false>>();
    cudaError_t e = cudaMalloc((void**)&b->layers_dev, sizeof(BatchLayer) * (size_t)L);
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->chunks_dev, sizeof(BatchChunk) * (chunks.size() + 1));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->task_layer_dev, sizeof(uint32_t) * (task_layer.size() + 1));
    if (e == cudaSuccess) e = cudaMemcpy(b->layers_dev, layers.data(), sizeof(BatchLayer) * (size_t)L, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !chunks.empty())
        e = cudaMemcpy(b->chunks_dev, chunks.data(), sizeof(BatchChunk) * chunks.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !task_layer.empty())
        e = cudaMemcpy(b->task_layer_dev, task_layer.data(), sizeof(uint32_t) * task_layer.size(), cudaMemcpyHostToDevice);
    // the handles take the batch's tables (a convolution reads the handle's device copy of the masks)
    for (int i = 0; i < L && e == cudaSuccess; ++i) {
        rtoss_packed* p = items[i].packed;
        if (memcmp(p->masks, items[i].masks_host, sizeof(uint16_t) * (size_t)items[i].P) != 0) {
            memset(p->masks, 0, sizeof(p->masks));
            memcpy(p->masks, items[i].masks_host, sizeof(uint16_t) * (size_t)items[i].P);
            e = cudaMemcpy(p->masks_dev, p->masks, sizeof(uint16_t) * 256, cudaMemcpyHostToDevice);
        }
    }
    cudaSetDevice(prev);
    if (e != cudaSuccess) {
        cudaGetLastError();
        rtoss_batch_destroy(b);
        set_err(ctx, "device allocation or upload failed");
        return RTOSS_ERR_ALLOC;
    }
    *out = b;
    return RTOSS_OK;
}

rtoss_status rtoss_batch_select_pack(rtoss_ctx* ctx, const rtoss_batch* b, void* cuda_stream) {
    if (!ctx) return RTOSS_ERR_INVALID_ARG;
    if (!b || b->device != ctx->device) {
        set_err(ctx, "null batch or batch of another device");
        return RTOSS_ERR_INVALID_ARG;
    }
    rtoss_device_guard on_device(ctx->device);   // the caller's current device comes back when the call returns
    cudaStream_t s = (cudaStream_t)cuda_stream;
    cudaError_t e = cudaSuccess;
    const unsigned cap = (unsigned)ctx->sm_count * 8u;
    if (b->n_chunks && b->threads == kSmallThreads) {
        e = rtoss_dev::launch_pdl(batch_select_pack_kernel<kSmallThreads>, b->n_chunks, kSmallThreads, 0, s, (const BatchLayer*)b->layers_dev,
                                  (const BatchChunk*)b->chunks_dev, b->n_chunks, (int)(b->n_tasks != 0));
    } else if (b->n_chunks) {
        const unsigned resident = (unsigned)ctx->sm_count * 6u;   // (what the kernel's launch bounds allow)
        const unsigned grid = b->n_chunks < resident ? b->n_chunks : resident;
        e = rtoss_dev::launch_pdl(batch_select_pack_kernel<kBatchThreads>, grid, kBatchThreads, 0, s, (const BatchLayer*)b->layers_dev,
                                  (const BatchChunk*)b->chunks_dev, b->n_chunks, (int)(b->n_tasks != 0));
    }
    if (e == cudaSuccess && b->n_tasks) {
        const unsigned grid = b->n_tasks < cap ? b->n_tasks : cap;
        e = b->sixteens ? rtoss_dev::launch_pdl(batch_order_kernel<true>, grid, rtoss_dev::kOrderThreads, 0, s, (const BatchLayer*)b->layers_dev,
                                                (const uint32_t*)b->task_layer_dev, b->n_tasks)
                        : rtoss_dev::launch_pdl(batch_order_kernel<false>, grid, rtoss_dev::kOrderWarps * 32, 0, s, (const BatchLayer*)b->layers_dev,
                                                (const uint32_t*)b->task_layer_dev, b->n_tasks);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        snprintf(ctx->err, sizeof(ctx->err), "batch launch: %s", cudaGetErrorString(e));
        return RTOSS_ERR_CUDA;
    }
    return RTOSS_OK;
}

void rtoss_batch_destroy(rtoss_batch* b) {
    if (!b) return;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(b->device);
    if (b->layers_dev) cudaFree(b->layers_dev);
    if (b->chunks_dev) cudaFree(b->chunks_dev);
    if (b->task_layer_dev) cudaFree(b->task_layer_dev);
    cudaSetDevice(prev);
    delete b;
}

}  // extern "C"
