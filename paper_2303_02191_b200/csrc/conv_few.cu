// Convolutions of few outputs on the FP32 FMA pipes (3x3 and 1x1): calls that would leave most SMs idle in the staged
// kernels (conv3x3_alu.cu, conv1x1_alu.cu), whose CTAs walk the input channels one chunk after the other -- load, wait,
// convert, barrier, compute -- so that a small image costs a chain of memory latencies and hardly any arithmetic.
//
// Here the input channels of a tile are dealt to the eight warps of a CTA (warp w takes channels w, w + 8, ...), every
// lane keeps four neighbouring output pixels of four filters, its windows come straight from global memory (one channel
// ahead), and the eight partial sums of an output are added up in shared memory at the end: no barrier inside the loop,
// four times as many CTAs, a chain of two or three latencies in all.  The weights of eight channels per warp are expanded at a
// time, a thread per (channel, filter); a handle's arrays may be read ahead of the wait for earlier kernels (conv_common.cuh),
// so the first expansion overlaps the kernel in front.
// Sums are fp32; an output's order of summation is fixed (channels of a warp ascending, then warps ascending).
#include "conv_common.cuh"

namespace {

using namespace rtoss_dev;

constexpr int kFewWarps = 8, kFewPx = 4, kFewCo = 4, kFewCh = 8;   // kFewCh: channels of a warp expanded at a time

struct FewArgs {
    const void* x;
    void* y;
    const void* val;
    const uint8_t* pid;
    const uint16_t* masks;
    const float* bias;
    int val_dtype;
    int N, Cin, Cout, H, W, Ho, Wo, k, P, act;
    int LX, LY, tiles_x, tiles_y;
    long long runs;                       // 1x1: full runs of nine
    long long x_img, x_ch, x_row, x_px;   // element strides of x
    long long y_img, y_ch, y_row, y_px;   // and of y
    int y_c_off;
};

// kVec: default layout, rows of a multiple of four pixels, 16-byte aligned -- a lane's four (stride 2: eight) columns are
// whole vectors, and the column on either side of them comes from the lane beside it.
template <typename T, int KS, int S, bool kVec>
__global__ void __launch_bounds__(kFewWarps * 32, 2) conv_few_kernel(const FewArgs a) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int WH = KS, WW = (kFewPx - 1) * S + KS, kSlots = KS == 3 ? 12 : 1;
    __shared__ __align__(16) float sW[kFewWarps][kFewCh * kFewCo * kSlots + 4];   // (+4: neighbouring channels on different banks)
    __shared__ uint16_t sM[256];
    __shared__ float sR[kFewWarps][kFewCo * kFewPx][33];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, co0 = blockIdx.y * kFewCo;
    int tile = blockIdx.x;
    const int tx = tile % a.tiles_x;
    tile /= a.tiles_x;
    const int ty = tile % a.tiles_y, n = tile / a.tiles_y;
    const int ly = lane / a.LX, lx = lane - ly * a.LX;   // (LX * LY is 32)
    const int ox = (tx * a.LX + lx) * kFewPx, oy = ty * a.LY + ly;
    constexpr int kPad = KS / 2;
    const int ix = ox * S - kPad, iy = oy * S - kPad;

    // A 3x3 kernel's dense weights: mask m, kept values v.
    auto put3 = [&](float* to, unsigned m, const float (&v)[9]) {
        float4* z = reinterpret_cast<float4*>(to);
        z[0] = z[1] = z[2] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 9; ++j)
            if (m) {   // value j belongs to the j-th kept tap
                to[__ffs(m) - 1] = v[j];
                m &= m - 1;
            }
    };
    // The first kFewCh channels of every warp, ahead of the wait: the block's threads take (channel, filter) pairs whose ids and
    // values are neighbours, so that a CTA asks L2 for every line once, and the masks come in once a CTA.  The reads have to come
    // from L2: nothing orders this SM's L1 behind the kernel that wrote the handle (conv_common.cuh).  fp32 and 16-bit calls of
    // 10 to 3000 CTAs, 260 of them, launches back to back, against each warp reading its own channels through L1: as fast on
    // average, 3x3 7->7 @11x106 x12 4.0 -> 4.6 us, fp32 1x1 calls of 200 to 450 CTAs up to 1.27 times slower (fewer registers
    // let four CTAs on an SM instead of three, which share the SMs out less evenly).  Each warp's own channels from L2: 3 to 6 %
    // slower, 5.2 us; with an acquire fence, which empties the L1 under the CTAs already running: 3 %, 1x1 46->323 @19x9 x2
    // 5.8 -> 8.7 us; behind the wait: 6 to 9 %.
    {
        const int ci = threadIdx.x % (kFewWarps * kFewCh), f = threadIdx.x / (kFewWarps * kFewCh), co = co0 + f;
        const bool real = ci < a.Cin && co < a.Cout;
        float* to = sW[ci % kFewWarps] + (ci / kFewWarps * kFewCo + f) * kSlots;
        unsigned p = 0;
        sM[threadIdx.x] = (int)threadIdx.x < a.P ? __ldcg(a.masks + threadIdx.x) : (uint16_t)0;   // (an id outside the table keeps nothing)
        if constexpr (KS == 3) {
            float v[9];
            const size_t kid = (size_t)co * a.Cin + ci;
            if (real) p = __ldcg(a.pid + kid);
            if (real) load_vals_cg(a.val, kid, a.k, a.val_dtype, v);
            __syncthreads();
            put3(to, real ? sM[p] : 0u, v);
        } else {
            const long long e = (long long)co * a.Cin + ci, g = e / 9;
            const int t = (int)(e - 9 * g);
            const bool kept = real && g < a.runs;
            if (kept) p = __ldcg(a.pid + g);
            __syncthreads();
            float w = 0.f;
            if (kept) {
                const unsigned m = sM[p];
                if (m & (1u << t)) w = load_val_cg(a.val, (size_t)(g * a.k + __popc(m & ((1u << t) - 1u))), a.val_dtype);
            }
            to[0] = w;
        }
        __syncthreads();
    }
    // The next ones, behind the wait, by the warp itself: a lane expands the kernel of channel warp + 8 (i0 + lane / 4), filter
    // co0 + lane % 4.
    auto expand = [&](int i0) {
        const int q = lane / kFewCo, f = lane % kFewCo, ci = warp + kFewWarps * (i0 + q), co = co0 + f;
        float* to = sW[warp] + lane * kSlots;
        const bool real = ci < a.Cin && co < a.Cout;
        if constexpr (KS == 3) {
            float v[9];
            unsigned m = 0;
            if (real) {
                const size_t kid = (size_t)co * a.Cin + ci;
                const unsigned p = __ldg(a.pid + kid);
#pragma unroll
                for (int j = 0; j < 9; ++j) v[j] = j < a.k ? load_val(a.val, kid * a.k + j, a.val_dtype) : 0.f;
                m = sM[p];
            }
            put3(to, m, v);
        } else {
            float w = 0.f;
            if (real) {
                const long long e = (long long)co * a.Cin + ci, g = e / 9;
                const int t = (int)(e - 9 * g);
                if (g < a.runs) {
                    const unsigned m = sM[__ldg(a.pid + g)];
                    if (m & (1u << t)) w = load_val(a.val, (size_t)(g * a.k + __popc(m & ((1u << t) - 1u))), a.val_dtype);
                }
            }
            to[0] = w;
        }
        __syncwarp();
    };
    const int mine = a.Cin > warp ? (a.Cin - warp + kFewWarps - 1) / kFewWarps : 0;   // this warp's channels
    // which values of the window lie inside the image
    unsigned inside = 0;
#pragma unroll
    for (int r = 0; r < WH; ++r)
#pragma unroll
        for (int c = 0; c < WW; ++c)
            if (oy < a.Ho && iy + r >= 0 && iy + r < a.H && ix + c >= 0 && ix + c < a.W) inside |= 1u << (r * WW + c);
    const T* __restrict__ xb = reinterpret_cast<const T*>(a.x) + (n * a.x_img + iy * a.x_row + ix * a.x_px);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // The next channel's window: as loaded (kVec: whole vectors, and the outer columns of the lanes at the ends of a row).
    constexpr int kVecs = S;   // vectors of four columns a row (from ix + kPad on)
    float next[WH][WW];
    auto fetch = [&](int i) {
        const T* p = xb + (warp + kFewWarps * i) * a.x_ch;
#pragma unroll
        for (int r = 0; r < WH; ++r) {
            if constexpr (kVec) {
                const T* row = p + r * a.x_row;
                float v[4 * kVecs];
#pragma unroll
                for (int h = 0; h < kVecs; ++h) {
                    const bool ok = inside & (1u << (r * WW + kPad + 4 * h));   // (a vector lies inside the row or outside)
                    if constexpr (sizeof(T) == 4) {
                        const float4 u = ok ? *reinterpret_cast<const float4*>(row + kPad + 4 * h) : make_float4(0.f, 0.f, 0.f, 0.f);
                        v[4 * h] = u.x, v[4 * h + 1] = u.y, v[4 * h + 2] = u.z, v[4 * h + 3] = u.w;
                    } else {
                        const uint2 u = ok ? *reinterpret_cast<const uint2*>(row + kPad + 4 * h) : make_uint2(0u, 0u);
                        const T* e = reinterpret_cast<const T*>(&u);
#pragma unroll
                        for (int c = 0; c < 4; ++c) v[4 * h + c] = to_f32<T>(e[c]);
                    }
                }
                if constexpr (KS == 3) {
                    next[r][0] = 0.f;
                    if (lx == 0 && (inside & (1u << (r * WW)))) next[r][0] = to_f32<T>(row[0]);
                    if constexpr (S == 1) {
                        next[r][WW - 1] = 0.f;
                        if (lx == a.LX - 1 && (inside & (1u << (r * WW + WW - 1)))) next[r][WW - 1] = to_f32<T>(row[WW - 1]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 4 * kVecs; ++c)
                    if (kPad + c < WW) next[r][kPad + c] = v[c];
            } else {
#pragma unroll
                for (int c = 0; c < WW; ++c) {
                    next[r][c] = 0.f;
                    if (inside & (1u << (r * WW + c))) next[r][c] = to_f32<T>(p[r * a.x_row + c * a.x_px]);
                }
            }
        }
    };
    float acc[kFewCo][kFewPx];
#pragma unroll
    for (int f = 0; f < kFewCo; ++f)
#pragma unroll
        for (int px = 0; px < kFewPx; ++px) acc[f][px] = 0.f;
    if (mine) fetch(0);
#pragma unroll 1
    for (int i = 0; i < mine; ++i) {
        if (i && i % kFewCh == 0) {
            __syncwarp();   // the warp's lanes have read the expansion before
            expand(i);
        }
        float win[WH][WW];
#pragma unroll
        for (int r = 0; r < WH; ++r)
#pragma unroll
            for (int c = 0; c < WW; ++c) win[r][c] = next[r][c];
        if (i + 1 < mine) fetch(i + 1);
        if constexpr (kVec && KS == 3) {
#pragma unroll
            for (int r = 0; r < WH; ++r) {   // the neighbour's last (first) column; beyond the image it is a zero there too
                const float left = __shfl_up_sync(0xFFFFFFFFu, win[r][4 * S], 1);
                if (lx != 0) win[r][0] = left;
                if constexpr (S == 1) {
                    const float right = __shfl_down_sync(0xFFFFFFFFu, win[r][1], 1);
                    if (lx != a.LX - 1) win[r][WW - 1] = right;
                }
            }
        }
#pragma unroll
        for (int f = 0; f < kFewCo; ++f) {
            const float* w = sW[warp] + (i % kFewCh * kFewCo + f) * kSlots;
            float wv[kSlots];
            if constexpr (KS == 3) {
#pragma unroll
                for (int h = 0; h < 3; ++h) *reinterpret_cast<float4*>(wv + 4 * h) = reinterpret_cast<const float4*>(w)[h];
            } else {
                wv[0] = w[0];
            }
#pragma unroll
            for (int r = 0; r < KS; ++r)
#pragma unroll
                for (int c = 0; c < KS; ++c)
#pragma unroll
                    for (int px = 0; px < kFewPx; ++px) acc[f][px] = fmaf(wv[r * KS + c], win[r][px * S + c], acc[f][px]);
        }
    }
#pragma unroll
    for (int f = 0; f < kFewCo; ++f)
#pragma unroll
        for (int px = 0; px < kFewPx; ++px) sR[warp][f * kFewPx + px][lane] = acc[f][px];
    __syncthreads();
    T* __restrict__ yb = reinterpret_cast<T*>(a.y) + n * a.y_img;
    for (int o = threadIdx.x; o < kFewCo * kFewPx * 32; o += kFewWarps * 32) {   // (filter, lane of the tile, pixel): neighbours along a row
        const int f = o / (kFewPx * 32), l = o / kFewPx % 32, px = o % kFewPx;
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < kFewWarps; ++w) sum += sR[w][f * kFewPx + px][l];
        const int row = l / a.LX, x = (tx * a.LX + l - row * a.LX) * kFewPx + px, y = ty * a.LY + row, co = co0 + f;
        if (x < a.Wo && y < a.Ho && co < a.Cout)
            yb[(a.y_c_off + co) * a.y_ch + y * a.y_row + x * a.y_px] = from_f32<T>(activate(sum + (a.bias ? __ldg(a.bias + co) : 0.f), a.act));
    }
}

// The lane arrangement (LX x LY lanes of four pixels) that covers the map with the fewest tiles, the wider one among equals.
long few_lanes(int Ho, int Wo, int* LX, int* LY) {
    long best = 0;
    for (int lx = 32; lx >= 1; lx >>= 1) {
        const int ly = 32 / lx;
        const long tiles = (long)((Wo + lx * kFewPx - 1) / (lx * kFewPx)) * ((Ho + ly - 1) / ly);
        if (!best || tiles < best) best = tiles, *LX = lx, *LY = ly;
    }
    return best;
}

template <typename T, bool kVec>
void launch_few(const FewArgs& a, int ks, int stride, dim3 grid, cudaStream_t s) {
    if (ks == 3 && stride == 1) rtoss_dev::launch_pdl(conv_few_kernel<T, 3, 1, kVec>, grid, kFewWarps * 32, 0, s, a);
    else if (ks == 3) rtoss_dev::launch_pdl(conv_few_kernel<T, 3, 2, kVec>, grid, kFewWarps * 32, 0, s, a);
    else if (stride == 1) rtoss_dev::launch_pdl(conv_few_kernel<T, 1, 1, kVec>, grid, kFewWarps * 32, 0, s, a);
    else rtoss_dev::launch_pdl(conv_few_kernel<T, 1, 2, kVec>, grid, kFewWarps * 32, 0, s, a);
}

}  // namespace

// Whole vectors of four columns (see the kernel)?
static bool few_vec(const rtoss_conv_desc* d, const void* x) {
    return d->layout == RTOSS_NCHW && d->W % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
}

// Is this a call for the kernel above?  Its time grows with its CTAs (tiles of 128 pixels x 4 filters) from the first on, that
// of the staged kernels in steps of a full device, so there is a number of CTAs up to which this one is faster.  420 calls of
// 300 to 9000 CTAs, both layouts, all types, 1 to 512 channels, this kernel's time / the staged one's:
//   3x3  at most 8 channels (one a warp: expansion and sum are all a CTA does)  315 CTAs 0.87, 560 0.99, 636 1.18, 660 0.73, 732 1.23,
//                  768 0.59, 900 1.11, 1000 1.37, 1050 2.07, 3528 1.95
//        9 to 16        664 0.44, 1020 0.57, 1092 0.88, 1290 1.04, 1590 1.25, 1848 1.63, 3871 1.71
//        more, default layout with whole vectors   1080 0.89, 3200 0.80 (64->64 @80x80 x4), 3840 0.75, 6400 1.48, 7020 1.40
//        more, other    1200 0.86, 1600 1.00, 3200 1.10, 5040 1.64; 16 bits channels last 1020 0.93, 1428 1.12, 1440 1.28
//        channels last in multiples of 8, which the staged kernel fetches as whole vectors   120 CTAs 0.64, 150 0.73, 240 0.98, 300 1.23,
//                  480 1.95, 640 1.33, 1260 2.88 (96->77 @23x104 x3 98 / 282 us)
//   1x1  at most 16 channels   3060 0.79, 3864 0.86, 4725 1.15, 5640 1.24
//        more           2560 0.29, 3570 0.64, 5220 0.86, 6400 1.19; without vectors 3840 0.84
// 16-bit calls that the tensor cores would take behind a layout pass (two launches, 5 us and more): only where a warp's
// share of the channels is short.  160 calls, by CTAs x channels per warp, this kernel / the tensor cores:
//   3x3, default layout, up to 48 channels   280 0.52, 480 0.69, 594 0.89, 600 1.12, 702 1.08, 1024 1.73; channels last, up to 16  504 0.85, 1056 2.08
//   1x1  at most 8 channels   360 0.64, 666 0.73, 750 1.07, 1302 1.56; up to 64, default layout   675 0.46, 1122 0.63, 1450 0.58, 1815 0.70, 1848 1.14;
//        channels last  600 0.90, 936 1.20, 1188 0.95, 1440 1.19
bool rtoss_few_eligible(const rtoss_packed* p, const rtoss_conv_desc* d, const void* x, bool repack) {
    if (p->ksize == 3 && p->Cin <= 4) return false;   // (stems have their own kernel)
    int lx, ly;
    const long long ctas = (long long)d->N * few_lanes((d->H - 1) / d->stride + 1, (d->W - 1) / d->stride + 1, &lx, &ly) * ((p->Cout + kFewCo - 1) / kFewCo);
    if (repack) {
        const long long steps = ctas * ((p->Cin + kFewWarps - 1) / kFewWarps);
        return p->ksize == 3 ? p->Cin <= (d->layout == RTOSS_NCHW ? 48 : 16) && steps <= 600 : p->Cin <= 64 && steps <= (p->Cin <= 8 ? 700 : d->layout == RTOSS_NCHW ? 1800 : 1200);
    }
    const bool vec = few_vec(d, x);
    if (p->ksize == 1) return ctas <= (vec && p->Cin > 16 ? 5000 : 4200);
    if (d->layout == RTOSS_NHWC && p->Cin % 8 == 0) return ctas <= 150;
    if (p->Cin <= 16) return ctas <= (p->Cin <= 8 ? 800 : 1200);
    return ctas <= (vec ? 4000 : d->layout == RTOSS_NHWC && d->io_dtype != RTOSS_F32 ? 1400 : 1600);
}

int rtoss_launch_conv_few(const rtoss_packed* p, const void* x, void* y, const rtoss_conv_desc* d, void* stream) {
    FewArgs a = {};
    a.x = x;
    a.y = y;
    a.val = p->val;
    a.pid = p->pid;
    a.masks = p->masks_dev;
    a.bias = d->bias_dev;
    a.val_dtype = (int)p->dtype;
    a.N = d->N;
    a.Cin = p->Cin;
    a.Cout = p->Cout;
    a.H = d->H;
    a.W = d->W;
    a.Ho = (d->H - 1) / d->stride + 1;
    a.Wo = (d->W - 1) / d->stride + 1;
    a.k = p->k;
    a.P = p->P;
    a.act = (int)d->act;
    a.runs = p->n_kernels;
    const long long cs = d->y_channel_stride ? d->y_channel_stride : p->Cout;
    if (d->layout == RTOSS_NCHW) {
        a.x_px = 1, a.x_row = d->W, a.x_ch = (long long)d->H * d->W, a.x_img = a.x_ch * p->Cin;
        a.y_px = 1, a.y_row = a.Wo, a.y_ch = (long long)a.Ho * a.Wo, a.y_img = a.y_ch * cs;
    } else {
        a.x_ch = 1, a.x_px = p->Cin, a.x_row = a.x_px * d->W, a.x_img = a.x_row * d->H;
        a.y_ch = 1, a.y_px = cs, a.y_row = cs * a.Wo, a.y_img = a.y_row * a.Ho;
    }
    a.y_c_off = d->y_channel_offset;
    const long tiles = few_lanes(a.Ho, a.Wo, &a.LX, &a.LY);
    a.tiles_x = (a.Wo + a.LX * kFewPx - 1) / (a.LX * kFewPx);
    a.tiles_y = (a.Ho + a.LY - 1) / a.LY;
    const dim3 grid((unsigned)(tiles * a.N), (unsigned)((a.Cout + kFewCo - 1) / kFewCo));
    cudaStream_t s = (cudaStream_t)stream;
    const bool vec = few_vec(d, x);
#define RTOSS_FEW(T_) (vec ? launch_few<T_, true>(a, p->ksize, d->stride, grid, s) : launch_few<T_, false>(a, p->ksize, d->stride, grid, s))
    switch (d->io_dtype) {
        case RTOSS_F32: RTOSS_FEW(float); break;
        case RTOSS_BF16: RTOSS_FEW(__nv_bfloat16); break;
        case RTOSS_F16: RTOSS_FEW(__half); break;
    }
#undef RTOSS_FEW
    return (int)cudaGetLastError();
}
