// 16-bit activations that the tensor path cannot read where they lie -- NCHW tensors, or channels-last ones whose pixels
// are no multiple of 16 bytes -- written once as channels-last rows of cin_p channels (a multiple of eight, the padding
// zero), which its TMA copies take.  The pass is a read and a write of the tensor (for a 128-channel 80x80 batch of eight
// 26 MB, mostly from and to L2: about 5 us); the FMA path, which used to take these calls, pays for the missing tensor cores
// ten times that and more.
#include <cuda_runtime.h>

#include "conv_common.cuh"

namespace {

using namespace rtoss_dev;

constexpr int kTileC = 64, kTileP = 64;   // channels x pixels a block turns
constexpr int kPitchW = 34;               // words per pixel row of the tile: 32 channel pairs + 2 (8-byte aligned; rows 8 apart fall 16 banks apart)

struct RepackArgs {
    const unsigned short* x;
    unsigned short* out;
    int Cin, cp;         // channels, channels per stored pixel
    int H, W, S, Wo;     // input image; every S-th row and column is kept
    long long plane;     // H * W
    int pixels;          // kept pixels per image
    int c_blocks, p_blocks;
};

// Eight pixels of one channel: v[i] = pixel p0 + i (zero beyond the image or the channels).
template <int VEC>   // bytes per load: 16 / 4 / 2 where planes start on such boundaries; 0: every S-th row and column
__device__ __forceinline__ uint4 load8(const RepackArgs& a, const unsigned short* src, int p0) {
    unsigned w[4] = {0, 0, 0, 0};
    if (VEC == 16) {
        if (p0 < a.pixels) return __ldg(reinterpret_cast<const uint4*>(src + p0));   // (the plane is a multiple of eight)
    } else if (VEC == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (p0 + 2 * i < a.pixels) w[i] = __ldg(reinterpret_cast<const unsigned*>(src + p0) + i);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (p0 + i < a.pixels) {
                long long at = p0 + i;
                if (VEC == 0) {
                    const int oy = (p0 + i) / a.Wo, ox = (p0 + i) - oy * a.Wo;
                    at = ((long long)oy * a.W + ox) * a.S;
                }
                w[i >> 1] |= (unsigned)__ldg(src + at) << (16 * (i & 1));
            }
        }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// NCHW: a thread takes eight pixels of two neighbouring channels, pairs them into words {channel c, channel c + 1} and
// stores them to the tile [pixel][channel pair]; the tile leaves as 16-byte pieces of eight channels.
template <int VEC>
__global__ void __launch_bounds__(256) repack_nchw_kernel(const RepackArgs a) {
    pdl_enter();
    __shared__ __align__(16) unsigned tile[kTileP * kPitchW];
    int b = blockIdx.x;
    const int pb = b % a.p_blocks;
    b /= a.p_blocks;
    const int cb = b % a.c_blocks, n = b / a.c_blocks;
    const int c0 = cb * kTileC, p0 = pb * kTileP;
    {
        // lanes: four groups of eight pixels (64 contiguous bytes of a plane) x eight channel pairs
        const int pg = (threadIdx.x & 3) | ((threadIdx.x >> 5) & 1) << 2;
        const int cpair = ((threadIdx.x >> 2) & 7) | (threadIdx.x >> 6) << 3;
        const int c = c0 + 2 * cpair, p = p0 + 8 * pg;
        uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
        if (c < a.Cin) lo = load8<VEC>(a, a.x + ((size_t)n * a.Cin + c) * a.plane, p);
        if (c + 1 < a.Cin) hi = load8<VEC>(a, a.x + ((size_t)n * a.Cin + c + 1) * a.plane, p);
        unsigned* t = tile + (8 * pg) * kPitchW + cpair;
        const unsigned l[4] = {lo.x, lo.y, lo.z, lo.w}, h[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            t[(2 * i) * kPitchW] = __byte_perm(l[i], h[i], 0x5410);
            t[(2 * i + 1) * kPitchW] = __byte_perm(l[i], h[i], 0x7632);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int item = (int)threadIdx.x + 256 * q, px = item >> 3, g = item & 7;
        const int p = p0 + px, c = c0 + 8 * g;
        if (p < a.pixels && c < a.cp) {
            const uint2* s = reinterpret_cast<const uint2*>(tile + px * kPitchW + 4 * g);
            const uint2 u = s[0], v = s[1];
            *reinterpret_cast<uint4*>(a.out + ((size_t)n * a.pixels + p) * a.cp + c) = make_uint4(u.x, u.y, v.x, v.y);
        }
    }
}

// Channels last, rows of Cin channels -> rows of cp: a thread writes one 16-byte piece.
template <int VEC>   // bytes per load: 8 / 4 / 2 as Cin allows
__global__ void __launch_bounds__(256) repack_nhwc_kernel(const RepackArgs a, unsigned pieces, unsigned per_px) {
    pdl_enter();
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < pieces; i += gridDim.x * 256u) {
        const unsigned px = i / per_px, g = i - px * per_px;
        size_t src = px;
        if (a.S > 1) {
            const unsigned n = px / (unsigned)a.pixels, r = px - n * (unsigned)a.pixels;
            const unsigned oy = r / (unsigned)a.Wo, ox = r - oy * (unsigned)a.Wo;
            src = (size_t)n * a.plane + ((size_t)oy * a.W + ox) * a.S;
        }
        const unsigned short* s = a.x + src * a.Cin + 8 * g;
        const int left = a.Cin - 8 * (int)g;   // channels of this piece that exist (the rest is padding)
        unsigned w[4] = {0, 0, 0, 0};
        if (VEC == 8) {
            if (left >= 4) {
                const uint2 u = __ldg(reinterpret_cast<const uint2*>(s));
                w[0] = u.x, w[1] = u.y;
            }
            if (left >= 8) {
                const uint2 u = __ldg(reinterpret_cast<const uint2*>(s) + 1);
                w[2] = u.x, w[3] = u.y;
            }
        } else if (VEC == 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (2 * j < left) w[j] = __ldg(reinterpret_cast<const unsigned*>(s) + j);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j < left) w[j >> 1] |= (unsigned)__ldg(s + j) << (16 * (j & 1));
        }
        reinterpret_cast<uint4*>(a.out)[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

}  // namespace

// x: N x Cin x H x W, 16-bit, in `layout`; out: [N][Ho][Wo][cp] with every S-th row and column (S = 1: all).
int rtoss_launch_repack16(const void* x, void* out, int N, int Cin, int cp, int H, int W, int S, rtoss_layout layout, void* stream) {
    RepackArgs a;
    a.x = static_cast<const unsigned short*>(x);
    a.out = static_cast<unsigned short*>(out);
    a.Cin = Cin, a.cp = cp, a.H = H, a.W = W, a.S = S;
    a.Wo = (W - 1) / S + 1;
    a.plane = (long long)H * W;
    a.pixels = ((H - 1) / S + 1) * a.Wo;
    a.c_blocks = (cp + kTileC - 1) / kTileC;
    a.p_blocks = (a.pixels + kTileP - 1) / kTileP;
    cudaStream_t s = (cudaStream_t)stream;
    if (layout == RTOSS_NCHW) {
        const long long blocks = (long long)N * a.c_blocks * a.p_blocks;
        if (blocks > 0x7FFFFFFFLL) return (int)cudaErrorInvalidValue;
        const dim3 grid((unsigned)blocks);
        if (S > 1) return (int)launch_pdl(repack_nchw_kernel<0>, grid, 256, 0, s, a);
        if (a.plane % 8 == 0) return (int)launch_pdl(repack_nchw_kernel<16>, grid, 256, 0, s, a);
        if (a.plane % 2 == 0) return (int)launch_pdl(repack_nchw_kernel<4>, grid, 256, 0, s, a);
        return (int)launch_pdl(repack_nchw_kernel<2>, grid, 256, 0, s, a);
    }
    const long long pieces = (long long)N * a.pixels * (cp / 8);
    if (pieces > 0x7FFFFFFFLL) return (int)cudaErrorInvalidValue;
    const dim3 grid((unsigned)(pieces < 148 * 8 * 256 ? (pieces + 255) / 256 : 148 * 8));
    const unsigned np = (unsigned)pieces, per = (unsigned)(cp / 8);
    if (Cin % 4 == 0) return (int)launch_pdl(repack_nhwc_kernel<8>, grid, 256, 0, s, a, np, per);
    if (Cin % 2 == 0) return (int)launch_pdl(repack_nhwc_kernel<4>, grid, 256, 0, s, a, np, per);
    return (int)launch_pdl(repack_nhwc_kernel<2>, grid, 256, 0, s, a, np, per);
}
