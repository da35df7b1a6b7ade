// Weight and bias gradients of the 3x3 convolutions on the tensor cores:
//   dw[tap][co][ci] = sum over pixels p of dout[p][co] in[p + shift(tap)][ci]
//   dbias[co]       = sum over pixels p of dout[p][co]
// -- a contraction over the pixels, the strided index of both NHWC operands.
//
// A warp owns a 16 (co) x 16 (ci) block of all nine taps: 18 m16n8k16
// accumulators (72 FP32 registers), A = dout^T and B = the input, both read
// from shared memory by transposing ldmatrix, so that a tap is only another
// start pixel of the same staged tile.  One step of 16 pixels is 10
// ldmatrix.x4 for 18 MMAs.  mma.sync and not tcgen05: the block's rows are 16
// output channels on most layers (tcgen05 takes 64 or 128), and at 18 MMAs per
// 10 shared-memory reads the step is bound by those reads, not by the MMAs.
//
// A CTA (8 warps) takes one such channel block and a contiguous range of
// 512-pixel tiles (TX x TY of one sample); the input tile with its one-pixel
// halo and the dout tile arrive by 16-byte cp.async into two buffers, pixels
// and channels outside the tensors as zeros.  The 16-byte halves of a pixel's
// 32 bytes are swapped for every other group of four pixels, which makes the
// eight rows of an ldmatrix hit all banks from any start pixel.  Products of
// BF16 are exact in FP32 and every sum is FP32: 16 pixels per MMA, the tiles of
// a warp in order, the warps in order, then the CTAs in order
// (k_wgrad_reduce_split) -- deterministic.
//
// Before: one thread per (co, ci) pair walked 2048 pixels by scalar FMAs with
// two-byte loads.  A training batch of 16 samples at 200 x 256 (forward, loss,
// gradients): 23.10 ms, of which 21.65 in that kernel; now 1.47 ms, 32 to 54 us
// per layer (60 to 140 TFLOP/s) with the sum over the CTAs.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "internal.h"

namespace pp {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int WG_WARPS = 8;
constexpr int WG_PIX = 512;                      // pixels per tile: four 16-pixel steps per warp
// Tiles per CTA at most: 32 MMAs of a warp, one after the other.  An MMA cuts its FP32 sum
// instead of rounding it, which drifts with the chain: 512 samples of 25 x 32, 64 -> 128
// channels, cut into 10 CTAs per block (5.4e-6 relative L2 error with normal values, 1.8e-5
// with positive ones), now 3.7e-7 and 5.6e-7; the scalar kernel's 2048 rounded additions
// have 4.6e-7 and 2.0e-7.
constexpr int WG_CHAIN = 8;
constexpr int WG_MAX_IN = (64 + 2) * (8 + 2);    // halo pixels of the largest tile shapes (64x8, 32x16, 16x32)
constexpr int WG_STAGE = (WG_MAX_IN + WG_PIX) * 32;

struct WgradArgs {
    const bf16 *in, *up;          // input; channels [0, cu) from up, of half the height and width, upsampled 2x
    int cu;
    const bf16 *dout;
    int cin, cout, n, h, wd;
    int tx, ty;                   // tile: tx pixels by ty rows, tx ty = WG_PIX
    int tiles_x, tiles_y, tiles;
    int per;                      // tiles per CTA
    int tci;                      // 16-channel blocks of the input
    float *part, *partb;          // [gridDim.x][9][cout][cin], [gridDim.x][cout]
};

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// 16 bytes global -> shared, zeros when !ok.
__device__ __forceinline__ void cp16(unsigned dst, const void *src, bool ok) {
    const int n = ok ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ unsigned pix_addr(unsigned base, int p, int half) {
    return base + 32u * (unsigned)p + 16u * (unsigned)(half ^ ((p >> 2) & 1));
}

__device__ __forceinline__ void ldsm4t(unsigned a, unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(a)
                 : "memory");
}

__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Stage tile t: the input halo (tx + 2) x (ty + 2) and dout tx x ty, 16
// channels (two 16-byte halves) of each pixel.
__device__ __forceinline__ void load_tile(const WgradArgs &a, int t, unsigned sm, int co0, int ci0) {
    const int bx = t % a.tiles_x, rest = t / a.tiles_x;
    const int x0 = bx * a.tx, y0 = (rest % a.tiles_y) * a.ty, s = rest / a.tiles_y;
    const int wx = a.tx + 2, nin = wx * (a.ty + 2);
    const size_t img = (size_t)s * a.h;
    for (int e = threadIdx.x; e < 2 * nin; e += WG_WARPS * 32) {
        const int p = e >> 1, half = e & 1;
        const int r = p / wx, y = y0 + r - 1, x = x0 + (p - r * wx) - 1, c = ci0 + 8 * half;
        const bool ok = (unsigned)y < (unsigned)a.h && (unsigned)x < (unsigned)a.wd && c < a.cin;
        const bf16 *src = a.in;
        if (ok)
            src = c < a.cu ? a.up + (((size_t)s * (a.h >> 1) + (y >> 1)) * (a.wd >> 1) + (x >> 1)) * a.cu + c
                           : a.in + ((img + y) * a.wd + x) * (a.cin - a.cu) + (c - a.cu);
        cp16(pix_addr(sm, p, half), src, ok);
    }
    const unsigned sd = sm + WG_MAX_IN * 32;
    const int sh = __ffs(a.tx) - 1;
    for (int e = threadIdx.x; e < 2 * WG_PIX; e += WG_WARPS * 32) {
        const int p = e >> 1, half = e & 1;
        const int y = y0 + (p >> sh), x = x0 + (p & (a.tx - 1)), c = co0 + 8 * half;
        const bool ok = y < a.h && x < a.wd && c < a.cout;
        cp16(pix_addr(sd, p, half), a.dout + (ok ? ((img + y) * a.wd + x) * a.cout + c : 0), ok);
    }
    cp_async_group_close();
}

__global__ void __launch_bounds__(WG_WARPS * 32, 2) k_wgrad_mma(const WgradArgs a) {
    extern __shared__ __align__(128) unsigned char wsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ci0 = 16 * ((int)blockIdx.y % a.tci), co0 = 16 * ((int)blockIdx.y / a.tci);
    const bool bias = ci0 == 0;
    const unsigned sm = smem_addr(wsm);
    const int t0 = (int)blockIdx.x * a.per, t1 = min(a.tiles, t0 + a.per);
    float acc[9][2][4], accb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[q][j][e] = 0.f;
    const int wx = a.tx + 2, sh = __ffs(a.tx) - 1;
    // this lane's row of the ldmatrix blocks: A blocks (k, co) = (0,0) (0,8) (8,0) (8,8), B (k, ci) = (0,0) (8,0) (0,8) (8,8)
    const int row = lane & 7, blk = lane >> 3;
    const int ka = row + 8 * (blk >> 1), ha = blk & 1, kb = row + 8 * (blk & 1), hb = blk >> 1;
    if (t0 < t1) load_tile(a, t0, sm, co0, ci0);
    for (int t = t0; t < t1; ++t) {
        const unsigned cur = sm + (unsigned)((t - t0) & 1) * WG_STAGE;
        if (t + 1 < t1) {
            load_tile(a, t + 1, sm + (unsigned)((t + 1 - t0) & 1) * WG_STAGE, co0, ci0);
            cp_async_group_wait<1>();
        } else {
            cp_async_group_wait<0>();
        }
        __syncthreads();
        const unsigned sd = cur + WG_MAX_IN * 32;
#pragma unroll 1
        for (int st = warp; st < WG_PIX / 16; st += WG_WARPS) {
            const int p = st * 16, r = p >> sh, x = p & (a.tx - 1);
            unsigned fa[4];
            ldsm4t(pix_addr(sd, p + ka, ha), fa[0], fa[1], fa[2], fa[3]);
            if (bias) mma16816(accb, fa, 0x3F803F80u, 0x3F803F80u);   // times ones: the sum over the pixels
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                unsigned b[4];
                ldsm4t(pix_addr(cur, (r + q / 3) * wx + x + q % 3 + kb, hb), b[0], b[1], b[2], b[3]);
                mma16816(acc[q][0], fa, b[0], b[1]);
                mma16816(acc[q][1], fa, b[2], b[3]);
            }
        }
        __syncthreads();   // the buffer is free for the load after the next
    }
    // the warps' sums in warp order
    float *red = reinterpret_cast<float *>(wsm);   // [9][16 co][16 ci], then the bias [16]
    const int g = lane >> 2, tq = lane & 3;
    for (int w = 0; w < WG_WARPS; ++w) {
        if (warp == w) {
#pragma unroll
            for (int q = 0; q < 9; ++q)
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float *d = red + (q * 16 + g + 8 * (e >> 1)) * 16 + 8 * j + 2 * tq + (e & 1);
                        *d = w ? *d + acc[q][j][e] : acc[q][j][e];
                    }
            if (tq == 0) {
                float *d = red + 9 * 256 + g;
                d[0] = w ? d[0] + accb[0] : accb[0];
                d[8] = w ? d[8] + accb[2] : accb[2];
            }
        }
        __syncthreads();
    }
    float *dst = a.part + (size_t)blockIdx.x * 9 * a.cout * a.cin;
    for (int e = threadIdx.x; e < 9 * 256; e += WG_WARPS * 32) {
        const int ci = ci0 + (e & 15), co = co0 + ((e >> 4) & 15), q = e >> 8;
        if (ci < a.cin && co < a.cout) dst[((size_t)q * a.cout + co) * a.cin + ci] = red[e];
    }
    if (bias && threadIdx.x < 16 && co0 + (int)threadIdx.x < a.cout)
        a.partb[(size_t)blockIdx.x * a.cout + co0 + threadIdx.x] = red[9 * 256 + threadIdx.x];
}

// Weight e's sum over the pixels of rows [row0, row1) of all images, by scalar FMAs:
// only products of pixels inside the image and gradients that are not zero.
__device__ __noinline__ float wgrad_scalar(const WgradArgs &a, int e, long row0, long row1) {
    const int ci = e % a.cin, co = e / a.cin % a.cout, tap = e / a.cin / a.cout;
    float s = 0.f;
    for (long r = row0; r < row1; ++r) {
        const long img = r / a.h * a.h;
        const int y = (int)(r - img) + tap / 3 - 1;
        if ((unsigned)y >= (unsigned)a.h) continue;
        for (int x0 = 0; x0 < a.wd; ++x0) {
            const float g = __bfloat162float(a.dout[(r * a.wd + x0) * a.cout + co]);
            const int x = x0 + tap % 3 - 1;
            if (g == 0.f || (unsigned)x >= (unsigned)a.wd) continue;
            const bf16 *v = ci < a.cu ? a.up + (((img >> 1) + (y >> 1)) * (a.wd >> 1) + (x >> 1)) * a.cu + ci
                                      : a.in + ((img + y) * a.wd + x) * (a.cin - a.cu) + (ci - a.cu);
            s = fmaf(g, __bfloat162float(*v), s);
        }
    }
    return s;
}

// Sum of the CTAs' partials: 32 outputs per block, each summed by eight
// threads over eighths of the partials, then those eight in order.  The MMAs also
// multiply the zeros around the images and gradients that are zero; where the other
// factor is infinite or NaN that gives NaN, so a weight whose sum is not finite is
// summed again without them (a diverged step: every weight takes the scalar loop).
__global__ void __launch_bounds__(256) k_wgrad_reduce_split(const __grid_constant__ WgradArgs a, int parts, float *__restrict__ dw,
                                                            float *__restrict__ db) {
    __shared__ float red[8][32];
    const float *__restrict__ part = a.part, *__restrict__ partb = a.partb;
    const int nw = 9 * a.cout * a.cin, cout = a.cout;
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
    const int e = (int)blockIdx.x * 32 + lane;   // weights, then biases
    const int eighth = (parts + 7) / 8, c0 = seg * eighth, c1 = min(parts, c0 + eighth);
    float s = 0.f;
    if (e < nw) {
        for (int c = c0; c < c1; ++c) s += part[(size_t)c * nw + e];
    } else if (e - nw < cout) {
        for (int c = c0; c < c1; ++c) s += partb[(size_t)c * cout + e - nw];
    }
    red[seg][lane] = s;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) s = k ? s + red[k][lane] : red[0][lane];   // (every segment the same sum)
    const bool again = e < nw && !isfinite(s);
    if (__any_sync(0xffffffffu, again)) {   // (the same in the block's eight warps)
        __syncthreads();
        const long rows = (long)a.n * a.h, eighth_r = (rows + 7) / 8;
        if (again) red[seg][lane] = wgrad_scalar(a, e, min(rows, seg * eighth_r), min(rows, (seg + 1) * eighth_r));
        __syncthreads();
        if (again)
            for (int k = 0; k < 8; ++k) s = k ? s + red[k][lane] : red[0][lane];
    }
    if (seg == 0) {
        if (e < nw) dw[e] = s;
        else if (db && e - nw < cout) db[e - nw] = s;
    }
}

}  // namespace

// 16-byte loads of eight channels: channel counts are multiples of 8 and the
// tensors 16-byte aligned; the caller's scalar kernel takes the rest.
bool wgrad_mma_takes(const void *up, int cu, const void *in, int cin, const void *dout, int cout) {
    return cin % 8 == 0 && cu % 8 == 0 && cout % 8 == 0 &&
           (((uintptr_t)in | (uintptr_t)up | (uintptr_t)dout) & 15) == 0;
}

cudaError_t launch_wgrad_mma(const void *up, int cu, const void *in, int cin, const void *dout, int cout, int n, int h, int wd, float *dw,
                             float *dbias, float *scratch, int max_parts, cudaStream_t st) {
    WgradArgs a{};
    a.in = (const bf16 *)in;
    a.up = (const bf16 *)up;
    a.cu = up ? cu : 0;
    a.dout = (const bf16 *)dout;
    a.cin = cin;
    a.cout = cout;
    a.n = n;
    a.h = h;
    a.wd = wd;
    // the widest tile of 64, 32 or 16 pixels that the image fills
    a.tx = wd >= 64 ? 64 : (wd > 16 ? 32 : 16);
    a.ty = WG_PIX / a.tx;
    a.tiles_x = (wd + a.tx - 1) / a.tx;
    a.tiles_y = (h + a.ty - 1) / a.ty;
    a.tiles = n * a.tiles_x * a.tiles_y;
    a.tci = (cin + 15) / 16;
    const int blocks = a.tci * ((cout + 15) / 16);
    // two CTAs per SM over all channel blocks, as many times as keep a CTA to WG_CHAIN
    // tiles; no more partials than the scratch holds (one per 2048 pixels)
    const int fill = (2 * kSMs + blocks - 1) / blocks;
    const long waves = std::max(1l, ((long)a.tiles + (long)fill * WG_CHAIN - 1) / ((long)fill * WG_CHAIN));
    const int parts = (int)std::max(1l, std::min({(long)max_parts, (long)a.tiles, fill * waves}));
    a.per = (a.tiles + parts - 1) / parts;
    const int used = (a.tiles + a.per - 1) / a.per;
    const int nw = 9 * cout * cin;
    a.part = scratch;
    a.partb = scratch + (size_t)used * nw;
    const int smem = 2 * WG_STAGE;
    cudaError_t e = cudaFuncSetAttribute(k_wgrad_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_wgrad_mma<<<dim3((unsigned)used, (unsigned)blocks), WG_WARPS * 32, smem, st>>>(a);
    k_wgrad_reduce_split<<<(unsigned)((nw + cout + 31) / 32), 256, 0, st>>>(a, used, dw, dbias);
    return cudaGetLastError();
}

}  // namespace pp
