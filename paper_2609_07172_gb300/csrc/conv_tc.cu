// 3x3 convolution of the learned warm start on the fifth-generation tensor
// cores: an implicit GEMM with tcgen05.mma (BF16 in, FP32 accumulated in
// tensor memory), operands staged by TMA.
//
// GEMM view: rows = output pixels (a tile of 128 consecutive pixels of one
// sample: 128 of one image row, or 128 / W whole rows when W < 128), columns =
// output channels (N = cout), reduction = (tap, input channel).  For tap
// (dy, dx) and a chunk of KC input channels the A operand of a tile is the
// input box [KC channels] x [the tile's pixels shifted by (dx, dy)]: one
// 4-D TMA load of the NHWC tensor, whose out-of-range coordinates (x = -1,
// x = W, y = -1, y = H) read zeros -- exactly the convolution's zero padding.
// The B operand is the weight slice w[tap][0:cout][c0:c0+KC] (K-major), one
// 3-D TMA load.  KC = 64, 32 or 16 channels make a 128-, 64- or 32-byte
// row, which TMA swizzles into the canonical K-major layout the MMA's shared
// memory descriptors name.
//
// Roles (192 threads): warp 4 issues the TMA loads into a ring of 4 stages (8
// for 16-channel chunks),
// warp 5 issues the MMAs (KC / 16 per stage, M = 128, N = cout, K = 16) into
// one of two TMEM accumulators, warps 0-3 drain an accumulator (tcgen05.ld,
// each warp its 32 TMEM lanes = 32 pixels), add the bias, apply ReLU and
// store BF16 and / or FP32 while the next tile accumulates into the other.
// CTAs are persistent over the tiles.  Every wait on an mbarrier is bounded;
// a wait that runs out sets an error flag (pic_nn_conv_tc_status), ends the
// CTA's loops, waits (bounded) for its own copies and MMAs, and frees its
// tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "internal.h"

namespace pp {

__device__ int g_conv_tc_error;   // 1 + the role whose wait ran out (0: none)

namespace {

typedef __nv_bfloat16 bf16;

constexpr int TC_M = 128;                      // pixels per tile (MMA M)
constexpr int TC_MAX_STAGES = 8;                 // ring slots: 8 for 16-channel chunks (a tile's 9 loads), else 4
constexpr int TC_THREADS = 192;                // warps 0-3 epilogue, 4 TMA, 5 MMA
constexpr unsigned TC_SPIN_LIMIT = 1u << 23;   // try_wait rounds before a wait gives up

struct ConvTCArgs {
    int n, h, wd, cin, cout;
    int kc, nchunks;                 // channels per stage, cin / kc
    int bx, by;                      // tile: bx pixels along x times by rows
    int tiles_x, tiles_y, tiles;
    unsigned a_bytes, b_bytes;       // TMA bytes of one stage
    unsigned stage_bytes;            // a_bytes + b_bytes rounded up to 1024
    unsigned tmem_cols;              // columns of one accumulator (power of two >= 32)
    unsigned idesc;                  // MMA instruction descriptor
    unsigned swz, sbo;               // shared-memory descriptor: layout type, 8-row stride
    const float *bias;
    bf16 *out;
    float *out32;
    int relu;
    int stages;                      // ring slots in use (<= TC_MAX_STAGES)
    // halo variant (k_conv3x3_tc_halo): no-swizzle K-major weights
    const bf16 *up;                  // CAT: channels [0, cu), of half the height and width
    int cu;
    bf16 *pool;                      // 2x2 averages of the output, or null
    unsigned lbo_b;                  // bytes from one 8-channel group of a tap's weights to the next
    unsigned w_bytes;                // all nine taps' weights (resident)
};

// No-swizzle K-major descriptor: 8-row core matrices of 16-byte rows; LBO =
// the step to the next 8 channels (K), SBO = 128 (the next 8 rows follow
// directly), so the start may sit on any 16-byte row.
__device__ __forceinline__ uint64_t smem_desc_plain(unsigned addr, unsigned lbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)(128u >> 4) << 32) | ((uint64_t)1 << 46);
}

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Wait for the completion of the phase with parity `parity`; false if the
// limit ran out or another role gave up (*abort set).
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int *abort) {
    for (unsigned it = 0; it < TC_SPIN_LIMIT; ++it) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 1023u) == 1023u && *abort) return false;
    }
    return false;
}

__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap *map, int c0, int c1, int c2,
                                            unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor (tcgen05): start address >> 4 (bits 0-13),
// leading-dimension byte offset >> 4 (16-29; not used by swizzled K-major
// operands whose K extent per MMA fits one swizzle row), stride-dimension byte
// offset >> 4 (32-45: from one 8-row group to the next), the fixed version
// bit 46, base offset 0 (1024-byte aligned stages), layout type (61-63).
__device__ __forceinline__ uint64_t smem_desc(unsigned addr, unsigned sbo, unsigned swz) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)swz << 61);
}

// One MMA, D (+)= A B, issued by the whole warp under a predicate (one lane's
// `one` is 1), the descriptors' halves apart: the upper words are constants of
// the kernel, the lower ones (start address >> 4) an addition per MMA.  Nothing
// diverges, so the operands stay in uniform registers -- an MMA issued inside a
// one-lane branch, its descriptors rebuilt from scratch, took about 360 cycles
// of the issuing thread and bound the halo kernel (see below).
__device__ __forceinline__ void umma_bf16_lo(unsigned tmem_d, unsigned alo, unsigned ahi, unsigned blo, unsigned bhi,
                                             unsigned idesc, unsigned acc, unsigned one) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "setp.ne.b32 q, %7, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(tmem_d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"(one)
        : "memory");
}
__device__ __forceinline__ unsigned elect_one() {
    unsigned one;
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(one));
    return one;
}
// Arrive on `bar` once every MMA the elected lane issued before has completed.
__device__ __forceinline__ void umma_commit_one(unsigned bar, unsigned one) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar),
        "r"(one)
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float (&v)[16]) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = __uint_as_float(r[e]);
}

__device__ __forceinline__ unsigned pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<unsigned *>(&v);
}

// The two values of a packed BF16 pair.
__device__ __forceinline__ float2 bf2(unsigned w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

__device__ __forceinline__ void tile_origin(const ConvTCArgs &a, int tile, int &nn, int &x0, int &y0) {
    const int tx = tile % a.tiles_x, rest = tile / a.tiles_x;
    x0 = tx * a.bx;
    y0 = (rest % a.tiles_y) * a.by;
    nn = rest / a.tiles_y;
}

__device__ __forceinline__ void give_up(volatile int *abort, int role) {
    *abort = 1;
    atomicCAS(&g_conv_tc_error, 0, 1 + role);
}

__global__ void __launch_bounds__(TC_THREADS, 1)
k_conv3x3_tc(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, const ConvTCArgs a) {
    extern __shared__ __align__(1024) unsigned char dsm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // stages on 1024-byte boundaries (the swizzle atoms), then the barriers
    const unsigned raw = smem_u32(dsm);
    const unsigned pad = (1024u - (raw & 1023u)) & 1023u;
    const unsigned stage0 = raw + pad;
    const int S = a.stages;
    unsigned char *tail = dsm + pad + S * a.stage_bytes;
    const unsigned full0 = smem_u32(tail);                   // [S] TMA bytes landed
    const unsigned empty0 = full0 + 8 * TC_MAX_STAGES;       // [S] stage read by the MMAs
    const unsigned tfull0 = empty0 + 8 * TC_MAX_STAGES;      // [2] accumulator complete
    const unsigned tempty0 = tfull0 + 16;                    // [2] accumulator drained
    const unsigned drain = tempty0 + 16;                     // every MMA of this CTA complete
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(tail + 8 * (2 * TC_MAX_STAGES + 5));
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *never = reinterpret_cast<volatile int *>(tmem_slot + 2);   // stays 0: a wait that ignores *abort
    const unsigned ncols = 2 * a.tmem_cols;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull0 + 8 * b, 1);
            mbar_init(tempty0 + 8 * b, 4 * 32);
        }
        mbar_init(drain, 1);
        *abort = 0;
        *never = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *tmem_slot;
    const int kiters = 9 * a.nchunks;

    if (warp == 4) {
        // ---------------- TMA producer
        if (lane == 0) {
            unsigned it = 0;
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x) {
                int nn, x0, y0;
                tile_origin(a, tile, nn, x0, y0);
                for (int k = 0; k < kiters; ++k, ++it) {
                    const unsigned s = it % S, u = it / S;
                    if (!mbar_wait(empty0 + 8 * s, (u & 1u) ^ 1u, abort)) {
                        give_up(abort, 0);
                        ok = false;
                        break;
                    }
                    const int tap = k / a.nchunks, c0 = (k - tap * a.nchunks) * a.kc;
                    const unsigned sa = stage0 + s * a.stage_bytes;
                    mbar_expect_tx(full0 + 8 * s, a.a_bytes + a.b_bytes);
                    tma_load_4d(sa, &ta, c0, x0 + tap % 3 - 1, y0 + tap / 3 - 1, nn, full0 + 8 * s);
                    tma_load_3d(sa + a.a_bytes, &tb, c0, 0, tap, full0 + 8 * s);
                }
            }
            // the last copies land before the CTA exits (on the normal path
            // the MMAs have consumed them already and these waits return at once)
            const unsigned first = it > (unsigned)S ? it - S : 0u;
            for (unsigned j = first; j < it; ++j)
                if (!mbar_wait(full0 + 8 * (j % S), (j / S) & 1u, never)) give_up(abort, 3);
        }
    } else if (warp == 5) {
        // ---------------- MMA issuer (the whole warp; one lane's MMAs and commits take effect)
        const unsigned one = elect_one();
        unsigned it = 0, tc = 0;
        bool ok = true;
        for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x, ++tc) {
            const unsigned buf = tc & 1u, u = tc >> 1;
            if (!mbar_wait(tempty0 + 8 * buf, (u & 1u) ^ 1u, abort)) {
                give_up(abort, 1);
                break;
            }
            tc_fence_after();
            const unsigned d = tmem + buf * a.tmem_cols;
            for (int k = 0; k < kiters; ++k, ++it) {
                const unsigned s = it % S, us = it / S;
                if (!mbar_wait(full0 + 8 * s, us & 1u, abort)) {
                    give_up(abort, 1);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const unsigned sa = stage0 + s * a.stage_bytes;
                const uint64_t da = smem_desc(sa, a.sbo, a.swz), db = smem_desc(sa + a.a_bytes, a.sbo, a.swz);
                for (int kk = 0; kk < a.kc / 16; ++kk)   // K = 16 BF16 = 32 bytes per MMA
                    umma_bf16_lo(d, (unsigned)da + 2u * kk, (unsigned)(da >> 32), (unsigned)db + 2u * kk,
                                 (unsigned)(db >> 32), a.idesc, (k | kk) != 0 ? 1u : 0u, one);
                umma_commit_one(empty0 + 8 * s, one);   // the stage is free once these MMAs have read it
            }
            if (!ok) break;
            umma_commit_one(tfull0 + 8 * buf, one);     // the tile's accumulator is complete
        }
        umma_commit_one(drain, one);
        if (!mbar_wait(drain, 0, never)) give_up(abort, 4);
    } else {
        // ---------------- epilogue: warp w drains TMEM lanes 32 w .. 32 w + 31
        const int row = threadIdx.x;   // pixel of the tile = TMEM lane
        unsigned tc = 0;
        for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, ++tc) {
            const unsigned buf = tc & 1u, u = tc >> 1;
            if (!mbar_wait(tfull0 + 8 * buf, u & 1u, abort)) {
                give_up(abort, 2);
                break;
            }
            tc_fence_after();
            int nn, x0, y0;
            tile_origin(a, tile, nn, x0, y0);
            const int x = x0 + row % a.bx, y = y0 + row / a.bx;
            const bool valid = y < a.h;
            const size_t p = ((size_t)nn * a.h + (valid ? y : 0)) * a.wd + x;
            const unsigned taddr = tmem + buf * a.tmem_cols + ((unsigned)(warp * 32) << 16);
            for (int c = 0; c < a.cout; c += 16) {
                float v[16];
                tmem_ld16(taddr + (unsigned)c, v);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    float t = v[e] + (a.bias ? a.bias[c + e] : 0.f);
                    v[e] = a.relu ? fmaxf(t, 0.f) : t;
                }
                if (!valid) continue;
                if (a.out) {
                    uint4 *o = reinterpret_cast<uint4 *>(a.out + p * a.cout + c);
                    o[0] = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
                    o[1] = make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]),
                                      pack2(v[14], v[15]));
                }
                if (a.out32) {
                    float4 *o = reinterpret_cast<float4 *>(a.out32 + p * a.cout + c);
#pragma unroll
                    for (int q = 0; q < 4; ++q) o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                }
            }
            tc_fence_before();
            mbar_arrive(tempty0 + 8 * buf);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    }
}

// Halo variant for image rows of 128 pixels or more and small weight sets (the
// full- and half-resolution layers, which are bound by data movement).  A tile
// is 128 pixels of two rows; per chunk of KC channels the four input rows
// y - 1 .. y + 2 over pixels x0 - 1 .. x0 + 128 are staged once, one row of KC
// channels per pixel (32- or 64-byte swizzle), and the nine taps of an output
// row are the same buffer seen from nine start rows, (r + 1 + dy) * 130 + 1 +
// dx: the swizzle is a function of the address bits, so a descriptor may start
// at any pixel of a buffer aligned to the pattern.  All nine taps' weights stay
// resident from the CTA's start.  A tile row then moves 2 * 130 * cin instead
// of 9 * 128 * cin input values.
//
// What bounded it before (clock64 in the roles): the MMA thread, which built
// two 64-bit descriptors per MMA inside a one-lane branch, about 360 cycles
// each with 9 to 18 per row; and the TMA engine, one request per staged row of
// 8 channels (780 to 1560 per output row at about 1.5 cycles).  65 samples of
// 200 x 256: 16 -> 16 channels 114 us, 32 -> 16 169 us.  With uniform issue
// (umma_bf16_lo), whole-pixel rows and two output rows per tile 60 and 77 us
// (three and two CTAs per SM).  What is left: an MMA of N = 16 costs the 32
// cycles of reading its 128 x 16 A operand (24 and 48 us), the staged rows about
// 1.5 cycles each, the bytes 31 and 47 us.
//
// CAT: the input is two tensors, channels [0, cu) from `up`, an image of half
// the height and width upsampled 2x (nearest), the others from `in` -- the
// decoder's concatenation, which is never written.  Four expander warps load
// up's pixels into registers a stage ahead and write each to the two pixels (and
// rows) it covers (32 -> 16 channels on 65 x 200 x 256: 73 us, against 169 for
// the convolution and 265 for writing the concatenation before).  MIX: a chunk holds 16 channels of each, in two buffers of
// 32-byte rows (KC = 32); otherwise a chunk lies in one tensor.
//
// pool: the 2x2 averages of the (BF16) output, from the two rows of the tile.
constexpr int TH_WX = TC_M + 2;                // pixels of a staged row
constexpr int TH_ROWS = 4 * TH_WX;             // staged pixels
constexpr int TH_EXPAND = 128;                 // expander threads (CAT)
constexpr int TH_UPIX = 3 * (TC_M / 2 + 2);    // up's pixels under a tile

template <int KC, bool CAT, bool MIX>
__global__ void __launch_bounds__(TC_THREADS + (CAT ? TH_EXPAND : 0), 1)
k_conv3x3_tc_halo(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, const ConvTCArgs a) {
    extern __shared__ __align__(1024) unsigned char dsm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned raw = smem_u32(dsm);
    const unsigned pad = (1024u - (raw & 1023u)) & 1023u;
    const unsigned wbase = raw + pad;                                  // resident weights
    const unsigned stage0 = wbase + ((a.w_bytes + 1023u) & ~1023u);   // halo tiles
    const int S = a.stages;
    unsigned char *tail = dsm + pad + ((a.w_bytes + 1023u) & ~1023u) + S * a.stage_bytes;
    const unsigned full0 = smem_u32(tail);
    const unsigned empty0 = full0 + 8 * TC_MAX_STAGES;
    const unsigned tfull0 = empty0 + 8 * TC_MAX_STAGES;
    const unsigned tempty0 = tfull0 + 16;
    const unsigned drain = tempty0 + 16;
    const unsigned wbar = drain + 8;                                   // weights landed
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(tail + 8 * (2 * TC_MAX_STAGES + 6));
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *never = reinterpret_cast<volatile int *>(tmem_slot + 2);
    float *bias = reinterpret_cast<float *>(tmem_slot + 4);           // [cout], zeros without a bias
    const unsigned ncols = 4 * a.tmem_cols;      // two sets of two accumulators (the tile's rows)
    const int cgroups = a.cin / 8;               // 8-channel groups per tap of the weights
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8 * s, CAT ? 1 + TH_EXPAND : 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull0 + 8 * b, 1);
            mbar_init(tempty0 + 8 * b, 4 * 32);
        }
        mbar_init(drain, 1);
        mbar_init(wbar, 1);
        *abort = 0;
        *never = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int c = threadIdx.x; c < a.cout; c += blockDim.x) bias[c] = a.bias ? a.bias[c] : 0.f;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *tmem_slot;

    if (warp == 4) {
        // ---------------- TMA producer: the weights once, then the halo tiles
        if (lane == 0) {
            mbar_expect_tx(wbar, a.w_bytes);
            for (int tap = 0; tap < 9; ++tap)
                for (int g = 0; g < cgroups; ++g)
                    tma_load_3d(wbase + (unsigned)(tap * cgroups + g) * a.lbo_b, &tb, 8 * g, 0, tap, wbar);
            unsigned it = 0;
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x) {
                int nn, x0, y0;
                tile_origin(a, tile, nn, x0, y0);
                for (int c = 0; c < a.nchunks; ++c, ++it) {
                    const unsigned s = it % S, u = it / S;
                    if (!mbar_wait(empty0 + 8 * s, (u & 1u) ^ 1u, abort)) {
                        give_up(abort, 0);
                        ok = false;
                        break;
                    }
                    const unsigned sa = stage0 + s * a.stage_bytes;
                    if (CAT && !MIX && c * KC < a.cu) {   // this chunk comes from the expanders alone
                        mbar_arrive(full0 + 8 * s);
                        continue;
                    }
                    mbar_expect_tx(full0 + 8 * s, a.a_bytes);
                    tma_load_4d(MIX ? sa + a.stage_bytes / 2 : sa, &ta, MIX ? 0 : c * KC - a.cu, x0 - 1, y0 - 1, nn,
                                full0 + 8 * s);
                }
            }
            const unsigned first = it > (unsigned)S ? it - S : 0u;
            for (unsigned j = first; j < it; ++j)
                if (!mbar_wait(full0 + 8 * (j % S), (j / S) & 1u, never)) give_up(abort, 3);
            if (!mbar_wait(wbar, 0, never)) give_up(abort, 3);
        }
    } else if (warp == 5) {
        // ---------------- MMA issuer (the whole warp; one lane's MMAs and commits take effect)
        const unsigned one = elect_one();
        unsigned it = 0, tc = 0;
        bool ok = mbar_wait(wbar, 0, abort);
        if (!ok) give_up(abort, 1);
        tc_fence_after();
        for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x, ++tc) {
            const unsigned buf = tc & 1u, u = tc >> 1;
            if (!mbar_wait(tempty0 + 8 * buf, (u & 1u) ^ 1u, abort)) {
                give_up(abort, 1);
                break;
            }
            tc_fence_after();
            const unsigned d = tmem + 2u * buf * a.tmem_cols;
            for (int c = 0; c < a.nchunks; ++c, ++it) {
                const unsigned s = it % S, us = it / S;
                if (!mbar_wait(full0 + 8 * s, us & 1u, abort)) {
                    give_up(abort, 1);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const unsigned sa = stage0 + s * a.stage_bytes;
                constexpr int ROW = MIX ? 32 : KC * 2;                       // bytes of a staged pixel
                const unsigned kstep = MIX ? a.stage_bytes / 2 >> 4 : 2u;    // the next 16 channels, 16-byte units
                const uint64_t da = smem_desc(sa, a.sbo, a.swz), db = smem_desc_plain(wbase, a.lbo_b);
                const unsigned alo = (unsigned)da, ahi = (unsigned)(da >> 32), bhi = (unsigned)(db >> 32);
                const unsigned bstep = 2u * a.lbo_b >> 4, btap = (unsigned)cgroups * a.lbo_b >> 4;
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    const unsigned ar = alo + (unsigned)r * (TH_WX * ROW / 16), dr = d + (unsigned)r * a.tmem_cols;
                    unsigned blo = (unsigned)db + (unsigned)c * (KC / 16) * bstep;
#pragma unroll
                    for (int tap = 0; tap < 9; ++tap, blo += btap)
#pragma unroll
                        for (int kk = 0; kk < KC / 16; ++kk)   // K = 16 BF16 = 32 bytes per MMA
                            umma_bf16_lo(dr, ar + ((tap / 3) * TH_WX + tap % 3) * (ROW / 16) + kk * kstep, ahi,
                                         blo + kk * bstep, bhi, a.idesc, (c | tap | kk) != 0 ? 1u : 0u, one);
                }
                umma_commit_one(empty0 + 8 * s, one);
            }
            if (!ok) break;
            umma_commit_one(tfull0 + 8 * buf, one);
        }
        umma_commit_one(drain, one);
        if (!mbar_wait(drain, 0, never)) give_up(abort, 4);
    } else if (warp < 4) {
        // ---------------- epilogue: warp w drains TMEM lanes 32 w .. 32 w + 31 (pixels) of the tile's two rows
        const int row = threadIdx.x;
        unsigned tc = 0;
        for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, ++tc) {
            const unsigned buf = tc & 1u, u = tc >> 1;
            int nn, x0, y0;
            tile_origin(a, tile, nn, x0, y0);
            const size_t p = ((size_t)nn * a.h + y0) * a.wd + x0 + row;
            const size_t pp = (((size_t)nn * (a.h >> 1) + (y0 >> 1)) * a.wd + x0 + row) >> 1;
            if (!mbar_wait(tfull0 + 8 * buf, u & 1u, abort)) {
                give_up(abort, 2);
                break;
            }
            tc_fence_after();
            const unsigned taddr = tmem + 2u * buf * a.tmem_cols + ((unsigned)(warp * 32) << 16);
            for (int c = 0; c < a.cout; c += 16) {
                unsigned q[2][8];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    float v[16];
                    tmem_ld16(taddr + (unsigned)r * a.tmem_cols + (unsigned)c, v);
                    const bool valid = y0 + r < a.h;
#pragma unroll
                    for (int e = 0; e < 16; e += 4) {
                        const float4 b = *reinterpret_cast<const float4 *>(bias + c + e);
                        v[e] += b.x, v[e + 1] += b.y, v[e + 2] += b.z, v[e + 3] += b.w;
                    }
                    if (a.relu)
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = fmaxf(v[e], 0.f);
#pragma unroll
                    for (int e = 0; e < 8; ++e) q[r][e] = pack2(v[2 * e], v[2 * e + 1]);
                    const size_t o = (p + (size_t)r * a.wd) * a.cout + c;
                    if (a.out && valid) {
                        uint4 *w = reinterpret_cast<uint4 *>(a.out + o);
                        w[0] = make_uint4(q[r][0], q[r][1], q[r][2], q[r][3]);
                        w[1] = make_uint4(q[r][4], q[r][5], q[r][6], q[r][7]);
                    }
                    if (a.out32 && valid) {
                        float4 *w = reinterpret_cast<float4 *>(a.out32 + o);
#pragma unroll
                        for (int e = 0; e < 4; ++e) w[e] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                    }
                }
                if (a.pool) {   // (h even) this pixel and its right neighbour, both rows; even lanes store
                    unsigned m[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const unsigned n0 = __shfl_down_sync(0xffffffffu, q[0][e], 1);
                        const unsigned n1 = __shfl_down_sync(0xffffffffu, q[1][e], 1);
                        const float2 f0 = bf2(q[0][e]), g0 = bf2(n0), f1 = bf2(q[1][e]), g1 = bf2(n1);
                        m[e] = pack2(0.25f * (f0.x + g0.x + f1.x + g1.x), 0.25f * (f0.y + g0.y + f1.y + g1.y));
                    }
                    if ((lane & 1) == 0) {
                        uint4 *w = reinterpret_cast<uint4 *>(a.pool + pp * a.cout + c);
                        w[0] = make_uint4(m[0], m[1], m[2], m[3]);
                        w[1] = make_uint4(m[4], m[5], m[6], m[7]);
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(tempty0 + 8 * buf);
        }
    } else if (CAT) {
        // ---------------- expanders: up's channels of a chunk, each pixel to the pixels and rows it covers
        const int t = (int)threadIdx.x - TC_THREADS;
        constexpr int G = (MIX ? 16 : KC) / 8;                        // 16-byte groups of a pixel
        constexpr int NP = (TH_UPIX * G + TH_EXPAND - 1) / TH_EXPAND;  // pieces per thread
        constexpr int UW = TC_M / 2 + 2;
        constexpr int ROW = 16 * G;
        const int uw = a.wd >> 1, uh = a.h >> 1;
        uint4 v[NP];
        auto load = [&](int tile, int c) {
            int nn, x0, y0;
            tile_origin(a, tile, nn, x0, y0);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const int e = t + j * TH_EXPAND, g = e % G, px = e / G;
                const int sy = px / UW, y = (y0 >> 1) - 1 + sy, x = (x0 >> 1) - 1 + (px - sy * UW);
                v[j] = make_uint4(0u, 0u, 0u, 0u);
                if (px < TH_UPIX && (unsigned)y < (unsigned)uh && (unsigned)x < (unsigned)uw)
                    v[j] = __ldg(reinterpret_cast<const uint4 *>(
                        a.up + (((size_t)nn * uh + y) * uw + x) * a.cu + (MIX ? 0 : c * KC) + 8 * g));
            }
        };
        unsigned it = 0;
        bool ok = true;
        if ((int)blockIdx.x < a.tiles) load(blockIdx.x, 0);
        for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x) {
            for (int c = 0; c < a.nchunks; ++c, ++it) {
                const unsigned s = it % S, u = it / S;
                if (!mbar_wait(empty0 + 8 * s, (u & 1u) ^ 1u, abort)) {
                    give_up(abort, 0);
                    ok = false;
                    break;
                }
                if (MIX || c * KC < a.cu) {
                    const unsigned sa = stage0 + s * a.stage_bytes;
#pragma unroll
                    for (int j = 0; j < NP; ++j) {
                        const int e = t + j * TH_EXPAND, g = e % G, px = e / G;
                        const int sy = px / UW, sx = px - sy * UW;
                        if (px >= TH_UPIX) continue;
#pragma unroll
                        for (int d = 0; d < 4; ++d) {
                            // staged rows of up's row sy: 0; 1, 2; 3 -- staged pixels of column sx: 2 sx - 1, 2 sx
                            const int r = sy == 0 ? 0 : (sy == 2 ? 3 : 1 + (d >> 1)), q = 2 * sx - 1 + (d & 1);
                            if ((d >> 1 && sy != 1) || q < 0 || q >= TH_WX) continue;
                            const unsigned pix = (unsigned)(r * TH_WX + q);
                            const unsigned sw = ROW == 32 ? (pix >> 2) & 1u : (pix >> 1) & 3u;   // swizzled 16-byte group
                            const unsigned at = sa + pix * ROW + (((unsigned)g ^ sw) << 4);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v[j].x), "r"(v[j].y),
                                         "r"(v[j].z), "r"(v[j].w)
                                         : "memory");
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // to the MMA's proxy
                }
                mbar_arrive(full0 + 8 * s);
                // the next chunk's pixels, in flight while the stage is used
                int c1 = c + 1, t1 = tile;
                if (c1 == a.nchunks) c1 = 0, t1 += gridDim.x;
                if (t1 < a.tiles && (MIX || c1 * KC < a.cu)) load(t1, c1);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    }
}

}  // namespace

// ------------------------------------------------------------------ host side
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

std::mutex g_tc_mutex;
EncodeTiledFn g_encode = nullptr;
bool g_encode_tried = false;

EncodeTiledFn encoder() {
    std::lock_guard<std::mutex> lock(g_tc_mutex);
    if (!g_encode_tried) {
        g_encode_tried = true;
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = (EncodeTiledFn)f;
        else
            cudaGetLastError();
    }
    return g_encode;
}

}  // namespace

namespace {

// Per device: SM count, shared memory per SM, and each kernel's registers per
// thread (fixed properties, queried once).
struct TCDeviceInfo {
    bool valid = false;
    int sms = 0, smem_sm = 0;
    int regs[5] = {0, 0, 0, 0, 0};   // kTCKernels
};
TCDeviceInfo g_tc_info[64];
// the generic variant, then the halo variants of 16 and 32 channels per chunk,
// of two inputs, and of two inputs mixed in a chunk
const void *const kTCKernels[5] = {
    (const void *)k_conv3x3_tc, (const void *)k_conv3x3_tc_halo<16, false, false>,
    (const void *)k_conv3x3_tc_halo<32, false, false>, (const void *)k_conv3x3_tc_halo<32, true, false>,
    (const void *)k_conv3x3_tc_halo<32, true, true>};

int conv_tc_occupancy(int which, int threads, size_t smem, unsigned tmem_cols_per_cta, int *grid_cap) {
    int dev = 0;
    PP_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        set_error("device ordinal %d beyond 64", dev);
        return PIC_POISSON_EINVAL;
    }
    TCDeviceInfo info;
    {
        std::lock_guard<std::mutex> lock(g_tc_mutex);
        info = g_tc_info[dev];
    }
    if (!info.valid) {
        PP_CUDA(cudaDeviceGetAttribute(&info.sms, cudaDevAttrMultiProcessorCount, dev));
        PP_CUDA(cudaDeviceGetAttribute(&info.smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
        for (int k = 0; k < 5; ++k) {
            cudaFuncAttributes fa;
            PP_CUDA(cudaFuncGetAttributes(&fa, kTCKernels[k]));
            info.regs[k] = fa.numRegs;
        }
        info.valid = true;
        std::lock_guard<std::mutex> lock(g_tc_mutex);
        g_tc_info[dev] = info;
    }
    // CTAs per SM: shared memory (1 KB reserved per CTA), registers, threads,
    // and tensor memory (512 columns per SM: no CTA waits for an allocation)
    const int regs = std::max(1, (info.regs[which] + 7) & ~7) * threads;
    const int occ = std::min({(int)(info.smem_sm / (smem + 1024)), 65536 / regs, 2048 / threads, 32,
                              (int)(512u / tmem_cols_per_cta)});
    *grid_cap = info.sms * std::max(1, occ);
    return PIC_POISSON_OK;
}

// (the kernels' ceiling, not this launch's size: other layers set it too, on other
// threads.  The most that a layer takes is 149 KB: 32 mixed channels to 80.)
constexpr size_t CONV_MAX_SMEM = 200 * 1024;
int set_smem(const void *kernel, size_t smem) {
    if (smem > CONV_MAX_SMEM) {
        set_error("conv3x3 (tcgen05): %zu bytes of shared memory, at most %zu", smem, CONV_MAX_SMEM);
        return PIC_POISSON_EINVAL;
    }
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CONV_MAX_SMEM);
    if (e == cudaSuccess)   // all of the SM's unified memory as shared memory, so several CTAs fit
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) {
        set_error("conv3x3 (tcgen05): %s", cudaGetErrorString(e));
        return PIC_POISSON_ECUDA;
    }
    return PIC_POISSON_OK;
}

// The halo variant's operands: swizzled 4-D boxes of a chunk's channels x 130
// pixels x 4 rows of the input, no-swizzle 3-D boxes of 8 channels x cout of
// each tap's weights.  1 when two inputs do not split into its chunks.
int launch_halo(ConvTCArgs a, const void *in, const void *w, EncodeTiledFn enc, cudaStream_t st) {
    a.kc = a.cin % 32 == 0 ? 32 : 16;
    a.nchunks = a.cin / a.kc;
    const bool cat = a.up != nullptr, mix = cat && a.cin == 32 && a.cu == 16;
    if (cat && !mix && (a.kc != 32 || a.cu % 32)) return 1;
    const int which = mix ? 4 : (cat ? 3 : (a.kc == 32 ? 2 : 1));
    const int tma_kc = mix ? 16 : a.kc;               // channels of a TMA box
    a.by = 2;
    a.tiles_y = (a.h + 1) / 2;
    const long tiles = (long)a.n * a.tiles_y * a.tiles_x;
    a.tiles = (int)tiles;
    a.a_bytes = (unsigned)(TH_ROWS * tma_kc * 2);      // TMA bytes of one chunk
    const unsigned buf_bytes = (a.a_bytes + 1023u) & ~1023u;
    a.stage_bytes = mix ? 2 * buf_bytes : buf_bytes;
    a.swz = tma_kc == 32 ? 4u : 6u;                   // 64- or 32-byte pixel rows
    a.sbo = 8u * (unsigned)(tma_kc * 2);
    a.lbo_b = (unsigned)a.cout * 16u;
    a.w_bytes = 9u * (unsigned)a.cout * (unsigned)a.cin * 2u;
    a.stages = a.kc == 16 ? 4 : 3;
    CUtensorMap ta, tb;
    const int cs = a.cin - a.cu;
    const cuuint64_t gdim_a[4] = {(cuuint64_t)cs, (cuuint64_t)a.wd, (cuuint64_t)a.h, (cuuint64_t)a.n};
    const cuuint64_t gstr_a[3] = {(cuuint64_t)cs * 2, (cuuint64_t)cs * 2 * a.wd, (cuuint64_t)cs * 2 * a.wd * a.h};
    const cuuint32_t box_a[4] = {(cuuint32_t)tma_kc, (cuuint32_t)TH_WX, 4, 1};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(in), gdim_a, gstr_a, box_a, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, tma_kc == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return 1;
    const cuuint64_t gdim_b[3] = {(cuuint64_t)a.cin, (cuuint64_t)a.cout, 9};
    const cuuint64_t gstr_b[2] = {(cuuint64_t)a.cin * 2, (cuuint64_t)a.cin * 2 * a.cout};
    const cuuint32_t box_b[3] = {8, (cuuint32_t)a.cout, 1};
    if (enc(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(w), gdim_b, gstr_b, box_b, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return 1;
    const size_t smem = 1024 + ((a.w_bytes + 1023u) & ~1023u) + (size_t)a.stages * a.stage_bytes +
                        8 * (2 * TC_MAX_STAGES + 6) + 16 + 128 * sizeof(float);
    int rc = set_smem(kTCKernels[which], smem);
    if (rc) return rc;
    const int threads = TC_THREADS + (cat ? TH_EXPAND : 0);
    int cap = 0;
    rc = conv_tc_occupancy(which, threads, smem, 4u * a.tmem_cols, &cap);
    if (rc) return rc;
    const int grid = std::min(a.tiles, cap);
    switch (which) {
    case 1: k_conv3x3_tc_halo<16, false, false><<<grid, threads, smem, st>>>(ta, tb, a); break;
    case 2: k_conv3x3_tc_halo<32, false, false><<<grid, threads, smem, st>>>(ta, tb, a); break;
    case 3: k_conv3x3_tc_halo<32, true, false><<<grid, threads, smem, st>>>(ta, tb, a); break;
    default: k_conv3x3_tc_halo<32, true, true><<<grid, threads, smem, st>>>(ta, tb, a); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("conv3x3 (tcgen05, halo) launch failed: %s", cudaGetErrorString(e));
        return PIC_POISSON_ECUDA;
    }
    return PIC_POISSON_OK;
}

// Tile shape of a W-wide image: 128 pixels of a row (W a multiple of 128) or
// 128 / W whole rows (W = 16, 32 or 64); 0 when the tensor-core path does not
// take this width.
int conv_tc_tile_x(int wd) {
    if (wd % TC_M == 0) return TC_M;
    if (wd == 16 || wd == 32 || wd == 64) return wd;
    return 0;
}

}  // namespace

// The tensor-core convolution, or 1 when it does not apply (the caller then
// runs the mma.sync kernel): cout a multiple of 16 up to 128, cin a multiple of
// 16, a tileable width, 16-byte aligned tensors and the driver's tensor-map
// encoder available.  0 on success, a PIC_POISSON_* error otherwise.
// up: the first cu of the cin channels come from it (half the height and
// width, upsampled 2x), the others from in; pool: also the 2x2 averages of the
// output.  Only the halo variant takes these (1 otherwise).
int launch_conv3x3_tc(const void *up, int cu, const void *in, int cin, const void *w, const float *bias, void *out,
                      float *out32, void *pool, int cout, int n, int h, int wd, int relu, cudaStream_t st) {
    const int bx = conv_tc_tile_x(wd);
    if (!bx || cout % 16 || cout > 128 || cin % 16 || ((uintptr_t)in & 15) || ((uintptr_t)w & 15) ||
        ((uintptr_t)out & 15) || ((uintptr_t)out32 & 15) || ((uintptr_t)up & 15) || ((uintptr_t)pool & 15))
        return 1;
    // halo variant: rows of 128 pixels and weights small enough to stay resident
    const unsigned w_all = 9u * (unsigned)cout * (unsigned)cin * 2u;
    const bool halo = bx == TC_M && w_all <= 48u * 1024u;
    if ((up || pool) && (!halo || h % 2)) return 1;
    EncodeTiledFn enc = encoder();
    if (!enc) return 1;
    ConvTCArgs a{};
    a.n = n;
    a.h = h;
    a.wd = wd;
    a.cin = cin;
    a.cout = cout;
    a.kc = cin % 64 == 0 ? 64 : (cin % 32 == 0 ? 32 : 16);
    a.nchunks = cin / a.kc;
    a.bx = bx;
    a.by = TC_M / bx;
    a.tiles_x = wd / bx;
    a.tiles_y = (h + a.by - 1) / a.by;
    const long tiles = (long)n * a.tiles_y * a.tiles_x;
    if (tiles > 0x7fffffffL) return 1;
    a.tiles = (int)tiles;
    a.a_bytes = (unsigned)(TC_M * a.kc * 2);
    a.b_bytes = (unsigned)(cout * a.kc * 2);
    a.stage_bytes = (a.a_bytes + a.b_bytes + 1023u) & ~1023u;
    a.tmem_cols = cout <= 32 ? 32u : (cout <= 64 ? 64u : 128u);
    // kind::f16 instruction descriptor: FP32 accumulator (bits 4-5 = 1), BF16 A
    // and B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at
    // bits 17-22, M >> 4 at bits 24-28
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(cout >> 3) << 17) | ((unsigned)(TC_M >> 4) << 24);
    // rows of kc BF16 = 32, 64 or 128 bytes: the matching swizzle, 8 rows per group
    a.swz = a.kc == 64 ? 2u : (a.kc == 32 ? 4u : 6u);
    a.sbo = 8u * (unsigned)(a.kc * 2);
    a.bias = bias;
    a.out = (bf16 *)out;
    a.out32 = out32;
    a.relu = relu;
    a.up = (const bf16 *)up;
    a.cu = up ? cu : 0;
    a.pool = (bf16 *)pool;
    if (halo) return launch_halo(a, in, w, enc, st);
    const CUtensorMapSwizzle sw = a.kc == 64 ? CU_TENSOR_MAP_SWIZZLE_128B
                                             : (a.kc == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    // activations: (c, x, y, n), zero fill outside
    CUtensorMap ta, tb;
    const cuuint64_t gdim_a[4] = {(cuuint64_t)cin, (cuuint64_t)wd, (cuuint64_t)h, (cuuint64_t)n};
    const cuuint64_t gstr_a[3] = {(cuuint64_t)cin * 2, (cuuint64_t)cin * 2 * wd, (cuuint64_t)cin * 2 * wd * h};
    const cuuint32_t box_a[4] = {(cuuint32_t)a.kc, (cuuint32_t)a.bx, (cuuint32_t)a.by, 1};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(in), gdim_a, gstr_a, box_a, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return 1;
    // weights [tap][cout][cin]: (c, co, tap)
    const cuuint64_t gdim_b[3] = {(cuuint64_t)cin, (cuuint64_t)cout, 9};
    const cuuint64_t gstr_b[2] = {(cuuint64_t)cin * 2, (cuuint64_t)cin * 2 * cout};
    const cuuint32_t box_b[3] = {(cuuint32_t)a.kc, (cuuint32_t)cout, 1};
    if (enc(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(w), gdim_b, gstr_b, box_b, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return 1;
    a.stages = a.kc == 16 ? 8 : 4;
    const size_t smem = 1024 + (size_t)a.stages * a.stage_bytes + 8 * (2 * TC_MAX_STAGES + 5) + 16;
    int rc = set_smem((const void *)k_conv3x3_tc, smem);
    if (rc) return rc;
    int cap = 0;
    rc = conv_tc_occupancy(0, TC_THREADS, smem, 2u * a.tmem_cols, &cap);
    if (rc) return rc;
    const int grid = std::min(a.tiles, cap);
    k_conv3x3_tc<<<grid, TC_THREADS, smem, st>>>(ta, tb, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("conv3x3 (tcgen05) launch failed: %s", cudaGetErrorString(e));
        return PIC_POISSON_ECUDA;
    }
    return PIC_POISSON_OK;
}

}  // namespace pp

// Status of the tensor-core convolution's bounded waits: 0 if none ran out
// since the last call, else 1 + the role (0 TMA, 1 MMA, 2 epilogue, 3 copy
// drain, 4 MMA drain) of the first that did; the flag is then cleared.
extern "C" int pic_nn_conv_tc_status(int *status) {
    pp::clear_error();
    if (!status) {
        pp::set_error("status is NULL");
        return PIC_POISSON_EINVAL;
    }
    int v = 0, zero = 0;
    PP_CUDA(cudaMemcpyFromSymbol(&v, pp::g_conv_tc_error, sizeof(int)));
    PP_CUDA(cudaMemcpyToSymbol(pp::g_conv_tc_error, &zero, sizeof(int)));
    *status = v;
    return PIC_POISSON_OK;
}
