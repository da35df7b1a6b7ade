// V-cycles in shared memory, one cluster per azimuthal mode: the lower levels of a
// hierarchy, all levels of a small one, or its whole solve.
//
// The modes are independent problems in (z, r).  Below a few hundred thousand
// entries a level kernel runs for 2 to 4 us whatever its size -- its launch and
// one trip through L2 -- and a V-cycle is 20 to 40 of them in a row.  Here a
// cluster of 1 to 8 blocks holds one mode's levels, from some level down to the
// exact solve of the coarsest, in its blocks' shared memory for whole V-cycles:
// each block owns the same range of rows (z) of every level and keeps a copy of
// the row next to it on either side, which its neighbours write when they write
// their own; a block barrier (some 80 cycles) or cluster barrier (500 cycles)
// takes the place of the end of a launch.  Every operation is the level kernels',
// in their order, so the results are theirs bit for bit.  An FP64 problem all of
// whose clusters are resident at a time is solved by one cooperative launch: the
// only word between clusters is the residual norm, added up once per cycle.
//
// Rows are stored by parity of i, [k][even cells | odd cells]: a half-sweep's
// reads and writes are then unit-stride (in cell order they are two apart, a
// two-way bank conflict on each 16-byte access).
//
// Bound by the latency of dependent steps (a half-sweep some 850 cycles in FP64,
// 290 in FP32, plus the barrier): levels of one cell per thread keep their
// coefficients in registers, and the level's description is read from shared
// memory.  Solves in one graph, us, by launches only (local_bottom = -1) / with the
// lower levels here (DEEP_MAX_WHOLE = 0) / as chosen: FP64 32 x 16 x 32 556 / 472 /
// 302, 90 x 32 x 70 528 / 530 / 342, 128 x 64 x 64 1,011 / 888 / 625, 152 x 32 x 90 (only
// the lower levels fit) 677 / 628; mixed 64 x 64 x 64 814 / 455 / 346, 128 x 64 x 96 876 /
// 578 / 467, 96 x 128 x 96 973 / 681 / 517, 192 x 32 x 192 1,182 / 788 / 631 us.
#include <algorithm>

#include "coarse.h"
#include "fastdiv.h"
#include "fixed.h"
#include "internal.h"

namespace pp {
namespace {

template <class T> __device__ __forceinline__ V2<T> mk(T x, T y) {
    V2<T> v;
    v.x = x;
    v.y = y;
    return v;
}

__device__ __forceinline__ int row_class(int k, int nz, int ncls) {
    return k == 0 ? 0 : (k == nz - 1 ? ncls - 1 : 1);
}

// Address of the same shared variable in block `rank` of the cluster.
template <class P> __device__ __forceinline__ P *peer(P *p, int rank) {
    unsigned long long o;
    asm("mapa.u64 %0, %1, %2;" : "=l"(o) : "l"((unsigned long long)p), "r"(rank));
    return reinterpret_cast<P *>(o);
}
__device__ __forceinline__ void cluster_sync(int C) {
    if (C == 1) {
        __syncthreads();
        return;
    }
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
template <int B> __device__ __forceinline__ void cp_async_bytes(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(B) : "memory");
}

// Tables of one smoothed level in shared memory, [ncls][nr] by parity of i like
// the rows, [nr] likewise.  Binary64: real part from hz .., imaginary part from
// the coefficients of fixed.h.
template <class T> struct Tab {
    T *hz, *hw, *he, *dg, *iv, *cz, *cw, *ce;
    int4 *hzw, *rzw;
    int2 *hev, *rdg, *rev;
};
template <class T> __host__ __device__ inline size_t tab_bytes(int nr, int ncls) {
    const size_t n = (size_t)ncls * nr;
    return sizeof(T) == 8 ? n * (5 * 8 + 16 + 8 + 8) + (size_t)nr * (3 * 8 + 16 + 8) : n * 5 * 4 + (size_t)nr * 3 * 4;
}
template <class T> __device__ __forceinline__ Tab<T> tab_of(unsigned char *p, int nr, int ncls) {
    const size_t n = (size_t)ncls * nr;
    Tab<T> t{};
    if constexpr (sizeof(T) == 8) {   // 16-byte entries first
        t.hzw = (int4 *)p;
        t.rzw = t.hzw + n;
        t.hev = (int2 *)(t.rzw + nr);
        t.rdg = t.hev + n;
        t.rev = t.rdg + n;
        p = (unsigned char *)(t.rev + nr);
    }
    t.hz = (T *)p;
    t.hw = t.hz + n;
    t.he = t.hw + n;
    t.dg = t.he + n;
    t.iv = t.dg + n;
    t.cz = t.iv + n;
    t.cw = t.cz + nr;
    t.ce = t.cw + nr;
    return t;
}

// One smoothed level as the block sees it, in shared memory (the kernel's argument
// indexed by a level costs a constant-cache miss or two per field and phase).
struct alignas(16) Lv {
    int nr, hr, nz, ncls;
    int row0, rows, before, rq;   // this block's rows; rows of the block before
    unsigned u, bh, b, tab;       // offsets; row 0 of u has a row of the blocks next to it on either side
    unsigned rhr, rnr;
    int fz, fr;
};

// What the functions below share: the kernel's argument, its shared memory and
// this block's share of the rows.
template <class T> struct Ctx {
    const DeepArg<T> &A;
    unsigned char *sm, *smb, *sma;   // own shared memory, that of the blocks before and after (or null)
    const Lv *lv;
    const int *own;                  // [ncz] of a coarsest row: block << 16 | row there
    int2 *ecol;                      // exponents of the columns of the exact solve
    unsigned rw;                     // reciprocal of this block's columns of the exact solve (fdiv)
    int C, rank, m, z0, z1, zb;      // coarsest rows [z0, z1) of this block, rows of the block before

    __device__ void sync() const { cluster_sync(C); }
    // v at row kl, place e of the array at offset `at` (row 0) with rows of nr, and in the
    // halo rows of the blocks next to this one.
    __device__ __forceinline__ void put(unsigned at, int kl, int e, int nr, int rows, int before, V2<T> v) const {
        const unsigned d = at + (unsigned)e * (unsigned)sizeof(V2<T>);
        const int w = nr * (int)sizeof(V2<T>);
        *(V2<T> *)(sm + (d + (unsigned)(kl * w))) = v;
        if (C > 1) {
            if (kl == 0 && smb) *(V2<T> *)(smb + (d + (unsigned)(before * w))) = v;
            if (kl == rows - 1 && sma) *(V2<T> *)(sma + (d - (unsigned)w)) = v;
        }
    }
};
__device__ __forceinline__ int pos(int i, int hr) { return (i & 1) * hr + (i >> 1); }

// One cell's share of a half-sweep: coefficients, b_hat and place.
template <class T> struct Cell {
    T hz, hw, he;
    int4 zw;
    int2 ev;
    V2<T> b;
    bool w, e;                    // has a west, an east neighbour
};
template <class T> __device__ __forceinline__ Cell<T> cell_of(const Tab<T> &t, const V2<T> *bh, int k, int o, int p, int ii,
                                                             int nr, int hr, int nz, int ncls) {
    const int e = p * hr + ii, tb = row_class(k, nz, ncls) * nr + e;
    Cell<T> c;
    c.hz = t.hz[tb];
    c.hw = t.hw[tb];
    c.he = t.he[tb];
    if constexpr (sizeof(T) == 8) {
        c.zw = t.hzw[tb];
        c.ev = t.hev[tb];
    }
    c.b = bh[o + e];
    c.w = 2 * ii + p > 0;
    c.e = 2 * ii + p + 1 < nr;
    return c;
}
template <class T> __device__ __forceinline__ V2<T> update(const Cell<T> &c, const V2<T> *u, int o, int p, int ii, int nr, int hr) {
    const V2<T> zero = mk<T>(0, 0), *r = u + o + p * hr + ii, *x = u + o + (1 - p) * hr + ii + p;
    const V2<T> us = *(r - nr), un = r[nr], uw = c.w ? *(x - 1) : zero, ue = c.e ? *x : zero;
    V2<T> v;
    v.x = fma(c.he, ue.x, fma(c.hw, uw.x, fma(c.hz, us.x + un.x, c.b.x)));
    if constexpr (sizeof(T) == 8) v.y = fx_update<true>(c.b.y, us.y, un.y, uw.y, ue.y, c.zw, c.ev);
    else v.y = fma(c.he, ue.y, fma(c.hw, uw.y, fma(c.hz, us.y + un.y, c.b.y)));
    return v;
}

// n red-black sweeps on level l.  With a cell of each colour per thread at most,
// its coefficients and b_hat stay in registers.
template <class T> __device__ __forceinline__ void sweeps(const Ctx<T> &X, int l, int n, bool skip_first_red) {
    const Lv v = X.lv[l];
    const V2<T> *u = (const V2<T> *)(X.sm + v.u), *bh = (const V2<T> *)(X.sm + v.bh);
    const Tab<T> t = tab_of<T>(X.sm + v.tab, v.nr, v.ncls);
    const int cells = v.rows * v.hr;
    if (cells <= DEEP_THREADS) {
        const bool on = (int)threadIdx.x < cells;
        const int c = on ? (int)threadIdx.x : 0;
        const int kl = (int)fdiv((unsigned)c, (unsigned)v.hr, v.rhr), ii = c - kl * v.hr, k = v.row0 + kl;
        const int p = k & 1, o = kl * v.nr;
        const Cell<T> cr = cell_of<T>(t, bh, k, o, p, ii, v.nr, v.hr, v.nz, v.ncls);
        const Cell<T> cb = cell_of<T>(t, bh, k, o, 1 - p, ii, v.nr, v.hr, v.nz, v.ncls);
        for (int s = 0; s < n; ++s) {
            if (s > 0 || !skip_first_red) {
                if (on) X.put(v.u, kl, p * v.hr + ii, v.nr, v.rows, v.before, update<T>(cr, u, o, p, ii, v.nr, v.hr));
                X.sync();
            }
            if (on) X.put(v.u, kl, (1 - p) * v.hr + ii, v.nr, v.rows, v.before, update<T>(cb, u, o, 1 - p, ii, v.nr, v.hr));
            X.sync();
        }
        return;
    }
    for (int s = skip_first_red ? 1 : 0; s < 2 * n; ++s) {
        for (int c = threadIdx.x; c < cells; c += DEEP_THREADS) {
            const int kl = (int)fdiv((unsigned)c, (unsigned)v.hr, v.rhr), ii = c - kl * v.hr, k = v.row0 + kl;
            const int p = (k + s) & 1, o = kl * v.nr;
            const Cell<T> cc = cell_of<T>(t, bh, k, o, p, ii, v.nr, v.hr, v.nz, v.ncls);
            X.put(v.u, kl, p * v.hr + ii, v.nr, v.rows, v.before, update<T>(cc, u, o, p, ii, v.nr, v.hr));
        }
        X.sync();
    }
}

// b - A u at place (p, ii) of row kl (as residual_at in mg.cu).
template <class T>
__device__ __forceinline__ V2<T> residual(const Lv &v, const Tab<T> &t, const V2<T> *u, const V2<T> *b, const V2<T> *bg, unsigned nm,
                                          int m, int kl, int p, int ii) {
    const int k = v.row0 + kl, o = kl * v.nr, e = p * v.hr + ii, i = 2 * ii + p;
    const V2<T> zero = mk<T>(0, 0), *r = u + o + e, *x = u + o + (1 - p) * v.hr + ii + p;
    const V2<T> us = *(r - v.nr), un = r[v.nr], uw = i > 0 ? *(x - 1) : zero, ue = i + 1 < v.nr ? *x : zero, uc = *r;
    const V2<T> bv = bg ? bg[((unsigned)k * (unsigned)v.nr + (unsigned)i) * nm + (unsigned)m] : b[o + e];
    const int tb = row_class(k, v.nz, v.ncls) * v.nr + e;
    const T cz = t.cz[e], cw = t.cw[e], ce = t.ce[e], d = t.dg[tb];
    V2<T> q;
    q.x = fma(-d, uc.x, fma(ce, ue.x, fma(cw, uw.x, fma(cz, us.x + un.x, bv.x))));
    if constexpr (sizeof(T) == 8) {
        const int4 zw = t.rzw[e];
        q.y = fx_residual<true>(bv.y, us.y, un.y, uw.y, ue.y, uc.y, make_int2(zw.x, zw.y), make_int2(zw.z, zw.w), t.rev[e],
                          t.rdg[tb], v.rq);
    } else {
        q.y = fma(-d, uc.y, fma(ce, ue.y, fma(cw, uw.y, fma(cz, us.y + un.y, bv.y))));
    }
    return q;
}

// Level l's residual summed into level l + 1 (as k_residual_restrict): its b and,
// where that level is smoothed, b_hat and the first red half-sweep from zero.
// NORM: the squared residuals are added up.
template <class T, bool NORM> __device__ __forceinline__ double restrict_level(const Ctx<T> &X, int l) {
    const Lv v = X.lv[l];
    const bool last = l + 1 == X.A.nl, red_only = X.A.red_only, both = v.fz == 2 && v.fr == 2;
    const int ncr = v.fr == 2 ? v.hr : v.nr, fz1 = v.fz - 1, crows = v.rows >> fz1, crow0 = v.row0 >> fz1, chr = ncr >> 1;
    const V2<T> *u = (const V2<T> *)(X.sm + v.u), *b = (const V2<T> *)(X.sm + v.b);
    const V2<T> *bg = l > 0 || X.A.top_b ? nullptr : X.A.lv[0].L.b;
    const Tab<T> t = tab_of<T>(X.sm + v.tab, v.nr, v.ncls);
    const unsigned nm = X.A.D.nm;
    Lv w = v;
    const T *civ = nullptr;
    if (!last) {
        w = X.lv[l + 1];
        civ = tab_of<T>(X.sm + w.tab, w.nr, w.ncls).iv;
    }
    const unsigned rcr = last ? 0u : w.rnr;
    const V2<T> zero = mk<T>(0, 0);
    const int nc = red_only ? (both ? 2 : 1) : v.fz * v.fr;
    double acc = 0.0;
    // cells (2K, 2I) and (2K + 1, 2I + 1) by two lanes next to each other; other shapes by one thread
    const bool pair = red_only && both;
    const int sh = pair ? 1 : 0, total = (crows * ncr) << sh;
    for (int base = 0; base < total; base += DEEP_THREADS) {
        const int f2 = base + (int)threadIdx.x, f = min(f2, total - 1) >> sh;
        const int Kl = last ? f / ncr : (int)fdiv((unsigned)f, (unsigned)ncr, rcr), I = f - Kl * ncr, K = crow0 + Kl;
        bool on = f2 < total;
        V2<T> sum;
        if (pair) {
            const int c = f2 & 1;
            const V2<T> r = residual<T>(v, t, u, b, bg, nm, X.m, 2 * Kl + c, c, I);
            sum = mk<T>(r.x + __shfl_xor_sync(0xffffffffu, r.x, 1), r.y + __shfl_xor_sync(0xffffffffu, r.y, 1));
            if (NORM && on) acc = fma((double)r.y, (double)r.y, fma((double)r.x, (double)r.x, acc));
            on = on && c == 0;
        } else {
            sum = zero;
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
                int kl, i;
                if (red_only) {
                    kl = v.fz * Kl + (v.fz == 2 ? (I & 1) : 0);
                    i = v.fr * I + (v.fr == 2 ? (K & 1) : 0);
                } else {
                    kl = v.fz * Kl + (v.fr == 2 ? (c >> 1) : c);
                    i = v.fr * I + (v.fr == 2 ? (c & 1) : 0);
                }
                const V2<T> r = residual<T>(v, t, u, b, bg, nm, X.m, kl, i & 1, i >> 1);
                sum = c == 0 ? r : mk<T>(sum.x + r.x, sum.y + r.y);
                if (NORM && on) acc = fma((double)r.y, (double)r.y, fma((double)r.x, (double)r.x, acc));
            }
        }
        if (!on) continue;
        V2<T> bhv = zero;
        const int e = last ? I : pos(I, chr);
        if (!last) {
            const T inv = civ[row_class(K, w.nz, w.ncls) * ncr + e];
            bhv = mk<T>(sum.x * inv, sum.y * inv);
        }
        if (last) {
            ((V2<T> *)(X.sm + X.A.bc))[Kl * ncr + e] = sum;
        } else {
            ((V2<T> *)(X.sm + w.b))[Kl * ncr + e] = sum;
            ((V2<T> *)(X.sm + w.bh))[Kl * ncr + e] = bhv;
            X.put(w.u, Kl, e, ncr, w.rows, w.before, (X.A.pre > 0 && ((K + I) & 1) == 0) ? bhv : zero);
        }
    }
    X.sync();
    return acc;
}

// Level l + 1's correction prolongated into level l (as k_prolong).  ASSIGN: u = P c
// (on the black cells where a red half-sweep follows).
template <class T, bool ASSIGN> __device__ __forceinline__ void prolong_level(const Ctx<T> &X, int l) {
    const Lv v = X.lv[l];
    const bool last = l + 1 == X.A.nl, cz2 = v.fz == 2, cr2 = v.fr == 2, black_only = ASSIGN ? X.A.pre > 0 : X.A.black_only != 0;
    const int nr = v.nr, hr = v.hr, ncr = cr2 ? hr : nr, fz1 = v.fz - 1, ncz = v.nz >> fz1, crow0 = v.row0 >> fz1, chr = ncr >> 1;
    const V2<T> *u = (const V2<T> *)(X.sm + v.u), *cu = (const V2<T> *)(X.sm + (last ? X.A.bc : X.lv[l + 1].u));
    auto at = [&](int K, int I) { return cu[(K - crow0) * ncr + (last ? I : pos(I, chr))]; };
    const int per = black_only ? hr : nr;
    for (int c = threadIdx.x; c < v.rows * per; c += DEEP_THREADS) {
        const int kl = (int)fdiv((unsigned)c, (unsigned)per, black_only ? v.rhr : v.rnr), k = v.row0 + kl;
        const int i = black_only ? 2 * (c - kl * hr) + ((k + 1) & 1) : c - kl * nr;
        const int K = cz2 ? (k >> 1) : k, I = cr2 ? (i >> 1) : i;
        const int K2 = K + ((k & 1) ? 1 : -1), I2 = I + ((i & 1) ? 1 : -1);
        const bool kin = K2 >= 0 && K2 < ncz, iin = I2 >= 0 && I2 < ncr;
        const int Kx = kin ? K2 : K, Ix = iin ? I2 : I, e = pos(i, hr);
        const V2<T> c0 = at(K, I);
        V2<T> x = ASSIGN ? mk<T>(0, 0) : u[kl * nr + e];
        if (cz2 && cr2) {
            const V2<T> c1 = at(K, Ix), c2 = at(Kx, I), c3 = at(Kx, Ix);
            const T w1 = iin ? T(0.1875) : T(-0.1875), w2 = kin ? T(0.1875) : T(-0.1875);
            const T w3 = iin == kin ? T(0.0625) : T(-0.0625);
            x.x = fma(w3, c3.x, fma(w2, c2.x, fma(w1, c1.x, fma(T(0.5625), c0.x, x.x))));
            if constexpr (sizeof(T) == 8) x.y = fx_bilinear(x.y, c0.y, c1.y, c2.y, c3.y, !iin, !kin);
            else x.y = fma(w3, c3.y, fma(w2, c2.y, fma(w1, c1.y, fma(T(0.5625), c0.y, x.y))));
        } else {
            const V2<T> c1 = cz2 ? at(Kx, I) : at(K, Ix);
            const T w1 = (cz2 ? kin : iin) ? T(0.25) : T(-0.25);
            x.x = fma(w1, c1.x, fma(T(0.75), c0.x, x.x));
            if constexpr (sizeof(T) == 8) x.y = fx_linear(x.y, c0.y, c1.y, cz2 ? !kin : !iin);
            else x.y = fma(w1, c1.y, fma(T(0.75), c0.y, x.y));
        }
        X.put(v.u, kl, e, nr, v.rows, v.before, x);
    }
    X.sync();
}

// Exact solve of the coarsest level (the separable, mirror-folded solve of
// k_coarse), right-hand side and solution in bc.  The transforms along z are
// independent by column and the tridiagonal solves by row, so the blocks split
// the columns for the one and the rows for the other; what crosses between them
// goes through shared memory of the cluster.
template <class T> __device__ __forceinline__ void exact_solve(const Ctx<T> &X) {
    const DeepArg<T> &A = X.A;
    const int ncr = A.D.nr, ncz = A.D.nz, C = X.C, hzc = ncz - ncz / 2, hc = ncz / 2, lw = ncr + 1;
    const int i0 = ncr * X.rank / C, w = ncr * (X.rank + 1) / C - i0;   // this block's columns
    const int lane = (int)(threadIdx.x & 31), warp = (int)(threadIdx.x >> 5);
    V2<T> *bc = (V2<T> *)(X.sm + A.bc), *ws = (V2<T> *)(X.sm + A.ws);
    auto at = [&](V2<T> *base, int k, int ld, int i) {   // entry of row k, wherever it lies
        const int o = X.own[k];
        return peer(base, o >> 16) + ((o & 0xffff) * ld + i0 + i);
    };
    auto store = [&](int k, int i, V2<T> x) {   // solution: into bc and the halo rows next to it
        const int o = X.own[k], q = o >> 16, kl = o & 0xffff;
        *(peer(bc, q) + (kl * ncr + i0 + i)) = x;
        if (C > 1) {
            const int b = ncz * q / C, e = ncz * (q + 1) / C;
            if (k == b && q > 0) *(peer(bc, q - 1) + ((b - ncz * (q - 1) / C) * ncr + i0 + i)) = x;
            if (k == e - 1 && q + 1 < C) *(peer(bc, q + 1) + (i0 + i - ncr)) = x;
        }
    };
    if constexpr (sizeof(T) == 8) {
        // in fixed point, a column's values aligned to its largest (fixed.h)
        int4 *fo = (int4 *)(X.sm + A.fo);
        const int2 *Vs = (const int2 *)(X.sm + A.V);
        for (int i = warp; i < w; i += DEEP_THREADS / 32) {
            V2<T> p = mk<T>(0, 0), q = p;
            const int km = ncz - 1 - lane;
            if (lane < hzc) {
                p = *at(bc, lane, ncr, i);
                if (km != lane) {
                    const V2<T> hi = *at(bc, km, ncr, i);
                    q = mk<T>(p.x - hi.x, p.y - hi.y);
                    p = mk<T>(p.x + hi.x, p.y + hi.y);
                }
            }
            const int ex = __reduce_max_sync(0xffffffffu, max(exp_bits(p.x), exp_bits(q.x)));
            const int ey = __reduce_max_sync(0xffffffffu, max(exp_bits(p.y), exp_bits(q.y)));
            if (lane < hzc) {
                fo[lane * w + i] = fx_split2(fx_align<5>(p.x, exp_bits(p.x), ex), fx_align<5>(p.y, exp_bits(p.y), ey));
                if (km != lane)
                    fo[km * w + i] = fx_split2(fx_align<5>(q.x, exp_bits(q.x), ex), fx_align<5>(q.y, exp_bits(q.y), ey));
            }
            if (lane == 0) X.ecol[i] = make_int2(ex, ey);
        }
        __syncthreads();
        for (int f = threadIdx.x; f < ncz * w; f += DEEP_THREADS) {
            const int j = (int)fdiv((unsigned)f, (unsigned)w, X.rw), i = f - j * w, n = (j & 1) == 0 ? hzc : hc;
            const int4 *col = fo + i + ((j & 1) == 0 ? 0 : (ncz - 1) * w);
            const int step = (j & 1) == 0 ? w : -w;
            FxSum ax, ay;
#pragma unroll 4
            for (int k = 0; k < n; ++k) {
                const int2 c = Vs[k * ncz + j];
                const int4 x = col[k * step];
                fx_mac(ax, x.x, x.y, c);
                fx_mac(ay, x.z, x.w, c);
            }
            const int2 e = X.ecol[i];
            *at(ws, j, lw, i) = mk<T>(fx_column(fx_total(ax), e.x), fx_column(fx_total(ay), e.y));
        }
    } else {
        V2<T> *fo = (V2<T> *)(X.sm + A.fo);
        const T *Vs = (const T *)(X.sm + A.V);
        for (int f = threadIdx.x; f < hzc * w; f += DEEP_THREADS) {
            const int k = (int)fdiv((unsigned)f, (unsigned)w, X.rw), i = f - k * w, km = ncz - 1 - k;
            const V2<T> lo = *at(bc, k, ncr, i);
            if (km == k) {
                fo[k * w + i] = lo;
            } else {
                const V2<T> hi = *at(bc, km, ncr, i);
                fo[k * w + i] = mk<T>(lo.x + hi.x, lo.y + hi.y);
                fo[km * w + i] = mk<T>(lo.x - hi.x, lo.y - hi.y);
            }
        }
        __syncthreads();
        for (int f = threadIdx.x; f < ncz * w; f += DEEP_THREADS) {
            const int j = (int)fdiv((unsigned)f, (unsigned)w, X.rw), i = f - j * w, n = (j & 1) == 0 ? hzc : hc;
            const V2<T> *col = fo + i + ((j & 1) == 0 ? 0 : (ncz - 1) * w);
            const int step = (j & 1) == 0 ? w : -w;
            T ax = 0, ay = 0;
#pragma unroll 4
            for (int k = 0; k < n; ++k) {
                const T c = Vs[k * ncz + j];
                const V2<T> x = col[k * step];
                ax = fma(c, x.x, ax);
                ay = fma(c, x.y, ay);
            }
            *at(ws, j, lw, i) = mk<T>(ax, ay);
        }
    }
    X.sync();
    tri_rows<T, 2>((T *)ws, (const T *)(X.sm + A.ps), (const T *)(X.sm + A.fs), (const T *)(X.sm + A.cs), (const T *)(X.sm + A.Q),
                   2 * (X.z1 - X.z0), ncr, lw);
    X.sync();
    if constexpr (sizeof(T) == 8) {
        int4 *fo = (int4 *)(X.sm + A.fo);
        const int2 *Vs = (const int2 *)(X.sm + A.V);
        for (int i = warp; i < w; i += DEEP_THREADS / 32) {
            V2<T> p = mk<T>(0, 0), q = p;
            if (lane < ncz) p = *at(ws, lane, lw, i);
            if (lane + 32 < ncz) q = *at(ws, lane + 32, lw, i);
            const int ex = __reduce_max_sync(0xffffffffu, max(exp_bits(p.x), exp_bits(q.x)));
            const int ey = __reduce_max_sync(0xffffffffu, max(exp_bits(p.y), exp_bits(q.y)));
            if (lane < ncz)
                fo[lane * w + i] = fx_split2(fx_align<5>(p.x, exp_bits(p.x), ex), fx_align<5>(p.y, exp_bits(p.y), ey));
            if (lane + 32 < ncz)
                fo[(lane + 32) * w + i] = fx_split2(fx_align<5>(q.x, exp_bits(q.x), ex), fx_align<5>(q.y, exp_bits(q.y), ey));
            if (lane == 0) X.ecol[i] = make_int2(ex, ey);
        }
        __syncthreads();
        // two threads per pair of rows (k, ncz-1-k): the sums over even and over odd j
        for (int base = 0; base < 2 * hzc * w; base += DEEP_THREADS) {
            const int f = base + (int)threadIdx.x, g = min(f >> 1, hzc * w - 1), h = f & 1;
            const int k = (int)fdiv((unsigned)g, (unsigned)w, X.rw), i = g - k * w, km = ncz - 1 - k;
            FxSum sx, sy;
            const int2 *c = Vs + k * ncz;
#pragma unroll 4
            for (int j = h; j < ncz; j += 2) {
                const int4 x = fo[j * w + i];
                fx_mac(sx, x.x, x.y, c[j]);
                fx_mac(sy, x.z, x.w, c[j]);
            }
            const fx ax = fx_total(sx), ay = fx_total(sy);
            const fx bx = __shfl_xor_sync(0xffffffffu, ax, 1), by = __shfl_xor_sync(0xffffffffu, ay, 1);
            const int2 e = X.ecol[i];
            if (f < 2 * hzc * w && (h == 0 || km != k))
                store(h ? km : k, i, mk<T>(fx_column(h ? bx - ax : ax + bx, e.x), fx_column(h ? by - ay : ay + by, e.y)));
        }
    } else {
        V2<T> *fo = (V2<T> *)(X.sm + A.fo);
        const T *Vs = (const T *)(X.sm + A.V);
        for (int f = threadIdx.x; f < ncz * w; f += DEEP_THREADS) {
            const int j = (int)fdiv((unsigned)f, (unsigned)w, X.rw), i = f - j * w;
            fo[f] = *at(ws, j, lw, i);
        }
        __syncthreads();
        for (int f = threadIdx.x; f < hzc * w; f += DEEP_THREADS) {
            const int k = (int)fdiv((unsigned)f, (unsigned)w, X.rw), i = f - k * w, km = ncz - 1 - k;
            T ex = 0, ey = 0, ox = 0, oy = 0;
#pragma unroll 2
            for (int j = 0; j + 1 < ncz; j += 2) {
                const T v0 = Vs[k * ncz + j], v1 = Vs[k * ncz + j + 1];
                const V2<T> a = fo[j * w + i], b = fo[(j + 1) * w + i];
                ex = fma(v0, a.x, ex);
                ey = fma(v0, a.y, ey);
                ox = fma(v1, b.x, ox);
                oy = fma(v1, b.y, oy);
            }
            if (ncz & 1) {
                const T c = Vs[k * ncz + ncz - 1];
                const V2<T> a = fo[(ncz - 1) * w + i];
                ex = fma(c, a.x, ex);
                ey = fma(c, a.y, ey);
            }
            store(k, i, mk<T>(ex + ox, ey + oy));
            if (km != k) store(km, i, mk<T>(ex - ox, ey - oy));
        }
    }
    X.sync();
}

// V-cycle from level `down` to the coarsest and back up to level `up`.
template <class T> __device__ __forceinline__ void vcycle(const Ctx<T> &X, int down, int up, bool skip) {
    const int nl = X.A.nl;
    for (int d = down; d < nl; ++d) {
        sweeps(X, d, X.A.pre, d > down ? X.A.pre > 0 : skip);
        restrict_level<T, false>(X, d);
    }
    exact_solve(X);
    for (int d = nl - 1; d >= up; --d) {
        prolong_level<T, false>(X, d);
        sweeps(X, d, X.A.post, false);
    }
}

// Level l's right-hand side summed into level l + 1 (as k_rhs_restrict), whose
// iterate becomes the first red half-sweep from zero.
template <class T> __device__ __forceinline__ void rhs_level(const Ctx<T> &X, int l) {
    const Lv v = X.lv[l];
    const bool last = l + 1 == X.A.nl;
    const int ncr = v.fr == 2 ? v.hr : v.nr, fz1 = v.fz - 1, crows = v.rows >> fz1, crow0 = v.row0 >> fz1, chr = ncr >> 1;
    const V2<T> *b = (const V2<T> *)(X.sm + v.b), *bg = X.A.lv[0].L.b, zero = mk<T>(0, 0);
    const Lv w = last ? v : X.lv[l + 1];
    const T *civ = last ? nullptr : tab_of<T>(X.sm + w.tab, w.nr, w.ncls).iv;
    const unsigned nm = X.A.D.nm;
    for (int f = threadIdx.x; f < crows * ncr; f += DEEP_THREADS) {
        const int Kl = f / ncr, I = f - Kl * ncr, K = crow0 + Kl;
        V2<T> sum = zero;
        for (int c = 0; c < v.fz * v.fr; ++c) {
            const int kl = v.fz * Kl + (v.fr == 2 ? (c >> 1) : c), i = v.fr * I + (v.fr == 2 ? (c & 1) : 0);
            const V2<T> x = l > 0 ? b[kl * v.nr + pos(i, v.hr)]
                                  : bg[((unsigned)(v.row0 + kl) * (unsigned)v.nr + (unsigned)i) * nm + (unsigned)X.m];
            sum = c == 0 ? x : mk<T>(sum.x + x.x, sum.y + x.y);
        }
        if (last) {
            ((V2<T> *)(X.sm + X.A.bc))[Kl * ncr + I] = sum;
            continue;
        }
        const int e = pos(I, chr);
        const T inv = civ[row_class(K, w.nz, w.ncls) * ncr + e];
        const V2<T> bhv = mk<T>(sum.x * inv, sum.y * inv);
        ((V2<T> *)(X.sm + w.b))[Kl * ncr + e] = sum;
        ((V2<T> *)(X.sm + w.bh))[Kl * ncr + e] = bhv;
        X.put(w.u, Kl, e, ncr, w.rows, w.before, (X.A.pre > 0 && ((K + I) & 1) == 0) ? bhv : zero);
    }
    X.sync();
}

// The full-multigrid start of a solve (as fmg_start in solve.cu): level 0 gets the
// prolongated solution of level 1.
template <class T> __device__ __forceinline__ void fmg(const Ctx<T> &X) {
    const int nl = X.A.nl;
    for (int l = 0; l < nl; ++l) rhs_level(X, l);
    int l = nl;   // level whose solution is known
    if (X.A.bottom) vcycle(X, --l, nl - 1, X.A.pre > 0);
    else exact_solve(X);
    while (l > 0) {
        prolong_level<T, true>(X, --l);
        if (l > 0) vcycle(X, l, l, false);
    }
}

// Norm of the residual over all modes and the convergence test (as k_check for one
// FP64 problem).  Every block adds its part; the first block of each cluster
// waits for all of them, adds them in the same order and tells its cluster.  The
// grid is resident as a whole (a cooperative launch); a wait that runs out all
// the same (Ctrl::polls) ends the solve with the status ECUDA and a NaN residual.
// Clusters whose own wait was met go on to the next test and give up there.
struct Test {
    double best, rr_first, rr;
    int stall, cycles, epoch, status;
};
__device__ __forceinline__ int converged(Ctrl *ctrl, Test &t) {
    const double tol = ctrl->tol, bb = ctrl->bnorm2[0];
    // far from the tolerance: no division, no square root
    if (tol > 0.0 && t.cycles < ctrl->max_cycles && bb > 0.0 && t.rr < 1e300 && t.rr > 1.001 * tol * tol * bb) return 0;
    const double rel = bb > 0.0 ? sqrt(t.rr / bb) : sqrt(t.rr);
    int stop = 0;
    if (isnan(rel) || isinf(rel)) {
        t.status = PIC_POISSON_ENONFINITE;
        return 1;
    }
    if (tol > 0.0) {
        stop = rel <= tol;
    } else if (rel < 0.5 * t.best) {   // halved since the last reference point
        t.best = rel;
        t.stall = 0;
    } else {
        stop = ++t.stall >= kFloorWindow;
    }
    if (!stop && t.cycles >= ctrl->max_cycles) {
        stop = 1;
        t.status = PIC_POISSON_ENOTCONVERGED;
    }
    return stop;
}
template <class T>
__device__ __forceinline__ bool test(const Ctx<T> &X, Ctrl *ctrl, double *partials, double acc, Test &t, double *red, int *s_stop) {
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    ++t.epoch;
    double *part = partials + (t.epoch & 1) * gridDim.x;   // (read until every block has come to the next test)
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int i = 0; i < DEEP_THREADS / 32; ++i) s += red[i];
            const int nt = X.A.lv[0].L.nt;
            __stcg(part + blockIdx.x, s * ((X.m == 0 || 2 * X.m == nt) ? 1.0 : 2.0));
            __threadfence();
            atomicAdd(&ctrl->arrived, 1u);
        }
        if (X.rank == 0) {
            int ok = 1;
            if (threadIdx.x == 0) {
                const unsigned want = (unsigned)t.epoch * gridDim.x;
                ok = 0;
                for (int n = 0, polls = ctrl->polls; n < polls && !ok; ++n) {
                    unsigned got;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(&ctrl->arrived) : "memory");
                    ok = got >= want;
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            double s = 0.0;
            if (ok)
                for (unsigned b = threadIdx.x; b < gridDim.x; b += 32) s += __ldcg(part + b);
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (threadIdx.x == 0) {
                t.rr = ok ? s : __longlong_as_double(0x7ff8000000000000ll);
                if (t.epoch == 1) t.rr_first = t.rr;
                int stop = 1;
                if (ok) stop = converged(ctrl, t);
                else t.status = PIC_POISSON_ECUDA;
                for (int r = 0; r < X.C; ++r) *peer(s_stop, r) = stop;
            }
        }
    }
    X.sync();
    return *s_stop != 0;
}

// SOLVE: the whole solve of one FP64 problem -- starting iterate (`start`: 0 the
// level's, 1 zero, 2 a full-multigrid pass), then V-cycles until the residual
// meets the test.  Else: `cycles` V-cycles on the first level of A, from zero
// (start 1) or from the level's iterate.
template <class T, bool SOLVE>
__global__ void __launch_bounds__(DEEP_THREADS, 1) k_deep(const __grid_constant__ DeepArg<T> A, int start, int cycles, Ctrl *ctrl,
                                                          double *partials) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ double red[DEEP_THREADS / 32];
    __shared__ int s_stop;
    __shared__ Lv slv[DEEP_LEVELS];
    __shared__ int own[DEEP_MAX_NZ];
    const int C = A.C, ncz = A.D.nz, ncr = A.D.nr, nm = A.D.nm;
    const int rank = C == 1 ? 0 : (int)(blockIdx.x % (unsigned)C), m = (int)(blockIdx.x / (unsigned)C);
    const int z0 = ncz * rank / C, z1 = ncz * (rank + 1) / C, zb = rank > 0 ? z0 - ncz * (rank - 1) / C : 0;
    const int w = ncr * (rank + 1) / C - ncr * rank / C;
    const unsigned rw = w ? 0xffffffffu / (unsigned)w : 0u;
    const Ctx<T> X{A, smraw, rank > 0 ? peer(smraw, rank - 1) : nullptr, rank + 1 < C ? peer(smraw, rank + 1) : nullptr,
                   slv, own, (int2 *)(smraw + A.ecol), rw, C, rank, m, z0, z1, zb};
    if (threadIdx.x < (unsigned)A.nl) {
        const DeepLevel<T> &v = A.lv[threadIdx.x];
        Lv &o = slv[threadIdx.x];
        o.nr = v.L.nr;
        o.hr = v.L.nr >> 1;
        o.nz = v.L.nz;
        o.ncls = v.L.ncls;
        o.row0 = v.zmul * z0;
        o.rows = v.zmul * (z1 - z0);
        o.before = v.zmul * zb;
        o.rq = v.L.rq;
        o.u = v.u;
        o.bh = v.bh;
        o.b = v.b;
        o.tab = v.tab;
        o.rhr = v.L.rhr;
        o.rnr = v.L.rnr;
        o.fz = v.fz;
        o.fr = v.fr;
    }
    for (int r = 0; r < C; ++r)
        for (int k = ncz * r / C + (int)threadIdx.x; k < ncz * (r + 1) / C; k += DEEP_THREADS) own[k] = r << 16 | (k - ncz * r / C);
    const V2<T> zero = mk<T>(0, 0);
    for (int l = 0; l <= A.nl; ++l) {   // halo rows (those beyond a wall stay zero)
        const int w = l < A.nl ? A.lv[l].L.nr : ncr, rows = l < A.nl ? A.lv[l].zmul * (z1 - z0) : z1 - z0;
        V2<T> *a = (V2<T> *)(smraw + (l < A.nl ? A.lv[l].u : A.bc));
        for (int f = threadIdx.x; f < w; f += DEEP_THREADS) a[f - w] = a[rows * w + f] = zero;
    }
    // tables, all in flight at once, before the wait for the kernel before
    for (int l = 0; l < A.nl; ++l) {
        const LevelDev<T> &L = A.lv[l].L;
        const Tab<T> t = tab_of<T>(smraw + A.lv[l].tab, L.nr, L.ncls);
        const int nr = L.nr, hr = nr >> 1;
        for (int f = threadIdx.x; f < L.ncls * nr; f += DEEP_THREADS) {
            const int cl = f / nr, d = cl * nr + pos(f - cl * nr, hr);
            const size_t g = (size_t)f * nm + m;
            cp_async_bytes<sizeof(T)>(t.hz + d, L.hz + g);
            cp_async_bytes<sizeof(T)>(t.hw + d, L.hw + g);
            cp_async_bytes<sizeof(T)>(t.he + d, L.he + g);
            cp_async_bytes<sizeof(T)>(t.dg + d, L.diag + g);
            cp_async_bytes<sizeof(T)>(t.iv + d, L.invd + g);
            if constexpr (sizeof(T) == 8) {
                cp_async_bytes<16>(t.hzw + d, L.hzw + g);
                cp_async_bytes<8>(t.hev + d, L.hev + g);
                cp_async_bytes<8>(t.rdg + d, L.rdg + g);
            }
        }
        for (int i = threadIdx.x; i < nr; i += DEEP_THREADS) {
            const int d = pos(i, hr);
            cp_async_bytes<sizeof(T)>(t.cz + d, L.cz + i);
            cp_async_bytes<sizeof(T)>(t.cw + d, L.cw + i);
            cp_async_bytes<sizeof(T)>(t.ce + d, L.ce + i);
            if constexpr (sizeof(T) == 8) {
                cp_async_bytes<16>(t.rzw + d, L.rzw + i);
                cp_async_bytes<8>(t.rev + d, L.rev + i);
            }
        }
    }
    {
        const int hzc = ncz - ncz / 2, lw = ncr + 1;
        T *Vs = (T *)(smraw + A.V), *ps = (T *)(smraw + A.ps), *cs = (T *)(smraw + A.cs), *fs = (T *)(smraw + A.fs);
        const T *V = A.D.Vl ? (const T *)A.D.Vl : A.D.V;
        for (int f = threadIdx.x; f < hzc * ncz; f += DEEP_THREADS) cp_async_bytes<sizeof(T)>(Vs + f, V + f);
        const size_t base = ((size_t)m * ncz + z0) * ncr;
        for (int f = threadIdx.x; f < (z1 - z0) * ncr; f += DEEP_THREADS) {
            const int j = f / ncr, i = f - j * ncr;
            cp_async_bytes<sizeof(T)>(ps + j * lw + i, A.D.piv + base + f);
            cp_async_bytes<sizeof(T)>(cs + j * lw + i, A.D.cpr + base + f);
            cp_async_bytes<sizeof(T)>(fs + j * lw + i, A.D.f + base + f);
        }
        if (ncr > TRI_SERIAL)
            for (int f = threadIdx.x; f < (z1 - z0) * TRI_Q; f += DEEP_THREADS)
                cp_async_bytes<sizeof(T)>((T *)(smraw + A.Q) + f, A.D.fq + ((size_t)m * ncz + z0) * TRI_Q + f);
    }
    __syncthreads();   // (the halo rows are zero before the copies below)
    pdl_wait();
    pdl_go();
    const LevelDev<T> &L0 = A.lv[0].L;
    const int nr = L0.nr, hr = nr >> 1, nz = L0.nz, row0 = A.lv[0].zmul * z0, rows = A.lv[0].zmul * (z1 - z0);
    V2<T> *u0 = (V2<T> *)(smraw + A.lv[0].u), *bh0 = (V2<T> *)(smraw + A.lv[0].bh), *b0 = (V2<T> *)(smraw + A.lv[0].b);
    // the levels' inputs, the iterates with the rows next to this block's
    for (int f = threadIdx.x; f < (rows + 2) * nr; f += DEEP_THREADS) {
        const int kl = (int)fdiv((unsigned)f, (unsigned)nr, L0.rnr) - 1, i = f - (kl + 1) * nr, k = row0 + kl;
        if (k < 0 || k >= nz) continue;
        const int d = kl * nr + pos(i, hr);
        const unsigned g = ((unsigned)k * (unsigned)nr + (unsigned)i) * (unsigned)nm + (unsigned)m;
        const bool here = kl >= 0 && kl < rows, red_cell = ((k + i) & 1) == 0;
        if (here) {
            cp_async_bytes<sizeof(V2<T>)>(bh0 + d, L0.bh + g);
            if (A.top_b && (!A.red_only || red_cell)) cp_async_bytes<sizeof(V2<T>)>(b0 + d, L0.b + g);
        }
        if (start == 0) cp_async_bytes<sizeof(V2<T>)>(u0 + d, L0.u + g);
        else if (!SOLVE && A.pre > 0 && red_cell) cp_async_bytes<sizeof(V2<T>)>(u0 + d, L0.bh + g);   // the first red half-sweep
        else u0[d] = zero;
    }
    cp_async_wait_all();
    X.sync();   // (every block of the cluster has started and loaded)
    if constexpr (SOLVE) {
        Test t{INFINITY, 0.0, 0.0, 0, 0, 0, PIC_POISSON_OK};
        if (start == 2) fmg(X);
        sweeps(X, 0, A.pre, false);
        while (!test(X, ctrl, partials, restrict_level<T, true>(X, 0), t, red, &s_stop)) {
            ++t.cycles;
            vcycle(X, 1, 0, A.pre > 0);
            sweeps(X, 0, A.pre, false);
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            const double bb = ctrl->bnorm2[0];
            ctrl->rel[0] = bb > 0.0 ? sqrt(t.rr / bb) : sqrt(t.rr);
            ctrl->rel_first[0] = bb > 0.0 ? sqrt(t.rr_first / bb) : sqrt(t.rr_first);
            ctrl->status[0] = t.status;
            ctrl->done[0] = 1;
            ctrl->done_cycles[0] = ctrl->cycles = t.cycles;
            ctrl->cont = 0;
        }
    } else {
        for (int c = 0; c < cycles; ++c) vcycle(X, 0, 0, c == 0 && start == 1 && A.pre > 0);
    }
    for (int f = threadIdx.x; f < rows * nr; f += DEEP_THREADS) {
        const int kl = (int)fdiv((unsigned)f, (unsigned)nr, L0.rnr), i = f - kl * nr;
        L0.u[((size_t)row0 * nr + f) * nm + m] = u0[kl * nr + pos(i, hr)];
    }
    // (a half-sweep, and so every way to here, ends with the cluster's barrier:
    // no block leaves while another still reads its shared memory)
}

}  // namespace

template <class T> size_t deep_layout(DeepArg<T> &A, int C) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 15) & ~size_t(15);
        return (unsigned)o;
    };
    const int ncz = A.D.nz, ncr = A.D.nr;
    const int rmax = (ncz + C - 1) / C, wmax = (ncr + C - 1) / C;
    A.C = C;
    for (int l = 0; l < A.nl; ++l) {
        DeepLevel<T> &v = A.lv[l];
        const size_t n = (size_t)v.zmul * rmax * v.L.nr * sizeof(V2<T>);
        v.u = take(n + 2 * (size_t)v.L.nr * sizeof(V2<T>)) + (unsigned)(v.L.nr * sizeof(V2<T>));
        v.bh = take(n);
        v.b = l > 0 || A.top_b ? take(n) : 0;
        v.tab = take(tab_bytes<T>(v.L.nr, v.L.ncls));
    }
    A.bc = take((size_t)(rmax + 2) * ncr * sizeof(V2<T>)) + (unsigned)(ncr * sizeof(V2<T>));
    A.fo = take((size_t)ncz * wmax * sizeof(V2<T>));
    A.ws = take((size_t)rmax * (ncr + 1) * sizeof(V2<T>));
    A.V = take((size_t)(ncz - ncz / 2) * ncz * sizeof(T));
    A.ps = take((size_t)rmax * (ncr + 1) * sizeof(T));
    A.cs = take((size_t)rmax * (ncr + 1) * sizeof(T));
    A.fs = take((size_t)rmax * (ncr + 1) * sizeof(T));
    A.Q = take((size_t)rmax * TRI_Q * sizeof(T));
    A.ecol = take((size_t)wmax * sizeof(int2));
    A.smem = (unsigned)off;
    return off;
}

namespace {
template <class T> void deep_config(const DeepArg<T> &A, cudaLaunchConfig_t &c, cudaLaunchAttribute *at, cudaStream_t st) {
    c.gridDim = dim3((unsigned)(A.D.nm * A.C));
    c.blockDim = dim3(DEEP_THREADS);
    c.dynamicSmemBytes = A.smem;
    c.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)A.C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    c.attrs = at;
    c.numAttrs = 1;
}
// (the limit, not this launch's size: other plans set it too, on other threads)
template <class K> cudaError_t deep_smem(K *k) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DEEP_MAX_SMEM);
}
}  // namespace

template <class T> int deep_resident(const DeepArg<T> &A) {
    if (deep_smem(k_deep<T, sizeof(T) == 8>) != cudaSuccess) return 0;
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[1]{};
    deep_config(A, c, at, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_deep<T, sizeof(T) == 8>, &c) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <class T>
cudaError_t launch_deep(const DeepArg<T> &A, bool from_zero, int cycles, cudaStream_t st) {
    cudaError_t e = deep_smem(k_deep<T, false>);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[2]{};
    deep_config(A, c, at, st);
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    c.numAttrs = 2;
    return cudaLaunchKernelEx(&c, k_deep<T, false>, A, from_zero ? 1 : 0, cycles, (Ctrl *)nullptr, (double *)nullptr);
}

cudaError_t launch_deep_solve(const DeepArg<double> &A, int start, Ctrl *ctrl, double *partials, cudaStream_t st) {
    cudaError_t e = deep_smem(k_deep<double, true>);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[2]{};
    deep_config(A, c, at, st);
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    c.numAttrs = 2;
    return cudaLaunchKernelEx(&c, k_deep<double, true>, A, start, 0, ctrl, partials);
}

template size_t deep_layout<double>(DeepArg<double> &, int);
template size_t deep_layout<float>(DeepArg<float> &, int);
template int deep_resident<double>(const DeepArg<double> &);
template int deep_resident<float>(const DeepArg<float> &);
template cudaError_t launch_deep<double>(const DeepArg<double> &, bool, int, cudaStream_t);
template cudaError_t launch_deep<float>(const DeepArg<float> &, bool, int, cudaStream_t);

}  // namespace pp
