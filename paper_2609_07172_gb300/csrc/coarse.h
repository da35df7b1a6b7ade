// Pieces of the separable coarsest-level solve, shared by k_coarse (mg.cu),
// k_bottom (bottom.cu) and k_deep (deep.cu), which give the same bits.
#pragma once

#include "fixed.h"
#include "internal.h"

namespace pp {

// The radial tridiagonal solves, one per axial eigenvector (and part), in place
// on rows of n entries: forward y_i = w_i piv_i + f_i y_(i-1) with
// f_i = -e_(i-1) piv_i, back x_i = y_i - cpr_i x_(i+1), with piv, f, cpr ([rows][lw])
// and Q ([rows][TRI_Q]) of the factorisation in shared memory.  E = 2: rows hold
// two parts interleaved, row g of `rows` is part g & 1 of row g / 2.
//
// A recurrence is a chain of FP64 operations of 64 cycles or more each (45 x 35:
// 14,000 cycles with a subtraction and a product per step).  Above 8 entries
// eight lanes share a row: each runs its eighth from zero, three shuffle steps
// with the products Q of the factors (tri_factors) give every lane the value
// that enters its eighth, and a second run gives the entries.
// (Q: [forward, back][step 1, 2, 4][lane])
constexpr int TRI_SERIAL = 8;
template <class T, int E>
__device__ __forceinline__ void tri_rows(T *ws, const T *ps, const T *fs, const T *cs, const T *Qs, int rows, int n, int lw) {
    if (n <= TRI_SERIAL) {   // one thread per row, over the first four warps (one per sub-partition)
        const int w = (int)(threadIdx.x >> 5), per = (rows + 3) >> 2;
        if (w < 4)
            for (int l = (int)(threadIdx.x & 31); l < per && w * per + l < rows; l += 32) {
                const int g = w * per + l;
                const size_t r = (size_t)(E == 2 ? g >> 1 : g) * lw;
                T *row = ws + r * E + (E == 2 ? (g & 1) : 0);
                T y = 0;
                for (int i = 0; i < n; ++i) {
                    y = fma(fs[r + i], y, row[E * i] * ps[r + i]);
                    row[E * i] = y;
                }
                for (int i = n - 2; i >= 0; --i) {
                    y = fma(-cs[r + i], y, row[E * i]);
                    row[E * i] = y;
                }
            }
        return;
    }
    constexpr unsigned FULL = 0xffffffffu;
    const int s = (int)(threadIdx.x & 7), len = (n + 7) >> 3, i0 = min(s * len, n), i1 = min(i0 + len, n);
    for (int base = (int)(threadIdx.x >> 5) * 4; base < rows; base += (int)(blockDim.x >> 5) * 4) {
        const int g = base + (int)((threadIdx.x >> 3) & 3);
        const bool on = g < rows;
        const size_t gr = on ? (size_t)(E == 2 ? g >> 1 : g) : 0, r = gr * lw;
        T *row = ws + r * E + (E == 2 ? (g & 1) : 0);
        const T *piv = ps + r, *f = fs + r, *c = cs + r, *Q = Qs + gr * TRI_Q + s;
        const int a = on ? i0 : 0, b = on ? i1 : 0;
        T y = 0;
        for (int i = a; i < b; ++i) {
            const T t = row[E * i] * piv[i];
            row[E * i] = t;
            y = fma(f[i], y, t);
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const T p = __shfl_up_sync(FULL, y, 1 << d, 8);
            if (s >= 1 << d) y = fma(Q[8 * d], p, y);
        }
        y = __shfl_up_sync(FULL, y, 1, 8);
        if (s == 0) y = 0;
        for (int i = a; i < b; ++i) {
            y = fma(f[i], y, row[E * i]);
            row[E * i] = y;
        }
        T x = 0;
        for (int i = b - 1; i >= a; --i) x = fma(i + 1 < n ? -c[i] : T(0), x, row[E * i]);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const T p = __shfl_down_sync(FULL, x, 1 << d, 8);
            if (s + (1 << d) < 8) x = fma(Q[24 + 8 * d], p, x);
        }
        x = __shfl_down_sync(FULL, x, 1, 8);
        if (s == 7) x = 0;
        for (int i = b - 1; i >= a; --i) {
            x = fma(i + 1 < n ? -c[i] : T(0), x, row[E * i]);
            row[E * i] = x;
        }
    }
}
// f and Q of one row from its pivots, multipliers and the off-diagonal.
template <class T> __device__ void tri_factors(const T *e, const T *piv, const T *cpr, int n, T *f, T *Q) {
    for (int i = 0; i < n; ++i) f[i] = i > 0 ? -e[i - 1] * piv[i] : T(0);
    const int len = (n + 7) >> 3;
    for (int s = 0; s < 8; ++s) {
        const int a = min(s * len, n), b = min(a + len, n);
        T p = 1, q = 1;
        for (int i = a; i < b; ++i) p *= f[i];
        for (int i = b - 1; i >= a; --i) q *= i + 1 < n ? -cpr[i] : T(0);
        Q[s] = p;
        Q[24 + s] = q;
    }
    for (int d = 1; d < 3; ++d)
        for (int s = 0; s < 8; ++s) {
            const int up = s - (1 << (d - 1)), dn = s + (1 << (d - 1));
            Q[8 * d + s] = up >= 0 ? Q[8 * (d - 1) + s] * Q[8 * (d - 1) + up] : Q[8 * (d - 1) + s];
            Q[24 + 8 * d + s] = dn < 8 ? Q[24 + 8 * (d - 1) + s] * Q[24 + 8 * (d - 1) + dn] : Q[24 + 8 * (d - 1) + s];
        }
}

// One real part's transforms by a whole block (nr x nz), mirror-folded.
// Binary64 in fixed point, V then as limbs (CoarseDev::Vl), each column aligned
// to its largest value: one warp per column, exponents in ecol [nr].  A lane takes one
// mirror pair and two rows, and a sum of 64 products fits FxSum:
static_assert(kMaxCoarseNz <= 64, "the planner's limit is the transforms'");

// bs [nz][nr] -> ws [nz][lw] = V^T b; bs is overwritten.
template <class T>
__device__ __forceinline__ void coarse_forward(T *bs, T *ws, const T *Vs, int *ecol, int nr, int nz, int lw) {
    const int h = nz >> 1, hz = nz - h;   // mirror pairs, rows with k <= nz-1-k
    if constexpr (sizeof(T) == 8) {
        const int lane = (int)(threadIdx.x & 31);
        int2 *xs = (int2 *)bs;
        for (int i = (int)(threadIdx.x >> 5); i < nr; i += (int)(blockDim.x >> 5)) {
            const int km = nz - 1 - lane;
            T p = 0, q = 0;
            if (lane < hz) {
                p = bs[lane * nr + i];
                if (km != lane) {
                    const T hi = bs[km * nr + i];
                    q = p - hi;
                    p = p + hi;
                }
            }
            const int em = __reduce_max_sync(0xffffffffu, max(exp_bits(p), exp_bits(q)));
            if (lane < hz) {
                xs[lane * nr + i] = fx_split(fx_align<5>(p, exp_bits(p), em));
                if (km != lane) xs[km * nr + i] = fx_split(fx_align<5>(q, exp_bits(q), em));
            }
            if (lane == 0) ecol[i] = em;
        }
        __syncthreads();
        const int2 *Vl = (const int2 *)Vs;
        for (int f = threadIdx.x; f < nz * nr; f += blockDim.x) {
            const int j = f / nr, i = f - j * nr, n = (j & 1) == 0 ? hz : h;
            const int2 *col = xs + i + ((j & 1) == 0 ? 0 : (nz - 1) * nr);
            const int step = (j & 1) == 0 ? nr : -nr;
            FxSum a;
#pragma unroll 4
            for (int k = 0; k < n; ++k) {
                const int2 x = col[k * step];
                fx_mac(a, x.x, x.y, Vl[k * nz + j]);
            }
            ws[j * lw + i] = fx_column(fx_total(a), ecol[i]);
        }
    } else {
        for (int f = threadIdx.x; f < h * nr; f += blockDim.x) {
            const int k = f / nr, i = f - k * nr;
            const T lo = bs[k * nr + i], hi = bs[(nz - 1 - k) * nr + i];
            bs[k * nr + i] = lo + hi;
            bs[(nz - 1 - k) * nr + i] = lo - hi;
        }
        __syncthreads();
        for (int f = threadIdx.x; f < nz * nr; f += blockDim.x) {
            const int j = f / nr, i = f - j * nr;
            T a = 0;
            if ((j & 1) == 0) {
                for (int k = 0; k < hz; ++k) a = fma(Vs[k * nz + j], bs[k * nr + i], a);
            } else {
                for (int k = 0; k < h; ++k) a = fma(Vs[k * nz + j], bs[(nz - 1 - k) * nr + i], a);
            }
            ws[j * lw + i] = a;
        }
    }
    __syncthreads();
}

// put(k, i, value) of V w for every row k and column i; ws is overwritten.
template <class T, class Put>
__device__ __forceinline__ void coarse_back(T *ws, const T *Vs, int *ecol, int nr, int nz, int lw, Put put) {
    const int hz = nz - (nz >> 1);
    if constexpr (sizeof(T) == 8) {
        const int lane = (int)(threadIdx.x & 31);
        int2 *xs = (int2 *)ws;
        for (int i = (int)(threadIdx.x >> 5); i < nr; i += (int)(blockDim.x >> 5)) {
            const T p = lane < nz ? ws[lane * lw + i] : T(0), q = lane + 32 < nz ? ws[(lane + 32) * lw + i] : T(0);
            const int em = __reduce_max_sync(0xffffffffu, max(exp_bits(p), exp_bits(q)));
            if (lane < nz) xs[lane * lw + i] = fx_split(fx_align<5>(p, exp_bits(p), em));
            if (lane + 32 < nz) xs[(lane + 32) * lw + i] = fx_split(fx_align<5>(q, exp_bits(q), em));
            if (lane == 0) ecol[i] = em;
        }
        __syncthreads();
        const int2 *Vl = (const int2 *)Vs;
        for (int f = threadIdx.x; f < hz * nr; f += blockDim.x) {
            const int k = f / nr, i = f - k * nr;
            FxSum e, o;
            for (int j = 0; j < nz; j += 2) {
                const int2 x = xs[j * lw + i];
                fx_mac(e, x.x, x.y, Vl[k * nz + j]);
                if (j + 1 < nz) {
                    const int2 y = xs[(j + 1) * lw + i];
                    fx_mac(o, y.x, y.y, Vl[k * nz + j + 1]);
                }
            }
            const fx se = fx_total(e), so = fx_total(o);
            put(k, i, fx_column(se + so, ecol[i]));
            if (nz - 1 - k != k) put(nz - 1 - k, i, fx_column(se - so, ecol[i]));
        }
    } else {
        for (int f = threadIdx.x; f < hz * nr; f += blockDim.x) {
            const int k = f / nr, i = f - k * nr;
            T e = 0, o = 0;
            for (int j = 0; j + 1 < nz; j += 2) {
                e = fma(Vs[k * nz + j], ws[j * lw + i], e);
                o = fma(Vs[k * nz + j + 1], ws[(j + 1) * lw + i], o);
            }
            if (nz & 1) e = fma(Vs[k * nz + nz - 1], ws[(nz - 1) * lw + i], e);
            put(k, i, e + o);
            if (nz - 1 - k != k) put(nz - 1 - k, i, e - o);
        }
    }
}

}  // namespace pp
