// Batched azimuthal real DFT (step a-1, fused with the right-hand side build)
// and its inverse (step a-8).
//
// Forward, Eq. azimuthal_dft with the 1/N_theta scale, then Eq. mode_rhs:
//   b_(i,k),m = s_i * (1/N) sum_j rho_(i,j,k) e^{-2 pi i m j / N} + b^D_(i,k) delta_m0
// Inverse (Sec. 3.1, inverse transform, no scale), with conjugate symmetry:
//   phi_j = sum_{m=0}^{N-1} phihat_m e^{2 pi i m j / N}
//
// Each CTA owns one axial plane k of one problem and TI = 32 consecutive radial
// columns; lane l of every warp works on column i0 + l, so global loads of rho
// (r fastest) and shared-memory accesses are contiguous across a warp.  A real
// sequence of length N is packed as z_n = x_2n + i x_2n+1 (n < M = N/2),
// transformed by an in-place radix-2 decimation-in-time FFT of length M in
// shared memory (bit-reversed load), and unpacked into the N/2+1 half-spectrum.
// The CTA's output is the contiguous mode-layout block of cells
// (k, i0 .. i0+TI-1), staged in shared memory and stored with coalesced writes.
// Problems of a batch may differ in size and N_theta; the dynamic shared
// memory is sized for the largest.
//
// Fixed point.  In binary64 the transforms were bound by the FP64 unit (89 %
// busy, 12 % of the bandwidth); every value between the conversions is a 64-bit
// integer instead (fixed.h).  A column's scale is set by the sum of its inputs'
// magnitudes, which bounds every intermediate value: the largest integer stays
// below 2^61 and one unit lies 2^-61 of that sum away -- for 128 inputs of equal
// size 2^-54 of one of them -- and additions round nothing.  Against a
// quadruple-precision transform of 8 to 256 points (plasma charge, smooth, spiked
// and near-constant columns) the results are within 4.6e-17 to 6.1e-17 forward
// and 1.3e-17 to 1.2e-16 inverse (relative L2), where binary64 butterflies had
// 8.1e-17 to 2.7e-16 both ways.  A butterfly is 16 integer multiply-adds and
// some 30 other integer instructions instead of six binary64 multiply-adds, 384
// issue slots of a scheduler.  Each thread applies two consecutive radix-2 stages to four
// values held in registers, halving the shared-memory round trips and barriers;
// the unpack (pack) of the real transform treats modes m and M - m together,
// sharing one twiddle product.  A column that holds an infinity or a NaN comes
// out as NaN; one of values near or below the normal range is scaled up first, and
// results below it are rounded to subnormals.
// The modes take the place of the transform's rows (X_M a row of its own), so
// that 256 points need 68 KB of shared memory and not 133, three blocks per SM
// instead of one: 128 x 256 x 96 forward 81 -> 52 us, and a batch's largest problem
// no longer costs the others their room.
// 512 x 128 x 400: forward 586 -> 306 us (with b_hat and the norm, in a solve,
// 653 -> 346), inverse 496 -> 274 us; both now bound by integer instructions
// and their latency (ALU pipe 47 to 52 %, three CTAs per SM).
#include "fixed.h"
#include "internal.h"

namespace pp {
namespace {

constexpr int TI = FFT_TI;
constexpr int LD = TI + 1;   // padded row of the transform buffer (conflict-free 16-byte lanes)
constexpr int NW = FFT_THREADS / 32;
// A column whose largest exponent field is below SMALL is scaled by 2^UP first (by
// integers: a column of zeros comes here too): beside larger values a subnormal is
// less than a unit of the column, so that the conversions take it for 0.
constexpr int SMALL = 64, UP = 128;
__device__ __noinline__ double2 scaled_up(double2 v) {
    double *x = &v.x;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const ufx b = (ufx)__double_as_longlong(x[i]), m = b & ~(1ull << 63);
        if (m == 0) continue;
        const int lz = __clzll((fx)m) - 11;      // of a subnormal: to bit 52
        const ufx r = m >> 52 ? b + ((ufx)UP << 52) : ((m << (lz & 63)) & ~(1ull << 52)) + ((ufx)(UP + 1 - lz) << 52) + (b & (1ull << 63));
        x[i] = __longlong_as_double((fx)r);
    }
    return v;
}
__device__ __forceinline__ void scale_up(double2 *e) {
    const double2 v = *e;
    if (((ufx)__double_as_longlong(v.x) | (ufx)__double_as_longlong(v.y)) << 1) *e = scaled_up(v);
}

template <int LG> __device__ __forceinline__ int bitrev(int n) {
    return LG == 0 ? 0 : (int)(__brev((unsigned)n) >> (32 - LG));
}

__device__ __forceinline__ int find_problem(const unsigned *__restrict__ start, int n, unsigned blk) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (start[mid] <= blk) lo = mid;
        else hi = mid;
    }
    return lo;
}

struct ci {
    fx x, y;
};

// w = e^{-i theta} (INVERSE: e^{+i theta}) as limbs of cos, -sin and +sin.
struct Tw {
    Limbs c, s, n;
};
template <bool INVERSE> __device__ __forceinline__ Tw twiddle(const int4 *__restrict__ tw, int t) {
    const int4 u = tw[2 * t], v = tw[2 * t + 1];
    const Limbs minus = {u.z, u.w}, plus = {v.x, v.y};   // -sin, +sin
    return {{u.x, u.y}, INVERSE ? plus : minus, INVERSE ? minus : plus};
}
// w z; |z| < 2^61 in either part
__device__ __forceinline__ ci tw_mul(const Tw &w, ci z) {
    return {fx_mul2(z.x, w.c, z.y, w.n), fx_mul2(z.y, w.c, z.x, w.s)};
}

__device__ __forceinline__ void add_sub(ci &a, ci &b) {
    const ci x = a;
    a = {x.x + b.x, x.y + b.y};
    b = {x.x - b.x, x.y - b.y};
}
// (top, bot) <- (top + w bot, top - w bot)
__device__ __forceinline__ void bfly(ci &top, ci &bot, const Tw &w) {
    bot = tw_mul(w, bot);
    add_sub(top, bot);
}
template <bool INVERSE> __device__ __forceinline__ ci quarter(ci z) {   // times -i (inverse: +i)
    return INVERSE ? ci{-z.y, z.x} : ci{z.y, -z.x};
}

__device__ __forceinline__ ci ld(const double2 *p) {
    const longlong2 v = *reinterpret_cast<const longlong2 *>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ void st(double2 *p, ci z) { *reinterpret_cast<longlong2 *>(p) = make_longlong2(z.x, z.y); }

// In-place radix-2 DIT FFT of length M on buf[M][LD] (bit-reversed input),
// two stages (h, 2h) per pass on four values per thread.  The first pass
// (or the first single stage when log2 M is odd) has twiddles 1 and -i only
// and is done with additions.  INVERSE: conjugated twiddles.  tw: e^{-2 pi i
// t / 2M}.  A warp's lanes hold columns, so its twiddles are uniform.
template <bool INVERSE, int LG>
__device__ __forceinline__ void fft_stages(double2 *buf, const int4 *__restrict__ tw, int lane, int warp) {
    constexpr int M = 1 << LG;
    if constexpr (LG & 1) {   // single stage h = 1
#pragma unroll
        for (int q0 = 0; q0 < (M >> 1); q0 += NW) {
            const int q = q0 + warp;
            if ((M >> 1) % NW && q >= (M >> 1)) break;
            double2 *x = buf + 2 * q * LD + lane;
            ci a = ld(x), b = ld(x + LD);
            add_sub(a, b);
            st(x, a);
            st(x + LD, b);
        }
    } else if constexpr (M >= 4) {   // stages 1 and 2: four-point DFTs
#pragma unroll
        for (int q0 = 0; q0 < (M >> 2); q0 += NW) {
            const int q = q0 + warp;
            if ((M >> 2) % NW && q >= (M >> 2)) break;
            double2 *x = buf + 4 * q * LD + lane;
            ci a0 = ld(x), a1 = ld(x + LD), a2 = ld(x + 2 * LD), a3 = ld(x + 3 * LD);
            add_sub(a0, a1);
            add_sub(a2, a3);
            add_sub(a0, a2);
            a3 = quarter<INVERSE>(a3);
            add_sub(a1, a3);
            st(x, a0);
            st(x + LD, a1);
            st(x + 2 * LD, a2);
            st(x + 3 * LD, a3);
        }
    }
    __syncthreads();
#pragma unroll
    for (int h = LG & 1 ? 2 : 4; 4 * h <= M; h <<= 2) {
#pragma unroll 2
        for (int q0 = 0; q0 < (M >> 2); q0 += NW) {
            const int q = q0 + warp;
            if ((M >> 2) % NW && q >= (M >> 2)) break;
            const int p = q & (h - 1);
            const int g = (q - p) << 2;   // (q / h) * 4h
            double2 *x = buf + (g + p) * LD + lane;
            ci a0 = ld(x), a1 = ld(x + h * LD), a2 = ld(x + 2 * h * LD), a3 = ld(x + 3 * h * LD);
            const Tw w1 = twiddle<INVERSE>(tw, p * (M / h));          // W_{2h}^p
            bfly(a0, a1, w1);
            bfly(a2, a3, w1);
            const Tw w2 = twiddle<INVERSE>(tw, p * (M / (2 * h)));    // W_{4h}^p; W_{4h}^{p+h} = -i (+i) times it
            bfly(a0, a2, w2);
            a3 = quarter<INVERSE>(tw_mul(w2, a3));
            add_sub(a1, a3);
            st(x, a0);
            st(x + h * LD, a1);
            st(x + 2 * h * LD, a2);
            st(x + 3 * h * LD, a3);
        }
        __syncthreads();
    }
}

// Bounds of a column (lane) over the block's warps: the largest exponent
// field, then the bits bl of the sum of magnitudes in units of 2^(em - 1043),
// sum < 2^bl of them.  HALVES: of the larger of the two sums over the even and
// the odd warps.  w: [FFT_THREADS / 32][32] words of shared memory each.
__device__ __forceinline__ int column_max(int v, int *w, int lane, int warp) {
    w[warp * 32 + lane] = v;
    __syncthreads();
    int m = 0;
#pragma unroll
    for (int q = 0; q < NW; ++q) m = max(m, w[q * 32 + lane]);
    return m;
}
__device__ __forceinline__ unsigned magnitude(double x, int em) {
    return ((((unsigned)__double2hiint(x) & 0xfffffu) | 0x100000u) >> min(em - f64_exp(x), 31)) + 1u;
}
template <bool HALVES> __device__ __forceinline__ int column_bits(unsigned v, int *w, int lane, int warp) {
    w[warp * 32 + lane] = (int)v;
    __syncthreads();
    unsigned s0 = 0, s1 = 0;
#pragma unroll
    for (int q = 0; q < NW; q += 2) {
        s0 += (unsigned)w[q * 32 + lane];
        s1 += (unsigned)w[q * 32 + 32 + lane];
    }
    return 32 - __clz((int)(HALVES ? max(s0, s1) : s0 + s1));
}

// Sum of v over the block, valid in thread 0; sh holds blockDim doubles.  The
// values go through shared memory and one warp adds them, so the reduction
// issues about blockDim/32 + 5 FP64 additions per block instead of 5 per
// thread.
__device__ __forceinline__ double block_sum(double v, double *sh) {
    __syncthreads();   // a previous reduction may still be reading sh
    sh[threadIdx.x] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        for (int j = threadIdx.x; j < (int)blockDim.x; j += 32) s += sh[j];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

// f(entry, mode, column) for this thread's entries of a block of n entries, mode fastest
// (the division by nm is carried along).
template <int nm, class F> __device__ __forceinline__ void entries(int n, F f) {
    constexpr int dm = FFT_THREADS % nm, dc = FFT_THREADS / nm;
    int m = (int)threadIdx.x % nm, c = (int)threadIdx.x / nm;
    for (int e = threadIdx.x; e < n; e += FFT_THREADS) {
        f(e, m, c);
        m += dm;
        c += dc;
        if (m >= nm) {
            m -= nm;
            ++c;
        }
    }
}

// LG = log2 M: the loops' bounds and the shared-memory offsets are constants.
template <int LG>
__device__ __forceinline__ void forward_body(const FFTProb &P, int lb, double2 *sm, double *red, int *wmax, int *wsum,
                                             double *__restrict__ partials) {
    constexpr int M = 1 << LG, nt = 2 * M, nm = M + 1;
    const int nr = P.nr, nz = P.nz;
    double2 *buf = sm;              // [M + 1][LD]

    const int tiles = (nr + TI - 1) / TI;
    const int k = lb / tiles;
    const int i0 = (lb - k * tiles) * TI;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = i0 + lane;
    const bool valid = i < nr;

    const double *src = P.rho + (size_t)k * nt * nr + i;
    int em = 0;
#pragma unroll 4
    for (int n = warp; n < M; n += NW) {
        double a = 0.0, b = 0.0;
        if (valid) {
            a = src[(size_t)(2 * n) * nr];
            b = src[(size_t)(2 * n + 1) * nr];
        }
        em = max(em, max(f64_exp(a), f64_exp(b)));
        buf[bitrev<LG>(n) * LD + lane] = make_double2(a, b);
    }
    em = column_max(em, wmax, lane, warp);
    int down = 0;
    if (em < SMALL && valid) {   // (values that may be subnormal: brought into the normal range)
        for (int n = warp; n < M; n += NW) {
            double2 *e = buf + bitrev<LG>(n) * LD + lane;
            scale_up(e);
        }
        down = UP;
        em = max(em, 1) + UP;
    }
    unsigned mag = 0;
#pragma unroll 4
    for (int n = warp; n < M; n += NW) {   // (a thread's own entries: no barrier between these passes)
        const double2 v = buf[bitrev<LG>(n) * LD + lane];
        mag += magnitude(v.x, em) + magnitude(v.y, em);
    }
    const int bl = column_bits<false>(mag, wsum, lane, warp);
#pragma unroll 4
    for (int n = warp; n < M; n += NW) {
        double2 *e = buf + bitrev<LG>(n) * LD + lane;
        const double2 v = *e;
        // sum of magnitudes < 2^61
        st(e, {f64_to_fx(v.x, em - f64_exp(v.x) + bl - 19), f64_to_fx(v.y, em - f64_exp(v.y) + bl - 19)});
    }
    __syncthreads();
    fft_stages<false, LG>(buf, P.tw, lane, warp);

    // Unpack, modes m and M - m together (W = e^{-2 pi i / N}, hs = s_i / (2N)):
    //   S = Z_m + conj Z_{M-m},  D = Z_m - conj Z_{M-m},  T = W^m D,
    //   X_m = hs (S - i T),  X_{M-m} = hs conj(S + i T);
    // X_0 = 2 hs (Re Z_0 + Im Z_0), X_M = 2 hs (Re Z_0 - Im Z_0), both exactly real.
    // |S - i T| = 2 |sum of the inputs times roots of unity| < 2^62; D is halved
    // for the product.  hs multiplies as a 63-bit mantissa.  In place: a pair's rows
    // are read and written by one thread, X_M takes the row after the last.
    // s_i, or per cell in a composite domain (zero outside its patches)
    const size_t si = valid ? (P.s_rows ? (size_t)k * nr + i : (size_t)i) : 0;
    const double hs = (P.s ? P.s[si] : 1.0) * P.half_inv_n;
    const fx hm = f64_exp(hs) ? (hs < 0.0 ? -(fx)f64_mant(hs) : (fx)f64_mant(hs)) : 0;
    const int be = em == 0x7ff ? FX_NAN : em - down + bl - 18 + f64_exp(hs) - 1021;   // biased exponent of r hm = 2^63 2^64
    const bool rare = fx_rare(be);
    auto out = [&](fx r, int e) { return fx_to_f64(__mul64hi(r, hm), e, rare); };
    double acc_in = 0.0, acc_edge = 0.0;   // Parseval weight 2 (0 < m < M) and 1 (m = 0, M)
    double2 *ob = buf + lane;
    for (int m = 1 + warp; 2 * m < M; m += NW) {
        const ci A = ld(buf + m * LD + lane), B = ld(buf + (M - m) * LD + lane);
        const ci S = {A.x + B.x, A.y - B.y};
        const ci T = tw_mul(twiddle<false>(P.tw, m), {(A.x - B.x) >> 1, (A.y + B.y) >> 1});   // W^m D / 2
        const double2 xm = make_double2(out(S.x + 2 * T.y, be), out(S.y - 2 * T.x, be));
        const double2 xp = make_double2(out(S.x - 2 * T.y, be), out(-S.y - 2 * T.x, be));
        ob[m * LD] = xm;
        ob[(M - m) * LD] = xp;
        acc_in = fma(xm.x, xm.x, fma(xm.y, xm.y, acc_in));
        acc_in = fma(xp.x, xp.x, fma(xp.y, xp.y, acc_in));
    }
    if (warp == 0) {
        const ci z = ld(buf + lane);
        double x0 = out(z.x + z.y, be + 1);
        const double xM = out(z.x - z.y, be + 1);
        if (P.bD && valid) x0 += P.bD[(size_t)k * nr + i];
        acc_edge = fma(x0, x0, fma(xM, xM, acc_edge));
        ob[0] = make_double2(x0, 0.0);
        ob[M * LD] = make_double2(xM, 0.0);
    }
    if (M >= 2 && warp == NW - 1) {   // m = M/2 pairs with itself: X = 2 hs conj Z
        const ci z = ld(buf + (M >> 1) * LD + lane);
        const double2 x = make_double2(out(z.x, be + 1), out(-z.y, be + 1));
        ob[(M >> 1) * LD] = x;
        acc_in = fma(x.x, x.x, fma(x.y, x.y, acc_in));
    }
    __syncthreads();
    const int ncols = min(TI, nr - i0);
    double2 *dst = P.b + ((size_t)k * nr + i0) * nm;
    entries<nm>(ncols * nm, [&](int f, int m, int c) { dst[f] = buf[m * LD + c]; });
    if (P.bh && P.invd) {
        // b_hat = b / diag for the smoother (row class of plane k, cells i0.., all modes)
        const int cls = P.rcls ? P.rcls[k] : (k == 0 ? 0 : (k == nz - 1 ? P.ncls - 1 : 1));
        const double *inv = P.invd + ((size_t)cls * nr + i0) * nm;
        double2 *dh = P.bh + ((size_t)k * nr + i0) * nm;
        entries<nm>(ncols * nm, [&](int f, int m, int c) {
            const double2 x = buf[m * LD + c];
            const double v = inv[f];
            dh[f] = make_double2(x.x * v, x.y * v);
        });
    }
    if (partials) {
        const double tot = block_sum(valid ? fma(2.0, acc_in, acc_edge) : 0.0, red);
        if (threadIdx.x == 0) partials[blockIdx.x] = tot;
    }
}

template <int LG>
__device__ __forceinline__ void inverse_body(const FFTProb &P, int lb, double2 *sm, int *wmax, int *wsum) {
    constexpr int M = 1 << LG, nt = 2 * M, nm = M + 1;
    const int nr = P.nr;
    double2 *buf = sm;              // [M + 1][LD]: X_m, then Z_m, in row(m)
    auto row = [](int m) { return (m == M ? M : bitrev<LG>(m)) * LD; };

    const int tiles = (nr + TI - 1) / TI;
    const int k = lb / tiles;
    const int i0 = (lb - k * tiles) * TI;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = i0 + lane;
    const bool valid = i < nr;
    const int ncols = min(TI, nr - i0);

    const double2 *src = P.uhat + ((size_t)k * nr + i0) * nm;
    entries<nm>(TI * nm, [&](int f, int m, int c) { buf[row(m) + c] = f < ncols * nm ? src[f] : make_double2(0.0, 0.0); });
    __syncthreads();

    // The column's bounds; X_0 and X_M enter through their real parts only.
    const double2 *ib = buf + lane;
    int em = 0;
    for (int m = warp; m <= M; m += NW) {
        const double2 x = ib[row(m)];
        em = max(em, max(f64_exp(x.x), m == 0 || m == M ? 0 : f64_exp(x.y)));
    }
    em = column_max(em, wmax, lane, warp);
    int down = 0;
    if (em < SMALL && valid) {   // (as in the forward transform; column_bits has a barrier)
        for (int m = warp; m <= M; m += NW) {
            double2 *e = buf + row(m) + lane;
            scale_up(e);
        }
        down = UP;
        em = max(em, 1) + UP;
    }
    unsigned mag = 0;
    for (int m = warp; m <= M; m += NW) {
        const double2 x = ib[row(m)];
        mag += magnitude(x.x, em) + (m == 0 || m == M ? 0u : magnitude(x.y, em));
    }
    const int bl = column_bits<true>(mag, wsum, lane, warp);
    // Sums of magnitudes of the even and of the odd modes < 2^59 (a warp's modes
    // have its parity, and so do m and M - m): the packed values of one parity and
    // their partial sums, all that a twiddle multiplies, stay below 2^61, the
    // last stage's sums of both below 2^62.
    auto in = [&](double v) { return f64_to_fx(v, em - f64_exp(v) + bl - 17); };

    // Pack, modes m and M - m together (w = e^{+2 pi i / N}):
    //   S = X_m + conj X_{M-m},  D = X_m - conj X_{M-m},  T = w^m D,
    //   Z_m = S + i T,  Z_{M-m} = conj(S - i T);
    // Z_0 = (X_0 + X_M) + i (X_0 - X_M).
    for (int m = 1 + warp; 2 * m < M; m += NW) {
        const double2 a = ib[row(m)], b = ib[row(M - m)];
        const ci A = {in(a.x), in(a.y)}, B = {in(b.x), in(b.y)};
        const ci S = {A.x + B.x, A.y - B.y};
        const ci T = tw_mul(twiddle<true>(P.tw, m), {A.x - B.x, A.y + B.y});
        st(buf + row(m) + lane, {S.x - T.y, S.y + T.x});
        st(buf + row(M - m) + lane, {S.x + T.y, T.x - S.y});
    }
    if (warp == 0) {
        const fx a = in(ib[0].x), b = in(ib[row(M)].x);
        st(buf + lane, {a + b, a - b});
    }
    if (M >= 2 && warp == NW - 1) {   // m = M/2 pairs with itself: Z = 2 conj X
        const double2 x = ib[row(M >> 1)];
        st(buf + row(M >> 1) + lane, {2 * in(x.x), -2 * in(x.y)});
    }
    __syncthreads();
    fft_stages<true, LG>(buf, P.tw, lane, warp);

    if (valid) {
        const int be = em == 0x7ff ? FX_NAN : em - down + bl - 16;
        const bool rare = fx_rare(be);
        double *dst = P.phi + (size_t)k * nt * nr + i;
#pragma unroll 4
        for (int n = warp; n < M; n += NW) {
            const ci z = ld(buf + n * LD + lane);
            dst[(size_t)(2 * n) * nr] = fx_to_f64(z.x, be, rare);
            dst[(size_t)(2 * n + 1) * nr] = fx_to_f64(z.y, be, rare);
        }
    }
}

// One instantiation per azimuthal size of a batch's problems.
#define PP_FFT_SWITCH(CALL)            \
    switch (P.log2M) {                 \
    case 0: CALL(0); break;            \
    case 1: CALL(1); break;            \
    case 2: CALL(2); break;            \
    case 3: CALL(3); break;            \
    case 4: CALL(4); break;            \
    case 5: CALL(5); break;            \
    case 6: CALL(6); break;            \
    default: CALL(7); break;           \
    }

__global__ void __launch_bounds__(FFT_THREADS, 3) k_forward(const FFTTab *__restrict__ tab, double *__restrict__ partials) {
    extern __shared__ double2 sm[];
    __shared__ double red[FFT_THREADS];
    __shared__ int wmax[FFT_THREADS], wsum[FFT_THREADS];
    const int pr = find_problem(tab->start, tab->n, blockIdx.x);
    const FFTProb P = tab->p[pr];
    const int lb = (int)(blockIdx.x - tab->start[pr]);
#define PP_CALL(LG) forward_body<LG>(P, lb, sm, red, wmax, wsum, partials)
    PP_FFT_SWITCH(PP_CALL)
#undef PP_CALL
}

__global__ void __launch_bounds__(FFT_THREADS, 3) k_inverse(const FFTTab *__restrict__ tab) {
    extern __shared__ double2 sm[];
    __shared__ int wmax[FFT_THREADS], wsum[FFT_THREADS];
    const int pr = find_problem(tab->start, tab->n, blockIdx.x);
    const FFTProb P = tab->p[pr];
    const int lb = (int)(blockIdx.x - tab->start[pr]);
#define PP_CALL(LG) inverse_body<LG>(P, lb, sm, wmax, wsum)
    PP_FFT_SWITCH(PP_CALL)
#undef PP_CALL
}

// Mode-layout initial iterate: b = guess, each CTA copying the cells of its
// plane k and radial tile (the same block ranges as the transforms).
__global__ void __launch_bounds__(FFT_THREADS) k_copy_guess(const FFTTab *__restrict__ tab) {
    const int pr = find_problem(tab->start, tab->n, blockIdx.x);
    const FFTProb P = tab->p[pr];
    const int nm = P.nt / 2 + 1;
    const int tiles = (P.nr + TI - 1) / TI;
    const int lb = (int)(blockIdx.x - tab->start[pr]);
    const int k = lb / tiles;
    const int i0 = (lb - k * tiles) * TI;
    const int ncols = min(TI, P.nr - i0);
    const size_t off = ((size_t)k * P.nr + i0) * nm;
    for (int f = threadIdx.x; f < ncols * nm; f += blockDim.x) P.b[off + f] = P.guess[off + f];
}

}  // namespace

cudaError_t launch_copy_guess(const FFTTab *tab, unsigned grid, cudaStream_t st) {
    k_copy_guess<<<grid, FFT_THREADS, 0, st>>>(tab);
    return cudaGetLastError();
}

size_t fft_smem_bytes(int nt) {
    return (size_t)(nt / 2 + 1) * LD * sizeof(double2);
}

cudaError_t launch_forward(const FFTTab *tab, unsigned grid, size_t smem, double *partials, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fft_smem_bytes(kMaxNtheta));
    if (e != cudaSuccess) return e;
    k_forward<<<grid, FFT_THREADS, smem, st>>>(tab, partials);
    return cudaGetLastError();
}

cudaError_t launch_inverse(const FFTTab *tab, unsigned grid, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fft_smem_bytes(kMaxNtheta));
    if (e != cudaSuccess) return e;
    k_inverse<<<grid, FFT_THREADS, smem, st>>>(tab);
    return cudaGetLastError();
}

}  // namespace pp
