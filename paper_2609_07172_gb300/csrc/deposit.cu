// Cloud-in-cell deposit of macro-particles to the cell-corner nodes and the
// projection of nodal density to cell-centred charge: the steps before the
// Poisson solve in the paper's particle-in-cell cycle (Sec. 2, and Sec.
// "Warp-aggregated cylindrical CIC deposition", Eqs. cic_weights,
// particle_cic_update, warp_aggregated_cic).
//
// Deposit.  A particle in cell (i, j, k) at normalised position (xi, eta,
// zeta) adds W w_r w_alpha w_z / V_nu to each of the cell's eight corner
// nodes (w^(0) = 1 - t, w^(1) = t; V_nu the node's cylindrical control
// volume, from cell centre to cell centre in r and z and cut at the walls, a
// full dalpha in alpha).  Aggregation (Eq. warp_aggregated_cic): a thread first
// sums its consecutive particles that share a cell; then lanes whose last
// cells agree -- runs of equal cell labels in lane order, which cell-sorted
// input makes long -- add their sums with a segmented scan of register
// shuffles; a run whose cell is the radial neighbour of the run before it takes
// over that run's four outer corners (the same nodes), across the warps of the
// block too; and the last lane of each run issues the run's FP64 atomic
// additions, each divided by the node's volume once: four per cell of sorted
// input instead of eight.  Particles outside the domain deposit nothing.
//
// Fixed point.  The FP64 unit (1/64 of the FP32 rate) bound this kernel: about
// 23 of its instructions per particle for the position and 16 per cell for the
// corners, 5.8 of the 5.8 ms per 105 M particles.  Offsets in the cell (64 fraction
// bits), their products and every sum are 64-bit integers instead (units of 2^-61): a
// cell's particles are summed as the eight moments 1, x, y, z, xy, xz, yz, xyz --
// sums that round nothing -- and the corner weights follow from them by exact
// subtractions.  Their error is absolute, three units per particle; a run with a
// corner sum below 2^47 units per particle (2^-14 of one; 2 to 3 % of single particles
// of a uniform density, one in 10^8 of four) goes to the nodes particle by particle
// in binary64, so that every weight holds 2^-45 of itself as double-float
// products did.  The position goes to a cell and an offset by one 64-bit
// multiplication; a particle near a cell boundary (2^-24 of a cell) or outside takes
// the binary64 arithmetic, which alone decides those cases, and one whose
// coordinate has bits below the fixed point's, close to the lower wall, takes that too.
// 210 M cell-sorted particles of two species, 4 per cell and species, at
// 512 x 128 x 400: 11.6 ms with double-float, now 2.5 (integer instructions and their
// issue, both two thirds busy).  In units of 2^-54 without the second way it was 2.3, but
// a weight of 1e-12 kept four digits; 96-bit products hold every weight without it and
// took 3.1.  Against a quadruple-precision deposit of 1.6 M particles the nodes are
// within 5.6e-14 (L2), all forms alike: the rounding of the node volumes.
//
// Non-uniform faces and composite domains (FACES): the cell comes
// from the face arrays (a bin lookup guesses, binary64 comparisons decide),
// the offsets from the cell's own faces; in a composite domain (Sec. 2.2) a
// particle in an inactive cell deposits nothing and a node's volume counts
// only its octants in active cells, so the projection below conserves the
// active cells' charge; inactive cells get rho = 0.
//
// Projection (Sec. 2, "volume-consistent projection to cell-centred
// charge"; the paper gives no formula -- the reading): each node's control
// volume is split into the octants inside its adjacent cells and an
// octant's charge goes to its cell, rho_q = charge * sum over the corners of
// q of n_nu V_(nu in q) / V_q.  The radial octant share is the exact r dr
// integral of the half cell (f_lo, f_hi below, f_lo + f_hi = 1), the
// azimuthal and axial ones are 1/2; so charge is conserved exactly:
// sum_q rho_q V_q = charge * sum_nu n_nu V_nu.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "plan.h"

namespace pp {
namespace {

typedef unsigned long long u64;

// One uniform axis in fixed point: x -> X = x 2^(62 - E) (|x| < 2^E over the
// domain), D = X - base in [0, span), and D 2^sh K / 2^64 = the position in
// cells with F fraction bits, the product's low word giving the bits below.
// K is cut by less than 2^-62 of it, and so is the position.  X is exact for
// |x| >= 2^(E - 10); below, or where the wall is cut, D is off by up to two units.
struct FixAxis {
    long long base;
    u64 span, K;
    int e1;                 // E + 1023
    int smax;               // shift up to which X is exact (0: the wall is cut)
    int sh, F;
};

struct DepositArgs {
    int nr, nt, nz;
    long long np;
    double r_in, z0, inv_dr, inv_da, inv_dz;
    FixAxis fr, fa, fz;
    double weight;
    int vec;                // the arrays allow 16-byte loads
    const double *r, *al, *z;
    const double *inv_vr;   // [nr + 1] 1 / (radial integral of r dr of node a's interval)
    const double *inv_vz;   // [nz + 1] 1 / (dalpha * axial length of node c's interval)
    double *nodes;          // (nz + 1, nt, nr + 1)
};

// Non-uniform faces or a composite domain: the cell is found
// on the face arrays -- a lookup bin guesses it, exact comparisons settle it.
struct DepositGeo {
    const double *rf, *zf;          // faces [nr + 1], [nz + 1]
    const double *inv_wr, *inv_wz;  // 1 / cell widths
    const int *rbin, *zbin;         // cell at the lower end of each bin
    int nrbin, nzbin;
    float r0f, z0f, inv_rbw, inv_zbw;
    const unsigned char *act;       // composite: active flags [nz][nr] (null: all active)
    const double *inv_v2;           // composite: 1 / node volumes of active octants [nz + 1][nr + 1]
};

// Cell of coordinate x on faces f[0..n] (max{a : f[a] <= x}), or -1 outside
// [f[0], f[n]).  The binary32 bin lookup only guesses; the binary64
// comparisons against the faces decide, so the cell is exactly the one the
// face array defines (a guess off by any amount still ends right, the loops
// are bounded by n).
__device__ __forceinline__ int find_cell(double x, const double *f, int n, const int *bin, int nbin, float x0,
                                         float inv_bw) {
    if (!(x >= f[0] && x < f[n])) return -1;   // NaN included
    int b = (int)(((float)x - x0) * inv_bw);
    b = b < 0 ? 0 : (b >= nbin ? nbin - 1 : b);
    int a = bin[b];
    while (a > 0 && x < f[a]) --a;
    while (a < n - 1 && x >= f[a + 1]) ++a;
    return a;
}

constexpr int DEP_PPT = 4;   // consecutive particles per thread
constexpr int DEP_THREADS = 256;
constexpr u64 DEP_NEAR = 1ull << 48;   // least D of a coordinate or wall that is cut

// A particle in its cell: indices and offsets, 64 fraction bits.
struct Place {
    int ir, ia, iz;
    u64 x, y, z;
};
// The same with binary64 offsets.
struct Spot {
    int ir, ia, iz;
    double x, y, z;
};

// A binary64 offset in [0, 1] as a 64-bit fraction (cut; 1 becomes 1 - 2^-64).
__device__ __forceinline__ u64 frac64(double f) {
    const unsigned hi = (unsigned)__double2hiint(f), lo = (unsigned)__double2loint(f);
    const int s = 1022 - (int)((hi >> 20) & 0x7ffu);   // 0 for [1/2, 1)
    if (s < 0) return ~0ull;
    if (s > 63) return 0ull;
    return ((((u64)((hi & 0xfffffu) | 0x100000u)) << 32 | lo) << 11) >> s;
}

// Cell and offset of x on a uniform axis; false where the binary64 arithmetic
// has to decide (outside, not finite, within 2^-24 of a cell boundary) or keeps
// more of the offset (`near` above: close to the lower wall).
__device__ __forceinline__ bool fix_place(const FixAxis &a, double x, int &cell, u64 &f) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int s = a.e1 - ((hi >> 20) & 0x7ff);
    u64 X = ((((u64)((hi & 0xfffff) | 0x100000)) << 32 | lo) << 10) >> min(max(s, 0), 63);
    if (hi < 0) X = 0ull - X;
    const u64 D = X - (u64)a.base, d = D << a.sh;
    const u64 t = __umul64hi(d, a.K);
    cell = (int)(t >> a.F);
    f = t << (64 - a.F) | (unsigned)((d * a.K) >> 32) >> (a.F - 32);   // (the low word's upper half: F >= 32, n < 2^30)
    return s >= 1 && D < a.span && (s <= a.smax || D >= DEP_NEAR) && (unsigned)(f >> 32) + 0x100u >= 0x200u;
}

// Cell and offsets of particle (r, al, z) by binary64 arithmetic; false when
// it is outside.
__device__ __forceinline__ bool locate(const DepositArgs &a, double r, double al, double z, Spot &q) {
    const double tr = (r - a.r_in) * a.inv_dr, ta = al * a.inv_da, tz = (z - a.z0) * a.inv_dz;
    const double fr = floor(tr), fa = floor(ta), fz = floor(tz);
    // in range before any conversion (NaN compares false)
    if (!(fr >= 0.0 && fr < (double)a.nr && fa >= 0.0 && fa < (double)a.nt && fz >= 0.0 && fz < (double)a.nz))
        return false;
    q = {(int)fr, (int)fa, (int)fz, tr - fr, ta - fa, tz - fz};   // exact differences, in [0, 1)
    return true;
}

// The same on face arrays; false also for a particle in an inactive cell.
__device__ __forceinline__ bool locate_faces(const DepositArgs &a, const DepositGeo &g, double r, double al, double z,
                                             Spot &q) {
    const double ta = al * a.inv_da, fa = floor(ta);
    if (!(fa >= 0.0 && fa < (double)a.nt)) return false;
    q.ir = find_cell(r, g.rf, a.nr, g.rbin, g.nrbin, g.r0f, g.inv_rbw);
    q.iz = find_cell(z, g.zf, a.nz, g.zbin, g.nzbin, g.z0f, g.inv_zbw);
    if (q.ir < 0 || q.iz < 0) return false;
    if (g.act && !g.act[(size_t)q.iz * a.nr + q.ir]) return false;   // inactive cell: nothing deposited
    q.ia = (int)fa;
    // the products may round to 1 at the upper face; the weights stay in [0, 1]
    q.x = fmin((r - g.rf[q.ir]) * g.inv_wr[q.ir], 1.0);
    q.y = ta - fa;
    q.z = fmin((z - g.zf[q.iz]) * g.inv_wz[q.iz], 1.0);
    return true;
}

// One particle's eight weights in binary64 straight to the nodes (21 FP64
// instructions beside the atomics).
template <bool V2D> __device__ __forceinline__ void spread(const DepositArgs &a, const double *inv_v2, const Spot &q) {
    const int ja = q.ia + 1 == a.nt ? 0 : q.ia + 1;
    const size_t rs = (size_t)a.nr + 1, ps = (size_t)a.nt * rs;
    const double w0 = 1.0 - q.y, wr[2] = {1.0 - q.x, q.x}, wz[2] = {1.0 - q.z, q.z};
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        const int nri = q.ir + d;
        const double f = V2D ? a.weight * wr[d] : a.weight * a.inv_vr[nri] * wr[d];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int nzi = q.iz + e;
            const double g = f * (V2D ? inv_v2[(size_t)nzi * rs + nri] * wz[e] : a.inv_vz[nzi] * wz[e]);
            double *p = a.nodes + (size_t)nzi * ps + nri;
            atomicAdd(p + (size_t)q.ia * rs, g * w0);
            atomicAdd(p + (size_t)ja * rs, g * q.y);
        }
    }
}
// Particle p by itself.
template <bool FACES, bool V2D> __device__ __noinline__ void stray(const DepositArgs &a, const DepositGeo &g, long long p) {
    Spot q;
    if (FACES ? locate_faces(a, g, a.r[p], a.al[p], a.z[p], q) : locate(a, a.r[p], a.al[p], a.z[p], q)) spread<V2D>(a, g.inv_v2, q);
}

// Moments of a cell's particles, the count apart.  A thread's (at most four) are in
// units of 2^-61; in a warp with a run over more than one lane all are cut to as many
// bits fewer as the longest run's sum needs.  Every sum stays below 2^63, two runs'
// below 2^64.
constexpr int DEP_UNIT = 61;
struct Moments {
    unsigned n;
    u64 m[7];   // x, y, z, xy, xz, yz, xyz
    __device__ __forceinline__ void clear() {
        n = 0;
#pragma unroll
        for (int e = 0; e < 7; ++e) m[e] = 0;
    }
    __device__ __forceinline__ void add(const Place &q) {
        constexpr int S = 64 - DEP_UNIT;
        const u64 y = q.y >> S, z = q.z >> S, yz = __umul64hi(q.y, z);
        ++n;
        m[0] += q.x >> S;
        m[1] += y;
        m[2] += z;
        m[3] += __umul64hi(q.x, y);
        m[4] += __umul64hi(q.x, z);
        m[5] += yz;
        m[6] += __umul64hi(q.x, yz);
    }
    // Corner sums (corner 4 dz + 2 dalpha + dr), each off by less than three units per
    // particle (four per lane where the moments are cut).  Returns whether every sum is
    // 2^47 units per particle or more, which makes that 2^-45 of it, the accuracy of
    // double-float products.
    __device__ __forceinline__ bool corners(u64 c[8], int unit) const {
        c[7] = m[6];
        c[3] = m[3] - m[6];
        c[5] = m[4] - m[6];
        c[6] = m[5] - m[6];
        c[1] = m[0] - m[3] - c[5];
        c[2] = m[1] - m[3] - c[6];
        c[4] = m[2] - m[4] - c[6];
        c[0] = ((u64)n << unit) - m[0] - c[2] - c[4] - c[6];
        int least = (int)(c[0] >> 32);
#pragma unroll
        for (int e = 1; e < 8; ++e) least = min(least, (int)(c[e] >> 32));
        return least >= (int)(n << 15);
    }
};

// The nearest binary64 value of c 2^-unit (integer instructions; the FP64 unit's
// conversion takes several of its slots).
__device__ __forceinline__ double to_f64(u64 c, int unit) {
    const int lz = __clzll((long long)c);
    const u64 m = c << (lz & 63);
    const u64 bits = ((u64)(unsigned)(1085 - unit - lz) << 52) + (m >> 11) + ((m >> 10) & 1u);
    return c ? __longlong_as_double((long long)bits) : 0.0;
}

// Add four corner sums to the nodes at radius index nri around cell (ia, iz):
// (alpha, z) = (0, 0), (1, 0), (0, 1), (1, 1).
template <bool V2D>
__device__ __forceinline__ void add4(const DepositArgs &a, const double *inv_v2, int unit, int nri, int ia, int iz, u64 c00,
                                     u64 c10, u64 c01, u64 c11) {
    const int ja = ia + 1 == a.nt ? 0 : ia + 1;
    const size_t rs = (size_t)a.nr + 1, ps = (size_t)a.nt * rs;
    double f0, f1;
    if (V2D) {   // composite domain: node volumes of active octants
        f0 = a.weight * inv_v2[(size_t)iz * rs + nri];
        f1 = a.weight * inv_v2[(size_t)(iz + 1) * rs + nri];
    } else {
        const double fr = a.weight * a.inv_vr[nri];
        f0 = fr * a.inv_vz[iz];
        f1 = fr * a.inv_vz[iz + 1];
    }
    double *p = a.nodes + (size_t)iz * ps + nri;
    atomicAdd(p + (size_t)ia * rs, to_f64(c00, unit) * f0);
    atomicAdd(p + (size_t)ja * rs, to_f64(c10, unit) * f0);
    atomicAdd(p + ps + (size_t)ia * rs, to_f64(c01, unit) * f1);
    atomicAdd(p + ps + (size_t)ja * rs, to_f64(c11, unit) * f1);
}

// FACES: face arrays or a composite domain; V2D: a composite domain.
//
// What a run's sums would not hold to 2^-45 goes to the nodes particle by particle
// in binary64: a run with a corner sum too small for its units, a particle that
// fix_place leaves to that arithmetic.  The block queues these and works on them
// together at its end -- an FP64 instruction of a warp holds the unit for 16
// cycles whether one lane needs it or all.
template <bool FACES, bool V2D>
__global__ void __launch_bounds__(DEP_THREADS) k_deposit(const __grid_constant__ DepositArgs a, const __grid_constant__ DepositGeo g) {
    constexpr int W = DEP_THREADS / 32;
    __shared__ long long s_first[W], s_last[W];   // labels of each warp's first and last lane
    __shared__ u64 s_hi[W][4];                    // outer corners of its last run
    __shared__ unsigned short s_queue[DEP_THREADS * DEP_PPT];
    __shared__ int s_queued;
    const long long b0 = (long long)blockIdx.x * (DEP_THREADS * DEP_PPT), t0 = b0 + (int)threadIdx.x * DEP_PPT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    if (threadIdx.x == 0) s_queued = 0;
    __syncthreads();
    auto queue = [&](unsigned mask) {             // of the thread's particles; a particle once
        while (mask) {
            const int t = __ffs((int)mask) - 1;
            mask &= mask - 1;
            s_queue[atomicAdd(&s_queued, 1)] = (unsigned short)(threadIdx.x * DEP_PPT + t);
        }
    };
    double pr[DEP_PPT], pa[DEP_PPT], pz[DEP_PPT];
    const int have_p = (int)min((long long)DEP_PPT, max(0ll, a.np - t0));
    if (a.vec && have_p == DEP_PPT) {
#pragma unroll
        for (int t = 0; t < DEP_PPT; t += 2) {
            const double2 u = __ldcs(reinterpret_cast<const double2 *>(a.r + t0 + t));
            const double2 v = __ldcs(reinterpret_cast<const double2 *>(a.al + t0 + t));
            const double2 w = __ldcs(reinterpret_cast<const double2 *>(a.z + t0 + t));
            pr[t] = u.x, pr[t + 1] = u.y, pa[t] = v.x, pa[t + 1] = v.y, pz[t] = w.x, pz[t + 1] = w.y;
        }
    } else {
#pragma unroll
        for (int t = 0; t < DEP_PPT; ++t)
            if (t < have_p) pr[t] = a.r[t0 + t], pa[t] = a.al[t0 + t], pz[t] = a.z[t0 + t];
    }
    Moments M;
    M.clear();
    int cr = 0, ca = 0, cz = 0;
    unsigned mine = 0, lone = 0;                  // particles of the current run, of the queue
    u64 c[8];
#pragma unroll
    for (int t = 0; t < DEP_PPT; ++t) {
        Place q;
        if (t >= have_p) continue;
        if constexpr (FACES) {
            Spot s;
            if (!locate_faces(a, g, pr[t], pa[t], pz[t], s)) continue;
            q = {s.ir, s.ia, s.iz, frac64(s.x), frac64(s.y), frac64(s.z)};
        } else if (!(fix_place(a.fr, pr[t], q.ir, q.x) & fix_place(a.fa, pa[t], q.ia, q.y) &
                     fix_place(a.fz, pz[t], q.iz, q.z))) {
            lone |= 1u << t;
            continue;
        }
        if (mine && (q.ir != cr || q.ia != ca || q.iz != cz)) {   // the finished run straight to the nodes
            if (M.corners(c, DEP_UNIT)) {
                add4<V2D>(a, g.inv_v2, DEP_UNIT, cr, ca, cz, c[0], c[2], c[4], c[6]);
                add4<V2D>(a, g.inv_v2, DEP_UNIT, cr + 1, ca, cz, c[1], c[3], c[5], c[7]);
            } else {
                lone |= mine;
            }
            M.clear();
            mine = 0;
        }
        cr = q.ir;
        ca = q.ia;
        cz = q.iz;
        mine |= 1u << t;
        M.add(q);
    }
    // runs of lanes with the same last cell (lanes with nothing left: a run each)
    const long long cell = mine ? ((long long)cz * a.nt + ca) * a.nr + cr : -1 - lane;
    const long long prev = __shfl_up_sync(full, cell, 1);
    const unsigned heads = __ballot_sync(full, lane == 0 || prev != cell);
    const unsigned upto = lane == 31 ? full : ((2u << lane) - 1u);
    const int start = 31 - __clz(heads & upto);   // first and last lane of this lane's run
    const int end = (heads & ~upto) ? __ffs((int)(heads & ~upto)) - 2 : 31;
    int unit = DEP_UNIT;                          // (the same for the whole warp)
    if (heads != full) {
        const int longest = (int)__reduce_max_sync(full, (unsigned)(lane - start)), cut = 32 - __clz(longest);
        unit -= cut;
#pragma unroll
        for (int e = 0; e < 7; ++e) M.m[e] >>= cut;
        for (int off = 1; off <= longest; off <<= 1) {
            const bool in = lane - off >= start;
            const unsigned yn = __shfl_up_sync(full, M.n, off);
            if (in) M.n += yn;
#pragma unroll
            for (int e = 0; e < 7; ++e) {
                const u64 y = __shfl_up_sync(full, M.m[e], off);
                if (in) M.m[e] += y;
            }
        }
    }
    const bool small = !M.corners(c, unit);
    if (__shfl_sync(full, small, end)) {          // (the run's sums are those of its last lane)
        lone |= mine;
        mine = 0;
    }
    if (lone) queue(lone);
    // the outer corners of the run before go to this run when its cell is the
    // radial neighbour (and its units are the same); the warps' ends meet through
    // shared memory
    const long long label = mine ? 64 * cell + unit : -2 - lane;
    const long long next = __shfl_down_sync(full, label, 1);
    if (lane == 0) s_first[warp] = label;
    if (lane == 31) {
        s_last[warp] = label;
#pragma unroll
        for (int e = 0; e < 4; ++e) s_hi[warp][e] = c[2 * e + 1];
    }
    __syncthreads();
    const int src = start > 0 ? start - 1 : 0;
    long long pl = __shfl_sync(full, label, src);
    u64 hi[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) hi[e] = __shfl_sync(full, c[2 * e + 1], src);
    if (start == 0) {
        pl = warp > 0 ? s_last[warp - 1] : -1;
#pragma unroll
        for (int e = 0; e < 4; ++e) hi[e] = s_hi[warp > 0 ? warp - 1 : 0][e];
    }
    if (mine && lane == end) {
        if (pl >= 0 && pl + 64 == label && cr > 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) c[2 * e] += hi[e];
        }
        add4<V2D>(a, g.inv_v2, unit, cr, ca, cz, c[0], c[2], c[4], c[6]);
        const long long nl = lane < 31 ? next : (warp + 1 < W ? s_first[warp + 1] : -1);
        if (!(nl == label + 64 && cr + 1 < a.nr)) add4<V2D>(a, g.inv_v2, unit, cr + 1, ca, cz, c[1], c[3], c[5], c[7]);
    }
    for (int e = threadIdx.x; e < s_queued; e += DEP_THREADS) stray<FACES, V2D>(a, g, b0 + s_queue[e]);
}

// The fixed-point form of a uniform axis of n cells over [lo, hi).
FixAxis fix_axis(double lo, double hi, int n) {
    FixAxis a{};
    int E = 0;
    std::frexp(std::max(std::fabs(lo), std::fabs(hi)), &E);
    a.e1 = E + 1023;
    a.base = (long long)std::ldexp(lo, 62 - E);   // (cut where lo has bits below 2^(E - 62))
    a.smax = std::ldexp((double)a.base, E - 62) == lo ? 10 : 0;
    a.span = (u64)((long long)std::ldexp(hi, 62 - E) - a.base);
    a.sh = 0;
    while (a.span && !((a.span << a.sh) >> 62)) ++a.sh;    // span 2^sh in [2^62, 2^63)
    int b = 0;
    while ((n >> (b + 1)) != 0) ++b;
    a.F = 61 - b;                                          // n 2^F in [2^61, 2^62)
    const u64 num = (u64)n << a.F, den = a.span << a.sh;   // K = floor(num 2^64 / den), num < den
    a.K = den ? (u64)(((unsigned __int128)num << 64) / den) : 0;
    if (num >= den || a.F < 32) a.span = 0;                // degenerate: every particle takes the binary64 arithmetic
    return a;
}

struct ProjectArgs {
    int nr, nt, nz, accumulate, walk;   // walk: axial cells per warp
    double charge;
    const double *flo, *fhi;   // [nr] radial shares of a cell's lower / upper corner nodes
    const double *nodes;
    double *rho;
    const unsigned char *act;  // MASK: active flags [nz][nr]; inactive cells get no charge
};

// A warp takes 31 consecutive radial cells (32 node radii) at one j and walks
// PROJ_K axial cells: a lane adds the two alpha nodes of its radius in a node
// plane once for the cells on both sides of the plane, adds two planes' sums,
// and gets the next radius' sum from the next lane -- 2 additions and 2
// multiply-adds per cell where one thread per cell took 7 and 4 FP64
// instructions, which bound the kernel (26.2 M cells: 545 us, now 264, the FP64 unit 72 % busy).
// Fewer cells per walk where that leaves too few warps (320 x 8 x 21: 7.1 -> 3.4 us).
constexpr int PROJ_K = 8, PROJ_WARPS = 8;

template <bool MASK>
__global__ void __launch_bounds__(PROJ_WARPS * 32) k_project(const ProjectArgs a) {
    const int lane = threadIdx.x & 31;
    const unsigned item = blockIdx.x * PROJ_WARPS + (threadIdx.x >> 5);   // (k block, j, radial block), radial fastest
    const unsigned rb = (unsigned)(a.nr + 30) / 31u, kb = (unsigned)(a.nz + a.walk - 1) / a.walk;
    if (item >= rb * (unsigned)a.nt * kb) return;
    const unsigned row = item / rb;
    const int i = (int)(item - row * rb) * 31 + lane;
    const int k0 = (int)(row / (unsigned)a.nt) * a.walk, j = (int)(row % (unsigned)a.nt);
    const int jn = j + 1 == a.nt ? 0 : j + 1;
    const size_t rs = (size_t)a.nr + 1, ps = (size_t)a.nt * rs;
    const int in = min(i, a.nr);                                           // (lanes beyond the last node radius)
    const bool cell = lane < 31 && i < a.nr;
    const double s = a.charge * 0.25;
    const double flo = cell ? s * a.flo[i] : 0.0, fhi = cell ? s * a.fhi[i] : 0.0;
    const double *n0 = a.nodes + (size_t)k0 * ps + (size_t)j * rs + in, *n1 = a.nodes + (size_t)k0 * ps + (size_t)jn * rs + in;
    double lower = *n0 + *n1;
    const int k1 = min(a.nz, k0 + a.walk);
    for (int k = k0; k < k1; ++k) {
        n0 += ps;
        n1 += ps;
        const double upper = *n0 + *n1, lo = lower + upper;
        const double hi = __shfl_down_sync(0xffffffffu, lo, 1);
        lower = upper;
        if (!cell) continue;
        const size_t e = ((size_t)k * a.nt + j) * a.nr + i;
        double v = fma(flo, lo, fhi * hi);
        if (MASK && !a.act[(size_t)k * a.nr + i]) v = 0.0;
        a.rho[e] = a.accumulate ? a.rho[e] + v : v;
    }
}

}  // namespace
}  // namespace pp

using namespace pp;

namespace {
int single(const pic_poisson_plan_s *P, const char *what) {
    if (P->n != 1) {
        set_error("%s needs a single-problem plan (this plan holds %d problems)", what, P->n);
        return PIC_POISSON_EINVAL;
    }
    return PIC_POISSON_OK;
}
}  // namespace

extern "C" int pic_poisson_deposit(pic_poisson_plan_t plan, const double *r_dev, const double *alpha_dev,
                                   const double *z_dev, long long np, double weight, double *nodes_dev) {
    int rc = plan_enter(plan);
    if (rc) return rc;
    rc = single(plan, "pic_poisson_deposit");
    if (rc) return rc;
    if (np < 0 || (np > 0 && (!r_dev || !alpha_dev || !z_dev)) || !nodes_dev) {
        set_error("pic_poisson_deposit: NULL pointer or negative count");
        return PIC_POISSON_EINVAL;
    }
    const ProblemPlan &q = plan->pr[0];
    if (np == 0) return PIC_POISSON_OK;
    const LevelHost &h = q.lv[0];
    DepositArgs a{};
    a.nr = h.nr;
    a.nt = q.d.ntheta;
    a.nz = h.nz;
    a.np = np;
    a.r_in = q.d.r_in;
    a.z0 = q.d.z0;
    a.inv_dr = 1.0 / h.dr;
    a.inv_da = q.d.ntheta / q.d.theta_span;
    a.inv_dz = 1.0 / h.dz;
    a.weight = weight;
    a.vec = ((reinterpret_cast<uintptr_t>(r_dev) | reinterpret_cast<uintptr_t>(alpha_dev) |
              reinterpret_cast<uintptr_t>(z_dev)) & 15) == 0;
    a.r = r_dev;
    a.al = alpha_dev;
    a.z = z_dev;
    a.inv_vr = q.dep_inv_vr;
    a.inv_vz = q.dep_inv_vz;
    a.nodes = nodes_dev;
    const bool gen = !q.uniform_r || !h.zf.empty() || q.act0;
    DepositGeo g{};
    if (gen) {
        g.rf = q.dep_rf;
        g.zf = q.dep_zf;
        g.inv_wr = q.dep_inv_wr;
        g.inv_wz = q.dep_inv_wz;
        g.rbin = q.dep_rbin;
        g.zbin = q.dep_zbin;
        g.nrbin = q.dep_nrbin;
        g.nzbin = q.dep_nzbin;
        g.r0f = (float)h.rf[0];
        g.z0f = (float)(h.zf.empty() ? q.d.z0 : h.zf[0]);
        g.inv_rbw = q.dep_inv_rbw;
        g.inv_zbw = q.dep_inv_zbw;
        g.act = q.act0;
        g.inv_v2 = q.dep_inv_v2;
    } else {
        a.fr = fix_axis(q.d.r_in, q.d.r_out, h.nr);
        a.fa = fix_axis(0.0, q.d.theta_span, q.d.ntheta);
        a.fz = fix_axis(q.d.z0, q.d.z1, h.nz);
    }
    const long long per = (long long)DEP_THREADS * DEP_PPT, blocks = (np + per - 1) / per;
    if (blocks > 0x7fffffffLL) {
        set_error("pic_poisson_deposit: too many particles for one launch (%lld)", np);
        return PIC_POISSON_EINVAL;
    }
    if (gen && g.inv_v2) k_deposit<true, true><<<(unsigned)blocks, DEP_THREADS, 0, plan->stream>>>(a, g);
    else if (gen) k_deposit<true, false><<<(unsigned)blocks, DEP_THREADS, 0, plan->stream>>>(a, g);
    else k_deposit<false, false><<<(unsigned)blocks, DEP_THREADS, 0, plan->stream>>>(a, g);
    PP_CUDA(cudaGetLastError());
    return PIC_POISSON_OK;
}

extern "C" int pic_poisson_project(pic_poisson_plan_t plan, const double *nodes_dev, double charge, int accumulate,
                                   double *rho_dev) {
    int rc = plan_enter(plan);
    if (rc) return rc;
    rc = single(plan, "pic_poisson_project");
    if (rc) return rc;
    if (!nodes_dev || !rho_dev) {
        set_error("pic_poisson_project: NULL pointer");
        return PIC_POISSON_EINVAL;
    }
    const ProblemPlan &q = plan->pr[0];
    const LevelHost &h = q.lv[0];
    ProjectArgs a{};
    a.nr = h.nr;
    a.nt = q.d.ntheta;
    a.nz = h.nz;
    a.accumulate = accumulate ? 1 : 0;
    a.charge = charge;
    a.flo = q.dep_flo;
    a.fhi = q.dep_fhi;
    a.nodes = nodes_dev;
    a.rho = rho_dev;
    a.act = q.act0;
    const size_t rows = (size_t)((a.nr + 30) / 31) * a.nt;   // of warps
    a.walk = (int)std::min<size_t>(std::max<size_t>(rows * a.nz / (kSMs * 64 * 2), 1), PROJ_K);
    const size_t items = rows * ((a.nz + a.walk - 1) / a.walk);
    const unsigned grid = (unsigned)((items + PROJ_WARPS - 1) / PROJ_WARPS);
    if (q.act0) k_project<true><<<grid, PROJ_WARPS * 32, 0, plan->stream>>>(a);
    else k_project<false><<<grid, PROJ_WARPS * 32, 0, plan->stream>>>(a);
    PP_CUDA(cudaGetLastError());
    return PIC_POISSON_OK;
}
