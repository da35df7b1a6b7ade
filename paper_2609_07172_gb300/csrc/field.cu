// Face-field reconstruction, the step that follows the Poisson solve in the
// paper's particle-in-cell cycle (Sec. 2: electric fields are stored on cell
// faces): E = -grad phi on every face of the three-dimensional cell grid,
// from the cell-centred potential.  Radial and axial faces use the distances
// of the operator's face conductances (appendix Eqs.
// interior_face_conductances, dirichlet_face_conductances): centre to centre
// between two cells, centre to face on a Dirichlet wall, where the potential
// is the wall value; azimuthal faces the arc r_i dalpha of the angular
// difference (Sec. 3.1), periodic.  So the face fluxes of a cell add up to its
// charge (discrete Gauss law): sum over faces of area E.n = rho V / eps0 for
// the discrete solution.
//
// Each cell writes its lower r, azimuthal (j + 1/2) and lower z face, and the cells
// next to the upper walls also the wall face: one subtraction and one product by a
// precomputed inverse distance per face.  With both in the FP64 unit the kernel
// took 401 us at 512 x 128 x 400 (845 MB, 123 us at the copy rate); with the
// products by integer multiplies, bit for bit those of binary64, and a walk along z
// that keeps factors and the plane before in registers 193 us, bound by latency and
// the subtractions (32 registers, eight blocks per SM and the next plane's load
// ahead of its use: 237 us with 48 registers and no load ahead).
// Non-uniform axial faces and composite domains take a variant with an axial
// distance table and, for patches, exposed faces (k_face_field_gen).
#include <algorithm>

#include "fixed.h"
#include "plan.h"

namespace pp {
namespace {

struct FieldArgs {
    int nr, nt, nz;
    double inv_dz, inv_hdz;                    // 1 / axial centre distance, 1 / centre-to-wall distance
    const double *inv_rd;                      // [nr + 1] 1 / radial distance across face a
    double phi_z0, phi_z1;
    const double *win, *wout;                  // [nz] r-wall potentials
    const double *inv_rda;                     // [nr] 1 / (r_i dalpha)
    const double *phi;                         // (nz, nt, nr)
    double *er, *ea, *ez;                      // (nz, nt, nr + 1), (nz, nt, nr), (nz + 1, nt, nr)
};

// A positive binary64 constant to multiply by: its mantissa in 64 bits (top bit
// set), exponent field and value.
struct Factor {
    ufx m;
    int e;
    double v;
};
__device__ __forceinline__ Factor factor(double c) { return {f64_mant(c) << 1, f64_exp(c), c}; }
// d c, rounded to nearest: the upper half of the mantissas' product, by integer
// multiplies.  What may be a tie (one product in a thousand), zeros, subnormals,
// infinities, NaN and results outside the normal range go to the FP64 unit.
// (Not inlined: predicated, that multiplication would hold the unit all the same.)
__device__ __noinline__ double times_f64(double d, double c) { return d * c; }
__device__ __forceinline__ double times(double d, const Factor &c) {
    const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
    const ufx p = __umul64hi(f64_mant(d), c.m);                // in [2^61, 2^63)
    const unsigned big = (unsigned)(p >> 62);
    const int E = e + c.e - 1023 + (int)big;                   // biased exponent, before a carry
    const ufx q = p << (1 - big);
    const ufx bits = ((q + (1ull << 9)) >> 10) + ((ufx)(unsigned)(E - 1) << 52);
    double r = __longlong_as_double((fx)(bits | (ufx)((unsigned)hi & 0x80000000u) << 32));
    if ((unsigned)(e - 1) >= 0x7feu || (unsigned)(E - 1) >= 0x7fdu || ((unsigned)q & 0x3ffu) == 0x200u) r = times_f64(d, c.v);
    return r;
}

// One thread per (j, i), r fastest, over `chunk` planes: the plane before stays in a
// register, the radial factors too.
__global__ void __launch_bounds__(256, 8) k_face_field(const FieldArgs a, int chunk) {
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x, nr = (unsigned)a.nr, plane = (unsigned)a.nt * nr;
    if (c >= plane) return;
    const unsigned j = c / nr, i = c - j * nr;
    const int k0 = (int)blockIdx.y * chunk, k1 = min(k0 + chunk, a.nz);
    const Factor fr = factor(a.inv_rd[i]), fa = factor(a.inv_rda[i]), fz = factor(a.inv_dz);
    const double inv_out = i + 1 == nr ? a.inv_rd[nr] : 0.0;
    const size_t e0 = (size_t)k0 * plane + c;
    const double *phi = a.phi + e0;
    // row j + 1 of the plane, periodic
    const double *next = a.phi + (e0 - c) + (j + 1 == (unsigned)a.nt ? i : c + nr);
    double *er = a.er + e0 + (size_t)k0 * a.nt + j, *ea = a.ea + e0, *ez = a.ez + e0;   // (er: rows of nr + 1)
    double ps = k0 > 0 ? *(phi - plane) : a.phi_z0, p = 0.0, pn = *phi;
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        p = pn;
        if (k + 1 < k1) pn = phi[plane];
        const double pw = i > 0 ? *(phi - 1) : a.win[k];
        *er = times(pw - p, fr);
        if (i + 1 == nr) er[1] = (p - a.wout[k]) * inv_out;
        *ea = times(p - *next, fa);
        *ez = k > 0 ? times(ps - p, fz) : (ps - p) * a.inv_hdz;
        ps = p;
        phi += plane;
        next += plane;
        er += plane + a.nt;
        ea += plane;
        ez += plane;
    }
    if (k1 == a.nz) *ez = (p - a.phi_z1) * a.inv_hdz;
}

// The same on non-uniform axial faces and composite domains.  Axial
// distances come from a table like the radial ones.  With MASK (a composite
// domain, Sec. 2.2): a face between an active and an inactive cell is a
// Dirichlet face at phi_exposed, differenced from the active cell's centre
// to the face (the distance of the exposed face's conductance); faces with no
// active cell on either side, wall faces of inactive cells included, get
// E = 0.  The plain kernel above is unchanged for plain plans.
struct FieldGenArgs {
    FieldArgs a;
    const double *inv_zd;                      // [nz + 1] 1 / axial distance across face c
    const double *inv_half;                    // 1 / centre-to-face: r lower, r upper [nr]; z lower, z upper [nz]
    const unsigned char *act;                  // [nz][nr] active flags (MASK)
    double pe;                                 // phi_exposed
};

template <bool MASK>
__global__ void __launch_bounds__(256) k_face_field_gen(const FieldGenArgs g) {
    const FieldArgs &a = g.a;
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned nr = (unsigned)a.nr, row_n = (unsigned)a.nz * (unsigned)a.nt;
    if (e >= row_n * nr) return;
    const unsigned row = e / nr;
    const int i = (int)(e - row * nr);
    const int k = (int)(row / (unsigned)a.nt), j = (int)(row - (unsigned)k * a.nt);
    const double p = a.phi[e];
    const bool ai = !MASK || g.act[(size_t)k * nr + i];
    const double *ihr_lo = g.inv_half, *ihr_hi = g.inv_half + a.nr;
    const double *ihz_lo = g.inv_half + 2 * a.nr, *ihz_hi = ihz_lo + a.nz;
    // radial face i
    const size_t fr = (size_t)row * (nr + 1) + i;
    double vr;
    if (i == 0) {
        vr = ai ? (a.win[k] - p) * a.inv_rd[0] : 0.0;
    } else {
        const bool aw = !MASK || g.act[(size_t)k * nr + i - 1];
        if (ai && aw) vr = (a.phi[e - 1] - p) * a.inv_rd[i];
        else if (aw) vr = (a.phi[e - 1] - g.pe) * ihr_hi[i - 1];   // exposed face east of cell i - 1
        else if (ai) vr = (g.pe - p) * ihr_lo[i];                  // exposed face west of cell i
        else vr = 0.0;
    }
    a.er[fr] = vr;
    if (i == a.nr - 1) a.er[fr + 1] = ai ? (p - a.wout[k]) * a.inv_rd[a.nr] : 0.0;
    // azimuthal face j + 1/2, periodic (both cells share the (r, z) cell's activity)
    const int jn = j + 1 == a.nt ? 0 : j + 1;
    a.ea[e] = ai ? (p - a.phi[((size_t)k * a.nt + jn) * nr + i]) * a.inv_rda[i] : 0.0;
    // axial face k
    const size_t plane = (size_t)a.nt * nr;
    double vz;
    if (k == 0) {
        vz = ai ? (a.phi_z0 - p) * g.inv_zd[0] : 0.0;
    } else {
        const bool as = !MASK || g.act[(size_t)(k - 1) * nr + i];
        if (ai && as) vz = (a.phi[e - plane] - p) * g.inv_zd[k];
        else if (as) vz = (a.phi[e - plane] - g.pe) * ihz_hi[k - 1];
        else if (ai) vz = (g.pe - p) * ihz_lo[k];
        else vz = 0.0;
    }
    a.ez[e] = vz;
    if (k == a.nz - 1) a.ez[e + plane] = ai ? (p - a.phi_z1) * g.inv_zd[a.nz] : 0.0;
}

}  // namespace
}  // namespace pp

using namespace pp;

extern "C" int pic_poisson_face_field(pic_poisson_plan_t plan, const double *phi_dev, double *er_dev, double *ea_dev,
                                      double *ez_dev) {
    int rc = plan_enter(plan);
    if (rc) return rc;
    if (plan->n != 1) {
        set_error("pic_poisson_face_field needs a single-problem plan (this plan holds %d problems)", plan->n);
        return PIC_POISSON_EINVAL;
    }
    if (!phi_dev || !er_dev || !ea_dev || !ez_dev) {
        set_error("NULL pointer");
        return PIC_POISSON_EINVAL;
    }
    const ProblemPlan &q = plan->pr[0];
    const LevelHost &h = q.lv[0];
    FieldArgs a{};
    a.nr = h.nr;
    a.nt = q.d.ntheta;
    a.nz = h.nz;
    a.inv_rd = q.finv_rd;
    a.inv_dz = 1.0 / h.dz;
    a.inv_hdz = 1.0 / (0.5 * h.dz);
    a.phi_z0 = q.d.phi_z0;
    a.phi_z1 = q.d.phi_z1;
    a.win = q.fwin;
    a.wout = q.fwout;
    a.inv_rda = q.finv_rda;
    a.phi = phi_dev;
    a.er = er_dev;
    a.ea = ea_dev;
    a.ez = ez_dev;
    const size_t n = (size_t)a.nz * a.nt * a.nr;
    const unsigned grid = (unsigned)((n + 255) / 256);
    if (h.act.empty() && h.zf.empty()) {
        // planes per block: as many as leave the chip twice the blocks it holds
        const unsigned cols = (unsigned)(((size_t)a.nt * a.nr + 255) / 256);
        // (and no more pieces than the grid's second dimension holds)
        const int fill = (int)std::min<size_t>(std::max<size_t>((size_t)cols * a.nz / (kSMs * 8 * 2), 1), 16);
        const int chunk = std::max(fill, (a.nz + 65534) / 65535);
        k_face_field<<<dim3(cols, (unsigned)((a.nz + chunk - 1) / chunk)), 256, 0, plan->stream>>>(a, chunk);
    } else {   // non-uniform axial faces and / or a composite domain
        FieldGenArgs g{};
        g.a = a;
        g.inv_zd = q.finv_zd;
        g.inv_half = q.finv_half;
        g.act = q.act0;
        g.pe = q.d.phi_exposed;
        if (q.act0) k_face_field_gen<true><<<grid, 256, 0, plan->stream>>>(g);
        else k_face_field_gen<false><<<grid, 256, 0, plan->stream>>>(g);
    }
    PP_CUDA(cudaGetLastError());
    return PIC_POISSON_OK;
}
