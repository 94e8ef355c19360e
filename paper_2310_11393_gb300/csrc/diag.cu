// Diagnostics kernels (off the stepping loop): charge density, Gauss-law residual,
// field and kinetic energies (Sec. 3.1, Eqs. L2_t and L2_t_cross use these integrals),
// energy-angle histograms (Sec. 4.2: angle measured from the propagation axis) and a
// point evaluator of the incident field.  Accumulation is in double precision.
#include <cuda_runtime.h>

#include <algorithm>

#include <mutex>

#include "beam.cuh"
#include "sff_common.cuh"
#include "sff_kernels.h"
#include "sim_internal.h"

namespace sff {

template <int D>
__device__ __forceinline__ void decode_cell_d(const SimDev& S, unsigned cl, int c[3])
{
    c[0] = (int)(cl & ((1u << S.cb[0]) - 1u));
    c[1] = 0;
    c[2] = 0;
    if constexpr (D > 1) c[1] = (int)((cl >> S.cb[0]) & ((1u << S.cb[1]) - 1u));
    if constexpr (D > 2) c[2] = (int)(cl >> (S.cb[0] + S.cb[1]));
}

// body(p) for every particle slot p of buffer set par, a block per tile (the tiles' occupied
// slots only: two to three times as many slots are in use as hold particles)
template <typename F>
__device__ __forceinline__ void for_particles(const SimDev& S, int par, F body)
{
    for (int t = blockIdx.x; t < S.nptiles; t += gridDim.x) {
        const long long p0 = S.toff[par][t];
        const int n = S.tnum[par][t];
        for (int i = threadIdx.x; i < n; i += blockDim.x) body(p0 + i);
    }
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// charge density scale * rho_e, rho_e = -sum w S(x - x_node), added on the primal nodes
// (array coordinates)
template <int D, typename R>
__global__ void k_charge(const SimDev* __restrict__ sim, double* __restrict__ rho, double scale)
{
    const SimDev& S = *sim;
    const int par = S.st->parity;
    for_particles(S, par, [&](long long p) {
        int c[3];
        decode_cell_d<D>(S, S.cell[par][p], c);
        double w[3][3];
        int lo[3] = {0, 0, 0};
        for (int d = 0; d < 3; ++d) {
            if (d < D) {
                const double o = (double)reinterpret_cast<const R*>(S.off[par][d])[p];
                const int h = o >= 0.5;
                const double dl = o - h;
                w[d][0] = 0.5 * (0.5 - dl) * (0.5 - dl);
                w[d][1] = 0.75 - dl * dl;
                w[d][2] = 0.5 * (0.5 + dl) * (0.5 + dl);
                lo[d] = c[d] + h - 1 + (d == 0 ? GX : G);
            } else {
                w[d][0] = 1.0;
                w[d][1] = w[d][2] = 0.0;
            }
        }
        const double q = -scale * (double)reinterpret_cast<const R*>(S.wgt[par])[p];
        const int nk = D > 2 ? 3 : 1, nj = D > 1 ? 3 : 1;
        for (int k = 0; k < nk; ++k)
            for (int j = 0; j < nj; ++j)
                for (int i = 0; i < 3; ++i)
                    atomicAdd(&rho[(long long)(lo[2] + k) * S.sz + (long long)(lo[1] + j) * S.sy + lo[0] + i],
                              q * w[0][i] * w[1][j] * w[2][k]);
    });
}

// max |div E - rho - rho_ion| over interior primal nodes; result as ordered bits
template <int D, typename R>
__global__ void k_gauss(const SimDev* __restrict__ sim, const double* __restrict__ rho, int n0, int n1, int n2,
                        unsigned long long* __restrict__ out)
{
    const SimDev& S = *sim;
    const R* F = reinterpret_cast<const R*>(S.F);
    const long long eb = (long long)comp_eb(S.st->parity) * S.sc;
    const long long total = (long long)n0 * n1 * n2;   // interior extents
    double worst = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total;
         k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k % n0) + 1;
        const int j = D > 1 ? (int)((k / n0) % n1) + 1 : 0;
        const int l = D > 2 ? (int)(k / ((long long)n0 * n1)) + 1 : 0;
        const long long o = (long long)(D > 2 ? l + G : 0) * S.sz + (long long)(D > 1 ? j + G : 0) * S.sy + (i + GX);
        double div = ((double)F[eb + o] - (double)F[eb + o - 1]) * S.inv_dx;
        if (D > 1) div += ((double)F[eb + S.sc + o] - (double)F[eb + S.sc + o - S.sy]) * S.inv_dx;
        if (D > 2) div += ((double)F[eb + 2 * S.sc + o] - (double)F[eb + 2 * S.sc + o - S.sz]) * S.inv_dx;
        const double r = fabs(div - rho[o] - S.rho_ion[o]);
        worst = fmax(worst, r);
    }
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(worst));
}

// Is component comp of the incident field identically zero (grid axes: the beam's z is x, its x
// is y, its y is z)?  The plane wave has E_y and B_z, the 2D Gaussian beam E_x, E_y and B_z; the
// focused pulses have no component odd in y (their own; grid z) in 2D, and RP no B along its axis.
template <int D>
__device__ __forceinline__ bool incident_zero(int beam, int comp)
{
    if (beam == BEAM_NONE) return true;
    if (beam == BEAM_PLANE) return comp != 1 && comp != 5;
    if (beam == BEAM_GAUSS2D) return comp != 0 && comp != 1 && comp != 5;
    if (beam == BEAM_LP || beam == BEAM_RP)
        return (D == 2 && comp != 0 && comp != 1 && comp != 5) || (beam == BEAM_RP && comp == 3);
    return false;
}

// 1/2 sum F^2 dx^dim over the points each component has: [0] scattered, [1] scattered + incident.
// A block takes 256 points of a row at a time: one double-precision phase reference per row
// segment (per point and component it was most of the kernel: FP64 runs at 1/64 of the FP32
// rate), the components in turn, those that are identically zero without the closed form.
// Double sums.  3D RP 512 x 256 x 256: 12.0 -> 4.8 ms with the particle part.
template <int D, typename R>
__global__ void __launch_bounds__(256) k_energy_fields(const SimDev* __restrict__ sim, double* __restrict__ acc)
{
    const SimDev& S = *sim;
    const R* F = reinterpret_cast<const R*>(S.F);
    const DevState* st = S.st;
    const long long eb = (long long)comp_eb(st->parity) * S.sc;
    const double t = (double)st->step * S.dt;
    const BeamC<R>& bc = beam_of<R>(S);
    const int m0 = S.n[0] + 1, m1 = D > 1 ? S.n[1] + 1 : 1, m2 = D > 2 ? S.n[2] + 1 : 1;
    const long long segs = (m0 + 255) / 256, total = segs * m1 * m2;
    __shared__ PhaseRef<R> s_pr;
    double es = 0.0, et = 0.0;
    // the segments of one place along x in turn: the phase reference changes with that place only
    long long ref_seg = -1;
    for (long long k = blockIdx.x; k < total; k += gridDim.x) {
        const long long rows = (long long)m1 * m2, seg = k / rows, row = k - seg * rows;
        if (seg != ref_seg) {
            __syncthreads();
            if (threadIdx.x == 0) s_pr = phase_ref<R>(S, t, (int)seg * 256);
            __syncthreads();
            ref_seg = seg;
        }
        const int g[3] = {(int)seg * 256 + (int)threadIdx.x, (int)(row % m1), (int)(row / m1)};
        if (g[0] >= m0) continue;
        const long long o = (long long)(D > 2 ? g[2] + G : 0) * S.sz + (long long)(D > 1 ? g[1] + G : 0) * S.sy +
                            (g[0] + GX);
#pragma unroll 1
        for (int comp = 0; comp < 6; ++comp) {
            const int c = comp % 3;
            bool has = true;
            R oo[3] = {R(0), R(0), R(0)};
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const bool stag = comp < 3 ? (d == c) : (d != c);
                if (stag) {
                    if (g[d] > S.n[d] - 1) has = false;
                    oo[d] = R(0.5);
                }
            }
            if (!has) continue;
            const double f = (double)F[eb + comp * S.sc + o];
            double h = f;
            if (!S.tf && !incident_zero<D>(S.beam, comp)) {
                R Ei[3], Bi[3];
                incident_at<D, R, true>(S, bc, s_pr, g, oo, Ei, Bi);
                const R e = c == 0 ? Ei[0] : (c == 1 ? Ei[1] : Ei[2]), b = c == 0 ? Bi[0] : (c == 1 ? Bi[1] : Bi[2]);
                h += (double)(comp < 3 ? e : b);
            }
            es += 0.5 * f * f;
            et += 0.5 * h * h;
        }
    }
    es = warp_sum(es);
    et = warp_sum(et);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&acc[0], es);
        atomicAdd(&acc[1], et);
    }
}

// [2] sum w (gamma - 1) of electrons in the box, [3] of exit records (times dx^dim on the host)
template <typename R>
__global__ void k_energy_particles(const SimDev* __restrict__ sim, long long nex, double* __restrict__ acc)
{
    const SimDev& S = *sim;
    const int par = S.st->parity;
    double ka = 0.0, ke = 0.0;
    for_particles(S, par, [&](long long p) {
        double u2 = 0.0;
        for (int d = 0; d < 3; ++d) {
            const double u = (double)reinterpret_cast<const R*>(S.mom[par][d])[p];
            u2 += u * u;
        }
        ka += (double)reinterpret_cast<const R*>(S.wgt[par])[p] * (sqrt(1.0 + u2) - 1.0);
    });
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < nex;
         p += (long long)gridDim.x * blockDim.x) {
        const double* e = S.exits + p * EXIT_DOUBLES;
        ke += e[3] * (sqrt(1.0 + e[0] * e[0] + e[1] * e[1] + e[2] * e[2]) - 1.0);
    }
    ka = warp_sum(ka);
    ke = warp_sum(ke);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&acc[2], ka);
        atomicAdd(&acc[3], ke);
    }
}

__device__ __forceinline__ void hist_add(double* bins, double ux, double uy, double uz, double w, int n_e, double e_max,
                                         int n_a)
{
    const double u2 = ux * ux + uy * uy + uz * uz;
    const double ek = sqrt(1.0 + u2) - 1.0;
    if (!(ek < e_max) || ek < 0.0) return;
    const double ang = atan2(sqrt(uy * uy + uz * uz), ux);   // from the +x (propagation) axis
    int ie = (int)(ek / e_max * n_e);
    int ia = (int)(ang / 3.14159265358979323846 * n_a);
    ie = min(max(ie, 0), n_e - 1);
    ia = min(max(ia, 0), n_a - 1);
    atomicAdd(&bins[(long long)ie * n_a + ia], w);
}

// The same for single-precision momenta: the bin from FP32 arithmetic wherever that cannot differ
// from the double one, i.e. unless it comes within its error of a bin's edge (2.1 M electrons,
// 96 x 36 bins: 0.53 -> 0.10 ms; the double functions run at 1/64 of the FP32 rate).  Errors:
// gamma - 1 = u^2/(gamma + 1) within 8 roundings of 2^-24 relative; the angle within 8 of pi.  The
// double gamma - 1 has its own, of 2^-53 gamma: they count where the bins are that narrow.
__device__ __forceinline__ void hist_add(double* bins, float ux, float uy, float uz, float w, int n_e, double e_max,
                                         int n_a)
{
    const float up2 = uy * uy + uz * uz, u2 = ux * ux + up2;
    const float scale = (float)n_e / (float)e_max;
    const float fe = u2 / (1.0f + sqrtf(1.0f + u2)) * scale;
    const float fa = atan2f(sqrtf(up2), ux) * ((float)n_a * 0.318309886f);
    const float de = 1e-6f * fe + 4.5e-16f * scale, da = 2e-6f * (float)n_a;
    const float ie = floorf(fe), ia = floorf(fa);
    const bool sure = fe - ie > de && fe - ie < 1.0f - de && fa - ia > da && fa - ia < 1.0f - da && u2 < 1e30f;
    if (!sure || n_e > (1 << 16) || n_a > (1 << 16)) {
        hist_add(bins, (double)ux, (double)uy, (double)uz, (double)w, n_e, e_max, n_a);
    } else if (ie < (float)n_e) {
        atomicAdd(&bins[(long long)(int)ie * n_a + min((int)ia, n_a - 1)], (double)w);
    }
}

// SHARED: each block adds up its own n_e * n_a bins in shared memory first (the hot bins of a
// thermal spectrum otherwise queue up in L2: 2.1 M electrons 0.44 ms).
template <typename R, bool SHARED>
__global__ void __launch_bounds__(512) k_histogram(const SimDev* __restrict__ sim, long long nex, int n_e, double e_max,
                                                   int n_a, double* __restrict__ out)
{
    extern __shared__ double s_bins[];
    const SimDev& S = *sim;
    const int par = S.st->parity;
    double* bins = SHARED ? s_bins : out;
    if constexpr (SHARED) {
        for (int i = threadIdx.x; i < n_e * n_a; i += blockDim.x) s_bins[i] = 0.0;
        __syncthreads();
    }
    for_particles(S, par, [&](long long p) {
        hist_add(bins, reinterpret_cast<const R*>(S.mom[par][0])[p], reinterpret_cast<const R*>(S.mom[par][1])[p],
                 reinterpret_cast<const R*>(S.mom[par][2])[p], reinterpret_cast<const R*>(S.wgt[par])[p], n_e, e_max, n_a);
    });
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < nex;
         p += (long long)gridDim.x * blockDim.x) {
        const double* e = S.exits + p * EXIT_DOUBLES;
        hist_add(bins, e[0], e[1], e[2], e[3], n_e, e_max, n_a);
    }
    if constexpr (SHARED) {
        __syncthreads();
        for (int i = threadIdx.x; i < n_e * n_a; i += blockDim.x)
            if (s_bins[i] != 0.0) atomicAdd(&out[i], s_bins[i]);
    }
}

// incident field at arbitrary points (x, y, z, t), grid coordinates
template <int D, typename R>
__global__ void k_eval_incident(const SimDev* __restrict__ sim, long long n, const double* __restrict__ pts,
                                double* __restrict__ out)
{
    const SimDev& S = *sim;
    const BeamC<R>& bc = beam_of<R>(S);
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        int c[3] = {0, 0, 0};
        R o[3] = {R(0), R(0), R(0)};
        for (int d = 0; d < D; ++d) {
            const double X = pts[4 * p + d] * S.inv_dx;
            const double fl = floor(X);
            c[d] = (int)fl;
            o[d] = R(X - fl);
        }
        R E[3], B[3];
        const PhaseRef<R> pr = phase_ref<R>(S, pts[4 * p + 3], c[0]);
        incident_at<D, R>(S, bc, pr, c, o, E, B);
        for (int d = 0; d < 3; ++d) {
            out[6 * p + d] = (double)E[d];
            out[6 * p + 3 + d] = (double)B[d];
        }
    }
}

// ---- state to and from the host layout ----------------------------------------------------
// The conversions between the device layout and the host arrays of the C-ABI run here, one
// piece of staging memory at a time, and the copy engine moves host doubles: 64 B per electron
// and 72 B per grid point at the link's rate (190-200 GB/s to and from host pages that are mapped
// already) instead of a pass of host threads over freshly mapped buffers.  Read-back of 2.1 M
// electrons 15-22 -> 4 ms, of 12 small simulations with their fields 21 -> 9 ms (what is left is
// mapping the caller's fresh output pages).

// first[t]: particles of the tiles before t in buffer set par, first[nptiles] their total
__global__ void __launch_bounds__(1024) k_tile_first(const SimDev* __restrict__ sim, int par, int* __restrict__ first)
{
    const SimDev& S = *sim;
    __shared__ int s_warp[32];
    const int tid = threadIdx.x, lane = tid & 31, n = S.nptiles;
    int carry = 0;
    for (int base = 0; base < n; base += 1024) {
        const int i = base + tid;
        const int v = i < n ? S.tnum[par][i] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[tid >> 5] = x;
        __syncthreads();
        int before = 0, all = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < (tid >> 5)) before += s_warp[w];
            all += s_warp[w];
        }
        if (i < n) first[i] = carry + before + x - v;
        carry += all;
        __syncthreads();
    }
    if (tid == 0) first[n] = carry;
}

// records k in [k0, k1) of PIC_DIAG_PARTICLES (tiles in order): x[3], u[3], w, id
template <int D, typename R>
__global__ void __launch_bounds__(128) k_pack_particles(const SimDev* __restrict__ sim, int par,
                                                        const int* __restrict__ first, long long k0, long long k1,
                                                        double2* __restrict__ out)
{
    const SimDev& S = *sim;
    for (int t = blockIdx.x; t < S.nptiles; t += gridDim.x) {
        const long long f = first[t], base = S.toff[par][t];
        const int i0 = (int)max(0ll, k0 - f), i1 = (int)min((long long)S.tnum[par][t], k1 - f);
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const long long p = base + i;
            int c[3];
            decode_cell_d<D>(S, S.cell[par][p], c);
            double r[8] = {0., 0., 0., 0., 0., 0., 0., 0.};
#pragma unroll
            for (int d = 0; d < D; ++d) r[d] = ((double)c[d] + (double)reinterpret_cast<const R*>(S.off[par][d])[p]) * S.dx;
#pragma unroll
            for (int d = 0; d < 3; ++d) r[3 + d] = (double)reinterpret_cast<const R*>(S.mom[par][d])[p];
            r[6] = (double)reinterpret_cast<const R*>(S.wgt[par])[p];
            r[7] = (double)S.pid[par][p];
            double2* o = out + 4 * (f + i - k0);
#pragma unroll
            for (int j = 0; j < 4; ++j) o[j] = make_double2(r[2 * j], r[2 * j + 1]);
        }
    }
}

// largest |w| (ordered bits) and first particle that pic_set_particles refuses: a coordinate
// outside [margin, n - margin) cells, an id outside [0, 2^31); x, w, id hold particles k0 ..
template <int D>
__global__ void k_check_particles(const SimDev* __restrict__ sim, long long k0, int n, const double* __restrict__ x,
                                  const double* __restrict__ w, const long long* __restrict__ id,
                                  unsigned long long* __restrict__ out)
{
    const SimDev& S = *sim;
    double wm = 0.0;
    unsigned long long bad = ~0ull;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        bool ok = id[p] >= 0 && id[p] < (1ll << 31);
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const double X = x[3 * p + d] / S.dx;
            ok = ok && X >= S.margin && X < S.n[d] - S.margin;
        }
        if (!ok) bad = min(bad, (unsigned long long)(k0 + p));
        wm = fmax(wm, fabs(w[p]));
    }
    unsigned long long wb = (unsigned long long)__double_as_longlong(wm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        bad = min(bad, __shfl_xor_sync(0xffffffffu, bad, o));
        wb = max(wb, __shfl_xor_sync(0xffffffffu, wb, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (bad != ~0ull) atomicMin(&out[0], bad);
        atomicMax(&out[1], wb);
    }
}

// particles k0 .. k0 + n - 1 from host layout into buffer set 1, linear order
template <int D, typename R>
__global__ void k_put_particles(const SimDev* __restrict__ sim, long long k0, int n, const double* __restrict__ x,
                                const double* __restrict__ u, const double* __restrict__ w,
                                const long long* __restrict__ id)
{
    const SimDev& S = *sim;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        unsigned cl = 0;
        int sh = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const double X = x[3 * p + d] / S.dx;
            const double fl = floor(X);
            R o = R(X - fl);
            if (sizeof(R) == 4 && o >= R(1)) o = R(0.99999994f);      // the float below 1
            reinterpret_cast<R*>(S.off[1][d])[k0 + p] = o;
            cl |= (unsigned)(int)fl << sh;
            sh += S.cb[d];
        }
        S.cell[1][k0 + p] = cl;
#pragma unroll
        for (int d = 0; d < 3; ++d) reinterpret_cast<R*>(S.mom[1][d])[k0 + p] = R(u[3 * p + d]);
        reinterpret_cast<R*>(S.wgt[1])[k0 + p] = R(w[p]);
        S.pid[1][k0 + p] = (unsigned)id[p];
    }
}

// is there a point of component comp (0..5 E, B; 6..8 J) at grid index g?
template <int D>
__device__ __forceinline__ bool comp_has(const SimDev& S, int comp, const int g[3])
{
    const int c = comp % 3;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const bool stag = (comp < 3 || comp >= 6) ? d == c : d != c;
        if (g[d] < 0 || g[d] > S.n[d] - (stag ? 1 : 0)) return false;
    }
    return true;
}

// components comp0 + blockIdx.y of E, B (of buffer set par) and of J (of the last step: in the
// other set) -> out[comp][ext_z][ext_y][ext_x], absent points 0
template <int D, typename R>
__global__ void k_get_field(const SimDev* __restrict__ sim, int par, int comp0, double* __restrict__ out0)
{
    const SimDev& S = *sim;
    const int comp = comp0 + blockIdx.y;
    const int fc = comp < 6 ? comp_eb(par) + comp : comp_j(1 - par) + comp - 6;
    const R* F = reinterpret_cast<const R*>(S.F) + (long long)fc * S.sc;
    const unsigned ex = S.n[0] + 1, ey = D > 1 ? S.n[1] + 1 : 1, ez = D > 2 ? S.n[2] + 1 : 1;
    double* out = out0 + (long long)blockIdx.y * ex * ey * ez;
    const unsigned rows = ey * ez, bpr = (ex + blockDim.x - 1) / blockDim.x;
    for (unsigned b = blockIdx.x; b < rows * bpr; b += gridDim.x) {
        const unsigned r = b / bpr, i = (b - r * bpr) * blockDim.x + threadIdx.x;
        if (i >= ex) continue;
        const int g[3] = {(int)i, (int)(r % ey), (int)(r / ey)};
        const long long o = (long long)(D > 2 ? g[2] + G : 0) * S.sz + (long long)(D > 1 ? g[1] + G : 0) * S.sy + (g[0] + GX);
        out[(long long)r * ex + i] = comp_has<D>(S, comp, g) ? (double)F[o] : 0.0;
    }
}

// in[comp][ext_z][ext_y][ext_x] -> components comp0 + blockIdx.y of E, B of buffer set par, every
// allocated point written (zero in the ghost region and at absent points)
template <int D, typename R>
__global__ void k_put_field(const SimDev* __restrict__ sim, int par, int comp0, const double* __restrict__ in0)
{
    const SimDev& S = *sim;
    const int comp = comp0 + blockIdx.y;
    R* F = reinterpret_cast<R*>(S.F) + (long long)(comp_eb(par) + comp) * S.sc;
    const unsigned ex = S.n[0] + 1, ey = D > 1 ? S.n[1] + 1 : 1;
    const double* in = in0 + (long long)blockIdx.y * ex * ey * (D > 2 ? S.n[2] + 1 : 1);
    const unsigned nx = S.na[0], ny = S.na[1], rows = ny * (unsigned)S.na[2], bpr = (nx + blockDim.x - 1) / blockDim.x;
    for (unsigned b = blockIdx.x; b < rows * bpr; b += gridDim.x) {
        const unsigned r = b / bpr, i = (b - r * bpr) * blockDim.x + threadIdx.x;
        if (i >= nx) continue;
        const int g[3] = {(int)i - GX, D > 1 ? (int)(r % ny) - G : 0, D > 2 ? (int)(r / ny) - G : 0};
        R v = R(0);
        if (comp_has<D>(S, comp, g)) v = R(in[((long long)g[2] * ey + g[1]) * ex + g[0]]);
        F[(long long)r * nx + i] = v;
    }
}

// ---- host wrappers ----
static int grid_for(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, (long long)device_sms() * 8)); }

#define SFF_DISPATCH3(dim, prec, FN, ...)                       \
    do {                                                        \
        if ((prec) == 0) {                                      \
            if ((dim) == 1) FN<1, double>(__VA_ARGS__);         \
            else if ((dim) == 2) FN<2, double>(__VA_ARGS__);    \
            else FN<3, double>(__VA_ARGS__);                    \
        } else {                                                \
            if ((dim) == 1) FN<1, float>(__VA_ARGS__);          \
            else if ((dim) == 2) FN<2, float>(__VA_ARGS__);     \
            else FN<3, float>(__VA_ARGS__);                     \
        }                                                       \
    } while (0)

// a block per tile
static int grid_tiles(int nptiles) { return std::max(1, std::min(nptiles, device_sms() * 8)); }

template <int D, typename R>
static void charge_t(const SimDev* sim, int nptiles, double* rho, double scale, cudaStream_t s)
{
    k_charge<D, R><<<grid_tiles(nptiles), 256, 0, s>>>(sim, rho, scale);
}
void launch_charge(const SimDev* sim, int dim, int prec, int nptiles, double* rho, cudaStream_t s, double scale)
{
    SFF_DISPATCH3(dim, prec, charge_t, sim, nptiles, rho, scale, s);
}

template <int D, typename R>
static void gauss_t(const SimDev* sim, const double* rho, const int n[3], unsigned long long* out, cudaStream_t s)
{
    const int n0 = n[0] - 1, n1 = D > 1 ? n[1] - 1 : 1, n2 = D > 2 ? n[2] - 1 : 1;
    const long long tot = (long long)n0 * n1 * n2;
    k_gauss<D, R><<<grid_for(tot), 256, 0, s>>>(sim, rho, n0, n1, n2, out);
}
void launch_gauss(const SimDev* sim, int dim, int prec, const int n[3], const double* rho, unsigned long long* out_bits,
                  cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, gauss_t, sim, rho, n, out_bits, s);
}

template <int D, typename R>
static void efield_t(const SimDev* sim, const int n[3], double* acc, cudaStream_t s)
{
    const long long segs = (n[0] + 256) / 256, rows = (D > 1 ? n[1] + 1LL : 1) * (D > 2 ? n[2] + 1LL : 1);
    const int grid = (int)std::min<long long>(segs * rows, (long long)device_sms() * 8);
    k_energy_fields<D, R><<<grid, 256, 0, s>>>(sim, acc);
}
void launch_energy_fields(const SimDev* sim, int dim, int prec, const int n[3], double* acc2, cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, efield_t, sim, n, acc2, s);
}

void launch_energy_particles(const SimDev* sim, int prec, int nptiles, long long n_exits, double* acc2, cudaStream_t s)
{
    const int grid = std::max(grid_tiles(nptiles), n_exits > 0 ? grid_for(n_exits) : 1);
    if (prec == 0) k_energy_particles<double><<<grid, 256, 0, s>>>(sim, n_exits, acc2);
    else k_energy_particles<float><<<grid, 256, 0, s>>>(sim, n_exits, acc2);
}

template <typename R>
static void hist_t(const SimDev* sim, int nptiles, long long n, long long nex, int n_e, double e_max, int n_a,
                   double* bins, cudaStream_t s)
{
    // bins in shared memory where they fit its default size and get enough electrons each to pay
    // for their clearing and the flush
    const long long nb = (long long)n_e * n_a;
    if (nb * 8 <= 48 * 1024 && n + nex >= 16 * nb) {
        k_histogram<R, true><<<std::max(1, std::min(nptiles, device_sms() * 4)), 512, (size_t)nb * 8, s>>>(
            sim, nex, n_e, e_max, n_a, bins);
    } else {
        const int grid = std::max(grid_tiles(nptiles), nex > 0 ? grid_for(nex) : 1);
        k_histogram<R, false><<<grid, 256, 0, s>>>(sim, nex, n_e, e_max, n_a, bins);
    }
}
void launch_histogram(const SimDev* sim, int prec, int nptiles, long long n_alive, long long n_exits, int n_e,
                      double e_max, int n_a, double* bins, cudaStream_t s)
{
    if (prec == 0) hist_t<double>(sim, nptiles, n_alive, n_exits, n_e, e_max, n_a, bins, s);
    else hist_t<float>(sim, nptiles, n_alive, n_exits, n_e, e_max, n_a, bins, s);
}

template <int D, typename R>
static void evalinc_t(const SimDev* sim, long long n, const double* pts, double* out, cudaStream_t s)
{
    if (n > 0) k_eval_incident<D, R><<<grid_for(n), 256, 0, s>>>(sim, n, pts, out);
}
void launch_eval_incident(const SimDev* sim, int dim, int prec, long long n, const double* pts, double* out,
                          cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, evalinc_t, sim, n, pts, out, s);
}

void launch_tile_first(const SimDev* sim, int par, int* first, cudaStream_t s)
{
    k_tile_first<<<1, 1024, 0, s>>>(sim, par, first);
}

template <int D, typename R>
static void pack_t(const SimDev* sim, int par, int nptiles, const int* first, long long k0, long long k1, double* out,
                   cudaStream_t s)
{
    const int grid = std::max(1, std::min(nptiles, device_sms() * 16));
    k_pack_particles<D, R><<<grid, 128, 0, s>>>(sim, par, first, k0, k1, reinterpret_cast<double2*>(out));
}
void launch_pack_particles(const SimDev* sim, int dim, int prec, int par, int nptiles, const int* first, long long k0,
                           long long k1, double* out, cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, pack_t, sim, par, nptiles, first, k0, k1, out, s);
}

void launch_check_particles(const SimDev* sim, int dim, long long k0, int n, const double* x, const double* w,
                            const long long* id, unsigned long long* out, cudaStream_t s)
{
    if (n <= 0) return;
    if (dim == 1) k_check_particles<1><<<grid_for(n), 256, 0, s>>>(sim, k0, n, x, w, id, out);
    else if (dim == 2) k_check_particles<2><<<grid_for(n), 256, 0, s>>>(sim, k0, n, x, w, id, out);
    else k_check_particles<3><<<grid_for(n), 256, 0, s>>>(sim, k0, n, x, w, id, out);
}

template <int D, typename R>
static void put_t(const SimDev* sim, long long k0, int n, const double* x, const double* u, const double* w,
                  const long long* id, cudaStream_t s)
{
    if (n > 0) k_put_particles<D, R><<<grid_for(n), 256, 0, s>>>(sim, k0, n, x, u, w, id);
}
void launch_put_particles(const SimDev* sim, int dim, int prec, long long k0, int n, const double* x, const double* u,
                          const double* w, const long long* id, cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, put_t, sim, k0, n, x, u, w, id, s);
}

template <int D, typename R>
static void getf_t(const SimDev* sim, long long points, int par, int comp0, int ncomp, double* out, cudaStream_t s)
{
    k_get_field<D, R><<<dim3(grid_for(points), ncomp), 256, 0, s>>>(sim, par, comp0, out);
}
void launch_get_field(const SimDev* sim, int dim, int prec, long long points, int par, int comp0, int ncomp,
                      double* out, cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, getf_t, sim, points, par, comp0, ncomp, out, s);
}
template <int D, typename R>
static void putf_t(const SimDev* sim, long long points, int par, int comp0, int ncomp, const double* in, cudaStream_t s)
{
    k_put_field<D, R><<<dim3(grid_for(points), ncomp), 256, 0, s>>>(sim, par, comp0, in);
}
void launch_put_field(const SimDev* sim, int dim, int prec, long long points, int par, int comp0, int ncomp,
                      const double* in, cudaStream_t s)
{
    SFF_DISPATCH3(dim, prec, putf_t, sim, points, par, comp0, ncomp, in, s);
}

}  // namespace sff

// ---- histogram with statically allocated bins (pic_histogram_static) ------------------------
// The bins live in this file-scope array, so the call path allocates nothing.  Host code only
// ever passes the array's device address, looked up once per device.
static __device__ __align__(256) double g_hist_bins[PIC_HIST_STATIC_MAX_BINS];

namespace {
std::mutex g_hist_mu;
double* g_hist_addr[64] = {nullptr};   // device address of g_hist_bins per device ordinal
}  // namespace

namespace {
// Makes `dev` the calling thread's current device for the guard's lifetime.
struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        ok = prev == dev || cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard()
    {
        if (ok && prev >= 0) cudaSetDevice(prev);
    }
};
}  // namespace

extern "C" pic_status pic_histogram_static(pic_sim* s, int n_e, double e_max, int n_a, double* host_out, void* stream)
{
    if (!s || !host_out || n_e <= 0 || n_a <= 0 || !(e_max > 0)) return PIC_EINVAL;
    if ((long long)n_e * n_a > PIC_HIST_STATIC_MAX_BINS) {
        s->err = "pic_histogram_static: n_e * n_a exceeds PIC_HIST_STATIC_MAX_BINS (16384)";
        return PIC_EINVAL;
    }
    // the simulation's device is current for the look-up and every launch below
    const int dev = s->device;
    DeviceGuard guard(dev);
    if (!guard.ok || dev < 0 || dev >= 64) {
        s->err = "pic_histogram_static: cannot make the simulation's device current";
        return PIC_ENODEV;
    }
    double* bins = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_hist_mu);
        if (!g_hist_addr[dev]) {
            // set-up, once per device, with that device current
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_hist_bins);
            if (e != cudaSuccess) {
                s->err = std::string("pic_histogram_static: cudaGetSymbolAddress failed: ") + cudaGetErrorString(e);
                return PIC_ECUDA;
            }
            g_hist_addr[dev] = static_cast<double*>(p);
        }
        bins = g_hist_addr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    sff::DevState ds;
    cudaError_t e = cudaMemcpyAsync(&ds, s->h.st, sizeof(sff::DevState), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        s->err = std::string("pic_histogram_static: ") + cudaGetErrorString(e);
        return PIC_ECUDA;
    }
    // the device status word, as pic_diag reads it
    if (ds.status & sff::FLAG_TIMEOUT) {
        s->err = "pic_histogram_static: a device wait timed out";
        return PIC_ETIMEOUT;
    }
    if (ds.status & sff::FLAG_CAPACITY) {
        s->err = "pic_histogram_static: a particle found no slot in its destination tile";
        return PIC_ECAPACITY;
    }
    const size_t nb = (size_t)n_e * n_a;
    e = cudaMemsetAsync(bins, 0, nb * sizeof(double), st);
    if (e == cudaSuccess) {
        sff::launch_histogram(s->d, s->cfg.precision, s->h.nptiles, ds.n_alive,
                              std::min<long long>(ds.n_exits, s->h.max_exits), n_e, e_max, n_a, bins, st);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(host_out, bins, nb * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        s->err = std::string("pic_histogram_static: ") + cudaGetErrorString(e);
        return PIC_ECUDA;
    }
    return PIC_OK;
}
