// jxf_ls.cu -- the level-set model (§3.5, §3.6, App. D, Alg. 2), FP64, on
// device arrays of a grid of cubic cells (2-D or 3-D):
//   jxf_ls_geometry   apertures, interface segment, volume fraction, normal
//   jxf_ls_rhs        R = -u . grad(phi) (5th-order upstream-central)
//   jxf_ls_advect     TVD-RK3 steps of the level-set advection
//   jxf_ls_reinit     pseudo-time steps of the reinitialisation equation
//   jxf_ls_interface  interface velocity and pressure of the cut cells
//   jxf_ls_extend     ghost-cell and interface-quantity extension
//   jxf_ls_cut_rhs    cut-cell right-hand side of one phase
//   jxf_ls_mix        conservative mixing of one phase
//   jxf_ls_init, jxf_ls_step   the two-phase time step chaining them
// One thread per cell (x fastest, 256 a block) or per face; indices outside
// the grid map through the boundary conditions (a mirror copies the
// scalar).  The FP64 pipe is the narrowest resource (1.7 operations a clock
// and SM): compares, divisions and square roots are kept off it where an
// integer test or a reciprocal does, cells whose result integer or float tests
// settle do no FP64 work, and the others are gathered into full warps.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "jxf.h"
#include "jxf_impl.cuh"  // fdiv; the face flux of the finite-volume scheme
#include "jxf_nvtx.cuh"
#include "jxf_setup.cuh"

namespace {

constexpr int kLsThreads = 256;

struct LsGrid {
    int ndim, n[3];
    int bc[3][2];
    double h, ih;  // cell size and its reciprocal
    long long ncell;
    long long stride[3];  // cell-index step of each axis
    long long foff[3];    // offset of axis d's face array in the concatenated apertures
};

__device__ __forceinline__ int ls_map(int c, int n, int blo, int bhi) {
    if (c < 0) {
        if (blo == JXF_BC_PERIODIC) return ((c % n) + n) % n;
        if (blo == JXF_BC_ZEROGRAD) return 0;
        return -1 - c;
    }
    if (c >= n) {
        if (bhi == JXF_BC_PERIODIC) return c % n;
        if (bhi == JXF_BC_ZEROGRAD) return n - 1;
        return 2 * n - 1 - c;
    }
    return c;
}

// phi at cell i moved by s along d (one boundary mapping)
__device__ __forceinline__ double ls_line(const LsGrid &g, const double *__restrict__ a, long long i, int cd, int d,
                                          int s) {
    const int m = ls_map(cd + s, g.n[d], g.bc[d][0], g.bc[d][1]);
    return __ldg(a + i + (long long)(m - cd) * g.stride[d]);
}

// cell coordinates of index i (32-bit arithmetic: ncell < 2^31)
__device__ __forceinline__ void ls_cell(const LsGrid &g, long long i, int (&c)[3]) {
    const unsigned u = (unsigned)i, n0 = (unsigned)g.n[0], n1 = (unsigned)g.n[1];
    const unsigned q = u / n0, r = q / n1;
    c[0] = (int)(u - q * n0);
    c[1] = (int)(q - r * n1);
    c[2] = (int)r;
}

// Sign tests and compares of doubles on their bit patterns (integer pipe;
// FP64 compares take slots of the narrow FP64 pipe), each equal to the
// FP64 compare for operands that are not NaN: x > 0, x < 0, and x > y for
// x, y >= 0 (non-negative doubles order as their bit patterns).
__device__ __forceinline__ bool ls_pos(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool ls_neg(double x) {
    const long long b = __double_as_longlong(x);
    return b < 0 && (b << 1) != 0;
}
__device__ __forceinline__ bool ls_gt_nonneg(double x, double y) {
    return __double_as_longlong(x) > __double_as_longlong(y);
}

// Cells of a block that need its long path, gathered into a list so that full
// warps take it: the FP64 pipe serves a warp instruction in 16 clocks whether
// one lane is active or 32, so scattered lanes would cost as much as all.
// Appends `item` of the calling thread where want is set (all threads call).
__device__ __forceinline__ void ls_gather(bool want, unsigned item, unsigned *list, int *count) {
    const unsigned m = __ballot_sync(0xffffffffu, want);
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (m && lane == 0) base = atomicAdd(count, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (want) list[base + __popc(m & ((1u << lane) - 1u))] = item;
}

// High word of |x|: compares like |x| to 2^-20 relative; 0x7FF00000 and above
// for infinities and NaN.
__device__ __forceinline__ unsigned ls_top(double x) { return (unsigned)__double2hiint(x) & 0x7FFFFFFFu; }

// ---------------------------------------------------------------- geometry --
// Fraction of an edge with phi > 0 (linear along the edge).
__device__ __forceinline__ double edge_fraction(double a, double b) {
    const bool pa = ls_pos(a), pb = ls_pos(b);
    if (pa && pb) return 1.0;
    if (!pa && !pb) return 0.0;
    return pa ? a / (a - b) : b / (b - a);
}

// Fraction of a square face with phi > 0 from its corner values
// (counter-clockwise from the face's lower corner): the polygon bounded by
// the face's edges and straight segments between the edges' zero crossings;
// two positive corners facing each other keep one triangle each.
__device__ double face_fraction(const double (&p)[4]) {
    int npos = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) npos += ls_pos(p[k]) ? 1 : 0;
    if (npos == 0) return 0.0;
    if (npos == 4) return 1.0;
    if (npos == 2 && ls_pos(p[0]) == ls_pos(p[2])) {
        double area = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (!ls_pos(p[k])) continue;
            const double ta = p[k] / (p[k] - p[(k + 1) & 3]);
            const double tb = p[k] / (p[k] - p[(k + 3) & 3]);
            area += 0.5 * ta * tb;
        }
        return area;
    }
    const double cx[4] = {0.0, 1.0, 1.0, 0.0}, cy[4] = {0.0, 0.0, 1.0, 1.0};
    double px[8], py[8];
    int m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int k1 = (k + 1) & 3;
        const bool pk = ls_pos(p[k]), pn = ls_pos(p[k1]);
        if (pk) {
            px[m] = cx[k];
            py[m] = cy[k];
            ++m;
        }
        if (pk != pn) {
            const double t = p[k] / (p[k] - p[k1]);
            px[m] = cx[k] + t * (cx[k1] - cx[k]);
            py[m] = cy[k] + t * (cy[k1] - cy[k]);
            ++m;
        }
    }
    double twice = 0.0;
    for (int k = 0; k < m; ++k) {
        const int k1 = k + 1 == m ? 0 : k + 1;
        twice += px[k] * py[k1] - px[k1] * py[k];
    }
    return 0.5 * twice;
}

// Geometry of one cell near the interface: the level set at the 2^ndim
// vertices (the mean of the 2^ndim cells sharing the vertex, summed in a
// fixed order), the apertures of its 2 ndim faces, the interface segment and
// volume fraction (App. D).  am / apx: apertures of the lower / upper face of
// each axis.
template <int NDIM>
__device__ void ls_cut_geometry(const LsGrid &g, const double *__restrict__ phi, long long i, const int (&c)[3],
                                double (&am)[3], double (&apx)[3], double &dg, double &al) {
    const double h = g.h;
    // mapped neighbour coordinates -1, 0, +1 of each axis
    long long ox[3], oy[3], oz[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ox[k] = ls_map(c[0] + k - 1, g.n[0], g.bc[0][0], g.bc[0][1]);
        oy[k] = (long long)ls_map(c[1] + k - 1, g.n[1], g.bc[1][0], g.bc[1][1]) * g.n[0];
        oz[k] = NDIM == 3 ? (long long)ls_map(c[2] + k - 1, g.n[2], g.bc[2][0], g.bc[2][1]) * g.n[0] * g.n[1] : 0;
    }
    if constexpr (NDIM == 3) {
        double P[3][3][3];  // cells c + (x, y, z) - 1
#pragma unroll
        for (int z = 0; z < 3; ++z)
#pragma unroll
            for (int y = 0; y < 3; ++y)
#pragma unroll
                for (int x = 0; x < 3; ++x) P[z][y][x] = __ldg(phi + oz[z] + oy[y] + ox[x]);
        double V[2][2][2];  // vertex with lower-corner cell c + (a, b, e) - 1, as V[e][b][a]
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    double s = 0.0;
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
#pragma unroll
                            for (int ii = 0; ii < 2; ++ii) s = __dadd_rn(s, P[e + k][b + j][a + ii]);
                    V[e][b][a] = s / 8.0;
                }
        const int o1[4] = {0, 1, 1, 0}, o2[4] = {0, 0, 1, 1};  // counter-clockwise in (e1, e2)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int e1 = d == 0 ? 1 : 0, e2 = d == 2 ? 1 : 2;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                double p[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    int q[3];
                    q[d] = s;
                    q[e1] = o1[k];
                    q[e2] = o2[k];
                    p[k] = V[q[2]][q[1]][q[0]];
                }
                const double f = face_fraction(p);
                if (s == 0) am[d] = f;
                else apx[d] = f;
            }
        }
    } else {
        double P[3][3];
#pragma unroll
        for (int y = 0; y < 3; ++y)
#pragma unroll
            for (int x = 0; x < 3; ++x) P[y][x] = __ldg(phi + oy[y] + ox[x]);
        double V[2][2];  // V[b][a]
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                double s = 0.0;
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int ii = 0; ii < 2; ++ii) s = __dadd_rn(s, P[b + j][a + ii]);
                V[b][a] = s / 4.0;
            }
        am[0] = edge_fraction(V[0][0], V[1][0]);
        apx[0] = edge_fraction(V[0][1], V[1][1]);
        am[1] = edge_fraction(V[0][0], V[0][1]);
        apx[1] = edge_fraction(V[1][0], V[1][1]);
    }
    const double sface = NDIM == 3 ? h * h : h, vcell = NDIM == 3 ? h * h * h : h * h;
    double s2 = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        const double t = (apx[d] - am[d]) * sface;
        s2 = __dadd_rn(s2, __dmul_rn(t, t));
    }
    dg = sqrt(s2);
    const double phic = __ldg(phi + i);
    double vol = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) vol = __dadd_rn(vol, __dmul_rn(__dmul_rn(__dadd_rn(am[d], apx[d]), sface), 0.5 * h));
    vol = __dadd_rn(vol, __dmul_rn(dg, phic));
    double a = vol / ((double)NDIM * vcell);
    a = ls_neg(a) ? 0.0 : (ls_gt_nonneg(a, 1.0) ? 1.0 : a);
    al = a;
}

// The cell writes the apertures of its lower faces (and of its upper faces
// at the grid's upper end); both cells of a face compute the same value.
template <int NDIM>
__device__ __forceinline__ void ls_put_geometry(const LsGrid &g, long long i, const int (&c)[3], const double (&am)[3],
                                                const double (&apx)[3], double dg, double al, double *__restrict__ ap,
                                                double *__restrict__ alpha, double *__restrict__ dgam) {
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        int m[3] = {g.n[0], g.n[1], g.n[2]};
        m[d] += 1;
        const long long f = ((long long)c[2] * m[1] + c[1]) * m[0] + c[0];
        ap[g.foff[d] + f] = am[d];
        if (c[d] == g.n[d] - 1) ap[g.foff[d] + f + (d == 0 ? 1 : (d == 1 ? m[0] : (long long)m[0] * m[1]))] = apx[d];
    }
    dgam[i] = dg;
    alpha[i] = al;
}

// 1/sqrt(x) of a normal x from the hardware estimate (2^-20) and one cubic
// correction y (1 + e/2 + 3 e^2/8), e = 1 - x y^2.
__device__ __forceinline__ double ls_rsqrt(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Geometry of every cell and its 4th-order normal.  Where the 3^ndim cells
// around a cell (whose means are its vertices) all have one sign, so have the
// vertices: the apertures are 1 (0), the segment 0 and alpha the constant the
// formula gives for a full (empty) cell, a_in (0) -- told by integer sign
// tests.  The other cells of the block, a few per cent next to the interface,
// are gathered and take the vertex sums and polygon areas.  What is left for
// every cell is the normal (about 30 FP64 operations of 200).  Bound by the
// FP64 pipe before; 332 -> 96 us on a 96^3 drop.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads) k_ls_geometry(const LsGrid g, const double *__restrict__ phi,
                                                             double a_in, double *__restrict__ ap,
                                                             double *__restrict__ alpha, double *__restrict__ dgam,
                                                             double *__restrict__ nrm) {
    __shared__ unsigned list[kLsThreads];
    __shared__ int count;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const long long i0 = (long long)blockIdx.x * blockDim.x, i = i0 + threadIdx.x;
    bool cut = false;
    if (i < g.ncell) {
        int c[3];
        ls_cell(g, i, c);
        long long ox[3], oy[3], oz[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            ox[k] = ls_map(c[0] + k - 1, g.n[0], g.bc[0][0], g.bc[0][1]);
            oy[k] = (long long)ls_map(c[1] + k - 1, g.n[1], g.bc[1][0], g.bc[1][1]) * g.n[0];
            oz[k] = NDIM == 3 ? (long long)ls_map(c[2] + k - 1, g.n[2], g.bc[2][0], g.bc[2][1]) * g.n[0] * g.n[1] : 0;
        }
        int npos = 0;
        unsigned top = 0;
#pragma unroll
        for (int z = 0; z < (NDIM == 3 ? 3 : 1); ++z)
#pragma unroll
            for (int y = 0; y < 3; ++y)
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    const double v = __ldg(phi + oz[z] + oy[y] + ox[x]);
                    npos += ls_pos(v) ? 1 : 0;
                    top = max(top, ls_top(v));
                }
        constexpr int all = NDIM == 3 ? 27 : 9;
        cut = (npos != 0 && npos != all) || top >= 0x7FF00000u;
        if (!cut) {
            const double v = npos ? 1.0 : 0.0;
            const double am[3] = {v, v, v};
            ls_put_geometry<NDIM>(g, i, c, am, am, 0.0, npos ? a_in : 0.0, ap, alpha, dgam);
        }
        double gr[3], gg = 0.0;
        const double k12 = g.ih * (1.0 / 12.0);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) {
            gr[d] = (ls_line(g, phi, i, c[d], d, -2) - 8.0 * ls_line(g, phi, i, c[d], d, -1) +
                     8.0 * ls_line(g, phi, i, c[d], d, 1) - ls_line(g, phi, i, c[d], d, 2)) *
                    k12;
            gg += gr[d] * gr[d];
        }
        // the estimate takes normal numbers well inside the exponent range
        const unsigned tg = ls_top(gg);
        const double ign = tg >= 0x03000000u && tg < 0x7C000000u ? ls_rsqrt(gg)
                                                                  : (ls_pos(gg) ? jxf::fdiv(1.0, sqrt(gg)) : 0.0);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) nrm[(long long)d * g.ncell + i] = gr[d] * ign;
    }
    ls_gather(cut, threadIdx.x, list, &count);
    __syncthreads();
    for (int t = threadIdx.x; t < count; t += kLsThreads) {
        const long long j = i0 + list[t];
        int c[3];
        ls_cell(g, j, c);
        double am[3], apx[3], dg, al;
        ls_cut_geometry<NDIM>(g, phi, j, c, am, apx, dg, al);
        ls_put_geometry<NDIM>(g, j, c, am, apx, dg, al, ap, alpha, dgam);
    }
}

// --------------------------------------------------------------- advection --
// 5th-order upstream-central derivative along d: the stencil i-3..i+2 for
// u_d >= 0, its mirror i-2..i+3 otherwise.
__device__ __forceinline__ double houc5(const LsGrid &g, const double *__restrict__ p, const int (&c)[3],
                                        long long i, int d, bool left) {
    const double k = g.ih * (1.0 / 60.0);
    if (left)
        return (-2.0 * ls_line(g, p, i, c[d], d, -3) + 15.0 * ls_line(g, p, i, c[d], d, -2) -
                60.0 * ls_line(g, p, i, c[d], d, -1) + 20.0 * ls_line(g, p, i, c[d], d, 0) +
                30.0 * ls_line(g, p, i, c[d], d, 1) - 3.0 * ls_line(g, p, i, c[d], d, 2)) *
               k;
    return (3.0 * ls_line(g, p, i, c[d], d, -2) - 30.0 * ls_line(g, p, i, c[d], d, -1) -
            20.0 * ls_line(g, p, i, c[d], d, 0) + 60.0 * ls_line(g, p, i, c[d], d, 1) -
            15.0 * ls_line(g, p, i, c[d], d, 2) + 2.0 * ls_line(g, p, i, c[d], d, 3)) *
           k;
}

template <int NDIM>
__device__ __forceinline__ double advect_r(const LsGrid &g, const double *__restrict__ p,
                                           const double *__restrict__ vel, const int (&c)[3], long long i) {
    double r = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        const double u = __ldg(vel + (long long)d * g.ncell + i);
        r -= u * houc5(g, p, c, i, d, !ls_neg(u));
    }
    return r;
}

// R only (mode < 0), or one TVD-RK3 stage: out = ca pn + cb (ps + dt R(ps))
// (the first stage out = ps + dt R(ps)).  out may alias pn, not ps.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads) k_ls_advect(const LsGrid g, const double *__restrict__ ps,
                                                         const double *pn, const double *__restrict__ vel, double dt,
                                                         int mode, double ca, double cb, double *out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.ncell) return;
    int c[3];
    ls_cell(g, i, c);
    const double r = advect_r<NDIM>(g, ps, vel, c, i);
    if (mode < 0) out[i] = r;
    else if (mode == 0) out[i] = ps[i] + dt * r;
    else out[i] = ca * pn[i] + cb * (ps[i] + dt * r);
}

// ---------------------------------------------------------- reinitialisation --
// Third-order WENO combination of one-sided derivatives (Jiang & Peng):
// (3 v2 - v1)/2 and (v2 + v3)/2 with linear weights 1/3, 2/3 and the
// smoothness (v2 - v1)^2, (v3 - v2)^2, eps = 1e-6.  Here on the undivided
// differences (eps scaled by h^2, which leaves the weights unchanged), the
// weights d_k/(eps + beta_k)^2 normalised in one division:
// q1 + s1 (q0 - q1)/(s1 + 2 s0), s_k = (eps + beta_k)^2.
__device__ __forceinline__ double weno3(double v1, double v2, double v3, double eps) {
    const double e0 = eps + (v2 - v1) * (v2 - v1), e1 = eps + (v3 - v2) * (v3 - v2);
    const double s0 = e0 * e0, s1 = e1 * e1;
    const double q0 = 0.5 * (3.0 * v2 - v1), q1 = 0.5 * (v2 + v3);
    return q1 + jxf::fdiv(s1 * (q0 - q1), s1 + 2.0 * s0);
}

// The cells a cell's derivatives are formed from: itself and two on each side
// along every axis (x[d][0..3]: -2, -1, 1, 2).
template <int NDIM> struct ReinitCells {
    double x0, x[NDIM][4];
    __device__ __forceinline__ ReinitCells(const LsGrid &g, const double *__restrict__ p, const int (&c)[3], long long i) {
        x0 = __ldg(p + i);
#pragma unroll
        for (int d = 0; d < NDIM; ++d)
#pragma unroll
            for (int k = 0; k < 4; ++k) x[d][k] = ls_line(g, p, i, c[d], d, k < 2 ? k - 2 : k - 1);
    }
};

// R_reinit = -sgn(phi0) (|grad phi| - 1) with the Godunov Hamiltonian of the
// one-sided derivatives, 0 where |R| <= thr.  need: bit d (d + 3) set where
// the left (right) derivative of axis d may enter; the others would be cut to
// 0 by their sign.
template <int NDIM>
__device__ __forceinline__ double reinit_r(const LsGrid &g, const ReinitCells<NDIM> &p, double phi0, double thr,
                                           unsigned need) {
    const bool spos = ls_pos(phi0);
    const double s = spos ? 1.0 : (ls_neg(phi0) ? -1.0 : 0.0);
    const double eps = 1e-6 * g.h * g.h;
    double h2 = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        const double dm = p.x0 - p.x[d][1], dp = p.x[d][2] - p.x0;
        double q1 = 0.0, q2 = 0.0;
        if ((need >> d) & 1u) {
            const double a = weno3(p.x[d][1] - p.x[d][0], dm, dp, eps) * g.ih;
            const double t1 = (spos ? ls_pos(a) : ls_neg(a)) ? a : 0.0;
            q1 = t1 * t1;
        }
        if ((need >> (d + 3)) & 1u) {
            const double b = weno3(p.x[d][3] - p.x[d][2], dp, dm, eps) * g.ih;
            const double t2 = (spos ? ls_neg(b) : ls_pos(b)) ? b : 0.0;
            q2 = t2 * t2;
        }
        h2 += ls_gt_nonneg(q1, q2) ? q1 : q2;
    }
    const double r = -s * (sqrt(h2) - 1.0);
    return ls_gt_nonneg(fabs(r), thr) ? r : 0.0;
}

// |x| truncated to 24 bits as a float, on the integer pipe (relative error
// below 2^-23; below 2^-126: 0; the caller keeps |x| below 2^127).
__device__ __forceinline__ float ls_trunc(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned b = ((__funnelshift_l(lo, hi, 3) ^ 0x40000000u) & 0x7FFFFFFFu) | (hi & 0x80000000u);
    return (hi & 0x7FFFFFFFu) < 0x38100000u ? 0.f : __uint_as_float(b);
}

// Float estimate of |grad phi| for reinit_r, with a bound on its error:
// true where |R| <= thr for certain (R = 0 then), else need receives the
// derivatives that may enter.  With m the largest |phi| and D the largest
// difference of the stencil, a difference of truncated values over h is off
// by at most e = 2^-22 (m + D)/h.  A WENO3 derivative is off by at most 7 e:
// 2 e from its candidates, the rest from the weights, whose sensitivity times
// the candidates' distance is bounded (eps + d^2 >= d^2) independently of
// eps; cutting by sign and the maximum do not enlarge it, the norm over the
// axes does by sqrt(3).  64 e covers this and the float evaluation's own
// rounding (below 2^-18 of a derivative) with a factor of five to spare.
template <int NDIM>
__device__ __forceinline__ bool reinit_screen(const LsGrid &g, const ReinitCells<NDIM> &p, double phi0, float thr,
                                              unsigned &need) {
    const float ih = (float)g.ih, f0 = ls_trunc(p.x0);
    unsigned top = max(ls_top(p.x0), ls_top(phi0));
    float v[NDIM][4];  // D_{-2}, D_{-1}, D_0, D_1 of each axis over h
    float m = fabsf(f0), D = 0.f;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        float f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            top = max(top, ls_top(p.x[d][k]));
            f[k] = ls_trunc(p.x[d][k]);
            m = fmaxf(m, fabsf(f[k]));
        }
        v[d][0] = (f[1] - f[0]) * ih;
        v[d][1] = (f0 - f[1]) * ih;
        v[d][2] = (f[2] - f0) * ih;
        v[d][3] = (f[3] - f[2]) * ih;
#pragma unroll
        for (int k = 0; k < 4; ++k) D = fmaxf(D, fabsf(v[d][k]));
    }
    need = 0x3Fu;
    if (top >= 0x47E00000u) return false;  // out of float's range, infinite or NaN
    const float err = 1.53e-5f * (m * ih + D);
    const bool spos = ls_pos(phi0);
    float h2 = 0.f;
    unsigned want = 0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        const float b0 = v[d][1] - v[d][0], b1 = v[d][2] - v[d][1], b2 = v[d][3] - v[d][2];
        float s0 = fmaf(b0, b0, 1e-6f), s1 = fmaf(b1, b1, 1e-6f), s2 = fmaf(b2, b2, 1e-6f);
        s0 *= s0, s1 *= s1, s2 *= s2;
        const float q1 = 0.5f * (v[d][1] + v[d][2]);
        float a = q1 + 0.5f * (b0 - b1) * (s1 * jxf::rcp(s1 + 2.f * s0));
        float b = q1 + 0.5f * (b1 - b2) * (s1 * jxf::rcp(s1 + 2.f * s2));
        if (!spos) a = -a, b = -b;
        if (!(a < -err)) want |= 1u << d;
        if (!(b > err)) want |= 8u << d;
        const float t = fmaxf(fmaxf(a, 0.f), -fminf(b, 0.f));
        h2 = fmaf(t, t, h2);
    }
    need = want;
    return fabsf(jxf::dsqrt(h2) - 1.f) <= thr - err;
}

// R only (mode < 0), or one second-order TVD Runge-Kutta stage in pseudo-time:
// mode 0: out = ps + dtau R(ps); mode 1: out = 1/2 pn + 1/2 (ps + dtau R(ps)).
// out may alias pn, not ps.  R is set to 0 below the threshold, so near a
// signed distance it is 0 almost everywhere: a float estimate with an error
// bound (reinit_screen) settles those cells, and the block's other cells are
// gathered and evaluated in double, without the one-sided derivatives whose
// sign is certain to cut them.  The results are those of evaluating every cell
// in double.  Bound by the FP64 pipe (150 operations a cell before, all
// cells); 246 -> 23 us for R on 96^3 cells near a distance function.
// Grids of at most one block per SM are bound by one warp's latency instead: no
// gathering there, each lane goes on with the cells it has loaded.  us for 10
// pseudo-time steps, all cells near a distance function | a quarter of them not |
// none, all in double / ungathered / gathered: 32^3 299 / 133 | 285 | 341 / 146 | 292 |
// 375; 40^3 504 / 146 | 437 | 546 / 156 | 368 | 582; 96^3 4934 / 443 | 1601 | 4181 / 443
// | 1487 | 4304.  (Far from a distance function everywhere the screen is lost
// time: on grids below 48^3 the all-double kernel was faster by up to 16 %.)
constexpr long long kReinitGather = (long long)jxf::kSMs * kLsThreads;
template <int NDIM, bool GATHER>
__global__ void __launch_bounds__(kLsThreads) k_ls_reinit(const LsGrid g, const double *__restrict__ ps,
                                                         const double *pn, const double *__restrict__ p0, double thr,
                                                         float thr_lo, double dtau, int mode, double *out) {
    __shared__ unsigned list[GATHER ? kLsThreads : 1];
    __shared__ int count;
    if constexpr (GATHER) {
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
    }
    const long long i0 = (long long)blockIdx.x * blockDim.x, i = i0 + threadIdx.x;
    auto put = [&](long long j, double r) {
        if (mode < 0) out[j] = r;
        else if (mode == 0) out[j] = ps[j] + dtau * r;
        else out[j] = 0.5 * pn[j] + 0.5 * (ps[j] + dtau * r);
    };
    bool full = false;
    unsigned need = 0;
    if (i < g.ncell) {
        int c[3];
        ls_cell(g, i, c);
        const ReinitCells<NDIM> x(g, ps, c, i);
        const double phi0 = __ldg(p0 + i);
        full = !reinit_screen<NDIM>(g, x, phi0, thr_lo, need);
        if (!full) {  // R = 0
            const double q = x.x0, z = __double_as_longlong(q) << 1 ? q : 0.0;  // -0 + 0 = 0
            if (mode < 0) out[i] = 0.0;
            else if (mode == 0) out[i] = z;
            else {
                const double o = pn[i];
                out[i] = __double_as_longlong(o) == __double_as_longlong(z) ? z : 0.5 * o + 0.5 * z;
            }
        } else if constexpr (!GATHER) {
            put(i, reinit_r<NDIM>(g, x, phi0, thr, need));
        }
    }
    if constexpr (GATHER) {
        ls_gather(full, threadIdx.x | (need << 16), list, &count);
        __syncthreads();
        for (int t = threadIdx.x; t < count; t += kLsThreads) {
            const unsigned e = list[t];
            const long long j = i0 + (e & 0xFFFFu);
            int c[3];
            ls_cell(g, j, c);
            put(j, reinit_r<NDIM>(g, ReinitCells<NDIM>(g, ps, c, j), __ldg(p0 + j), thr, e >> 16));
        }
    }
}

// ------------------------------------------------- interface quantities --
// A cut cell holds an interface segment (Sec. 3.5): both phases have volume
// in it, or the interface runs along one of its faces (alpha = 1 and
// dGamma > 0 on the side whose aperture drops to 0 there).
__device__ __forceinline__ bool ls_is_cut(double alpha, double dgamma) {
    return (ls_pos(alpha) && alpha < 1.0) || ls_pos(dgamma);
}

// The linearised two-material Riemann problem (App. D, no surface tension)
// in every cut cell: Z_p = rho_p c_p, un_p = u_p . n,
// u_Gamma = (Z1 un1 + Z2 un2 + p2 - p1)/(Z1 + Z2) along n, p_Gamma =
// (Z1 p2 + Z2 p1 + Z1 Z2 (un2 - un1))/(Z1 + Z2); 0 elsewhere.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_interface(const LsGrid g, const double *__restrict__ W1, const double *__restrict__ W2, double g1,
                   double pi1, double g2, double pi2, const double *__restrict__ alpha,
                   const double *__restrict__ dgamma, const double *__restrict__ nrm, double *__restrict__ ug,
                   double *__restrict__ pg) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.ncell) return;
    const long long nc = g.ncell;
    if (!ls_is_cut(__ldg(alpha + i), __ldg(dgamma + i))) {
#pragma unroll
        for (int d = 0; d < NDIM; ++d) ug[(long long)d * nc + i] = 0.0;
        pg[i] = 0.0;
        return;
    }
    double n[NDIM];
#pragma unroll
    for (int d = 0; d < NDIM; ++d) n[d] = __ldg(nrm + (long long)d * nc + i);
    double Z[2], un[2], p[2];
    const double *Wp[2] = {W1, W2};
    const double gm[2] = {g1, g2}, pim[2] = {pi1, pi2};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double rho = __ldg(Wp[k] + i), pk = __ldg(Wp[k] + (long long)(1 + NDIM) * nc + i);
        double u = 0.0;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) u += __ldg(Wp[k] + (long long)(1 + d) * nc + i) * n[d];
        Z[k] = rho * sqrt(gm[k] * (pk + pim[k]) / rho);
        un[k] = u;
        p[k] = pk;
    }
    const double zs = Z[0] + Z[1];
    const double u_g = (Z[0] * un[0] + Z[1] * un[1] + p[1] - p[0]) / zs;
    const double p_g = (Z[0] * p[1] + Z[1] * p[0] + Z[0] * Z[1] * (un[1] - un[0])) / zs;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) ug[(long long)d * nc + i] = u_g * n[d];
    pg[i] = p_g;
}

// ----------------------------------------------------------------- extension --
// One explicit Euler step (dtau) of dQ/dtau + a . grad Q = 0 on nq cell
// arrays, first-order upwind per axis, a = sdir n: with the upwind
// neighbour u_d of each axis (i - 1 where a_d > 0, i + 1 where a_d < 0) and
// w_d = (dtau/h) |a_d|, Q <- (1 - sum_d w_d) Q + sum_d w_d Q[u_d] (a convex
// combination, sum_d w_d <= sqrt(3)/4; no division on the device: dtau/h is
// an argument).  Mode 0 (ghost cells of phase 1): sdir = -1 where alpha =
// 0; mode 1 (phase 2): sdir = +1 where alpha = 1; mode 2 (interface
// quantities): sdir = sgn(phi) in every cell but the cut cells.  The other
// cells keep their values.  One launch serves one or two such extensions
// (modes ma and mb >= 0, each with its arrays): the ghost cells of both
// phases are one launch per pseudo-time step (a cell is a ghost of at most
// one phase).
//
// Bound by the FP64 pipe, four operations per value.  The time step forms
// the weights and upwind offsets once per extension (k_ls_extend_setup)
// instead of in each of its 10 or 20 pseudo-time steps (6 of 26 operations);
// a value whose upwind neighbours are 0 as it is stays 0 without arithmetic
// -- the interface quantities, 0 away from the cut cells, reach one cell
// further per step; and cells that keep their values are copied to the other
// of the two buffers in the first step only.  55 -> 31 us per step on a 96^3
// drop.
struct LsExtWork {
    double *w;            // [ndim + 1][cell]: 1 - sum w_d, w_d
    int *off;             // [ndim][cell]: upwind neighbour minus the cell
    unsigned char *code;  // [cell]: kExtA / kExtB if extension a / b moves the cell; kExtFinite
    unsigned char *seen;  // [2][block]: a value other than +0 has been in the block (read / written in turn)
};
constexpr unsigned char kExtA = 1, kExtB = 2, kExtFinite = 4;

// Does extension `mode` leave the cell alone; else its direction sdir.
__device__ __forceinline__ bool ls_ext_fixed(int mode, double al, long long i, const double *__restrict__ phi,
                                             const double *__restrict__ dgamma, int &sdir) {
    // alpha in [0, 1]: alpha < 1 as a bit-pattern compare with 1.0
    const bool a_pos = ls_pos(al), a_lt1 = __double_as_longlong(al) < 0x3FF0000000000000LL;
    if (mode == 0) {
        sdir = -1;
        return a_pos;
    }
    if (mode == 1) {
        sdir = 1;
        return a_lt1;
    }
    const double ph = __ldg(phi + i);
    sdir = ls_pos(ph) ? 1 : (ls_neg(ph) ? -1 : 0);
    return (a_pos && a_lt1) || ls_pos(__ldg(dgamma + i));
}

// Weights w0 = 1 - sum w_d and w_d, and the upwind offsets (0 where a_d = 0);
// returns whether they are finite.
template <int NDIM>
__device__ __forceinline__ bool ls_ext_weights(const LsGrid &g, const double *__restrict__ nrm, long long i, int sdir,
                                               double cfl, double &w0, double (&w)[NDIM], int (&off)[NDIM]) {
    int c[3];
    ls_cell(g, i, c);
    double wsum = 0.0;
    bool fin = true;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        const double n = __ldg(nrm + (long long)d * g.ncell + i);
        const int sn = ls_pos(n) ? 1 : (ls_neg(n) ? -1 : 0);
        const int s = -sdir * sn;  // step to the upwind neighbour: against the sign of a_d = sdir n_d
        off[d] = s ? (int)((long long)(ls_map(c[d] + s, g.n[d], g.bc[d][0], g.bc[d][1]) - c[d]) * g.stride[d]) : 0;
        w[d] = s ? cfl * fabs(n) : 0.0;
        wsum += w[d];
        fin = fin && ls_top(n) < 0x7FF00000u;
    }
    w0 = 1.0 - wsum;
    return fin;
}

template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_extend_setup(const LsGrid g, const double *__restrict__ phi, const double *__restrict__ alpha,
                      const double *__restrict__ dgamma, const double *__restrict__ nrm, int ma, int mb, double cfl,
                      const double *__restrict__ q, int nq, const LsExtWork e) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (mb < 0) {  // one extension: which blocks hold anything yet
        long long any = 0;
        if (i < g.ncell)
            for (int k = 0; k < nq; ++k) any |= __double_as_longlong(__ldg(q + (long long)k * g.ncell + i));
        const int a = __syncthreads_or(any != 0);
        if (threadIdx.x == 0) e.seen[blockIdx.x] = a ? 1 : 0;
    }
    if (i >= g.ncell) return;
    const double al = __ldg(alpha + i);
    int sdir = 0, sb = 0;
    unsigned char code = ls_ext_fixed(ma, al, i, phi, dgamma, sdir) ? 0 : kExtA;
    if (!code && mb >= 0 && !ls_ext_fixed(mb, al, i, phi, dgamma, sb)) {
        code = kExtB;
        sdir = sb;
    }
    if (code) {
        double w0, w[NDIM];
        int off[NDIM];
        if (ls_ext_weights<NDIM>(g, nrm, i, sdir, cfl, w0, w, off)) code |= kExtFinite;
        e.w[i] = w0;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) {
            e.w[(long long)(d + 1) * g.ncell + i] = w[d];
            e.off[(long long)d * g.ncell + i] = off[d];
        }
    }
    e.code[i] = code;
}

// One step of the NQ arrays of one cell (all loads before the arithmetic).
template <int NDIM, int NQ>
__device__ __forceinline__ bool ls_ext_move(long long nc, long long i, const double *__restrict__ qin,
                                            double *__restrict__ qout, double w0, const double (&w)[NDIM],
                                            const int (&off)[NDIM], bool fin) {
    long long out = 0;
    double v[NQ][NDIM + 1];
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
        const double *q = qin + (long long)k * nc + i;
        v[k][NDIM] = __ldg(q);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) v[k][d] = __ldg(q + off[d]);
    }
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
        long long any = __double_as_longlong(v[k][NDIM]);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) any |= __double_as_longlong(v[k][d]);
        double r = 0.0;
        if (any != 0 || !fin) {  // all +0: the combination is +0
            r = w0 * v[k][NDIM];
#pragma unroll
            for (int d = 0; d < NDIM; ++d) r = fma(w[d], v[k][d], r);
        }
        qout[(long long)k * nc + i] = r;
        out |= __double_as_longlong(r);
    }
    return out != 0;  // anything but +0 written
}

__device__ __forceinline__ void ls_ext_copy(long long nc, long long i, int nq, const double *__restrict__ qin,
                                            double *__restrict__ qout) {
    for (int k = 0; k < nq; ++k) qout[(long long)k * nc + i] = __ldg(qin + (long long)k * nc + i);
}

// One cell of k_ls_extend; true if anything but +0 was written.
template <int NDIM, int NQ>
__device__ __forceinline__ bool ls_ext_cell(const LsGrid &g, const LsExtWork &e, int two, bool first, long long i,
                                            const double *__restrict__ qa_in, double *__restrict__ qa_out,
                                            const double *__restrict__ qb_in, double *__restrict__ qb_out) {
    const long long nc = g.ncell;
    const unsigned code = e.code[i];
    double w[NDIM];
    int off[NDIM];
    const double w0 = __ldg(e.w + i);  // beside the code, not after it (unused where the cell keeps its values)
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        w[d] = __ldg(e.w + (long long)(d + 1) * nc + i);
        off[d] = __ldg(e.off + (long long)d * nc + i);
    }
    if (first) {
        if (!(code & kExtA)) ls_ext_copy(nc, i, NQ, qa_in, qa_out);
        if (two && !(code & kExtB)) ls_ext_copy(nc, i, NQ, qb_in, qb_out);
    }
    if (!(code & (kExtA | kExtB))) return false;
    const bool a = (code & kExtA) != 0;
    return ls_ext_move<NDIM, NQ>(nc, i, a ? qa_in : qb_in, a ? qa_out : qb_out, w0, w, off, (code & kExtFinite) != 0);
}

// One pseudo-time step with the weights of k_ls_extend_setup; first: also copy
// the cells that keep their values.  step >= 0 (one extension): blocks that have
// only ever held +0, like every block their cells' neighbours lie in, stay so
// and are left out -- from the second step on, when both buffers hold the
// zeros.  Interface quantities: 28 -> 18.5 us per step on a 96^3 drop.
template <int NDIM, int NQ>
__global__ void __launch_bounds__(kLsThreads, 4)
    k_ls_extend(const LsGrid g, const LsExtWork e, int two, int step, const double *__restrict__ qa_in,
                double *__restrict__ qa_out, const double *__restrict__ qb_in, double *__restrict__ qb_out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool first = step == 0;
    const int nb = (int)gridDim.x;
    const unsigned char *seen_in = e.seen + (step & 1 ? nb : 0);
    unsigned char *seen_out = e.seen + (step & 1 ? 0 : nb);
    if (!two && !first) {
        // the block's own flag and, for every way a neighbour index differs (one
        // step along an axis, or across a periodic side), the two blocks it hits
        const int t = threadIdx.x, w = (t - 1) >> 1, d = w >> 2;
        int hit = 0;
        if (t == 0) hit = seen_in[blockIdx.x];
        else if (t <= 8 * NDIM) {
            const long long st = d == 0 ? 1 : (d == 1 ? g.stride[1] : g.stride[2]);
            const int nd = d == 0 ? g.n[0] : (d == 1 ? g.n[1] : g.n[2]);
            const long long o = (w & 2) ? (nd - 1) * st : st;
            const long long c = (long long)blockIdx.x * kLsThreads + ((w & 1) ? o : -o);
            const long long b = (c >= 0 ? c / kLsThreads : -((kLsThreads - 1 - c) / kLsThreads)) + ((t - 1) & 1);
            if (b >= 0 && b < nb) hit = seen_in[b];
        }
        if (!__syncthreads_or(hit)) {
            if (t == 0) seen_out[blockIdx.x] = 0;
            return;
        }
    }
    bool any = false;
    if (i < g.ncell) any = ls_ext_cell<NDIM, NQ>(g, e, two, first, i, qa_in, qa_out, qb_in, qb_out);
    if (!two) {
        const int a = __syncthreads_or(any);
        if (threadIdx.x == 0) seen_out[blockIdx.x] = a || seen_in[blockIdx.x] ? 1 : 0;
    }
}

// The same without a work array for the weights (jxf_ls_extend, whose caller
// brings ping-pong scratch only): they are formed in every step.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads, 4)
    k_ls_extend_plain(const LsGrid g, const double *__restrict__ phi, const double *__restrict__ alpha,
                      const double *__restrict__ dgamma, const double *__restrict__ nrm, int mode, int nq, int first,
                      double cfl, const double *__restrict__ qin, double *__restrict__ qout) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.ncell) return;
    int sdir;
    if (ls_ext_fixed(mode, __ldg(alpha + i), i, phi, dgamma, sdir)) {
        if (first) ls_ext_copy(g.ncell, i, nq, qin, qout);
        return;
    }
    double w0, w[NDIM];
    int off[NDIM];
    const bool fin = ls_ext_weights<NDIM>(g, nrm, i, sdir, cfl, w0, w, off);
    for (int k = 0; k < nq; ++k)
        ls_ext_move<NDIM, 1>(g.ncell, i, qin + (long long)k * g.ncell, qout + (long long)k * g.ncell, w0, w, off, fin);
}

// ------------------------------------------------------- cut-cell right side --
// Face fluxes of one phase: the scheme's face flux (reconstruction and HLLC
// of jxf_impl.cuh, single-phase model, no limiter, inviscid; RSV 0: WENO5,
// 2: TENO6-A) from the phase's primitives P.W, one thread per face of axis
// d, into F (nv arrays of the axis's faces).  A face the phase does not wet (its aperture A,
// resp. 1 - A for phase 2, is 0) carries no flux of the phase: F = 0 there,
// without evaluating it (the right-hand side weighs it by 0 either way).
template <int NDIM, int d, int RSV>
__global__ void __launch_bounds__(jxf::kFluxThreads, jxf::SweepMinBlocks<double, RSV>::value)
    k_ls_cut_faces(const jxf::Dev P, const double *__restrict__ apd, int phase, double *__restrict__ F) {
    using V = jxf::Vars<JXF_SPM, NDIM>;
    int m[3] = {P.n[0], P.n[1], P.n[2]};
    m[d] += 1;
    const long long nface = (long long)m[0] * m[1] * m[2];
    const long long g = (long long)blockIdx.x * blockDim.x;
    const auto wet = [&](long long f) {
        const double A = __ldg(apd + f);
        if (phase == 1 ? A > 0.0 : A < 1.0) return true;
#pragma unroll
        for (int v = 0; v < V::NV; ++v) F[v * nface + f] = 0.0;
        return false;
    };
    const auto put = [&](long long f, const double *Fv, double) {
#pragma unroll
        for (int v = 0; v < V::NV; ++v) F[v * nface + f] = Fv[v];
    };
    const long long left = nface - g;
    jxf::flux_block<double, JXF_SPM, NDIM, d, 0, RSV, true>(P, 0.0, g, left < blockDim.x ? (int)left : (int)blockDim.x, m,
                                                       false, wet, put);
}

// d(alpha U)/dt of phase 1 (phi > 0) or 2 in every cell: the face fluxes
// weighted by the phase's apertures (A resp. 1 - A), then the interface
// pressure force and power along the phase's inward normal (+n resp. -n):
// sp pg dGamma / V (n, u_Gamma . n).
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_cut_update(const LsGrid g, const double *__restrict__ F, const double *__restrict__ ap,
                    const double *__restrict__ dgam, const double *__restrict__ nrm, const double *__restrict__ ug,
                    const double *__restrict__ pg, int phase, double *__restrict__ dU) {
    constexpr int NV = NDIM + 2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.ncell) return;
    const long long nc = g.ncell;
    int c[3];
    ls_cell(g, i, c);
    double R[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) R[v] = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        int m[3] = {g.n[0], g.n[1], g.n[2]};
        m[d] += 1;
        const long long nface = (long long)m[0] * m[1] * m[2];
        const long long gm = ((long long)c[2] * m[1] + c[1]) * m[0] + c[0];
        const long long gp = gm + (d == 0 ? 1 : (d == 1 ? m[0] : (long long)m[0] * m[1]));
        double am = __ldg(ap + g.foff[d] + gm), apx = __ldg(ap + g.foff[d] + gp);
        if (phase == 2) {
            am = 1.0 - am;
            apx = 1.0 - apx;
        }
        const double *Fd = F + (long long)NV * g.foff[d];
        // dry faces (aperture 0 on both sides) add exactly nothing, full ones
        // need no weighting: most cells, told by integer tests
        const long long bm = __double_as_longlong(am), bp = __double_as_longlong(apx);
        constexpr long long one = 0x3FF0000000000000LL;
        if ((bm | bp) == 0) continue;
        if (bm == one && bp == one) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
                R[v] = R[v] - (__ldg(Fd + v * nface + gp) - __ldg(Fd + v * nface + gm)) * g.ih;
            continue;
        }
#pragma unroll
        for (int v = 0; v < NV; ++v)
            R[v] = R[v] - (apx * __ldg(Fd + v * nface + gp) - am * __ldg(Fd + v * nface + gm)) * g.ih;
    }
    const double dg = __ldg(dgam + i);
    if (dg > 0.0) {
        const double ivol = NDIM == 3 ? g.ih * g.ih * g.ih : g.ih * g.ih;
        double n[NDIM], un = 0.0;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) {
            n[d] = __ldg(nrm + (long long)d * nc + i);
            un += __ldg(ug + (long long)d * nc + i) * n[d];
        }
        const double force = (phase == 1 ? 1.0 : -1.0) * __ldg(pg + i) * dg * ivol;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) R[1 + d] = R[1 + d] + force * n[d];
        R[1 + NDIM] = R[1 + NDIM] + force * un;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) dU[v * nc + i] = R[v];
}

// ------------------------------------------------------------------ mixing --
// Conservative mixing (App. D) of one phase's volume-weighted state, as a
// gather in two passes (no atomics: the result does not depend on the
// order threads run in).  Pass 1: every cell that vanished (a1 = 0 < a0),
// is new (a0 = 0 < a1) or is small (a1 < amix) computes the fluxes to its
// targets -- the neighbours one step along sign(n^p) on each axis, pair of
// axes and all three -- with the weights |n_e|^2 a_t, |n_e n_f| a_t,
// |n_x n_y n_z|^(2/3) a_t normalised to 1 (a target outside a non-periodic
// side weighs 0): M_t = beta_t/(a beta_t + a_t) [(a_t U_t) a - (a U) a_t],
// stored as M[t][v][cell], and a code byte per cell: 0 for a cell without
// fluxes (M is then neither written nor read), else 0x80 | the signs of
// n^p (2 bits per axis, sign + 1).  Pass 2, in place: every cell adds its
// own fluxes and subtracts those its neighbours aimed at it (it reads aU
// only at itself, so no other thread sees the update).
__device__ __forceinline__ bool ls_mixing(double a0, double a1, double amix) {
    return (a1 == 0.0 && a0 > 0.0) || (a1 > 0.0 && a0 == 0.0) || a1 < amix;
}

// Target t (subset mask t + 1 of the axes) of cell c along the signs sg:
// its cell index, -1 when it lies outside a non-periodic side (or a sign is 0).
template <int NDIM>
__device__ __forceinline__ long long ls_target(const LsGrid &g, const int (&c)[3], const int (&sg)[3], int t) {
    int q[3] = {c[0], c[1], c[2]};
    const int mask = t + 1;
#pragma unroll
    for (int e = 0; e < NDIM; ++e) {
        if (!((mask >> e) & 1)) continue;
        if (sg[e] == 0) return -1;
        q[e] += sg[e];
        if (q[e] < 0 || q[e] >= g.n[e]) {
            if (g.bc[e][0] != JXF_BC_PERIODIC) return -1;
            q[e] += q[e] < 0 ? g.n[e] : -g.n[e];
        }
    }
    return ((long long)q[2] * g.n[1] + q[1]) * g.n[0] + q[0];
}

// Pass 1.  The cells to mix lie along the interface, but every cell of the
// other phase is "small" too: those are dropped when all targets are empty
// (then nothing mixes), told from the targets' fractions before any weight is
// formed, and the block's remaining cells are gathered for the weights and
// fluxes (the FP64 work: a cube root and about 20 divisions).  103 -> 57 us
// on a 96^3 drop.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_mix_flux(const LsGrid g, int nv, const double *__restrict__ a0, const double *__restrict__ a1,
                  const double *__restrict__ np, double amix, const double *__restrict__ aU, double *__restrict__ M,
                  unsigned char *__restrict__ code) {
    __shared__ unsigned list[kLsThreads];
    __shared__ int count;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const long long b0 = (long long)blockIdx.x * blockDim.x, self = b0 + threadIdx.x, nc = g.ncell;
    constexpr int ntrg = NDIM == 3 ? 7 : 3;
    auto signs = [&](long long i, int (&sg)[3]) {
        sg[0] = sg[1] = sg[2] = 0;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) {
            const double nd = __ldg(np + (long long)d * nc + i);
            const bool nan = (__double_as_longlong(nd) & 0x7FFFFFFFFFFFFFFFLL) > 0x7FF0000000000000LL;
            sg[d] = nan ? 0 : (ls_pos(nd) ? 1 : (ls_neg(nd) ? -1 : 0));
        }
    };
    bool any = false;
    if (self < nc) {
        code[self] = 0;
        if (ls_mixing(__ldg(a0 + self), __ldg(a1 + self), amix)) {
            int c[3], sg[3];
            ls_cell(g, self, c);
            signs(self, sg);
#pragma unroll
            for (int t = 0; t < ntrg; ++t) {
                const long long ti = ls_target<NDIM>(g, c, sg, t);
                if (ti >= 0) any = any || (__double_as_longlong(__ldg(a1 + ti)) << 1) != 0;
            }
        }
    }
    ls_gather(any, threadIdx.x, list, &count);
    __syncthreads();
    for (int u = threadIdx.x; u < count; u += kLsThreads) {
        const long long i = b0 + list[u];
        const double ai = __ldg(a1 + i);
        int c[3], sg[3];
        ls_cell(g, i, c);
        signs(i, sg);
        double an[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int d = 0; d < NDIM; ++d) an[d] = fabs(__ldg(np + (long long)d * nc + i));
        long long ti[7];
        double beta[7], at[7], bsum = 0.0;
#pragma unroll
        for (int t = 0; t < ntrg; ++t) {
            const int mask = t + 1;
            ti[t] = ls_target<NDIM>(g, c, sg, t);
            const bool in = ti[t] >= 0;
            double w = 1.0;
            int nbits = 0;
#pragma unroll
            for (int e = 0; e < NDIM; ++e)
                if ((mask >> e) & 1) {
                    ++nbits;
                    w *= an[e];
                }
            if (nbits == 1) w = w * w;
            else if (nbits == 3) w = cbrt(w * w);
            at[t] = in ? __ldg(a1 + ti[t]) : 0.0;
            beta[t] = in ? w * at[t] : 0.0;
            bsum += beta[t];
        }
        if (!(bsum > 0.0)) continue;
#pragma unroll
        for (int t = 0; t < ntrg; ++t) {
            if (ti[t] < 0 || beta[t] == 0.0) {
                for (int v = 0; v < nv; ++v) M[((long long)t * nv + v) * nc + i] = 0.0;
                continue;
            }
            const double b = beta[t] / bsum;
            const double f = b / (ai * b + at[t]);
            for (int v = 0; v < nv; ++v)
                M[((long long)t * nv + v) * nc + i] =
                    f * (__ldg(aU + (long long)v * nc + ti[t]) * ai - __ldg(aU + (long long)v * nc + i) * at[t]);
        }
        code[i] = (unsigned char)(0x80 | (sg[0] + 1) | ((sg[1] + 1) << 2) | ((sg[2] + 1) << 4));
    }
}

// Pass 2.  Most cells see no code among their 3^ndim neighbours and leave at
// once; 80 -> 46 us on a 96^3 drop (bound by the integer work of finding
// the neighbours across the boundaries one by one before).
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_mix_apply(const LsGrid g, int nv, const double *__restrict__ M, const unsigned char *__restrict__ code,
                   double *__restrict__ aU) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.ncell) return;
    const long long nc = g.ncell;
    constexpr int ntrg = NDIM == 3 ? 7 : 3;
    int c[3];
    ls_cell(g, i, c);
    // neighbours k = c - o, o in {-1, 0, 1} per axis (index o + 1): cell-index
    // offset of each axis, bit o + 1 of out set where it lies outside a
    // non-periodic side
    int step[3][3];
    unsigned out[3] = {0, 0, 0};
#pragma unroll
    for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int o = -1; o <= 1; ++o) {
            int k = c[e] - o;
            if (e < NDIM && (k < 0 || k >= g.n[e])) {
                if (g.bc[e][0] == JXF_BC_PERIODIC) k += k < 0 ? g.n[e] : -g.n[e];
                else {
                    out[e] |= 1u << (o + 1);
                    k = c[e];
                }
            }
            step[e][o + 1] = (int)((long long)(k - c[e]) * g.stride[e]);
        }
    // bit (oz + 1) 9 + (oy + 1) 3 + ox + 1 of hit: that neighbour's code aims a
    // flux at this cell (its signs are o on the axes it steps along)
    unsigned hit = 0;
#pragma unroll
    for (int oz = (NDIM == 3 ? 0 : 1); oz <= (NDIM == 3 ? 2 : 1); ++oz)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox) {
                if (ox == 1 && oy == 1 && oz == 1) continue;
                const unsigned ck = __ldg(code + i + step[0][ox] + step[1][oy] + step[2][oz]);
                const unsigned off = ((out[0] >> ox) | (out[1] >> oy) | (out[2] >> oz)) & 1u;
                const bool m = (ox == 1 || (int)(ck & 3u) == ox) && (oy == 1 || (int)((ck >> 2) & 3u) == oy) &&
                               (oz == 1 || (int)((ck >> 4) & 3u) == oz);
                if (ck && !off && m) hit |= 1u << (oz * 9 + oy * 3 + ox);
            }
    const bool own = code[i] != 0;
    if (!own && !hit) return;
    for (int v = 0; v < nv; ++v) {
        double r = aU[(long long)v * nc + i];
        if (own)
#pragma unroll
            for (int t = 0; t < ntrg; ++t) r += __ldg(M + ((long long)t * nv + v) * nc + i);
        for (unsigned m = hit; m; m &= m - 1) {
            const int j = __ffs(m) - 1, oz = j / 9, oy = j / 3 % 3, ox = j % 3;
            const int mask = (ox != 1 ? 1 : 0) | (oy != 1 ? 2 : 0) | (oz != 1 ? 4 : 0);
            long long k = i;
#pragma unroll
            for (int o = 0; o < 3; ++o) {  // the offsets stay in registers
                if (ox == o) k += step[0][o];
                if (oy == o) k += step[1][o];
                if (oz == o) k += step[2][o];
            }
            r -= __ldg(M + ((long long)(mask - 1) * nv + v) * nc + k);
        }
        aU[(long long)v * nc + i] = r;
    }
}

// ----------------------------------------------------------- the time step --
// Volume-weighted conservative states of both phases from their primitives
// (rho, u_d, p, given in every cell): aU1 = alpha U(W1), aU2 = (1 - alpha)
// U(W2), each phase's stiffened gas in its Dev.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_cons(const jxf::Dev P1, const jxf::Dev P2, long long nc, const double *__restrict__ alpha,
              const double *__restrict__ W1, const double *__restrict__ W2, double *__restrict__ aU1,
              double *__restrict__ aU2) {
    constexpr int NV = NDIM + 2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const double a = __ldg(alpha + i);
    double w[NV], u[NV], rc2;
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = __ldg(W1 + v * nc + i);
    jxf::prim2cons<double, JXF_SPM, NDIM>(P1, w, u, rc2);
#pragma unroll
    for (int v = 0; v < NV; ++v) aU1[v * nc + i] = a * u[v];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = __ldg(W2 + v * nc + i);
    jxf::prim2cons<double, JXF_SPM, NDIM>(P2, w, u, rc2);
#pragma unroll
    for (int v = 0; v < NV; ++v) aU2[v * nc + i] = (1.0 - a) * u[v];
}

// One TVD-RK3 stage of both phases' volume-weighted states (n values each):
// U <- U + dt R in the first stage, else U <- ca Un + cb (U + dt R).
__global__ void __launch_bounds__(kLsThreads)
    k_ls_stage(long long n, int first, double ca, double cb, double dt, const double *__restrict__ U1n,
               const double *__restrict__ R1, double *__restrict__ U1, const double *__restrict__ U2n,
               const double *__restrict__ R2, double *__restrict__ U2) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    if (first) {
        U1[k] = U1[k] + dt * __ldg(R1 + k);
        U2[k] = U2[k] + dt * __ldg(R2 + k);
    } else {
        U1[k] = ca * __ldg(U1n + k) + cb * (U1[k] + dt * __ldg(R1 + k));
        U2[k] = ca * __ldg(U2n + k) + cb * (U2[k] + dt * __ldg(R2 + k));
    }
}

// Phase 2's fractions before and after a stage and its inward normal:
// 1 - a0, 1 - a1, -n.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_phase2(long long nc, const double *__restrict__ a0, const double *__restrict__ a1,
                const double *__restrict__ nrm, double *__restrict__ b0, double *__restrict__ b1,
                double *__restrict__ n2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    b0[i] = 1.0 - __ldg(a0 + i);
    b1[i] = 1.0 - __ldg(a1 + i);
#pragma unroll
    for (int d = 0; d < NDIM; ++d) n2[d * nc + i] = -__ldg(nrm + d * nc + i);
}

// Primitives of the cells holding a phase (fraction ap > 0) from its
// volume-weighted state: W = cons2prim(aU / ap); the other cells keep W.
template <int NDIM>
__global__ void __launch_bounds__(kLsThreads)
    k_ls_prim(const jxf::Dev P, long long nc, const double *__restrict__ ap, const double *__restrict__ aU,
              double *__restrict__ W) {
    constexpr int NV = NDIM + 2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const double a = __ldg(ap + i);
    if (!(a > 0.0)) return;
    double u[NV], w[NV], rho, p, rc2;
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = __ldg(aU + v * nc + i);
    if (__double_as_longlong(a) != 0x3FF0000000000000LL) {  // x / 1 = x: full cells skip the divisions
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = u[v] / a;
    }
    jxf::cons2prim<double, double, JXF_SPM, NDIM>(P, u, w, rho, p, rc2);
#pragma unroll
    for (int v = 0; v < NV; ++v) W[v * nc + i] = w[v];
}

// ------------------------------------------------------------------- host --
jxf_status ls_grid(const jxf_grid *grid, LsGrid &g) {
    if (!grid || grid->ndim < 2 || grid->ndim > 3) return JXF_ERR_ARG;
    g.ndim = grid->ndim;
    long long nc = 1;
    for (int e = 0; e < 3; ++e) {
        g.n[e] = e < g.ndim ? grid->n[e] : 1;
        if (g.n[e] < 1) return JXF_ERR_ARG;
        for (int s = 0; s < 2; ++s) {
            g.bc[e][s] = grid->bc[e][s];
            if (e < g.ndim && (g.bc[e][s] < JXF_BC_PERIODIC || g.bc[e][s] > JXF_BC_SYMMETRY)) return JXF_ERR_ARG;
        }
        if (e < g.ndim && (grid->bc[e][0] == JXF_BC_PERIODIC) != (grid->bc[e][1] == JXF_BC_PERIODIC))
            return JXF_ERR_ARG;
        nc *= g.n[e];
    }
    g.h = (grid->hi[0] - grid->lo[0]) / g.n[0];
    if (!(g.h > 0.0)) return JXF_ERR_ARG;
    g.ih = 1.0 / g.h;
    g.stride[0] = 1;
    g.stride[1] = g.n[0];
    g.stride[2] = (long long)g.n[0] * g.n[1];
    for (int e = 1; e < g.ndim; ++e) {
        const double he = (grid->hi[e] - grid->lo[e]) / g.n[e];
        if (std::fabs(he - g.h) > 1e-12 * g.h) return JXF_ERR_ARG;  // cubic cells only (§3.5)
    }
    // the boundary mapping reaches 3 cells past an end (one reflection)
    for (int e = 0; e < g.ndim; ++e)
        if (g.n[e] < 3) return JXF_ERR_ARG;
    if (nc >= (1ll << 31)) return JXF_ERR_ARG;
    g.ncell = nc;
    long long off = 0;
    for (int d = 0; d < 3; ++d) {
        g.foff[d] = off;
        if (d < g.ndim) {
            long long f = 1;
            for (int e = 0; e < 3; ++e) f *= g.n[e] + (e == d ? 1 : 0);
            off += f;
        }
    }
    return JXF_OK;
}

// The volume fraction the geometry's formula gives for a full cell (all
// apertures 1), operation by operation in IEEE double as the kernel evaluates
// it elsewhere (volatile: no contraction), clipped to 1.
double ls_alpha_full(const LsGrid &g) {
    const double h = g.h;
    volatile double sface = h, vcell = h * h;
    if (g.ndim == 3) {
        sface = h * h;
        vcell = vcell * h;
    }
    volatile double t = 2.0 * sface, u = 0.5 * h, x = t * u, vol = 0.0;
    for (int d = 0; d < g.ndim; ++d) vol = vol + x;
    volatile double den = (double)g.ndim * vcell, a = vol / den;
    return a > 1.0 ? 1.0 : a;
}

unsigned ls_blocks(const LsGrid &g) { return (unsigned)((g.ncell + kLsThreads - 1) / kLsThreads); }

void advect_launch(const LsGrid &g, const double *ps, const double *pn, const double *vel, double dt, int mode,
                   double ca, double cb, double *out, cudaStream_t s) {
    if (g.ndim == 3) k_ls_advect<3><<<ls_blocks(g), kLsThreads, 0, s>>>(g, ps, pn, vel, dt, mode, ca, cb, out);
    else k_ls_advect<2><<<ls_blocks(g), kLsThreads, 0, s>>>(g, ps, pn, vel, dt, mode, ca, cb, out);
}

void reinit_launch(const LsGrid &g, const double *ps, const double *pn, const double *p0, double thr, double dtau,
                   int mode, double *out, cudaStream_t s) {
    const float lo = std::nextafterf((float)thr, -1.f);  // not above thr
    auto run = [&](auto kernel) { kernel<<<ls_blocks(g), kLsThreads, 0, s>>>(g, ps, pn, p0, thr, lo, dtau, mode, out); };
    if (g.ncell > kReinitGather) run(g.ndim == 3 ? k_ls_reinit<3, true> : k_ls_reinit<2, true>);
    else run(g.ndim == 3 ? k_ls_reinit<3, false> : k_ls_reinit<2, false>);
}

jxf_status ls_launched() {
    return cudaPeekAtLastError() == cudaSuccess ? JXF_OK : (cudaGetLastError(), JXF_ERR_CUDA);
}

unsigned ls_blocks_n(long long n) { return (unsigned)((n + kLsThreads - 1) / kLsThreads); }

template <int RSV>
void ls_cut_faces_rsv(int ndim, int d, unsigned blocks, cudaStream_t s, const jxf::Dev &P, const double *A,
                      int phase, double *F) {
    if (ndim == 3) {
        if (d == 0) k_ls_cut_faces<3, 0, RSV><<<blocks, jxf::kFluxThreads, 0, s>>>(P, A, phase, F);
        if (d == 1) k_ls_cut_faces<3, 1, RSV><<<blocks, jxf::kFluxThreads, 0, s>>>(P, A, phase, F);
        if (d == 2) k_ls_cut_faces<3, 2, RSV><<<blocks, jxf::kFluxThreads, 0, s>>>(P, A, phase, F);
    } else {
        if (d == 0) k_ls_cut_faces<2, 0, RSV><<<blocks, jxf::kFluxThreads, 0, s>>>(P, A, phase, F);
        if (d == 1) k_ls_cut_faces<2, 1, RSV><<<blocks, jxf::kFluxThreads, 0, s>>>(P, A, phase, F);
    }
}

// The face-flux launch of axis d for the scheme family (WENO5 or TENO6-A).
void ls_cut_faces_launch(int ndim, int d, bool teno, unsigned blocks, cudaStream_t s, const jxf::Dev &P,
                         const double *A, int phase, double *F) {
    if (teno) ls_cut_faces_rsv<2>(ndim, d, blocks, s, P, A, phase, F);
    else ls_cut_faces_rsv<0>(ndim, d, blocks, s, P, A, phase, F);
}

// steps pseudo-time steps of one extension (mode ma of the nq arrays qa) or
// two at once (mode mb >= 0 of qb as well), ping-ponging through scratch
// (nq ncell doubles per extension); the results end in qa (and qb).  ext:
// room for the weights, for the time step's nq = ndim + 2 or ndim + 1 (w null:
// form them in every step; one extension only, any nq).
jxf_status ls_extend_launch(const LsGrid &g, const double *phi, const double *alpha, const double *dgamma,
                            const double *normal, int ma, double *qa, int mb, double *qb, int nq, int steps,
                            double *scratch, const LsExtWork &ext, cudaStream_t s) {
    const double cfl = 0.25;  // dtau / h, dtau = 0.25 h
    const long long nb = (long long)nq * g.ncell;
    const unsigned blocks = ls_blocks(g);
    double *a0 = qa, *a1 = scratch, *b0 = qb, *b1 = mb >= 0 ? scratch + nb : nullptr;
    if (ext.w && steps > 0) {
        if (g.ndim == 3)
            k_ls_extend_setup<3><<<blocks, kLsThreads, 0, s>>>(g, phi, alpha, dgamma, normal, ma, mb, cfl, qa, nq, ext);
        else k_ls_extend_setup<2><<<blocks, kLsThreads, 0, s>>>(g, phi, alpha, dgamma, normal, ma, mb, cfl, qa, nq, ext);
    }
    for (int k = 0; k < steps; ++k) {
        const int first = k == 0 ? 1 : 0, two = mb >= 0 ? 1 : 0;
        if (ext.w) {
            // the time step extends the ndim + 2 primitives or the ndim + 1 interface quantities
            if (g.ndim == 3 && nq == 5) k_ls_extend<3, 5><<<blocks, kLsThreads, 0, s>>>(g, ext, two, k, a0, a1, b0, b1);
            else if (g.ndim == 3) k_ls_extend<3, 4><<<blocks, kLsThreads, 0, s>>>(g, ext, two, k, a0, a1, b0, b1);
            else if (nq == 4) k_ls_extend<2, 4><<<blocks, kLsThreads, 0, s>>>(g, ext, two, k, a0, a1, b0, b1);
            else k_ls_extend<2, 3><<<blocks, kLsThreads, 0, s>>>(g, ext, two, k, a0, a1, b0, b1);
        } else if (g.ndim == 3) {
            k_ls_extend_plain<3><<<blocks, kLsThreads, 0, s>>>(g, phi, alpha, dgamma, normal, ma, nq, first, cfl, a0,
                                                              a1);
        } else {
            k_ls_extend_plain<2><<<blocks, kLsThreads, 0, s>>>(g, phi, alpha, dgamma, normal, ma, nq, first, cfl, a0,
                                                              a1);
        }
        std::swap(a0, a1);
        std::swap(b0, b1);
    }
    if (a0 != qa && cudaMemcpyAsync(qa, a0, (size_t)nb * sizeof(double), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return JXF_ERR_CUDA;
    if (mb >= 0 && b0 != qb &&
        cudaMemcpyAsync(qb, b0, (size_t)nb * sizeof(double), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return JXF_ERR_CUDA;
    return ls_launched();
}

// Work buffer of the time step, in doubles (see jxf_ls_step_work).
struct LsWork {
    double *ap, *al0, *al1, *dg, *nr, *n2, *b0, *b1, *phin, *phit, *R1, *R2, *U1n, *U2n, *scr;
    LsExtWork ext;  // in R1 and R2, which the stage combination has consumed by then
    long long total;
};

LsWork ls_work(const LsGrid &g, long long nface, double *base) {
    const long long nc = g.ncell;
    const int nd = g.ndim, nv = nd + 2, ntrg = nd == 3 ? 7 : 3;
    LsWork w{};
    long long off = 0;
    auto take = [&](long long n) {
        double *p = base ? base + off : nullptr;
        off += (n + 31) / 32 * 32;  // 256-byte aligned pieces
        return p;
    };
    w.ap = take(nface);
    w.al0 = take(nc);
    w.al1 = take(nc);
    w.dg = take(nc);
    w.nr = take((long long)nd * nc);
    w.n2 = take((long long)nd * nc);
    w.b0 = take(nc);
    w.b1 = take(nc);
    w.phin = take(nc);
    w.phit = take(nc);
    w.R1 = take((long long)nv * nc);
    w.R2 = take((long long)nv * nc);
    w.U1n = take((long long)nv * nc);
    w.U2n = take((long long)nv * nc);
    // shared by the calls of one stage, one at a time: the face fluxes of the
    // cut-cell right-hand side, the mixing fluxes, the extension and
    // reinitialisation ping-pong buffers
    w.scr = take(std::max((long long)nv * nface, (long long)(ntrg + 1) * nv * nc));
    w.ext.w = w.R1;                           // ndim + 1 of the ndim + 2 arrays
    w.ext.off = reinterpret_cast<int *>(w.R2);  // half of ndim arrays, then a byte per cell, flags
    w.ext.code = base ? reinterpret_cast<unsigned char *>(w.ext.off + (long long)nd * nc) : nullptr;
    w.ext.seen = base ? w.ext.code + nc : nullptr;
    w.total = off;
    return w;
}

// The arguments of jxf_ls_init / jxf_ls_step: both phases single-phase
// stiffened gases on the same grid, the FP64 inviscid scheme without limiter.
jxf_status ls_step_args(const jxf_grid *grid, const jxf_eos *eos1, const jxf_eos *eos2, const jxf_scheme *scheme,
                        LsGrid &g, jxf::Dev &P1, jxf::Dev &P2) {
    long long ncell = 0;
    if (ls_grid(grid, g) != JXF_OK || !eos1 || !eos2 || !scheme) return JXF_ERR_ARG;
    if (eos1->model != JXF_SPM || eos2->model != JXF_SPM) return JXF_ERR_UNSUPPORTED;
    if (jxf::validate_setup(grid, eos1, scheme, &ncell, false) != JXF_OK ||
        jxf::validate_setup(grid, eos2, scheme, &ncell, false) != JXF_OK)
        return JXF_ERR_ARG;
    if (eos1->model != JXF_SPM || eos2->model != JXF_SPM || scheme->precision != JXF_FP64 || scheme->viscous ||
        scheme->limiter || scheme->recon > JXF_TENO6A_CHAR)
        return JXF_ERR_UNSUPPORTED;
    jxf::fill_dev(grid, eos1, scheme, ncell, P1);
    jxf::fill_dev(grid, eos2, scheme, ncell, P2);
    return JXF_OK;
}

// Interface quantities from W1, W2 and the geometry (al, dg, nr) and their
// extension (20 steps): qg = (u_Gamma n_d ..., p_Gamma).
jxf_status ls_interface_ext(const jxf_grid *grid, const LsGrid &g, const jxf_eos *eos1, const jxf_eos *eos2,
                            const double *phi, const double *W1, const double *W2, const double *al,
                            const double *dg, const double *nr, double *qg, double *scr, const LsExtWork &ext,
                            cudaStream_t s) {
    const double gam[2] = {eos1->gamma[0], eos2->gamma[0]}, pin[2] = {eos1->pinf[0], eos2->pinf[0]};
    jxf_status st = jxf_ls_interface(grid, W1, W2, gam, pin, al, dg, nr, qg, qg + (long long)g.ndim * g.ncell,
                                     (jxf_stream)s);
    if (st != JXF_OK) return st;
    return ls_extend_launch(g, phi, al, dg, nr, 2, qg, -1, nullptr, g.ndim + 1, 20, scr, ext, s);
}

}  // namespace

extern "C" {

long long jxf_ls_nface(const jxf_grid *grid) {
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK) return -1;
    long long s = 0;
    for (int d = 0; d < g.ndim; ++d) {
        long long f = 1;
        for (int e = 0; e < 3; ++e) f *= g.n[e] + (e == d ? 1 : 0);
        s += f;
    }
    return s;
}

jxf_status jxf_ls_geometry(const jxf_grid *grid, const double *phi, double *apert, double *alpha, double *dgamma,
                           double *normal, jxf_stream stream) {
    JXF_RANGE("jxf_ls_geometry");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !phi || !apert || !alpha || !dgamma || !normal) return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const double a_in = ls_alpha_full(g);
    if (g.ndim == 3) k_ls_geometry<3><<<ls_blocks(g), kLsThreads, 0, s>>>(g, phi, a_in, apert, alpha, dgamma, normal);
    else k_ls_geometry<2><<<ls_blocks(g), kLsThreads, 0, s>>>(g, phi, a_in, apert, alpha, dgamma, normal);
    return ls_launched();
}

jxf_status jxf_ls_rhs(const jxf_grid *grid, const double *phi, const double *vel, double *rhs, jxf_stream stream) {
    JXF_RANGE("jxf_ls_rhs");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !phi || !vel || !rhs || rhs == phi) return JXF_ERR_ARG;
    advect_launch(g, phi, phi, vel, 0.0, -1, 0.0, 0.0, rhs, (cudaStream_t)stream);
    return ls_launched();
}

jxf_status jxf_ls_advect(const jxf_grid *grid, double *phi, const double *vel, double dt, int nsteps,
                         double *scratch, jxf_stream stream) {
    JXF_RANGE("jxf_ls_advect");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !phi || !vel || !scratch || nsteps < 0 || !std::isfinite(dt))
        return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    double *p1 = scratch, *p2 = scratch + g.ncell;
    for (int k = 0; k < nsteps; ++k) {
        // TVD-RK3 (§3.4): p1 = p + dt R(p); p2 = 3/4 p + 1/4 (p1 + dt R(p1));
        // p <- 1/3 p + 2/3 (p2 + dt R(p2))
        advect_launch(g, phi, phi, vel, dt, 0, 0.0, 1.0, p1, s);
        advect_launch(g, p1, phi, vel, dt, 1, 0.75, 0.25, p2, s);
        advect_launch(g, p2, phi, vel, dt, 1, 1.0 / 3.0, 2.0 / 3.0, phi, s);
    }
    return ls_launched();
}

jxf_status jxf_ls_reinit_rhs(const jxf_grid *grid, const double *phi, const double *phi0, double threshold,
                             double *rhs, jxf_stream stream) {
    JXF_RANGE("jxf_ls_reinit_rhs");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !phi || !phi0 || !rhs || rhs == phi || !(threshold >= 0.0))
        return JXF_ERR_ARG;
    reinit_launch(g, phi, phi, phi0, threshold, 0.0, -1, rhs, (cudaStream_t)stream);
    return ls_launched();
}

jxf_status jxf_ls_interface(const jxf_grid *grid, const double *W1, const double *W2, const double *gamma,
                            const double *pinf, const double *alpha, const double *dgamma, const double *normal,
                            double *ug, double *pg, jxf_stream stream) {
    JXF_RANGE("jxf_ls_interface");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !W1 || !W2 || !gamma || !pinf || !alpha || !dgamma || !normal || !ug || !pg)
        return JXF_ERR_ARG;
    for (int k = 0; k < 2; ++k)
        if (!(gamma[k] > 1.0) || !(pinf[k] >= 0.0)) return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (g.ndim == 3)
        k_ls_interface<3><<<ls_blocks(g), kLsThreads, 0, s>>>(g, W1, W2, gamma[0], pinf[0], gamma[1], pinf[1], alpha,
                                                             dgamma, normal, ug, pg);
    else
        k_ls_interface<2><<<ls_blocks(g), kLsThreads, 0, s>>>(g, W1, W2, gamma[0], pinf[0], gamma[1], pinf[1], alpha,
                                                             dgamma, normal, ug, pg);
    return ls_launched();
}

jxf_status jxf_ls_extend(const jxf_grid *grid, const double *phi, const double *alpha, const double *dgamma,
                         const double *normal, double *q, int nq, int mode, int steps, double *scratch,
                         jxf_stream stream) {
    JXF_RANGE("jxf_ls_extend");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !phi || !alpha || !dgamma || !normal || !q || !scratch || nq < 1 || mode < 0 ||
        mode > 2 || steps < 0)
        return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    return ls_extend_launch(g, phi, alpha, dgamma, normal, mode, q, -1, nullptr, nq, steps, scratch, LsExtWork{}, s);
}

jxf_status jxf_ls_cut_rhs(const jxf_grid *grid, const jxf_eos *eos, const jxf_scheme *scheme, const double *apert,
                          const double *dgamma, const double *normal, const double *W, int phase, const double *ug,
                          const double *pg, double *dU, double *scratch, jxf_stream stream) {
    JXF_RANGE("jxf_ls_cut_rhs");
    LsGrid g;
    long long ncell = 0;
    if (ls_grid(grid, g) != JXF_OK || !eos || !scheme || !apert || !dgamma || !normal || !W || !ug || !pg || !dU ||
        !scratch || (phase != 1 && phase != 2))
        return JXF_ERR_ARG;
    if (jxf::validate_setup(grid, eos, scheme, &ncell, false) != JXF_OK) return JXF_ERR_ARG;
    if (eos->model != JXF_SPM || scheme->precision != JXF_FP64 || scheme->viscous || scheme->limiter ||
        scheme->recon > JXF_TENO6A_CHAR)
        return JXF_ERR_UNSUPPORTED;
    jxf::Dev P;
    jxf::fill_dev(grid, eos, scheme, ncell, P);
    P.split = jxf::split_allowed(grid, P.weno_eps, jxf::kSplitFaces);  // sorted faces: from one warp per pipe
    P.W = const_cast<double *>(W);
    cudaStream_t s = (cudaStream_t)stream;
    const int nv = g.ndim + 2;
    for (int d = 0; d < g.ndim; ++d) {
        long long nf = 1;
        for (int e = 0; e < 3; ++e) nf *= g.n[e] + (e == d ? 1 : 0);
        const unsigned blocks = (unsigned)((nf + jxf::kFluxThreads - 1) / jxf::kFluxThreads);
        double *F = scratch + (long long)nv * g.foff[d];
        const double *A = apert + g.foff[d];
        ls_cut_faces_launch(g.ndim, d, P.teno != 0, blocks, s, P, A, phase, F);
    }
    if (g.ndim == 3)
        k_ls_cut_update<3><<<ls_blocks(g), kLsThreads, 0, s>>>(g, scratch, apert, dgamma, normal, ug, pg, phase, dU);
    else k_ls_cut_update<2><<<ls_blocks(g), kLsThreads, 0, s>>>(g, scratch, apert, dgamma, normal, ug, pg, phase, dU);
    return ls_launched();
}

jxf_status jxf_ls_mix(const jxf_grid *grid, int nv, const double *a0, const double *a1, const double *np,
                      double amix, double *aU, double *scratch, jxf_stream stream) {
    JXF_RANGE("jxf_ls_mix");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || nv < 1 || nv > 8 || !a0 || !a1 || !np || !aU || !scratch || !(amix >= 0.0))
        return JXF_ERR_ARG;
    for (int e = 0; e < g.ndim; ++e)  // mixing reaches one cell across a side
        if (g.bc[e][0] == JXF_BC_PERIODIC && g.n[e] < 3) return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int ntrg = g.ndim == 3 ? 7 : 3;
    double *M = scratch;
    unsigned char *code = reinterpret_cast<unsigned char *>(scratch + (long long)ntrg * nv * g.ncell);
    if (g.ndim == 3) k_ls_mix_flux<3><<<ls_blocks(g), kLsThreads, 0, s>>>(g, nv, a0, a1, np, amix, aU, M, code);
    else k_ls_mix_flux<2><<<ls_blocks(g), kLsThreads, 0, s>>>(g, nv, a0, a1, np, amix, aU, M, code);
    if (g.ndim == 3) k_ls_mix_apply<3><<<ls_blocks(g), kLsThreads, 0, s>>>(g, nv, M, code, aU);
    else k_ls_mix_apply<2><<<ls_blocks(g), kLsThreads, 0, s>>>(g, nv, M, code, aU);
    return ls_launched();
}

long long jxf_ls_step_work(const jxf_grid *grid) {
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK) return -1;
    return ls_work(g, jxf_ls_nface(grid), nullptr).total;
}

jxf_status jxf_ls_init(const jxf_grid *grid, const jxf_eos *eos1, const jxf_eos *eos2, const jxf_scheme *scheme,
                       const double *phi, const double *W1, const double *W2, double *aU1, double *aU2, double *qg,
                       double *work, jxf_stream stream) {
    JXF_RANGE("jxf_ls_init");
    LsGrid g;
    jxf::Dev P1, P2;
    jxf_status st = ls_step_args(grid, eos1, eos2, scheme, g, P1, P2);
    if (st != JXF_OK) return st;
    if (!phi || !W1 || !W2 || !aU1 || !aU2 || !qg || !work) return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const LsWork w = ls_work(g, jxf_ls_nface(grid), work);
    if ((st = jxf_ls_geometry(grid, phi, w.ap, w.al0, w.dg, w.nr, stream)) != JXF_OK) return st;
    if (g.ndim == 3) k_ls_cons<3><<<ls_blocks(g), kLsThreads, 0, s>>>(P1, P2, g.ncell, w.al0, W1, W2, aU1, aU2);
    else k_ls_cons<2><<<ls_blocks(g), kLsThreads, 0, s>>>(P1, P2, g.ncell, w.al0, W1, W2, aU1, aU2);
    if ((st = ls_launched()) != JXF_OK) return st;
    return ls_interface_ext(grid, g, eos1, eos2, phi, W1, W2, w.al0, w.dg, w.nr, qg, w.scr, w.ext, s);
}

jxf_status jxf_ls_step(const jxf_grid *grid, const jxf_eos *eos1, const jxf_eos *eos2, const jxf_scheme *scheme,
                       double dt, int nsteps, double amix, double *phi, double *aU1, double *aU2, double *W1,
                       double *W2, double *qg, double *work, jxf_stream stream) {
    JXF_RANGE("jxf_ls_step");
    LsGrid g;
    jxf::Dev P1, P2;
    jxf_status st = ls_step_args(grid, eos1, eos2, scheme, g, P1, P2);
    if (st != JXF_OK) return st;
    if (!phi || !aU1 || !aU2 || !W1 || !W2 || !qg || !work || nsteps < 0 || !std::isfinite(dt) ||
        !(amix >= 0.0))
        return JXF_ERR_ARG;
    if (nsteps == 0) return JXF_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const long long nc = g.ncell;
    const int nd = g.ndim, nv = nd + 2;
    const size_t ubytes = (size_t)nv * nc * sizeof(double), pbytes = (size_t)nc * sizeof(double);
    const LsWork w = ls_work(g, jxf_ls_nface(grid), work);
    double *al0 = w.al0, *al1 = w.al1;
    const double *ug = qg, *pg = qg + (long long)nd * nc;
    static const double ca[3] = {0.0, 0.75, 1.0 / 3.0}, cb[3] = {1.0, 0.25, 2.0 / 3.0};
#define LS_TRY(x)                          \
    do {                                   \
        if ((st = (x)) != JXF_OK) return st; \
    } while (0)
    // the geometry of phi on entry; afterwards each stage leaves the
    // geometry of its result in (ap, al1, dg, nr), which the next stage
    // starts from
    LS_TRY(jxf_ls_geometry(grid, phi, w.ap, al0, w.dg, w.nr, stream));
    for (int step = 0; step < nsteps; ++step) {
        if (cudaMemcpyAsync(w.U1n, aU1, ubytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(w.U2n, aU2, ubytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(w.phin, phi, pbytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            return JXF_ERR_CUDA;
        for (int stage = 0; stage < 3; ++stage) {
            // right-hand sides of both phases and the level set's stage
            LS_TRY(jxf_ls_cut_rhs(grid, eos1, scheme, w.ap, w.dg, w.nr, W1, 1, ug, pg, w.R1, w.scr, stream));
            LS_TRY(jxf_ls_cut_rhs(grid, eos2, scheme, w.ap, w.dg, w.nr, W2, 2, ug, pg, w.R2, w.scr, stream));
            advect_launch(g, phi, w.phin, ug, dt, stage == 0 ? 0 : 1, ca[stage], cb[stage], w.phit, s);
            k_ls_stage<<<ls_blocks_n((long long)nv * nc), kLsThreads, 0, s>>>(
                (long long)nv * nc, stage == 0, ca[stage], cb[stage], dt, w.U1n, w.R1, aU1, w.U2n, w.R2, aU2);
            LS_TRY(ls_launched());
            if (cudaMemcpyAsync(phi, w.phit, pbytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
                return JXF_ERR_CUDA;
            if (stage == 2) LS_TRY(jxf_ls_reinit(grid, phi, 10, 5e-2, w.scr, stream));
            // the new geometry, mixing against it, the phases' primitives and
            // ghost cells, the interface quantities
            LS_TRY(jxf_ls_geometry(grid, phi, w.ap, al1, w.dg, w.nr, stream));
            if (nd == 3) k_ls_phase2<3><<<ls_blocks(g), kLsThreads, 0, s>>>(nc, al0, al1, w.nr, w.b0, w.b1, w.n2);
            else k_ls_phase2<2><<<ls_blocks(g), kLsThreads, 0, s>>>(nc, al0, al1, w.nr, w.b0, w.b1, w.n2);
            LS_TRY(jxf_ls_mix(grid, nv, al0, al1, w.nr, amix, aU1, w.scr, stream));
            LS_TRY(jxf_ls_mix(grid, nv, w.b0, w.b1, w.n2, amix, aU2, w.scr, stream));
            if (nd == 3) {
                k_ls_prim<3><<<ls_blocks(g), kLsThreads, 0, s>>>(P1, nc, al1, aU1, W1);
                k_ls_prim<3><<<ls_blocks(g), kLsThreads, 0, s>>>(P2, nc, w.b1, aU2, W2);
            } else {
                k_ls_prim<2><<<ls_blocks(g), kLsThreads, 0, s>>>(P1, nc, al1, aU1, W1);
                k_ls_prim<2><<<ls_blocks(g), kLsThreads, 0, s>>>(P2, nc, w.b1, aU2, W2);
            }
            LS_TRY(ls_launched());
            LS_TRY(ls_extend_launch(g, phi, al1, w.dg, w.nr, 0, W1, 1, W2, nv, 10, w.scr, w.ext, s));
            LS_TRY(ls_interface_ext(grid, g, eos1, eos2, phi, W1, W2, al1, w.dg, w.nr, qg, w.scr, w.ext, s));
            std::swap(al0, al1);
        }
    }
#undef LS_TRY
    return JXF_OK;
}

jxf_status jxf_ls_reinit(const jxf_grid *grid, double *phi, int steps, double threshold, double *scratch,
                         jxf_stream stream) {
    JXF_RANGE("jxf_ls_reinit");
    LsGrid g;
    if (ls_grid(grid, g) != JXF_OK || !phi || !scratch || steps < 0 || !(threshold >= 0.0)) return JXF_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    double *p0 = scratch, *p1 = scratch + g.ncell;
    if (steps == 0) return JXF_OK;
    if (cudaMemcpyAsync(p0, phi, (size_t)g.ncell * sizeof(double), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return JXF_ERR_CUDA;
    const double dtau = 0.25 * g.h;
    for (int k = 0; k < steps; ++k) {
        // second-order TVD Runge-Kutta: p1 = p + dtau R(p); p <- 1/2 p + 1/2 (p1 + dtau R(p1))
        reinit_launch(g, phi, phi, p0, threshold, dtau, 0, p1, s);
        reinit_launch(g, p1, phi, p0, threshold, dtau, 1, phi, s);
    }
    return ls_launched();
}

}  // extern "C"
