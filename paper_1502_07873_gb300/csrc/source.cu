// Source discretisation and medium coefficients (device side).
//
//  - k_sources: for every solve, the perturbed parameter vector theta +/- d_j e_j
//    (central finite differences, 2*7 + 1 solves per node), the regularised
//    delta / delta' weights of Sec. 3.3.2 item 2 (six points k-2..k+3, fourth-order
//    moments, C^2 in x_s) combined into the force density f = M grad(delta)
//    (Eq. source), and the Gaussian source time function of Sec. 4.1
//    S(t) = w/sqrt(2 pi) exp(-w^2 (t - t_s)^2 / 2) sampled at every step.
//    All of it in FP64, stored in the stencil's precision.
//  - k_rows: per-row stencil coefficients of the leap-frog update for a medium
//    layered in depth (lambda = rho (vp^2 - 2 vs^2), mu = rho vs^2, Sec. 2.1).
#include <algorithm>

#include "oed_internal.cuh"

namespace oed {

// Regularised delta and delta' at nodes k-2..k+3 for offset a = (x_s - x_k)/h
// (Sec. 3.3.2 item 2).  Horner form of the printed polynomials.
__device__ void delta_weights(double a, double h, double *d, double *dp)
{
    const double P = a * a * a * a * a *
                     (5.0 / 3.0 + a * (-7.0 / 24.0 + a * (-17.0 / 12.0 + a * (9.0 / 8.0 - a / 4.0))));
    const double R = a * a * a * a * (-25.0 / 12.0 + a * (-3.0 / 4.0 + a * (59.0 / 12.0 + a * (-4.0 + a))));
    const double ih = 1.0 / h, ih2 = ih * ih;
    d[0] = (a * (1.0 / 12.0 + a * (-1.0 / 24.0 + a * (-1.0 / 12.0 - 19.0 / 24.0 * a))) + P) * ih;
    d[1] = (a * (-2.0 / 3.0 + a * (2.0 / 3.0 + a * (1.0 / 6.0 + 4.0 * a))) - 5.0 * P) * ih;
    d[2] = (1.0 + a * a * (-5.0 / 4.0 - 97.0 / 12.0 * a * a) + 10.0 * P) * ih;
    d[3] = (a * (2.0 / 3.0 + a * (2.0 / 3.0 + a * (-1.0 / 6.0 + 49.0 / 6.0 * a))) - 10.0 * P) * ih;
    d[4] = (a * (-1.0 / 12.0 + a * (-1.0 / 24.0 + a * (1.0 / 12.0 - 33.0 / 8.0 * a))) + 5.0 * P) * ih;
    d[5] = (5.0 / 6.0 * a * a * a * a - P) * ih;
    dp[0] = (-1.0 / 12.0 + a * (1.0 / 12.0 + a * (1.0 / 4.0 + 2.0 / 3.0 * a)) + R) * ih2;
    dp[1] = (2.0 / 3.0 + a * (-4.0 / 3.0 + a * (-1.0 / 2.0 - 7.0 / 2.0 * a)) - 5.0 * R) * ih2;
    dp[2] = (a * (5.0 / 2.0 + 22.0 / 3.0 * a * a) + 10.0 * R) * ih2;
    dp[3] = (-2.0 / 3.0 + a * (-4.0 / 3.0 + a * (1.0 / 2.0 - 23.0 / 3.0 * a)) - 10.0 * R) * ih2;
    dp[4] = (1.0 / 12.0 + a * (1.0 / 12.0 + a * (-1.0 / 4.0 + 4.0 * a)) + 5.0 * R) * ih2;
    dp[5] = (-5.0 / 6.0 * a * a * a - R) * ih2;
}

// d/dx_s of the six delta and delta' weights (the forcing derivative of a
// sensitivity solve, Alg. 1 step 2): (1/h) d/dalpha of the printed polynomials.
__device__ void delta_weights_dxs(double a, double h, double *d, double *dp)
{
    const double Pp = a * a * a * a * (25.0 / 3.0 + a * (-7.0 / 4.0 + a * (-119.0 / 12.0 + a * (9.0 - 9.0 / 4.0 * a))));
    const double Rp = a * a * a * (-25.0 / 3.0 + a * (-15.0 / 4.0 + a * (59.0 / 2.0 + a * (-28.0 + 8.0 * a))));
    const double ih2 = 1.0 / (h * h), ih3 = ih2 / h;
    d[0] = (1.0 / 12.0 + a * (-1.0 / 12.0 + a * (-1.0 / 4.0 - 19.0 / 6.0 * a)) + Pp) * ih2;
    d[1] = (-2.0 / 3.0 + a * (4.0 / 3.0 + a * (1.0 / 2.0 + 16.0 * a)) - 5.0 * Pp) * ih2;
    d[2] = (a * (-5.0 / 2.0 - 97.0 / 3.0 * a * a) + 10.0 * Pp) * ih2;
    d[3] = (2.0 / 3.0 + a * (4.0 / 3.0 + a * (-1.0 / 2.0 + 98.0 / 3.0 * a)) - 10.0 * Pp) * ih2;
    d[4] = (-1.0 / 12.0 + a * (-1.0 / 12.0 + a * (1.0 / 4.0 - 33.0 / 2.0 * a)) + 5.0 * Pp) * ih2;
    d[5] = (10.0 / 3.0 * a * a * a - Pp) * ih2;
    dp[0] = (1.0 / 12.0 + a * (1.0 / 2.0 + 2.0 * a) + Rp) * ih3;
    dp[1] = (-4.0 / 3.0 + a * (-1.0 - 21.0 / 2.0 * a) - 5.0 * Rp) * ih3;
    dp[2] = (5.0 / 2.0 + 22.0 * a * a + 10.0 * Rp) * ih3;
    dp[3] = (-4.0 / 3.0 + a * (1.0 - 23.0 * a) - 10.0 * Rp) * ih3;
    dp[4] = (1.0 / 12.0 + a * (-1.0 / 2.0 + 12.0 * a) + 5.0 * Rp) * ih3;
    dp[5] = (-5.0 / 2.0 * a * a - Rp) * ih3;
}

// d2/dx_s2 of the six delta and delta' weights (the forcing's second derivatives,
// Alg. 1 step 9; the regularised delta is C^2 in x_s): (1/h^2) d2/dalpha2 of the
// printed polynomials.
__device__ void delta_weights_dxs2(double a, double h, double *d, double *dp)
{
    const double Ppp = a * a * a * (100.0 / 3.0 + a * (-35.0 / 4.0 + a * (-119.0 / 2.0 + a * (63.0 - 18.0 * a))));
    const double Rpp = a * a * (-25.0 + a * (-15.0 + a * (295.0 / 2.0 + a * (-168.0 + 56.0 * a))));
    const double h3 = h * h * h, h4 = h3 * h;
    d[0] = (-1.0 / 12.0 + a * (-1.0 / 2.0 - 19.0 / 2.0 * a) + Ppp) / h3;
    d[1] = (4.0 / 3.0 + a * (1.0 + 48.0 * a) - 5.0 * Ppp) / h3;
    d[2] = (-5.0 / 2.0 - 97.0 * a * a + 10.0 * Ppp) / h3;
    d[3] = (4.0 / 3.0 + a * (-1.0 + 98.0 * a) - 10.0 * Ppp) / h3;
    d[4] = (-1.0 / 12.0 + a * (1.0 / 2.0 - 99.0 / 2.0 * a) + 5.0 * Ppp) / h3;
    d[5] = (10.0 * a * a - Ppp) / h3;
    dp[0] = (1.0 / 2.0 + 4.0 * a + Rpp) / h4;
    dp[1] = (-1.0 - 21.0 * a - 5.0 * Rpp) / h4;
    dp[2] = (44.0 * a + 10.0 * Rpp) / h4;
    dp[3] = (1.0 - 46.0 * a - 10.0 * Rpp) / h4;
    dp[4] = (-1.0 / 2.0 + 24.0 * a + 5.0 * Rpp) / h4;
    dp[5] = (-5.0 * a - Rpp) / h4;
}

struct FdStep {
    double d[kNT];
};

// S(t) of the given kind: OED_STF_GAUSS (Sec. 4.1, w = omega_s) or OED_STF_RICKER
// ((1 - 2a) e^{-a}, a = (pi w (t - ts))^2, w the peak frequency)
__device__ __forceinline__ double stf_value(int kind, double t, double ts, double ws)
{
    const double u = t - ts;
    if (kind == OED_STF_RICKER) {
        double a = 3.141592653589793 * ws * u;
        a = a * a;
        return (1.0 - 2.0 * a) * exp(-a);
    }
    return ws * 0.3989422804014327 * exp(-0.5 * ws * ws * u * u);   // w / sqrt(2 pi) e^{...}
}

// All solves of one node.  per_node = 1: the node itself (forward map);
// per_node = 15: centre and theta +/- d_j e_j (pairs Jacobian); per_node = 7:
// solve j carries the FP64 difference of the theta + d_j e_j and theta - d_j e_j
// forcings (difference Jacobian; by linearity of the scheme in the forcing its
// seismogram is exactly g(theta + d_j e_j) - g(theta - d_j e_j)), or with sens the analytic
// derivative of the forcing (Alg. 1 step 2).  Spatial part of a solve on its 6x6 support,
// corner (kx - 2, kz - 2), entry (b, a) at node (kx - 2 + a, kz - 2 + b):
//   f_x = m_xx delta'(x) delta(z) + m_xz delta(x) delta'(z)
//   f_z = m_xz delta'(x) delta(z) + m_zz delta(x) delta'(z)
// For j = x_s, z_s and the moments the two 6x6 patches of a difference solve are subtracted
// on their 7x7 union; for j = t_s, omega_s the time function differs.
//
// A node's solves share almost everything: at most three positions per axis (the node's and
// the two perturbed ones, a lane each for the weights) and five time functions.  One block
// per solve with one thread for its patch, and an exponential per solve and step, took
// 0.80 ms for 2048 nodes of 7 solves of 50 steps (the FP64 pipe, mostly one lane of it);
// this form 0.09 ms.  Block y of a node takes a part of its time steps, block 0 the patches too.
template <typename real>
__global__ void __launch_bounds__(128) k_sources(const double *__restrict__ theta_nodes, int per_node, int sens,
                                                 int stf_kind, FdStep step, Geometry g,
                                                 const RowCoef<real> *__restrict__ rows,
                                                 SourceDesc<real> *__restrict__ src, real *__restrict__ stf,
                                                 double *__restrict__ theta_out)
{
    const int node = blockIdx.x, tid = threadIdx.x;
    const bool diff = per_node == kND && !sens, pairs = per_node == kNP;
    __shared__ double th[kNT], thp[kNT], thm[kNT];   // the node, + d_j and - d_j in each entry
    __shared__ double W[2][3][4][6];                 // axis, position (node, +, -), delta, delta', and their d/dx_s
    __shared__ int cell[2][3], fin[2][3];            // first node of the weights + 2; usable position
    __shared__ int corner[kNP][3];                   // patch corner and whether it fits, per solve
    if (tid < kNT) {
        const double v = theta_nodes[(size_t)node * kNT + tid];
        th[tid] = v;
        thp[tid] = v + step.d[tid];
        thm[tid] = v - step.d[tid];
    }
    __syncthreads();
    // entry j of solve p's parameter vector
    auto param = [&](int p, int j) {
        return pairs && p > 0 && (p - 1) / 2 == j ? ((p - 1) & 1 ? thm[j] : thp[j]) : th[j];
    };
    // position (0 node, 1 +, 2 -) of solve p on an axis
    auto position = [&](int p, int axis) { return pairs && p > 0 && (p - 1) / 2 == axis ? 1 + ((p - 1) & 1) : 0; };
    if (blockIdx.y == 0) {
        if (tid < 6) {
            const int axis = tid / 3, v = tid % 3;
            if (v == 0 || diff || pairs) {
                const double q = (v == 0 ? th : v == 1 ? thp : thm)[axis] / g.h, fl = floor(q);
                const bool ok = isfinite(q) && fabs(fl) < 1e9;
                fin[axis][v] = ok;
                cell[axis][v] = ok ? (int)fl : 0;
                delta_weights(q - fl, g.h, W[axis][v][0], W[axis][v][1]);
                if (sens) delta_weights_dxs(q - fl, g.h, W[axis][v][2], W[axis][v][3]);
            }
        }
        __syncthreads();
        if (tid < per_node) {
            const int p = tid;
            int i0, j0, span = 6;   // span: 6 or 7 nodes of the patch actually used
            bool ok;
            if (diff && p != 2 && p != 3) {
                const int px = p == 0, pz = p == 1;   // the axis that is perturbed has positions 1 and 2
                const int xa = cell[0][px], xb = cell[0][2 * px], za = cell[1][pz], zb = cell[1][2 * pz];
                ok = fin[0][px] && fin[0][2 * px] && fin[1][pz] && fin[1][2 * pz];
                i0 = min(xa, xb) - 2;
                j0 = min(za, zb) - 2;
                ok = ok && max(xa, xb) - min(xa, xb) <= 1 && max(za, zb) - min(za, zb) <= 1;
                if (xa != xb || za != zb) span = 7;
            } else {
                const int vx = position(p, 0), vz = position(p, 1);
                ok = fin[0][vx] && fin[1][vz];
                i0 = cell[0][vx] - 2;
                j0 = cell[1][vz] - 2;
            }
            ok = ok && i0 >= 1 && i0 + span - 1 <= g.nx - 2 && j0 >= 0 && j0 + span - 1 <= g.nz - 2;
            corner[p][0] = ok ? i0 : -100;
            corner[p][1] = ok ? j0 : -100;
            corner[p][2] = ok;
            SourceDesc<real> &d = src[(size_t)node * per_node + p];
            d.i0 = corner[p][0];
            d.j0 = corner[p][1];
            d.ok = ok;
        }
        __syncthreads();
        for (int k = tid; k < per_node * kPatch * kPatch; k += blockDim.x) {
            const int p = k / (kPatch * kPatch), e = k % (kPatch * kPatch), b = e / kPatch, a = e % kPatch;
            double vx = 0.0, vz = 0.0;
            // M grad(delta) of positions (px, pz) with moments m at support entry (bb, aa)
            auto force = [&](int px, int pz, double mxx, double mxz, double mzz, int bb, int aa, double &fx, double &fz) {
                fx = fz = 0.0;
                if ((unsigned)aa >= 6u || (unsigned)bb >= 6u) return;
                const double dx = W[0][px][0][aa], dpx = W[0][px][1][aa], dz = W[1][pz][0][bb], dpz = W[1][pz][1][bb];
                fx = mxx * dpx * dz + mxz * dx * dpz;
                fz = mxz * dpx * dz + mzz * dx * dpz;
            };
            if (sens) {
                if (a < 6 && b < 6) {
                    const double dx = W[0][0][0][a], dpx = W[0][0][1][a], ex = W[0][0][2][a], epx = W[0][0][3][a];
                    const double dz = W[1][0][0][b], dpz = W[1][0][1][b], ez = W[1][0][2][b], epz = W[1][0][3][b];
                    const double mxx = th[4], mxz = th[5], mzz = th[6];
                    if (p == 0) {
                        vx = mxx * epx * dz + mxz * ex * dpz;
                        vz = mxz * epx * dz + mzz * ex * dpz;
                    } else if (p == 1) {
                        vx = mxx * dpx * ez + mxz * dx * epz;
                        vz = mxz * dpx * ez + mzz * dx * epz;
                    } else if (p == 2 || p == 3) {
                        vx = mxx * dpx * dz + mxz * dx * dpz;
                        vz = mxz * dpx * dz + mzz * dx * dpz;
                    } else if (p == 4) {
                        vx = dpx * dz;
                    } else if (p == 5) {
                        vx = dx * dpz;
                        vz = dpx * dz;
                    } else {
                        vz = dx * dpz;
                    }
                }
            } else if (diff && p != 2 && p != 3) {
                const int px = p == 0, pz = p == 1;
                const int xa = cell[0][px], xb = cell[0][2 * px], za = cell[1][pz], zb = cell[1][2 * pz];
                if (corner[p][2]) {
                    double gx, gz;
                    force(px, pz, p == 4 ? thp[4] : th[4], p == 5 ? thp[5] : th[5], p == 6 ? thp[6] : th[6],
                          b - (za - min(za, zb)), a - (xa - min(xa, xb)), vx, vz);
                    force(2 * px, 2 * pz, p == 4 ? thm[4] : th[4], p == 5 ? thm[5] : th[5], p == 6 ? thm[6] : th[6],
                          b - (zb - min(za, zb)), a - (xb - min(xa, xb)), gx, gz);
                    vx = vx - gx;
                    vz = vz - gz;
                }
            } else {
                force(position(p, 0), position(p, 1), param(p, 4), param(p, 5), param(p, 6), b, a, vx, vz);
            }
            const int j = corner[p][1] + b;
            const double rf = (corner[p][2] && j <= g.nz - 1) ? (double)rows[j].rf : 0.0;
            SourceDesc<real> &d = src[(size_t)node * per_node + p];
            d.wx[e] = (real)(vx * rf);
            d.wz[e] = (real)(vz * rf);
        }
        for (int k = tid; k < per_node * kNT; k += blockDim.x)
            theta_out[(size_t)node * per_node * kNT + k] = param(k / kNT, k % kNT);
    }
    const double ts = th[2], ws = th[3];
    real *out = stf + (size_t)node * per_node * g.nsteps;
    for (int m = blockIdx.y * blockDim.x + tid; m < g.nsteps; m += gridDim.y * blockDim.x) {
        const double t = m * g.dt;
        const double S = stf_value(stf_kind, t, ts, ws);
        double v2 = S, v3 = S;   // solves of t_s and omega_s: difference or derivative
        if (sens) {   // (Gaussian only, the host refuses sensitivity solves for any other kind)
            v2 *= ws * ws * (t - ts);                        // dS/dt_s
            v3 *= 1.0 / ws - ws * (t - ts) * (t - ts);       // dS/domega_s
        } else if (diff) {
            v2 = stf_value(stf_kind, t, thp[2], ws) - stf_value(stf_kind, t, thm[2], ws);
            v3 = stf_value(stf_kind, t, ts, thp[3]) - stf_value(stf_kind, t, ts, thm[3]);
        }
        for (int p = 0; p < per_node; p++) {
            double v = S;
            if (pairs) {
                if (p == 5) v = stf_value(stf_kind, t, thp[2], ws);
                if (p == 6) v = stf_value(stf_kind, t, thm[2], ws);
                if (p == 7) v = stf_value(stf_kind, t, ts, thp[3]);
                if (p == 8) v = stf_value(stf_kind, t, ts, thm[3]);
            } else if (per_node == kND) {
                if (p == 2) v = v2;
                if (p == 3) v = v3;
            }
            out[(size_t)p * g.nsteps + m] = (real)v;
        }
    }
}

// Per-row coefficients (one thread per row).
template <typename real>
__global__ void k_rows(Geometry g, int nlayers, const double *__restrict__ lay,
                       RowCoef<real> *__restrict__ rows, FacCoef<real> *__restrict__ fac)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= g.nz) return;
    auto layer_of = [&](int jj) {
        const double z = (jj < 0 ? 0 : (jj >= g.nz ? g.nz - 1 : jj)) * g.h;
        int l = 0;
        for (int q = 0; q < nlayers; q++)
            if (z >= lay[q]) l = q;
        return l;
    };
    auto lam = [&](int jj) {
        int l = layer_of(jj);
        double vp = lay[nlayers + l], vs = lay[2 * nlayers + l], rho = lay[3 * nlayers + l];
        return rho * (vp * vp - 2.0 * vs * vs);
    };
    auto mu = [&](int jj) {
        int l = layer_of(jj);
        double vs = lay[2 * nlayers + l], rho = lay[3 * nlayers + l];
        return rho * vs * vs;
    };
    const int l = layer_of(j);
    const double vp = lay[nlayers + l], vs = lay[2 * nlayers + l], rho = lay[3 * nlayers + l];
    const double h2 = g.h * g.h;
    const double r = g.dt * g.dt / rho;
    const double lc = lam(j), mc = mu(j), pc = lc + 2.0 * mc;
    RowCoef<double> c;
    c.axx = pc * r / h2;
    c.azx = mc * r / h2;
    c.rf = r;
    c.cp = vp * g.dt / g.h;
    c.cs = vs * g.dt / g.h;
    c.pad = 0.0;
    if (j == 0) {
        const double l1 = lam(1), m1 = mu(1), p1 = l1 + 2.0 * m1;
        c.axzp = 2.0 * 0.5 * (mc + m1) * r / h2;
        c.axzm = 0.0;
        c.azzp = 2.0 * 0.5 * (pc + p1) * r / h2;
        c.azzm = 0.0;
        c.lx = lc * r / (2.0 * h2);
        c.mxp = m1 * r / (2.0 * h2);
        c.mxm = mc * r / (2.0 * h2);
        c.mz = mc * r / (2.0 * h2);
        c.lzp = l1 * r / (2.0 * h2);
        c.lzm = lc * r / (2.0 * h2);
    } else {
        const double ls = lam(j + 1), ms = mu(j + 1), ps = ls + 2.0 * ms;
        const double ln = lam(j - 1), mn = mu(j - 1), pn = ln + 2.0 * mn;
        c.axzp = 0.5 * (mc + ms) * r / h2;
        c.axzm = 0.5 * (mn + mc) * r / h2;
        c.azzp = 0.5 * (pc + ps) * r / h2;
        c.azzm = 0.5 * (pn + pc) * r / h2;
        c.lx = lc * r / (4.0 * h2);
        c.mxp = ms * r / (4.0 * h2);
        c.mxm = mn * r / (4.0 * h2);
        c.mz = mc * r / (4.0 * h2);
        c.lzp = ls * r / (4.0 * h2);
        c.lzm = ln * r / (4.0 * h2);
    }
    RowCoef<real> o;
    o.axx = (real)c.axx; o.azx = (real)c.azx; o.axzp = (real)c.axzp; o.axzm = (real)c.axzm;
    o.azzp = (real)c.azzp; o.azzm = (real)c.azzm; o.lx = (real)c.lx; o.mxp = (real)c.mxp;
    o.mxm = (real)c.mxm; o.mz = (real)c.mz; o.lzp = (real)c.lzp; o.lzm = (real)c.lzm;
    o.rf = (real)c.rf; o.cp = (real)c.cp; o.cs = (real)c.cs; o.pad = (real)0;
    rows[j] = o;
    FacCoef<double> f;
    f.axx = c.axx; f.axzp = c.axzp; f.naxzm = -c.axzm;
    f.azx = c.azx; f.azzp = c.azzp; f.nazzm = -c.azzm;
    f.px = c.lx + c.mxp;
    f.pz = c.mz + c.lzp;
    f.nqx = j == 0 ? c.mxm - c.lx : -(c.lx + c.mxm);
    f.nqz = j == 0 ? c.lzm - c.mz : -(c.mz + c.lzm);
    FacCoef<real> q;
    q.axx = (real)f.axx; q.axzp = (real)f.axzp; q.naxzm = (real)f.naxzm; q.px = (real)f.px;
    q.nqx = (real)f.nqx; q.azx = (real)f.azx; q.azzp = (real)f.azzp; q.nazzm = (real)f.nazzm;
    q.pz = (real)f.pz; q.nqz = (real)f.nqz; q.cp = (real)c.cp; q.cs = (real)c.cs;
    // for the dual problem: the centre coefficients of B and those of the absorbing nodes
    q.pad0 = (real)2 - (real)2 * q.axx - q.axzp + q.naxzm;
    q.pad1 = (real)2 - (real)2 * q.azx - q.azzp + q.nazzm;
    q.pad2 = (real)1 - q.cp;
    q.pad3 = (real)1 - q.cs;
    fac[j] = q;
}

void launch_rows(oed_ctx *ctx, cudaStream_t s)
{
    const int nl = (int)ctx->z_top.size();
    std::vector<double> lay(4 * nl);
    for (int l = 0; l < nl; l++) {
        lay[l] = ctx->z_top[l];
        lay[nl + l] = ctx->vp[l];
        lay[2 * nl + l] = ctx->vs[l];
        lay[3 * nl + l] = ctx->rho[l];
    }
    double *d_lay = nullptr;
    cudaMallocAsync((void **)&d_lay, sizeof(double) * lay.size(), s);
    cudaMemcpyAsync(d_lay, lay.data(), sizeof(double) * lay.size(), cudaMemcpyHostToDevice, s);
    const int nb = (ctx->g.nz + 127) / 128;
    if (ctx->precision == OED_FP64)
        k_rows<double><<<nb, 128, 0, s>>>(ctx->g, nl, d_lay, (RowCoef<double> *)ctx->d_rows,
                                           (FacCoef<double> *)ctx->d_fac);
    else
        k_rows<float><<<nb, 128, 0, s>>>(ctx->g, nl, d_lay, (RowCoef<float> *)ctx->d_rows,
                                          (FacCoef<float> *)ctx->d_fac);
    cudaFreeAsync(d_lay, s);
    cudaStreamSynchronize(s);   // the host vector `lay` must outlive the copy
}

// Cost gradient and H_II from the dual solve (Alg. 1 steps 9-10, Eq. H2_numerics).
// The forcing of a solve is S(t) W on the 6x6 patch, W = dt^2/nu_row P(x_s, z_s, M),
//   P_x = m_xx d'(x) d(z) + m_xz d(x) d'(z),   P_z = m_xz d'(x) d(z) + m_zz d(x) d'(z),
// with d, d' the delta / delta' weights.  acc[t][c][node] = sum_m lambda^{m+1} S_t(t_m)
// (t = S, S_ts, S_w, S_tsts, S_tsw, S_ww), so with dJ/d(S W)^m = lambda^{m+1}
//   d2J/dth_p dth_q = sum_c sum_node acc[time part of (p,q)] * d^k W / (space part of (p,q))
// where t_s, omega_s differentiate S, x_s and z_s the weights of their axis, m_k
// select their moment term (d2/dm dm = 0).  H_II = -d2J (added to H), grad = -dJ.
// One block per solve; thread t < 28 takes the upper-triangle pair t, 28 <= t < 35
// the gradient entry t - 28.
template <typename real>
__global__ void __launch_bounds__(64) k_hii_combine(const double *__restrict__ theta, const double *__restrict__ acc,
                                                    const SourceDesc<real> *__restrict__ src,
                                                    const RowCoef<real> *__restrict__ rows, Geometry g,
                                                    double *__restrict__ H, double *__restrict__ grad,
                                                    int *__restrict__ status)
{
    const int s = blockIdx.x, t = threadIdx.x;
    const double *th = theta + (size_t)s * kNT;
    __shared__ double W[2][3][2][6];   // axis, derivative order, delta / delta', node
    __shared__ double rf[6];
    const bool ok = src[s].ok;
    if (t == 0 && ok) {
        for (int axis = 0; axis < 2; axis++) {
            const double q = th[axis] / g.h, al = q - floor(q);
            delta_weights(al, g.h, W[axis][0][0], W[axis][0][1]);
            delta_weights_dxs(al, g.h, W[axis][1][0], W[axis][1][1]);
            delta_weights_dxs2(al, g.h, W[axis][2][0], W[axis][2][1]);
        }
        for (int b = 0; b < 6; b++) rf[b] = (double)rows[src[s].j0 + b].rf;
    }
    __syncthreads();
    if (t >= 35) return;
    int p, q;
    if (t < 28) {   // upper-triangle pair number t
        p = 0;
        int r = t;
        while (r >= kNT - p) {
            r -= kNT - p;
            p++;
        }
        q = p + r;
    } else {
        p = t - 28;
        q = -1;
    }
    if (!ok) {
        if (t < 28) {
            H[(size_t)s * 49 + p * kNT + q] = NAN;
            H[(size_t)s * 49 + q * kNT + p] = NAN;
        } else if (grad) {
            grad[(size_t)s * kNT + p] = NAN;
        }
        if (t == 0 && status) status[s] = OED_EINVAL;
        return;
    }
    // derivative orders of the two axes, the time part and the moment selection
    const int ordx = (p == 0) + (q == 0), ordz = (p == 1) + (q == 1);
    const int nt = (p == 2 || p == 3) + (q == 2 || q == 3);
    const int nm = (p >= 4) + (q >= 4);
    double v = 0.0;
    if (nm < 2) {
        int tk;   // S-derivative index of acc
        if (nt == 0)
            tk = 0;
        else if (nt == 1)
            tk = (p == 2 || q == 2) ? 1 : 2;
        else
            tk = (p == 2 && q == 2) ? 3 : ((p == 3 && q == 3) ? 5 : 4);
        const double *ac = acc + (size_t)s * 6 * 2 * kPatch * kPatch + (size_t)tk * 2 * kPatch * kPatch;
        // moment terms of each component: (moment index, kind of the x factor; z factor the other)
        const int tm[2][2] = {{4, 5}, {5, 6}};
        const int xk[2][2] = {{1, 0}, {1, 0}};
        for (int c = 0; c < 2; c++)
            for (int b = 0; b < 6; b++)
                for (int a = 0; a < 6; a++) {
                    double P = 0.0;
                    for (int k = 0; k < 2; k++) {
                        const int mk = tm[c][k];
                        double coef = th[mk];
                        if (nm == 1) coef = (p == mk || q == mk) ? 1.0 : 0.0;
                        P += coef * W[0][ordx][xk[c][k]][a] * W[1][ordz][1 - xk[c][k]][b];
                    }
                    v += ac[c * kPatch * kPatch + b * kPatch + a] * rf[b] * P;
                }
    }
    if (t < 28) {
        H[(size_t)s * 49 + p * kNT + q] -= v;
        if (q != p) H[(size_t)s * 49 + q * kNT + p] -= v;
    } else if (grad) {
        grad[(size_t)s * kNT + p] = -v;
    }
    if (t == 0 && status) status[s] = 0;
}

void launch_hii_combine(const oed_ctx *ctx, int nsolve, const double *acc, double *H, double *grad, int *status,
                        cudaStream_t st)
{
    if (nsolve <= 0) return;
    if (ctx->precision == OED_FP64)
        k_hii_combine<double><<<nsolve, 64, 0, st>>>(ctx->d_theta, acc, (const SourceDesc<double> *)ctx->d_src,
                                                     (const RowCoef<double> *)ctx->d_rows, ctx->g, H, grad,
                                                     status);
    else
        k_hii_combine<float><<<nsolve, 64, 0, st>>>(ctx->d_theta, acc, (const SourceDesc<float> *)ctx->d_src,
                                                    (const RowCoef<float> *)ctx->d_rows, ctx->g, H, grad, status);
}

void launch_sources(const oed_ctx *ctx, const double *theta_nodes, int nnode, int per_node,
                    const double *step, cudaStream_t s)
{
    const int sens = (per_node == kND && ctx->jac_mode == OED_JAC_SENSITIVITY) ? 1 : 0;
    FdStep st;
    for (int j = 0; j < kNT; j++) st.d[j] = step ? step[j] : 0.0;
    if (nnode <= 0) return;
    // few nodes: their time steps are spread over several blocks
    const int parts = std::max(1, std::min((ctx->g.nsteps + 127) / 128, 2 * ctx->sms / nnode));
    const dim3 grid(nnode, parts);
    if (ctx->precision == OED_FP64)
        k_sources<double><<<grid, 128, 0, s>>>(theta_nodes, per_node, sens, ctx->stf, st, ctx->g,
                                               (const RowCoef<double> *)ctx->d_rows, (SourceDesc<double> *)ctx->d_src,
                                               (double *)ctx->d_stf, ctx->d_theta);
    else
        k_sources<float><<<grid, 128, 0, s>>>(theta_nodes, per_node, sens, ctx->stf, st, ctx->g,
                                              (const RowCoef<float> *)ctx->d_rows, (SourceDesc<float> *)ctx->d_src,
                                              (float *)ctx->d_stf, ctx->d_theta);
}

}  // namespace oed
