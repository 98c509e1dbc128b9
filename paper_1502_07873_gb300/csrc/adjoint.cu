// The dual (adjoint) problem of Eq. Dual_problems for Alg. 1 steps 6-10: the
// transpose of the discrete scheme, run backwards in time from receiver weights.
//
// For J = sum_m sum_{r,c} w^m_{r,c} g^m_{r,c} (w = C^-1 r, the data-side derivative
// of the cost) the derivative of J with respect to every value of the forcing is
// obtained from
//   lambda^m = R^T w^m + B^T lambda^{m+1} + E^T lambda^{m+2},   m = nsteps .. 1,
//   lambda^{nsteps+1} = lambda^{nsteps+2} = 0,   dJ/d(S W)^{m-1} = lambda^m,
// where u^{m+1} = B u^m + E u^{m-1} + (forcing) is the node update of
// stencil_cell.cuh (E = -I on interior and surface nodes, 0 on absorbing nodes) and
// R samples the receivers.  B^T is applied in gather form: node j collects, from
// every node i whose update reads u_j, the coefficient of u_j in that update times
// lambda_i, with the coefficients of node i's row (FacCoef).  Interior node i reads
// its 3x3 neighbourhood; the surface row reads its own row in place of the row
// above; an absorbing node reads itself and its inward neighbour.
//
// Like the forward kernels, lambda^m overwrites lambda^{m+2} in place (a node reads
// only its own lambda^{m+2}).  After each step a small kernel per solve adds the
// receiver weights and accumulates, for the source patch, the time sums
//   acc[s][c][node] += lambda^m(node, c) * S_s(t_{m-1}),   s = S, S_t, S_w, S_tt, S_tw, S_ww,
// from which the forcing's first and second parameter derivatives give the cost
// gradient and H_II (source.cu, k_hii_combine).
#include <algorithm>

#include "oed_internal.cuh"

namespace oed {

template <typename real>
struct AdjArgs {
    const real *cur;    // lambda^{m+1}
    real *nxt;          // lambda^{m+2} in, lambda^m out
    const FacCoef<real> *fac;
    Geometry g;
};

template <typename real>
__device__ __forceinline__ bool interior(const Geometry &g, int i, int j)
{
    return i >= 1 && i <= g.nx - 2 && j >= 0 && j <= g.nz - 2;
}

// (B^T lambda)(i, j) for both components plus E^T lambda^{m+2}.
template <typename real>
__global__ void __launch_bounds__(256) k_adjoint_step(AdjArgs<real> a)
{
    const Geometry &g = a.g;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int s = blockIdx.z;
    if (i >= g.nx || j >= g.nz) return;
    const real *lx = a.cur + (size_t)s * g.solve_stride;
    const real *lz = lx + g.comp_stride;
    real *ox = a.nxt + (size_t)s * g.solve_stride;
    real *oz = ox + g.comp_stride;
    auto LX = [&](int ii, int jj) { return lx[(size_t)jj * g.xp + ii]; };
    auto LZ = [&](int ii, int jj) { return lz[(size_t)jj * g.xp + ii]; };
    const FacCoef<real> *F = a.fac;
    const bool side = (i == 0 || i == g.nx - 1);
    const bool bottom = !side && j == g.nz - 1;
    const bool inner = !side && !bottom;
    real sx = 0, sz = 0;
    // the node's own update
    if (inner) {
        const FacCoef<real> &K = F[j];
        sx = ((real)2 - (real)2 * K.axx - K.axzp + K.naxzm) * LX(i, j);
        sz = ((real)2 - (real)2 * K.azx - K.azzp + K.nazzm) * LZ(i, j);
    } else if (side) {
        sx = ((real)1 - F[j].cp) * LX(i, j);
        sz = ((real)1 - F[j].cs) * LZ(i, j);
    } else {
        sx = ((real)1 - F[g.nz - 1].cs) * LX(i, j);
        sz = ((real)1 - F[g.nz - 1].cp) * LZ(i, j);
    }
    // west / east neighbours on the same row (this node is their east / west)
    if (interior<real>(g, i - 1, j)) {
        sx += F[j].axx * LX(i - 1, j);
        sz += F[j].azx * LZ(i - 1, j);
    }
    if (interior<real>(g, i + 1, j)) {
        sx += F[j].axx * LX(i + 1, j);
        sz += F[j].azx * LZ(i + 1, j);
    }
    // the row above (this node is its south) and the row below (this node is its north)
    if (j >= 1 && interior<real>(g, i, j - 1)) {
        sx += F[j - 1].axzp * LX(i, j - 1);
        sz += F[j - 1].azzp * LZ(i, j - 1);
    }
    if (interior<real>(g, i, j + 1)) {
        sx -= F[j + 1].naxzm * LX(i, j + 1);
        sz -= F[j + 1].nazzm * LZ(i, j + 1);
    }
    // cross terms: u_x(i,j) enters the u_z update of the diagonal neighbours and vice versa
    if (j >= 1) {
        if (interior<real>(g, i - 1, j - 1)) {   // this node is their south-east
            sx += F[j - 1].pz * LZ(i - 1, j - 1);
            sz += F[j - 1].px * LX(i - 1, j - 1);
        }
        if (interior<real>(g, i + 1, j - 1)) {   // south-west
            sx -= F[j - 1].pz * LZ(i + 1, j - 1);
            sz -= F[j - 1].px * LX(i + 1, j - 1);
        }
    }
    if (interior<real>(g, i - 1, j + 1)) {       // north-east of the row below
        sx += F[j + 1].nqz * LZ(i - 1, j + 1);
        sz += F[j + 1].nqx * LX(i - 1, j + 1);
    }
    if (interior<real>(g, i + 1, j + 1)) {       // north-west
        sx -= F[j + 1].nqz * LZ(i + 1, j + 1);
        sz -= F[j + 1].nqx * LX(i + 1, j + 1);
    }
    if (j == 0) {   // the surface row's cross terms read its own row: east / west of row 0
        if (interior<real>(g, i - 1, 0)) {
            sx += F[0].nqz * LZ(i - 1, 0);
            sz += F[0].nqx * LX(i - 1, 0);
        }
        if (interior<real>(g, i + 1, 0)) {
            sx -= F[0].nqz * LZ(i + 1, 0);
            sz -= F[0].nqx * LX(i + 1, 0);
        }
    }
    // absorbing nodes whose inward neighbour is this node
    if (i == 1) {
        sx += F[j].cp * LX(0, j);
        sz += F[j].cs * LZ(0, j);
    }
    if (i == g.nx - 2) {
        sx += F[j].cp * LX(g.nx - 1, j);
        sz += F[j].cs * LZ(g.nx - 1, j);
    }
    if (j == g.nz - 2 && i >= 1 && i <= g.nx - 2) {
        sx += F[g.nz - 1].cs * LX(i, g.nz - 1);
        sz += F[g.nz - 1].cp * LZ(i, g.nz - 1);
    }
    const size_t o = (size_t)j * g.xp + i;
    if (inner) {   // E^T lambda^{m+2}
        sx -= ox[o];
        sz -= oz[o];
    }
    ox[o] = sx;
    oz[o] = sz;
}

// The same in FP64, where the pipe (two lanes per clock and SM) is the bound and only its
// issue slots count: 16 per node and a little per row segment, against 37 with a branch per
// neighbour and the centre coefficients formed anew at every node.  A thread takes a column's
// segment of up to ZS rows, threads are packed densely over solves, segments and columns, the
// east - west differences of a row serve the rows above and below it, and the boundary nodes
// take the slots of the interior with selected operands: a neighbour that is no interior node
// enters as zero, the absorbing nodes' terms in the place of the missing neighbour's.
struct AdjRow {
    double w[2], c[2], e[2];   // lambda at i-1, i, i+1 (u_x, then u_z)
    double d[2];               // west - east, interior nodes only
};

template <int ZS>
__global__ void __launch_bounds__(128) k_adjoint64(AdjArgs<double> a, int nseg, unsigned nthr)
{
    const Geometry &g = a.g;
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nthr) return;
    const unsigned per = (unsigned)g.nx * (unsigned)nseg;
    const int s = (int)(t / per);
    const unsigned q = t - (unsigned)s * per;
    const int seg = (int)(q / (unsigned)g.nx), i = (int)(q - (unsigned)seg * (unsigned)g.nx);
    const int j0 = (int)((long long)g.nz * seg / nseg), j1 = (int)((long long)g.nz * (seg + 1) / nseg);
    const double *__restrict__ cur = a.cur + (size_t)s * g.solve_stride + i;
    double *__restrict__ nxt = a.nxt + (size_t)s * g.solve_stride + i;
    const bool side = i == 0 || i == g.nx - 1, hasw = i > 0, hase = i < g.nx - 1;
    const bool inw = i - 1 >= 1, ine = i + 1 <= g.nx - 2;   // the west / east column holds interior nodes
    auto load = [&](int j, AdjRow &r) {
        const bool in = j >= 0 && j < g.nz, rowin = in && j <= g.nz - 2;
        const size_t o = (size_t)(in ? j : 0) * g.xp;
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const double *u = cur + k * g.comp_stride + o;
            r.c[k] = in ? __ldg(u) : 0.0;
            r.w[k] = in && hasw ? __ldg(u - 1) : 0.0;
            r.e[k] = in && hase ? __ldg(u + 1) : 0.0;
            r.d[k] = (rowin && inw ? r.w[k] : 0.0) - (rowin && ine ? r.e[k] : 0.0);
        }
    };
    AdjRow n, c, so;
    load(j0 - 1, n);
    load(j0, c);
#pragma unroll
    for (int k0 = 0; k0 < ZS; k0++) {
        const int j = j0 + k0;
        if (j >= j1) break;
        const bool bottom = j == g.nz - 1, inner = !side && !bottom;
        const size_t o = (size_t)j * g.xp;
        const FacCoef<double> K = a.fac[j], Kn = a.fac[j > 0 ? j - 1 : 0], Ks = a.fac[bottom ? j : j + 1];
        const double ox = __ldcs(nxt + o), oz = __ldcs(nxt + g.comp_stride + o);
        load(j + 1, so);
        // the node's own update and E^T lambda^{m+2}; pad0 .. pad3: centre coefficients of u_x, u_z
        // and 1 - c_p, 1 - c_s
        double sx = fma(side ? K.pad2 : (bottom ? K.pad3 : K.pad0), c.c[0], inner ? -ox : 0.0);
        double sz = fma(side ? K.pad3 : (bottom ? K.pad2 : K.pad1), c.c[1], inner ? -oz : 0.0);
        // west and east neighbours on the row, or the absorbing side node whose inward neighbour this is
        const double axx = bottom ? 0.0 : K.axx, azx = bottom ? 0.0 : K.azx;
        sx = fma(i == 1 ? K.cp : (inw ? axx : 0.0), c.w[0], sx);
        sz = fma(i == 1 ? K.cs : (inw ? azx : 0.0), c.w[1], sz);
        sx = fma(i == g.nx - 2 ? K.cp : (ine ? axx : 0.0), c.e[0], sx);
        sz = fma(i == g.nx - 2 ? K.cs : (ine ? azx : 0.0), c.e[1], sz);
        // the row above (this node is its south) and the row below (its north, or the absorbing bottom)
        const bool last = j == g.nz - 2;
        sx = fma(side ? 0.0 : Kn.axzp, n.c[0], sx);
        sz = fma(side ? 0.0 : Kn.azzp, n.c[1], sz);
        sx = fma(side ? 0.0 : (last ? Ks.cs : -Ks.naxzm), so.c[0], sx);
        sz = fma(side ? 0.0 : (last ? Ks.cp : -Ks.nazzm), so.c[1], sz);
        // cross terms: u_x(i,j) enters the u_z update of the diagonal neighbours and vice versa
        sx = fma(Kn.pz, n.d[1], sx);
        sz = fma(Kn.px, n.d[0], sz);
        sx = fma(Ks.nqz, so.d[1], sx);
        sz = fma(Ks.nqx, so.d[0], sz);
        if (j == 0) {   // the surface row's cross terms read its own row
            sx = fma(K.nqz, c.d[1], sx);
            sz = fma(K.nqx, c.d[0], sz);
        }
        nxt[o] = sx;
        nxt[g.comp_stride + o] = sz;
        n = c;
        c = so;
    }
}

static void adjoint_step(const AdjArgs<float> &a, int nsolve, int, cudaStream_t st)
{
    const dim3 blk(32, 8, 1), grd((a.g.nx + 31) / 32, (a.g.nz + 7) / 8, nsolve);
    k_adjoint_step<float><<<grd, blk, 0, st>>>(a);
}

static void adjoint_step(const AdjArgs<double> &a, int nsolve, int sms, cudaStream_t st)
{
    constexpr int ZS = 4;   // 8 and 12 measured equal on 256 and 1000 solves of 101x76
    const int nseg = segments64((long long)a.g.nx * nsolve, a.g.nz, ZS, 16.0, 8.0, sms);
    const long long per = (long long)a.g.nx * nseg;
    const int most = (int)std::max(1LL, std::min((long long)nsolve, (1LL << 31) / per));   // 32-bit thread numbers
    for (int s0 = 0; s0 < nsolve; s0 += most) {
        const int ns = std::min(most, nsolve - s0);
        AdjArgs<double> b = a;
        b.cur += (size_t)s0 * a.g.solve_stride;
        b.nxt += (size_t)s0 * a.g.solve_stride;
        const unsigned nthr = (unsigned)(per * ns);
        k_adjoint64<ZS><<<(nthr + 63) / 64, 64, 0, st>>>(b, nseg, nthr);
    }
}

// S and its first and second derivatives in (t_s, omega_s): tau = t - t_s,
// L = log S, dL/dt_s = w^2 tau, dL/dw = 1/w - w tau^2, d2L/dt_s2 = -w^2,
// d2L/dt_s dw = 2 w tau, d2L/dw2 = -1/w^2 - tau^2, d2S = S (dL dL + d2L).
__device__ void stf_derivs(double t, double ts, double w, double *out)
{
    const double tau = t - ts;
    const double S = w * 0.3989422804014327 * exp(-0.5 * w * w * tau * tau);   // w / sqrt(2 pi)
    const double Lt = w * w * tau, Lw = 1.0 / w - w * tau * tau;
    out[0] = S;
    out[1] = S * Lt;
    out[2] = S * Lw;
    out[3] = S * (Lt * Lt - w * w);
    out[4] = S * (Lt * Lw + 2.0 * w * tau);
    out[5] = S * (Lw * Lw - 1.0 / (w * w) - tau * tau);
}

// One block per solve: add R^T w^m (duplicate receivers summed by the first of them,
// in receiver order), then accumulate the patch's time sums.
template <typename real>
__global__ void __launch_bounds__(128) k_adjoint_post(real *lam, const double *__restrict__ w,
                                                      const int *__restrict__ rec,
                                                      const SourceDesc<real> *__restrict__ src,
                                                      const double *__restrict__ theta, double *acc,
                                                      Geometry g, int m)
{
    const int s = blockIdx.x;
    real *lx = lam + (size_t)s * g.solve_stride;
    real *lz = lx + g.comp_stride;
    const double *wm = w + ((size_t)s * g.nlev + m) * g.nrec * 2;
    for (int q = threadIdx.x; q < 2 * g.nrec; q += blockDim.x) {
        const int r = q >> 1, c = q & 1, node = rec[r];
        bool first = true;
        for (int k = 0; k < r; k++) first = first && rec[k] != node;
        if (!first) continue;
        double v = 0.0;
        for (int k = r; k < g.nrec; k++)
            if (rec[k] == node) v += wm[k * 2 + c];
        real *p = (c ? lz : lx) + node;
        *p = (real)((double)*p + v);
    }
    __syncthreads();
    __shared__ double sd[6];
    const SourceDesc<real> *sdesc = src + s;
    if (!sdesc->ok) return;
    if (threadIdx.x == 0) stf_derivs((m - 1) * g.dt, theta[(size_t)s * kNT + 2], theta[(size_t)s * kNT + 3], sd);
    __syncthreads();
    const int k = threadIdx.x;
    if (k < 2 * kPatch * kPatch) {
        const int c = k / (kPatch * kPatch), ab = k % (kPatch * kPatch);
        const int b = ab / kPatch, a2 = ab % kPatch;
        const int ii = sdesc->i0 + a2, jj = sdesc->j0 + b;
        if (ii >= 0 && ii < g.nx && jj >= 0 && jj < g.nz) {
            const double v = (double)(c ? lz : lx)[(size_t)jj * g.xp + ii];
            double *ac = acc + (size_t)s * 6 * 2 * kPatch * kPatch;
#pragma unroll
            for (int t = 0; t < 6; t++) ac[(t * 2 + c) * kPatch * kPatch + ab] += v * sd[t];
        }
    }
}

// w = (y - g) / sigma^2 in FP64 from the traces of the primal solves
template <typename real>
__global__ void k_residual(const real *__restrict__ trace, const double *__restrict__ y, double inv_s2,
                           size_t count, double *__restrict__ w)
{
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < count;
         k += (size_t)gridDim.x * blockDim.x)
        w[k] = (y[k] - (double)trace[k]) * inv_s2;
}

template <typename real>
static void adjoint_impl(const oed_ctx *ctx, int nsolve, const double *y, double sigma, double *w,
                         double *acc, cudaStream_t st)
{
    const Geometry &g = ctx->g;
    const size_t cnt = (size_t)nsolve * g.nlev * g.nrec * 2;
    k_residual<real><<<(int)std::min<size_t>((cnt + 255) / 256, 4096), 256, 0, st>>>(
        (const real *)ctx->d_trace, y, 1.0 / (sigma * sigma), cnt, w);
    const size_t bytes = (size_t)nsolve * g.solve_stride * sizeof(real);
    cudaMemsetAsync(ctx->d_u0, 0, bytes, st);
    cudaMemsetAsync(ctx->d_u1, 0, bytes, st);
    cudaMemsetAsync(acc, 0, sizeof(double) * (size_t)nsolve * 6 * 2 * kPatch * kPatch, st);
    AdjArgs<real> a;
    a.fac = (const FacCoef<real> *)ctx->d_fac;
    a.g = g;
    real *A = (real *)ctx->d_u0, *B = (real *)ctx->d_u1;
    for (int m = g.nsteps; m >= 1; m--) {
        const int k = g.nsteps - m;
        a.cur = (k & 1) ? B : A;   // lambda^{m+1}
        a.nxt = (k & 1) ? A : B;   // lambda^{m+2} -> lambda^m
        adjoint_step(a, nsolve, ctx->sms, st);
        k_adjoint_post<real><<<nsolve, 128, 0, st>>>(a.nxt, w, ctx->d_rec, (const SourceDesc<real> *)ctx->d_src,
                                                     ctx->d_theta, acc, g, m);
    }
}

void launch_adjoint(const oed_ctx *ctx, int nsolve, const double *y, double sigma, double *w, double *acc,
                    cudaStream_t st)
{
    if (ctx->precision == OED_FP64)
        adjoint_impl<double>(ctx, nsolve, y, sigma, w, acc, st);
    else
        adjoint_impl<float>(ctx, nsolve, y, sigma, w, acc, st);
}

}  // namespace oed
