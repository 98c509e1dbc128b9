// Batched leap-frog time stepping of the 2-D elastic wave equation
// (Sec. 3.3.1: Eqs. interior_disc, absorbing_disc, full_discrete, Full_Disc).
//
// One launch advances every solve of the batch by one step:
//   interior and surface nodes:  u^{m+1} = 2u^m - u^{m-1} + dt^2/nu (A_h u^m + f^m)
//   absorbing nodes (sides, bottom; first-order Clayton-Engquist, forward in time,
//   upwind in space):            u^{m+1} = u^m + c dt/h (u_inward^m - u^m)
// with A_h the second-order operator built from D+, D-, D0 and a summation-by-parts
// closure on the free surface, and f^m = S(t_m) M grad(delta) on the 7x7 source patch.
//
// Memory layout: u[solve][component][z][xp] with xp a multiple of 32, so every warp
// reads and writes whole 128-byte lines.  u^{m+1} overwrites u^{m-1} in place (each
// node reads only its own u^{m-1}), so a solve needs two level buffers.
// Each thread owns one column i and ZS consecutive rows.  It issues all of its
// loads first (rows j-1 .. j+ZS of u^m at columns i-1, i, i+1, both components,
// and its ZS values of u^{m-1}), so each thread keeps ~8 ZS independent loads in
// flight, then computes and stores its ZS nodes.  Horizontal neighbours are L1
// hits and the two halo rows of a segment are L2 hits, so HBM traffic is the
// algorithmic minimum: read u^m and u^{m-1}, write u^{m+1}, two components each
// (24 B per cell-update in FP32).
//
// The same launch gathers the receiver samples of level m from its input u^m
// (Eq. forward_model), so the seismograms need no extra pass over the field.
#include <algorithm>
#include <cmath>

#include "stencil_cell.cuh"

namespace oed {

template <typename real>
struct StepArgs {
    const real *cur;               // u^m
    real *nxt;                     // u^{m-1} in, u^{m+1} out
    const FacCoef<real> *fac;      // [nz]
    const SourceDesc<real> *src;   // [nsolve]
    const real *stf;               // [nsolve][nsteps]
    real *trace;                   // [nsolve][nlev][nrec][2]
    const int *rec;                // [nrec]
    Geometry g;
    int m;
};

template <typename real>
__device__ __forceinline__ void load3(const real *__restrict__ p, int im, int i, int ip, real *v)
{
    v[0] = __ldg(p + im);
    v[1] = __ldg(p + i);
    v[2] = __ldg(p + ip);
}

template <typename real, int ZS>
__global__ void __launch_bounds__(256) k_step(StepArgs<real> a)
{
    const Geometry &g = a.g;
    const int s = blockIdx.z;
    const size_t base = (size_t)s * g.solve_stride;
    const real *__restrict__ cx = a.cur + base;
    const real *__restrict__ cz = cx + g.comp_stride;

    if (blockIdx.x == 0 && blockIdx.y == 0) {
        // receiver samples of level m (the input field)
        const int t = threadIdx.y * blockDim.x + threadIdx.x;
        real *tr = a.trace + ((size_t)s * g.nlev + a.m) * g.nrec * 2;
        for (int q = t; q < 2 * g.nrec; q += blockDim.x * blockDim.y)
            tr[q] = (q & 1 ? cz : cx)[a.rec[q >> 1]];
    }

    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int jb = (blockIdx.y * blockDim.y + threadIdx.y) * ZS;
    if (i >= g.nx || jb >= g.nz) return;

    real *__restrict__ px = a.nxt + base;
    real *__restrict__ pz = px + g.comp_stride;
    const int im = i > 0 ? i - 1 : 0;
    const int ip = i < g.nx - 1 ? i + 1 : g.nx - 1;
    const int side = (i == 0) ? 1 : ((i == g.nx - 1) ? 2 : 0);
    const int jlast = g.nz - 1;

    // Issue every load of this thread before any arithmetic: rows jb-1 .. jb+ZS of
    // u^m (three columns, two components) and rows jb .. jb+ZS-1 of u^{m-1}.  Rows
    // outside the grid are clamped (their values are never used).
    real X[ZS + 2][3], Z[ZS + 2][3], XM[ZS], ZM[ZS];
#pragma unroll
    for (int k = 0; k < ZS + 2; k++) {
        int j = jb - 1 + k;
        j = j < 0 ? 0 : (j > jlast ? jlast : j);
        const size_t o = (size_t)j * g.xp;
        load3(cx + o, im, i, ip, X[k]);
        load3(cz + o, im, i, ip, Z[k]);
    }
#pragma unroll
    for (int k = 0; k < ZS; k++) {
        const int j = jb + k < jlast ? jb + k : jlast;
        const size_t o = (size_t)j * g.xp + i;
        XM[k] = __ldcs(px + o);   // read once, never reused: streaming
        ZM[k] = __ldcs(pz + o);
    }
    const int si = i - a.src[s].i0;
    const int sj = a.src[s].j0;
    const bool scol = (unsigned)si < (unsigned)kPatch;
    const real S = scol ? a.stf[(size_t)s * g.nsteps + a.m] : (real)0;

#pragma unroll
    for (int k = 0; k < ZS; k++) {
        const int j = jb + k;
        if (j > jlast) break;
        const FacCoef<real> K = a.fac[j];
        real ux, uz;
        node_update(K, X[k], X[k + 1], X[k + 2], Z[k], Z[k + 1], Z[k + 2], XM[k], ZM[k], side,
                    j == jlast, j == 0, ux, uz);
        const int b = j - sj;
        if (scol && (unsigned)b < (unsigned)kPatch && !side && j != jlast) {
            ux = add_force(ux, S, a.src[s].wx[b * kPatch + si]);
            uz = add_force(uz, S, a.src[s].wz[b * kPatch + si]);
        }
        const size_t o = (size_t)j * g.xp + i;
        __stcs(px + o, ux);   // u^{m+1} is next read one full step later: streaming
        __stcs(pz + o, uz);
    }
}

// The FP64 step.  FP64 runs at two lanes per clock and SM here, 64 times below FP32, so a
// warp's FP64 instruction holds its scheduler's pipe for 64 clocks: the pipe bounds the
// kernel and everything else (loads, selects, index arithmetic) is free beside it.  The
// split therefore saves FP64 issue slots only:
//  - a thread owns a column pair (the first difference between its columns serves both) and
//    up to ZS rows, each row's differences formed once as it enters as the south row;
//  - threads are packed densely over (solve, row segment, pair), so no lanes idle at the right
//    edge of a grid, and the segments of a grid are equally long to one row;
//  - the surface row, the bottom row and the side columns take the slots of the interior
//    update with selected operands instead of branches of their own (the rounding is that of
//    node_update in each case).
// 81x41, 240 solves: 25 slots per cell-update against 38 for the kernel of one column and
// four rows per thread that it replaces.
struct Row64 {
    double ca[2], cb[2];   // centre values, u_x then u_z
    double da[2], db[2];   // east - west differences
    double va[2], vb[2];   // south row minus this row
};

template <int ZS>
__global__ void __launch_bounds__(256) k_step64(StepArgs<double> a, int npair, int nseg, unsigned nthr)
{
    const Geometry &g = a.g;
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    const int nq = 2 * g.nrec;
    const unsigned per = (unsigned)npair * (unsigned)nseg;
    if (t >= nthr) return;
    const int s = (int)(t / per);
    const unsigned w = t - (unsigned)s * per;
    const int seg = (int)(w / (unsigned)npair), p = (int)(w - (unsigned)seg * (unsigned)npair);
    const size_t base = (size_t)s * g.solve_stride;
    const double *__restrict__ cur = a.cur + base;
    double *__restrict__ nxt = a.nxt + base;
    if (seg == 0)   // receiver samples of level m (the input field)
        for (int q = p; q < nq; q += npair)
            a.trace[((size_t)s * g.nlev + a.m) * nq + q] = cur[(q & 1) * g.comp_stride + a.rec[q >> 1]];

    const int c = 2 * p, last = g.nx - 1;
    // (ZS = 1: one row each, without the divisions)
    const int j0 = ZS == 1 ? seg : (int)((long long)g.nz * seg / nseg);
    const int j1 = ZS == 1 ? seg + 1 : (int)((long long)g.nz * (seg + 1) / nseg);
    const bool sideA = c == 0 || c == last, sideB = c + 1 == last, hasB = c + 1 <= last;
    const int iw = c > 0 ? c - 1 : 0, ie = c + 2 <= last ? c + 2 : last;
    // row j of u^m as seen by the pair; outside the grid the neighbour is the node itself
    auto load = [&](int j, Row64 &r, double (&la)[2], double (&lb)[2]) {
        const size_t o = (size_t)(j < g.nz - 1 ? j : g.nz - 1) * g.xp;
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const double *u = cur + k * g.comp_stride + o;
            const double2 v = __ldg(reinterpret_cast<const double2 *>(u + c));
            const double xw = __ldg(u + iw), xe = __ldg(u + ie);
            const double xb = hasB ? v.y : v.x;
            r.ca[k] = v.x;
            r.cb[k] = xb;
            const double f = xb - v.x;
            la[k] = f - (v.x - xw);
            lb[k] = (xe - xb) - f;
            r.da[k] = xb - xw;
            r.db[k] = xe - v.x;
        }
    };
    auto south = [](Row64 &n, const Row64 &s_) {
#pragma unroll
        for (int k = 0; k < 2; k++) {
            n.va[k] = s_.ca[k] - n.ca[k];
            n.vb[k] = s_.cb[k] - n.cb[k];
        }
    };
    // u^{m+1} of one component at one node: K1 .. K5 the operator's coefficients in op_x's order
    auto node = [](double K1, double K2, double K3, double K4, double K5, double cside, double cbot, double uc, double um,
                   double lap, double vs, double vn, double ds, double dn, bool side, bool bottom) {
        const double a1 = fma(side ? cside : K1, lap, side ? uc : uc - um);
        const double a2 = fma(K2, vs, a1);
        const double a3 = fma(bottom ? -cbot : K3, vn, bottom ? uc : a2);
        const double a5 = fma(K5, dn, fma(K4, ds, a3));
        const double u = uc + a5;
        return side ? a1 : (bottom ? a3 : u);
    };
    const int sj = a.src[s].j0, si = c - a.src[s].i0;
    const bool scolA = (unsigned)si < (unsigned)kPatch, scolB = hasB && (unsigned)(si + 1) < (unsigned)kPatch;
    const double S = scolA || scolB ? a.stf[(size_t)s * g.nsteps + a.m] : 0.0;

    Row64 n, ce, so;
    double la[2], lb[2], sa[2], sb[2];
    load(j0, ce, la, lb);
    if (j0 == 0) {   // no north differences, cross terms on the row itself
        n = ce;
#pragma unroll
        for (int k = 0; k < 2; k++) n.va[k] = n.vb[k] = 0.0;
    } else {
        load(j0 - 1, n, sa, sb);
        south(n, ce);
    }
#pragma unroll
    for (int i = 0; i < ZS; i++) {
        const int j = j0 + i;
        if (j >= j1) break;
        const bool bottom = j == g.nz - 1;
        const FacCoef<double> K = a.fac[j];
        const size_t o = (size_t)j * g.xp + c;
        const double2 mx = __ldcs(reinterpret_cast<const double2 *>(nxt + o));
        const double2 mz = __ldcs(reinterpret_cast<const double2 *>(nxt + g.comp_stride + o));
        load(j + 1, so, sa, sb);
        south(ce, so);
        double xa = node(K.axx, K.axzp, K.naxzm, K.px, K.nqx, K.cp, K.cs, ce.ca[0], mx.x, la[0], ce.va[0], n.va[0],
                         so.da[1], n.da[1], sideA, bottom);
        double za = node(K.azx, K.azzp, K.nazzm, K.pz, K.nqz, K.cs, K.cp, ce.ca[1], mz.x, la[1], ce.va[1], n.va[1],
                         so.da[0], n.da[0], sideA, bottom);
        double xb = node(K.axx, K.axzp, K.naxzm, K.px, K.nqx, K.cp, K.cs, ce.cb[0], mx.y, lb[0], ce.vb[0], n.vb[0],
                         so.db[1], n.db[1], sideB, bottom);
        double zb = node(K.azx, K.azzp, K.nazzm, K.pz, K.nqz, K.cs, K.cp, ce.cb[1], mz.y, lb[1], ce.vb[1], n.vb[1],
                         so.db[0], n.db[0], sideB, bottom);
        const int b = j - sj;
        if ((unsigned)b < (unsigned)kPatch && (scolA || scolB)) {
            const SourceDesc<double> &d = a.src[s];
            if (scolA) {
                xa = add_force(xa, S, d.wx[b * kPatch + si]);
                za = add_force(za, S, d.wz[b * kPatch + si]);
            }
            if (scolB) {
                xb = add_force(xb, S, d.wx[b * kPatch + si + 1]);
                zb = add_force(zb, S, d.wz[b * kPatch + si + 1]);
            }
        }
        if (!hasB) xb = zb = 0.0;   // the padding column stays zero
        __stcs(reinterpret_cast<double2 *>(nxt + o), make_double2(xa, xb));
        __stcs(reinterpret_cast<double2 *>(nxt + g.comp_stride + o), make_double2(za, zb));
        n = ce;
        ce = so;
#pragma unroll
        for (int k = 0; k < 2; k++) {
            la[k] = sa[k];
            lb[k] = sb[k];
        }
    }
}

// Receiver samples of one level (used for the last level after the final step).
template <typename real>
__global__ void k_gather(const real *__restrict__ cur, real *__restrict__ trace,
                         const int *__restrict__ rec, Geometry g, int m, int nsolve)
{
    const int s = blockIdx.x;
    if (s >= nsolve) return;
    const real *cx = cur + (size_t)s * g.solve_stride;
    const real *cz = cx + g.comp_stride;
    real *tr = trace + ((size_t)s * g.nlev + m) * g.nrec * 2;
    for (int q = threadIdx.x; q < 2 * g.nrec; q += blockDim.x)
        tr[q] = (q & 1 ? cz : cx)[rec[q >> 1]];
}

// Row segments for the FP64 kernels, columns of which (over all solves) take a thread each: up to zs
// rows a segment, shorter where that spreads the columns over more of the schedulers (four per SM,
// each with its own FP64 pipe).  A segment of r rows takes per r + once issue slots of its pipe; the
// warps go round the pipes, half of a partly filled last round overlaps the others, and a thread's
// rows follow one another, which a pipe with one or two warps does not hide (latency per row).  A
// fit to 47 batches of six grids (9x9 to 401x201, 1 to 3000 solves): 1 to 1.5% slower than the best
// segment length on average.  Counted in whole rounds and without the latency it was 8% and up to
// 39%: 15 solves of 81x41 482 us for 60 steps against 370 in one-row segments.  These have a kernel
// without the divisions of the general one (ZS = 1; one solve of 201x101 318 -> 298 us).
int segments64(long long columns, int nz, int zs, double per, double once, int sms)
{
    constexpr double kLatency = 8.0;
    const double pipes = 4.0 * sms;
    int best = (nz + zs - 1) / zs;
    double least = 0.0;
    for (int r = zs; r >= 1; r--) {
        const int nseg = (nz + r - 1) / r, rows = (nz + nseg - 1) / nseg;
        const double warps = (double)columns * nseg / 32.0 / pipes;
        const double cost = std::max(1.0, 0.5 * (warps + std::ceil(warps))) * (per * rows + once) + kLatency * rows;
        if (r == zs || cost < least) {
            least = cost;
            best = nseg;
        }
    }
    return best;
}

// One step of nsolve solves with the context's launch shape.
template <typename real, int ZS>
static void launch_one(const oed_ctx *ctx, int nsolve, const StepArgs<real> &a, cudaStream_t st)
{
    const Geometry &g = ctx->g;
    const int wz = ctx->tune.wz;
    if constexpr (sizeof(real) == 8) {
        const int npair = (g.nx + 1) / 2, nseg = segments64((long long)npair * nsolve, g.nz, ZS, 23.0, 10.0, ctx->sms);
        const long long per = (long long)npair * nseg;
        // 32-bit thread numbers: a batch past them goes in several launches
        const int most = (int)std::max(1LL, std::min((long long)nsolve, (1LL << 31) / per));
        for (int s0 = 0; s0 < nsolve; s0 += most) {
            const int ns = std::min(most, nsolve - s0);
            StepArgs<double> b = a;
            b.cur += (size_t)s0 * g.solve_stride;
            b.nxt += (size_t)s0 * g.solve_stride;
            b.src += s0;
            b.stf += (size_t)s0 * g.nsteps;
            b.trace += (size_t)s0 * g.nlev * g.nrec * 2;
            const unsigned nthr = (unsigned)(per * ns);
            const auto kernel = nseg == g.nz ? k_step64<1> : k_step64<ZS>;
            kernel<<<(nthr + 32 * wz - 1) / (32 * wz), 32 * wz, 0, st>>>(b, npair, nseg, nthr);
        }
    } else {
        const int rows_per_block = wz * ZS;
        dim3 grid((g.nx + 31) / 32, (g.nz + rows_per_block - 1) / rows_per_block, nsolve);
        k_step<real, ZS><<<grid, dim3(32, wz), 0, st>>>(a);
    }
}

template <typename real, int ZS>
static void launch_steps_zs(const oed_ctx *ctx, int nsolve, cudaStream_t st, cudaEvent_t ev0,
                            cudaEvent_t ev1)
{
    const Geometry &g = ctx->g;
    real *u0 = (real *)ctx->d_u0, *u1 = (real *)ctx->d_u1;
    StepArgs<real> a;
    a.fac = (const FacCoef<real> *)ctx->d_fac;
    a.src = (const SourceDesc<real> *)ctx->d_src;
    a.stf = (const real *)ctx->d_stf;
    a.trace = (real *)ctx->d_trace;
    a.rec = ctx->d_rec;
    a.g = g;
    // external event records so they become event nodes of a captured graph
    if (ev0) cudaEventRecordWithFlags(ev0, st, cudaEventRecordExternal);
    for (int m = 0; m < g.nsteps; m++) {
        a.cur = (m & 1) ? u1 : u0;
        a.nxt = (m & 1) ? u0 : u1;
        a.m = m;
        launch_one<real, ZS>(ctx, nsolve, a, st);
    }
    if (ev1) cudaEventRecordWithFlags(ev1, st, cudaEventRecordExternal);
    const real *last = (g.nsteps & 1) ? u1 : u0;
    k_gather<real><<<nsolve, 128, 0, st>>>(last, (real *)ctx->d_trace, ctx->d_rec, g, g.nsteps,
                                           nsolve);
}

template <typename real>
static void launch_steps(const oed_ctx *ctx, int nsolve, cudaStream_t st, cudaEvent_t ev0,
                         cudaEvent_t ev1)
{
    switch (ctx->tune.zs) {
    case 2: launch_steps_zs<real, 2>(ctx, nsolve, st, ev0, ev1); break;
    case 8: launch_steps_zs<real, 8>(ctx, nsolve, st, ev0, ev1); break;
    default: launch_steps_zs<real, 4>(ctx, nsolve, st, ev0, ev1); break;
    }
}

// Autotuner probe: nrep stencil launches for nsolve solves with the context's
// current tuning, bracketed by ev0 / ev1 (fields and traces are scratch here).
template <typename real, int ZS>
static void probe_zs(const oed_ctx *ctx, int nsolve, int nrep, cudaStream_t st, cudaEvent_t ev0,
                     cudaEvent_t ev1)
{
    const Geometry &g = ctx->g;
    StepArgs<real> a;
    a.fac = (const FacCoef<real> *)ctx->d_fac;
    a.src = (const SourceDesc<real> *)ctx->d_src;
    a.stf = (const real *)ctx->d_stf;
    a.trace = (real *)ctx->d_trace;
    a.rec = ctx->d_rec;
    a.g = g;
    cudaEventRecord(ev0, st);
    for (int m = 0; m < nrep; m++) {
        a.cur = (real *)((m & 1) ? ctx->d_u1 : ctx->d_u0);
        a.nxt = (real *)((m & 1) ? ctx->d_u0 : ctx->d_u1);
        a.m = m % g.nsteps;
        launch_one<real, ZS>(ctx, nsolve, a, st);
    }
    cudaEventRecord(ev1, st);
}

template <typename real>
static void probe_real(const oed_ctx *ctx, int nsolve, int nrep, cudaStream_t st, cudaEvent_t ev0,
                       cudaEvent_t ev1)
{
    switch (ctx->tune.zs) {
    case 2: probe_zs<real, 2>(ctx, nsolve, nrep, st, ev0, ev1); break;
    case 8: probe_zs<real, 8>(ctx, nsolve, nrep, st, ev0, ev1); break;
    default: probe_zs<real, 4>(ctx, nsolve, nrep, st, ev0, ev1); break;
    }
}

// Fill the level buffers the autotuner's probes run on with a deterministic pattern of
// order-one values (a hash of the index): the probes then time the kernels on data like
// a running solve's rather than on zeros, on which some kernels run at another speed.
template <typename real>
__global__ void k_fill_probe(real *__restrict__ u, size_t n, unsigned salt)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const unsigned h = ((unsigned)i ^ salt) * 2654435761u;
        u[i] = (real)((double)(h >> 8) * (1.0 / 16777216.0) - 0.5);
    }
}

// Source patches without weight, spread over the grid as a batch's are: a multi-step kernel's tiles
// and strips with a source take longer, and those of a corner are slow without one.
template <typename real>
__global__ void k_fill_probe_src(SourceDesc<real> *__restrict__ src, int nsolve, int nx, int nz)
{
    const int s = blockIdx.x;
    SourceDesc<real> &d = src[s];
    if (threadIdx.x == 0) {
        const unsigned h = ((unsigned)s + 1u) * 2654435761u;
        d.i0 = 1 + (int)((h >> 16) % (unsigned)max(1, nx - kPatch - 1));
        d.j0 = (int)(((h & 0xffffu) * 40503u >> 8) % (unsigned)max(1, nz - kPatch));
        d.ok = 1;
    }
    for (int k = threadIdx.x; k < kPatch * kPatch; k += blockDim.x) d.wx[k] = d.wz[k] = (real)0;
}

void launch_fill_probe(const oed_ctx *ctx, int nsolve, cudaStream_t st)
{
    if (ctx->d_u2) {
        k_fill_probe_src<float><<<nsolve, 64, 0, st>>>((SourceDesc<float> *)ctx->d_src, nsolve, ctx->g.nx, ctx->g.nz);
        cudaMemsetAsync(ctx->d_stf, 0, (size_t)nsolve * ctx->g.nsteps * sizeof(float), st);
    }
    size_t per = ctx->g.solve_stride;
    if (ctx->d_u2) per = per > strip_stride(ctx->g) ? per : strip_stride(ctx->g);
    const size_t n = (size_t)nsolve * per;
    void *lv[4] = {ctx->d_u0, ctx->d_u1, ctx->d_u2, ctx->d_u3};
    for (int k = 0; k < 4; k++) {
        if (!lv[k]) continue;
        if (ctx->precision == OED_FP64)
            k_fill_probe<double><<<152 * 8, 256, 0, st>>>((double *)lv[k], n, 0x9e3779b9u * (k + 1));
        else
            k_fill_probe<float><<<152 * 8, 256, 0, st>>>((float *)lv[k], n, 0x9e3779b9u * (k + 1));
    }
}

void launch_step_probe(const oed_ctx *ctx, int nsolve, int nrep, cudaStream_t st, cudaEvent_t ev0,
                       cudaEvent_t ev1)
{
    if (ctx->precision == OED_FP64)
        probe_real<double>(ctx, nsolve, nrep, st, ev0, ev1);
    else
        probe_real<float>(ctx, nsolve, nrep, st, ev0, ev1);
}

// Zero both level buffers (u^0 = u^{-1} = 0, Eq. elastic_2nd) and run all steps;
// ev0 / ev1 (may be null) bracket the stencil launches.
cudaError_t launch_forward_steps(const oed_ctx *ctx, int nsolve, cudaStream_t st, cudaEvent_t ev0,
                                 cudaEvent_t ev1)
{
    if (ctx->tune.C == -2) {   // the multi-step kernel's strip layout
        const size_t pb = 2 * (size_t)nsolve * strip_stride(ctx->g) * sizeof(float);
        cudaMemsetAsync(ctx->d_u0, 0, pb, st);
        cudaMemsetAsync(ctx->d_u2, 0, pb, st);
        return launch_steps_strip(ctx, nsolve, st, ev0, ev1, 0);
    }
    if (ctx->tune.C == -3) {   // the two-step kernel's paired layout
        const size_t pb = (size_t)nsolve * paired_stride(ctx->g) * sizeof(float);
        void *lv[4] = {ctx->d_u0, ctx->d_u1, ctx->d_u2, ctx->d_u3};
        for (void *p : lv) cudaMemsetAsync(p, 0, pb, st);
        const float *last = nullptr;
        const cudaError_t e = launch_steps_tma2(ctx, nsolve, st, ev0, ev1, 0, &last);
        if (e != cudaSuccess) return e;
        launch_tma2_gather(ctx, nsolve, last, ctx->g.nsteps, st);
        return cudaGetLastError();
    }
    const size_t bytes = (size_t)nsolve * ctx->g.solve_stride * ctx->elem;
    cudaMemsetAsync(ctx->d_u0, 0, bytes, st);
    cudaMemsetAsync(ctx->d_u1, 0, bytes, st);
    if (ctx->tune.C == -1) {
        const cudaError_t e = launch_steps_tma(ctx, nsolve, st, ev0, ev1, 0);
        if (e != cudaSuccess) return e;
        const float *last = (const float *)((ctx->g.nsteps & 1) ? ctx->d_u1 : ctx->d_u0);
        k_gather<float><<<nsolve, 128, 0, st>>>(last, (float *)ctx->d_trace, ctx->d_rec, ctx->g,
                                                ctx->g.nsteps, nsolve);
        return cudaGetLastError();
    }
    if (ctx->precision == OED_FP64)
        launch_steps<double>(ctx, nsolve, st, ev0, ev1);
    else
        launch_steps<float>(ctx, nsolve, st, ev0, ev1);
    return cudaGetLastError();
}

template <typename real>
__global__ void k_trace_f64(const real *__restrict__ trace, const SourceDesc<real> *__restrict__ src,
                            Geometry g, int nsolve, double *__restrict__ out)
{
    const size_t per = (size_t)g.nlev * g.nrec * 2;
    const size_t n = per * nsolve;
    const double nan = __longlong_as_double(0x7ff8000000000000ULL);
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x) {
        const int s = (int)(k / per);
        out[k] = src[s].ok ? (double)trace[k] : nan;
    }
}

void launch_trace_to_f64(const oed_ctx *ctx, int nsolve, double *g, cudaStream_t st)
{
    const size_t n = (size_t)ctx->g.nlev * ctx->g.nrec * 2 * nsolve;
    const int blocks = (int)((n + 255) / 256 < 152 * 16 ? (n + 255) / 256 : 152 * 16);
    if (ctx->precision == OED_FP64)
        k_trace_f64<double><<<blocks, 256, 0, st>>>((const double *)ctx->d_trace,
                                                    (const SourceDesc<double> *)ctx->d_src,
                                                    ctx->g, nsolve, g);
    else
        k_trace_f64<float><<<blocks, 256, 0, st>>>((const float *)ctx->d_trace,
                                                   (const SourceDesc<float> *)ctx->d_src, ctx->g,
                                                   nsolve, g);
}

}  // namespace oed
