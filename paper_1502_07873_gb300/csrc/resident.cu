// Cluster-resident time stepping: one thread-block cluster integrates one solve
// through all of its time steps with the wavefield held in distributed shared
// memory (Sec. 3.3.1, Eq. Full_Disc; the node update of stencil_cell.cuh).
//
// CTA r of a cluster of C owns rows [r R, min((r+1) R, nz)) of the grid, both
// components and both time levels, in its shared memory:
//     A, B : [R][rs] float2,   coef : [R] KP (FacCoef in (x, z) pairs)
// A row stores the even columns' (x, z) in sq = npair + 2 float2 slots, then the odd
// columns' in sq more; slot q of each half belongs to the column pair p = q - 1, and
// slots 0 and npair + 1 (columns -2, -1, nx..) are zero
// ghosts.  A thread owning pair p reads its whole neighbourhood, both components at
// once, with four 64-bit loads (its two columns, the west column from the odd half
// and the east column from the even half), each at an 8-byte stride across the
// warp: no bank conflicts.  Level m lives in A (m
// even) or B (m odd); u^{m+1} overwrites u^{m-1} in place.  The rows just above
// and below a CTA's slab are read straight from the neighbouring CTA's shared
// memory (mapa + ld.shared::cluster).  One cluster barrier (arrive.release /
// wait.acquire) per step orders the writes of step m before the reads of step
// m+1 and the reads of step m before the overwrites of step m+1; every thread of
// every CTA executes the same number of barriers.  Threads are packed densely
// over (row segment, column pair); each marches down its segment.  A row enters
// the register window once, as the south row, where its second differences and
// east - west differences are formed; its south differences are formed when the
// next row arrives, and all of them serve it again as the centre and north row.
// The surface row, the bottom row and the rows whose neighbour lives in another
// CTA are peeled off the main loop, and so are the march's last one to three rows
// (the only ones that do not prefetch): the unrolled march body has no branch.  The
// absorbing side columns are left out of the march (its stores to them go to ghost
// slots that no thread reads) and written by a separate edge warp from u^m alone, so
// the warps that hold a side column march exactly like the others; the same warp adds
// the source term to the patch nodes once the march warps that own them have stored
// them (named barrier 1).  The arithmetic runs on packed
// (x, z) pairs (.f32x2).  HBM traffic is only the seismogram samples and the source
// time function: the wavefield never leaves the chip, so this kernel is bound by the
// shared-memory pipe (eight 64-bit accesses per column pair, row and step) and the per-step
// barrier, not by HBM.  Large launches: 81x41 867 Gcell-upd/s (three CTAs an SM), 101x76, two
// layers, 722, 151x76, three layers, 784, 201x101 706, 401x201 696 (clusters of six: 138 of 152 SMs
// have a CTA).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "pair_math.cuh"

namespace oed {

// Block size and register cap: registers are split over the SM's four schedulers
// (16 K each), so 20 warps of 96 registers is the most one CTA can hold (the packed
// update needs about 90).  The last warp is the edge warp.
constexpr int kResThreads = 640;
constexpr int kResRegs = 96;
constexpr int kEdgeRec = 6;   // receiver offsets a lane of the edge warp keeps (96 receivers)
constexpr int kEdgeRows = 2;  // rows of the slab whose absorbing speeds a lane of it keeps
constexpr size_t kSmemPerSm = 228 * 1024;   // shared memory of an SM, 1 KB of it reserved per CTA

struct ResArgs {
    const FacCoef<float> *fac;     // [nz]
    const SourceDesc<float> *src;  // [nsolve]
    const float *stf;              // [nsolve][nsteps]
    float *trace;                  // [nsolve][nlev][nrec][2]
    const int *rec;                // [nrec]
    Geometry g;
    int R;                         // rows per CTA
    int sq;                        // float2 slots per half row, npair + 2
    int rs;                        // float2 slots per row, 2 sq and the padding
    int npair;                     // column pairs per row, (nx + 1) / 2
    int np;                        // threads per segment, npair and the idle ones
    int shift;                     // 1: segments start below the surface row
    int nseg;                      // row segments per column pair
    int rps;                       // rows per segment (the last takes what is left)
    int nmarch;                    // threads of the march warps; the last warp is the edge warp
};

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n"
                 "barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// The end of a step: the edge warp and the march warps reach it from loops of their own
template <bool ONE>
__device__ __forceinline__ void step_barrier()
{
    if (ONE)
        asm volatile("barrier.sync.aligned 0;" ::: "memory");
    else
        cluster_barrier();
}

// shared::cta address of a local pointer, and its image in CTA `rank` of the cluster
__device__ __forceinline__ unsigned smem_addr(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned remote_addr(unsigned local, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}

__device__ __forceinline__ float2 lds2(unsigned a)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void sts2(unsigned a, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

__device__ __forceinline__ float2 ld_cluster2(unsigned addr)
{
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

// A shared row holds the even columns' (x, z) in its first sq float2 slots and the odd
// columns' in the next sq: slot q of each half belongs to the column pair p = q - 1, so
// the pair of a thread is (E[q], O[q]), its west column O[q-1] and its east column
// E[q+1] -- four 64-bit loads at an 8-byte stride across the warp, no bank conflicts.
// Addresses are 32-bit shared ones: a is the thread's even slot of a row, so8 the bytes from
// the even half to the odd one.
__device__ __forceinline__ float4 pair_at(unsigned a, unsigned so8)
{
    const float2 e = lds2(a), o = lds2(a + so8);
    return make_float4(e.x, e.y, o.x, o.y);
}

// The pair's slots in the level being written (u^{m-1} in, u^{m+1} out), at per-thread
// byte offsets offE (column c) and offO (column c + 1) from a: 0 and so8 for interior pairs.  A
// side column is written by the edge warp, not by the march, so its thread's slot is moved to a
// ghost slot that no thread reads (even slot 0, or slot npair + 1 of either half): the march's
// stores stay unconditional.  (The ghost column nx of an odd width is read by the thread of the
// side column nx - 1 alone, whose results are not used.)
__device__ __forceinline__ float4 pair_at_n(unsigned a, int offE, int offO)
{
    const float2 e = lds2(a + offE), o = lds2(a + offO);
    return make_float4(e.x, e.y, o.x, o.y);
}

__device__ __forceinline__ void pair_put_n(unsigned a, int offE, int offO, float4 u)
{
    sts2(a + offE, make_float2(u.x, u.y));
    sts2(a + offO, make_float2(u.z, u.w));
}

__device__ __forceinline__ void load_row(unsigned a, unsigned so8, Row2P &r)
{
    const float4 m = pair_at(a, so8);
    row_fromP(lds2(a + so8 - 8u), m, lds2(a + 8u), r);
}

// the same slots of a row in CTA `nb` of the cluster
__device__ __forceinline__ float4 pair_at_remote(unsigned a, unsigned so8, unsigned nb)
{
    const unsigned b = remote_addr(a, nb);
    const float2 e = ld_cluster2(b), o = ld_cluster2(b + so8);
    return make_float4(e.x, e.y, o.x, o.y);
}

__device__ __forceinline__ void load_row_remote(unsigned a, unsigned so8, unsigned nb, Row2P &r)
{
    const unsigned b = remote_addr(a, nb);
    const float2 e = ld_cluster2(b), o = ld_cluster2(b + so8);
    row_fromP(ld_cluster2(b + so8 - 8u), make_float4(e.x, e.y, o.x, o.y), ld_cluster2(b + 8u), r);
}

// slot of column i within a shared row, and the float offset of its component comp
__device__ __forceinline__ int node_slot(int i, int sq) { return (i & 1) ? sq + (i >> 1) + 1 : (i >> 1) + 1; }
__device__ __forceinline__ int node_off(int i, int comp, int sq) { return 2 * node_slot(i, sq) + comp; }

// HOM: the medium is homogeneous, so every march row has the coefficients of row 1.
// ONE: clusters of one CTA, no remote rows and a CTA barrier in place of the cluster's.
template <bool HOM, bool ONE>
__global__ void __maxnreg__(kResRegs) k_resident(ResArgs a)
{
    extern __shared__ float4 smem4[];
    const Geometry &g = a.g;
    const unsigned rank = ONE ? 0 : cluster_rank();
    const int s = blockIdx.y;
    const int R = a.R, sq = a.sq;
    const int j0 = (int)rank * R;
    const int nrows = max(0, min(R, g.nz - j0));
    const int RS = a.rs;
    float2 *A = reinterpret_cast<float2 *>(smem4), *B = A + R * RS;
    KP *coef = reinterpret_cast<KP *>(smem4 + R * RS);
    const unsigned level0 = smem_addr(A), lvl8 = 8u * (unsigned)(R * RS);   // shared address of level A; B is lvl8 on
    const int tid = threadIdx.x;
    const int nthr = blockDim.x;

    for (int k = tid; k < R * RS; k += nthr) smem4[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int k = tid; k < nrows; k += nthr) coef[k] = pack_coef(a.fac[j0 + k]);

    // march threads are packed densely over (segment, pair): a warp may straddle two
    // segments.  The last warp (the edge warp) takes the absorbing side columns, which
    // the march does not store, and the receiver samples: side columns read only u^m, so
    // this needs no synchronisation with the march, and no march warp is slowed down by
    // the absorbing patch of a side column.
    const bool edge = tid >= a.nmarch;
    const int p = tid % a.np;
    const int c = 2 * p;
    const int seg = tid / a.np;
    const bool active = !edge && seg < a.nseg && p < a.npair;
    const int kind = (c == 0 ? 1 : 0) | (c + 1 == g.nx - 1 ? 2 : 0) | (c == g.nx - 1 ? 4 : 0);
    const unsigned so8 = 8u * (unsigned)sq, rs8 = 8u * (unsigned)RS;   // bytes: half row, row
    const int offE = (kind & 1) ? -8 : ((kind & 4) ? 8 : 0);
    const int offO = (int)so8 + ((kind & 2) ? 8 : 0);
    // The rows are cut into segments of rps rows.  The surface row, and the slab's last row, are no
    // march rows; the segments that hold them take them besides.  With shift the surface row is not
    // counted, so that the lanes of a warp that straddles segments run the same loop.
    const bool top = rank == 0 && seg == 0;
    const int shift = ONE ? 1 : (rank == 0 ? a.shift : 0);
    const int l0 = seg * a.rps + (top ? 1 : shift);     // first march row
    const int l1 = seg == a.nseg - 1 ? nrows : min((seg + 1) * a.rps + shift, nrows);
    const bool rows = active && (top || l0 < l1);
    const unsigned slot0 = level0 + 8u * (unsigned)(l0 * RS + p + 1);
    const SourceDesc<float> *sd = a.src + s;
    const int sj = sd->j0, si0 = sd->i0;
    const int siA = c - sd->i0, siB = c + 1 - sd->i0;
    const bool scolA = (unsigned)siA < (unsigned)kPatch;
    const bool scolB = c + 1 < g.nx && (unsigned)siB < (unsigned)kPatch;
    const float *stf = a.stf + (size_t)s * g.nsteps;
    // The source term of the patch nodes is added by the edge warp once the march warps
    // that own patch nodes of this CTA have stored them: those warps arrive at named
    // barrier 1 after their march (without waiting), the edge warp waits there.  The
    // count is fixed per CTA, so every step's barrier completes.
    const int srow0 = max(sj, j0), srow1 = min(sj + kPatch, j0 + nrows);   // patch rows in this CTA
    const bool patch = rows && (scolA || scolB) && sj + kPatch > j0 + (top ? 0 : l0) && sj < j0 + l1;
    const bool patch_warp = __any_sync(0xffffffffu, patch);
    float *trace = a.trace + (size_t)s * g.nlev * g.nrec * 2;
    // The march keeps its rows' coefficients in registers instead of reloading them row by
    // row: in a homogeneous medium they are the CTA's, otherwise where the march rows of every
    // lane of a warp (its segment's, without the surface row and the slab's last row, which are
    // peeled) have one set each, as anywhere but around a layer interface.
    const int lfirst = HOM ? (rank == 0 ? 1 : 0) : l0, llast = min(l1, nrows - 1);
    __syncthreads();
    const KP K0 = coef[min(lfirst, nrows - 1)];
    // Elsewhere bit k says that the k-th march row has other coefficients than the one before
    // (from row 31 on, where the shifted-in sign says so, every row reloads): the warps at a layer
    // interface, which the others wait for, loaded four 16-byte words a row (401x201, three
    // layers: 618 -> 637 Gcell-upd/s; 101x76, two: 634 -> 667).
    int change = 0;
    if (!HOM && active)
        for (int k = lfirst + 1; k < llast; k++)
            if (!kp_equal(coef[k], coef[k - 1])) change |= k - lfirst < 31 ? 1 << (k - lfirst) : -1;
    const bool unif = HOM || __all_sync(0xffffffffu, change == 0) != 0;
    const int npw = __syncthreads_count(patch_warp && (tid & 31) == 0);
    if (!ONE) cluster_barrier();

    if (edge) {
        // What the edge warp needs of a step beside u^m it holds in registers: on the step's
        // critical path (the source term comes last, behind the march warps that own the patch)
        // stand one wait, one shared load, one fma and one store.  (With the time function, the
        // receivers' columns and the weights read in the step: one solve of 81x41 in seven CTAs
        // 0.419 ms for 400 steps against 0.309; 2048 solves 655 Gcell-upd/s against 708.)
        const int e = tid - a.nmarch;
        int ro[kEdgeRec];
#pragma unroll
        for (int k = 0; k < kEdgeRec; k++) {
            const int q = e + 32 * k;
            ro[k] = rank == 0 && q < 2 * g.nrec ? node_off(a.rec[q >> 1], q & 1, sq) : -1;
        }
        constexpr int kNodes = (kPatch * kPatch + 31) / 32;
        int po[kNodes];
        float wx[kNodes], wz[kNodes];
#pragma unroll
        for (int k = 0; k < kNodes; k++) {
            const int q = e + 32 * k, bb = q / kPatch, ai = q - bb * kPatch, j = sj + bb;
            po[k] = -1;
            if (q < kPatch * kPatch && j >= srow0 && j < srow1) {
                po[k] = (j - j0) * RS * 2 + node_off(si0 + ai, 0, sq);
                wx[k] = sd->wx[q];
                wz[k] = sd->wz[q];
            }
        }
        const int oL = node_slot(0, sq), oL1 = node_slot(1, sq);
        const int oR = node_slot(g.nx - 1, sq), oR1 = node_slot(g.nx - 2, sq);
        float2 sc[kEdgeRows];   // absorbing speeds of the lane's rows
#pragma unroll
        for (int k = 0; k < kEdgeRows; k++)
            sc[k] = e + 32 * k < nrows ? coef[e + 32 * k].c : make_float2(0.0f, 0.0f);
        float S = stf[0];
        for (int m = 0; m < g.nsteps; m++) {
            const float *cf = reinterpret_cast<const float *>((m & 1) ? B : A);   // u^m
            float *nf = reinterpret_cast<float *>((m & 1) ? A : B);               // u^{m+1}
            const float Sn = m + 1 < g.nsteps ? stf[m + 1] : 0.0f;
            float *tr = trace + (size_t)m * g.nrec * 2;
#pragma unroll
            for (int k = 0; k < kEdgeRec; k++)
                if (ro[k] >= 0) tr[e + 32 * k] = cf[ro[k]];
            if (rank == 0)
                for (int q = e + 32 * kEdgeRec; q < 2 * g.nrec; q += 32)
                    tr[q] = cf[node_off(a.rec[q >> 1], q & 1, sq)];
            // side columns 0 and nx-1 (first-order absorbing, from the inward neighbour;
            // they take precedence at the surface and bottom corners)
            auto side = [&](int l, float2 k) {
                const float2 *cr = reinterpret_cast<const float2 *>(cf) + l * RS;
                float2 *nr = reinterpret_cast<float2 *>(nf) + l * RS;
                const float2 L = cr[oL], L1 = cr[oL1], Q = cr[oR], Q1 = cr[oR1];
                nr[oL] = make_float2(absorb(L.x, L1.x, k.x), absorb(L.y, L1.y, k.y));
                nr[oR] = make_float2(absorb(Q.x, Q1.x, k.x), absorb(Q.y, Q1.y, k.y));
            };
#pragma unroll
            for (int k = 0; k < kEdgeRows; k++)
                if (e + 32 * k < nrows) side(e + 32 * k, sc[k]);
            for (int l = e + 32 * kEdgeRows; l < nrows; l += 32) side(l, coef[l].c);
            // source term: u^{m+1} += dt^2/nu f^m on the patch nodes of this CTA, added last
            // as in the node update of the streaming kernel
            if (npw > 0) {
                asm volatile("bar.sync 1, %0;" :: "r"(32 * (npw + 1)) : "memory");
#pragma unroll
                for (int k = 0; k < kNodes; k++)
                    if (po[k] >= 0) {
                        nf[po[k]] = add_force(nf[po[k]], S, wx[k]);
                        nf[po[k] + 1] = add_force(nf[po[k] + 1], S, wz[k]);
                    }
            }
            S = Sn;
            step_barrier<ONE>();
        }
    }
    for (int m = edge ? g.nsteps : 0; m < g.nsteps; m++) {   // the march warps
        // this thread's even slot in its segment's first row
        const unsigned cur = slot0 + ((m & 1) ? lvl8 : 0u), nxt = slot0 + ((m & 1) ? 0u : lvl8);
        if (rows) {
            Row2P rn, rc, rs;   // the rows l - 1 and l
            int l = l0;
            if (ONE || l > 0)
                load_row(cur - rs8, so8, rn);
            else
                load_row_remote(cur + (R - 1) * rs8, so8, rank - 1, rn);
            if (ONE || l < nrows)
                load_row(cur, so8, rc);
            else   // a one-row slab below the surface
                load_row_remote(cur - rs8, so8, rank + 1, rc);
            southP(rn, rc);
            if (top) {   // surface row: no north differences, cross terms on the row itself
                Row2P nt = rn;
                nt.va = nt.vb = make_float2(0.0f, 0.0f);
                float4 u = pair_at_n(nxt - rs8, offE, offO);
                const KP K = coef[0];
                pair_updateP(K, nt, rn, rc, u);
                pair_put_n(nxt - rs8, offE, offO, u);
            }
            // rows whose south neighbour is a local row and that are not the bottom row:
            // unrolled by three with the three window rows taking turns
            const int lstop = min(l1, nrows - 1);
            if (l < lstop) {
                // Four shared addresses move down with the march: the even and odd slots of the row
                // to fetch, and of the row whose u^{m-1} is fetched with it and that is stored next
                unsigned pe = cur + rs8, po = pe + so8, we = nxt + offE, wo = nxt + offO;
                const KP *cf = coef + l;
                // the loads of the next row are issued before the update of this one
                float4 pm, pu;
                float2 pw, px;
                auto fetch = [&] {
                    const float2 e = lds2(pe), o = lds2(po);
                    pm = make_float4(e.x, e.y, o.x, o.y);
                    pw = lds2(po - 8u);
                    px = lds2(pe + 8u);
                    const float2 a0 = lds2(we), b0 = lds2(wo);
                    pu = make_float4(a0.x, a0.y, b0.x, b0.y);
                };
                fetch();
                // pf: a row below the south row exists, prefetch it (every row but the last)
                // unifK: each lane's march rows share its K0 (no coefficient loads)
                auto march = [&](auto unifK) {
                    KP K = K0;
                    int cg = change;
                    auto row = [&](auto pf, const Row2P &wn, Row2P &wc, Row2P &ws) {
                        row_fromP(pw, pm, px, ws);
                        float4 u = pu;
                        const unsigned se = we, so = wo;
                        if constexpr (decltype(pf)::value) {
                            pe += rs8;
                            po += rs8;
                            we += rs8;
                            wo += rs8;
                            fetch();
                        }
                        southP(wc, ws);
                        if constexpr (!decltype(unifK)::value) {
                            if (cg & 1) K = *cf;
                            cg >>= 1;
                        }
                        pair_updateP(K, wn, wc, ws, u);
                        sts2(se, make_float2(u.x, u.y));
                        sts2(so, make_float2(u.z, u.w));
                        cf++;
                    };
                    const std::true_type P{};
                    const std::false_type N{};
                    for (; l + 3 < lstop; l += 3) {
                        row(P, rn, rc, rs);   // window (n, c, s)
                        row(P, rc, rs, rn);   // row l+2 lands in rn
                        row(P, rs, rn, rc);   // row l+3 lands in rc
                    }
                    // one to three rows left, the last without prefetch; the window ends
                    // as (rn, rc) = (north, centre) of the row after the march
                    const int r = lstop - l;
                    if (r == 3) {
                        row(P, rn, rc, rs);
                        row(P, rc, rs, rn);
                        row(N, rs, rn, rc);
                    } else if (r == 2) {
                        row(P, rn, rc, rs);
                        row(N, rc, rs, rn);
                        const Row2P t = rn;
                        rn = rs;
                        rc = t;
                    } else {
                        row(N, rn, rc, rs);
                        rn = rc;
                        rc = rs;
                    }
                    l = lstop;
                };
                // a warp-uniform choice: a branch inside the march body would split the
                // unrolled rows into separate blocks and cost the scheduler its overlap
                if (HOM || unif)
                    march(std::true_type{});
                else
                    march(std::false_type{});
            }
            // what is left: a last interior row whose south neighbour sits in CTA rank+1,
            // or the absorbing bottom row
            if (l < l1) {
                const unsigned lr = (unsigned)(l - l0) * rs8;
                const KP K = coef[l];
                float4 u = pair_at_n(nxt + lr, offE, offO);
                if (ONE || j0 + l == g.nz - 1) {
                    const float4 nv = ONE || l > 0 ? pair_at(cur + lr - rs8, so8)
                                                   : pair_at_remote(cur + (R - 1) * rs8, so8, rank - 1);
                    absorbingP(K.c, nv, rc, true, 0, u);
                } else {
                    load_row_remote(cur - (unsigned)l0 * rs8, so8, rank + 1, rs);
                    southP(rc, rs);
                    pair_updateP(K, rn, rc, rs, u);
                }
                pair_put_n(nxt + lr, offE, offO, u);
            }
        }
        if (patch_warp)
            asm volatile("bar.arrive 1, %0;" :: "r"(32 * (npw + 1)) : "memory");
        step_barrier<ONE>();
    }
    if (rank == 0) {
        const float *row0 = reinterpret_cast<const float *>((g.nsteps & 1) ? B : A);
        for (int q = tid; q < 2 * g.nrec; q += nthr)
            trace[(size_t)g.nsteps * g.nrec * 2 + q] = row0[node_off(a.rec[q >> 1], q & 1, sq)];
    }
}

// Shape of the resident launch for a grid: cluster size C (1..8) and rows per CTA,
// or C = 0 when the two levels do not fit in C CTAs of shared memory.
struct ResShape {
    int C, R, sq, rs, shift, npair, np, nseg, rps, nmarch, threads;
    size_t smem;
};

// kmax: the most CTAs one SM gets of the launch, so the most that are worth planning for.
//
// The slab's rows go to nseg segments of rps rows, the last takes what is left.  With no more
// than one CTA an SM the step's latency counts: the fewest rows a thread.  Otherwise the plan of
// the highest product of
//   sqrt(the share of the warps' lanes and rows that hold nodes; the longest segment sets the step),
//   rows / (rows + 3): what a segment costs besides its rows (the row above it, its start),
//   warps / (warps + 15): all CTAs' warps on the SM, which hide each other's latency,
//   balance^(1/6): a CTA's warps go to the SM's four schedulers in turn,
//   0.92 where straddling warps have bank conflicts, else 0.97 where the edge warp has.
// A fit to 1050 plans of 29 grids: it takes one 1.9% slower than the best on average.  Against as
// many segments as a share of the registers' warps allows, scored by warps and CTAs alone,
// Gcell-upd/s: 41x21 325 -> 551, 50x50 612 -> 717, 64x64 743 -> 803, 81x41 766 -> 867, 101x101 666 ->
// 722, 101x76 668 -> 722 (two layers), 161x81 in clusters of two 684 -> 738; 401x201 in clusters of six 640 and
// 643; a few lose: 61x31 774 -> 755, 91x61 777 -> 736, 221x60 826 -> 784, 301x151 656 -> 642.
//
// A warp that straddles two segments reads two runs of slots: without bank conflicts if a
// segment's first slot lies as many slots behind the one before, modulo the 16 slots of a
// 64-bit access, as its first thread lies threads behind.  Rows get up to 15 slots of padding
// for that and segments up to 15 idle threads, as far as the warps and the CTAs per SM allow; an
// odd row also spreads the edge warp's column over the banks.  Gcell-upd/s without and with: 61x31
// 672 and 774, 81x41 712 and 766, 121x61 606 and 663, 151x76 712 and 777, 201x101 662 and 711,
// 401x201 684 and 696 (the side columns' 64-bit accesses included).
//
// Segments that start below the surface row (shift) have the same number of march rows, so a
// straddling warp does not diverge (81x41 766 -> 830 Gcell-upd/s, 201x101 in clusters of two 674 -> 701),
// but the first one takes a row more, and a cluster waits for it: not where straddling warps are
// few, from four warps a segment on (301x151 in clusters of four 601 and 624, 351x176 in clusters
// of six 553 and 563).
static ResShape resident_shape(const Geometry &g, int C, int kmax = 1)
{
    ResShape r{};
    const int npair = (g.nx + 1) / 2;
    if (npair > kResThreads - 32 || C < 1 || C > 8) return r;
    const int R = (g.nz + C - 1) / C;
    if ((C - 1) * R >= g.nz) return r;   // a CTA would own no rows
    const int sq = npair + 2;   // ghost slots on both sides
    auto bytes = [&](int rs) { return (size_t)R * rs * sizeof(float4) + (size_t)R * sizeof(KP); };
    // 392 bytes short of the limit: which grids count as on chip decides the workspace and which
    // launch shapes are accepted, and stays what it was with the source weights in shared memory
    if (bytes(2 * sq) + 392 > 227 * 1024) return r;
    r.shift = C == 1 || npair < 128;
    const int top = C == 1, most = std::min((kResThreads - 32) / npair, R);
    double best = -1.0;
    for (int n = 1; n <= most; n++)
        for (int d = -2; d <= 1; d++) {
            const int rps = (R + n - 1) / n + d, last = R - top - (n - 1) * rps;
            if (rps < 1 || last < 1 || (n == 1 && d != 0)) continue;
            const int rows = n == 1 ? R : std::max(rps + top, last);
            const int warps = (npair * n + 31) / 32;
            int k = std::min((int)(kSmemPerSm / (bytes(2 * sq) + 1024)), kResThreads / 32 / (warps + 1));
            k = std::max(1, std::min(k, kmax));
            int np = npair, rs = 2 * sq;
            bool found = false;
            for (int odd = 1; odd >= 0 && !found; odd--)
                for (int p = npair; p < npair + 16 && p * n <= 32 * warps && !found; p++)
                    for (int q = 2 * sq + odd; q < 2 * sq + 16 && !found; q += 2)
                        if ((n == 1 || (rps * q - p) % 16 == 0) && bytes(q) <= 227 * 1024 &&
                            k * (bytes(q) + 1024) <= kSmemPerSm) {
                            found = true;
                            np = p;
                            rs = q;
                        }
            const double full = (double)npair * R / (32.0 * warps * rows);
            const double sched = warps / (4.0 * ((warps + 3) / 4));
            const double score = kmax == 1 ? 1.0 / (rows + 0.01 * n)
                                           : sqrt(full) * rps / (rps + 3.0) * (k * warps) / (k * warps + 15.0) *
                                                 cbrt(sqrt(sched)) * (found ? (rs & 1 ? 1.0 : 0.97) : 0.92);
            if (score > best) {
                best = score;
                r.rs = rs;
                r.np = np;
                r.nseg = n;
                r.rps = rps;
                r.nmarch = 32 * warps;
            }
        }
    r.C = C;
    r.R = R;
    r.sq = sq;
    r.npair = npair;
    r.threads = r.nmarch + 32;
    r.smem = bytes(r.rs);
    return r;
}

// Smallest cluster that holds an FP32 grid, or 0 if none does.
int resident_fits(const Geometry &g)
{
    for (int C = 1; C <= 8; C++)
        if (resident_shape(g, C).C) return C;
    return 0;
}

// The same for a context (0 for FP64 contexts).
int resident_cluster_size(const oed_ctx *ctx)
{
    return ctx->precision == OED_FP32 ? resident_fits(ctx->g) : 0;
}

using ResKernel = void (*)(ResArgs);
static const ResKernel kResKernels[4] = {k_resident<false, false>, k_resident<false, true>, k_resident<true, false>,
                                         k_resident<true, true>};

// The kernel's dynamic shared-memory limit is always set to the device's opt-in
// maximum (launches may use less): a fixed value, so concurrent callers with
// different grids never lower it under each other.
static cudaError_t set_smem_limit()
{
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    for (ResKernel k : kResKernels) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static ResKernel resident_kernel(const oed_ctx *ctx, int C)
{
    bool hom = true;
    for (size_t l = 1; l < ctx->vp.size(); l++)
        hom &= ctx->vp[l] == ctx->vp[0] && ctx->vs[l] == ctx->vs[0] && ctx->rho[l] == ctx->rho[0];
    return kResKernels[2 * hom + (C == 1)];
}

int resident_max_active_clusters(const oed_ctx *ctx, int C)
{
    const ResShape r = resident_shape(ctx->g, C);
    if (!r.C) return 0;
    set_smem_limit();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r.C, 1, 1);
    cfg.blockDim = dim3(r.threads, 1, 1);
    cfg.dynamicSmemBytes = r.smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = r.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, resident_kernel(ctx, C), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// All nsteps steps of nsolve solves in one launch (grid: C CTAs per solve).
cudaError_t launch_resident(const oed_ctx *ctx, int C, int nsolve, cudaStream_t st, cudaEvent_t ev0,
                            cudaEvent_t ev1, int nsteps_override)
{
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const ResShape r = resident_shape(ctx->g, C, (int)(((long long)nsolve * C + nsm - 1) / nsm));
    if (!r.C) return cudaErrorInvalidValue;
    set_smem_limit();
    ResArgs a;
    a.fac = (const FacCoef<float> *)ctx->d_fac;
    a.src = (const SourceDesc<float> *)ctx->d_src;
    a.stf = (const float *)ctx->d_stf;
    a.trace = (float *)ctx->d_trace;
    a.rec = ctx->d_rec;
    a.g = ctx->g;
    if (nsteps_override > 0 && nsteps_override < a.g.nsteps) a.g.nsteps = nsteps_override;
    a.R = r.R;
    a.sq = r.sq;
    a.rs = r.rs;
    a.np = r.np;
    a.shift = r.shift;
    a.npair = r.npair;
    a.nseg = r.nseg;
    a.rps = r.rps;
    a.nmarch = r.nmarch;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r.C, nsolve, 1);
    cfg.blockDim = dim3(r.threads, 1, 1);
    cfg.dynamicSmemBytes = r.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = r.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (ev0) cudaEventRecord(ev0, st);
    cudaError_t e = cudaLaunchKernelEx(&cfg, resident_kernel(ctx, C), a);
    if (ev1) cudaEventRecord(ev1, st);
    return e;
}

}  // namespace oed
