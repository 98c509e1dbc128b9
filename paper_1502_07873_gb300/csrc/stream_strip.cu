// Several leap-frog steps per pass for grids whose wavefield does not fit the
// cluster-resident kernel (Sec. 3.3.1, Eq. Full_Disc; the packed node update of
// pair_math.cuh, so the bits are those of every other stencil kernel).
//
// A warp marches down a strip of 64 columns over a band of rows once per pass, T steps
// deep: when row z of u^m and u^{m-1} arrives, step 1 completes row z-1 of u^{m+1}, step 2
// row z-2 of u^{m+2} from it, ..., step T row z-T of u^{m+T}.  A lane owns a column pair; the
// rows in flight (two per step) stay in its registers and the west and east columns come
// from the neighbouring lanes by shuffles, so the steps need no shared memory, no barrier
// and no second trip to HBM.  Rows move in chunks of three, prefetched by cp.async, 16 bytes
// a lane, into a ring in shared memory that only the lane itself reads.  A strip's outer T
// columns and a band's outer T rows are computed by both neighbours: the own tile is 64 - 2H
// columns wide (H = T rounded up to even).  HBM traffic per cell-update is 32 / T bytes (two
// levels read and two written per T steps).  Levels live in two buffers used in alternation:
// a pass reads (u^{m-1}, u^m) from one and writes (u^{m+T-1}, u^{m+T}) to the other, so no
// strip overwrites what its neighbours still read.
//
// Most chunks run in a branch-free body in which the window rows take turns in the
// registers, with the rows' coefficients held in registers too: it needs the rows in
// flight to share them (each packed row holds the end of its run of equal rows).  Chunks
// that hold the surface or the bottom row, a row next to a layer interface or a row of the
// source patch go through a general body; the strips that hold a side column have a
// branch-free body of their own.
//
// What bounds it: HBM, with T = 4 at 8 B per cell-update (801x401, three layers, 672
// solves: 705 Gcell-upd/s, 83% of the measured copy rate; 70 solves of 1601x801: 730), and
// with few solves the blocks that do not fill the chip evenly (56 solves: 559; 7 of
// 1601x801: 535).  The two-step tile kernel runs these at 362, 340 and 325; it keeps the cases
// that this one is slower on: one or two solves, whose passes wait for the longest band,
// media with an interface every few rows (the general body takes about three times the
// plain one's time a row) and grids of few rows (stream_tma2.cu; oed_autotune chooses).  T = 2 (16 B) 390, T = 3 560: two more steps of registers
// cost less than their bytes.  Eight warps an SM at up to 255 registers: twelve at 168
// spill (673 on the 672 solves), sixteen much more (360).
#include <cmath>
#include <type_traits>

#include "pair_math.cuh"

namespace oed {

constexpr int kStripSteps = 4;    // T of the main passes
constexpr int kStripWarps = 8;    // resident warps per SM the registers are capped for
constexpr int kChunk = 3;         // rows per chunk
constexpr int kRingChunks = 4;    // chunks in the prefetch ring
constexpr int kRunCap = 512;      // longest run of equal rows that is looked up at once
constexpr int kChunkBytes = kChunk * 2 * 32 * (int)sizeof(float4);   // both levels of a chunk
constexpr int kRingBytes = kRingChunks * kChunkBytes;
constexpr int kStripSmem = kRingBytes + 8 * (int)sizeof(KP);   // and the coefficients of a general chunk

struct StripArgs {
    const float *in;              // u^{m-1} and u^m (strip layout)
    float *out;                   // u^{m+T-1} and u^{m+T}: the other buffer
    const KP *kp;                 // [nz] the rows' coefficients as (x, z) pairs
    const SourceDesc<float> *src;
    const float *stf;
    float *trace;
    const int *rec;
    Geometry g;
    int m, nsolve, nstrip, nband;
    int sq;                       // a level's row holds 2 sq column slots
    size_t pst;                   // floats per solve of a level pair
    int last;                     // the time loop ends with this pass: its level is sampled, not stored
};

// a grid row of one step's input level in the window of a lane
struct StripRow {
    float2 ca, cb;   // the pair's values
    float2 pa, pb;   // a lap + (u - previous level): the start of the operator sum
    float2 da, db;   // east - west differences, swapped (pair_math.cuh)
    float2 va, vb;   // south row minus this row
};

__device__ __forceinline__ float2 shfl2(float2 v, int lane_from)
{
    return make_float2(__shfl_sync(0xffffffffu, v.x, lane_from), __shfl_sync(0xffffffffu, v.y, lane_from));
}

// a new row enters the window: v its pair, um the previous level's
__device__ __forceinline__ void strip_feed(StripRow &s, float4 v, float4 um, float2 Ka)
{
    s.ca = make_float2(v.x, v.y);
    s.cb = make_float2(v.z, v.w);
    const float2 w = make_float2(__shfl_up_sync(0xffffffffu, v.z, 1), __shfl_up_sync(0xffffffffu, v.w, 1));
    const float2 e = make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
    const float2 t = sub2(s.cb, s.ca);
    const float2 la = sub2(t, sub2(s.ca, w));
    const float2 lb = sub2(sub2(e, s.cb), t);
    s.da = make_float2(v.w - w.y, v.z - w.x);
    s.db = make_float2(e.y - v.y, e.x - v.x);
    s.pa = fma2(Ka, la, sub2(s.ca, make_float2(um.x, um.y)));
    s.pb = fma2(Ka, lb, sub2(s.cb, make_float2(um.z, um.w)));
}

// the next level of row c (pair_updateP's operations in its order); nva .. ndb the north
// row's south and east - west differences
__device__ __forceinline__ float4 strip_update(const KP &K, float2 nva, float2 nvb, float2 nda, float2 ndb,
                                               StripRow &c, const StripRow &s)
{
    c.va = sub2(s.ca, c.ca);
    c.vb = sub2(s.cb, c.cb);
    float2 A = fma2(K.vs, c.va, c.pa);
    A = fma2(K.vn, nva, A);
    A = fma2(K.ds, s.da, A);
    A = fma2(K.dn, nda, A);
    float2 B = fma2(K.vs, c.vb, c.pb);
    B = fma2(K.vn, nvb, B);
    B = fma2(K.ds, s.db, B);
    B = fma2(K.dn, ndb, B);
    const float2 xa = add2(c.ca, A), xb = add2(c.cb, B);
    return make_float4(xa.x, xa.y, xb.x, xb.y);
}

// absorbing side columns (kind as in stencil_cell.cuh)
__device__ __forceinline__ void strip_side(float2 cpcs, const StripRow &c, int kind, float4 &u)
{
    const float cp = cpcs.x, cs = cpcs.y;
    if (kind & 1) {
        u.x = absorb(c.ca.x, c.cb.x, cp);
        u.y = absorb(c.ca.y, c.cb.y, cs);
    }
    if (kind & 2) {
        u.z = absorb(c.cb.x, c.ca.x, cp);
        u.w = absorb(c.cb.y, c.ca.y, cs);
    }
    if (kind & 4) {   // column nx-1: its east - west difference is -west (the ghost east is 0)
        u.x = absorb(c.ca.x, -c.da.y, cp);
        u.y = absorb(c.ca.y, -c.da.x, cs);
        u.z = 0.0f;
        u.w = 0.0f;
    }
}

__device__ __forceinline__ void cp_async16(unsigned dst, const char *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ float4 lds4(unsigned a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}

__device__ __forceinline__ void sts4(unsigned a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// a row's coefficients from shared memory
__device__ __forceinline__ KP ring_coef(unsigned d)
{
    const float4 u = lds4(d), v = lds4(d + 16), w = lds4(d + 32);
    KP k;
    k.a = make_float2(u.x, u.y);
    k.vs = make_float2(u.z, u.w);
    k.vn = make_float2(v.x, v.y);
    k.ds = make_float2(v.z, v.w);
    k.dn = make_float2(w.x, w.y);
    k.c = make_float2(w.z, w.w);
    return k;
}

// first row of band b of nband: the row that the first row of a chunk completes
template <int T>
__device__ __forceinline__ int band_row(int nz, int nband, int b)
{
    if (b == 0 || b == nband) return b ? nz : 0;
    return (int)((long long)nz * b / nband + T) / kChunk * kChunk - T;
}

template <int T>
__global__ void __launch_bounds__(32, kStripWarps) k_strip(const __grid_constant__ StripArgs a)
{
    constexpr int H = (T + 1) / 2 * 2, W = 64 - 2 * H;
    extern __shared__ float4 ring[];
    const Geometry &g = a.g;
    const int nz = g.nz;
    const int lane = threadIdx.x;
    const unsigned q = blockIdx.x / (unsigned)a.nstrip;
    const int strip = (int)(blockIdx.x - q * (unsigned)a.nstrip);
    const int s = (int)(q / (unsigned)a.nband);
    const int band = (int)(q - (unsigned)s * (unsigned)a.nband);
    const int z0 = band_row<T>(nz, a.nband, band), z1 = band_row<T>(nz, a.nband, band + 1);
    const int x0 = strip * W;
    const int c = x0 - H + 2 * lane;                   // the pair's first column
    const bool valid = c >= 0 && c < g.nx;
    const int kind = (c == 0 ? 1 : 0) | (c + 1 == g.nx - 1 ? 2 : 0) | (c == g.nx - 1 ? 4 : 0);
    const bool side = x0 == 0 || x0 + W + H >= g.nx;   // the strip holds a side column
    const SourceDesc<float> *src = a.src + s;
    const int sj0 = src->j0, si0 = src->i0;
    const bool has_src = si0 + kPatch > x0 - H && si0 < x0 - H + 64;
    const bool store = valid && c >= x0 && c < x0 + W && !a.last;

    // rows taken: zs .. z1 + T - 1 (those past nz - 1 are not used); row z completes row z - T.
    // Chunks start at multiples of three, so none of them mixes rows of two bands.
    const int zs = max(0, z0 + T - (2 * T + kChunk - 1) / kChunk * kChunk), zload = min(z1 + T, nz);
    const size_t ls = 16 * (size_t)a.sq, rs = 2 * ls;  // bytes per level of a row, per row
    // column c sits in slot c + 4 of the row; the pairs outside the grid read the zero slots 0, 1
    const unsigned at = valid ? 8u * (unsigned)(c + 4) : 0u;
    const char *pin = reinterpret_cast<const char *>(a.in) + ((size_t)s * a.pst * 4 + zs * rs);   // next chunk fetched
    char *pout = reinterpret_cast<char *>(a.out) + ((size_t)s * a.pst * 4 + (zs - T) * (ptrdiff_t)rs);   // row z - T
    const unsigned base = (unsigned)__cvta_generic_to_shared(ring) + lane * 16;
    int zf = zs;                                       // its first row
    auto fetch = [&](unsigned d) {
#pragma unroll
        for (int i = 0; i < kChunk; i++) {
            if (zf + i < zload) {
                cp_async16(d + i * 1024, pin + i * rs + at);
                cp_async16(d + i * 1024 + 512, pin + (i * rs + ls) + at);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        pin += kChunk * rs;
        zf += kChunk;
    };
#pragma unroll
    for (int i = 0; i < kRingChunks - 1; i++) fetch(base + i * kChunkBytes);

    StripRow wn[T], wc[T], ws[T];
#pragma unroll
    for (int k = 0; k < T; k++) wn[k] = wc[k] = StripRow{};
    unsigned rd = base, fr = base + (kRingChunks - 1) * kChunkBytes;   // chunk read now, chunk read before

    int z = zs;         // first row of the chunk
    auto arrived = [&] { asm volatile("cp.async.wait_group %0;" ::"n"(kRingChunks - 2) : "memory"); };
    auto next = [&] {   // to the next chunk; the slot of the one before this is filled again
        z += kChunk;
        pout += kChunk * rs;
        fetch(fr);
        fr = rd;
        rd += kChunkBytes;
        if (rd == base + kRingBytes) rd = base;
    };
    while (z < z1 + T) {
        // how far the rows from z on are plain: past the surface rows, before the bottom, clear
        // of the source patch, one set of coefficients over the T + 1 rows in flight, and for
        // the stores either all of their rows z - T in the band or none
        int clean = 0;
        if (z > T) {
            int e = nz - 1;
            if (has_src && z < sj0 + kPatch + T) e = min(e, z > sj0 ? 0 : sj0 + 1);
            e = min(e, z < z0 + T ? z0 + T : z1 + T);
            if (e >= z + kChunk) clean = min(e, __float_as_int(a.kp[z - T].pad0.x));
        }
        auto put = [&](bool st, int i, float4 um, float4 v) {
            if (st) {
                *reinterpret_cast<float4 *>(pout + i * rs + at) = um;
                *reinterpret_cast<float4 *>(pout + (i * rs + ls) + at) = v;
            }
        };
        if (z + kChunk <= clean) {
            const KP K = a.kp[z];
            const bool st = store && z >= z0 + T;
            auto plain = [&](auto sidec) {
                constexpr bool SIDE = decltype(sidec)::value;
                auto row = [&](int i, StripRow(&n)[T], StripRow(&cc)[T], StripRow(&so)[T]) {
                    float4 um = lds4(rd + i * 1024), v = lds4(rd + i * 1024 + 512);
#pragma unroll
                    for (int k = 0; k < T; k++) {
                        strip_feed(so[k], v, um, K.a);
                        v = strip_update(K, n[k].va, n[k].vb, n[k].da, n[k].db, cc[k], so[k]);
                        if (SIDE) strip_side(K.c, cc[k], kind, v);
                        um = make_float4(cc[k].ca.x, cc[k].ca.y, cc[k].cb.x, cc[k].cb.y);
                    }
                    put(st, i, um, v);
                };
#pragma unroll 1
                do {
                    arrived();
                    row(0, wn, wc, ws);
                    row(1, wc, ws, wn);
                    row(2, ws, wn, wc);
                    next();
                } while (z + kChunk <= clean);
            };
            if (side)
                plain(std::true_type{});
            else
                plain(std::false_type{});
#pragma unroll
            for (int k = 0; k < T; k++) wn[k].ca = wn[k].cb = make_float2(0.0f, 0.0f);   // not read from here on
        } else {
            // receiver samples of a level from its surface row u
            auto sample = [&](int level, float4 u) {
                float *trace = a.trace + ((size_t)s * g.nlev + level) * g.nrec * 2;
                for (int r0 = 0; r0 < g.nrec; r0 += 32) {
                    const int r = r0 + lane;
                    const int x = r < g.nrec ? a.rec[r] : -1;
                    const int from = ((x - (x0 - H)) >> 1) & 31;
                    const float2 ua = shfl2(make_float2(u.x, u.y), from), ub = shfl2(make_float2(u.z, u.w), from);
                    if (x >= x0 && x < x0 + W) *reinterpret_cast<float2 *>(trace + r * 2) = (x & 1) ? ub : ua;
                }
            };
            // coefficients of the rows z - T .. z + 2 in flight, one 16-byte piece a lane
            static_assert(T + kChunk <= 8, "eight rows of coefficients");
            const unsigned kb = base - lane * 16 + kRingBytes;
            __syncwarp();
            sts4(kb + lane * 16, reinterpret_cast<const float4 *>(a.kp + min(max(z - T + (lane >> 2), 0), nz - 1))[lane & 3]);
            __syncwarp();
            arrived();
#pragma unroll 1
            for (int i = 0; i < kChunk; i++) {
                float4 um = lds4(rd + i * 1024), v = lds4(rd + i * 1024 + 512);
                if (z + i == 0) sample(a.m, v);
#pragma unroll
                for (int k = 0; k < T; k++) {
                    const int r = z + i - k - 1;   // row r + 1 enters the step, row r is completed
                    const unsigned kr = kb + (unsigned)(i - k - 1 + T) * (unsigned)sizeof(KP);   // row r
                    strip_feed(ws[k], v, um, ring_coef(kr + (unsigned)sizeof(KP)).a);
                    float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (r >= 0 && r < nz) {
                        const KP Kr = ring_coef(kr);
                        const bool top = r == 0;   // no north differences, cross terms on the row itself
                        const float2 zero = make_float2(0.0f, 0.0f);
                        u = strip_update(Kr, top ? zero : wn[k].va, top ? zero : wn[k].vb,
                                         top ? wc[k].da : wn[k].da, top ? wc[k].db : wn[k].db, wc[k], ws[k]);
                        if (r == nz - 1) {
                            u.x = absorb(wc[k].ca.x, wn[k].ca.x, Kr.c.y);
                            u.y = absorb(wc[k].ca.y, wn[k].ca.y, Kr.c.x);
                            u.z = absorb(wc[k].cb.x, wn[k].cb.x, Kr.c.y);
                            u.w = absorb(wc[k].cb.y, wn[k].cb.y, Kr.c.x);
                        }
                        if (side) strip_side(Kr.c, wc[k], kind, u);
                        const int b = r - sj0;
                        if (has_src && (unsigned)b < (unsigned)kPatch) {
                            const int ia = c - si0, ib = c + 1 - si0;
                            const float f = a.stf[(size_t)s * g.nsteps + a.m + k];
                            if ((unsigned)ia < (unsigned)kPatch) {
                                u.x = add_force(u.x, f, src->wx[b * kPatch + ia]);
                                u.y = add_force(u.y, f, src->wz[b * kPatch + ia]);
                            }
                            if (c + 1 < g.nx && (unsigned)ib < (unsigned)kPatch) {
                                u.z = add_force(u.z, f, src->wx[b * kPatch + ib]);
                                u.w = add_force(u.w, f, src->wz[b * kPatch + ib]);
                            }
                        }
                        if (top && z0 == 0 && (k + 1 < T || a.last)) sample(a.m + k + 1, u);
                    }
                    um = make_float4(wc[k].ca.x, wc[k].ca.y, wc[k].cb.x, wc[k].cb.y);
                    v = u;
                    wn[k] = wc[k];
                    wc[k] = ws[k];
                }
                put(store && z + i >= z0 + T && z + i < z1 + T, i, um, v);
            }
            next();
        }
    }
}

// The rows' coefficients as (x, z) pairs, the form the packed update reads, each with the
// end of the run of rows that share its coefficients (an int in pad0.x, capped).
__global__ void k_pack_kp(const FacCoef<float> *__restrict__ fac, int nz, KP *__restrict__ kp)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nz) return;
    KP k = pack_coef(fac[j]);
    int e = j + 1;
    while (e < nz && e - j < kRunCap && kp_equal(k, pack_coef(fac[e]))) e++;
    k.pad0.x = __int_as_float(e);
    kp[j] = k;
}

// ---------------------------------------------------------------- host side

void launch_pack_kp(const oed_ctx *ctx, cudaStream_t st)
{
    if (!ctx->d_kp) return;
    k_pack_kp<<<(ctx->g.nz + 127) / 128, 128, 0, st>>>((const FacCoef<float> *)ctx->d_fac, ctx->g.nz,
                                                       (KP *)ctx->d_kp);
}

int strip_prepare(oed_ctx *ctx)
{
    int dev = 0, nsm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_strip<kStripSteps>, 32, kStripSmem) != cudaSuccess ||
        per_sm < 1)
        return 0;
    ctx->strip_sms = nsm;
    return nsm;
}

template <int T>
static cudaError_t strip_pass(StripArgs a, int nsm, cudaStream_t st)
{
    constexpr int W = 64 - 2 * ((T + 1) / 2 * 2);
    a.nstrip = (a.g.nx + W - 1) / W;
    // bands: more of them fill the chip when there are few strips, but each costs about 22 rows
    // more (2 T rows computed twice, its start).  Blocks run in waves of the warps that the chip
    // holds; the last, partly filled one costs as much as the others.  A fit to 1 to 16 bands on
    // nine batches (801x401, 1601x801, 701x351, 501x501; 7 to 105 solves): the rule's choice is
    // 0.2% slower than the best on average.  Against a wave's cost spread over its blocks, Gcell-upd/s:
    // 28 solves of 801x401 443 -> 476, 49 of 701x351 492 -> 512, 56 of 801x401 543 -> 559, 7 of
    // 1601x801 519 -> 535.
    const double strips = (double)a.nsolve * a.nstrip;
    double best = 0.0;
    for (int nb = 1; nb <= 64 && a.g.nz / nb >= 4 * T; nb++) {
        const double waves = std::ceil(strips * nb / (nsm * kStripWarps));
        const double cost = waves * ((double)a.g.nz / nb + 22.0);
        if (nb == 1 || cost < best) {
            best = cost;
            a.nband = nb;
        }
    }
    const long long blocks = (long long)a.nsolve * a.nstrip * a.nband;
    if (blocks > 2147483647LL) return cudaErrorInvalidValue;
    k_strip<T><<<(unsigned)blocks, 32, kStripSmem, st>>>(a);
    return cudaSuccess;
}

// nsteps (or nsteps_override) steps of nsolve solves: passes over the two buffers (d_u0, d_u1)
// and (d_u2, d_u3) in alternation, all in the strip layout, the last ones shorter when the
// count asks for it.  Every level is sampled at the receivers, the last one too.
// The caller zeroes the buffers (strip_stride floats per solve and level).
cudaError_t launch_steps_strip(const oed_ctx *ctx, int nsolve, cudaStream_t st, cudaEvent_t ev0, cudaEvent_t ev1,
                               int nsteps_override)
{
    const Geometry &g = ctx->g;
    if (ctx->strip_sms < 1 || !ctx->d_u2 || !ctx->d_kp) return cudaErrorInvalidConfiguration;
    float *pair[2] = {(float *)ctx->d_u0, (float *)ctx->d_u2};   // d_u1, d_u3 follow their partners
    StripArgs a;
    a.kp = (const KP *)ctx->d_kp;
    a.src = (const SourceDesc<float> *)ctx->d_src;
    a.stf = (const float *)ctx->d_stf;
    a.trace = (float *)ctx->d_trace;
    a.rec = ctx->d_rec;
    a.g = g;
    a.nsolve = nsolve;
    a.nband = 1;
    a.sq = strip_sq(g);
    a.pst = 2 * strip_stride(g);
    const int nsteps = (nsteps_override > 0 && nsteps_override < g.nsteps) ? nsteps_override : g.nsteps;
    tma_record(ev0, st);
    cudaError_t e = cudaSuccess;
    for (int m = 0, pr = 0; m < nsteps && e == cudaSuccess; pr ^= 1) {
        const int left = nsteps - m;
        const int T = left < kStripSteps ? left : kStripSteps;
        a.in = pair[pr];
        a.out = pair[pr ^ 1];
        a.m = m;
        a.last = T == left && nsteps == g.nsteps;   // (a probe's last pass stores like the others)
        e = T == 4   ? strip_pass<4>(a, ctx->strip_sms, st)
            : T == 3 ? strip_pass<3>(a, ctx->strip_sms, st)
            : T == 2 ? strip_pass<2>(a, ctx->strip_sms, st)
                     : strip_pass<1>(a, ctx->strip_sms, st);
        m += T;
    }
    tma_record(ev1, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace oed
