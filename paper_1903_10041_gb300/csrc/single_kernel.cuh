// Persistent single-instance solve kernel: the whole ADMM loop of App. A on
// the device, one cooperative launch per solve.
//
// Work split.  The columns (j, k) are taken in j-major order and cut into
// one contiguous range per CTA of (nearly) equal length: either every row j
// cut into the same number of pieces (no CTA straddles two rows), or, for
// short rows, flat chunks of `chunk` columns, where the row segments of one
// CTA are worked on side by side by disjoint warps (or, when the segments are
// long, one after another by all warps).  The thread that owns a column
// updates all m sources of it in registers (step (a) sweeps the sources in
// order, so the Gauss-Seidel sums over l != i stay local), then steps (e)
// and (f) for that column.  The per-(i, j) sums over k that steps (b) and
// (d) and the residuals need are segmented reductions: each CTA reduces each
// row segment it owns (warp shuffles, then shared memory) into a partial
// record; after one grid barrier every CTA adds the records of each row in
// a fixed order and runs the per-(i, j) scalar steps (b), (c), (d), (g),
// (h), (i), the residuals and the stop test redundantly, so all CTAs hold
// identical scalars and take the same stop decision without a second
// barrier.  Partial records are double-buffered by iteration parity.
//
// Identities used (derived from steps (b) and (g)): after every iteration
// lambda^(i,j) is constant over k and z_k = g_k(x_k) + zeta with
// zeta = lambda_new - lambda_old, so theta_k = z_k + lambda =
// g_k(x~_k) + zeta + lambda needs no per-element z or lambda.  The zero start
// (z = 0, the paper's iteration from zeros) is flagged `cold`, where
// theta = 0 instead.
//
// Small problems (template CL, single_shape): the CTAs are one thread-block
// cluster, each with one piece of one row; the records stay in shared memory,
// one hardware cluster barrier (380 cycles; __syncthreads for one CTA) takes
// the grid barrier's place (2400) and the scalar phase reads the records
// through distributed shared memory instead of L2.
//
// Precision variants (template PREC):
//   ADMM_FP64             one column per thread, dense column space (rs = n);
//   ADMM_MIXED            FP32 storage and element work on column pairs
//                         (float2, paired FP32 instructions) over a padded
//                         column space (rs = ld); the
//                         capacity sums over k are accumulated per thread in
//                         float-float (about 48 bits) and reduced in FP64; the
//                         column state s, mu is stored and updated in
//                         float-float; the cubic's branch is decided as FP64
//                         would decide it;
//   ADMM_MIXED_FP64CUBIC  as ADMM_MIXED with the cubic step in FP64.
// The per-(i, j) scalar steps, residuals and stop test are FP64 in all three.
#pragma once
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "mixed_elem.cuh"
#include "quartic64.cuh"

namespace admm_impl {

namespace {

struct Sm {
    double *lam, *zeta, *h, *p, *nu, *x1, *rho, *flags; // mirror of the scalar state
    double *x0;   // [mq]
    double *x1n;  // [kMaxM]
    double *red;  // [kSingleWarpsMax][kMaxM][3]
    double *mx;   // [kSingleWarpsMax][8]
    double *bc;   // [16] broadcast: [0] r, [1] sigma, [2] adaptation factor, [3] kappa, [4..6] rho_3/2, rho_4/2,
                  //      rho_1/2, [7] int flags of a check (converged, penalties changed), [8..9] floats rho_1,
                  //      rho_3, rho_4, rho_1/2
    int *segof;   // [kSingleWarpsMax] segment (within the pass) of each warp
    int *rfirst;  // [q] first CTA whose columns touch row j
    int *rcnt;    // [q] how many do
    double *crec; // [2][kMaxM][4] this CTA's record (cluster variant)
    double *ccm;  // [2][2] its column maxima (cluster variant)
    float *uoff;  // [mq] zeta + lambda in FP32 (mixed variants)
    float *x1nu;  // [mq] x1 + nu in FP32 (mixed variants)
    double *zl;   // [mq] zeta + lambda (FP64 variant; the storage of uoff, x1nu)
};

// Bytes of the shared state carve() lays out, rounded up to 16: the rolling
// stage of the mixed kernels (m <= 4) starts there.
__host__ __device__ inline size_t single_carve_bytes(int m, int q)
{
    const int mq = m * q;
    const size_t b = sizeof(double) * ((size_t)scal_size(m, q) + mq + kMaxM + kSingleWarpsMax * kMaxM * 3 +
                                       kSingleWarpsMax * 8 + 16 + kSingleWarpsMax) +
                     sizeof(float) * 2 * (size_t)mq + sizeof(int) * 2 * (size_t)q +
                     sizeof(double) * (2 * kMaxM * 4 + 4);
    return (b + 15) / 16 * 16;
}

__device__ __forceinline__ Sm carve(double *base, int m, int q)
{
    const int mq = m * q;
    Sm s;
    s.lam = base;
    s.zeta = base + mq;
    s.h = base + 2 * mq;
    s.p = base + 3 * mq;
    s.nu = base + 4 * mq;
    s.x1 = base + 5 * mq;
    s.rho = s.x1 + m;
    s.flags = s.rho + 4;
    double *t = base + scal_size(m, q);
    s.x0 = t;
    t += mq;
    s.x1n = t;
    t += kMaxM;
    s.red = t;
    t += kSingleWarpsMax * kMaxM * 3;
    s.mx = t;
    t += kSingleWarpsMax * 8;
    s.bc = t;
    t += 16;
    s.segof = (int *)t;
    t += kSingleWarpsMax;
    s.uoff = (float *)t;
    s.x1nu = s.uoff + mq;
    s.zl = t;
    s.rfirst = (int *)(t + mq);
    s.rcnt = s.rfirst + q;
    s.crec = t + mq + q;
    s.ccm = s.crec + 2 * kMaxM * 4;
    return s;
}

// Per-iteration constants of the FP64 element update, the same in every thread.
struct Iter64 {
    double rho3h, rho4h, hr1, iq, iqh; // rho_3/2, rho_4/2, rho_1/2, 1/q, 1/(2q)
    float hr1f;
};

// ---------------------------------------------------------------------------
// FP64 phase 1: step (a) for all sources of column (j, k), then (e), (f).
// Bound by the FP64 pipe (64 cycles per warp instruction and scheduler), so
// what counts is the number of FP64-pipe instructions: per column 3m - 5 for
// the sums over the other sources (prefix of the new x, suffix of the old),
// 3 for rho_3 (s + y + mu)/2, 2 for (e), (f), and per element 3 for C and Dh
// and the root (elem_min64_seeded), 21 in all with losses and 7 without.
// Measured on n = 1000, m = 2, q = 50 (PHEV): 24.8 -> 16.7 us per iteration; n = 4099, m = 3, q = 7: 33.6 -> 23.3.
// (e), (f): with v = sum_i x - y - mu, s = max(0, v) and mu + s - sum_i x + y
// = max(0, -v), the same values as the literal sums to rounding.
// ---------------------------------------------------------------------------
template <int M>
__device__ __forceinline__ void column64(const SingleArgs &a, const Sm &sm, const Iter64 &ic, int j, int k, bool check,
                                         bool cold, double mu_div, double *gs, double *dmx, double *dmn,
                                         double &cm_r, double &cm_s, double *rec, int rstep)
{
    const int m = a.m, q = a.q, ld = a.ld;
    const double *F2 = (const double *)a.f2, *F1 = (const double *)a.f1;
    const double *G2 = (const double *)a.g2, *G1 = (const double *)a.g1, *G0 = (const double *)a.g0;
    const double *LO = (const double *)a.lo, *HI = (const double *)a.hi, *Y = (const double *)a.y;
    double *X = (double *)a.x, *Sv = (double *)a.s, *MU = (double *)a.mu;
    const bool jac = a.sweep == ADMM_JACOBI;

    double xt[M], suf[M]; // x~ and its sums over the sources after i
#pragma unroll
    for (int i = 0; i < M; ++i)
        if (i < m) xt[i] = X[((size_t)i * q + j) * ld + k];
    const size_t col = (size_t)j * ld + k;
    const double st = Sv[col], yv = Y[col];
    double mu = MU[col];
    if (__double_as_longlong(mu_div) != 0x3ff0000000000000ll) mu = mu / mu_div; // not 1.0
#pragma unroll
    for (int i = M - 2; i >= 0; --i)
        if (i + 1 < m) suf[i] = i + 2 < m ? xt[i + 1] + suf[i + 1] : xt[i + 1];
    const double rb = ic.rho3h * ((st + yv) + mu);

    double pre = 0.0, sx = 0.0, dx = 0.0; // sums of the x that step (a) uses, of the new x and of x - x~ so far
#pragma unroll
    for (int i = 0; i < M; ++i) {
        if (i < m) {
            const size_t e = ((size_t)i * a.cq + (size_t)j * a.cj) * ld + k; // coefficient element
            const double a2 = F2[e], a1 = F1[e], b2 = G2[e], b1 = G1[e];
            const int pr = i * q + j;
            const double others = i == 0 ? (m > 1 ? suf[0] : 0.0) : (i + 1 < m ? pre + suf[i] : pre);
            double C = fma(a2, ic.iq, ic.rho3h), Dh = fma(a1, ic.iqh, fma(ic.rho3h, others, -rb));
            if (k == 0) {
                C += ic.rho4h;
                Dh -= ic.rho4h * (sm.x1[i] + sm.nu[pr]);
            }
            const double lo = LO[(size_t)i * ld + k], hi = HI[(size_t)i * ld + k];
            double xn, gq = 0.0, gq_old = 0.0;
            // b2 = b1 = 0 (either sign of zero), tested on the integer pipes: no loss on this
            // element (g = beta_0), the terms in beta_2, beta_1 vanish
            if (((__double_as_longlong(b2) | __double_as_longlong(b1)) << 1) == 0) {
                xn = elem_min64_linear(C, Dh, lo, hi);
            } else {
                // u = theta - beta_0 (theta = z + lambda)
                const double t = fma(b2, xt[i], b1);
                const double u = cold ? -G0[e] : fma(t, xt[i], sm.zl[pr]);
                xn = elem_min64_seeded({b2, b1, u, C, Dh, ic.hr1}, ic.hr1f, lo, hi, a.xmin_mode);
                const double tn = fma(b2, xn, b1);
                gs[i] = fma(tn, xn, gs[i]);
                if (check) {
                    gq = tn * xn;
                    gq_old = t * xt[i];
                }
            }
            if (check) {
                // z_k - z~_k = D_k + (lambda_new - lambda - zeta); D_k = g(x) - g(x~),
                // or g(x) at the zero start where z~ = 0.
                const double dk = cold ? gq + G0[e] : gq - gq_old;
                dmx[i] = max_ord(dmx[i], dk);
                dmn[i] = min_ord(dmn[i], dk);
                dx += xn - xt[i];
            }
            sx = i == 0 ? xn : sx + xn;
            if (jac) pre = i == 0 ? xt[i] : pre + xt[i];
            else pre = sx;
            X[((size_t)i * q + j) * ld + k] = xn;
            if (k == 0) rec[i * rstep] = xn;
        }
    }
    const double v = (sx - yv) - mu;
    const bool pos = __double_as_longlong(v) > 0;
    const double sn = pos ? v : 0.0;             // (e)
    const double mun = pos ? 0.0 : -v;           // (f)
    if (check) {
        cm_r = max_ord(cm_r, fabs((sn - sx) + yv));
        cm_s = max_ord(cm_s, fabs((sn - st) - dx));
    }
    Sv[col] = sn;
    MU[col] = mun;
}

// Warp plan of one pass over the row segments jb..je (at most NWP rows, the
// CTA's warp count) of the chunk [c0, c1): segment s gets warps
// [W_s, W_s+1) with W_s = s + floor((NWP - ns) * (columns before s) /
// (columns in the pass)),
// at least one warp each and the rest in proportion to length, so the
// segments of a CTA run side by side.  The plan depends only on the launch
// shape, so it is the same in every iteration.
struct SegPlan {
    int j;          // row of this warp's segment
    int seg;        // its index within the pass (j - jb)
    int lw, nw;     // this warp's index among the segment's warps, their count
    int kb, ke;     // the segment's columns k of row j
};

template <int NWP>
__device__ __forceinline__ SegPlan seg_plan(int64_t c0, int64_t c1, int64_t rs, int jb, int je, int w)
{
    SegPlan p{};
    const int ns = je - jb + 1;
    if (ns == 1) {
        p.j = jb;
        p.lw = w;
        p.nw = NWP;
    } else {
        const int64_t b0 = max(c0, (int64_t)jb * rs), b1 = min(c1, (int64_t)(je + 1) * rs);
        const float scale = (float)(NWP - ns) / (float)(b1 - b0);
        int wlo = 0, whi = NWP;
        for (int t = 0; t < ns; ++t) {
            const int64_t before = max(c0, (int64_t)(jb + t) * rs) - b0;
            const int ws = t + (int)floorf(scale * (float)before);
            if (ws <= w) {
                p.seg = t;
                wlo = ws;
            } else {
                whi = min(whi, ws);
            }
        }
        p.lw = w - wlo;
        p.nw = whi - wlo;
        p.j = jb + p.seg;
    }
    const int64_t r0 = (int64_t)p.j * rs;
    p.kb = (int)(max(c0, r0) - r0);
    p.ke = (int)(min(c1, r0 + rs) - r0);
    return p;
}

// Rows per pass for the chunk [c0, c1) spanning rows jf..jl: all of them
// side by side (NWP per pass), or one at a time on all warps when that
// takes fewer rounds of column work (long segments, where splitting the
// warps unevenly costs more than the extra reduction barrier, counted as a
// quarter round).  unit: columns per thread and round.
template <int NWP>
__device__ __noinline__ int pass_rows(int64_t c0, int64_t c1, int64_t rs, int jf, int jl, int unit)
{
    const int ns = jl - jf + 1;
    if (ns == 1 || ns > NWP) return NWP;
    int64_t conc = 0, seq4 = (int64_t)(ns - 1); // seq in quarter rounds
    for (int w = 0; w < NWP; ++w) {
        const SegPlan sp = seg_plan<NWP>(c0, c1, rs, jf, jl, w);
        if (sp.lw != 0) continue;
        const int64_t v = (sp.ke - sp.kb + unit - 1) / unit;
        conc = max(conc, (v + 32 * sp.nw - 1) / (32 * sp.nw));
        seq4 += 4 * ((v + 32 * NWP - 1) / (32 * NWP));
    }
    return 4 * conc <= seq4 ? NWP : 1;
}

// Columns [c0, c1) of this CTA.
__device__ __forceinline__ void cta_columns(const SingleArgs &a, int unit, int64_t &c0, int64_t &c1)
{
    if (a.pieces > 0) {
        const int j = (int)blockIdx.x / a.pieces, t = (int)blockIdx.x - j * a.pieces;
        c0 = (int64_t)j * a.rs + piece_bound(t, a.rs, a.pieces, unit);
        c1 = (int64_t)j * a.rs + piece_bound(t + 1, a.rs, a.pieces, unit);
    } else {
        c0 = (int64_t)blockIdx.x * a.chunk;
        c1 = min(c0 + a.chunk, a.ncols);
    }
}

// CTAs whose columns touch row j: the first and how many.
__device__ __forceinline__ void row_ctas(const SingleArgs &a, int j, int &first, int &cnt)
{
    if (a.pieces > 0) {
        first = j * a.pieces;
        cnt = a.pieces;
        return;
    }
    const int64_t rbeg = (int64_t)j * a.rs;
    first = (int)(rbeg / a.chunk);
    cnt = (int)((rbeg + a.rs - 1) / a.chunk) - first + 1;
}

// Records of one iteration parity: planes of S = sum g, max D and min D,
// each [q][m][nbp] with a pair's records contiguous in the CTAs touching the
// row, then x at k = 0 as [m][q].  The scalar phase of every CTA reads them
// all, so what counts is the number of 32-byte sectors: with the records of
// one CTA contiguous instead, each sector held one wanted value (n = 1e5, m =
// 4, q = 20: 79.5 -> 76.1 us per iteration; n = 1000, q = 50 PHEV mixed 7.5 ->
// 6.1, FP64 12.2 -> 11.4; n = 10007, m = 6, q = 11: 23.5 -> 21.5).
struct Recs {
    double *s;      // plane of S; the others follow at + plane
    size_t plane;   // q m nbp
    int m, nbp;
    __device__ __forceinline__ size_t at(int i, int j, int t) const { return ((size_t)j * m + i) * nbp + t; }
    __device__ __forceinline__ double *x0() const { return s + 3 * plane; }
};
__device__ __forceinline__ Recs records(const SingleArgs &a, int par)
{
    Recs r;
    r.m = a.m;
    r.nbp = record_pad(a.nbmax);
    r.plane = (size_t)a.q * a.m * r.nbp;
    r.s = a.part + (size_t)par * (3 * r.plane + record_pad(a.q * a.m)); // 32-byte aligned, as the pairs are
    return r;
}
// Writes this CTA's record of (row j, source i); lo, hi on check iterations.
template <bool CL>
__device__ __forceinline__ void put_record(const SingleArgs &a, const Sm &sm, int par, int j, int i, double v, bool check,
                                           double hi, double lo)
{
    if constexpr (CL) {
        double *rec = sm.crec + (par * kMaxM + i) * 4;
        rec[0] = v;
        rec[1] = hi;
        rec[2] = lo;
    } else {
        const Recs r = records(a, par);
        const size_t e = r.at(i, j, (int)blockIdx.x - sm.rfirst[j]);
        r.s[e] = v;
        if (check) {
            r.s[r.plane + e] = hi;
            r.s[2 * r.plane + e] = lo;
        }
    }
}

// Reduction of one pass of row segments into their partial records, and (on
// check iterations) of the CTA's column maxima: warp sums of all sources at
// once by shuffles, then per (segment, source) the sum over that segment's
// warps by the 16 lanes of a half warp, in a fixed order.
template <int M, int NWP, bool CL>
__device__ __forceinline__ void flush_segments(const SingleArgs &a, int par, int jb, int ns, double *gs, double *dmx,
                                               double *dmn, double cm_r, double cm_s, bool check, int m,
                                               const SegPlan &sp, const Sm &sm)
{
    static_assert(NWP <= 16, "a half warp covers the warps");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto add = [](double k, double s, int o) { return k + __shfl_xor_sync(0xffffffffu, s, o); };
    auto mx = [](double k, double s, int o) { return max_ord(k, __shfl_xor_sync(0xffffffffu, s, o)); };
    auto mn = [](double k, double s, int o) { return min_ord(k, __shfl_xor_sync(0xffffffffu, s, o)); };
    const int src = slot_of<M>(lane);
    const double v = warp_many<M>(gs, add);
    if (lane % (32 / M) == 0) sm.red[(w * kMaxM + src) * 3] = v;
    if (check) {
        const double hi = warp_many<M>(dmx, mx), lo = warp_many<M>(dmn, mn);
        cm_r = warp_max_nonneg(cm_r);
        cm_s = warp_max_nonneg(cm_s);
        if (lane % (32 / M) == 0) {
            sm.red[(w * kMaxM + src) * 3 + 1] = hi;
            sm.red[(w * kMaxM + src) * 3 + 2] = lo;
        }
        if (lane == 0) {
            sm.mx[w * 8] = cm_r;
            sm.mx[w * 8 + 1] = cm_s;
        }
    }
    if (lane == 0) sm.segof[w] = sp.seg;
    __syncthreads();
    const int hl = lane & 15;
    for (int t = 2 * w + (lane >> 4); t - (lane >> 4) < ns * m; t += 2 * NWP) { // a half warp per (segment, source)
        const int sg = t / m, i = t - sg * m;
        const bool in = t < ns * m && hl < NWP && sm.segof[hl < NWP ? hl : 0] == sg;
        double r = in ? sm.red[(hl * kMaxM + i) * 3] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        double hi = 0.0, lo = 0.0;
        if (check) {
            hi = in ? sm.red[(hl * kMaxM + i) * 3 + 1] : -INFINITY;
            lo = in ? sm.red[(hl * kMaxM + i) * 3 + 2] : INFINITY;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                hi = mx(hi, hi, o);
                lo = mn(lo, lo, o);
            }
        }
        if (hl == 0 && t < ns * m) {
            put_record<CL>(a, sm, par, jb + sg, i, r, check, hi, lo);
        }
    }
}

// Mixed variant, on the FP32 pipes: float-float sums and FP32 max / min in
// a fixed order; only the finished records are converted to FP64.
template <int M, int NWP, bool CL>
__device__ __forceinline__ void flush_segments32(const SingleArgs &a, int par, int jb, int ns, const float2 *ghi,
                                                 const float2 *glo, float *fmx, float *fmn, float cm_r, float cm_s,
                                                 bool check, int m, const SegPlan &sp, const Sm &sm)
{
    float *red = (float *)sm.red; // [NWP][kMaxM][4] floats
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto add = [](FF k, FF s, int o) {
        return ff_add(k, FF{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o)});
    };
    auto mx = [](float k, float s, int o) { return fmaxf(k, __shfl_xor_sync(0xffffffffu, s, o)); };
    auto mn = [](float k, float s, int o) { return fminf(k, __shfl_xor_sync(0xffffffffu, s, o)); };
    FF g[M];
#pragma unroll
    for (int i = 0; i < M; ++i) g[i] = lanes_sum(ghi[i], glo[i]);
    const int src = slot_of<M>(lane);
    const FF v = warp_many<M>(g, add);
    float *rw = red + (w * kMaxM + src) * 4;
    if (lane % (32 / M) == 0) {
        rw[0] = v.hi;
        rw[1] = v.lo;
    }
    if (check) {
        const float hi = warp_many<M>(fmx, mx), lo = warp_many<M>(fmn, mn);
        cm_r = warp_max_nonneg(cm_r);
        cm_s = warp_max_nonneg(cm_s);
        if (lane % (32 / M) == 0) {
            rw[2] = hi;
            rw[3] = lo;
        }
        if (lane == 0) {
            sm.mx[w * 8] = f32_to_f64_nan(cm_r);
            sm.mx[w * 8 + 1] = f32_to_f64_nan(cm_s);
        }
    }
    if (lane == 0) sm.segof[w] = sp.seg;
    __syncthreads();
    const int hl = lane & 15;
    for (int t = 2 * w + (lane >> 4); t - (lane >> 4) < ns * m; t += 2 * NWP) { // a half warp per (segment, source)
        const int sg = t / m, i = t - sg * m;
        const bool in = t < ns * m && hl < NWP && sm.segof[hl < NWP ? hl : 0] == sg;
        const float *rr = red + (hl * kMaxM + i) * 4;
        FF r = in ? FF{rr[0], rr[1]} : FF{0.0f, 0.0f};
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) r = add(r, r, o);
        float hi = 0.0f, lo = 0.0f;
        if (check) {
            hi = in ? rr[2] : -INFINITY;
            lo = in ? rr[3] : INFINITY;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                hi = mx(hi, hi, o);
                lo = mn(lo, lo, o);
            }
        }
        if (hl == 0 && t < ns * m) {
            put_record<CL>(a, sm, par, jb + sg, i, f32_to_f64_nan(r.hi) + f32_to_f64_nan(r.lo), check,
                           f32_to_f64_nan(hi), f32_to_f64_nan(lo));
        }
    }
}

// The values derived from the penalties that the next iterations read (by one thread).
__device__ __forceinline__ void derive_penalties(const Sm &sm, int n)
{
    const double r1 = sm.rho[0], r2 = sm.rho[1], r3 = sm.rho[2], r4 = sm.rho[3];
    sm.bc[3] = r2 / fma((double)n, r2, r1); // kappa of step (b)
    sm.bc[4] = 0.5 * r3;
    sm.bc[5] = 0.5 * r4;
    sm.bc[6] = 0.5 * r1;
    float *f = (float *)(sm.bc + 8);
    f[0] = (float)r1;
    f[1] = (float)r3;
    f[2] = (float)r4;
    f[3] = (float)(0.5 * r1);
}

// NT: threads of a CTA, one CTA per SM.  FP64 takes 384 (168 registers).  The
// mixed kernel takes 256 (255 registers, at most 32 bytes spilled) where one pass
// covers the columns, and 384 (168) where a thread has several: two CTAs of 256
// at 128 registers keep a third more warps but spill about 500 bytes a thread, and
// the reloads come back through an L1 that the stage's copies sweep (n = 1e5, m = 4,
// q = 20: 76.1 -> 66.7 us per iteration; 320 threads 72.3, 448 79.5; n = 10007, m =
// 6, q = 11: 21.5 -> 18.8).  384 spill 156 bytes stored and 88 loaded at M = 4, 360 and
// 392 at M = 8, none at M = 2.
template <int M, int PREC, int NT, bool CL>
__global__ void __launch_bounds__(NT, 1) single_kernel(SingleArgs a)
{
    namespace cg = cooperative_groups;
    constexpr int NWP = NT / 32;
    extern __shared__ double smem[];
    constexpr bool MIXED = PREC != ADMM_FP64;
    constexpr int VW = kMixedVW;
    const int m = a.m, q = a.q, n = a.n, mq = m * q, rs = a.rs;
    const Sm sm = carve(smem, m, q);
    auto team_sync = [&]() {
        if (a.grid > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    for (int t = threadIdx.x; t < scal_size(m, q); t += NT) smem[t] = a.scal[t];
    __syncthreads();
    for (int pr = threadIdx.x; pr < mq; pr += NT) {
        if constexpr (MIXED) {
            sm.uoff[pr] = (float)(sm.zeta[pr] + sm.lam[pr]);
            sm.x1nu[pr] = (float)(sm.x1[pr / q] + sm.nu[pr]);
        } else {
            sm.zl[pr] = sm.zeta[pr] + sm.lam[pr];
        }
    }
    for (int j = threadIdx.x; j < q; j += NT) row_ctas(a, j, sm.rfirst[j], sm.rcnt[j]);
    if (threadIdx.x == 0) derive_penalties(sm, n);
    const double iq64 = 1.0 / (double)q, nd = (double)n;
    const float iq = 1.0f / (float)q;
    // lanes that share the records of one pair in the scalar phase
    int gsh = 0;
    while ((CL ? 2 : 4) << gsh <= a.nbmax && gsh < 5 && (mq << (gsh + 1)) <= NT) ++gsh;
    const int G = 1 << gsh;
    bool cold = sm.flags[0] != 0.0;
    double mu_div = sm.flags[1];
    __syncthreads();

    int64_t c0, c1;
    cta_columns(a, MIXED ? VW : 1, c0, c1);
    const int jf = (int)(c0 / rs), jl = (int)((c1 - 1) / rs);
    const int prows = pass_rows<NWP>(c0, c1, rs, jf, jl, MIXED ? VW : 1);
    const SegPlan sp0 = seg_plan<NWP>(c0, c1, rs, jf, min(jl, jf + prows - 1), threadIdx.x >> 5);
    unsigned nbar = 0;
    unsigned esc = 0;
    bool ok = true, conv = false;
    int it, ncheck = a.check_every; // iterations up to the next check
    double res[7] = {0, 0, 0, 0, 0, 0, 0}; // r1 r2 r3 r4 s1 s2 s3 (unscaled s)
    double r_last = INFINITY, s_last = INFINITY;
    const float *fp = (const float *)(sm.bc + 8);

    for (it = 1; it <= a.max_iter; ++it) {
        const bool check = --ncheck == 0 || it == a.max_iter;
        if (ncheck == 0) ncheck = a.check_every;
        const int par = it & 1;
        double cm_r = 0.0, cm_s = 0.0;
        float fcr = 0.0f, fcs = 0.0f;
        Iter64 ic;
        if constexpr (!MIXED) {
            ic.rho3h = sm.bc[4];
            ic.rho4h = sm.bc[5];
            ic.hr1 = sm.bc[6];
            ic.hr1f = fp[3];
            ic.iq = iq64;
            ic.iqh = 0.5 * iq64;
        }

        // ---- phase 1: element updates and segment partials --------------
        // The rows j the chunk touches are taken prows at a time; within a
        // pass every row segment gets its own warps, so its segments run
        // concurrently and one reduction barrier closes them all.
        for (int jb = jf; jb <= jl; jb += prows) {
            const int ns = min(jl, jb + prows - 1) - jb + 1;
            if (jb > jf) __syncthreads(); // the previous pass has been reduced
            const SegPlan sp = jb == jf ? sp0 : seg_plan<NWP>(c0, c1, rs, jb, jb + ns - 1, threadIdx.x >> 5);
            const int j = sp.j;
            // x of source i at k = 0 goes to rec[i * rstep]
            double *rec = CL ? sm.crec + par * kMaxM * 4 + 3 : records(a, par).x0() + j;
            const int rstep = CL ? 4 : q;
            // row-local column range of the segment (k), and this thread's start and step
            const int kb = sp.kb, ke = sp.ke;
            const int first = sp.lw * 32 + (threadIdx.x & 31), stride = sp.nw * 32;
            if constexpr (!MIXED) {
                double gs[M], dmx[M], dmn[M];
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    gs[i] = 0.0;
                    dmx[i] = -INFINITY;
                    dmn[i] = INFINITY;
                }
                for (int k = kb + first; k < ke; k += stride)
                    column64<M>(a, sm, ic, j, k, check, cold, mu_div, gs, dmx, dmn, cm_r, cm_s, rec, rstep);
                flush_segments<M, NWP, CL>(a, par, jb, ns, gs, dmx, dmn, cm_r, cm_s, check, m, sp, sm);
            } else {
                float2 ghi[M], glo[M]; // per-lane capacity sums of the column pairs
                float fmx[M], fmn[M];
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    ghi[i] = make_float2(0.0f, 0.0f);
                    glo[i] = make_float2(0.0f, 0.0f);
                    fmx[i] = -INFINITY;
                    fmn[i] = INFINITY;
                }
                const float rho1 = fp[0], rho3 = fp[1], rho4 = fp[2], mudf = f64_to_f32_int(mu_div);
                const ElemF32 ea = {(const float *)a.f2, (const float *)a.f1, (const float *)a.g2,
                                    (const float *)a.g1, (const float *)a.g0, (const float *)a.lo,
                                    (const float *)a.hi, (const float *)a.y,  (float *)a.x,
                                    (float *)a.s,        (float *)a.mu,       (float *)a.s_lo,
                                    (float *)a.mu_lo,    a.n,                 a.m,
                                    a.q,                 a.ld,                a.sweep,
                                    a.xmin_mode,         a.cq,                a.cj,
                                    a.dbg};
                const int kn = min(ke, n); // padding columns k >= n are skipped
                const bool tiny_c = tiny_rho3(rho3);
                // PLAIN: not a check iteration, not cold, no pending mu divisor (nine iterations in
                // ten), a normal rho_3, with those branches and their registers compiled out of the
                // loop (n = 1e5, m = 4, q = 20: 91.3 -> 80.2 us per iteration).  Not for M = 8, where
                // two copies spill more than the branches cost (m = 6: 23.0 -> 25.9).
                auto columns = [&](auto plain) {
                    constexpr bool PLAIN = decltype(plain)::value;
                    const bool chk = !PLAIN && check, cld = !PLAIN && cold;
                    const float mud = PLAIN ? 1.0f : mudf;
                    if constexpr (M <= 4) {
                        // every input through the warp's rolling cp.async stage (each CTA keeps its
                        // columns for the whole launch, so its L1 never holds another SM's lines)
                        float2 *stw = (float2 *)((char *)smem + single_carve_bytes(m, q)) +
                                      (size_t)(threadIdx.x >> 5) * roll_slots<M>() * 32 + (threadIdx.x & 31);
                        const int k00 = kb + first * VW;
                        roll_prologue<M>(ea, j, k00, k00 < kn, stw);
                        for (int k0 = k00; k0 < kn; k0 += stride * VW) {
                            const int k0n = k0 + stride * VW < kn ? k0 + stride * VW : -1;
                            vec32<M, VW, PREC == ADMM_MIXED_FP64CUBIC, STAGE_ROLL>(
                                ea, sm.uoff, sm.x1nu, j, k0, chk, cld, PLAIN, mud, rho1, rho3, rho4, iq, ghi, glo,
                                fmx, fmn, fcr, fcs, esc, rec, rstep, stw, k0n);
                        }
                        cp_async_wait0();
                    } else {
                        for (int k0 = kb + first * VW; k0 < kn; k0 += stride * VW) {
                            if constexpr (NT > kBlock) // several vectors per thread: fetch the next one into L2
                                if (k0 + stride * VW < kn) prefetch_vec32<M>(ea, j, k0 + stride * VW, cld);
                            vec32<M, VW, PREC == ADMM_MIXED_FP64CUBIC>(ea, sm.uoff, sm.x1nu, j, k0, chk, cld,
                                                                       PLAIN, mud, rho1, rho3, rho4, iq, ghi, glo,
                                                                       fmx, fmn, fcr, fcs, esc, rec, rstep);
                        }
                    }
                };
                if (M > 4 || check || cold || mudf != 1.0f || tiny_c) columns(std::false_type{});
                else columns(std::true_type{});
                flush_segments32<M, NWP, CL>(a, par, jb, ns, ghi, glo, fmx, fmn, fcr, fcs, check, m, sp, sm);
            }
        }
        if (check && threadIdx.x == 0) { // the CTA's column maxima (the last pass holds the largest so far)
            double v0 = 0.0, v1 = 0.0;
            for (int w = 0; w < NWP; ++w) {
                v0 = max_nonneg(v0, sm.mx[w * 8]);
                v1 = max_nonneg(v1, sm.mx[w * 8 + 1]);
            }
            double *cm = CL ? sm.ccm + par * 2 : a.cpart + ((size_t)par * a.grid + blockIdx.x) * 4;
            cm[0] = v0;
            cm[1] = v1;
        }
        if constexpr (CL) {
            team_sync();
        } else {
            ++nbar;
            if (!grid_barrier(a.bar, nbar * (unsigned)a.grid, a.status, a.spin_ns, ADMM_ETIMEOUT)) {
                ok = false;
                break;
            }
        }
        cold = false;
        mu_div = 1.0; // the pending mu rescale has been applied

        // ---- phase 2: per-(i, j) scalar steps, redundantly in every CTA ---
        // Two independent chains on different warps: the mean over j of step (c)
        // with (h), one warp per source from the last warp down, and steps (b),
        // (d), (g), (i) per pair, G lanes sharing a pair's records; one CTA barrier
        // closes both.  Bound by latency: the records' L2 round trip and a chain
        // of about 15 FP64 instructions of 64 cycles.  With the reductions above,
        // per iteration (us): n = 1000, q = 50 PHEV FP64 16.7 -> 12.1, mixed
        // 10.0 -> 7.7; n = 4099, m = 3, q = 7 FP64 23.3 -> 15.2; n = 10007, m = 6,
        // q = 11 mixed 31.4 -> 24.0; n = 100 FP64 1.8x.
        const Recs rr = records(a, par);
        // the cluster variant's records: CTA j * pieces + t holds record t of row j
        auto remote = [&](int j, int t, int i, int e) {
            const double *p = sm.crec + (par * kMaxM + i) * 4 + e;
            return a.grid == 1 ? p : (const double *)cg::this_cluster().map_shared_rank((double *)p, j * a.pieces + t);
        };
        double r1m = 0.0, r2m = 0.0, r3m = 0.0, r4m = 0.0, s1m = 0.0, s2m = 0.0, s3m = 0.0;
        {
            const int lane = threadIdx.x & 31;
            for (int i = NWP - 1 - (int)(threadIdx.x >> 5); i < m; i += NWP) {
                double sum = 0.0;
                for (int j = lane; j < q; j += 32) {
                    // x at k = 0: FP64 in the FP64 kernel, FP32 in the slot's first four bytes in the mixed ones
                    double x0;
                    if constexpr (CL) x0 = MIXED ? f32_to_f64_nan(*(const float *)remote(j, 0, i, 3)) : *remote(j, 0, i, 3);
                    else x0 = MIXED ? f32_to_f64_nan(__ldcg((const float *)(rr.x0() + i * q + j))) : ldcg(rr.x0() + i * q + j);
                    const double d = x0 - sm.nu[i * q + j];
                    sm.x0[i * q + j] = x0;
                    sum = j == lane ? d : sum + d;
                }
                const double x1n = __dmul_rn(warp_sum(sum), iq64);    // (c), the mean over j
                for (int j = lane; j < q; j += 32) {
                    const int pr = i * q + j;
                    const double d = x1n - sm.x0[pr], nun = sm.nu[pr] + d; // (h)
                    sm.nu[pr] = nun;
                    if (MIXED) sm.x1nu[pr] = f64_to_f32_nan(x1n + nun);
                    if (check) r4m = max_nonneg(r4m, fabs(d));
                }
                if (lane == 0) sm.x1[i] = x1n;
            }
        }
        const double kappa = sm.bc[3];
        for (int p0 = 0; p0 < mq; p0 += NT >> gsh) {
            if (p0 + (int)((threadIdx.x & ~31u) >> gsh) >= mq) break; // the whole warp is past the pairs
            const int pq = p0 + (int)(threadIdx.x >> gsh), sub = threadIdx.x & (G - 1);
            const bool in = pq < mq;
            const int pr = in ? pq : mq - 1;
            const int i = pr / q, j = pr - i * q;
            const int nb = sm.rcnt[j];
            const double g0s = a.sumg0[pr], ci = a.c[i];
            // records of row j, every G-th (pair) per lane; a fixed order of the sums
            double S = 0.0, dmx = -INFINITY, dmn = INFINITY;
            if constexpr (CL) {
                for (int t = sub; t < nb; t += G) {
                    const double v = *remote(j, t, i, 0);
                    S = t == sub ? v : S + v;
                    if (check) {
                        dmx = max_ord(dmx, *remote(j, t, i, 1));
                        dmn = min_ord(dmn, *remote(j, t, i, 2));
                    }
                }
            } else {
                // two records per load, neighbouring lanes on neighbouring pairs of records; the
                // padding past nb is not added
                const double *rs = rr.s + rr.at(i, j, 0);
#pragma unroll 4
                for (int t = 2 * sub; t < nb; t += 2 * G) {
                    const double2 v = __ldcg((const double2 *)(rs + t));
                    const double w = t + 1 < nb ? v.x + v.y : v.x;
                    S = t == 2 * sub ? w : S + w;
                }
                if (check)
                    for (int t = sub; t < nb; t += G) {
                        dmx = max_ord(dmx, ldcg(rs + rr.plane + t));
                        dmn = min_ord(dmn, ldcg(rs + 2 * rr.plane + t));
                    }
            }
            for (int o = G >> 1; o > 0; o >>= 1) {
                S += __shfl_xor_sync(0xffffffffu, S, o);
                if (check) {
                    dmx = max_ord(dmx, __shfl_xor_sync(0xffffffffu, dmx, o));
                    dmn = min_ord(dmn, __shfl_xor_sync(0xffffffffu, dmn, o));
                }
            }
            const double lam = sm.lam[pr], zeta = sm.zeta[pr], hh = sm.h[pr], pp = sm.p[pr];
            const double W = fma(-nd, lam, S + g0s);                  // 1'(g(x) - lambda)
            const double lamn = __dmul_rn(kappa, (hh + pp) - W);      // (b) + (g); never fused into later sums,
                                                                      // which a resumed solve forms from lamn
            const double Z = fma(nd, lamn, W);                        // 1'z
            const double hn = min_ord(Z - pp, ci);                    // (d)
            const double e = hn - Z, zn = lamn - lam;
            if (check && in) { // a lane past the pairs may see the last pair's new scalars
                r2m = max_nonneg(r2m, fabs(zn));
                r3m = max_nonneg(r3m, fabs(e));
                const double dl = zn - zeta;
                s1m = max_nonneg(s1m, max_nonneg(fabs(dmx + dl), fabs(dmn + dl)));
                s2m = max_nonneg(s2m, fabs(hn - hh));
            }
            __syncwarp(); // the lanes of a pair have read its scalars
            if (in && sub == 0) {
                sm.lam[pr] = lamn;
                sm.zeta[pr] = zn;
                sm.h[pr] = hn;
                sm.p[pr] = pp + e;                                    // (i)
                if (MIXED) sm.uoff[pr] = f64_to_f32_nan(zn + lamn);
                else sm.zl[pr] = zn + lamn;
            }
        }
        if (check) { // maxima over the CTA, and over the CTAs' columns
            for (int b = threadIdx.x; b < a.grid; b += NT) {
                const double *cm = CL ? sm.ccm + par * 2 : a.cpart + ((size_t)par * a.grid + b) * 4;
                if (CL && a.grid > 1) cm = cg::this_cluster().map_shared_rank((double *)cm, b);
                r1m = max_nonneg(r1m, CL ? cm[0] : ldcg(cm));
                s3m = max_nonneg(s3m, CL ? cm[1] : ldcg(cm + 1));
            }
            double v[8] = {r1m, r2m, r3m, r4m, s1m, s2m, s3m, 0.0};
            auto mx = [](double k, double s, int o) { return max_nonneg(k, __shfl_xor_sync(0xffffffffu, s, o)); };
            const double r = warp_many<8>(v, mx);
            if ((threadIdx.x & 3) == 0) sm.mx[(threadIdx.x >> 5) * 8 + ((threadIdx.x & 31) >> 2)] = r;
        }
        __syncthreads();
        if (check) {
            // thread 0 takes the stop decision and the adaptation of Sec. IV-A and passes them on
            int *dec = (int *)(sm.bc + 7);
            if (threadIdx.x == 0) {
                double v[7];
#pragma unroll
                for (int t = 0; t < 7; ++t) {
                    v[t] = 0.0;
                    for (int w = 0; w < NWP; ++w) v[t] = max_nonneg(v[t], sm.mx[w * 8 + t]);
                    res[t] = v[t];
                }
                const double r = max_nonneg(max_nonneg(v[0], v[1]), max_nonneg(v[2], v[3]));
                const double sg = max_nonneg(max_nonneg(sm.rho[0] * v[4], sm.rho[1] * v[5]), sm.rho[2] * v[6]);
                r_last = r;
                s_last = sg;
                const bool cv = r < a.r_tol && sg < a.s_tol;
                double f = 1.0;
                if (!cv && a.adapt && it < a.max_iter && it >= a.adapt_start) { // Sec. IV-A, duals rescaled
                    const double ratio = r / sg, target = a.adapt_target;
                    if (ratio > 1.2 * target) f = a.tau;
                    else if (ratio < 0.8 * target) f = 1.0 / a.tau;
                }
                dec[0] = cv;
                dec[1] = f != 1.0;
                sm.bc[2] = f;
                if (f != 1.0) {
                    for (int t = 0; t < 4; ++t) sm.rho[t] *= f;
                    derive_penalties(sm, n);
                }
            }
            __syncthreads();
            if (dec[0]) {
                conv = true;
                break;
            }
            if (dec[1]) {
                const double f = sm.bc[2];
                for (int pr = threadIdx.x; pr < mq; pr += NT) {
                    const double l = sm.lam[pr] / f, nu = sm.nu[pr] / f;
                    sm.lam[pr] = l;
                    sm.p[pr] /= f;
                    sm.nu[pr] = nu;
                    if (MIXED) {
                        sm.uoff[pr] = (float)(sm.zeta[pr] + l);
                        sm.x1nu[pr] = (float)(sm.x1[pr / q] + nu);
                    } else {
                        sm.zl[pr] = sm.zeta[pr] + l;
                    }
                }
                mu_div = f;
                __syncthreads();
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        sm.flags[0] = cold ? 1.0 : 0.0;
        sm.flags[1] = mu_div;
    }
    __syncthreads();
    const int iters = it > a.max_iter ? a.max_iter : it;

    // ---- objective (1/q) sum f(x) of eq. (2): one more barrier -----------
    if (ok) {
        double acc = 0.0;
        for (int64_t cc = c0 + threadIdx.x; cc < c1; cc += NT) {
            const int j = (int)(cc / rs), k = (int)(cc - (int64_t)j * rs);
            if (k >= n) continue;
            for (int i = 0; i < m; ++i) {
                const size_t e = ((size_t)i * q + j) * a.ld + k;
                const size_t ec = ((size_t)i * a.cq + (size_t)j * a.cj) * a.ld + k; // coefficient element
                double f2, f1, f0, x;
                if constexpr (MIXED) {
                    f2 = ((const float *)a.f2)[ec];
                    f1 = ((const float *)a.f1)[ec];
                    f0 = ((const float *)a.f0)[ec];
                    x = ((const float *)a.x)[e];
                } else {
                    f2 = ((const double *)a.f2)[ec];
                    f1 = ((const double *)a.f1)[ec];
                    f0 = ((const double *)a.f0)[ec];
                    x = ((const double *)a.x)[e];
                }
                acc += f2 * x * x + f1 * x + f0;
            }
        }
        acc = warp_sum(acc);
        double escd = warp_sum((double)esc);
        if ((threadIdx.x & 31) == 0) {
            sm.mx[(threadIdx.x >> 5) * 8] = acc;
            sm.mx[(threadIdx.x >> 5) * 8 + 1] = escd;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0, te = 0.0;
            for (int w = 0; w < NWP; ++w) {
                t += sm.mx[w * 8];
                te += sm.mx[w * 8 + 1];
            }
            a.cpart[(size_t)blockIdx.x * 4 + 2] = t;
            a.cpart[(size_t)blockIdx.x * 4 + 3] = te;
        }
        if constexpr (CL) {
            team_sync(); // every CTA is past its last read of another's shared memory too
        } else {
            ++nbar;
            ok = grid_barrier(a.bar, nbar * (unsigned)a.grid, a.status, a.spin_ns, ADMM_ETIMEOUT);
        }
    }
    if (blockIdx.x == 0) {
        for (int t = threadIdx.x; t < scal_size(m, q); t += NT) a.scal[t] = smem[t];
        if (threadIdx.x == 0) {
            double obj = 0.0, escs = 0.0;
            if (ok)
                for (int b = 0; b < a.grid; ++b) {
                    obj += ldcg(a.cpart + (size_t)b * 4 + 2);
                    escs += ldcg(a.cpart + (size_t)b * 4 + 3);
                }
            a.info[0] = iters;
            a.info[1] = conv ? 1.0 : 0.0;
            a.info[2] = r_last;
            a.info[3] = s_last;
            for (int t = 0; t < 4; ++t) a.info[4 + t] = res[t];
            for (int t = 0; t < 3; ++t) a.info[8 + t] = res[4 + t] * sm.rho[t];
            a.info[11] = obj / (double)q;
            a.info[12] = ok ? 0.0 : (double)ld_volatile_i32(a.status);
            a.info[13] = escs;
        }
    }
}

} // namespace

} // namespace admm_impl
