// sweep2d_f64.cu -- FP64 transport sweep of one source iteration in 2D (arXiv:1712.01132, Sec. 3.1
// step i with the quadrature of step iii fused).
//
// What bounds it: GB300 issues an FP64 warp instruction once per ~65 cycles on a sub-partition, so a
// point costs a warp (operations) x 65 cycles and the wavefront's critical path is counted in points.
// The kernel therefore spreads the points of a band over warps and spends as few FP64 operations on a
// point as the scheme allows:
//   * Persistent CTAs take (problem, quadrant, band) items in band order.  A warp owns RPW rows of the
//     band (two rows of 16 velocities, or one row of 32) for the whole band; all its x1 carries are
//     registers.  A step of a warp is one column of its rows, the upper row a column behind the lower; a
//     warp follows the warp below it (same velocities) through a progress word in shared memory, so the
//     band's rows are swept at the same time on the SM's four sub-partitions.  A row takes its x2 upstream
//     values from the row below through shared memory (or, inside a warp, by a shuffle from the lower half).
//   * Three more warps keep everything else off the arithmetic: one copies the edge of the band below from
//     global memory into a ring in shared memory as soon as it is published, one builds the points' records,
//     one publishes this band's own edge column by column.
//   * Eq. 10 at a point takes seven FP64 operations (source 2, each axis 2, denominator 1):
//       h = R [ a + b1 v1 + b2 v2 + A1 (x + k h(x - 2 s1 e1)) + A2 (y + k' h(x - 2 s2 e2)) ]
//     with (A, k) = (2 |v|/dx, -1/4) for the second-order stencil, (|v|/dx, 0) for the first-order one,
//     and x = h(x - s1 e1) or the wall term: the same rounding as coefficients (2, -1/2), without the
//     multiplications by 0, 1 and 2.
//   * The moments take three more and no additions across lanes: the sweeping warps leave their h of the
//     last 16 columns in shared memory and moment warps sum them transposed (a lane per point, velocity by
//     velocity), on the FP64 time that the sweeping warps' latencies leave free.  The 16-velocity groups'
//     sums are added in group order.
// Measured, per sweep, against one warp per 32 velocities walking 8 x 8-point tiles one point at a time: 540 x
// 540 carpet, 8 x 8 velocities 5.93 -> 0.98 ms; 32 x 32 cell, 16 x 16 velocities 311 -> 90 us.  A step of eight
// warps on fluid columns takes ~1760 cycles (256 against 512 columns), of which its 80 FP64 instructions need ~1300
// at the SM's rate of one per ~16 cycles.  A band costs, beyond the steps of its rows, the hop through global
// memory (publish, poll, load): ~5000 cycles with 16 velocities a quadrant, ~8600 with 64 (2 against 8 bands).
#include <cuda_runtime.h>

#include <cstdint>

#include "dvm_device.cuh"
#include "dvm_internal.h"
#include "sweep2d_f64_waits.h"

namespace dvm {

namespace {

using f64waits::kBlk;             // columns of a moment block
constexpr int kRing = 2 * kBlk;   // columns of the h and record rings
constexpr int kMaxWarps = 16;     // sweeping warps of a CTA

// Moment warps beside W sweeping warps.  Three more load the edge below and the records and publish the edge above: at
// most 20 in all, but 23 with 16 sweeping warps, for which one moment warp is too few (200 x 160 points, 32^2 velocities
// 1963 us an iteration with one, 1500 with four; 22^2 in bands of 4 rows 1203 and 805).  More of them beside 13 to 15
// sweeping warps lose up to 6 %.
__host__ __device__ constexpr int moment_warps(int W) { return W < 17 - W ? W : (W < 16 ? 17 - W : 4); }

// Record of a point for one quadrant: {a, b1} {b2, E1} {E2, bits}, bits = stencil case of x1 | case of
// x2 << 2 | fluid << 4 | index of the denominator << 5; with specular wall parts the faces {upstream x1, x2, downstream x1, x2}.
struct alignas(16) Rec {
    double a, b1, b2, E1, E2;
    int bits, pad;
};

__device__ __forceinline__ int ld_acquire_cta(const int* p) {
    int v;
    asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_cta(int* p, int v) {
    asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

// a where p, else b, without a branch (the compiler may turn ?: on FP64 operands into divergent code)
__device__ __forceinline__ double sel(bool p, double a, double b) {
    double r;
    asm("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\tselp.f64 %0, %1, %2, q;\n\t}" : "=d"(r) : "d"(a), "d"(b), "r"((int)p));
    return r;
}

// barrier of the sweeping warps
__device__ __forceinline__ void barrier_warps(int nthreads) { asm volatile("barrier.cta.sync 1, %0;" ::"r"(nthreads) : "memory"); }

// Spin until the shared-memory flag reaches target; false when *stop is set or the bound expires: the warp then sets
// s_dead, with which the CTA leaves the item and the kernel's status is set.  (What these waits wait for is bounded
// itself by the waits on the band below; this is the second line.)
__device__ __forceinline__ bool spin_shared(const int* flag, int target, const int* stop, long long limit_ns) {
    if (ld_acquire_cta(flag) >= target) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned k = 1;; ++k) {
        if (ld_acquire_cta(flag) >= target) return true;
        if (ld_volatile(stop)) return ld_acquire_cta(flag) >= target;
        if ((k & 1023u) == 0u && (long long)(global_ns() - t0) > limit_ns) return false;
    }
}

template <int RPW> struct HRing {   // h of a warp's last kRing columns: [column][row][velocity + pad]
    static constexpr int VL = 32 / RPW;
    static constexpr int stride = VL + 1;
    static constexpr int doubles = kRing * RPW * stride;
};

}  // namespace

// (MAXW: the most warps of a CTA, which bounds the registers of a thread)
template <int RPW, bool XS, bool SPEC, int MAXW>
__global__ void __launch_bounds__(32 * MAXW) sweep2d_f64_kernel(const SweepArgs2D<double> a, const int NC, const int PR,
                                                                  const int TP) {
    constexpr int VL = 32 / RPW;                     // velocities per warp
    constexpr int HS = HRing<RPW>::stride;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    __shared__ int s_dead;                           // a wait gave up: the item is abandoned
    __shared__ int s_avail;                          // columns of the edge ring filled
    __shared__ int s_col[kMaxWarps];                 // steps (columns of its lower row) a sweeping warp has finished
    __shared__ int s_mom[kMaxWarps];                 // blocks summed, per sweeping warp
    __shared__ int s_rec[kMaxWarps];                 // blocks whose records are in place, per unit
    __shared__ int s_cnt[2 * kMaxWarps];             // group sums written, per block parity and unit
    const int W = PR * NC;                           // sweeping warps: unit p (RPW rows), velocity group cc
    const int NMW = moment_warps(W);
    const int NLc = NC * VL;                         // velocities swept
    const int ER = 2 * TP;                           // columns of the edge ring (a power of two)
    double* hring = reinterpret_cast<double*>(smem_raw);              // [W][kRing][RPW][HS]
    double* wtab = hring + (size_t)W * HRing<RPW>::doubles;           // [NLc][4]: W, W v1, W v2, -
    double* rtab = wtab + (size_t)NLc * 4;                            // [4][NLc]: reciprocal denominators
    double* ering = rtab + (size_t)NLc * 4;                           // [ER][2][NLc]
    double* part = ering + (size_t)ER * 2 * NLc;                      // [2][W][3][32]
    Rec* recs = reinterpret_cast<Rec*>(part + (size_t)2 * W * 3 * 32);        // [PR][kRing][RPW]
    int4* faces = reinterpret_cast<int4*>(recs + (size_t)PR * kRing * RPW);   // [PR][kRing][RPW] with SPEC
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = warp / NC, cc = warp - p * NC;
    const int rw = lane / VL;                        // row of the unit this lane sweeps
    const int vl = lane - rw * VL;
    const int vel = cc * VL + vl;                    // velocity slot of the quadrant
    const size_t NL = (size_t)a.NL;

    for (;;) {
        if (threadIdx.x == 0) {
            s_item = ld_volatile(a.status) ? a.nitems : atomicAdd(a.ticket, 1);
            s_avail = s_dead = 0;
        }
        if (threadIdx.x < kMaxWarps) s_col[threadIdx.x] = s_mom[threadIdx.x] = s_rec[threadIdx.x] = s_cnt[threadIdx.x] = s_cnt[kMaxWarps + threadIdx.x] = 0;
        __syncthreads();
        const int it = s_item;
        if (it >= a.nitems) return;
        const SweepItem item = a.items[it];
        const Prob2D<double>* __restrict__ P = a.prob + item.prob;
        const int q = item.quad, band = item.band;
        const int n1 = P->n1, n2 = P->n2, N = P->N;
        const int s1neg = q & 1, s2neg = (q >> 1) & 1;
        const int4 binfo = P->bands[q * P->nbands + band];
        const int row0 = binfo.x, nrows = binfo.y, below = binfo.z, above = binfo.w;
        const int par = a.parity;
        const int nblk = (n1 + kBlk - 1) / kBlk;
        const long long limit = f64waits::inner_bound(a.timeout_ns);     // of the waits inside the CTA
        if (warp < W) {
            const int yo = row0 + p * RPW + rw;                       // this lane's oriented row
            const bool myrow = p * RPW + rw < nrows;
            const bool top = p * RPW + rw == nrows - 1;               // the band's top row
            const bool topwarp = p == (nrows - 1) / RPW;
            const bool myunit = p * RPW < nrows;                      // the unit has a row of this band
            double v1, v2, a1, a2, a1f, a2f;
            const bool o2 = P->order == 2;
            {
                const double* lc = P->lanec + ((size_t)q * NL + vel) * kLaneConsts;
                v1 = lc[0]; v2 = lc[1]; a1 = lc[2]; a2 = lc[3];
                a1f = o2 ? 2.0 * a1 : a1;
                a2f = o2 ? 2.0 * a2 : a2;
                if (p == 0 && rw == 0) {
                    for (int k = 0; k < 4; ++k) rtab[k * NLc + vel] = lc[7 + k];
                    double* w = wtab + (size_t)vel * 4;
                    w[0] = lc[4];
                    w[1] = lc[5];
                    w[2] = lc[6];
                    w[3] = 0.0;
                }
            }
            const double kk = o2 ? -0.25 : 0.0;
            double* hr = hring + (size_t)warp * HRing<RPW>::doubles;
            const double* hb = hr - (size_t)NC * HRing<RPW>::doubles;      // the unit below, same velocities
            const double* hb2 = hb - (size_t)NC * HRing<RPW>::doubles;     // and the one below that (RPW = 1)
            Rec* rc = recs + (size_t)p * kRing * RPW;
            int4* fc = faces + (size_t)p * kRing * RPW;
            // specular wall parts: face stores of the previous iteration (read) and of this one (written)
            const double* fprev1 = nullptr;
            const double* fprev2 = nullptr;
            double* fnext1 = nullptr;
            double* fnext2 = nullptr;
            const double spec = SPEC ? P->spec : 0.0;
            if constexpr (SPEC) {   // x1 faces are told apart by the quadrant's x2 sign bit, x2 faces by its x1 bit
                const size_t plane = (size_t)P->nfaces * 2 * NL;
                fprev1 = P->F + par * plane + (size_t)s2neg * NL + vel;
                fprev2 = P->F + par * plane + (size_t)s1neg * NL + vel;
                fnext1 = P->F + (par ^ 1) * plane + (size_t)s2neg * NL + vel;
                fnext2 = P->F + (par ^ 1) * plane + (size_t)s1neg * NL + vel;
            }
            // x1 upstream of a row's first column: lagged slot 0 (the x1 ghosts) or the slot of an x1 subdomain
            auto gx = [&](int parity, int slot) -> double* {
                return P->gx1 + ((((size_t)(parity * 4 + q) * P->nxslots + slot) * n2 + yo) * 2) * NL + vel;
            };
            double hx1 = 0.0, hx2 = 0.0;
            if (myrow) {
                const double* g = gx(par, 0);
                hx1 = g[0];
                hx2 = g[NL];
            }
            int xsp = 1, xnext = (XS && P->nxslots > 1) ? P->xslot_col[q * P->nxslots + 1] : n1 + 1;
            // top edge: the ring slot of the band above, or the x2 layers of the next iteration (Eq. 8 /
            // periodic: the reflected quadrant reads the same slot)
            double* et = nullptr;
            if (topwarp) {
                if (above < 0) {
                    et = P->edge + ((size_t)(q * 2 * P->nslots + (-1 - above)) * n1) * 2 * NL + vel;
                } else {
                    const int qd = (above > 0 || P->lateral == 1) ? q : (q ^ 2);
                    et = P->glat + (((size_t)((par ^ 1) * 4 + qd) * P->nslots + above) * n1) * 2 * NL + vel;
                }
            }
            // x2 upstream values of the unit's lower row: the edge ring (unit 0) or the h of the rows below
            const double* ub1 = p == 0 ? ering + vel : (RPW == 2 ? hb + HS + vl : hb + vl);
            const double* ub2 = p == 0 ? ering + NLc + vel : (RPW == 2 ? hb + vl : (p == 1 ? ering + vel : hb2 + vl));
            const bool e1 = p == 0, e2 = p == 0 || (RPW == 1 && p == 1);      // from the edge ring
            const int um1 = e1 ? ER - 1 : kRing - 1, um2 = e2 ? ER - 1 : kRing - 1;
            const int us1 = e1 ? 2 * NLc : RPW * HS, us2 = e2 ? 2 * NLc : RPW * HS;
            const double* rt = rtab + vel;
            double h = 0.0, hy1 = 0.0;
            int bad = 0;                                  // a wait gave up
            const int steps = n1 + RPW - 1;
            // What a point needs beside its x2 upstream values, prepared at the end of the step before:
            // S, the x1 term, coefficients, and the lower row's last values for the upper row
            double S = 0.0, t1 = 0.0, A1 = a1, A2 = a2, ky = 0.0, Ey = 0.0, Rv = 0.0, s1 = 0.0, s2 = 0.0;
            bool wally = false, act = false;
            auto prepare = [&](int c, const Rec& r) {     // of this lane's column c with record r
                const bool in = myrow && (unsigned)c < (unsigned)n1;
                if constexpr (XS) {                       // a new x1 subdomain: its carry comes from a lagged slot
                    if (in && c == xnext) {
                        double* go = gx(par ^ 1, xsp);
                        go[0] = hx1;
                        go[NL] = hx2;
                        const double* gi = gx(par, xsp);
                        hx1 = gi[0];
                        hx2 = gi[NL];
                        ++xsp;
                        xnext = xsp < P->nxslots ? P->xslot_col[q * P->nxslots + xsp] : n1 + 1;
                    }
                }
                const int ca = r.bits & 3, cb = (r.bits >> 2) & 3;
                Rv = rt[((r.bits >> 5) & 3) * NLc];       // (masked: a lane off the band may hold a record not yet written)
                act = __any_sync(0xffffffffu, in && (r.bits & 16)) != 0;
                if (act) {
                    double x = sel(ca == 2, r.E1, hx1);
                    Ey = r.E2;
                    if constexpr (SPEC) {                 // + (1 - alpha) h'(x, reflected v) at walls
                        const int4 f = in ? fc[(c & (kRing - 1)) * RPW + rw] : make_int4(-1, -1, -1, -1);
                        if (f.x >= 0) x = fma(spec, fprev1[(size_t)f.x * 2 * NL], x);
                        if (f.y >= 0) Ey = fma(spec, fprev2[(size_t)f.y * 2 * NL], Ey);
                    }
                    S = fma(r.b2, v2, fma(r.b1, v1, r.a));
                    t1 = fma(sel(ca == 0, kk, 0.0), hx2, x);
                    A1 = sel(ca == 0, a1f, a1);
                    A2 = sel(cb == 0, a2f, a2);
                    ky = sel(cb == 0, kk, 0.0);
                    wally = cb == 2;
                }
                if constexpr (RPW == 2) {
                    s1 = __shfl_up_sync(0xffffffffu, h, 16);
                    s2 = __shfl_up_sync(0xffffffffu, hy1, 16);
                }
            };
            // before the records of column cn are read, at the start of a block: they are in place, and the h of
            // two blocks ago, which this block overwrites, has been summed and read by the rows above
            const bool above1 = (p + 1) * RPW < nrows, above2 = RPW == 1 && (p + 2) * RPW < nrows;
            auto block_ready = [&](int cn) {
                const int k = cn / kBlk;
                if (!spin_shared(&s_rec[p], f64waits::records_of_block(k), &s_dead, limit)) bad = 1;
                if (k >= 2) {
                    if (!spin_shared(&s_mom[warp], f64waits::own_moments(k), &s_dead, limit)) bad = 1;
                    if (above1 && !spin_shared(&s_col[warp + NC], f64waits::rows_above(k), &s_dead, limit)) bad = 1;
                    if (above2 && !spin_shared(&s_col[warp + 2 * NC], f64waits::rows_above(k), &s_dead, limit)) bad = 1;
                }
                bad = __any_sync(0xffffffffu, bad);
            };
            // before column c of the lower row is swept: its x2 upstream values are there (the edge of the band
            // below, or the unit below has finished the step in which its top row sweeps the column)
            const int* upflag = p == 0 ? &s_avail : &s_col[warp - NC];
            const int uplag = p == 0 ? 1 : f64waits::row_below(0, RPW);
            int seen = 0;                                 // progress already observed
            auto column_ready = [&](int c) {
                if (c < n1 && c + uplag > seen) {
                    // (the least that any lane has acquired: another lane's value would order nothing for this one)
                    seen = __reduce_min_sync(0xffffffffu, spin_shared(upflag, c + uplag, &s_dead, limit) ? ld_acquire_cta(upflag) : -1);
                    bad |= seen < 0;
                }
            };
            barrier_warps(W * 32);                        // the tables are in place
            if (myunit) {
                block_ready(0);
                // (after a wait that gave up the ring holds no record: its face numbers must not be followed)
                if (!SPEC || !bad) prepare(-rw, rc[((-rw) & (kRing - 1)) * RPW + rw]);
                for (int clow = 0; clow < steps; ++clow) {
                    const int c = clow - rw;              // this lane's column
                    const int cn = clow + 1;              // the lower row's next one
                    if ((cn & (kBlk - 1)) == 0 && cn < n1) block_ready(cn);
                    const Rec rn = rc[((cn - rw) & (kRing - 1)) * RPW + rw];
                    column_ready(clow);
                    if (bad) break;
                    // (lanes without a point of their own this step load and compute too; they keep nothing)
                    double u1 = ub1[(c & um1) * us1], u2 = ub2[(c & um2) * us2];
                    if constexpr (RPW == 2) {
                        u1 = sel(rw, s1, u1);
                        u2 = sel(rw, s2, u2);
                    }
                    double hn = 0.0;                      // solid points: 0, which no fluid point reads
                    if (act) {
                        const double t2 = fma(ky, u2, sel(wally, Ey, u1));
                        hn = fma(A1, t1, fma(A2, t2, S)) * Rv;
                    }
                    if (myrow && (unsigned)c < (unsigned)n1) {
                        h = hn;
                        hy1 = u1;
                        hx2 = hx1;
                        hx1 = h;
                        hr[((c & (kRing - 1)) * RPW + rw) * HS + vl] = h;
                        if (top) {
                            double* e = et + (size_t)c * 2 * NL;
                            e[0] = h;
                            e[NL] = u1;
                        }
                        if constexpr (SPEC) {   // molecules moving into a downstream face
                            const int4 f = fc[(c & (kRing - 1)) * RPW + rw];
                            if (f.z >= 0) fnext1[(size_t)f.z * 2 * NL] = h;
                            if (f.w >= 0) fnext2[(size_t)f.w * 2 * NL] = h;
                        }
                        if (c == n1 - 1) {   // x1 layers of the next iteration
                            double* g1 = gx(par ^ 1, 0);
                            g1[0] = hx1;
                            g1[NL] = hx2;
                        }
                    }
                    __syncwarp();
                    if (lane == 0) st_release_cta(&s_col[warp], cn);
                    prepare(cn - rw, rn);
                }
            }
            if (bad && lane == 0) *reinterpret_cast<volatile int*>(&s_dead) = 1;
        } else if (warp < W + NMW) {
            // moments: lane = point of a block (with 32 velocities a warp's lanes are 16 points x two halves of
            // the velocities); every sweeping warp's block is one velocity group's sum
            const int mpt = RPW == 2 ? lane : (lane & 15), mgrp = RPW == 2 ? 0 : lane >> 4;
            bool dead = false;
            for (int kb = 0; kb < nblk && !dead; ++kb) {
                for (int w = warp - W; w < W && !dead; w += NMW) {
                    const int pw = w / NC, cw = w - pw * NC;
                    if (pw * RPW >= nrows) {              // a unit off the band
                        if (lane == 0) st_release_cta(&s_mom[w], kb + 1);
                        continue;
                    }
                    dead = __any_sync(0xffffffffu, !spin_shared(&s_col[w], f64waits::swept(kb, n1, RPW), &s_dead, limit));
                    if (dead) break;
                    const double* hv = hring + (size_t)w * HRing<RPW>::doubles + ((kb & 1) * kBlk * RPW + mpt) * HS + mgrp * 16;
                    const double* wt = wtab + (size_t)(cw * VL + mgrp * 16) * 4;
                    double m[3] = {0.0, 0.0, 0.0};
#pragma unroll 4
                    for (int l = 0; l < 16; ++l) {
                        const double2 wa = *reinterpret_cast<const double2*>(wt + l * 4);
                        const double x = hv[l];
                        m[0] = fma(wa.x, x, m[0]);
                        m[1] = fma(wa.y, x, m[1]);
                        m[2] = fma(wt[l * 4 + 2], x, m[2]);
                    }
                    if constexpr (RPW == 1) {
#pragma unroll
                        for (int j = 0; j < 3; ++j) m[j] += __shfl_xor_sync(0xffffffffu, m[j], 16);
                    }
                    bool write = true;
                    if (NC > 1) {   // the last group of the unit to come adds the groups' sums in group order
                        // this parity's sums and count are free: every group is past block kb - 2 (a lane per group)
                        const bool free = kb < 2 || lane >= NC ||
                                          spin_shared(&s_mom[pw * NC + lane], f64waits::group_moments(kb), &s_dead, limit);
                        dead = !__all_sync(0xffffffffu, free);
                        if (dead) break;
                        __syncwarp();
                        double* d = part + ((size_t)(kb & 1) * W + w) * 3 * 32 + lane;
                        d[0] = m[0];
                        d[32] = m[1];
                        d[64] = m[2];
                        __threadfence_block();
                        __syncwarp();
                        int prev = lane == 0 ? atomicAdd(&s_cnt[(kb & 1) * kMaxWarps + pw], 1) : 0;
                        prev = __shfl_sync(0xffffffffu, prev, 0);
                        write = prev == ((kb >> 1) + 1) * NC - 1;
                        if (write) {
                            __threadfence_block();
                            __syncwarp();                 // lane 0's count, then every lane's reads of the sums
                            const double* o = part + ((size_t)(kb & 1) * W + pw * NC) * 3 * 32 + lane;
#pragma unroll
                            for (int j = 0; j < 3; ++j) {
                                m[j] = 0.0;
                                for (int k = 0; k < NC; ++k) m[j] += o[(k * 3 + j) * 32];
                            }
                        }
                    }
                    const int col = kb * kBlk + mpt / RPW, rr = pw * RPW + mpt % RPW;
                    if (write && mgrp == 0 && col < n1 && rr < nrows) {
                        const int x = s1neg ? n1 - 1 - col : col;
                        const int y = s2neg ? n2 - 1 - (row0 + rr) : row0 + rr;
                        double* o = P->P + (size_t)q * 3 * N + (size_t)y * n1 + x;
                        o[0] = m[0];
                        o[N] = m[1];
                        o[2 * (size_t)N] = m[2];
                    }
                    __syncwarp();
                    if (lane == 0) st_release_cta(&s_mom[w], kb + 1);
                }
            }
            if (dead && lane == 0) *reinterpret_cast<volatile int*>(&s_dead) = 1;
        } else if (warp == W + NMW) {
            // the two rows below this band, column by column: the band below's top edge once it is
            // published, or lagged layers (the x2 ghosts at the domain face, the halo of a subdomain)
            const double* eb = below >= 0 ? P->glat + (((size_t)(par * 4 + q) * P->nslots + below) * n1) * 2 * NL
                                          : P->edge + ((size_t)(q * 2 * P->nslots + (-1 - below)) * n1) * 2 * NL;
            const int* flag = P->prog + q * P->nbands + band - 1;
            int seen = below < 0 ? 0 : n1;
            const int ng = NLc / 16;                                  // groups of 16 velocities
            for (int c0 = 0, n = 0; c0 < n1; c0 += n) {
                // every lane waits for itself (a shuffle orders no memory), and the least that any has seen counts
                if (seen <= c0) seen = __reduce_min_sync(0xffffffffu, wait_geq_value(flag, c0 + 1, a.status, a.timeout_ns));
                int ok = seen >= 0;
                // as many columns as are there, up to half the ring.  The slot of column c is free when unit 0
                // (and with one row per unit also unit 1, which reads it as its second upstream row) is past c
                n = min(min(seen, n1) - c0, TP);
                for (int w = 0; ok && c0 + n > ER && w < (RPW == 1 ? 2 : 1) * NC; ++w)
                    if ((w < NC || nrows > 1) && !spin_shared(&s_col[w], c0 + n - ER, &s_dead, limit)) ok = 0;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) *reinterpret_cast<volatile int*>(&s_dead) = 1;
                    break;
                }
                // items of 16 velocities (eight lanes x 16 bytes), four at a time: (column, layer) cl, group gr
                const int items = n * 2 * ng;
                int cl = (lane >> 3) / ng, gr = (lane >> 3) - cl * ng;
#pragma unroll 4
                for (int k = lane >> 3; k < items; k += 4) {
                    const int v = gr * 8 + (lane & 7);
                    const double2 d = __ldcg(reinterpret_cast<const double2*>(eb + ((size_t)c0 * 2 + cl) * NL) + v);
                    reinterpret_cast<double2*>(ering + (size_t)(((c0 + (cl >> 1)) & (ER - 1)) * 2 + (cl & 1)) * NLc)[v] = d;
                    gr += 4;
                    while (gr >= ng) {
                        gr -= ng;
                        ++cl;
                    }
                }
                __syncwarp();
                if (lane == 0) st_release_cta(&s_avail, c0 + n);
            }
        } else if (warp == W + NMW + 1) {
            // records of a block's points, unit by unit (a lane per point): the loads of the next unit or block
            // are on their way while the sweep runs
            const int lcol = RPW == 2 ? lane >> 1 : lane & 15, lrow = RPW == 2 ? (lane & 1) : 0;
            const int nun = (nrows + RPW - 1) / RPW;
            bool ok = true;
            for (int k = it == -2 - a.withhold_item ? nblk : 0; k < nblk && ok; ++k) {   // (test hook: no records at all)
                for (int pu = 0; pu < nun; ++pu) {
                    int code = kSolidBit;
                    double2 ab = make_double2(0.0, 0.0);
                    double b2 = 0.0, E1 = 0.0, E2 = 0.0;
                    int4 f = make_int4(-1, -1, -1, -1);
                    const int ic = k * kBlk + lcol, lr = pu * RPW + lrow;
                    if (ic < n1 && lr < nrows) {
                        const int x = s1neg ? n1 - 1 - ic : ic;
                        const int y = s2neg ? n2 - 1 - (row0 + lr) : row0 + lr;
                        const int id = y * n1 + x;
                        code = P->code[id];
                        ab = reinterpret_cast<const double2*>(P->src)[2 * (size_t)id];
                        b2 = P->src[4 * (size_t)id + 2];
                        E1 = P->E[4 * (size_t)id + s1neg];
                        E2 = P->E[4 * (size_t)id + 2 + s2neg];
                        if constexpr (SPEC) {
                            const int* fi = P->face_id;
                            f = make_int4(fi[(0 + s1neg) * (size_t)N + id], fi[(2 + s2neg) * (size_t)N + id],
                                          fi[(1 - s1neg) * (size_t)N + id], fi[(3 - s2neg) * (size_t)N + id]);
                        }
                    }
                    // the buffer's last reader is the unit's top row at the end of block k - 2
                    for (int w = pu * NC; k >= 2 && ok && w < (pu + 1) * NC; ++w)
                        ok = spin_shared(&s_col[w], f64waits::record_readers(k, RPW), &s_dead, limit);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    if (lane < kBlk * RPW) {
                        const int o = (pu * kRing + (k & 1) * kBlk + lcol) * RPW + lrow;
                        Rec* r = recs + o;
                        const bool fluid = !(code & kSolidBit);
                        const int ca = (code >> (2 * s1neg)) & 3, cb = (code >> (2 * (2 + s2neg))) & 3;
                        r->a = fluid ? ab.x : 0.0;
                        r->b1 = fluid ? ab.y : 0.0;
                        r->b2 = fluid ? b2 : 0.0;
                        r->E1 = fluid ? E1 : 0.0;
                        r->E2 = fluid ? E2 : 0.0;
                        // first-order denominator of an axis when either upstream point is solid (cases 1, 2);
                        // a solid point is a point between walls without a source: h = 0
                        r->bits = fluid ? (ca | (cb << 2) | 16 | (ca != 0 ? 32 : 0) | (cb != 0 ? 64 : 0)) : (2 | (2 << 2) | 96);
                        if constexpr (SPEC) faces[o] = fluid ? f : make_int4(-1, -1, -1, -1);
                    }
                    __syncwarp();
                    if (lane == 0) st_release_cta(&s_rec[pu], k + 1);
                }
            }
            if (!ok && lane == 0) *reinterpret_cast<volatile int*>(&s_dead) = 1;
        } else if (lane == 0 && above < 0 && it != a.withhold_item) {
            // publish this band's top edge as the top row (row `ft` of unit `pt`) sweeps it, whatever is new at a time
            const int pt = (nrows - 1) / RPW, ft = (nrows - 1) % RPW;
            bool ok = true;
            for (int done = 0; done < n1;) {
                int m = n1;
                for (int w = pt * NC; ok && w < (pt + 1) * NC; ++w) {
                    ok = spin_shared(&s_col[w], done + 1 + ft, &s_dead, limit);
                    m = min(m, ld_acquire_cta(&s_col[w]) - ft);
                }
                if (!ok) break;
                done = m;
                publish_gpu(P->prog + q * P->nbands + band, done);
            }
            if (!ok) *reinterpret_cast<volatile int*>(&s_dead) = 1;
        }
        __syncthreads();
        if (s_dead) {   // some wait gave up: the host learns of it here, also where no other band waits for this item
            if (threadIdx.x == 0) atomicCAS(a.status, 0, -4);
            return;
        }
        __syncthreads();
    }
}

// Shape of a CTA for nvq velocities per quadrant: rows per warp, velocity groups (warps per unit of rows),
// units per band and half the columns of the ring that holds the edge of the band below.
//   * Two rows of 16 velocities per warp up to 256 velocities (less padding: 16 velocities a quadrant fill a
//     warp), one row of 32 above (so that 512 velocities still take 16 warps).
//   * Eight sweeping warps per CTA (two per sub-partition) unless band_rows asks otherwise.  Fewer rows per band
//     cost more hops from band to band, more rows share the SM's FP64 units.  An iteration on the 32 x 32 cell with
//     64 velocities a quadrant takes 126, 101 and 111 us with 4, 8 and 16 warps, on the 540 x 540 carpet with 16
//     velocities 1.57, 1.04, 0.98 and 1.47 ms with 2, 4, 8 and 16.  Five to eight groups leave one unit, two rows a
//     band: two units (band_rows 4) are faster on large domains (200 x 160 points, 81 velocities a quadrant 809 and
//     682 us, 121 897 and 805).
Shape2DF64 sweep2d_f64_shape(int nvq, int band_rows, int tile_x1, size_t smem_limit, int spec) {
    Shape2DF64 s;
    s.rpw = nvq <= 256 ? 2 : 1;
    s.groups = (nvq + 32 / s.rpw - 1) / (32 / s.rpw);
    const int most = kMaxWarps / s.groups;
    int units = band_rows > 0 ? (band_rows + s.rpw - 1) / s.rpw : 8 / s.groups;
    s.units = units < 1 ? 1 : (units > most ? most : units);
    s.rows = s.units * s.rpw;
    if (band_rows > 0 && band_rows < s.rows) s.rows = band_rows;
    s.tile = (tile_x1 == 16 ? 16 : 8) / 2;
    while (s.tile > 2 && sweep2d_f64_smem(s, spec) > smem_limit) s.tile /= 2;
    while (s.units > 1 && sweep2d_f64_smem(s, spec) > smem_limit) {
        --s.units;
        if (s.rows > s.units * s.rpw) s.rows = s.units * s.rpw;
    }
    return s;
}

size_t sweep2d_f64_smem(const Shape2DF64& s, int spec) {
    const size_t W = (size_t)s.units * s.groups, NLc = (size_t)s.groups * (32 / s.rpw);
    const size_t hd = s.rpw == 2 ? HRing<2>::doubles : HRing<1>::doubles;
    return sizeof(double) * (W * hd + NLc * 8 + (size_t)2 * s.tile * 2 * NLc + 2 * W * 3 * 32) +
           (size_t)s.units * kRing * s.rpw * (sizeof(Rec) + (spec ? sizeof(int4) : 0));
}

namespace {

template <int RPW, bool XS, bool SPEC>
cudaError_t run_t(const SweepArgs2D<double>* a, const Shape2DF64& s, int grid, cudaStream_t st, int* blocks_per_sm) {
    const size_t smem = sweep2d_f64_smem(s, SPEC);
    const int W = s.units * s.groups, warps = W + moment_warps(W) + 3, threads = 32 * warps;
    auto kern = warps <= 20 ? sweep2d_f64_kernel<RPW, XS, SPEC, 20> : sweep2d_f64_kernel<RPW, XS, SPEC, 23>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (blocks_per_sm) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, threads, smem);
    kern<<<grid, threads, smem, st>>>(*a, s.groups, s.units, s.tile);
    return cudaGetLastError();
}

cudaError_t run(const SweepArgs2D<double>* a, const Shape2DF64& s, int xs, int spec, int grid, cudaStream_t st, int* bps) {
    if (s.rpw == 2) {
        if (spec) return xs ? run_t<2, true, true>(a, s, grid, st, bps) : run_t<2, false, true>(a, s, grid, st, bps);
        return xs ? run_t<2, true, false>(a, s, grid, st, bps) : run_t<2, false, false>(a, s, grid, st, bps);
    }
    if (spec) return xs ? run_t<1, true, true>(a, s, grid, st, bps) : run_t<1, false, true>(a, s, grid, st, bps);
    return xs ? run_t<1, true, false>(a, s, grid, st, bps) : run_t<1, false, false>(a, s, grid, st, bps);
}

}  // namespace

// xs: x1 subdomains (lagged x1 halos); a.spec: specular wall parts (Eq. 5)
cudaError_t launch_sweep2d_f64(const SweepArgs2D<double>& a, const Shape2DF64& s, int xs, int grid, cudaStream_t st) {
    return run(&a, s, xs, a.spec, grid, st, nullptr);
}

cudaError_t sweep2d_f64_occupancy(const Shape2DF64& s, int xs, int spec, int* blocks_per_sm) {
    return run(nullptr, s, xs, spec, 0, nullptr, blocks_per_sm);
}

}  // namespace dvm
