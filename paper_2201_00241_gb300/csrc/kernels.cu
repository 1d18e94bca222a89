// kernels.cu -- FP64 device kernels of librh (sm_103a).
//
// The hot path (Algorithm 2 of arXiv 2201.00241) is FP64-ALU-bound on GB300:
// one FP64 pipe per SM sub-partition retires one warp-wide DFMA per 64 cycles
// (about 1.2 TFLOP/s for the chip) and masked-off lanes cost the same issue
// slot.  The kernels are therefore organised to keep every lane of every
// DFMA useful:
//
//  * Directions are independent, so the direction kernel gives each CTA its
//    own slice of the N directions and runs every step of Algorithm 2 on it
//    (SpMul, both triangular sweeps, the projection, both transposed sweeps,
//    SpMulAdd) with only CTA-local barriers: no grid-wide synchronisation.
//  * Inside a CTA the work of a level is flattened over (bus, direction)
//    pairs; in narrow levels near the top of the elimination tree each row's
//    dot product is further split over adjacent lanes of a warp and summed with
//    shuffles, so that more warps issue FP64 work and a level needs one barrier.
//  * A bus is a block of one (PV) or two (PQ) variables whose rows share the
//    same columns outside the bus; one load of x_c feeds two FMAs.
//  * Right-hand sides are interleaved, row-major [row][ld]: the D directions
//    of a CTA are contiguous in each row.
#include <cstdio>
#include <mutex>

#include "../../include/rh.h"
#include "rh_kernels.h"

namespace rh {

namespace {

// Direction CTAs: 384 threads, 2 resident per SM (80 registers).  With 24 warps per
// SM either way, 2 CTAs of 384 run the full 9241-bus Hessian in 6.47 ms against
// 7.39 ms for 3 of 256: more directions per CTA put fewer buses (with different
// row lengths) in a warp and more items in every level.
constexpr int kDirThreads = 384;
constexpr int kDirCtasPerSm = 2;
constexpr int kPartCap = 4096;   // doubles of the CTA's dense-tail rows (T x directions)
constexpr int kDMax = 256;       // max directions per CTA

// Index checks of the bounds-checking build (-DRH_BOUNDS): a failed check sets a
// bit of g_bounds_err and the access is skipped (never a trap, never an early
// return that a barrier would wait for); rh_bounds_check reads the word.  In the
// normal build every check is the constant true and compiles away.
#ifdef RH_BOUNDS
__device__ unsigned int g_bounds_err;
__device__ __forceinline__ bool inb(long long i, long long n) {
    const bool ok = i >= 0 && i < n;
    if (!ok) atomicOr(&g_bounds_err, 1u);
    return ok;
}
#else
__device__ __forceinline__ constexpr bool inb(long long, long long) { return true; }
#endif

__device__ __forceinline__ unsigned long long ordered_bits(double v) {
    // |v| as a bit pattern whose unsigned order is the numeric order (NaN above inf)
    return (unsigned long long)__double_as_longlong(fabs(v));
}

// ---------------------------------------------------------------------------
// power flow: injections (eq. 2), residual (eq. 3), Jacobians
// ---------------------------------------------------------------------------

__global__ void k_injections(PfGrid g, PfState s) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_bus) return;
    double vi = s.vm[i], ai = s.va[i], p = 0.0, q = 0.0;
    for (int t = g.yp[i]; t < g.yp[i + 1]; t++) {
        int j = g.yj[t];
        double sn, cs;
        sincos(ai - s.va[j], &sn, &cs);
        p += s.vm[j] * (g.G[t] * cs + g.B[t] * sn);
        q += s.vm[j] * (g.G[t] * sn - g.B[t] * cs);
    }
    s.P[i] = vi * p;
    s.Q[i] = vi * q;
}

// One thread per bus: injections, the two residual rows of the bus and the
// Jacobian entries of those rows, scattered into the fixed LU / J_p slots.
// the four derivatives of admittance entry t into their slots of A (J_x) or J_p
__device__ __forceinline__ void jac_store(const PfGrid& g, int t, const double (&d)[4], double* A, double* jpv,
                                          unsigned long long& jm) {
    for (int u = 0; u < 4; u++) {
        const int dst = g.jac_dst[4 * t + u];
        if (dst >= 0) {
            if (!inb(dst, g.nnz_a)) continue;
            A[dst] = d[u];
            const unsigned long long b = ordered_bits(d[u]);
            jm = b > jm ? b : jm;
        } else if (dst <= -2) {
            if (!inb(-(dst + 2), g.nnz_jp)) continue;
            jpv[-(dst + 2)] = d[u];
        }
    }
}

__device__ __forceinline__ void k_pf_eval_body(PfGrid g, PfState s, double* gres, double* A, double* jpv,
                          unsigned long long* gmax, unsigned long long* jmax, int want_jac) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_bus) return;
    const double vi = s.vm[i], ai = s.va[i];
    const int rP = g.qth[i];
    const bool jac = want_jac && rP >= 0;
    double P = 0.0, Q = 0.0;
    unsigned long long jm = 0;
    int tdiag = -1;
    // one pass over the admittance row: the injection sums and, for j != i, the
    // off-diagonal Jacobian entries from the same sin/cos of theta_i - theta_j
    for (int t = g.yp[i]; t < g.yp[i + 1]; t++) {
        const int j = g.yj[t];
        double sn = 0.0, cs = 1.0;
        if (j != i) sincos(ai - s.va[j], &sn, &cs);
        else tdiag = t;
        const double vj = s.vm[j], Gij = g.G[t], Bij = g.B[t];
        P += vj * (Gij * cs + Bij * sn);
        Q += vj * (Gij * sn - Bij * cs);
        if (jac && j != i) {
            double d[4];  // dP/dtheta_j, dP/dv_j, dQ/dtheta_j, dQ/dv_j
            d[0] = vi * vj * (Gij * sn - Bij * cs);
            d[1] = vi * (Gij * cs + Bij * sn);
            d[2] = -vi * vj * (Gij * cs + Bij * sn);
            d[3] = vi * (Gij * sn - Bij * cs);
            jac_store(g, t, d, A, jpv, jm);
        }
    }
    P *= vi;
    Q *= vi;
    s.P[i] = P;
    s.Q[i] = Q;
    const int rQ = g.qv[i];
    if (rP < 0) return;  // slack: no rows
    if (gres) {
        double gp = P - s.pg[i] + s.pd[i];
        gres[rP] = gp;
        unsigned long long m = ordered_bits(gp);
        if (rQ >= 0) {
            double gq = Q + s.qd[i];
            gres[rQ] = gq;
            unsigned long long mq = ordered_bits(gq);
            m = mq > m ? mq : m;
        }
        atomicMax(gmax, m);
    }
    if (!want_jac) return;
    if (tdiag >= 0) {
        const double Gii = g.G[tdiag], Bii = g.B[tdiag];
        double d[4];
        d[0] = -Q - Bii * vi * vi;
        d[1] = P / vi + Gii * vi;
        d[2] = P - Gii * vi * vi;
        d[3] = Q / vi - Bii * vi;
        jac_store(g, tdiag, d, A, jpv, jm);
    }
    if (g.ip_pg[i] >= 0) jpv[g.pg_slot[i]] = -1.0;
    atomicMax(jmax, jm);
}
__global__ void k_pf_eval(PfGrid g, PfState s, double* gres, double* A, double* jpv,
                          unsigned long long* gmax, unsigned long long* jmax, int want_jac) {
    pdl_wait();
    pdl_trigger();
    k_pf_eval_body(g, s, gres, A, jpv, gmax, jmax, want_jac);
}

// Per-state preparation of the assembly: sin and cos of every bus angle (the
// assembly then forms sin and cos of each angle difference with two products), and,
// with zero, A (the slots the assembly and the refactorisation fill), the maxima and
// the pivot flag cleared.
__device__ __forceinline__ void pf_prep_body(const PfGrid& g, const PfState& s, double* A, unsigned long long* umax,
                                             int* err, int zero) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    if (zero) {
        for (int64_t k = i0; k < g.nnz_a; k += stride) A[k] = 0.0;
        if (i0 == 0) {
            umax[0] = 0ull;
            umax[1] = 0ull;
            if (err) *err = 0;
        }
    }
    if (s.sc)
        for (int64_t b = i0; b < g.n_bus; b += stride) {
            double sn, cs;
            sincos(s.va[b], &sn, &cs);
            s.sc[2 * b] = sn;
            s.sc[2 * b + 1] = cs;
        }
}
__global__ void k_pf_prep(PfGrid g, PfState s, double* A, unsigned long long* umax, int* err, int zero) {
    pdl_wait();
    pf_prep_body(g, s, A, umax, err, zero);
}

// The same evaluation with one admittance entry per lane: warp w takes the buses
// [pf_wb[w], pf_wb[w + 1]) (at most 32 entries together).  Each lane forms its
// entry's sin/cos, the two injection terms and, off the diagonal, its four Jacobian
// entries; after a warp barrier the lane of each bus sums its row's terms in row
// order and finishes the bus (residual, diagonal Jacobian block) as above.  The
// maxima go through one atomic per warp.  Blocks of kPfWarps warps.
constexpr int kPfWarps = 4;
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
        v = u > v ? u : v;
    }
    return v;
}
__device__ __forceinline__ void pf_eval_warp_body(const PfGrid& g, const PfState& s, double* gres, double* A,
                                                  double* jpv, unsigned long long* gmax, unsigned long long* jmax,
                                                  int want_jac) {
    __shared__ double sh[kPfWarps][96];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int w = blockIdx.x * kPfWarps + wl;
    if (w >= g.n_pfw) return;                                   // warp-uniform
    double* sw = sh[wl];
    const int b0 = g.pf_wb[w], b1 = g.pf_wb[w + 1];
    const int e0 = g.yp[b0], e1 = g.yp[b1];
    const int t = e0 + lane;
    unsigned long long jm = 0, gm = 0;
    double vj = 0.0, xp = 0.0, xq = 0.0;
    if (t < e1) {
        const int i = g.yrow[t], j = g.yj[t];
        double sn = 0.0, cs = 1.0;
        if (j != i) {
            if (s.sc) {            // sin / cos of theta_i - theta_j from the buses' own
                const double si = s.sc[2 * i], ci = s.sc[2 * i + 1], sj = s.sc[2 * j], cj = s.sc[2 * j + 1];
                sn = fma(si, cj, -(ci * sj));
                cs = fma(ci, cj, si * sj);
            } else {
                sincos(s.va[i] - s.va[j], &sn, &cs);
            }
        }
        vj = s.vm[j];
        const double Gij = g.G[t], Bij = g.B[t];
        xp = Gij * cs + Bij * sn;
        xq = Gij * sn - Bij * cs;
        if (want_jac && j != i && g.qth[i] >= 0) {
            const double vi = s.vm[i];
            double d[4];  // dP/dtheta_j, dP/dv_j, dQ/dtheta_j, dQ/dv_j
            d[0] = vi * vj * xq;
            d[1] = vi * xp;
            d[2] = -vi * vj * xp;
            d[3] = vi * xq;
            jac_store(g, t, d, A, jpv, jm);
        }
    }
    sw[lane] = vj;
    sw[32 + lane] = xp;
    sw[64 + lane] = xq;
    __syncwarp();
    const int i = b0 + lane;
    if (i < b1) {
        const double vi = s.vm[i];
        double P = 0.0, Q = 0.0;
        int tdiag = -1;
        for (int tt = g.yp[i]; tt < g.yp[i + 1]; tt++) {
            const int k = tt - e0;
            P += sw[k] * sw[32 + k];
            Q += sw[k] * sw[64 + k];
            if (g.yj[tt] == i) tdiag = tt;
        }
        P *= vi;
        Q *= vi;
        s.P[i] = P;
        s.Q[i] = Q;
        const int rP = g.qth[i], rQ = g.qv[i];
        if (rP >= 0) {                                          // the slack has no rows
            if (gres) {
                const double gp = P - s.pg[i] + s.pd[i];
                gres[rP] = gp;
                gm = ordered_bits(gp);
                if (rQ >= 0) {
                    const double gq = Q + s.qd[i];
                    gres[rQ] = gq;
                    const unsigned long long mq = ordered_bits(gq);
                    gm = mq > gm ? mq : gm;
                }
            }
            if (want_jac) {
                if (tdiag >= 0) {
                    const double Gii = g.G[tdiag], Bii = g.B[tdiag];
                    double d[4];
                    d[0] = -Q - Bii * vi * vi;
                    d[1] = P / vi + Gii * vi;
                    d[2] = P - Gii * vi * vi;
                    d[3] = Q / vi - Bii * vi;
                    jac_store(g, tdiag, d, A, jpv, jm);
                }
                if (g.ip_pg[i] >= 0) jpv[g.pg_slot[i]] = -1.0;
            }
        }
    }
    gm = warp_max_u64(gm);
    jm = warp_max_u64(jm);
    if (lane == 0) {
        if (gres) atomicMax(gmax, gm);
        if (want_jac) atomicMax(jmax, jm);
    }
}
__global__ void __launch_bounds__(32 * kPfWarps) k_pf_eval_warp(PfGrid g, PfState s, double* gres, double* A,
                                                                double* jpv, unsigned long long* gmax,
                                                                unsigned long long* jmax, int want_jac) {
    pdl_wait();
    pdl_trigger();
    pf_eval_warp_body(g, s, gres, A, jpv, gmax, jmax, want_jac);
}

__device__ __forceinline__ void k_newton_update_body(PfGrid g, PfState s, const double* dx) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_bus) return;
    if (g.qth[i] >= 0) s.va[i] -= dx[g.qth[i]];
    if (g.qv[i] >= 0) s.vm[i] -= dx[g.qv[i]];
}
__global__ void k_newton_update(PfGrid g, PfState s, const double* dx) {
    pdl_wait();
    pdl_trigger();
    k_newton_update_body(g, s, dx);
}

// ---------------------------------------------------------------------------
// coloured forward-mode Jacobian (section 4.2.2, Fig. 2)
// ---------------------------------------------------------------------------
// A dual number carries a value and CH tangent components.  Every variable of
// x and p is seeded with the unit tangent of its column colour, so the
// tangent c of a residual row is the sum of that row's derivatives over the
// columns of colour c, which the colouring makes a single entry.  Colours are
// processed CH at a time (one grid row per chunk; the values are recomputed in
// every chunk, as in chunked forward mode).

template <int CH>
struct Dual {
    double v;
    double d[CH];
};

template <int CH>
__device__ __forceinline__ Dual<CH> dual_seed(double v, int k) {
    Dual<CH> r;
    r.v = v;
#pragma unroll
    for (int m = 0; m < CH; m++) r.d[m] = (m == k) ? 1.0 : 0.0;
    return r;
}

template <int CH>
__global__ void __launch_bounds__(128) k_jac_ad(PfGrid g, PfState s, const int* __restrict__ col_th,
                                                const int* __restrict__ col_v, const int* __restrict__ col_pg,
                                                double* A, double* jpv, unsigned long long* jmax) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_bus || g.qth[i] < 0) return;      // the slack has no rows
    const int c0 = blockIdx.y * CH;
    const Dual<CH> th_i = dual_seed<CH>(s.va[i], col_th[i] - c0);
    const Dual<CH> v_i = dual_seed<CH>(s.vm[i], col_v[i] - c0);
    // P_i / v_i and Q_i / v_i accumulated over the admittance row (eq. 2)
    Dual<CH> p = dual_seed<CH>(0.0, -1), q = dual_seed<CH>(0.0, -1);
    for (int t = g.yp[i]; t < g.yp[i + 1]; t++) {
        const int j = g.yj[t];
        const double G = g.G[t], B = g.B[t];
        const int kth = col_th[j] - c0, kv = col_v[j] - c0;
        double sn, cs;
        sincos(th_i.v - s.va[j], &sn, &cs);
        const double vj = s.vm[j];
        const double gc = G * cs + B * sn, gs = G * sn - B * cs;   // value parts of the two brackets
        p.v = fma(vj, gc, p.v);
        q.v = fma(vj, gs, q.v);
#pragma unroll
        for (int m = 0; m < CH; m++) {
            // d(theta_i - theta_j); d cos = -sin d(.), d sin = cos d(.)
            const double da = th_i.d[m] - (m == kth ? 1.0 : 0.0);
            const double dvj = (m == kv) ? 1.0 : 0.0;
            const double dgc = (B * cs - G * sn) * da;              // d(G cos + B sin)
            const double dgs = (G * cs + B * sn) * da;              // d(G sin - B cos)
            p.d[m] = fma(vj, dgc, fma(dvj, gc, p.d[m]));
            q.d[m] = fma(vj, dgs, fma(dvj, gs, q.d[m]));
        }
    }
    // g_P = v_i p - Pg_i + Pd_i,  g_Q = v_i q + Qd_i
    Dual<CH> gP, gQ;
    const int kpg = col_pg[i] - c0;
    gP.v = v_i.v * p.v;
    gQ.v = v_i.v * q.v;
#pragma unroll
    for (int m = 0; m < CH; m++) {
        gP.d[m] = fma(v_i.v, p.d[m], v_i.d[m] * p.v) - (m == kpg ? 1.0 : 0.0);
        gQ.d[m] = fma(v_i.v, q.d[m], v_i.d[m] * q.v);
    }
    // uncompress: each structural entry reads the tangent of its column's colour
    unsigned long long jm = 0;
    for (int t = g.yp[i]; t < g.yp[i + 1]; t++) {
        const int j = g.yj[t];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int dst = g.jac_dst[4 * t + u];
            if (dst == -1) continue;
            const int k = ((u & 1) ? col_v[j] : col_th[j]) - c0;
            if (k < 0 || k >= CH) continue;
            double val = 0.0;
#pragma unroll
            for (int m = 0; m < CH; m++)
                if (m == k) val = (u < 2) ? gP.d[m] : gQ.d[m];
            if (dst >= 0) {
                A[dst] = val;
                const unsigned long long b = ordered_bits(val);
                jm = b > jm ? b : jm;
            } else {
                jpv[-(dst + 2)] = val;
            }
        }
    }
    if (kpg >= 0 && kpg < CH) {
        double val = 0.0;
#pragma unroll
        for (int m = 0; m < CH; m++)
            if (m == kpg) val = gP.d[m];
        jpv[g.pg_slot[i]] = val;
    }
    if (jm) atomicMax(jmax, jm);
}

// ---------------------------------------------------------------------------
// fixed-pattern LU refactorisation (row-wise elimination, static pivots)
// ---------------------------------------------------------------------------

// Right-looking refactorisation, pivot steps of every sparse bus k, once all
// levels are done.  Bus block (theta, v) of a PQ bus:
//   u_tt = a_tt, l_vt = a_vt / u_tt, u_vv = a_vv - l_vt u_tv,
//   U row of v:    u_vj = a_vj - l_vt u_tj,
//   L columns:     l_jt = a_jt / u_tt,  l_jv = (a_jv - l_jt u_tv) / u_vv
// for every later variable j of the bus's pattern (a PV bus has theta only), with
// 1/u_tt, l_vt, 1/u_vv, u_tv from the bus's pivot job.  Thread x < n_piv does bus
// x's block, the others one entry j each (positions a_tj, a_vj, a_jt, a_jv).
__device__ __forceinline__ void k_rf_pivot_body(const RfGrid& g, int64_t x) {
    const int64_t e = x - g.n_piv;
    int k = 0, qt = 0, dt = 0, n_rows = 0;
    int4 p = make_int4(-1, -1, -1, -1);             // a_tj, a_vj, a_jt, a_jv
    if (e < 0) {
        k = (int)x;
        qt = g.q0[k];
        dt = g.diagpos[qt];
        n_rows = g.nv[k];
    } else if (e < g.n_pe) {
        k = g.pe_bus[e];
        p = g.pe_pos[e];
    }
    pdl_wait();
    pdl_trigger();
    if (e < 0) {
        const double tau = 1e-14 * __longlong_as_double((long long)*g.jmax);
        const double4_32a pq = g.piv[k];
        if (!(fabs(g.A[dt]) > tau)) atomicOr(g.err, 1);
        g.invdiag[qt] = pq.x;
        if (n_rows == 2) {
            const int dv = g.diagpos[qt + 1];
            if (!(inb(dv, g.nnz) && inb(qt + 1, g.n_x))) return;
            const double uvv = fma(-pq.y, pq.w, g.A[dv]);
            g.A[dv - 1] = pq.y;
            g.A[dv] = uvv;
            g.invdiag[qt + 1] = pq.z;
            if (!(fabs(uvv) > tau)) atomicOr(g.err, 1);
        }
        return;
    }
    if (e >= g.n_pe) return;
    if (!(inb(k, g.n_piv) && inb(p.x, g.nnz) && inb(p.z, g.nnz) && (p.y < 0 || (inb(p.y, g.nnz) && inb(p.w, g.nnz)))))
        return;
    const double4_32a pq = g.piv[k];
    const double lt = g.A[p.z] * pq.x;
    g.A[p.z] = lt;
    if (p.y >= 0) {
        g.A[p.y] = fma(-pq.y, g.A[p.x], g.A[p.y]);
        g.A[p.w] = fma(-lt, pq.w, g.A[p.w]) * pq.z;
    }
}
__global__ void k_rf_pivot(RfGrid g) {
    k_rf_pivot_body(g, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// Pivot quantities of a bus from its block [a_tt a_tv; a_vt a_vv]: 1/u_tt,
// l_vt = a_vt / u_tt, and 1/u_vv = a_tt / det (u_vv = det / a_tt, det = a_tt a_vv -
// a_vt a_tv), so that the two reciprocals 1/a_tt and 1/det are independent (it
// and idet given).  Stored as {1/u_tt, l_vt, 1/u_vv, u_tv}.
__device__ __forceinline__ double rf_det(double att, double atv, double avt, double avv) {
    return fma(att, avv, -(avt * atv));
}
__device__ __forceinline__ void rf_piv_store(const RfGrid& g, int j, double att, double atv, double avt, double it,
                                             double idet, bool two) {
    double lvt = 0.0, iv = 0.0, utv = 0.0;
    if (two) {
        utv = atv;
        lvt = avt * it;
        iv = att * idet;
    }
    if (inb(j, g.n_piv)) {
        double4_32a r;
        r.x = it; r.y = lvt; r.z = iv; r.w = utv;
        g.piv[j] = r;
    }
}
// Pivot jobs of the leaves (buses whose block no level updates), before the
// first level: one thread per job, the block read from A.
__device__ __forceinline__ void k_rf_leaf_piv_body(const RfGrid& g, int njob) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    int pp[4] = {-1, -1, -1, -1}, bus = 0;
    if (q < njob) {
        for (int e = 0; e < 4; e++) pp[e] = g.piv_pos[4 * q + e];
        bus = g.piv_bus[q];
    }
    pdl_wait();
    pdl_trigger();
    if (q >= njob) return;
    double v[4];
    for (int e = 0; e < 4; e++) v[e] = (pp[e] >= 0 && inb(pp[e], g.nnz)) ? g.A[pp[e]] : 0.0;
    const bool two = pp[3] >= 0;
    const double it = 1.0 / v[0];
    const double idet = two ? 1.0 / rf_det(v[0], v[1], v[2], v[3]) : 0.0;
    rf_piv_store(g, bus, v[0], v[1], v[2], it, idet, two);
}
__global__ void k_rf_leaf_piv(RfGrid g, int njob) {
    k_rf_leaf_piv_body(g, njob);
}

// Update step of one level: every target entry a_ij of the level subtracts
// sum_k l_ik u_kj over the buses k of the level whose pattern holds i and j
// (fixed order: bus, then theta before v).  Bus k's pivot step has not run:
// l_it, l_iv and u_vj are formed from k's raw entries and its pivot quantities
// with the operations of the pivot step, so the factors equal those of a pivot
// step before every level, while the pivot steps of all sparse buses run once,
// in one launch, at the end.  The pivot quantities (1/u_tt, l_vt, 1/u_vv, u_tv)
// are formed once per bus by its pivot job, in the launch of the last level
// that updates k's block (the leaves' in a launch before the first level).  No
// entry a group reads is a target of the same level (its bus would depend on
// the level's own buses).
__device__ __forceinline__ double rf_group(const RfGrid& g, int2 d, int2 tu, int2 vu, double acc) {
    if (tu.x < 0) return acc;
    if (!(inb(d.x, g.n_piv) && inb(tu.x, g.nnz) && inb(tu.y, g.nnz) &&
          (d.y < 0 || (inb(vu.x, g.nnz) && inb(vu.y, g.nnz)))))
        return acc;
    const double4_32a pq = g.piv[d.x];
    const double lt = g.A[tu.x] * pq.x;
    const double ut = g.A[tu.y];
    if (d.y >= 0) {
        const double lv = fma(-lt, pq.w, g.A[vu.x]) * pq.z;
        const double uv = fma(-pq.y, ut, g.A[vu.y]);
        acc = fma(lt, ut, acc);
        return fma(lv, uv, acc);
    }
    return fma(lt, ut, acc);
}

// Targets [t0, t0 + nt) of one level; the first 4 * njob of them are the quads of
// the level's pivot jobs j0 .. j0 + njob - 1 (lane e of job q: entry e of the bus's
// block a_tt, a_tv, a_vt, a_vv, a target of this level or an empty lane).
//
// The plan's arrays do not change, so a thread reads its target's groups and its pivot
// job's positions before it waits for the previous level, and the next level's CTAs start
// as soon as this one's wait is over: between two levels only the values' loads, their
// FMAs and the hand-over remain.  First-order derivatives at 9241 buses 894 -> 783 us (74
// launches), eight Newton re-solves at 1354 buses 1203 -> 1124 us.
struct RfPre {
    int p, pos3, pp, bus;
    int2 d, tu, vu, x[2][3];
    int64_t x0, x1;
};
__device__ __forceinline__ void rf_load(const RfGrid& g, int64_t t0, int64_t nt, int j0, int njob, int64_t tl,
                                        RfPre& r) {
    r.p = r.pos3 = r.pp = -1;
    r.bus = 0;
    r.d = make_int2(0, 0);
    r.tu = r.vu = make_int2(-1, 0);
    r.x0 = r.x1 = 0;
    if (tl < nt) {
        const int64_t t = t0 + tl;
        r.p = g.tgt_pos[t];
        r.d = g.grp[3 * t];
        r.tu = g.grp[3 * t + 1];
        r.vu = g.grp[3 * t + 2];
        r.x0 = g.xptr[t];
        r.x1 = g.xptr[t + 1];
    }
    if (tl < 4 * (int64_t)njob) {
        const int64_t q = j0 + (tl >> 2);
        r.pos3 = g.piv_pos[4 * q + 3];
        r.pp = g.piv_pos[4 * q + (tl & 3)];
        r.bus = g.piv_bus[q];
    }
#pragma unroll
    for (int m = 0; m < 2; m++)
#pragma unroll
        for (int k = 0; k < 3; k++) r.x[m][k] = r.x0 + m < r.x1 ? g.xgrp[3 * (r.x0 + m) + k] : make_int2(-1, 0);
}
// All lanes of a warp call it with consecutive tl.
__device__ __forceinline__ void rf_apply(const RfGrid& g, int njob, int64_t tl, const RfPre& r) {
    double nv = 0.0;
    if (r.p >= 0 && inb(r.p, g.nnz)) {
        double acc = rf_group(g, r.d, r.tu, r.vu, 0.0);
        if (r.x0 < r.x1) acc = rf_group(g, r.x[0][0], r.x[0][1], r.x[0][2], acc);
        if (r.x0 + 1 < r.x1) acc = rf_group(g, r.x[1][0], r.x[1][1], r.x[1][2], acc);
        int64_t c = r.x0 + 2;
        for (; c + 1 < r.x1; c += 2) {
            const int2 da = g.xgrp[3 * c], tua = g.xgrp[3 * c + 1], vua = g.xgrp[3 * c + 2];
            const int2 db = g.xgrp[3 * c + 3], tub = g.xgrp[3 * c + 4], vub = g.xgrp[3 * c + 5];
            acc = rf_group(g, da, tua, vua, acc);
            acc = rf_group(g, db, tub, vub, acc);
        }
        if (c < r.x1) acc = rf_group(g, g.xgrp[3 * c], g.xgrp[3 * c + 1], g.xgrp[3 * c + 2], acc);
        nv = g.A[r.p] - acc;
        g.A[r.p] = nv;
    }
    // pivot jobs: the quads are whole within a warp, and a warp that holds any of
    // them runs the shuffles with all its lanes
    if (tl - (int64_t)(threadIdx.x & 31) < 4 * (int64_t)njob) {
        const int e = (int)(tl & 3);
        const bool mine = tl < 4 * (int64_t)njob;
        double v = nv;
        if (mine && r.p < 0) v = (r.pp >= 0 && inb(r.pp, g.nnz)) ? g.A[r.pp] : 0.0;
        const int b = (int)(threadIdx.x & 28);
        const double att = __shfl_sync(0xffffffffu, v, b);
        const double atv = __shfl_sync(0xffffffffu, v, b + 1);
        const double avt = __shfl_sync(0xffffffffu, v, b + 2);
        const double avv = __shfl_sync(0xffffffffu, v, b + 3);
        // the two reciprocals in one division: 1/a_tt on lane 0 of the quad, 1/det on lane 3
        const double x = e == 0 ? att : (e == 3 && r.pos3 >= 0 ? rf_det(att, atv, avt, avv) : 1.0);
        const double rx = 1.0 / x;
        const double idet = __shfl_sync(0xffffffffu, rx, b + 3);
        if (mine && e == 0) rf_piv_store(g, r.bus, att, atv, avt, rx, idet, r.pos3 >= 0);
    }
}
__device__ __forceinline__ void k_rf_update_body(const RfGrid& g, int64_t t0, int64_t nt, int j0, int njob) {
    const int64_t tl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    RfPre r;
    rf_load(g, t0, nt, j0, njob, tl, r);
    pdl_wait();
    pdl_trigger();
    rf_apply(g, njob, tl, r);
}

// Levels l0 .. l1 - 1, of at most kRfThreads targets each, in one CTA: a CTA barrier between
// two of them takes less than a launch.  A thread reads its target's groups of the next
// level before the barrier.  The reduced Hessian at 118 buses (13 levels) 176 -> 172 us.
// (Wider levels on a cluster of 8 CTAs with a cluster barrier between them were slower
// than their launches: eight re-solves at 1354 buses 1081 -> 1113 us.)
constexpr int kRfThreads = 512;
__device__ __forceinline__ void rf_levels_body(const RfGrid& g, int l0, int l1) {
    int4 lv = g.lev[l0];                                    // first target, targets, first pivot job, jobs
    RfPre r;
    rf_load(g, lv.x, lv.y, lv.z, lv.w, threadIdx.x, r);
    pdl_wait();
    pdl_trigger();
    for (int l = l0; l < l1; l++) {
        rf_apply(g, lv.w, threadIdx.x, r);
        if (l + 1 < l1) {
            lv = g.lev[l + 1];
            rf_load(g, lv.x, lv.y, lv.z, lv.w, threadIdx.x, r);
            __syncthreads();
        }
    }
}
__global__ void __launch_bounds__(kRfThreads) k_rf_levels(RfGrid g, int l0, int l1) { rf_levels_body(g, l0, l1); }
__global__ void k_rf_update(RfGrid g, int64_t t0, int64_t nt, int j0, int njob) {
    k_rf_update_body(g, t0, nt, j0, njob);
}

// Dense trailing block [t0, n_x) as a tiled right-looking LU over TB x TB tiles
// of a row-major scratch copy, spread over many SMs (GB300 runs FP64 on the
// CUDA cores at 2 lane-FMAs per clock per SM, so one CTA would need T^3 / 3
// FMAs on a single SM).  Static diagonal pivots, unit lower L.  One launch per
// tile column: launch k (k = -1 .. nt - 1) factors column c = k + 1 and holds
//   panel CTAs     one per tile (i, c) and (c, i), i > c: the tile and the
//                  diagonal tile take their last update (column k), the
//                  diagonal tile is factored, and L_ic = A_ic U_cc^{-1} or
//                  U_ci = L_cc^{-1} A_ci is stored
//   a diagonal CTA that factors tile (k, k) once more and stores its L and U:
//                  the panel CTAs of launch k - 1 read that tile, so it is only
//                  overwritten one launch later
//   trailing CTAs  A_ij -= L_ik U_kj for every tile i, j > c.
// Every CTA that needs the factored diagonal tile factors it itself from the
// same inputs with the same code, so all copies agree bit for bit; no launch
// reads a tile that another of its CTAs writes.  The diagonal tile is
// eliminated without divisions (cross-multiplied steps with an exact
// power-of-two rescale): the trailing block after step j is s_{j+1} times the
// ordinary one, so u_rc = a_rc / s_r (r <= c), l_rc = a_rc / a_cc (r > c) and
// 1 / u_cc = s_c / a_cc, with one division per column for 1 / a_cc.
constexpr int kTailTB = 16;

// Entry (i, j) of the dense tail's triangles of the unit-diagonal factors L'', U' and of
// their transposes, from a_ij, a_ji, the smaller index's diagonal and both inverse diagonals.
__device__ __forceinline__ void tail_tri(double* triLd, double* triUd, double* triUtd, double* triLtd, int T, int i,
                                         int j, double aij, double aji, double amin, double ii, double ij) {
    if (i > j) {
        const int o = j * (T - 1) - j * (j - 1) / 2 + (i - j - 1);
        triLd[o] = aij * amin * ii;                   // L''_ij
        triUtd[o] = aji * ij;                         // (U'^T)_ij = U'_ji
    } else if (i < j) {
        const int o = j * (j - 1) / 2 + i;
        triUd[o] = aij * ii;                          // U'_ij
        triLtd[o] = aji * amin * ij;                  // (L''^T)_ij = L''_ji
    }
}

__device__ __forceinline__ void k_tail_gather_body(RfGrid g) {
    const int T = g.T;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int p = idx < T * T ? g.tail_pos[idx] : -1;
    pdl_wait();
    pdl_trigger();
    if (idx >= T * T) return;
    g.tailD[idx] = (p >= 0 && inb(p, g.nnz)) ? g.A[p] : 0.0;
}
__global__ void k_tail_gather(RfGrid g) {
    k_tail_gather_body(g);
}

// Entry p of a TB x TB tile in shells of decreasing min(r, c) (p = 0 is the
// last diagonal entry): the entries with r, c > j are exactly p < (TB-1-j)^2.
__device__ __forceinline__ void tail_shell_entry(int p, int& r, int& c) {
    constexpr int TB = kTailTB;
    int q = (int)sqrtf((float)p);
    q += (q + 1) * (q + 1) <= p;
    q -= q * q > p;
    const int m = TB - 1 - q, o = p - q * q;
    r = o <= q ? m : m + (o - q);
    c = o == 0 ? m : (o <= q ? m + o : m);
}

// Eliminates the tile at D (leading dimension ld, unit-padded beyond kb) without
// divisions: afterwards D[r][c] = s_{min(r,c)} a_rc (a the ordinary elimination's values
// when the entry is final), S[c] = s_c and Rd[c] = 1 / D[c][c].  Run by the CTA's first
// 256 threads, which meet at named barrier 1.
__device__ __forceinline__ void tail_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void tail_factor(double* D, int ld, int kb, double* S, double* Rd) {
    constexpr int TB = kTailTB;
    const int t = threadIdx.x;
    int er = 0, ec = 0;
    tail_shell_entry(min(t, (TB - 1) * (TB - 1) - 1), er, ec);
    double own = D[er * ld + ec];
#pragma unroll
    for (int j = 0; j < TB - 1; j++) {
        if (j >= kb - 1) break;
        const int na = (TB - 1 - j) * (TB - 1 - j);
        if ((t & ~31) < na) {                            // the same for the warp
            const double d = D[j * ld + j];
            const int sh = pivot_shift(d);
            double v = fma(d, own, -(D[er * ld + j] * D[j * ld + ec]));
            if (sh) v = scale_pow2(v, sh);
            if (t < na) {
                own = v;
                D[er * ld + ec] = v;
            }
        }
        tail_sync();
    }
    if (t < 32) {
        // s_t: the product of the scaled pivots before t
        const double d = t < kb - 1 ? D[t * ld + t] : 1.0;
        double st = scale_pow2(d, pivot_shift(d));
        st = __shfl_up_sync(0xffffffffu, st, 1);
        if (t == 0) st = 1.0;
#pragma unroll
        for (int o = 1; o < TB; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, st, o);
            if (t >= o) st *= u;
        }
        if (t < TB) {
            S[t] = t < kb ? st : 0.0;
            Rd[t] = t < kb ? 1.0 / D[t * ld + t] : 0.0;
        }
    }
    tail_sync();
}

// Loads a TB x TB tile of the row-major T x T scratch at (i0, j0), rb x cb live.
__device__ __forceinline__ void tail_load(double (*X)[kTailTB + 1], const double* D, int T, int i0, int j0, int rb,
                                          int cb) {
    const int r = threadIdx.x / kTailTB, c = threadIdx.x % kTailTB;   // lanes along a row (coalesced)
    X[r][c] = (r < rb && c < cb) ? D[(size_t)(i0 + r) * T + j0 + c] : 0.0;
}

// The diagonal tile of column c0 / TB with its last update (column kk0 / TB,
// if kk0 >= 0): Dk = A_cc - L_ck U_kc, unit-padded beyond kb.  Uses Lk and Uk.
__device__ __forceinline__ void tail_diag_tile(const RfGrid& g, int c0, int kb, int kk0, double (*Dk)[kTailTB + 1],
                                               double (*Lk)[kTailTB + 1], double (*Uk)[kTailTB + 1]) {
    constexpr int TB = kTailTB;
    const int T = g.T, t = threadIdx.x, r = t / TB, c = t % TB;
    const double* D = g.tailD;
    const double a = (r < kb && c < kb) ? D[(size_t)(c0 + r) * T + c0 + c] : (r == c ? 1.0 : 0.0);
    if (kk0 >= 0) {
        tail_load(Lk, D, T, c0, kk0, kb, TB);
        tail_load(Uk, D, T, kk0, c0, TB, kb);
    }
    __syncthreads();
    double acc = 0.0;
    if (kk0 >= 0) {
#pragma unroll
        for (int q = 0; q < TB; q++) acc = fma(Lk[r][q], Uk[q][c], acc);
    }
    Dk[r][c] = a - acc;
    __syncthreads();
}

__device__ __forceinline__ void k_tail_step_body(RfGrid g, int k) {
    constexpr int TB = kTailTB;
    __shared__ double Dk[TB][TB + 1];
    __shared__ double X[TB][TB + 1];
    __shared__ double Lk[TB][TB + 1];
    __shared__ double Uk[TB][TB + 1];
    __shared__ double Xk[TB][TB + 1];
    __shared__ double S[TB], Rd[TB];
    const int T = g.T, nt = (T + TB - 1) / TB;
    const int t = threadIdx.x;
    const int c = k + 1, c0 = c * TB, k0 = k * TB;
    const int U = c < nt ? nt - c - 1 : 0;
    double* D = g.tailD;
    int b = (int)blockIdx.x;
    if (b < 2 * U) {
        // panel CTA: tile (i, c) (L) for b < U, tile (c, i) (U) otherwise
        const bool ltile = b < U;
        const int o0 = c0 + ((ltile ? b : b - U) + 1) * TB, ob = min(TB, T - o0);
        const int kb = min(TB, T - c0);
        // own tile and its last update: A_ic - L_ik U_kc, or A_ci - L_ck U_ki
        if (ltile) {
            tail_load(X, D, T, o0, c0, ob, kb);
            if (k >= 0) tail_load(Xk, D, T, o0, k0, ob, TB);   // L_ik
        } else {
            tail_load(X, D, T, c0, o0, kb, ob);
            if (k >= 0) tail_load(Xk, D, T, k0, o0, TB, ob);   // U_ki
        }
        tail_diag_tile(g, c0, kb, k >= 0 ? k0 : -1, Dk, Lk, Uk);   // its barriers also cover X, Xk
        if (k >= 0) {
            const int r = t / TB, cc = t % TB;
            double acc = 0.0;
#pragma unroll
            for (int q = 0; q < TB; q++)
                acc = ltile ? fma(Xk[r][q], Uk[q][cc], acc) : fma(Lk[r][q], Xk[q][cc], acc);
            X[r][cc] -= acc;
        }
        tail_factor(&Dk[0][0], TB + 1, kb, S, Rd);   // begins by reading only Dk; its barriers cover X
        // multipliers in place: u_jc / u_jj = Dk[j][c] Rd[j] above the diagonal,
        // l_rj = Dk[r][j] Rd[j] below it
        {
            const int r = t / TB, cc = t % TB;
            if (r != cc) Dk[r][cc] *= Rd[min(r, cc)];
            __syncthreads();
        }
        if (ltile) {
            // X U_cc = A_ic, unscaled (x_rj u_jj), with the multipliers u_jc / u_jj;
            // the rows are independent, each in TB lanes (one per column)
            const int r = t / TB, cl = t % TB;
            double x = X[r][cl];
#pragma unroll
            for (int j = 0; j < TB - 1; j++) {
                if (j < kb - 1) {
                    const double xj = __shfl_sync(0xffffffffu, x, j, TB);
                    if (cl > j) x = fma(-xj, Dk[j][cl], x);
                }
            }
            // 1 / u_cc = s_c / Dk[c][c]
            if (r < ob && cl < kb) D[(size_t)(o0 + r) * T + c0 + cl] = x * (S[cl] * Rd[cl]);
        } else {
            // L_cc Y = A_ci with unit L; the columns are independent, each in TB
            // lanes (one per row)
            const int col = t / TB, r = t % TB;
            double y = X[r][col];
#pragma unroll
            for (int j = 0; j < TB - 1; j++) {
                if (j < kb - 1) {
                    const double yj = __shfl_sync(0xffffffffu, y, j, TB);
                    if (r > j) y = fma(-Dk[r][j], yj, y);
                }
            }
            if (r < kb && col < ob) D[(size_t)(c0 + r) * T + o0 + col] = y;
        }
        return;
    }
    b -= 2 * U;
    if (k >= 0 && b == 0) {
        // diagonal CTA: factor tile (k, k) with its last update (column k - 1) and store
        // U (r <= c: Dk / s_r) and L (r > c: Dk / Dk[c][c])
        const int kb = min(TB, T - k0);
        tail_diag_tile(g, k0, kb, k >= 1 ? k0 - TB : -1, Dk, Lk, Uk);
        tail_factor(&Dk[0][0], TB + 1, kb, S, Rd);
        const int r = t / TB, cl = t % TB;
        if (t < TB) Xk[0][t] = t < kb ? 1.0 / S[t] : 0.0;
        __syncthreads();
        if (r < kb && cl < kb) D[(size_t)(k0 + r) * T + k0 + cl] = r > cl ? Dk[r][cl] * Rd[cl] : Dk[r][cl] * Xk[0][r];
        return;
    }
    if (k >= 0) b -= 1;
    if (k < 0 || b >= U * U) return;
    // trailing tile (i, j), i, j > c: A_ij -= L_ik U_kj
    const int bi = b / U, bj = b % U;
    const int i0 = c0 + (bi + 1) * TB, j0 = c0 + (bj + 1) * TB;
    const int ib = min(TB, T - i0), jb = min(TB, T - j0);
    const int r = t / TB, cc = t % TB;
    const double a = (r < ib && cc < jb) ? D[(size_t)(i0 + r) * T + j0 + cc] : 0.0;
    tail_load(Lk, D, T, i0, k0, ib, TB);
    tail_load(Uk, D, T, k0, j0, TB, jb);
    __syncthreads();
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < TB; q++) acc = fma(Lk[r][q], Uk[q][cc], acc);
    if (r < ib && cc < jb) D[(size_t)(i0 + r) * T + j0 + cc] = a - acc;
}
__global__ void __launch_bounds__(256) k_tail_step(RfGrid g, int k) {
    pdl_wait();
    pdl_trigger();
    k_tail_step_body(g, k);
}

__device__ __forceinline__ void k_tail_scatter_body(RfGrid g) {
    const int T = g.T;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= T * T) return;
    const int p = g.tail_pos[idx];
    const double v = g.tailD[idx];
    if (p >= 0 && inb(p, g.nnz)) g.A[p] = v;
    const int i = idx / T, j = idx - i * T;
    if (i == j) {
        g.invdiag[g.t0 + i] = 1.0 / v;
        const double tau = 1e-14 * __longlong_as_double((long long)*g.jmax);
        if (!(fabs(v) > tau)) atomicOr(g.err, 1);
    }
}
__global__ void k_tail_scatter(RfGrid g) {
    pdl_wait();
    k_tail_scatter_body(g);
}

// The whole dense tail of T <= kTailOne in one CTA, beside the pivot steps (which touch no
// entry of it): LU in shared memory over the same tiles, then the factor, its inverse
// diagonal and the sweeps' triangles.  Such a tail has 2-4 tiles: launched tile by tile it is
// mostly launches, loads and one diagonal tile factored in every CTA, where one SM needs
// few FP64 cycles for all of it (T^3 / 3 multiply-adds at 2 a cycle).  A refactorisation's
// launches after the last level, 5 + ceil(T / 16) of them and k_build_tail, are one: the
// reduced Hessian at 118 buses (T = 16) 185 -> 175 us, eight re-solves at 1354 buses (T = 48)
// 1124 -> 1092 us.  T = 80 would need 95 k cycles of the SM's FP64 pipes (T = 48: 38 k), more
// than the launches it saves.
constexpr int kTailThreads = 512;
struct TailOne {
    double M[kTailOne][kTailOne + 1];
    double Mk[kTailTB][kTailTB + 1];   // multipliers of the current diagonal tile
    double S[kTailTB], Rd[kTailTB], inv[kTailOne];
};
__device__ __forceinline__ void tail_one(const RfGrid& g, TailOne& s) {
    constexpr int TB = kTailTB, LD = kTailOne + 1, Q = kTailOne * kTailOne / kTailThreads;
    const int T = g.T, nt = (T + TB - 1) / TB, Tp = nt * TB, t = threadIdx.x;
    int pos[Q];
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int e = t + q * kTailThreads, i = e / Tp, j = e - i * Tp;
        pos[q] = e < Tp * Tp && i < T && j < T ? g.tail_pos[i * T + j] : -1;
        if (pos[q] >= 0 && !inb(pos[q], g.nnz)) pos[q] = -1;
    }
    pdl_wait();
    pdl_trigger();
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int e = t + q * kTailThreads, i = e / Tp, j = e - i * Tp;
        if (e < Tp * Tp) s.M[i][j] = pos[q] >= 0 ? g.A[pos[q]] : (i == j && i >= T ? 1.0 : 0.0);
    }
    __syncthreads();
    for (int k0 = 0; k0 < Tp; k0 += TB) {
        const int kb = min(TB, T - k0), R = Tp - k0 - TB;
        if (t < 256) {
            tail_factor(&s.M[k0][k0], LD, kb, s.S, s.Rd);
            // l_rc = D[r][c] / D[c][c] (the multiplier too), u_rc = D[r][c] / s_r with u_rc / u_rr the multiplier
            const int r = t / TB, c = t % TB;
            const double v = s.M[k0 + r][k0 + c], m = v * s.Rd[min(r, c)];
            if (r != c) s.Mk[r][c] = m;
            s.M[k0 + r][k0 + c] = r > c ? m : (r < kb ? v * (1.0 / s.S[r]) : v);
        }
        __syncthreads();
        // panels, TB lanes to a row below (X U_kk = A_ik) or a column to the right (L_kk Y = A_kj)
        for (int h = t / TB; h < 2 * R; h += kTailThreads / TB) {
            const bool low = h < R;                       // the same for the warp
            const int o = k0 + TB + (low ? h : h - R), l = t % TB;
            double* at = low ? &s.M[o][k0 + l] : &s.M[k0 + l][o];
            double x = *at;
#pragma unroll
            for (int j = 0; j < TB - 1; j++) {
                const double xj = __shfl_sync(0xffffffffu, x, j, TB);
                if (l > j) x = fma(-xj, low ? s.Mk[j][l] : s.Mk[l][j], x);
            }
            *at = low ? x * (s.S[l] * s.Rd[l]) : x;
        }
        __syncthreads();
        for (int e = t; e < R * R; e += kTailThreads) {
            const int i = k0 + TB + e / R, j = k0 + TB + e % R;
            double acc = 0.0;
#pragma unroll
            for (int q = 0; q < TB; q++) acc = fma(s.M[i][k0 + q], s.M[k0 + q][j], acc);
            s.M[i][j] -= acc;
        }
        __syncthreads();
    }
    if (t < T) {
        const double v = s.M[t][t], tau = 1e-14 * __longlong_as_double((long long)*g.jmax), r = 1.0 / v;
        s.inv[t] = r;
        g.invdiag[g.t0 + t] = r;
        if (!(fabs(v) > tau)) atomicOr(g.err, 1);
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int e = t + q * kTailThreads, i = e / Tp, j = e - i * Tp;
        if (e >= Tp * Tp || i >= T || j >= T) continue;
        if (pos[q] >= 0) g.A[pos[q]] = s.M[i][j];
        else s.M[i][j] = 0.0;                             // structurally zero
    }
    __syncthreads();
    for (int e = t; e < T * T; e += kTailThreads) {
        const int i = e / T, j = e - i * T;
        tail_tri(g.triLd, g.triUd, g.triUtd, g.triLtd, T, i, j, s.M[i][j], s.M[j][i], s.M[i > j ? j : i][i > j ? j : i],
                 s.inv[i], s.inv[j]);
    }
}
__device__ __forceinline__ void rf_finish_body(const RfGrid& g) {
    __shared__ TailOne tail;
    if (blockIdx.x == 0) tail_one(g, tail);
    else k_rf_pivot_body(g, (int64_t)(blockIdx.x - 1) * kTailThreads + threadIdx.x);
}
__global__ void __launch_bounds__(kTailThreads) k_rf_finish(RfGrid g) { rf_finish_body(g); }

// Transposed copies of the factor values and of J_p, and the unit-diagonal
// factors of the direction kernel.  With D = diag(U), J_x = L U = D L'' U' where
// L'' = D^-1 L D and U' = D^-1 U are both unit triangular:
//   l''_qc = l_qc u_cc / u_qq (c < q),   u'_qc = u_qc / u_qq (c > q).
// J_x z = b is then L'' y = D^-1 b, U' z = y, and J_x^T psi = r is U'^T u = r,
// L''^T w = u, psi = D^-1 w: no sweep multiplies by a pivot, and D^-1 folds into
// the rows of J_p (SpMul's right-hand sides, SpMulAdd's J_p^T psi).  One thread
// per position of A (row arow[i], column col[i]) and per entry of J_p.
__device__ __forceinline__ double unit_scale(const double* A, const int* diagpos, const double* invdiag, int r,
                                             int c) {
    return c < r ? A[diagpos[c]] * invdiag[r] : (c > r ? invdiag[r] : 0.0);
}
__global__ void k_transpose_values(int nnz, const int* __restrict__ tpos, const int* __restrict__ arow,
                                   const int* __restrict__ col, const int* __restrict__ diagpos,
                                   const double* __restrict__ A, const double* __restrict__ invdiag,
                                   double* __restrict__ Ad, double* __restrict__ Atd,
                                   int nnz_jp, const int* __restrict__ jpt_src, const int* __restrict__ jpt_row,
                                   const double* __restrict__ jpv, double* __restrict__ jptv,
                                   double* __restrict__ jptvd) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nnz) {
        const int r = arow[i], c = col[i];
        const double at = A[tpos[i]];
        Ad[i] = r == c ? 1.0 : A[i] * unit_scale(A, diagpos, invdiag, r, c);
        Atd[i] = r == c ? 1.0 : at * unit_scale(A, diagpos, invdiag, c, r);
    }
    if (i < nnz_jp) {
        const double v = jpv[jpt_src[i]];
        jptv[i] = v;
        jptvd[i] = v * invdiag[jpt_row[i]];
    }
}

// The four packed triangles of the dense tail for the sweeps, one thread per
// (i, j) of the T x T block; pos maps (i, j) to A (-1: structurally zero).
// x[r] *= s[r] for the first n rows of an n x N row-major block (leading dimension ld)
__global__ void k_scale_rows(int n, int N, const double* __restrict__ s, double* x, int64_t ld) {
    const int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= (int64_t)n * N) return;
    const int r = (int)(it / N), c = (int)(it - (int64_t)r * N);
    x[(int64_t)r * ld + c] *= s[r];
}

// The dense tail's triangles of the unit-diagonal factors L'', U' and their transposes.
__global__ void k_build_tail(int T, int t0, const int* __restrict__ pos, const double* __restrict__ A,
                             const double* __restrict__ invdiag, double* triLd, double* triUd, double* triUtd,
                             double* triLtd) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= T * T) return;
    int i = idx / T, j = idx - i * T;
    if (i == j) return;
    int pij = pos[idx], pji = pos[j * T + i];
    tail_tri(triLd, triUd, triUtd, triLtd, T, i, j, pij >= 0 ? A[pij] : 0.0, pji >= 0 ? A[pji] : 0.0,
             A[pos[i > j ? j * T + j : i * T + i]], invdiag[t0 + i], invdiag[t0 + j]);
}

// ---------------------------------------------------------------------------
// the direction kernel: Algorithm 2 for a slice of directions per CTA
// ---------------------------------------------------------------------------

// Narrow levels (fewer than blockDim / 2 (bus, direction) items): every row's dot
// product is split over ks adjacent lanes of a warp, ks a power of two up to the
// cap (at most 32) and at most half the row, as long as the items still fit in the
// CTA's threads.  1: no split.
__device__ __forceinline__ int split_lanes(int nb, int D, int maxext, int cap) {
    const int base = nb * D;
    if (2 * base > (int)blockDim.x) return 1;
    int ks = 1;
    while (2 * ks <= cap && 2 * base * ks <= (int)blockDim.x && 2 * ks <= maxext) ks *= 2;
    return ks;
}

// a0 -= sum_e v0[e] x[col[e]], a1 -= sum_e v1[e] x[col[e]] over e in [e0, e1) of
// one bus block (two rows sharing their columns when TWO).  Unrolled by 4 so
// that each lane has four independent loads in flight, with one FMA chain per
// row: the FP64 pipe takes one warp instruction per 64 cycles per sub-partition,
// far longer than the chain's latency, so a second accumulator would only cost
// an extra FP64 add.
//
// TWO is chosen per warp (any lane with a second row): a predicated FP64
// instruction occupies the pipe even with its lanes off, so warps of
// single-row buses must not issue the second row at all.  In a mixed warp the
// single-row lanes run the second row on a copy of their first (r1 == r0) and
// ignore the result.
// CMASK: x of a row whose bit in cmask is clear is zero and is not read.
__device__ __forceinline__ bool mask_get(const unsigned* m, int q) { return (m[q >> 5] >> (q & 31)) & 1u; }
template <bool CMASK>
__device__ __forceinline__ double ldx(const double* X, int i, int64_t ld, int64_t c, const unsigned* cmask,
                                      int nrows) {
    return (inb(i, nrows) && (!CMASK || mask_get(cmask, i))) ? X[(int64_t)i * ld + c] : 0.0;
}
// n, or 0 when a row part [r0, r0 + n) or [r1, r1 + n) would leave the nnz
// positions of the pattern (bounds build only; the item is then left as it is)
__device__ __forceinline__ int part_len(int n, int r0, int r1, int nnz) {
    return (inb(r0, nnz + 1) && inb(r0 + n, nnz + 1) && inb(r1, nnz + 1) && inb(r1 + n, nnz + 1)) ? n : 0;
}
// X[q][c] = v for a row q that must lie below nrows (checked in the bounds build)
__device__ __forceinline__ void stx(double* X, int q, int64_t ld, int64_t c, double v, int nrows) {
    if (inb(q, nrows)) X[(int64_t)q * ld + c] = v;
}
template <bool TWO, bool CMASK = false>
__device__ __forceinline__ void block_sub(const int* __restrict__ col, const double* __restrict__ vals, int r0, int r1,
                                          int e0, int e1, const double* X, int64_t ld, int64_t c, double& a0,
                                          double& a1, const unsigned* cmask = nullptr, int nrows = 0x7fffffff) {
    int e = e0;
    for (; e + 4 <= e1; e += 4) {
        const int i0 = col[r0 + e], i1 = col[r0 + e + 1], i2 = col[r0 + e + 2], i3 = col[r0 + e + 3];
        const double x0 = ldx<CMASK>(X, i0, ld, c, cmask, nrows), x1 = ldx<CMASK>(X, i1, ld, c, cmask, nrows);
        const double x2 = ldx<CMASK>(X, i2, ld, c, cmask, nrows), x3 = ldx<CMASK>(X, i3, ld, c, cmask, nrows);
        a0 = fma(-vals[r0 + e], x0, a0);
        a0 = fma(-vals[r0 + e + 1], x1, a0);
        a0 = fma(-vals[r0 + e + 2], x2, a0);
        a0 = fma(-vals[r0 + e + 3], x3, a0);
        if constexpr (TWO) {
            a1 = fma(-vals[r1 + e], x0, a1);
            a1 = fma(-vals[r1 + e + 1], x1, a1);
            a1 = fma(-vals[r1 + e + 2], x2, a1);
            a1 = fma(-vals[r1 + e + 3], x3, a1);
        }
    }
    for (; e < e1; e++) {
        const double xv = ldx<CMASK>(X, col[r0 + e], ld, c, cmask, nrows);
        a0 = fma(-vals[r0 + e], xv, a0);
        if constexpr (TWO) a1 = fma(-vals[r1 + e], xv, a1);
    }
}

// a0 -= sum v0[e] x[col[e]], a1 likewise, over e = e0, e0 + step, ... < n: the share of
// one lane of a split row (adjacent lanes read adjacent entries)
template <bool TWO, bool CMASK>
__device__ __forceinline__ void strided_sub(const int* __restrict__ col, const double* __restrict__ vals, int r0,
                                            int r1, int e, int n, int step, const double* X, int64_t ld, int64_t c,
                                            double& a0, double& a1, const unsigned* cmask, int nrows) {
    for (; e + step < n; e += 2 * step) {
        const int i0 = col[r0 + e], i1 = col[r0 + e + step];
        const double x0 = ldx<CMASK>(X, i0, ld, c, cmask, nrows), x1 = ldx<CMASK>(X, i1, ld, c, cmask, nrows);
        a0 = fma(-vals[r0 + e], x0, a0);
        a0 = fma(-vals[r0 + e + step], x1, a0);
        if constexpr (TWO) {
            a1 = fma(-vals[r1 + e], x0, a1);
            a1 = fma(-vals[r1 + e + step], x1, a1);
        }
    }
    if (e < n) {
        const double xv = ldx<CMASK>(X, col[r0 + e], ld, c, cmask, nrows);
        a0 = fma(-vals[r0 + e], xv, a0);
        if constexpr (TWO) a1 = fma(-vals[r1 + e], xv, a1);
    }
}

// sum of a lane's partial sums over the ks adjacent lanes of its item (all 32 lanes of
// the warp take part; ks divides 32)
__device__ __forceinline__ void split_sum(int ks, bool wtwo, double& s0, double& s1) {
    for (int off = ks >> 1; off > 0; off >>= 1) {
        s0 += __shfl_down_sync(0xffffffffu, s0, off, ks);
        if (wtwo) s1 += __shfl_down_sync(0xffffffffu, s1, off, ks);
    }
}

// warp-uniform choice of the two-row path (lanes that left the item loop do not vote)
__device__ __forceinline__ bool warp_any(bool p) { return __any_sync(__activemask(), p); }

// forward sweep over the L pattern: x_q = b_q - sum_{c<q} v_qc x_c
template <bool TWO>
__device__ __forceinline__ void fwd_finish(const DirGrid& g, const double* __restrict__ vals, double* X, int64_t ld,
                                           int64_t c, int q, bool two, int pos_vt, double a0, double a1) {
    stx(X, q, ld, c, a0, g.n_x);
    if constexpr (TWO) {
        a1 = fma(-vals[pos_vt], a0, a1);
        if (two) stx(X, q + 1, ld, c, a1, g.n_x);
    }
}

// One level of a sweep is flattened over (bus, direction) items, or, when the
// level is too narrow to give every warp work, over (bus, direction, lane of the
// row) with the row's lanes adjacent in a warp.  Each bus block is described by one packed slot
//   forward:  {q, n, rp, rpv}  theta row q, n columns left of the bus, L parts of
//             the theta row at rp and of the v row at rpv (-1 for a PV bus)
//   backward: {q, n, ue0, ue1} U parts right of the bus at ue0 / ue1 (-1: PV)
// so an item needs a single dependent load before its row data; the next
// item's slot is prefetched while the current one is computed.
// EXT: subtract the row parts only (the dense tail's external phase), no finish.
// mask (optional, forward L sweep with identity W): bit q is set for the theta row q of
// every bus whose x can be nonzero for this CTA's directions; every processed bus
// activates its tree parent, an inactive bus only stores its zeros.  seed: the buses
// whose right-hand side was written (zeroed, then the J_p entries scattered); every
// other active bus has b = 0, so V need not be zeroed beforehand.
__device__ __forceinline__ void mask_set(unsigned* m, int q) { atomicOr(m + (q >> 5), 1u << (q & 31)); }
// activate a bus given its encoded theta row (theta row * 2 + 1 if it has a v row)
__device__ __forceinline__ void mask_bus(unsigned* m, int enc) {
    if (enc < 0) return;
    mask_set(m, enc >> 1);
    if (enc & 1) mask_set(m, (enc >> 1) + 1);
}
template <bool EXT = false, bool CMASK = false>
__device__ void sweep_fwd(const DirGrid& g, const LevelSet& ls, const double* __restrict__ vals, double* X,
                          int64_t ld, int c0, int D, double* part, unsigned* mask = nullptr,
                          const unsigned* seed = nullptr, const unsigned* cmask = nullptr) {
    for (int lev = 0; lev < ls.n_lev; lev++) {
        const int b0 = ls.ptr[lev], nb = ls.ptr[lev + 1] - b0;
        const int4* __restrict__ slots = ls.slots + b0;
        const int ks = split_lanes(nb, D, ls.maxext[lev], g.ks_cap);
        if (ks == 1) {
            const int items = nb * D;
            int it = threadIdx.x;
            int bi = it / D;
            int4 nxt = it < items ? slots[bi] : make_int4(0, 0, 0, -1);
            for (; it < items; it += blockDim.x) {
                const int4 sl = nxt;
                const int d = it - bi * D;
                const int it2 = it + blockDim.x, bi2 = it2 / D;
                if (it2 < items) nxt = slots[bi2];
                const int q = sl.x, rp = sl.z;
                bi = bi2;
                const bool two = sl.w >= 0;
                const int64_t c = c0 + d;
                if (mask && !(inb(q, g.n_x) && mask_get(mask, q))) continue;   // outside the reach: x = 0, never read
                const int rpv = two ? sl.w : rp;
                const int n = part_len(sl.y, rp, rpv, g.nnz);
                const bool has_b = !seed || mask_get(seed, q);
                double a0 = (has_b && inb(q, g.n_x)) ? X[(int64_t)q * ld + c] : 0.0;
                double a1 = (two && has_b && inb(q + 1, g.n_x)) ? X[(int64_t)(q + 1) * ld + c] : 0.0;
                if (warp_any(two)) {
                    block_sub<true, CMASK>(g.col, vals, rp, rpv, 0, n, X, ld, c, a0, a1, cmask, g.n_x);
                    if (EXT) {
                        stx(X, q, ld, c, a0, g.n_x);
                        if (two) stx(X, q + 1, ld, c, a1, g.n_x);
                    } else {
                        fwd_finish<true>(g, vals, X, ld, c, q, two, rpv + n, a0, a1);
                    }
                } else {
                    block_sub<false, CMASK>(g.col, vals, rp, rpv, 0, n, X, ld, c, a0, a1, cmask, g.n_x);
                    if (EXT) stx(X, q, ld, c, a0, g.n_x);
                    else fwd_finish<false>(g, vals, X, ld, c, q, two, rpv + n, a0, a1);
                }
                if (mask) mask_bus(mask, g.bparent[q]);
            }
        } else {
            // narrow level: each row split over ks adjacent lanes, summed by shuffles
            const int total = nb * D * ks;
            const int lane = (int)(threadIdx.x & 31);
            for (int w0 = (int)threadIdx.x - lane; w0 < total; w0 += blockDim.x) {     // warp-uniform
                const int it = w0 + lane, sli = it & (ks - 1), item = it / ks;
                const bool valid = it < total;
                const int bi = valid ? item / D : 0, d = valid ? item - bi * D : 0;
                const int4 sl = valid ? slots[bi] : make_int4(0, 0, 0, -1);
                const int q = sl.x, rp = sl.z;
                const bool two = sl.w >= 0;
                const int rpv = two ? sl.w : rp;
                const bool act = valid && !(mask && !(inb(q, g.n_x) && mask_get(mask, q)));
                const int n = act ? part_len(sl.y, rp, rpv, g.nnz) : 0;
                const int64_t c = c0 + d;
                const bool fin = act && sli == 0;          // the lane that finishes the item
                const bool has_b = fin && (!seed || mask_get(seed, q));
                const double b0 = (has_b && inb(q, g.n_x)) ? X[(int64_t)q * ld + c] : 0.0;
                const double b1 = (two && has_b && inb(q + 1, g.n_x)) ? X[(int64_t)(q + 1) * ld + c] : 0.0;
                const bool wtwo = __any_sync(0xffffffffu, two);   // every lane of the warp is here
                double s0 = 0.0, s1 = 0.0;
                if (wtwo) strided_sub<true, CMASK>(g.col, vals, rp, rpv, sli, n, ks, X, ld, c, s0, s1, cmask, g.n_x);
                else strided_sub<false, CMASK>(g.col, vals, rp, rpv, sli, n, ks, X, ld, c, s0, s1, cmask, g.n_x);
                split_sum(ks, wtwo, s0, s1);
                if (!fin) continue;
                const double a0 = b0 + s0, a1 = b1 + s1;
                if (EXT) {
                    stx(X, q, ld, c, a0, g.n_x);
                    if (two) stx(X, q + 1, ld, c, a1, g.n_x);
                } else if (two) {
                    fwd_finish<true>(g, vals, X, ld, c, q, two, rpv + n, a0, a1);
                } else {
                    fwd_finish<false>(g, vals, X, ld, c, q, two, rpv + n, a0, a1);
                }
                if (mask) mask_bus(mask, g.bparent[q]);
            }
        }
        __syncthreads();
    }
}

// backward sweep over the U pattern: x_q = b_q - sum_{c>q} v_qc x_c
template <bool TWO>
__device__ __forceinline__ void bwd_finish(const DirGrid& g, const double* __restrict__ vals, double* X, int64_t ld,
                                           int64_t c, int q, bool two, int pos_tv, double a0, double a1) {
    if constexpr (TWO) {
        if (two) stx(X, q + 1, ld, c, a1, g.n_x);
        a0 = fma(-vals[pos_tv], two ? a1 : 0.0, a0);
    }
    stx(X, q, ld, c, a0, g.n_x);
}

// rmask (optional): right-hand side rows whose bit is clear are zero and are not read
__device__ void sweep_bwd(const DirGrid& g, const LevelSet& ls, const double* __restrict__ vals, double* X,
                          int64_t ld, int c0, int D, double* part, const unsigned* rmask = nullptr) {
    for (int lev = 0; lev < ls.n_lev; lev++) {
        const int b0 = ls.ptr[lev], nb = ls.ptr[lev + 1] - b0;
        const int4* __restrict__ slots = ls.slots + b0;
        const int ks = split_lanes(nb, D, ls.maxext[lev], g.ks_cap);
        if (ks == 1) {
            const int items = nb * D;
            int it = threadIdx.x;
            int bi = it / D;
            int4 nxt = it < items ? slots[bi] : make_int4(0, 0, 0, -1);
            for (; it < items; it += blockDim.x) {
                const int4 sl = nxt;
                const int d = it - bi * D;
                const int it2 = it + blockDim.x, bi2 = it2 / D;
                if (it2 < items) nxt = slots[bi2];
                const int q = sl.x, ue0 = sl.z;
                const bool two = sl.w >= 0;
                const int ue1 = two ? sl.w : ue0;
                const int n = part_len(sl.y, ue0 - 1, ue1, g.nnz);
                const int64_t c = c0 + d;
                const bool has_b = !rmask || mask_get(rmask, q);
                double a0 = (has_b && inb(q, g.n_x)) ? X[(int64_t)q * ld + c] : 0.0;
                double a1 = (two && has_b && inb(q + 1, g.n_x)) ? X[(int64_t)(q + 1) * ld + c] : 0.0;
                if (warp_any(two)) {
                    block_sub<true>(g.col, vals, ue0, ue1, 0, n, X, ld, c, a0, a1, nullptr, g.n_x);
                    bwd_finish<true>(g, vals, X, ld, c, q, two, ue0 - 1, a0, a1);
                } else {
                    block_sub<false>(g.col, vals, ue0, ue1, 0, n, X, ld, c, a0, a1, nullptr, g.n_x);
                    bwd_finish<false>(g, vals, X, ld, c, q, two, ue0 - 1, a0, a1);
                }
                bi = bi2;
            }
        } else {
            // narrow level: each row split over ks adjacent lanes, summed by shuffles
            const int total = nb * D * ks;
            const int lane = (int)(threadIdx.x & 31);
            for (int w0 = (int)threadIdx.x - lane; w0 < total; w0 += blockDim.x) {     // warp-uniform
                const int it = w0 + lane, sli = it & (ks - 1), item = it / ks;
                const bool valid = it < total;
                const int bi = valid ? item / D : 0, d = valid ? item - bi * D : 0;
                const int4 sl = valid ? slots[bi] : make_int4(0, 0, 0, -1);
                const int q = sl.x, ue0 = sl.z;
                const bool two = sl.w >= 0;
                const int ue1 = two ? sl.w : ue0;
                const int n = valid ? part_len(sl.y, ue0 - 1, ue1, g.nnz) : 0;
                const int64_t c = c0 + d;
                const bool fin = valid && sli == 0;
                const bool has_b = fin && (!rmask || mask_get(rmask, q));
                const double b0 = (has_b && inb(q, g.n_x)) ? X[(int64_t)q * ld + c] : 0.0;
                const double b1 = (two && has_b && inb(q + 1, g.n_x)) ? X[(int64_t)(q + 1) * ld + c] : 0.0;
                const bool wtwo = __any_sync(0xffffffffu, two);   // every lane of the warp is here
                double s0 = 0.0, s1 = 0.0;
                if (wtwo) strided_sub<true, false>(g.col, vals, ue0, ue1, sli, n, ks, X, ld, c, s0, s1, nullptr, g.n_x);
                else strided_sub<false, false>(g.col, vals, ue0, ue1, sli, n, ks, X, ld, c, s0, s1, nullptr, g.n_x);
                split_sum(ks, wtwo, s0, s1);
                if (!fin) continue;
                if (two) bwd_finish<true>(g, vals, X, ld, c, q, two, ue0 - 1, b0 + s0, b1 + s1);
                else bwd_finish<false>(g, vals, X, ld, c, q, two, ue0 - 1, b0 + s0, b1 + s1);
            }
        }
        __syncthreads();
    }
}

// Dense trailing block [t0, t0 + T) of a sweep, column-oriented in shared memory.
// xt[i * D + d] holds row t0 + i of the CTA's directions; tri_g is the packed
// strictly-triangular block (column j contiguous); each column step is
// y_i -= tri_ij y_j.  With tri != NULL the
// triangle is first staged in shared memory (one CTA per SM); with tri == NULL
// it is read through L1, where it is shared by all the CTAs of the SM.
__device__ __forceinline__ int lpack_off(int j, int T) { return j * (T - 1) - j * (j - 1) / 2; }  // rows j+1..T-1
__device__ __forceinline__ int upack_off(int j) { return j * (j - 1) / 2; }                      // rows 0..j-1

// The solve runs over blocks of kTailB columns with two barriers per block:
// the block's diagonal part is solved inside warps (16 lanes hold the block's
// rows of one direction and pass each finished value along with a shuffle),
// then every row below (above, for the backward solve) takes the block's
// contribution in one CTA-wide pass.
constexpr int kTailB = 16;

__device__ __forceinline__ double tri_l(const double* src, int T, int i, int j) { return src[lpack_off(j, T) + (i - j - 1)]; }
__device__ __forceinline__ double tri_u(const double* src, int i, int j) { return src[upack_off(j) + i]; }

template <class Grid>
__device__ void tail_fwd(const Grid& g, const double* __restrict__ tri_g, double* X, int64_t ld, int c0, int D,
                         double* xt, double* tri) {
    const int T = g.T, t0 = g.t0;
    const int ntri = T * (T - 1) / 2;
    if (tri)
        for (int i = threadIdx.x; i < ntri; i += blockDim.x) tri[i] = tri_g[i];
    const double* src = tri ? tri : tri_g;
    for (int it = threadIdx.x; it < T * D; it += blockDim.x) {
        int i = it / D, d = it - i * D;
        xt[it] = X[(int64_t)(t0 + i) * ld + c0 + d];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, l = lane & 15;
    const int hw = (int)(threadIdx.x >> 4), nhw = (int)(blockDim.x >> 4);
    const unsigned hmask = (lane < 16) ? 0x0000ffffu : 0xffff0000u;
    for (int b0 = 0; b0 < T; b0 += kTailB) {
        const int bn = min(kTailB, T - b0);
        // (1) diagonal block: rows b0 + l of direction d, one half-warp per direction
        if (hw < D) {
            double a[kTailB];
#pragma unroll
            for (int m = 0; m < kTailB; m++) a[m] = (m < l && l < bn) ? tri_l(src, T, b0 + l, b0 + m) : 0.0;
            for (int d = hw; d < D; d += nhw) {
                double v = l < bn ? xt[(b0 + l) * D + d] : 0.0;
#pragma unroll
                for (int m = 0; m < kTailB - 1; m++) {
                    const double ym = __shfl_sync(hmask, v, m, 16);
                    v = fma(-a[m], ym, v);
                }
                if (l < bn) xt[(b0 + l) * D + d] = v;
            }
        }
        __syncthreads();
        // (2) rows below the block take its contribution
        const int n = (T - b0 - bn) * D;
        for (int it = threadIdx.x; it < n; it += blockDim.x) {
            const int i = b0 + bn + it / D, d = it % D;
            double v = xt[i * D + d];
            for (int m = 0; m < bn; m++) v = fma(-tri_l(src, T, i, b0 + m), xt[(b0 + m) * D + d], v);
            xt[i * D + d] = v;
        }
        __syncthreads();
    }
    for (int it = threadIdx.x; it < T * D; it += blockDim.x) {
        int i = it / D, d = it - i * D;
        X[(int64_t)(t0 + i) * ld + c0 + d] = xt[it];
    }
    __syncthreads();
}

template <class Grid>
__device__ void tail_bwd(const Grid& g, const double* __restrict__ tri_g, double* X, int64_t ld, int c0, int D,
                         double* xt, double* tri) {
    const int T = g.T, t0 = g.t0;
    const int ntri = T * (T - 1) / 2;
    if (tri)
        for (int i = threadIdx.x; i < ntri; i += blockDim.x) tri[i] = tri_g[i];
    const double* src = tri ? tri : tri_g;
    for (int it = threadIdx.x; it < T * D; it += blockDim.x) {
        int i = it / D, d = it - i * D;
        xt[it] = X[(int64_t)(t0 + i) * ld + c0 + d];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, l = lane & 15;
    const int hw = (int)(threadIdx.x >> 4), nhw = (int)(blockDim.x >> 4);
    const unsigned hmask = (lane < 16) ? 0x0000ffffu : 0xffff0000u;
    for (int be = T; be > 0; be -= kTailB) {
        const int b0 = be > kTailB ? be - kTailB : 0, bn = be - b0;
        // (1) diagonal block, bottom-up: row b0 + l takes the finished values of the rows after it
        if (hw < D) {
            double a[kTailB];
#pragma unroll
            for (int m = 0; m < kTailB; m++) a[m] = (l < m && m < bn) ? tri_u(src, b0 + l, b0 + m) : 0.0;
            for (int d = hw; d < D; d += nhw) {
                double v = l < bn ? xt[(b0 + l) * D + d] : 0.0;
#pragma unroll
                for (int m = kTailB - 1; m > 0; m--) {
                    const double ym = __shfl_sync(hmask, v, m, 16);
                    v = fma(-a[m], ym, v);
                }
                if (l < bn) xt[(b0 + l) * D + d] = v;
            }
        }
        __syncthreads();
        // (2) rows above the block take its contribution
        const int n = b0 * D;
        for (int it = threadIdx.x; it < n; it += blockDim.x) {
            const int i = it / D, d = it - i * D;
            double v = xt[i * D + d];
            for (int m = 0; m < bn; m++) v = fma(-tri_u(src, i, b0 + m), xt[(b0 + m) * D + d], v);
            xt[i * D + d] = v;
        }
        __syncthreads();
    }
    for (int it = threadIdx.x; it < T * D; it += blockDim.x) {
        int i = it / D, d = it - i * D;
        X[(int64_t)(t0 + i) * ld + c0 + d] = xt[it];
    }
    __syncthreads();
}

// Projection (eq. 11/13): y = [lambda^T Hess g + Hess f] v for v = (z, w).
// Gathered bus by bus over the incident branches (no atomics, deterministic):
//   y_v(b)  = d2_b dv_b + A_b dth_b + sum_e ( K_e dv_j - a_e dth_j )
//   y_th(b) = A_b dv_b  + C_b dth_b + sum_e ( b_e dv_j - c_e dth_j )
// plus c''_slack (grad P_slack . v) grad P_slack and c''_k w_Pg_k.
__device__ __forceinline__ double flip_sign(double v, bool flip) {
    // negation through the sign bit (an integer operation, not an FP64 instruction)
    return __longlong_as_double(__double_as_longlong(v) ^ (flip ? (long long)0x8000000000000000ULL : 0LL));
}

// Buses are visited in the order tp_bus (degree descending), so the lanes of a
// warp mostly share their incidence count; each output is one FMA chain; the
// slack-neighbour and Pg terms, which few buses have, are only issued by warps
// that hold such a bus (a predicated FP64 instruction costs its issue slot).
// fold_ut: the launch runs the U'^T sweep over the sparse levels next; its level 0
// (buses without L entries outside their block, so x_theta = b_theta and, for a PQ
// bus, x_v = b_v - u'_tv x_theta) is done here and the sweep starts at level 1.
__device__ void tproj(const DirGrid& g, const double* V, double* T, int64_t ld, int c0, int D, double* sref,
                      bool fold_ut) {
    double c2r = *g.c2ref;
    for (int d = threadIdx.x; d < D; d += blockDim.x) {
        double s = 0.0;
        for (int e = 0; e < g.n_gref; e++)
            if (inb(g.gref_row[e], g.zero_row + 1)) s = fma(g.gref_val[e], V[(int64_t)g.gref_row[e] * ld + c0 + d], s);
        sref[d] = c2r * s;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < g.n_bus * D; it += blockDim.x) {
        int bi = it / D, d = it - bi * D;
        int b = g.tp_bus[bi];
        int64_t c = c0 + d;
        int rth = g.uth[b], rv = g.uv[b];
        const int rows = g.zero_row + 1;
        double dth = inb(rth, rows) ? V[(int64_t)rth * ld + c] : 0.0, dv = inb(rv, rows) ? V[(int64_t)rv * ld + c] : 0.0;
        double ab = g.asum[b];
        double yv = fma(g.d2[b], dv, ab * dth);
        double yth = fma(ab, dv, g.csum[b] * dth);
        int e = g.inc_ptr[b];
        const int e1 = g.inc_ptr[b + 1];
        for (; e + 2 <= e1; e += 2) {
            const int t0 = g.inc_uth[e], v0 = g.inc_uv[e], t1 = g.inc_uth[e + 1], v1 = g.inc_uv[e + 1];
            const double dthj0 = inb(t0, rows) ? V[(int64_t)t0 * ld + c] : 0.0;
            const double dvj0 = inb(v0, rows) ? V[(int64_t)v0 * ld + c] : 0.0;
            const double dthj1 = inb(t1, rows) ? V[(int64_t)t1 * ld + c] : 0.0;
            const double dvj1 = inb(v1, rows) ? V[(int64_t)v1 * ld + c] : 0.0;
            const double4_32a cf0 = g.inc_coef[e], cf1 = g.inc_coef[e + 1];
            yv = fma(cf0.x, dvj0, yv);
            yv = fma(cf0.y, dthj0, yv);
            yth = fma(cf0.z, dvj0, yth);
            yth = fma(cf0.w, dthj0, yth);
            yv = fma(cf1.x, dvj1, yv);
            yv = fma(cf1.y, dthj1, yv);
            yth = fma(cf1.z, dvj1, yth);
            yth = fma(cf1.w, dthj1, yth);
        }
        if (warp_any(e < e1)) {
            if (e < e1) {
                const double4_32a cf = g.inc_coef[e];
                const double dthj = inb(g.inc_uth[e], rows) ? V[(int64_t)g.inc_uth[e] * ld + c] : 0.0;
                const double dvj = inb(g.inc_uv[e], rows) ? V[(int64_t)g.inc_uv[e] * ld + c] : 0.0;
                yv = fma(cf.x, dvj, yv);
                yv = fma(cf.y, dthj, yv);
                yth = fma(cf.z, dvj, yth);
                yth = fma(cf.w, dthj, yth);
            }
        }
        const bool hg = g.has_gref[b];
        if (warp_any(hg)) {
            if (hg) {
                yv = fma(sref[d], g.gref_v[b], yv);
                yth = fma(sref[d], g.gref_th[b], yth);
            }
        }
        if (rth != g.zero_row && inb(rth, rows)) T[(int64_t)rth * ld + c] = flip_sign(yth, true);
        const int l0 = fold_ut ? g.tp_l0[b] : -1;
        if (warp_any(l0 >= 0)) {
            if (l0 >= 0) yv = fma(-g.Atd[l0], yth, yv);   // T_v = -yv + u'_tv yth
        }
        if (inb(rv, rows)) T[(int64_t)rv * ld + c] = flip_sign(yv, rv < g.n_x);
        const int pr = g.pg_row[b];
        if (warp_any(pr >= 0)) {
            if (pr >= 0 && inb(pr, rows)) T[(int64_t)pr * ld + c] = g.pg_curv[b] * V[(int64_t)pr * ld + c];
        }
    }
}

// identity W: the column of direction j of the launch (and of its HW, relative to col0)
__device__ __forceinline__ int id_col(const DirLaunch& L, int j) { return L.colmap ? L.colmap[L.col0 + j] : L.col0 + j; }

// HW = Y_p + J_p^T Psi (Algorithm 2, SpMulAdd): one lane per p row k, directions
// blocked W at a time, so a warp's stores of one direction are consecutive.
template <int W>
__device__ __forceinline__ void muladd_row(const DirGrid& g, const DirLaunch& L, const double* T, int64_t ld, int c0,
                                           int d0, int k) {
    double h[W];
#pragma unroll
    for (int w = 0; w < W; w++) h[w] = T[(int64_t)(g.n_x + k) * ld + d0 + w];
    const int t1 = g.jpt_ptr[k + 1];
    for (int t = g.jpt_ptr[k]; t < t1; t++) {
        const double v = g.jptvd[t];
        if (!inb(g.jpt_row[t], g.n_x)) continue;
        const double* pr = T + (int64_t)g.jpt_row[t] * ld + d0;
#pragma unroll
        for (int w = 0; w < W; w++) h[w] = fma(v, pr[w], h[w]);
    }
#pragma unroll
    for (int w = 0; w < W; w++) L.HW[(int64_t)(id_col(L, c0 + d0 + w) - L.col0) * L.ldhw + k] = h[w];
}

// Algorithm 2 for the directions owned by CTA `cta` of launch L on grid g.
__device__ __forceinline__ void dirs_body(const DirGrid& g, const DirLaunch& L, const int cta, double* part,
                                          double* sref, unsigned* mask_smem) {
    const int c0 = (int)((int64_t)cta * L.N / L.n_cta);
    const int c1 = (int)((int64_t)(cta + 1) * L.N / L.n_cta);
    const int D = c1 - c0;
    if (D <= 0) return;
    // this CTA's directions: row r, local direction d at base[r * ld + d]
    const int64_t ld = L.ld;
    {
        // the CTA's last element lies in the buffers (bounds build; the condition is
        // the same for every thread of the CTA, so leaving here skips no barrier)
        const int64_t first = L.cta_stride ? (int64_t)cta * L.cta_stride : (int64_t)c0;
        const int64_t last = first + (int64_t)g.zero_row * ld + D - 1;
        if (!inb((L.cta_stride ? 0 : c0) + D - 1, ld) || (L.ws_elems > 0 && !inb(last, L.ws_elems))) return;
    }
    const int64_t base = L.cta_stride ? (int64_t)cta * L.cta_stride : (int64_t)c0;
    double* V = L.V + base;
    double* T = L.T + base;
    if (L.phases & PH_WLOAD) {
        for (int it = threadIdx.x; it < g.n_p * D; it += blockDim.x) {
            int k = it / D, d = it - k * D;
            int64_t c = c0 + d;
            double w = L.W ? L.W[c * L.ldw + k] : (k == id_col(L, (int)c) ? 1.0 : 0.0);
            V[(int64_t)(g.n_x + k) * ld + d] = w;
        }
        for (int d = threadIdx.x; d < D; d += blockDim.x) V[(int64_t)g.zero_row * ld + d] = 0.0;
        __syncthreads();
    }
    unsigned* seed = nullptr;
    if ((L.phases & PH_SPMUL) && !L.W && L.use_reach) {
        // identity W with the reach-restricted forward sweep: only the buses of this
        // CTA's J_p columns (all their rows, every direction) and the dense tail are
        // zeroed before the scatter; the forward sweep writes the other rows of the
        // reach, and the rows outside it are zero and never read
        seed = mask_smem + (g.n_x + 31) / 32;
        for (int i = threadIdx.x; i < (g.n_x + 31) / 32; i += blockDim.x) seed[i] = 0u;
        for (int it = threadIdx.x; it < g.T * D; it += blockDim.x) {
            const int i = it / D, d = it - i * D;
            V[(int64_t)(g.t0 + i) * ld + d] = 0.0;
        }
        __syncthreads();
        for (int d = threadIdx.x / 8; d < D; d += blockDim.x / 8) {
            const int k = id_col(L, c0 + d);
            for (int t = g.jpt_ptr[k] + (threadIdx.x & 7); t < g.jpt_ptr[k + 1]; t += 8) {
                const int qb = g.qtheta[g.jpt_row[t]];
                const bool two = qb + 1 < g.n_x && g.qtheta[qb + 1] == qb;
                mask_set(seed, qb);
                if (two) mask_set(seed, qb + 1);
                for (int e = 0; e < D; e++) {
                    V[(int64_t)qb * ld + e] = 0.0;
                    if (two) V[(int64_t)(qb + 1) * ld + e] = 0.0;
                }
            }
        }
        __syncthreads();
        for (int d = threadIdx.x / 8; d < D; d += blockDim.x / 8) {
            const int k = id_col(L, c0 + d);
            for (int t = g.jpt_ptr[k] + (threadIdx.x & 7); t < g.jpt_ptr[k + 1]; t += 8)
                V[(int64_t)g.jpt_row[t] * ld + d] = -g.jptvd[t];
        }
        __syncthreads();
    } else if ((L.phases & PH_SPMUL) && !L.W) {
        // identity W: -B column c is minus column col0 + c of J_p; zero the x rows
        // (stores only), then scatter the few entries of each column
        const int rstep = (int)blockDim.x / D;
        if (threadIdx.x < rstep * D) {
            const int d = threadIdx.x % D;
            for (int r = threadIdx.x / D; r < g.n_x; r += rstep) V[(int64_t)r * ld + d] = 0.0;
        }
        __syncthreads();
        for (int d = threadIdx.x / 8; d < D; d += blockDim.x / 8) {
            const int k = id_col(L, c0 + d);
            for (int t = g.jpt_ptr[k] + (threadIdx.x & 7); t < g.jpt_ptr[k + 1]; t += 8)
                V[(int64_t)g.jpt_row[t] * ld + d] = -g.jptvd[t];
        }
        __syncthreads();
    } else if (L.phases & PH_SPMUL) {
        // rows of J_p without entries: -B is zero there (stores only, no loads)
        for (int it = threadIdx.x; it < g.n_jp_zero * D; it += blockDim.x) {
            int r = it / D, d = it - r * D;
            V[(int64_t)g.jp_zero_rows[r] * ld + d] = 0.0;
        }
        for (int it = threadIdx.x; it < g.n_jp_rows * D; it += blockDim.x) {
            int r = it / D, d = it - r * D;
            const int q = g.jp_rows[r];
            double s = 0.0;
            for (int t = g.jp_ptr[q]; t < g.jp_ptr[q + 1]; t++)
                s = fma(g.jpv[t], V[(int64_t)(g.n_x + g.jp_col[t]) * ld + d], s);
            V[(int64_t)q * ld + d] = -s * g.invdiag[q];     // D^-1 B for the unit-diagonal factors
        }
        __syncthreads();
    }
    if (L.use_tail) {
        // identity W: the reach of B's columns (one bit per row; L, U and the tail's
        // external phase in this launch); rows outside it are zero in Z's forward sweep
        unsigned* mask = nullptr;
        if ((L.phases & PH_L) && L.use_reach) {
            mask = mask_smem;
            if (L.reach) {
                const int words = L.reach->words;
                const unsigned* m = L.reach->masks + (int64_t)cta * words;
                for (int i = threadIdx.x; i < words; i += blockDim.x) mask[i] = m[i];
            } else if (seed) {
                for (int i = threadIdx.x; i < (g.n_x + 31) / 32; i += blockDim.x) mask[i] = seed[i];
            } else {
                for (int i = threadIdx.x; i < (g.n_x + 31) / 32; i += blockDim.x) mask[i] = 0u;
                __syncthreads();
                for (int d = threadIdx.x / 8; d < D; d += blockDim.x / 8) {
                    const int k = id_col(L, c0 + d);
                    for (int t = g.jpt_ptr[k] + (threadIdx.x & 7); t < g.jpt_ptr[k + 1]; t += 8) {
                        const int qb = g.qtheta[g.jpt_row[t]];
                        mask_set(mask, qb);
                        if (qb + 1 < g.n_x && g.qtheta[qb + 1] == qb) mask_set(mask, qb + 1);
                    }
                }
            }
            __syncthreads();
        }
        if (L.phases & PH_L) {
            if (mask && L.reach) {
                // the CTA's reach, level by level, precomputed: nothing to skip or grow
                const ReachSched& R = *L.reach;
                const int m0 = R.lev0[cta];
                const LevelSet rs = {R.nlev[cta], R.ptr + m0 + cta, R.slots, R.maxext + m0};
                sweep_fwd<false, true>(g, rs, g.Ad, V, ld, 0, D, part, nullptr, seed, mask);
                sweep_fwd<true, true>(g, g.ef, g.Ad, V, ld, 0, D, part, nullptr, nullptr, mask);
            } else if (mask) {
                sweep_fwd<false, true>(g, g.sf, g.Ad, V, ld, 0, D, part, mask, seed, mask);
                sweep_fwd<true, true>(g, g.ef, g.Ad, V, ld, 0, D, part, nullptr, nullptr, mask);
            } else {
                sweep_fwd(g, g.sf, g.Ad, V, ld, 0, D, part);
                sweep_fwd<true>(g, g.ef, g.Ad, V, ld, 0, D, part);
            }
            tail_fwd(g, g.triLd, V, ld, 0, D, part, nullptr);
        }
        if (L.phases & PH_U) {
            tail_bwd(g, g.triUd, V, ld, 0, D, part, nullptr);
            sweep_bwd(g, g.sb, g.Ad, V, ld, 0, D, part, mask);
        }
    } else {
        if (L.phases & PH_L) sweep_fwd(g, g.lf, g.Ad, V, ld, 0, D, part);
        if (L.phases & PH_U) sweep_bwd(g, g.lb, g.Ad, V, ld, 0, D, part);
    }
    const bool fold_ut = (L.phases & PH_TPROJ) && (L.phases & PH_UT) && L.use_tail && g.sf.n_lev > 0;
    if (L.phases & PH_TPROJ) {
        tproj(g, V, T, ld, 0, D, sref, fold_ut);
        __syncthreads();
    }
    if (L.use_tail) {
        if (L.phases & PH_UT) {
            LevelSet sf = g.sf;
            if (fold_ut) {   // level 0 was done by the projection
                sf.n_lev -= 1;
                sf.ptr += 1;
                sf.maxext += 1;
            }
            sweep_fwd(g, sf, g.Atd, T, ld, 0, D, part);
            sweep_fwd<true>(g, g.ef, g.Atd, T, ld, 0, D, part);
            tail_fwd(g, g.triUtd, T, ld, 0, D, part, nullptr);
        }
        if (L.phases & PH_LT) {
            // psi is only read by SpMulAdd here: rows outside J_p and its ancestors are skipped
            tail_bwd(g, g.triLtd, T, ld, 0, D, part, nullptr);
            sweep_bwd(g, (L.phases & PH_MULADD) ? g.sbr : g.sb, g.Atd, T, ld, 0, D, part);
        }
    } else {
        if (L.phases & PH_UT) sweep_fwd(g, g.lf, g.Atd, T, ld, 0, D, part);
        if (L.phases & PH_LT) sweep_bwd(g, g.lb, g.Atd, T, ld, 0, D, part);
    }
    if (L.phases & PH_MULADD) {
        for (int k = threadIdx.x; k < g.n_p; k += blockDim.x) {
            int d0 = 0;
            for (; d0 + 8 <= D; d0 += 8) muladd_row<8>(g, L, T, ld, c0, d0, k);
            if (d0 + 4 <= D) { muladd_row<4>(g, L, T, ld, c0, d0, k); d0 += 4; }
            if (d0 + 2 <= D) { muladd_row<2>(g, L, T, ld, c0, d0, k); d0 += 2; }
            if (d0 < D) muladd_row<1>(g, L, T, ld, c0, d0, k);
        }
    }
}

__global__ void __launch_bounds__(kDirThreads, kDirCtasPerSm) k_dirs(DirGrid g, DirLaunch L) {
    __shared__ double part[kPartCap];
    __shared__ double sref[kDMax];
    extern __shared__ unsigned mask_smem[];
    dirs_body(g, L, blockIdx.x, part, sref, mask_smem);
}

// Several (grid, W block) items in one launch: CTA b belongs to the item i with
// cta_ptr[i] <= b < cta_ptr[i + 1]; the item descriptors travel in the kernel
// parameters and are copied to shared memory.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_dirs_batch(DirBatch B) {
    __shared__ double part[kPartCap];
    __shared__ double sref[kDMax];
    __shared__ DirGrid sg;
    __shared__ DirLaunch sl;
    int item = 0;
    while (item + 1 < B.n_items && (int)blockIdx.x >= B.cta_ptr[item + 1]) item++;
    if (threadIdx.x == 0) {
        sg = B.g[item];
        sl = B.l[item];
    }
    __syncthreads();
    dirs_body(sg, sl, (int)blockIdx.x - B.cta_ptr[item], part, sref, nullptr);
    pdl_wait();      // beside k_dir1_batch: what follows this launch follows both
}

// Sweeps of a right-hand side held in shared memory.  There is nothing to coalesce, so
// each row takes a group of G adjacent lanes (a power of two, at most 16 for the two rows
// of a bus, 32 for one): the lanes stride over the row and combine their sums with warp
// shuffles in log2(G) steps, and the first lane of the bus finishes it.
//
// The schedule is laid out on the host (line_steps in api.cu) as steps of one descriptor
// per thread, {q, base, b, w}: theta row of the bus (-1: idle lane), the warp's first entry
// in the line arrays, the bus's place in the schedule, and w (see LineBits).  Entry k of the
// warp's lane l is at base + 32 k + l of the column indices and of the values, which
// k_line_values copies there from the factors (negated) before the solve: every load of a
// warp is one contiguous run.  Read from the factors' rows instead, a warp's load touches a
// 32-byte sector per row for 8 bytes, and one SM's L2 path bounds the solve: 1.25 M cycles for
// the two sweeps of the 9241-bus grid.
//
// A descriptor's address depends on the step's number alone, so the descriptors are read
// three steps ahead and the row data one step ahead, while a step is reduced and finished;
// between two barriers a level reads x from shared memory, multiplies, shuffles and
// finishes.  A lone warp issues an instruction every 4-5 cycles, so a narrow level is given
// to one half of the warps and the next to the other half: a half loads its row data while
// the other computes.  Wide levels take all warps for as many rounds as they need.  FP64
// instructions hold a sub-partition's pipe 64 cycles whatever their lanes do, so line_steps
// counts those of each level's busiest sub-partition and longest warp for each group size
// and takes the least.
// (Spreading a level over a thread-block cluster with x replicated through distributed
// shared memory was slower: more CTAs do not shorten a level's chain, and a cluster
// barrier costs more than a CTA barrier.)
struct LineAhead {
    int i[kLinePre];
    double u[kLinePre];        // the switch of line_sweep names all eight
    double vt;                 // the bus's own off-diagonal entry
};

__device__ __forceinline__ void line_ahead(const LineSched& sc, const int4 d, LineAhead& p) {
    const int cnt = d.w & kLineCntMask;                    // the same for the whole warp
    const int at = d.y + (threadIdx.x & 31);
#pragma unroll
    for (int k = 0; k < kLinePre; k++)
        if (k < cnt && inb(at + 32 * k, sc.n_ent)) {
            p.i[k] = sc.col[at + 32 * k];
            p.u[k] = sc.val[at + 32 * k];
        }
    if (d.z >= 0 && inb(d.z, sc.n_vt)) p.vt = sc.vt[d.z];
}

// x_q = b_q - sum v_qc x_c over the schedule's levels; in a bus of two rows the theta row
// is solved first (FWD) or the v row.  X: n_x rows and the pads' zero.
template <bool FWD, int NT>
__device__ void line_sweep(const LineSched& sc, double* X, const int n_x) {
    const int n_steps = sc.n;
    if (n_steps <= 0) return;
    const int4* my = sc.steps + threadIdx.x;
    auto desc = [&](int st) { return st < n_steps ? my[st * NT] : make_int4(-1, 0, -1, 0); };
    int4 d = desc(0), d1 = desc(1), d2 = desc(2);
    LineAhead p;
#pragma unroll
    for (int k = 0; k < kLinePre; k++) {
        p.i[k] = 0;
        p.u[k] = 0.0;
    }
    p.vt = 0.0;
    line_ahead(sc, d, p);
    for (int st = 0; st < n_steps; st++) {
        const int4 d3 = desc(st + 3);
        const int w = d.w;
        if (w & kLineActive) {                             // the same for the whole warp
            const int q = d.x, lg = (w >> kLineLg) & 7, cnt = w & kLineCntMask, wlg = (w >> kLineWlg) & 7;
            const int G = 1 << lg, row = (w & kLineSplit) && (threadIdx.x & G) ? 1 : 0;
            // the first lane of a row starts from its right-hand side
            double s = q >= 0 && (threadIdx.x & (G - 1)) == 0 && inb(q + row, n_x) ? X[q + row] : 0.0;
            double xv[kLinePre];
#pragma unroll
            for (int k = 0; k < kLinePre; k++) xv[k] = k < cnt && inb(p.i[k], n_x + 1) ? X[p.i[k]] : 0.0;
            // Jumps, not predicates: a predicated-off FP64 instruction still takes its 64 cycles.
            // Unrolled with `if (k < cnt)`, a level of 16-lane rows cost 2000 cycles for any cnt;
            // so it costs 1700, and the two sweeps of the 9241-bus grid 494 k cycles for 580 k.
            switch (cnt) {
                default: s = fma(p.u[7], xv[7], s); [[fallthrough]];
                case 7: s = fma(p.u[6], xv[6], s); [[fallthrough]];
                case 6: s = fma(p.u[5], xv[5], s); [[fallthrough]];
                case 5: s = fma(p.u[4], xv[4], s); [[fallthrough]];
                case 4: s = fma(p.u[3], xv[3], s); [[fallthrough]];
                case 3: s = fma(p.u[2], xv[2], s); [[fallthrough]];
                case 2: s = fma(p.u[1], xv[1], s); [[fallthrough]];
                case 1: s = fma(p.u[0], xv[0], s); [[fallthrough]];
                case 0: break;
            }
            for (int k = kLinePre; k < cnt; k += 4) {      // rows of more than kLinePre G entries
                const int at = d.y + (threadIdx.x & 31) + 32 * k;
                int c[4];
                double u[4];
#pragma unroll
                for (int m = 0; m < 4; m++) {
                    const bool in = k + m < cnt && inb(at + 32 * m, sc.n_ent);
                    c[m] = in ? sc.col[at + 32 * m] : 0;
                    u[m] = in ? sc.val[at + 32 * m] : 0.0;
                }
#pragma unroll
                for (int m = 0; m < 4; m++)
                    if (k + m < cnt && inb(c[m], n_x + 1)) s = fma(u[m], X[c[m]], s);
            }
            auto halve = [&](int o) {
                const double t = __shfl_down_sync(0xffffffffu, s, 1 << o);
                if (o < lg) s += t;
            };
            switch (wlg) {
                case 5: halve(4); [[fallthrough]];
                case 4: halve(3); [[fallthrough]];
                case 3: halve(2); [[fallthrough]];
                case 2: halve(1); [[fallthrough]];
                case 1: halve(0); [[fallthrough]];
                default: break;
            }
            const double s1 = __shfl_sync(0xffffffffu, s, (threadIdx.x + G) & 31);
            if (q >= 0 && (threadIdx.x & ((w & kLineSplit ? 2 * G : G) - 1)) == 0 &&
                inb(w & kLineSplit ? q + 1 : q, n_x)) {
                if (!(w & kLineSplit)) {
                    X[q] = s;
                } else if (w & kLineExt) {
                    X[q] = s;
                    X[q + 1] = s1;
                } else {
                    X[FWD ? q : q + 1] = FWD ? s : s1;
                    X[FWD ? q + 1 : q] = FWD ? fma(p.vt, s, s1) : fma(p.vt, s1, s);
                }
            }
        }
        if (d1.w & kLineActive) line_ahead(sc, d1, p);
        if (w & kLineSync) __syncthreads();                // the same for every thread of the step
        d = d1;
        d1 = d2;
        d2 = d3;
    }
}

// The line arrays' values from the factors: entry i is minus the entry of the unit-diagonal
// factors L'', U' (see k_transpose_values) at position map[i], or (trans) of their transpose
// there; 0 for a pad.
__device__ __forceinline__ void line_values_body(const LineGrid& g, bool trans, double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_line) return;
    const int m = g.map[i];
    double v = 0.0;
    if (m >= 0 && inb(m, g.nnz) && inb(g.tpos[m], g.nnz)) {
        const int r = g.arow[m], c = g.col[m];
        v = trans ? -(g.A[g.tpos[m]] * unit_scale(g.A, g.diagpos, g.invdiag, c, r))
                  : -(g.A[m] * unit_scale(g.A, g.diagpos, g.invdiag, r, c));
    }
    out[i] = v;
}
// blockIdx.y 0: of the factors into `line`, 1: of their transpose into `tline`
__global__ void k_line_values(const __grid_constant__ LineGrid g) {
    pdl_wait();
    line_values_body(g, blockIdx.y != 0, blockIdx.y ? g.tline : g.line);
}

// The factor copies that a Newton step leaves out (see enqueue_factor_copies), from those it
// makes: entry i of `line` is minus L'' or U' at position map[i], the tail's block is in
// triLd and triUd, or, where every level is swept (use_tail 0), in `line` too.  Writes what
// k_transpose_values and k_build_tail write from the same factors (Ad, Atd and the tail's
// triangles; inside the tail up to the order of two multiplications).  A holds the next
// Jacobian by then.  One thread an entry, bound by the latency of its loads and scattered
// stores: 7 us at 118 and 1354 buses, 35 us at 9241 (320 k threads), for the first solve
// after a power flow instead of in each of its Newton steps.
__global__ void k_copies_from_lines(const __grid_constant__ LineGrid g, const __grid_constant__ LineCopies o,
                                    int use_tail) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int T = g.T, t0 = g.t0;
    auto lower = [&](int r, int c) { return c * (T - 1) - c * (c - 1) / 2 + (r - c - 1); };   // r > c
    auto upper = [&](int r, int c) { return c * (c - 1) / 2 + r; };                           // r < c
    auto put = [&](int p, double v) {
        if (!inb(p, g.nnz) || !inb(g.tpos[p], g.nnz)) return;
        o.Ad[p] = v;
        o.Atd[g.tpos[p]] = v;
    };
    if (i < g.n_line) {
        const int m = g.map[i];
        if (m < 0) return;
        if (!inb(m, g.nnz)) return;
        const double v = -g.line[i];
        put(m, v);
        const int r = g.arow[m] - t0, c = g.col[m] - t0;
        if (use_tail || r < 0 || c < 0) return;
        (r > c ? o.triLd[lower(r, c)] : o.triUd[upper(r, c)]) = v;
        (r > c ? o.triLtd[upper(c, r)] : o.triUtd[lower(c, r)]) = v;
        return;
    }
    i -= g.n_line;
    if (i < g.n_x) {
        put(g.diagpos[i], 1.0);
        return;
    }
    i -= g.n_x;
    if (!use_tail || i >= (int64_t)T * T) return;
    const int r = (int)(i / T), c = (int)(i % T), p = o.tail_pos[i];
    if (r == c) return;
    const double v = r > c ? g.triLd[lower(r, c)] : g.triUd[upper(r, c)];
    (r > c ? o.triLtd[upper(c, r)] : o.triUtd[lower(c, r)]) = v;
    if (p >= 0) put(p, v);
}

// One right-hand side, one CTA, x held in shared memory for the whole sweep
// (Newton steps and the first-order adjoint).  Dynamic shared memory holds
// X[n_x] | a zero | the packed tail triangle (use_tail) | kSolve1Part doubles of scratch
// (the tail's right-hand side).  With the tail, the dense top block is solved
// column by column in shared memory, as in k_dirs, instead of as one sparse
// level per variable.
constexpr int kSolve1Part = 2047;
template <int NT>
__device__ __forceinline__ void k_solve1_body(const LineGrid& g, const double* x, double* out, bool trans,
                                              int use_tail) {
    extern __shared__ double X[];
    double* tri = X + g.n_x + 1;
    double* part = tri + (use_tail ? (size_t)g.T * (g.T - 1) / 2 : 0);
    // J_x = D L'' U': the right-hand side of J_x z = b enters as D^-1 b, and the solution
    // D psi of J_x^T leaves as psi
    for (int q = threadIdx.x; q < g.n_x; q += NT) X[q] = trans ? x[q] : x[q] * g.invdiag[q];
    if (threadIdx.x == 0) X[g.n_x] = 0.0;                  // the pads' column
    __syncthreads();
    line_sweep<true, NT>(trans ? g.tup : g.up, X, g.n_x);
    if (use_tail) {
        tail_fwd(g, trans ? g.triUtd : g.triLd, X, 1, 0, 1, part, tri);
        tail_bwd(g, trans ? g.triLtd : g.triUd, X, 1, 0, 1, part, tri);
    }
    line_sweep<false, NT>(trans ? g.tdown : g.down, X, g.n_x);
    __syncthreads();
    for (int q = threadIdx.x; q < g.n_x; q += NT) out[q] = trans ? X[q] * g.invdiag[q] : X[q];
}
template <int NT>
__global__ void __launch_bounds__(NT, kLineRegs / NT)
    k_solve1(const __grid_constant__ LineGrid g, const double* x, double* out, int trans, int use_tail) {
    pdl_wait();
    if (NT == 256) pdl_trigger();
    k_solve1_body<NT>(g, x, out, trans, use_tail);
}

// Algorithm 2 with one direction per CTA and x in shared memory: few directions, where
// k_dirs has one or two a CTA and every level costs it the latency of slot, row and x loads
// from L2.  The sweeps are line_sweep's, on the values k_line_values laid out, so a level
// costs its multiplications, shuffles and one barrier; the projection reads x at random from
// shared memory and passes through Y (in L2) to the transposed sweeps' x.  The chain of
// levels bounds it on small networks and the SM's FP64 pipes on large ones: one product at
// 118 buses 108 -> 63 us, 45 at 2869 buses 513 -> 233, 256 at 9241 buses 2046 -> 1465.
//   phases SPMUL L U (x is left in V), TPROJ UT LT MULADD (x from V), or all of them
template <int NT>
__device__ __forceinline__ void dir1_body(const DirGrid& g, const LineGrid& s, const DirLaunch& L, const int c,
                                          int use_tail) {
    extern __shared__ double X[];
    double* tri = X + g.n_x + 1;
    double* part = tri + (use_tail ? (size_t)s.T * (s.T - 1) / 2 : 0);
    const int rows = g.zero_row + 1;
    if (L.ws_elems > 0 && !inb((int64_t)(c + 1) * rows - 1, L.ws_elems)) return;
    double* V = L.V + (int64_t)c * rows;
    double* Y = L.T + (int64_t)c * rows;
    const double* __restrict__ W = L.W ? L.W + (int64_t)c * L.ldw : nullptr;
    const int id = id_col(L, c);
    if (threadIdx.x == 0) X[g.n_x] = 0.0;                  // the pads' column
    if (L.phases & PH_SPMUL) {
        // D^-1 B, B = -J_p w, or minus column id of J_p
        for (int q = threadIdx.x; q < g.n_x; q += NT) X[q] = 0.0;
        __syncthreads();
        if (W) {
            for (int r = threadIdx.x; r < g.n_jp_rows; r += NT) {
                const int q = g.jp_rows[r];
                double a = 0.0;
                for (int t = g.jp_ptr[q]; t < g.jp_ptr[q + 1]; t++) a = fma(g.jpv[t], W[g.jp_col[t]], a);
                if (inb(q, g.n_x)) X[q] = -a * g.invdiag[q];
            }
        } else {
            for (int t = g.jpt_ptr[id] + threadIdx.x; t < g.jpt_ptr[id + 1]; t += NT)
                if (inb(g.jpt_row[t], g.n_x)) X[g.jpt_row[t]] = -g.jptvd[t];
        }
        __syncthreads();
        line_sweep<true, NT>(s.up, X, g.n_x);
        if (use_tail) {
            tail_fwd(s, s.triLd, X, 1, 0, 1, part, tri);
            tail_bwd(s, s.triUd, X, 1, 0, 1, part, tri);
        }
        line_sweep<false, NT>(s.down, X, g.n_x);
        __syncthreads();
    }
    if (!(L.phases & PH_TPROJ)) {
        for (int q = threadIdx.x; q < g.n_x; q += NT) V[q] = X[q];
        return;
    }
    if (!(L.phases & PH_SPMUL)) {
        for (int q = threadIdx.x; q < g.n_x; q += NT) X[q] = V[q];
        __syncthreads();
    }
    // entry r of v = (z, w, 0)
    auto v_at = [&](int r) {
        if (!inb(r, rows) || r == g.zero_row) return 0.0;
        return r < g.n_x ? X[r] : (W ? W[r - g.n_x] : (r - g.n_x == id ? 1.0 : 0.0));
    };
    if (threadIdx.x < 32) {
        double a = 0.0;
        for (int e = threadIdx.x; e < g.n_gref; e += 32) a = fma(g.gref_val[e], v_at(g.gref_row[e]), a);
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (threadIdx.x == 0) part[0] = *g.c2ref * a;
    }
    __syncthreads();
    const double sref = part[0];
    // projection (see tproj)
    for (int bi = threadIdx.x; bi < g.n_bus; bi += NT) {
        const int b = g.tp_bus[bi], rth = g.uth[b], rv = g.uv[b];
        const double dth = v_at(rth), dv = v_at(rv), ab = g.asum[b];
        double yv = fma(g.d2[b], dv, ab * dth);
        double yth = fma(ab, dv, g.csum[b] * dth);
        int e = g.inc_ptr[b];
        const int e1 = g.inc_ptr[b + 1];
        for (; e + 2 <= e1; e += 2) {
            const double th0 = v_at(g.inc_uth[e]), v0 = v_at(g.inc_uv[e]);
            const double th1 = v_at(g.inc_uth[e + 1]), v1 = v_at(g.inc_uv[e + 1]);
            const double4_32a cf0 = g.inc_coef[e], cf1 = g.inc_coef[e + 1];
            yv = fma(cf0.x, v0, yv);
            yv = fma(cf0.y, th0, yv);
            yth = fma(cf0.z, v0, yth);
            yth = fma(cf0.w, th0, yth);
            yv = fma(cf1.x, v1, yv);
            yv = fma(cf1.y, th1, yv);
            yth = fma(cf1.z, v1, yth);
            yth = fma(cf1.w, th1, yth);
        }
        if (warp_any(e < e1)) {
            if (e < e1) {
                const double th0 = v_at(g.inc_uth[e]), v0 = v_at(g.inc_uv[e]);
                const double4_32a cf = g.inc_coef[e];
                yv = fma(cf.x, v0, yv);
                yv = fma(cf.y, th0, yv);
                yth = fma(cf.z, v0, yth);
                yth = fma(cf.w, th0, yth);
            }
        }
        const bool hg = g.has_gref[b];
        if (warp_any(hg)) {
            if (hg) {
                yv = fma(sref, g.gref_v[b], yv);
                yth = fma(sref, g.gref_th[b], yth);
            }
        }
        if (rth != g.zero_row && inb(rth, rows)) Y[rth] = flip_sign(yth, true);
        if (inb(rv, rows)) Y[rv] = flip_sign(yv, rv < g.n_x);
        const int pr = g.pg_row[b];
        if (warp_any(pr >= 0)) {
            if (pr >= 0 && inb(pr, rows)) Y[pr] = g.pg_curv[b] * v_at(pr);
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < g.n_x; q += NT) X[q] = Y[q];
    __syncthreads();
    line_sweep<true, NT>(s.tup, X, g.n_x);
    if (use_tail) {
        tail_fwd(s, s.triUtd, X, 1, 0, 1, part, tri);
        tail_bwd(s, s.triLtd, X, 1, 0, 1, part, tri);
    }
    line_sweep<false, NT>(s.tdown, X, g.n_x);
    __syncthreads();
    double* HW = L.HW + (int64_t)(id - L.col0) * L.ldhw;
    for (int k = threadIdx.x; k < g.n_p; k += NT) {
        double h = Y[g.n_x + k];
        for (int t = g.jpt_ptr[k]; t < g.jpt_ptr[k + 1]; t++)
            if (inb(g.jpt_row[t], g.n_x)) h = fma(g.jptvd[t], X[g.jpt_row[t]], h);
        HW[k] = h;
    }
}

template <int NT>
__global__ void __launch_bounds__(NT, kLineRegs / NT)
    k_dir1(const __grid_constant__ DirGrid g, const __grid_constant__ LineGrid s, const __grid_constant__ DirLaunch L,
           int use_tail) {
    dir1_body<NT>(g, s, L, blockIdx.x, use_tail);
}

// Items of a batched launch, the directions of item i in CTAs [cta_ptr[i], cta_ptr[i + 1]).
// The launch of the batch's other items may start beside this one.
__global__ void __launch_bounds__(512, kLineRegs / 512) k_dir1_batch(const __grid_constant__ Dir1Batch B) {
    pdl_trigger();
    int i = 0;
    while (i + 1 < B.n_items && (int)blockIdx.x >= B.cta_ptr[i + 1]) i++;
    dir1_body<512>(B.g[i], B.s[i], B.l[i], (int)blockIdx.x - B.cta_ptr[i], B.l[i].use_tail);
}

// ---------------------------------------------------------------------------
// adjoint (eq. 7) and the per-state second-order coefficients
// ---------------------------------------------------------------------------

// Block 0: the slack cost derivatives, grad P_slack, the right-hand side
// -grad_x f = -c'_slack grad_x P_slack of the adjoint system (the rest of rhs is
// zeroed), one thread per admittance entry of the slack.  Block 1: F = sum over
// generators of c2 (S Pg)^2 + c1 S Pg in a fixed order.  Both are single blocks on the
// critical path, bound by their chains of loads; as one thread and a block of 256 after it
// they took 15 + 47 us at 9241 buses.  With k_adjoint_coef, first-order derivatives at 9241
// buses 783 -> 707 us, the reduced Hessian at 118 buses 217 -> 185 us.
constexpr int kAdjThreads = 1024;
__global__ void __launch_bounds__(kAdjThreads) k_adjoint_rhs(PfGrid g, PfState s, AdjData a) {
    const double S = g.base_mva;
    const int r = g.ref;
    if (blockIdx.x == 0) {
        for (int q = threadIdx.x; q < a.n_rhs; q += kAdjThreads) a.rhs[q] = 0.0;
        __syncthreads();
        const double vr = s.vm[r], Pr = s.P[r];
        const double cref = 2.0 * g.c2[r] * S * S * (Pr + s.pd[r]) + g.c1[r] * S;
        if (threadIdx.x == 0) {
            *a.cref = cref;
            *a.c2ref = 2.0 * g.c2[r] * S * S;
        }
        const int t0 = g.yp[r], td = g.ydiag[r];
        for (int t = t0 + threadIdx.x; t < g.yp[r + 1]; t += kAdjThreads) {
            const int j = g.yj[t], n = 2 * (t - t0) - (t > td);    // two entries a neighbour, one for the slack
            if (j == r) {
                const double dv = Pr / vr + g.G[t] * vr;
                a.gref_v[r] = dv;
                a.gref_th[r] = 0.0;
                a.gref_row[n] = a.uv[r];
                a.gref_val[n] = dv;
                continue;
            }
            double sn, cs;
            sincos(s.va[r] - s.va[j], &sn, &cs);
            const double vj = s.vm[j];
            const double dth = vr * vj * (g.G[t] * sn - g.B[t] * cs);
            const double dv = vr * (g.G[t] * cs + g.B[t] * sn);
            a.gref_th[j] = dth;
            a.gref_v[j] = dv;
            a.gref_row[n] = a.uth[j];
            a.gref_val[n] = dth;
            a.gref_row[n + 1] = a.uv[j];
            a.gref_val[n + 1] = dv;
            a.rhs[g.qth[j]] = -cref * dth;
            if (g.qv[j] >= 0) a.rhs[g.qv[j]] = -cref * dv;
        }
        return;
    }
    __shared__ double red[32];
    double acc = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < g.n_bus; i += kAdjThreads) {
        // a PQ bus has no generator
        const double pg = g.qv[i] >= 0 ? 0.0 : (i == r ? s.P[i] + s.pd[i] : s.pg[i]);
        const double P = S * pg, c = g.c2[i] * P * P + g.c1[i] * P;
        if (g.qv[i] < 0) acc += c;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = red[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) *a.F = acc;
    }
}

// Bus weights mu, nu from lambda (mu_slack = c'_slack) and the coefficients of every
// incident branch for the gathered projection.
// With alpha = G(mu_i + mu_j) - B(nu_i + nu_j), beta = B(mu_i - mu_j) + G(nu_i - nu_j),
// t = theta_i - theta_j, the branch term of sum mu P + nu Q is
// v_i v_j (alpha cos t + beta sin t); K = alpha cos t + beta sin t,
// M = dK/dt, a = v_j M, b = v_i M, c = -v_i v_j K.
struct CoefBus {
    double mu, nu, v;
};
constexpr int kCoefThreads = 128;
__device__ __forceinline__ CoefBus coef_bus(const PfGrid& g, const PfState& s, const CoefData& c, int i) {
    return {g.qth[i] >= 0 ? c.lam[g.qth[i]] : *c.cref, g.qv[i] >= 0 ? c.lam[g.qv[i]] : 0.0, s.vm[i]};
}
// admittance entry t = (i, j), j != i: its coefficients, and a and c for the bus's sums
__device__ __forceinline__ double4_32a coef_entry(const PfGrid& g, const PfState& s, const CoefData& c, int t, int i,
                                                  const CoefBus& bi, double& a, double& cc) {
    const int j = g.yj[t];
    const CoefBus bj = coef_bus(g, s, c, j);
    const double Gij = g.G[t], Bij = g.B[t];
    const double alpha = Gij * (bi.mu + bj.mu) - Bij * (bi.nu + bj.nu);
    const double beta = Bij * (bi.mu - bj.mu) + Gij * (bi.nu - bj.nu);
    double sn, cs;
    sincos(s.va[i] - s.va[j], &sn, &cs);
    const double K = alpha * cs + beta * sn;
    const double M = -alpha * sn + beta * cs;
    a = bj.v * M;
    cc = -bi.v * bj.v * K;
    return make_double4_32a(K, -a, bi.v * M, -cc);
}
__device__ __forceinline__ void coef_finish(const PfGrid& g, const CoefData& c, int i, const CoefBus& bi, double sa,
                                            double sc) {
    c.d2[i] = 2.0 * (bi.mu * g.G[g.ydiag[i]] - bi.nu * g.B[g.ydiag[i]]);
    c.asum[i] = sa;
    c.csum[i] = sc;
    c.pg_curv[i] = g.ip_pg[i] >= 0 ? 2.0 * g.c2[i] * g.base_mva * g.base_mva : 0.0;
}
// one thread per bus (a network with a bus of more than 32 entries)
__device__ __forceinline__ void coef_by_bus(const PfGrid& g, const PfState& s, const CoefData& c, int i) {
    if (i >= g.n_bus) return;
    const CoefBus bi = coef_bus(g, s, c, i);
    double sa = 0.0, sc = 0.0;
    int e = c.inc_ptr[i];
    for (int t = g.yp[i]; t < g.yp[i + 1]; t++) {
        if (g.yj[t] == i) continue;
        double a, cc;
        c.coef[e++] = coef_entry(g, s, c, t, i, bi, a, cc);
        sa += a;
        sc += cc;
    }
    coef_finish(g, c, i, bi, sa, sc);
}
// One admittance entry per lane, on the warps of k_pf_eval_warp: a sincos is a long chain
// of dependent FP64 instructions, and a thread per bus runs one after the other.  The
// lane of each bus adds its row's terms in row order.
__device__ __forceinline__ void coef_by_warp(const PfGrid& g, const PfState& s, const CoefData& c, int w) {
    __shared__ double sh[kCoefThreads / 32][64];
    if (w >= g.n_pfw) return;                                   // warp-uniform
    const int lane = threadIdx.x & 31;
    double* sw = sh[threadIdx.x >> 5];
    const int b0 = g.pf_wb[w], b1 = g.pf_wb[w + 1], e0 = g.yp[b0], t = e0 + lane;
    double a = 0.0, cc = 0.0;
    if (t < g.yp[b1]) {
        const int i = g.yrow[t], td = g.ydiag[i];
        if (t != td)
            c.coef[c.inc_ptr[i] + (t - g.yp[i]) - (t > td)] = coef_entry(g, s, c, t, i, coef_bus(g, s, c, i), a, cc);
    }
    sw[lane] = a;
    sw[32 + lane] = cc;
    __syncwarp();
    const int i = b0 + lane;
    if (i < b1) {
        double sa = 0.0, sc = 0.0;
        for (int tt = g.yp[i]; tt < g.yp[i + 1]; tt++) {        // the diagonal's terms are zero
            sa += sw[tt - e0];
            sc += sw[32 + tt - e0];
        }
        coef_finish(g, c, i, coef_bus(g, s, c, i), sa, sc);
    }
}

// grad F = grad_p f + J_p^T lambda, one thread per bus (its v and Pg entries).
__device__ __forceinline__ void gradient_bus(const PfGrid& g, const PfState& s, const CoefData& c, int i) {
    if (i >= g.n_bus) return;
    const int kv = g.ip_v[i];
    if (kv >= 0) {
        double h = *c.cref * c.gref_v[i];
        for (int t = c.jpt_ptr[kv]; t < c.jpt_ptr[kv + 1]; t++) h = fma(c.jptv[t], c.lam[c.jpt_row[t]], h);
        c.grad[kv] = h;
    }
    const int kp = g.ip_pg[i];
    if (kp >= 0) {
        const double S = g.base_mva;
        double h = 2.0 * g.c2[i] * S * S * s.pg[i] + g.c1[i] * S;
        for (int t = c.jpt_ptr[kp]; t < c.jpt_ptr[kp + 1]; t++) h = fma(c.jptv[t], c.lam[c.jpt_row[t]], h);
        c.grad[kp] = h;
    }
}

// What follows from lambda: the projection's coefficients (the first n_coef blocks) and
// grad F (the others); as two kernels with a thread per bus 33 + 11 us at 9241 buses.
__global__ void __launch_bounds__(kCoefThreads) k_adjoint_coef(PfGrid g, PfState s, CoefData c, int n_coef) {
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x >= n_coef) gradient_bus(g, s, c, ((int)blockIdx.x - n_coef) * kCoefThreads + (int)threadIdx.x);
    else if (g.n_pfw > 0) coef_by_warp(g, s, c, (int)(blockIdx.x * (kCoefThreads / 32) + (threadIdx.x >> 5)));
    else coef_by_bus(g, s, c, (int)(blockIdx.x * kCoefThreads + threadIdx.x));
}

// external column-major <-> internal row-major with a row map
__global__ void k_scatter_rows(int n_rows, int N, const int* map, const double* src, int64_t lds, double* dst,
                               int64_t ldd, double scale_x, int n_x) {
    int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= (int64_t)n_rows * N) return;
    int c = (int)(it / n_rows), r = (int)(it - (int64_t)c * n_rows);
    double v = src[(int64_t)c * lds + r];
    dst[(int64_t)map[r] * ldd + c] = r < n_x ? scale_x * v : v;
}

__global__ void k_gather_rows(int n_rows, int N, const int* map, const double* src, int64_t lds, double* dst,
                              int64_t ldd, double scale_x, int n_x) {
    int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= (int64_t)n_rows * N) return;
    int c = (int)(it / n_rows), r = (int)(it - (int64_t)c * n_rows);
    double v = src[(int64_t)map[r] * lds + c];
    dst[(int64_t)c * ldd + r] = r < n_x ? scale_x * v : v;
}

int blocks_for(int64_t n, int t) { return (int)((n + t - 1) / t); }

// ---------------------------------------------------------------------------
// Newton power flow over several grids of one topology: item blockIdx.y
// ---------------------------------------------------------------------------
__global__ void k_pf_eval_batch(PfBatch B) {
    pdl_wait();
    pdl_trigger();
    const PfBatchItem& it = B.it[blockIdx.y];
    k_pf_eval_body(it.g, it.s, it.x, it.A, it.jpv, it.umax, it.umax + 1, 1);
}
__global__ void k_pf_prep_batch(PfBatch B) {
    const PfBatchItem& it = B.it[blockIdx.y];
    pf_prep_body(it.g, it.s, it.A, it.umax, nullptr, 1);
}
__global__ void __launch_bounds__(32 * kPfWarps) k_pf_eval_warp_batch(PfBatch B) {
    pdl_wait();
    pdl_trigger();
    const PfBatchItem& it = B.it[blockIdx.y];
    pf_eval_warp_body(it.g, it.s, it.x, it.A, it.jpv, it.umax, it.umax + 1, 1);
}

__global__ void k_batch_status(PfBatch B, double* out) {
    const int i = threadIdx.x;
    if (i >= B.n) return;
    out[2 * i] = __longlong_as_double((long long)B.it[i].umax[0]);
    out[2 * i + 1] = (double)B.it[i].err[0];
}

__global__ void k_newton_update_batch(PfBatch B) {
    pdl_wait();
    pdl_trigger();
    const PfBatchItem& it = B.it[blockIdx.y];
    k_newton_update_body(it.g, it.s, it.x);
}

__global__ void k_rf_update_batch(RfBatch B, int64_t t0, int64_t nt, int j0, int njob) {
    k_rf_update_body(B.g[blockIdx.y], t0, nt, j0, njob);
}
__global__ void __launch_bounds__(kRfThreads) k_rf_levels_batch(RfBatch B, int l0, int l1) {
    rf_levels_body(B.g[blockIdx.y], l0, l1);
}
__global__ void k_rf_leaf_piv_batch(RfBatch B, int njob) {
    k_rf_leaf_piv_body(B.g[blockIdx.y], njob);
}
__global__ void k_rf_pivot_batch(RfBatch B) {
    k_rf_pivot_body(B.g[blockIdx.y], (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}
__global__ void __launch_bounds__(kTailThreads) k_rf_finish_batch(RfBatch B) { rf_finish_body(B.g[blockIdx.y]); }
__global__ void k_tail_gather_batch(RfBatch B) {
    k_tail_gather_body(B.g[blockIdx.y]);
}
__global__ void __launch_bounds__(256) k_tail_step_batch(RfBatch B, int k) {
    pdl_wait();
    pdl_trigger();
    k_tail_step_body(B.g[blockIdx.y], k);
}
__global__ void k_tail_scatter_batch(RfBatch B) {
    pdl_wait();
    k_tail_scatter_body(B.g[blockIdx.y]);
}

// the single solves' tail triangles, of the unit-diagonal factors L'' and U'
__global__ void k_tail_tri_batch(TriBatch B) {
    const int i = blockIdx.y, T = B.T;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= T * T) return;
    const int r = idx / T, c = idx - r * T;
    if (r == c) return;
    const int p = B.pos[i][idx];
    const double a = p >= 0 ? B.A[i][p] : 0.0, ir = B.invdiag[i][B.t0 + r];     // as k_build_tail, bit for bit
    if (r > c) B.triLd[i][c * (T - 1) - c * (c - 1) / 2 + (r - c - 1)] = a * B.A[i][B.pos[i][c * T + c]] * ir;
    else B.triUd[i][c * (c - 1) / 2 + r] = a * ir;
}

__global__ void k_line_values_batch(const __grid_constant__ Solve1Batch B) {
    pdl_wait();
    pdl_trigger();
    line_values_body(B.g[blockIdx.y], false, B.g[blockIdx.y].line);
}

template <int NT>
__global__ void __launch_bounds__(NT, kLineRegs / NT)
    k_solve1_batch(const __grid_constant__ Solve1Batch B, int use_tail) {
    pdl_wait();
    pdl_trigger();
    k_solve1_body<NT>(B.g[blockIdx.x], B.x[blockIdx.x], B.x[blockIdx.x], false, use_tail);
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

void launch_injections(const PfGrid& g, const PfState& s, cudaStream_t st) {
    if (g.n_bus > 0) k_injections<<<blocks_for(g.n_bus, 128), 128, 0, st>>>(g, s);
}

static unsigned prep_blocks(const PfGrid& g) {
    const int64_t n = g.nnz_a > g.n_bus ? g.nnz_a : g.n_bus;
    const int64_t b = (n + 1023) / 1024;             // four entries per thread
    return (unsigned)(b < 1 ? 1 : (b > 1024 ? 1024 : b));
}
void launch_pf_prep(const PfGrid& g, const PfState& s, double* A, unsigned long long* umax, int* err, bool zero,
                    bool chained, cudaStream_t st) {
    launch_pdl(chained, k_pf_prep, dim3(prep_blocks(g)), dim3(256), 0, st, g, s, A, umax, err, zero ? 1 : 0);
}
void launch_pf_prep_batch(const PfBatch& B, cudaStream_t st) {
    if (B.n > 0) k_pf_prep_batch<<<dim3(prep_blocks(B.it[0].g), (unsigned)B.n), 256, 0, st>>>(B);
}

void launch_pf_eval(const PfGrid& g, const PfState& s, double* gres, double* A, double* jpv,
                    unsigned long long* gmax, unsigned long long* jmax, bool want_jac, cudaStream_t st) {
    if (g.n_pfw > 0)
        launch_pdl(true, k_pf_eval_warp, dim3((g.n_pfw + kPfWarps - 1) / kPfWarps), dim3(32 * kPfWarps), 0, st, g, s,
                   gres, A, jpv, gmax, jmax, want_jac ? 1 : 0);
    else if (g.n_bus > 0)
        launch_pdl(true, k_pf_eval, dim3(blocks_for(g.n_bus, 64)), dim3(64), 0, st, g, s, gres, A, jpv, gmax, jmax,
                   want_jac ? 1 : 0);
}

cudaError_t launch_jac_ad(const PfGrid& g, const PfState& s, const int* col_th, const int* col_v, const int* col_pg,
                          int n_colors, double* A, double* jpv, unsigned long long* jmax, cudaStream_t st) {
    constexpr int CH = 8;
    if (g.n_bus == 0 || n_colors == 0) return cudaSuccess;
    dim3 grid((unsigned)blocks_for(g.n_bus, 128), (unsigned)((n_colors + CH - 1) / CH));
    k_jac_ad<CH><<<grid, 128, 0, st>>>(g, s, col_th, col_v, col_pg, A, jpv, jmax);
    return cudaGetLastError();
}

void launch_newton_update(const PfGrid& g, const PfState& s, const double* dx, bool chained, cudaStream_t st) {
    if (g.n_bus > 0) launch_pdl(chained, k_newton_update, dim3(blocks_for(g.n_bus, 128)), dim3(128), 0, st, g, s, dx);
}

// L2 prefetch of read-only arrays: one bulk prefetch of up to kPrefetchChunk bytes
// per thread (TMA units of many SMs at once).  The refactorisation's level data
// (tens of MB on the 9241-bus grid) is otherwise read from HBM level by level,
// after the direction sweeps of the previous state evicted it from L2.
constexpr unsigned long long kPrefetchChunk = 4096;
__global__ void k_prefetch_l2(PrefetchList L) {
    const unsigned long long c = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (L.n <= 0 || c >= L.first[L.n]) return;
    int a = 0;
    while (a + 1 < L.n && c >= L.first[a + 1]) a++;
    const unsigned long long off = (c - L.first[a]) * kPrefetchChunk;
    if (off >= L.bytes[a]) return;
    unsigned long long n = L.bytes[a] - off;
    if (n > kPrefetchChunk) n = kPrefetchChunk;
    n &= ~15ull;
    if (n)
        asm volatile("{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %0;\n\tcp.async.bulk.prefetch.L2.global [ga], %1;\n\t}"
                     :: "l"(L.p[a] + off), "r"((unsigned)n) : "memory");
}

void launch_prefetch_l2(const PrefetchList& in, cudaStream_t st) {
    PrefetchList L = in;
    L.first[0] = 0;
    for (int a = 0; a < L.n; a++) L.first[a + 1] = L.first[a] + (L.bytes[a] + kPrefetchChunk - 1) / kPrefetchChunk;
    const unsigned long long nc = L.n > 0 ? L.first[L.n] : 0;
    if (nc > 0) k_prefetch_l2<<<(unsigned)((nc + 31) / 32), 32, 0, st>>>(L);
}

// The first of the last levels that one CTA runs in one launch (n_lev: none; a single level
// is no gain).
static int rf_one_cta(const int64_t* tgt_lev_ptr_host, int n_lev) {
    int l = n_lev;
    while (l > 0 && tgt_lev_ptr_host[l] - tgt_lev_ptr_host[l - 1] <= kRfThreads) l--;
    return n_lev - l > 1 ? l : n_lev;
}

cudaError_t launch_refactor(const RfGrid& g, const int* lev_ptr_host, const int64_t* tgt_lev_ptr_host,
                            const int* piv_lev_ptr_host, int n_lev, cudaStream_t st) {
    (void)lev_ptr_host;
    cudaError_t e = cudaSuccess;
    bool pdl = false;   // the first launch follows an event wait
    auto chk = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        pdl = true;
    };
    if (n_lev > 0 && piv_lev_ptr_host[0] > 0)
        chk(launch_pdl(pdl, k_rf_leaf_piv, dim3(blocks_for(piv_lev_ptr_host[0], 128)), dim3(128), 0, st, g,
                       piv_lev_ptr_host[0]));
    const int l0 = rf_one_cta(tgt_lev_ptr_host, n_lev);
    for (int lev = 0; lev < l0; lev++) {
        const int64_t t0 = tgt_lev_ptr_host[lev], nt = tgt_lev_ptr_host[lev + 1] - t0;
        const int j0 = piv_lev_ptr_host[lev], njob = piv_lev_ptr_host[lev + 1] - j0;
        if (nt > 0) chk(launch_pdl(pdl, k_rf_update, dim3(blocks_for(nt, 256)), dim3(256), 0, st, g, t0, nt, j0, njob));
    }
    if (l0 < n_lev) chk(launch_pdl(pdl, k_rf_levels, dim3(1), dim3(kRfThreads), 0, st, g, l0, n_lev));
    if (tail_in_one(g.T)) {
        chk(launch_pdl(pdl, k_rf_finish, dim3(1 + blocks_for((int64_t)g.n_piv + g.n_pe, kTailThreads)),
                       dim3(kTailThreads), 0, st, g));
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    if (g.n_piv + g.n_pe > 0)
        chk(launch_pdl(pdl, k_rf_pivot, dim3(blocks_for((int64_t)g.n_piv + g.n_pe, 256)), dim3(256), 0, st, g));
    if (g.T > 0) {
        const int TT = g.T * g.T, nt = (g.T + kTailTB - 1) / kTailTB;
        chk(launch_pdl(pdl, k_tail_gather, dim3(blocks_for(TT, 256)), dim3(256), 0, st, g));
        for (int k = -1; k < nt; k++) {
            const int c = k + 1, U = c < nt ? nt - c - 1 : 0;
            const int grid = 2 * U + (k >= 0 ? 1 + U * U : 0);
            if (grid > 0) chk(launch_pdl(pdl, k_tail_step, dim3(grid), dim3(kTailTB * kTailTB), 0, st, g, k));
        }
        chk(launch_pdl(pdl, k_tail_scatter, dim3(blocks_for(TT, 256)), dim3(256), 0, st, g));
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The dynamic shared-memory limit is a per-kernel attribute of each device's
// context: raise it on every device once, to that device's maximum (minus the
// kernel's static shared memory), for every kernel that can need more than the
// 48 KB default.  The SM count is cached per device too.
constexpr int kMaxDevices = 64;
std::mutex g_dev_mu;
bool g_prepared[kMaxDevices];
int g_n_sm[kMaxDevices];

cudaError_t prepare_kernels() {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_dev_mu);
    if (g_prepared[dev]) return cudaSuccess;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const void* fns[8] = {(const void*)k_dirs, (const void*)k_solve1<256>, (const void*)k_solve1<512>,
                          (const void*)k_solve1_batch<256>, (const void*)k_solve1_batch<512>,
                          (const void*)k_dir1<256>, (const void*)k_dir1<512>, (const void*)k_dir1_batch};
    for (const void* f : fns) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, f);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
        if (e != cudaSuccess) return e;
    }
    // the batched direction kernel's shapes: shared memory before L1, so that the
    // shape's resident CTAs fit an SM (6 x 35 KB for 128 threads)
    const void* shapes[4] = {(const void*)k_dirs_batch<128, 6>, (const void*)k_dirs_batch<192, 4>,
                             (const void*)k_dirs_batch<256, 3>, (const void*)k_dirs_batch<kDirThreads, kDirCtasPerSm>};
    for (const void* f : shapes) {
        e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
    }
    g_prepared[dev] = true;
    return cudaSuccess;
}

void launch_transpose_values(int nnz, const int* tpos, const int* arow, const int* col, const int* diagpos,
                             const double* A, const double* invdiag, double* Ad, double* Atd, int nnz_jp,
                             const int* jpt_src, const int* jpt_row, const double* jpv, double* jptv, double* jptvd,
                             cudaStream_t st) {
    int n = nnz > nnz_jp ? nnz : nnz_jp;
    if (n > 0)
        k_transpose_values<<<blocks_for(n, 256), 256, 0, st>>>(nnz, tpos, arow, col, diagpos, A, invdiag, Ad, Atd, nnz_jp,
                                                               jpt_src, jpt_row, jpv, jptv, jptvd);
}

// SMs of the current device (1 if the query fails)
int num_sms() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 1;
    std::lock_guard<std::mutex> lock(g_dev_mu);
    if (g_n_sm[dev] == 0) {
        int n = 0;
        g_n_sm[dev] = (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) ? n : 1;
    }
    return g_n_sm[dev];
}

int dirs_cta_slots_for(int n_sm) { return kDirCtasPerSm * n_sm; }

int dirs_ctas_for(int N, int slots) {
    int G = N < slots ? N : slots;
    int need = (N + kDMax - 1) / kDMax;
    if (G < need) G = need;
    return G < 1 ? 1 : G;
}

int dirs_default_ctas(int N) { return dirs_ctas_for(N, kDirCtasPerSm * num_sms()); }

int dirs_tail_cap() { return kPartCap; }

bool dirs_tail_fits(int T, int N, int n_cta) {
    if (T <= 1 || n_cta <= 0) return false;
    int dmax = (N + n_cta - 1) / n_cta;
    return (int64_t)T * dmax <= kPartCap;      // the tail rows of the CTA's directions sit in `part`
}

void launch_dirs(const DirGrid& g, const DirLaunch& L, cudaStream_t st) {
    if (L.N <= 0 || L.n_cta <= 0) return;
    // active and seed masks, one bit per row each
    size_t smem = (L.use_tail && L.use_reach) ? 2 * (((size_t)g.n_x + 127) / 128 * 16) : 0;
    k_dirs<<<L.n_cta, kDirThreads, smem, st>>>(g, L);
}

// Compiled CTA shapes of the batched direction kernel: threads x resident CTAs per
// SM, 768 threads an SM each (the register bound of the 384 x 2 shape); the
// static shared memory (dense-tail rows, reference row, item descriptors) is
// about 35 KB a CTA, 210 KB an SM at 6 CTAs.
int dirs_batch_ctas_per_sm(int threads) {
    switch (threads) {
        case 128: return 6;
        case 192: return 4;
        case 256: return 3;
        case 384: return 2;
        default: return 0;
    }
}
bool dirs_batch_shape_ok(int threads) { return dirs_batch_ctas_per_sm(threads) > 0; }

cudaError_t launch_dirs_batch(const DirBatch& B, int threads, bool beside, cudaStream_t st) {
    const int n = B.n_items > 0 ? B.cta_ptr[B.n_items] : 0;
    if (n <= 0) return cudaSuccess;
    const dim3 grid((unsigned)n), block((unsigned)threads);
    switch (threads) {
        case 128: return launch_pdl(beside, k_dirs_batch<128, 6>, grid, block, 0, st, B);
        case 192: return launch_pdl(beside, k_dirs_batch<192, 4>, grid, block, 0, st, B);
        case 256: return launch_pdl(beside, k_dirs_batch<256, 3>, grid, block, 0, st, B);
        default: return launch_pdl(beside, k_dirs_batch<kDirThreads, kDirCtasPerSm>, grid, dim3(kDirThreads), 0, st, B);
    }
}

void launch_scale_rows(int n, int N, const double* s, double* x, int64_t ld, cudaStream_t st) {
    if ((int64_t)n * N > 0) k_scale_rows<<<blocks_for((int64_t)n * N, 256), 256, 0, st>>>(n, N, s, x, ld);
}

void launch_build_tail(int T, int t0, const int* pos, const double* A, const double* invdiag, double* triLd,
                       double* triUd, double* triUtd, double* triLtd, cudaStream_t st) {
    if (T > 1 && !tail_in_one(T))
        k_build_tail<<<blocks_for((int64_t)T * T, 256), 256, 0, st>>>(T, t0, pos, A, invdiag, triLd, triUd, triUtd,
                                                                      triLtd);
}

void launch_line_values(const LineGrid& g, bool transposed_too, cudaStream_t st) {
    if (g.n_line > 0)
        launch_pdl(true, k_line_values, dim3((unsigned)blocks_for(g.n_line, 256), transposed_too ? 2u : 1u), dim3(256), 0,
                   st, g);
}

cudaError_t launch_copies_from_lines(const LineGrid& g, const LineCopies& o, bool use_tail, cudaStream_t st) {
    const int64_t n = (int64_t)g.n_line + g.n_x + (use_tail ? (int64_t)g.T * g.T : 0);
    if (n > 0) k_copies_from_lines<<<blocks_for(n, 256), 256, 0, st>>>(g, o, use_tail ? 1 : 0);
    return cudaGetLastError();
}

void launch_adjoint_rhs(const PfGrid& g, const PfState& s, const AdjData& a, cudaStream_t st) {
    k_adjoint_rhs<<<2, kAdjThreads, 0, st>>>(g, s, a);
}

// Small grids take CTAs of 256 threads: their levels do not fill more warps, and idle
// warps cost issue slots and barrier time at every step.
int line_threads(int n_x) { return n_x <= 1024 ? 256 : 512; }

static size_t solve1_smem(int n_x, int T, bool tail) {
    return ((size_t)n_x + 1 + (tail ? (size_t)T * (T - 1) / 2 : 0) + kSolve1Part) * sizeof(double);
}

int solve1_mode(int n_x, int T) {
    const size_t cap = 227 * 1024;
    if (T > 1 && T <= kSolve1Part && solve1_smem(n_x, T, true) <= cap) return 2;
    return solve1_smem(n_x, T, false) <= cap ? 1 : 0;
}

cudaError_t launch_dir1_batch(const Dir1Batch& B, cudaStream_t st) {
    if (B.n_items <= 0) return cudaSuccess;
    size_t smem = 0;
    for (int i = 0; i < B.n_items; i++) smem = std::max(smem, solve1_smem(B.s[i].n_x, B.s[i].T, B.l[i].use_tail != 0));
    k_dir1_batch<<<B.cta_ptr[B.n_items], 512, smem, st>>>(B);
    return cudaGetLastError();
}

cudaError_t launch_dir1(const DirGrid& g, const LineGrid& s, const DirLaunch& L, bool use_tail, cudaStream_t st) {
    const size_t smem = solve1_smem(s.n_x, s.T, use_tail);
    if (line_threads(s.n_x) == 256) k_dir1<256><<<L.N, 256, smem, st>>>(g, s, L, use_tail ? 1 : 0);
    else k_dir1<512><<<L.N, 512, smem, st>>>(g, s, L, use_tail ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_solve1(const LineGrid& g, const double* x, double* out, bool trans, bool use_tail, bool chained,
                          cudaStream_t st) {
    const size_t smem = solve1_smem(g.n_x, g.T, use_tail);
    const bool small = line_threads(g.n_x) == 256;
    return launch_pdl(chained, small ? k_solve1<256> : k_solve1<512>, dim3(1), dim3(small ? 256 : 512), smem, st, g, x,
                      out, trans ? 1 : 0, use_tail ? 1 : 0);
}

int dirs_cta_slots() { return kDirCtasPerSm * num_sms(); }
int dirs_batch_slots(int threads) { return dirs_batch_ctas_per_sm(threads) * num_sms(); }

void launch_adjoint_coef(const PfGrid& g, const PfState& s, const CoefData& c, bool chained, cudaStream_t st) {
    const int n_coef = g.n_pfw > 0 ? blocks_for(g.n_pfw, kCoefThreads / 32) : blocks_for(g.n_bus, kCoefThreads);
    launch_pdl(chained, k_adjoint_coef, dim3(n_coef + blocks_for(g.n_bus, kCoefThreads)), dim3(kCoefThreads), 0, st, g, s, c,
               n_coef);
}

void launch_scatter_rows(int n_rows, int N, const int* map, const double* src, int64_t lds, double* dst,
                         int64_t ldd, double scale_x, int n_x, cudaStream_t st) {
    int64_t n = (int64_t)n_rows * N;
    if (n > 0) k_scatter_rows<<<blocks_for(n, 256), 256, 0, st>>>(n_rows, N, map, src, lds, dst, ldd, scale_x, n_x);
}

void launch_pf_eval_batch(const PfBatch& B, cudaStream_t st) {
    if (B.n > 0 && B.it[0].g.n_pfw > 0)
        launch_pdl(true, k_pf_eval_warp_batch,
                   dim3((unsigned)((B.it[0].g.n_pfw + kPfWarps - 1) / kPfWarps), (unsigned)B.n), dim3(32 * kPfWarps), 0, st, B);
    else if (B.n > 0 && B.max_bus > 0)
        launch_pdl(true, k_pf_eval_batch, dim3((unsigned)blocks_for(B.max_bus, 64), (unsigned)B.n), dim3(64), 0, st, B);
}

void launch_batch_status(const PfBatch& B, double* out, cudaStream_t st) {
    if (B.n > 0) k_batch_status<<<1, 32, 0, st>>>(B, out);
}

void launch_newton_update_batch(const PfBatch& B, bool chained, cudaStream_t st) {
    if (B.n > 0 && B.max_bus > 0)
        launch_pdl(chained, k_newton_update_batch, dim3((unsigned)blocks_for(B.max_bus, 128), (unsigned)B.n), dim3(128), 0,
                   st, B);
}

cudaError_t launch_refactor_batch(const RfBatch& B, const int* lev_ptr_host, const int64_t* tgt_lev_ptr_host,
                                  const int* piv_lev_ptr_host, int n_lev, cudaStream_t st) {
    if (B.n <= 0) return cudaSuccess;
    const unsigned n = (unsigned)B.n;
    (void)lev_ptr_host;
    cudaError_t e = cudaSuccess;
    bool pdl = false;   // the first launch follows an event wait
    auto chk = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        pdl = true;
    };
    if (n_lev > 0 && piv_lev_ptr_host[0] > 0)
        chk(launch_pdl(pdl, k_rf_leaf_piv_batch, dim3((unsigned)blocks_for(piv_lev_ptr_host[0], 128), n), dim3(128), 0, st,
                       B, piv_lev_ptr_host[0]));
    const int l0 = rf_one_cta(tgt_lev_ptr_host, n_lev);
    for (int lev = 0; lev < l0; lev++) {
        const int64_t t0 = tgt_lev_ptr_host[lev], nt = tgt_lev_ptr_host[lev + 1] - t0;
        const int j0 = piv_lev_ptr_host[lev], njob = piv_lev_ptr_host[lev + 1] - j0;
        if (nt > 0)
            chk(launch_pdl(pdl, k_rf_update_batch, dim3((unsigned)blocks_for(nt, 256), n), dim3(256), 0, st, B, t0, nt, j0,
                           njob));
    }
    if (l0 < n_lev) chk(launch_pdl(pdl, k_rf_levels_batch, dim3(1, n), dim3(kRfThreads), 0, st, B, l0, n_lev));
    const int64_t np = (int64_t)B.g[0].n_piv + B.g[0].n_pe;
    if (tail_in_one(B.g[0].T)) {
        chk(launch_pdl(pdl, k_rf_finish_batch, dim3((unsigned)(1 + blocks_for(np, kTailThreads)), n), dim3(kTailThreads),
                       0, st, B));
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    if (np > 0) chk(launch_pdl(pdl, k_rf_pivot_batch, dim3((unsigned)blocks_for(np, 256), n), dim3(256), 0, st, B));
    const int T = B.g[0].T;
    if (T > 0) {
        const int TT = T * T, nt = (T + kTailTB - 1) / kTailTB;
        chk(launch_pdl(pdl, k_tail_gather_batch, dim3((unsigned)blocks_for(TT, 256), n), dim3(256), 0, st, B));
        for (int k = -1; k < nt; k++) {
            const int c = k + 1, U = c < nt ? nt - c - 1 : 0;
            const int grid = 2 * U + (k >= 0 ? 1 + U * U : 0);
            if (grid > 0)
                chk(launch_pdl(pdl, k_tail_step_batch, dim3((unsigned)grid, n), dim3(kTailTB * kTailTB), 0, st, B, k));
        }
        chk(launch_pdl(pdl, k_tail_scatter_batch, dim3((unsigned)blocks_for(TT, 256), n), dim3(256), 0, st, B));
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

void launch_tail_tri_batch(const TriBatch& B, cudaStream_t st) {
    if (B.n > 0 && B.T > 1 && !tail_in_one(B.T))
        k_tail_tri_batch<<<dim3((unsigned)blocks_for((int64_t)B.T * B.T, 256), (unsigned)B.n), 256, 0, st>>>(B);
}

cudaError_t launch_solve1_batch(const Solve1Batch& B, bool use_tail, int n_x, int T, cudaStream_t st) {
    if (B.n <= 0) return cudaSuccess;
    const int nl = B.g[0].n_line;      // one topology: the same for every item
    if (nl > 0) {
        const cudaError_t e = launch_pdl(true, k_line_values_batch, dim3((unsigned)blocks_for(nl, 256), (unsigned)B.n),
                                         dim3(256), 0, st, B);
        if (e != cudaSuccess) return e;
    }
    const bool small = line_threads(n_x) == 256;
    return launch_pdl(nl > 0, small ? k_solve1_batch<256> : k_solve1_batch<512>, dim3((unsigned)B.n),
                      dim3(small ? 256 : 512), solve1_smem(n_x, T, use_tail), st, B, use_tail ? 1 : 0);
}

void launch_gather_rows(int n_rows, int N, const int* map, const double* src, int64_t lds, double* dst,
                        int64_t ldd, double scale_x, int n_x, cudaStream_t st) {
    int64_t n = (int64_t)n_rows * N;
    if (n > 0) k_gather_rows<<<blocks_for(n, 256), 256, 0, st>>>(n_rows, N, map, src, lds, dst, ldd, scale_x, n_x);
}

}  // namespace rh

// Whether this build checks indices (-DRH_BOUNDS), and the error word of `device`,
// which the call reads and clears.
extern "C" rh_status rh_bounds_check(int32_t device, int32_t* enabled, uint32_t* errors) {
    if (!enabled || !errors) return RH_EINVAL;
    *errors = 0;
#ifdef RH_BOUNDS
    *enabled = 1;
    if (cudaSetDevice(device) != cudaSuccess) return RH_ECUDA;
    unsigned int e = 0, z = 0;
    if (cudaMemcpyFromSymbol(&e, rh::g_bounds_err, sizeof(e)) != cudaSuccess) return RH_ECUDA;
    if (cudaMemcpyToSymbol(rh::g_bounds_err, &z, sizeof(z)) != cudaSuccess) return RH_ECUDA;
    *errors = e;
#else
    (void)device;
    *enabled = 0;
#endif
    return RH_OK;
}
