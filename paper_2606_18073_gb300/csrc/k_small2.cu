// Latency-optimised FP64 small phase of one sGKS iteration (the default path).
//
// k_qr_append (K2): rank-one append to the sketched QR factors S_A A W = Q_A R_A and
//   S_L L W = Q_L R_L (eq. updqr and the formulas under it; classical Gram-Schmidt applied
//   `cgs_passes` times), plus the new d_A entry q_A^T S_A b (eq. dA_update).  Grid = two
//   thread-block clusters: cluster 0 appends to (Q_A, R_A), cluster 1 to (Q_L, R_L).  CTA r of
//   a cluster owns rows [r R, (r+1) R) of the s-dimensional sketch space and stages its slice
//   of Q (all d columns) in shared memory with coalesced loads, so each projection pass is
//   one local matrix-vector product, one all-to-all push of d partial dot products through
//   distributed shared memory, one cluster barrier and one local update; one more exchange gives the
//   norm and the new d_A entry.  A barrier after pushes costs about a microsecond and sets the pace, so
//   there are three of them (one per pass and one for the scalars), and what earlier iterations wrote is
//   loaded before the preceding kernel has finished (programmatic dependent launch).
// k_stacked_solve (K3): the projected problem of eq. (projected_sketched_bis),
//   y = argmin ||[R_A; sqrt(lam) R_L] y - [d_A; 0]||, by the same classical Gram-Schmidt
//   append on the stacked 2d x d matrix M (rows in creation order: A-row j, L-row j).  An
//   explicit orthonormal factor Q_T (2d x d) gives M = Q_T T with T upper triangular;
//   z = Q_T^T [d_A; 0] gains one entry per step.  T^{-1} is bordered one column at a time
//   (X' = [[X, -X t / theta], [0, 1 / theta]]) and kept in both column- and row-major order,
//   so y = X z and the refinement's X X^T g are warp-per-row products.
// k_refine_solve2: y -= X X^T g with g the FP64 sum of the refinement partials.
//
// All cluster-wide scalars are reduced in the same order in every CTA (deterministic).  The
// two clusters of k_qr_append never wait on each other and never write the shared `stop` /
// `status` words; k_stacked_solve (one cluster) reads their per-launch results and decides.
#include <math.h>

#include "ff.cuh"
#include "sgks_internal.cuh"

namespace sgks {

// FP64 on GB300: a warp's FP64 instruction takes its quarter of the SM for 64 cycles, whatever its lanes do
// and whether or not it depends on the one before; the quarters run side by side.  What counts is thus
// the number of FP64 warp instructions per quarter: sums run with one accumulator per lane, the lanes per
// sum are chosen for each step (best_group), and independent scalars go to different warps.  Every order
// is fixed and the same in every CTA, so all CTAs obtain bit-identical values.
// lanes (a power of two, as its logarithm) that share one sum of `len` products when the CTA forms `items`
// of them: the fewest FP64 warp instructions on the busiest quarter of the SM
__device__ __forceinline__ int best_group(int items, int len) {
    int best = 0, cost = 0x7fffffff;
#pragma unroll
    for (int lg = 0; lg <= 5; ++lg) {
        const int warps = ((items << lg) + 31) >> 5;
        const int c = ((warps + 3) >> 2) * (((len + (1 << lg) - 1) >> lg) + lg);
        if (c < cost) {
            cost = c;
            best = lg;
        }
    }
    return best;
}

// out(i, sum over k < len of term(i, k)) for i < items, 2^lg lanes per sum; out is called in the lanes
// lane, lane + 2^lg, ... of the group, which it is told.
template <typename Term, typename Out>
__device__ __forceinline__ void group_sums(int items, int len, int lg, Term term, Out out) {
    const int g = 1 << lg;
    for (int base = 0; base < (items << lg); base += kThreads) {
        const int t = base + threadIdx.x, i = t >> lg, l = t & (g - 1);
        if (base + (int)(threadIdx.x & ~31) >= (items << lg)) break;   // a warp without work
        const bool act = i < items;
        double a = 0.0;
        if (act)
#pragma unroll 4
            for (int k = l; k < len; k += g) a = term(i, k, a);
        for (int o = g >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (act) out(i, a, l, g);
    }
}

// In the calling warp: the sum of v(i) over i < count (<= kThreads), in every lane.
template <typename V>
__device__ __forceinline__ double warp_total(int count, V v) {
    const int lane = lane_id();
    double a = lane < count ? v(lane) : 0.0;
    for (int i = lane + 32; i < count; i += 32) a += v(i);
    for (int o = count > 16 ? 16 : (count > 8 ? 8 : (count > 4 ? 4 : 2)); o > 0; o >>= 1)
        a += __shfl_xor_sync(0xffffffffu, a, o);
    return __shfl_sync(0xffffffffu, a, 0);
}

// Copies `total` values with the CTA's threads: each thread issues up to eight loads (ld(idx))
// before it stores them (st(idx, value)).
template <typename Ld, typename St>
__device__ __forceinline__ void stage_batched(int total, Ld ld, St st) {
    constexpr int U = 8;
    for (int base = threadIdx.x; base < total; base += U * kThreads) {
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * kThreads;
            v[u] = idx < total ? ld(idx) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * kThreads;
            if (idx < total) st(idx, v[u]);
        }
    }
}

// sqrt(a) and 1 / sqrt(a) (0 for a = 0).  The library's square root and division are long dependent chains,
// and a dependent FP64 operation takes ~68 cycles here: 2.7 us for both on one thread.  From the FP32
// reciprocal root y of the mantissa m (a = m 4^k, 1 <= m < 4), r = 1 - m y^2 ~ 2^-21, one step of the third
// order, y (1 + r / 2 + 3 r^2 / 8), gives 1 / sqrt(m) to about an ulp (the binomial series of (1 - r)^(-1/2));
// the root s = m y and its reciprocal then each take one Newton correction from their exact residuals
// (Markstein 1990), nine dependent operations in all.
__device__ __forceinline__ void root_pair(double a, double* root, double* inv) {
    const int hi = __double2hiint(a), e = (hi >> 20) - 1023;
    if (hi < 0x00100000 || hi >= 0x7ff00000) {   // 0, subnormal, negative, infinite or NaN
        *root = sqrt(a);
        *inv = *root == 0.0 ? 0.0 : 1.0 / *root;
        return;
    }
    const int k2 = e & ~1;   // even part of the exponent
    const double m = __hiloint2double(hi - (k2 << 20), __double2loint(a));
    const double y0 = (double)rsqrtf((float)m);
    const double r = fma(-(m * y0), y0, 1.0);
    const double y = fma(y0 * r, fma(0.375, r, 0.5), y0);
    const double s0 = m * y;
    const double s = fma(fma(-s0, s0, m), 0.5 * y, s0);
    const double z = fma(fma(-s, y, 1.0), y, y);
    const int half = k2 / 2;
    *root = __hiloint2double(__double2hiint(s) + half * 0x100000, __double2loint(s));
    *inv = __hiloint2double(__double2hiint(z) - half * 0x100000, __double2loint(z));
}

// y_i, and its float-float copy where a batch keeps one
__device__ __forceinline__ void put_y(const Small& S, int i, double y) {
    S.y[i] = y;
    if (S.y2) S.y2[(size_t)i * S.y2_stride] = dsplit(y);
}

// v into element idx of `local` in every CTA of the cluster, by the lanes first, first + step, ...
template <int CS>
__device__ __forceinline__ void push(cg::cluster_group& cl, double* local, int idx, double v, int first, int step) {
    for (int r = first; r < CS; r += step) cl.map_shared_rank(local, r)[idx] = v;
}

// Shared-memory plan of k_qr_append (doubles): Qs[dq_max * RP] | v[R] | sb[R] | cbuf[2*CS*dm] |
// c[dm] | p[dm] | red[3*CS] | scratch[8].  nbuf: halves of cbuf, one where two do not fit.
__host__ __device__ inline size_t qr_append_smem(int s, int dm, int cs, int nbuf) {
    const int R = (s + cs - 1) / cs, RP = R | 1;
    return sizeof(double) * ((size_t)dm * RP + 2 * (size_t)R + nbuf * (size_t)cs * dm + 2 * (size_t)dm + 3 * cs + 8);
}

// k_stacked_solve (doubles): QTs[dm * RP2] | v[R2] | da[R2] | cbuf[nbuf*CS*dm] | c[dm] | tau[dm] | red[2*CS] |
// scratch[8].  It bounds dm below 420 (227 KB), so a CTA's rows R2 <= 105 < kThreads.
__host__ __device__ inline size_t stacked_smem(int dm, int cs, int nbuf) {
    const int R2 = (2 * dm + cs - 1) / cs, RP2 = R2 | 1;
    return sizeof(double) * ((size_t)dm * RP2 + 2 * (size_t)R2 + nbuf * (size_t)cs * dm + 2 * (size_t)dm + 2 * cs + 8);
}

template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kThreads)
    k_qr_append(Dims D, Small S0, const Small* __restrict__ Sarr, int nbuf) {
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();   // every CTA of the cluster has started once the matching wait returns
    const int rank = (int)cl.block_rank();
    const int fac = (blockIdx.x / CS) & 1;  // 0: S_A A W, 1: S_L L W
    const Small S = Sarr ? Sarr[blockIdx.x / (2 * CS)] : S0;
    const int tid = threadIdx.x, warp = warp_id(), lane = lane_id();
    const int s = D.s, dm = D.dmax;
    const int R = (s + CS - 1) / CS, RP = R | 1;
    const int i0 = rank * R;
    const int nr = max(0, min(s, i0 + R) - i0);

    extern __shared__ __align__(16) double sm[];
    double* Qs = sm;                               // [dq][RP]
    double* v = Qs + (size_t)dm * RP;              // [R]
    double* sb = v + R;                            // [R]
    double* cbuf = sb + R;                         // [nbuf][CS][dm], the halves in turn
    double* c = cbuf + nbuf * (size_t)CS * dm;     // [dm]
    double* p = c + dm;                            // [dm]
    double* red = p + dm;                          // [3][CS]
    double* scratch = red + 3 * CS;                // [8]

    double* Q = fac ? S.QL : S.QA;
    double* Rm = fac ? S.RL : S.RA;
    const double* part = fac ? S.partL : S.partA;
    const int np = fac ? D.npL : D.npA;
    const DevScalars* sc = S.sc;

    // Before the kernel in front of this one (the sketch) has finished: the Q slice, which earlier
    // iterations wrote (coalesced along rows of each column, eight loads per thread in flight before
    // their stores: the global source could alias the shared destination as far as the compiler
    // knows, so a plain copy loop would wait for each load in turn).
    const int dq = min(__ldcg(&sc->d), dm);
    stage_batched(dq * nr, [&](int idx) {
        const int j = idx / nr, li = idx - j * nr;
        return __ldcg(Q + (size_t)j * s + i0 + li);
    }, [&](int idx, double val) {
        const int j = idx / nr, li = idx - j * nr;
        Qs[(size_t)j * RP + li] = val;
    });
    const bool own = tid < nr;   // nr <= kMaxS / 8 = kThreads
    if (fac == 0 && own) sb[tid] = __ldcg(S.Sb + i0 + tid);
    for (int j = tid; j < dq; j += kThreads) p[j] = 0.0;
    const int lg_dot = best_group(dq, nr), lg_sum = best_group(dq, CS), lg_upd = best_group(nr, dq);
    pdl_wait();   // the new sketched column and the stop flag are valid from here on
    pdl_trigger();
    cl.barrier_wait();
    if (sc->stop) return;
    if (sc->status == ST_SKETCH || dq >= dm) return;   // k_stacked_solve reports it

    // own row of the new sketched column
    if (np == 1) {
        if (own) v[tid] = __ldcg(part + i0 + tid) * D.sketch_scale;
    } else {   // several sketch partials: warp per row, lanes over the partials
        for (int li = warp; li < nr; li += kWarps) {
            double a = 0.0;
            for (int b = lane; b < np; b += 32) a += part[(size_t)b * s + i0 + li];
            a = warp_sum(a);
            if (lane == 0) v[li] = a * D.sketch_scale;
        }
    }
    __syncthreads();
    for (int pass = 0; pass < D.cgs_passes; ++pass) {
        double* cb = cbuf + (nbuf == 2 ? (size_t)(pass & 1) * CS * dm : 0);
        // partial c_j over own rows, pushed to every CTA
        group_sums(dq, nr, lg_dot, [&](int j, int k, double a) { return fma(Qs[(size_t)j * RP + k], v[k], a); },
                   [&](int j, double a, int l, int g) { push<CS>(cl, cb + (size_t)rank * dm, j, a, l, g); });
        if (pass == 0) {
            if (warp == kWarps - 1) {   // ||u||^2 for the breakdown test
                const double un = warp_total(nr, [&](int i) { return v[i] * v[i]; });
                push<CS>(cl, red, rank, un, lane, 32);
            }
        } else if (rank == 0) {
            for (int j = tid; j < dq; j += kThreads) p[j] += c[j];
        }
        // The pushes of all CTAs have landed.  With two halves the next pass fills the other one, and the
        // pass after it comes behind a further barrier; with one, a second barrier ends the pass.
        cl.sync();
        group_sums(dq, CS, lg_sum, [&](int j, int k, double a) { return a + cb[(size_t)k * dm + j]; },
                   [&](int j, double a, int l, int) { if (l == 0) c[j] = a; });
        __syncthreads();
        // v -= Q c over own rows
        group_sums(nr, dq, lg_upd, [&](int i, int k, double a) { return fma(Qs[(size_t)k * RP + i], c[k], a); },
                   [&](int i, double a, int l, int) { if (l == 0) v[i] -= a; });
        if (nbuf == 1) cl.sync();
        else __syncthreads();
    }
    // ||v||^2 and v^T S_A b (the d_A entry is q^T S_A b = v^T S_A b / rho) in one exchange
    if (warp == 0) {
        const double rr = warp_total(nr, [&](int i) { return v[i] * v[i]; });
        push<CS>(cl, red + CS, rank, rr, lane, 32);
    } else if (warp == 1 && fac == 0) {
        const double dp = warp_total(nr, [&](int i) { return v[i] * sb[i]; });
        push<CS>(cl, red + 2 * CS, rank, dp, lane, 32);
    } else if (warp >= 2 && rank == 0) {
        for (int j = tid - 64; j < dq; j += kThreads - 64) p[j] += c[j];
    }
    cl.sync();
    // the scalars, each in a warp of its own, broadcast through shared memory
    if (warp < 3) {
        const double a = warp_total(CS, [&](int i) { return red[(warp == 0 ? CS : (warp == 1 ? 0 : 2 * CS)) + i]; });
        if (warp == 0) {
            double rho, inv;
            root_pair(a, &rho, &inv);
            if (lane == 0) {
                scratch[0] = rho;
                scratch[1] = inv;
                scratch[2] = isfinite(a) ? 1.0 : 0.0;
            }
        } else if (warp == 1) {
            double un, unused;
            root_pair(a, &un, &unused);
            if (lane == 0) {
                scratch[3] = 1e-13 * un;
                scratch[4] = isfinite(a) ? 1.0 : 0.0;
            }
        } else if (lane == 0) {
            scratch[5] = a;
        }
    }
    __syncthreads();
    const bool brk = !(scratch[0] > scratch[3]);
    const double rho = brk ? 0.0 : scratch[0], inv = brk ? 0.0 : scratch[1];
    if (rank == 0 && tid == 0) {
        double* out = S.qr_out + 4 * fac;
        out[0] = rho;
        out[1] = brk ? 1.0 : 0.0;
        out[2] = scratch[2] != 0.0 && scratch[4] != 0.0 ? 1.0 : 0.0;
        out[3] = fac || brk ? 0.0 : scratch[5] * inv;
    }
    if (own) Q[(size_t)dq * s + i0 + tid] = v[tid] * inv;   // new Q column over own rows
    if (rank == 0)
        for (int j = tid; j <= dq; j += kThreads) Rm[(size_t)dq * dm + j] = j < dq ? p[j] : rho;
}

template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kThreads)
    k_stacked_solve(Dims D, Small S0, const Small* __restrict__ Sarr, int nbuf) {
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();
    const Small S = Sarr ? Sarr[blockIdx.x / CS] : S0;
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = lane_id(), warp = warp_id();
    const int gw = warp * CS + rank, GW = CS * kWarps;   // a row of X per warp, spread over the CTAs first
    const int dm = D.dmax, ldT = 2 * dm;
    DevScalars* sc = S.sc;
    const int R2 = (2 * dm + CS - 1) / CS, RP2 = R2 | 1;
    const int r0 = rank * R2;

    extern __shared__ __align__(16) double sm[];
    double* Qs = sm;                                // [dq][RP2]
    double* v = Qs + (size_t)dm * RP2;              // [R2]
    double* da = v + R2;                            // [R2] own rows of [d_A; 0]
    double* cbuf = da + R2;                         // [nbuf][CS][dm], the halves in turn
    double* c = cbuf + nbuf * (size_t)CS * dm;      // [dm]
    double* tau = c + dm;                           // [dm]
    double* red = tau + dm;                         // [2][CS]
    double* scratch = red + 2 * CS;                 // [8]

    // Before k_qr_append has finished: what earlier iterations wrote.  The Q_T slice (column j is zero
    // below row 2j+2), the thread's row of [d_A; 0], and the warp's row of X with its part of z.
    const int dq = min(__ldcg(&sc->d), dm);
    const int N2 = 2 * dq + 2;
    const int nr = max(0, min(N2, r0 + R2) - r0);
    stage_batched(dq * nr, [&](int idx) {
        const int j = idx / nr, lr = idx - j * nr, row = r0 + lr;
        return row < 2 * j + 2 ? __ldcg(S.QT + (size_t)j * ldT + row) : 0.0;
    }, [&](int idx, double val) {
        const int j = idx / nr, lr = idx - j * nr;
        Qs[(size_t)j * RP2 + lr] = val;
    });
    for (int j = tid; j < dq; j += kThreads) tau[j] = 0.0;
    const bool own = tid < nr;
    const int orow = r0 + tid, oj = orow >> 1;
    if (own) da[tid] = !(orow & 1) && oj < dq ? __ldcg(S.dA + oj) : 0.0;
    const int lg_dot = best_group(dq, nr), lg_sum = best_group(dq, CS), lg_upd = best_group(nr, dq);
    const double sl = sqrt(S.lam);
    constexpr int XP = 4;   // entries of a row of X per lane held in registers (128 columns)
    double xpre[XP], zpre[XP];
#pragma unroll
    for (int u = 0; u < XP; ++u) {
        const int j = gw + lane + 32 * u;
        xpre[u] = gw < dq && j < dq ? __ldcg(S.Xr + (size_t)gw * dm + j) : 0.0;
        zpre[u] = gw < dq && j < dq ? __ldcg(S.z + j) : 0.0;
    }
    pdl_wait();   // the new columns of R_A, R_L and the append's results are valid from here on
    cl.barrier_wait();
    if (sc->stop) return;
    const double rhoA = S.qr_out[0], rhoL = S.qr_out[4];
    const bool brA = S.qr_out[1] != 0.0, brL = S.qr_out[5] != 0.0;
    const bool finite = S.qr_out[2] != 0.0 && S.qr_out[6] != 0.0;
    const int bad = (sc->status == ST_SKETCH) ? ST_SKETCH : (dq >= dm ? ST_FULL : (!finite ? ST_NONFINITE : (brA && brL ? ST_BREAKDOWN : 0)));
    if (bad) {
        cl.sync();   // every CTA has read stop / d / status before they change
        if (rank == 0 && tid == 0) {
            sc->status = bad;
            sc->stop = 1;
        }
        return;
    }
    const double dnew = S.qr_out[3];
    // own row of the new stacked column [p_A; sqrt(lam) p_L] in creation order
    if (own) {
        const double pn = oj < dq ? __ldcg(((orow & 1) ? S.RL : S.RA) + (size_t)dq * dm + oj) : ((orow & 1) ? rhoL : rhoA);
        v[tid] = (orow & 1) ? sl * pn : pn;
        if (oj == dq && !(orow & 1)) da[tid] = dnew;
    }
    __syncthreads();
    for (int pass = 0; pass < D.cgs_passes; ++pass) {   // as in k_qr_append
        double* cb = cbuf + (nbuf == 2 ? (size_t)(pass & 1) * CS * dm : 0);
        group_sums(dq, nr, lg_dot, [&](int j, int k, double a) { return fma(Qs[(size_t)j * RP2 + k], v[k], a); },
                   [&](int j, double a, int l, int g) { push<CS>(cl, cb + (size_t)rank * dm, j, a, l, g); });
        if (pass > 0)
            for (int j = tid; j < dq; j += kThreads) tau[j] += c[j];
        cl.sync();
        group_sums(dq, CS, lg_sum, [&](int j, int k, double a) { return a + cb[(size_t)k * dm + j]; },
                   [&](int j, double a, int l, int) { if (l == 0) c[j] = a; });
        __syncthreads();
        group_sums(nr, dq, lg_upd, [&](int i, int k, double a) { return fma(Qs[(size_t)k * RP2 + i], c[k], a); },
                   [&](int i, double a, int l, int) { if (l == 0) v[i] -= a; });
        if (nbuf == 1) cl.sync();
        else __syncthreads();
    }
    // ||v||^2 and v^T [d_A; 0] (the new entry of z is that divided by theta) in one exchange
    if (warp == 0) {
        const double rr = warp_total(nr, [&](int i) { return v[i] * v[i]; });
        push<CS>(cl, red, rank, rr, lane, 32);
    } else if (warp == 1) {
        const double zp = warp_total(nr, [&](int i) { return v[i] * da[i]; });
        push<CS>(cl, red + CS, rank, zp, lane, 32);
    } else {
        for (int j = tid - 64; j < dq; j += kThreads - 64) tau[j] += c[j];
    }
    cl.sync();
    if (warp < 2) {
        const double a = warp_total(CS, [&](int i) { return red[warp * CS + i]; });
        if (warp == 0) {
            double th, it;
            root_pair(a, &th, &it);   // > 0: at least one of rho_A, rho_L is nonzero
            if (lane == 0) {
                scratch[0] = th;
                scratch[1] = it;
            }
        } else if (lane == 0) {
            scratch[2] = a;
        }
    }
    __syncthreads();
    const double theta = scratch[0], itheta = scratch[1], zn = scratch[2] * itheta;
    if (own) S.QT[(size_t)dq * ldT + orow] = v[tid] * itheta;   // new Q_T column
    if (rank == 0) {
        for (int j = tid; j <= dq; j += kThreads) S.Tm[(size_t)dq * dm + j] = j < dq ? tau[j] : theta;
        if (tid == 0) {
            S.dA[dq] = dnew;
            S.z[dq] = zn;
        }
    }
    // X = T^{-1}: new column -X tau / theta (row i of X in the row-major copy), X[dq][dq] = 1/theta;
    // then y_i = sum_{j >= i} X(i, j) z_j with the same warp per row.
    for (int i = gw; i <= dq; i += GW) {
        const double* xr = S.Xr + (size_t)i * dm;
        double a = 0.0, b = 0.0;
#pragma unroll
        for (int u = 0; u < XP; ++u) {
            const int j = i + lane + 32 * u;
            if (j < dq) {
                const double x = i == gw ? xpre[u] : __ldcg(xr + j);
                a += x * tau[j];
                b += x * (i == gw ? zpre[u] : __ldcg(S.z + j));
            }
        }
        for (int j = i + lane + 32 * XP; j < dq; j += 32) {
            const double x = __ldcg(xr + j);
            a += x * tau[j];
            b += x * __ldcg(S.z + j);
        }
        // both sums at once: the lower half of the warp finishes a, the upper half b
        const bool up = lane & 16;
        double f = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
        a = __shfl_sync(0xffffffffu, f, 0);
        b = __shfl_sync(0xffffffffu, f, 16);
        const double xn = i < dq ? -a * itheta : itheta;
        b = fma(xn, zn, b);
        if (lane == 0) {
            S.X[(size_t)dq * dm + i] = xn;
            S.Xr[(size_t)i * dm + dq] = xn;
            put_y(S, i, b);
        }
    }
    if (rank == 0 && tid == 0) sc->d = dq + 1;
}

// y -= X X^T g on one cluster, g_j the fixed-order sum of the npart refinement partials S.gpart[b][j]; warp
// per output, lanes over the sum.  X is older than the kernel in front of this one, so the warp's first
// column and row of it are loaded before that one has finished.
template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kThreads)
    k_refine_solve2(Dims D, Small S0, const Small* __restrict__ Sarr, int npart) {
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();
    const Small S = Sarr ? Sarr[blockIdx.x / CS] : S0;
    extern __shared__ __align__(16) double sm[];
    double *g = sm, *h = sm + D.dmax;
    const int rank = (int)cl.block_rank(), lane = lane_id();
    const int gw = warp_id() * CS + rank, GW = CS * kWarps;
    const int dm = D.dmax, d = min(__ldcg(&S.sc->d), dm);
    constexpr int XP = 4;
    double xc[XP], xr[XP];   // X(j, gw) for j = lane + 32 u <= gw; X(gw, j) for j = gw + lane + 32 u
#pragma unroll
    for (int u = 0; u < XP; ++u) {
        const int j = lane + 32 * u;
        xc[u] = gw < d && j <= gw ? __ldcg(S.X + (size_t)gw * dm + j) : 0.0;
        xr[u] = gw < d && gw + j < d ? __ldcg(S.Xr + (size_t)gw * dm + gw + j) : 0.0;
    }
    pdl_wait();
    cl.barrier_wait();
    if (S.sc->stop) return;
    for (int j = gw; j < d; j += GW) {   // g_j: lanes over the partials, pushed to every CTA
        double a = 0.0;
#pragma unroll 4
        for (int b = lane; b < npart; b += 32) a += __ldcg(S.gpart + (size_t)b * dm + j);
        a = warp_sum(a);
        push<CS>(cl, g, j, a, lane, 32);
    }
    cl.sync();
    for (int i = gw; i < d; i += GW) {   // h = X^T g: column i of X (contiguous) with g[0..i]
        const double* x = S.X + (size_t)i * dm;
        double a = 0.0;
#pragma unroll
        for (int u = 0; u < XP; ++u) {
            const int j = lane + 32 * u;
            if (j <= i) a += (i == gw ? xc[u] : __ldcg(x + j)) * g[j];
        }
        for (int j = lane + 32 * XP; j <= i; j += 32) a += __ldcg(x + j) * g[j];
        a = warp_sum(a);
        push<CS>(cl, h, i, a, lane, 32);
    }
    cl.sync();
    for (int i = gw; i < d; i += GW) {   // y_i -= (X h)_i: row i of X (row-major copy)
        const double* x = S.Xr + (size_t)i * dm;
        double a = 0.0;
#pragma unroll
        for (int u = 0; u < XP; ++u) {
            const int j = i + lane + 32 * u;
            if (j < d) a += (i == gw ? xr[u] : __ldcg(x + j)) * h[j];
        }
        for (int j = i + lane + 32 * XP; j < d; j += 32) a += __ldcg(x + j) * h[j];
        a = warp_sum(a);
        if (lane == 0) put_y(S, i, S.y[i] - a);
    }
}

// ----------------------------------------------------------------------------- launchers
static size_t smem_limit() {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return (size_t)optin;
}

// halves of cbuf: two when the plan with two fits
static int halves(size_t two) { return two <= smem_limit() ? 2 : 1; }

template <int CS>
static cudaError_t config2(int s, int dm, size_t limit) {
    if (qr_append_smem(s, dm, CS, 1) > limit || stacked_smem(dm, CS, 1) > limit) return cudaErrorInvalidValue;
    cudaError_t e;
    if (CS > 8) {
        e = cudaFuncSetAttribute(k_qr_append<CS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stacked_solve<CS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_refine_solve2<CS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    e = allow_smem(k_qr_append<CS>, qr_append_smem(s, dm, CS, halves(qr_append_smem(s, dm, CS, 2))));
    if (e == cudaSuccess) e = allow_smem(k_stacked_solve<CS>, stacked_smem(dm, CS, halves(stacked_smem(dm, CS, 2))));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * CS);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = qr_append_smem(s, dm, CS, halves(qr_append_smem(s, dm, CS, 2)));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    e = cudaOccupancyMaxActiveClusters(&ncl, (void*)k_qr_append<CS>, &cfg);
    if (e != cudaSuccess) return e;
    return ncl >= 2 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

// Chooses the cluster size of the fast small path; returns an error if it cannot be used
// (the caller then falls back to the global-memory path of k_small.cu).
cudaError_t configure_small_fast(int* cluster_out, int s, int dm) {
    const size_t limit = smem_limit();
    cudaError_t e = config2<16>(s, dm, limit);
    if (e == cudaSuccess) {
        *cluster_out = 16;
        return e;
    }
    cudaGetLastError();
    e = config2<8>(s, dm, limit);
    if (e == cudaSuccess) *cluster_out = 8;
    else cudaGetLastError();
    return e;
}

template <int CS>
static cudaError_t qr_append_cs(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr, int ninst) {
    const int nbuf = halves(qr_append_smem(D.s, D.dmax, CS, 2));
    carveout_once((const void*)k_qr_append<CS>);
    return launch_pdl(k_qr_append<CS>, 2 * CS * ninst, kThreads, qr_append_smem(D.s, D.dmax, CS, nbuf), st, D, S, Sarr, nbuf);
}

template <int CS>
static cudaError_t stacked_solve_cs(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr, int ninst) {
    const int nbuf = halves(stacked_smem(D.dmax, CS, 2));
    carveout_once((const void*)k_stacked_solve<CS>);
    return launch_pdl(k_stacked_solve<CS>, CS * ninst, kThreads, stacked_smem(D.dmax, CS, nbuf), st, D, S, Sarr, nbuf);
}

cudaError_t launch_qr_append(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr, int ninst) {
    return D.cluster2 == 16 ? qr_append_cs<16>(D, S, st, Sarr, ninst) : qr_append_cs<8>(D, S, st, Sarr, ninst);
}

cudaError_t launch_stacked_solve(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr, int ninst) {
    return D.cluster2 == 16 ? stacked_solve_cs<16>(D, S, st, Sarr, ninst) : stacked_solve_cs<8>(D, S, st, Sarr, ninst);
}

cudaError_t launch_refine_solve2(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr, int ninst,
                                 int npart) {
    const int np = npart >= 0 ? npart : D.refine_np;
    const size_t smem = 2 * sizeof(double) * (size_t)D.dmax;
    if (D.cluster2 == 16) {
        carveout_once((const void*)k_refine_solve2<16>);
        return launch_pdl(k_refine_solve2<16>, 16 * ninst, kThreads, smem, st, D, S, Sarr, np);
    } else {
        carveout_once((const void*)k_refine_solve2<8>);
        return launch_pdl(k_refine_solve2<8>, 8 * ninst, kThreads, smem, st, D, S, Sarr, np);
    }
    return cudaGetLastError();
}

}  // namespace sgks
