// Internal declarations shared by the CUDA translation units of the sGKS library.
// Device-side operator rows (A, A^T, L, L^T L), the sparse-sign hash, warp reductions,
// and the launcher prototypes that the host orchestration (sgks_api.cu) calls.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <string>
#include <vector>
#include <stdint.h>

#include "../../include/sgks.h"

namespace cg = cooperative_groups;

namespace sgks {

constexpr int kThreads = 256;           // threads of every bulk kernel
constexpr int kWarps = kThreads / 32;
constexpr int kMaxS = 2048;             // largest sketch size supported
constexpr int kMaxZeta = 16;
constexpr int kClusterMax = 16;         // CTAs of the small FP64 cluster kernels
constexpr int kMaxDraws = 256;
constexpr int kFastK = 9;               // largest psf side of the register-blocked conv kernels

// ------------------------------------------------------------------------------ status
enum DevStatus : int { ST_OK = 0, ST_BREAKDOWN = 1, ST_STOPPED = 2, ST_NONFINITE = 3, ST_SKETCH = 4,
                       ST_FULL = 5, ST_TIMEOUT = 6 };

// Scalars that live on the device and are updated by the kernels, so that one captured
// graph of a step replays for every iteration.
struct DevScalars {
    int d;          // columns of W currently in the sketched QR factors
    int iter;       // iterations done since the setup
    int stop;       // nonzero: later kernels of the solve do nothing
    int status;     // DevStatus
    int ka_done;    // block counter of the combine kernel's last-block reduction
    int tol_on;     // RC stopping test active
    double tol;
    double rc_last, rre_last, rre0;
    double xt2;     // ||x_true||^2
};

// ----------------------------------------------------------------------- operator views
template <typename T, typename V>
struct DevA {
    int kind;            // SGKS_OP_*
    int64_t m, n;
    int64_t nnz;         // CSR: stored entries (0 for the other kinds)
    const int32_t* rp;   // CSR
    const int32_t* ci;
    const V* val;
    const int32_t* trp;  // CSR of A^T
    const int32_t* tci;
    const V* tval;
    // A^T once more in 32-row slices with each slice's entries interleaved by row: entry k of row
    // 32 g + t at sl_off[g] + 32 k + t (sl_len[i] entries in row i; the tail of a shorter row is
    // padding that is never read).  A warp then reads the k-th entries of 32 consecutive rows
    // together: for rows that are neighbouring pixels of a ray-based operator those entries are
    // neighbouring rays, so the gathers of e fall on few cache lines, and no row needs a
    // cross-lane sum.  Built when n >= 155,648 (enough slices to fill the GPU) and either the form
    // is FP64 or rows hold fewer than 96 entries on average; sl_off = nullptr otherwise (long FP32
    // rows run faster with 32 lanes per row, small operators with rows spread over every warp).
    const int64_t* sl_off;   // [ceil(n / 32) + 1]
    const int32_t* sl_len;   // [n]
    const int32_t* sl_ci;
    const V* sl_val;
    const T* dense;      // row-major m x ld
    int64_t ld;
    int nx, ny, kh, kw;  // conv2d
    const T* psf;
    // conv2d with a square K x K psf, K <= kFastK, and nx % 4 == 0: the tap values as launch
    // parameters (read from the constant bank by the register-blocked kernels of k_conv.cu);
    // kfast = K, or 0 when those kernels do not apply.
    int kfast;
    T tk[kFastK * kFastK];
};

struct DevL {
    int kind;            // SGKS_REG_*
    int nx, ny, nt;
    int64_t n, p;
};

// --------------------------------------------------------------------------- utilities
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }

// ---------------------------------------------------------- bulk copies (TMA) and mbarriers
// One elected thread moves a contiguous global range into shared memory with cp.async.bulk and
// an mbarrier counts the bytes; the other threads wait on the barrier's phase.  Every wait is
// bounded: after kWaitTries unsuccessful try_wait rounds it reports failure, and the caller
// records ST_TIMEOUT, drains its own copies (again bounded) and returns.
constexpr int kWaitTries = 1 << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// orders this thread's earlier generic-proxy shared-memory accesses before later bulk copies
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// dst and src 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// one arrival (release at CTA scope) on a barrier counting thread arrivals
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    for (int i = 0; i < kWaitTries; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// the same with a caller-chosen number of rounds (0: report failure without waiting)
__device__ __forceinline__ bool mbar_wait_n(uint64_t* bar, uint32_t parity, int tries) {
    for (int i = 0; i < tries; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// ----------------------------------------------------- programmatic dependent launch (PDL)
// The kernels of one iteration follow each other on one stream.  Launched with the
// programmatic-serialization attribute (launch_pdl), a kernel starts as soon as every CTA of the
// kernel before it has exited or called pdl_trigger, without waiting for that grid's completion
// to be processed; its CTAs then wait in pdl_wait until the predecessor has finished and its writes
// are visible.  This overlaps each kernel's launch and CTA start-up with its predecessor.  Rules:
// - every kernel launched with launch_pdl calls pdl_wait, in every CTA, before it writes global memory
//   and before it reads what its predecessor or any kernel still running may write;
// - a kernel calls pdl_trigger only after its own pdl_wait, also where it is launched plainly today (the
//   wait then does nothing).  So when a kernel starts, its predecessor has passed its wait, and everything
//   before the predecessor is complete and visible;
// - what may be read before pdl_wait is therefore what neither the predecessor nor this kernel writes: data
//   fixed since the handle's creation (sketch entries, k_sketch.cu) and the factors and scalars that
//   earlier kernels left (k_small2.cu: d, Q_A, Q_L, Q_T, X, z, d_A and S_A b, which the sketch, gradient
//   and refinement kernels in front of it only read).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel's CTAs start while this one still runs (its pdl_wait returns when this one has
// finished); after pdl_wait, see above.  Used where the next kernel is one of the small FP64 cluster
// kernels: 16 to 64 CTAs that fit beside the others and have an earlier state to load (k_small2.cu).  Before
// a large kernel it does not pay: the waiting CTAs hold SM resources through the whole predecessor.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// SGKS_PDL=0 in the environment launches plainly (for comparison); default on.
bool pdl_enabled();

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Quotient of a non-negative index by a positive divisor, as a 32-bit division when both fit in
// 32 bits (a 64-bit division is a long instruction sequence; the stencil and convolution rows
// decompose an index for every row they compute).
__device__ __forceinline__ int64_t qdiv(int64_t a, int64_t b) {
    return (((uint64_t)a | (uint64_t)b) >> 32) == 0 ? (int64_t)((uint32_t)a / (uint32_t)b) : a / b;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename T>
__device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }

// Warp sum of a per-lane partial: FP32 shuffles for the FP32 form (FP32 accumulation),
// FP64 for the FP64 form; the cross-warp and cross-CTA sums are FP64 in both.
template <typename T>
__device__ __forceinline__ double warp_sum_acc(T v) { return (double)warp_sum(v); }

// Sums over the warp of R values per lane: at each step half of the lanes take over half of the
// values, until a lane holds one row's sum; lane & (32 / R - 1) == 0 then holds row lane / (32 / R).
template <int R, typename T>
__device__ __forceinline__ T warp_sum_rows(T (&a)[R]) {
    const int lane = lane_id();
    int off = 16;
#pragma unroll
    for (int h = R / 2; h >= 1; h >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T keep = up ? a[i + h] : a[i], send = up ? a[i] : a[i + h];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    T v = a[0];
    for (; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Sum of part[0 .. nb) over the calling warp (lanes over the entries), in every lane.
__device__ __forceinline__ double warp_sum_parts(const double* part, int nb, int stride = 1) {
    double a = 0.0;
#pragma unroll 4
    for (int b = lane_id(); b < nb; b += 32) a += __ldcg(part + (size_t)b * stride);
    return warp_sum(a);
}

// acc[j] += sum over q < rows of Q[j ld + q] us[q], j < d: two columns per warp and step, lanes over the
// rows, products in T; the two sums share their reduction (an FP64 warp instruction takes a quarter of the
// SM for 64 clocks).  us and acc in shared memory, acc[j] owned by the warp that takes column j.
template <typename T>
__device__ __forceinline__ void tile_dots(const T* __restrict__ Q, size_t ld, const T* us, int rows, int d, double* acc) {
    for (int j = 2 * warp_id(); j < d; j += 2 * kWarps) {
        const T *q0 = Q + (size_t)j * ld, *q1 = j + 1 < d ? q0 + ld : q0;
        T a0 = T(0), a1 = T(0);
#pragma unroll 4
        for (int q = lane_id(); q < rows; q += 32) {
            const T u = us[q];
            a0 += q0[q] * u;
            a1 += q1[q] * u;
        }
        double s[2] = {(double)a0, (double)a1};
        const double v = warp_sum_rows<2>(s);
        const int c = j + (lane_id() >> 4);
        if ((lane_id() & 15) == 0 && c < d) acc[c] += v;
    }
}

// Fixed pairwise tree over N values with a stride (deterministic, log2 depth).
template <int N>
__device__ __forceinline__ double tree_sumd(const double* a, int stride = 1) {
    if constexpr (N == 1) {
        return a[0];
    } else {
        return tree_sumd<N / 2>(a, stride) + tree_sumd<N / 2>(a + (N / 2) * stride, stride);
    }
}

// Shared-memory carveout: when SGKS_CARVEOUT (0..100) is set, every library kernel gets that
// preferred carveout on its first launch, so consecutive kernels need no SM reconfiguration.
void carveout_once(const void* kernel);

// More than 48 KB of shared memory has to be allowed kernel by kernel, and the limit belongs to the process: a
// handle of another size, or another host thread between this call and the launch, changes it for everyone.  So it
// is only ever raised, at once to all that a CTA can have.  cudaErrorInvalidValue where that is less than `bytes`.
cudaError_t allow_smem(const void* kernel, size_t bytes);
template <typename... KArgs>
cudaError_t allow_smem(void (*kernel)(KArgs...), size_t bytes) {
    return allow_smem((const void*)kernel, bytes);
}

// SplitMix64 output function (Steele, Lea, Flood 2014).
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__host__ __device__ __forceinline__ uint64_t sketch_key_host_dev(uint64_t seed, int stream) {
    uint64_t z = 2ull * seed + (uint64_t)stream;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Rows and signs of the sparse-sign column j: the k-th accepted draw is the first draw
// c (counting on from the previous acceptance) whose row differs from rows[0..k-1].
// Returns false when the 256-draw limit is hit.
template <int ZMAX>
__device__ __forceinline__ bool sparse_sign_column(uint64_t key, uint64_t j, int s, int zeta,
                                                   int (&rows)[ZMAX], uint32_t& negmask) {
    int c = 0;
    bool ok = true;
    negmask = 0u;
#pragma unroll
    for (int k = 0; k < ZMAX; ++k) {
        rows[k] = -1;
        if (k < zeta) {
            while (true) {
                if (c >= kMaxDraws) { ok = false; rows[k] = 0; break; }
                const uint64_t hv = mix64(key ^ ((j << 8) | (uint64_t)c));
                ++c;
                const int r = (int)(((hv >> 32) * (uint64_t)s) >> 32);
                bool dup = false;
#pragma unroll
                for (int t = 0; t < ZMAX; ++t)
                    if (t < k && rows[t] == r) dup = true;
                if (!dup) {
                    rows[k] = r;
                    if (hv & 1ull) negmask |= (1u << k);
                    break;
                }
            }
        }
    }
    return ok;
}

// --------------------------------------------------------------- rows of A (forward)
// Warp-cooperative rows (CSR, dense): every lane returns the full row value.
template <typename T, typename V>
__device__ __forceinline__ T a_row_warp(const DevA<T, V>& A, int64_t j, const T* __restrict__ x) {
    const int lane = lane_id();
    T acc = T(0);
    if (A.kind == SGKS_OP_CSR) {
        const int b = A.rp[j], e = A.rp[j + 1];
        int k = b + lane;
        for (; k + 96 < e; k += 128) {
            const int c0 = ldg(A.ci + k), c1 = ldg(A.ci + k + 32), c2 = ldg(A.ci + k + 64), c3 = ldg(A.ci + k + 96);
            const T v0 = (T)ldg(A.val + k), v1 = (T)ldg(A.val + k + 32), v2 = (T)ldg(A.val + k + 64),
                    v3 = (T)ldg(A.val + k + 96);
            acc += v0 * ldg(x + c0);
            acc += v1 * ldg(x + c1);
            acc += v2 * ldg(x + c2);
            acc += v3 * ldg(x + c3);
        }
        for (; k < e; k += 32) acc += (T)ldg(A.val + k) * ldg(x + ldg(A.ci + k));
    } else {  // dense row-major
        const T* row = A.dense + j * A.ld;
        for (int64_t k = lane; k < A.n; k += 32) acc += ldg(row + k) * ldg(x + k);
    }
    return warp_sum(acc);
}

// Rows i0 + t GW (t < 32) of a CSR matrix times x, LPR lanes per row (32 / LPR rows at a time):
// lane l of a row's group sums the entries b + l, b + l + LPR, ... and the group combines them by
// a fixed xor tree; the result of row i0 + t GW ends in lane t (0 past nrows).  Short rows take
// fewer lanes, so that a row does not pay a 32-lane reduction for a few dozen entries (in FP64
// each reduction step is a warp instruction on GB300's narrow FP64 pipe).
template <typename T, typename V, int LPR>
__device__ __forceinline__ T csr_rows_rr(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                         const V* __restrict__ val, const T* __restrict__ x, int64_t i0, int64_t GW,
                                         int64_t nrows) {
    constexpr int RPW = 32 / LPR;
    const int lane = lane_id(), sub = lane / LPR, sl = lane % LPR;
    T mine = T(0);
#pragma unroll 1
    for (int p = 0; p < LPR; ++p) {
        if (i0 + (int64_t)(p * RPW) * GW >= nrows) break;   // warp-uniform: rows grow with t
        const int64_t row = i0 + (int64_t)(p * RPW + sub) * GW;
        T acc = T(0);
        if (row < nrows) {
            const int b = rp[row], e = rp[row + 1];
#pragma unroll 4
            for (int k = b + sl; k < e; k += LPR) acc += (T)ldg(val + k) * ldg(x + ldg(ci + k));
        }
#pragma unroll
        for (int off = LPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        const int s = lane - p * RPW;   // this lane's row within the pass, if any
        const T v = __shfl_sync(0xffffffffu, acc, (s >= 0 && s < RPW ? s : 0) * LPR);
        if (s >= 0 && s < RPW) mine = v;
    }
    return mine;
}

// Rows 32 g .. 32 g + 31 of A^T v from the interleaved slices: lane t returns row 32 g + t (0
// past the last row).  Each lane runs its own row with eight entries in flight, entry k going to
// accumulator k mod 8; the accumulators are summed pairwise at the end.
template <typename T, typename V>
__device__ __forceinline__ T sell_rows(const DevA<T, V>& A, const T* __restrict__ v, int64_t g, int64_t rows) {
    constexpr int U = 8;
    const int lane = lane_id();
    const int64_t row = g * 32 + lane;
    if (row >= rows) return T(0);
    const int len = A.sl_len[row];
    const int64_t o = A.sl_off[g] + lane;
    const int32_t* ci = A.sl_ci + o;
    const V* va = A.sl_val + o;
    T acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) acc[u] = T(0);
    int k = 0;
    for (; k + U <= len; k += U) {
        int c[U];
        T w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = ldg(ci + 32 * (k + u));
            w[u] = (T)ldg(va + 32 * (k + u));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] += w[u] * ldg(v + c[u]);
    }
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (k + u < len) acc[u] += (T)ldg(va + 32 * (k + u)) * ldg(v + ldg(ci + 32 * (k + u)));
    return ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
}

// lanes per CSR row for rows of `avg` entries on average
inline int csr_lanes_per_row(int64_t nnz, int64_t rows) {
    const int64_t avg = rows > 0 ? nnz / rows : 0;
    return avg >= 96 ? 32 : (avg >= 48 ? 16 : (avg >= 16 ? 8 : 4));
}

// Thread-level rows (2D convolution).
template <typename T, typename V>
__device__ __forceinline__ T a_row_conv(const DevA<T, V>& A, const T* __restrict__ psf_s, int64_t j,
                                        const T* __restrict__ x) {
    const int nx = A.nx, ny = A.ny, kh = A.kh, kw = A.kw;
    const int iy = (int)qdiv(j, nx), ix = (int)(j - (int64_t)iy * nx);
    T acc = T(0);
    for (int a = 0; a < kh; ++a) {
        const int yy = iy - a + kh / 2;
        if (yy < 0 || yy >= ny) continue;
        const T* xr = x + (int64_t)yy * nx;
        const T* pr = psf_s + a * kw;
        for (int c = 0; c < kw; ++c) {
            const int xx = ix - c + kw / 2;
            if (xx >= 0 && xx < nx) acc += pr[c] * ldg(xr + xx);
        }
    }
    return acc;
}

// --------------------------------------------------------------- rows of A^T (adjoint)
template <typename T, typename V>
__device__ __forceinline__ T at_row_warp(const DevA<T, V>& A, int64_t i, const T* __restrict__ e) {
    const int lane = lane_id();
    T acc = T(0);
    if (A.kind == SGKS_OP_CSR) {
        const int b = A.trp[i], en = A.trp[i + 1];
        int k = b + lane;
        for (; k + 96 < en; k += 128) {
            const int c0 = ldg(A.tci + k), c1 = ldg(A.tci + k + 32), c2 = ldg(A.tci + k + 64),
                      c3 = ldg(A.tci + k + 96);
            const T v0 = (T)ldg(A.tval + k), v1 = (T)ldg(A.tval + k + 32), v2 = (T)ldg(A.tval + k + 64),
                    v3 = (T)ldg(A.tval + k + 96);
            acc += v0 * ldg(e + c0);
            acc += v1 * ldg(e + c1);
            acc += v2 * ldg(e + c2);
            acc += v3 * ldg(e + c3);
        }
        for (; k < en; k += 32) acc += (T)ldg(A.tval + k) * ldg(e + ldg(A.tci + k));
    } else {  // dense: column i
        for (int64_t k = lane; k < A.m; k += 32) acc += ldg(A.dense + k * A.ld + i) * ldg(e + k);
    }
    return warp_sum(acc);
}

template <typename T, typename V>
__device__ __forceinline__ T at_row_conv(const DevA<T, V>& A, const T* __restrict__ psf_s, int64_t i,
                                         const T* __restrict__ e) {
    const int nx = A.nx, ny = A.ny, kh = A.kh, kw = A.kw;
    const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
    T acc = T(0);
    for (int a = 0; a < kh; ++a) {
        const int yy = iy + a - kh / 2;
        if (yy < 0 || yy >= ny) continue;
        const T* er = e + (int64_t)yy * nx;
        const T* pr = psf_s + a * kw;
        for (int c = 0; c < kw; ++c) {
            const int xx = ix + c - kw / 2;
            if (xx >= 0 && xx < nx) acc += pr[c] * ldg(er + xx);
        }
    }
    return acc;
}

// -------------------------------------------------------------- rows of L and of L^T L
// The stencil rows read the vector through an accessor X(q) (element q of the vector), so the
// same definitions serve the single-instance layout (X(q) = x[q]) and the instance-interleaved
// batched layout (X(q) = x[q * B + b]).
template <typename T>
struct Unit {
    const T* __restrict__ p;
    __device__ __forceinline__ T operator()(int64_t q) const { return ldg(p + q); }
};
template <typename T>
struct Strided {
    const T* __restrict__ p;
    int64_t st;
    __device__ __forceinline__ T operator()(int64_t q) const { return ldg(p + q * st); }
};

// VV values of consecutive instances handled as one number by the stencil rows (elementwise
// arithmetic, the same operations per instance as with T), so that one index decomposition of
// a row serves all VV instances.
template <typename T, int VV>
struct VecN {
    T v[VV];
    __device__ __forceinline__ VecN() {}
    __device__ __forceinline__ VecN(T s) {
#pragma unroll
        for (int k = 0; k < VV; ++k) v[k] = s;
    }
    __device__ __forceinline__ VecN& operator+=(const VecN& o) {
#pragma unroll
        for (int k = 0; k < VV; ++k) v[k] += o.v[k];
        return *this;
    }
    __device__ __forceinline__ VecN& operator-=(const VecN& o) {
#pragma unroll
        for (int k = 0; k < VV; ++k) v[k] -= o.v[k];
        return *this;
    }
};
template <typename T, int VV>
__device__ __forceinline__ VecN<T, VV> operator+(VecN<T, VV> a, const VecN<T, VV>& b) { return a += b; }
template <typename T, int VV>
__device__ __forceinline__ VecN<T, VV> operator-(VecN<T, VV> a, const VecN<T, VV>& b) { return a -= b; }
template <typename T, int VV>
__device__ __forceinline__ VecN<T, VV> operator*(const VecN<T, VV>& a, const VecN<T, VV>& b) {
    VecN<T, VV> r;
#pragma unroll
    for (int k = 0; k < VV; ++k) r.v[k] = a.v[k] * b.v[k];
    return r;
}
// element q of VV interleaved instance vectors: p[q st + k], k < VV
template <typename T, int VV>
struct StridedVec {
    const T* __restrict__ p;
    int64_t st;
    __device__ __forceinline__ VecN<T, VV> operator()(int64_t q) const {
        VecN<T, VV> r;
#pragma unroll
        for (int k = 0; k < VV; ++k) r.v[k] = ldg(p + q * st + k);
        return r;
    }
};

template <typename T, typename X>
__device__ __forceinline__ T l_row_x(const DevL& L, int64_t k, const X& x) {
    const int nx = L.nx, ny = L.ny;
    switch (L.kind) {
        case SGKS_REG_FD1:
            return x(k + 1) - x(k);
        case SGKS_REG_GRAD2D: {
            const int64_t nh = (int64_t)ny * (nx - 1);
            if (k < nh) {
                const int64_t iy = qdiv(k, nx - 1), ix = k - iy * (nx - 1);
                const int64_t q = iy * nx + ix;
                return x(q + 1) - x(q);
            }
            const int64_t q = k - nh;  // (iy, ix) with iy < ny-1
            return x(q + nx) - x(q);
        }
        case SGKS_REG_LAPLACE2D: {
            const int iy = (int)qdiv(k, nx), ix = (int)(k - (int64_t)iy * nx);
            T v = T(4) * x(k);
            if (ix > 0) v -= x(k - 1);
            if (ix < nx - 1) v -= x(k + 1);
            if (iy > 0) v -= x(k - nx);
            if (iy < ny - 1) v -= x(k + nx);
            return v;
        }
        default: {  // SPACETIME
            const int64_t per = (int64_t)ny * (nx - 1), per2 = (int64_t)(ny - 1) * nx;
            const int64_t n1 = per * L.nt, n2 = per2 * L.nt;
            const int64_t fr = (int64_t)nx * ny;
            if (k < n1) {
                const int64_t t = qdiv(k, per), r = k - t * per;
                const int64_t iy = qdiv(r, nx - 1), ix = r - iy * (nx - 1);
                const int64_t q = t * fr + iy * nx + ix;
                return x(q + 1) - x(q);
            }
            if (k < n1 + n2) {
                const int64_t kk = k - n1;
                const int64_t t = qdiv(kk, per2), r = kk - t * per2;
                const int64_t q = t * fr + r;
                return x(q + nx) - x(q);
            }
            const int64_t q = k - n1 - n2;
            return x(q + fr) - x(q);
        }
    }
}

// (L^T L x)_i, fused: for a first-difference block D along one axis, (D^T D x)_i =
// [i not last](x_i - x_{i+1}) + [i not first](x_i - x_{i-1}).
template <typename T, typename X>
__device__ __forceinline__ T fd_pair_x(const X& x, int64_t i, int64_t stride, int pos, int len) {
    const T xi = x(i);
    T v = T(0);
    if (pos < len - 1) v += xi - x(i + stride);
    if (pos > 0) v += xi - x(i - stride);
    return v;
}

template <typename T, typename X>
__device__ __forceinline__ T lap5_x(const X& x, int iy, int ix, int nx, int ny) {
    const int64_t q = (int64_t)iy * nx + ix;
    T v = T(4) * x(q);
    if (ix > 0) v -= x(q - 1);
    if (ix < nx - 1) v -= x(q + 1);
    if (iy > 0) v -= x(q - nx);
    if (iy < ny - 1) v -= x(q + nx);
    return v;
}

template <typename T, typename X>
__device__ __forceinline__ T ltl_row_x(const DevL& L, int64_t i, const X& x) {
    const int nx = L.nx, ny = L.ny;
    switch (L.kind) {
        case SGKS_REG_FD1:
            return fd_pair_x<T>(x, i, 1, (int)i, nx);
        case SGKS_REG_GRAD2D: {
            const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
            return fd_pair_x<T>(x, i, 1, ix, nx) + fd_pair_x<T>(x, i, nx, iy, ny);
        }
        case SGKS_REG_LAPLACE2D: {  // L symmetric: L^T L = L^2, 13-point stencil
            const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
            T v = T(4) * lap5_x<T>(x, iy, ix, nx, ny);
            if (ix > 0) v -= lap5_x<T>(x, iy, ix - 1, nx, ny);
            if (ix < nx - 1) v -= lap5_x<T>(x, iy, ix + 1, nx, ny);
            if (iy > 0) v -= lap5_x<T>(x, iy - 1, ix, nx, ny);
            if (iy < ny - 1) v -= lap5_x<T>(x, iy + 1, ix, nx, ny);
            return v;
        }
        default: {  // SPACETIME
            const int64_t fr = (int64_t)nx * ny;
            const int t = (int)qdiv(i, fr);
            const int64_t r = i - (int64_t)t * fr;
            const int iy = (int)qdiv(r, nx), ix = (int)(r - (int64_t)iy * nx);
            return fd_pair_x<T>(x, i, 1, ix, nx) + fd_pair_x<T>(x, i, nx, iy, ny) + fd_pair_x<T>(x, i, fr, t, L.nt);
        }
    }
}


// (L^T v)_i for v of length p (used by sgks_apply only).
template <typename T, typename X>
__device__ __forceinline__ T lt_row_x(const DevL& L, int64_t i, const X& v) {
    const int nx = L.nx, ny = L.ny;
    switch (L.kind) {
        case SGKS_REG_FD1: {
            T a = T(0);
            if (i < nx - 1) a -= v(i);
            if (i > 0) a += v(i - 1);
            return a;
        }
        case SGKS_REG_GRAD2D: {
            const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
            const int64_t nh = (int64_t)ny * (nx - 1);
            T a = T(0);
            const int64_t h = (int64_t)iy * (nx - 1) + ix;
            if (ix < nx - 1) a -= v(h);
            if (ix > 0) a += v(h - 1);
            if (iy < ny - 1) a -= v(nh + i);
            if (iy > 0) a += v(nh + i - nx);
            return a;
        }
        case SGKS_REG_LAPLACE2D: {
            const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
            return lap5_x<T>(v, iy, ix, nx, ny);
        }
        default: {
            const int64_t fr = (int64_t)nx * ny;
            const int t = (int)qdiv(i, fr);
            const int64_t r = i - (int64_t)t * fr;
            const int iy = (int)qdiv(r, nx), ix = (int)(r - (int64_t)iy * nx);
            const int64_t per = (int64_t)ny * (nx - 1), per2 = (int64_t)(ny - 1) * nx;
            const int64_t n1 = per * L.nt, n2 = per2 * L.nt;
            T a = T(0);
            const int64_t h = (int64_t)t * per + (int64_t)iy * (nx - 1) + ix;
            if (ix < nx - 1) a -= v(h);
            if (ix > 0) a += v(h - 1);
            const int64_t g = n1 + (int64_t)t * per2 + r;
            if (iy < ny - 1) a -= v(g);
            if (iy > 0) a += v(g - nx);
            const int64_t q = n1 + n2 + i;
            if (t < L.nt - 1) a -= v(q);
            if (t > 0) a += v(q - fr);
            return a;
        }
    }
}

template <typename T>
__device__ __forceinline__ T l_row(const DevL& L, int64_t k, const T* __restrict__ x) {
    return l_row_x<T>(L, k, Unit<T>{x});
}
template <typename T>
__device__ __forceinline__ T ltl_row(const DevL& L, int64_t i, const T* __restrict__ x) {
    return ltl_row_x<T>(L, i, Unit<T>{x});
}
template <typename T>
__device__ __forceinline__ T lt_row(const DevL& L, int64_t i, const T* __restrict__ v) {
    return lt_row_x<T>(L, i, Unit<T>{v});
}

// Rows [base, base + 32) of the gradient r = A^T e + lam L^T L x (eq. gradient), lane l holding
// row base + l (0 beyond n): warp-cooperative A^T rows (CSR, dense) or one convolution row per
// lane (psf_s: the taps in shared memory).
template <typename T, typename V, bool WARPA>
__device__ __forceinline__ T grad_value(const DevA<T, V>& A, const DevL& L, const T* psf_s, const T* e, const T* x,
                                        double lam, int64_t base, int64_t n) {
    const int lane = lane_id();
    const int64_t i = base + lane;
    T adj = T(0);
    if (WARPA && A.kind == SGKS_OP_CSR && A.sl_off) {   // base is a multiple of 32: one slice of A^T
        adj = sell_rows(A, e, base >> 5, n);
    } else if (WARPA) {
        for (int r = 0; r < 32; ++r) {
            const int64_t ii = base + r;
            if (ii >= n) break;
            const T v = at_row_warp(A, ii, e);
            if (lane == r) adj = v;
        }
    } else if (i < n) {
        adj = at_row_conv(A, psf_s, i, e);
    }
    if (i >= n) return T(0);
    return adj + (T)lam * ltl_row<T>(L, i, x);
}

// ------------------------------------------------------------------------- workspace
template <typename T>
struct Bulk {                 // solver-precision arrays
    T* W;                     // [dmax][n]
    T* AW;                    // [dmax][m]
    T* x;                     // working x = W y (n)
    T* xs;                    // last accepted iterate x_k (n)
    T* e;                     // A x - b (m)
    const T* b;               // (m), handle-owned copy of the right-hand side
    const T* xtrue;           // (n) or null
    T* tmp_m;                 // scratch (m)
    T* tmp_p;                 // scratch (p)
};

// fp32x form: FP32 storage of W and b, float-float pairs (hi, lo) for A W, x, e.
struct BulkX {
    float* W;                 // [dmax][n]
    float2* AW;               // [dmax][m]
    float2* x;                // working x = W y
    float2* xs;               // last accepted iterate x_k
    float2* e;                // A x - b
    const float* b;           // handle-owned copy
    const float* xtrue;       // or null
    float* tmp_m;
    double* tmp_p;            // L w for the Gaussian sketch
};

struct Small {                // FP64 state of the sketched QR and projected solve
    double *QA, *QL, *RA, *RL;
    double *G, *X, *Tm, *zf, *dA, *y, *Sb;
    double *QT, *Xr, *z;      // fast path: orthonormal factor of [R_A; sqrt(lam) R_L], row-major T^{-1}, z
    double *qr_out;           // [8] per-launch results of k_qr_append (rho, breakdown, finite, d_A entry)
    double *partA, *partL;    // sketch partials [nb][s]
    double *gpart;            // refinement partials [nb][dmax]
    double *kapart;           // combine-kernel norm partials [nb][4]
    double *rc_hist, *rre_hist;
    DevScalars* sc;
    double lam;               // regularization parameter of this instance
    float2* y2;               // batched compensated forms: y split into (hi, lo), y2[j * y2_stride]; or null
    int y2_stride;
};

// Sparse-sign sketches stored by sketch rows: entries [ptr[r], ptr[r+1]) of idx hold the
// column index of S with the sign in bit 31 (set = -1), columns ascending.
struct SketchCSR {
    const int32_t* ptrA;
    const uint32_t* idxA;
    const int32_t* ptrL;
    const uint32_t* idxL;
};

// Dense sketches (k_dense.cu): a matrix-vector product in row groups and nc column chunks of C, its
// partials and the arrival counter of each row group (zero between launches).
struct DensePlan {
    int64_t C;
    int nc, groups;
};
struct DenseWork {
    double* part;
    int* cnt;
};

// S_A and S_L re-blocked by chunks of C columns (batched compensated forms, k_sketchx.cu): nA chunks of
// u = A w, then nL of t = L w.  The s sketch rows of a chunk, sorted by their number of entries, form
// `groups` groups of four; group id = chunk groups + g holds the rows row[4 id ..] (-1: none) and the
// quads goff[id] .. goff[id+1]: quad k is four entries (column in the chunk | sign << 31) of each of the
// four rows, at ent[4 k + place in the group]; column C holds 0.
struct SketchChunks {
    int C, nA, nL, groups;
    const int32_t* goff;
    const int32_t* row;
    const uint4* ent;
};

// ------------------------------------------------------------------------ launchers
struct Dims {
    int64_t n, m, p;
    int s, zeta, dmax, ell;
    int nbA, nbL;             // blocks of the sketch kernel for the A rows and the L rows (multiples of 8)
    int npA, npL;             // sketch partials (one per cluster of 8 blocks; 1 for the dense sketch)
    int nbG;                  // blocks of the gradient kernels (n / kThreads tiles)
    int refine_np;            // refinement partials S.gpart holds (nbG, or nbG / 8 from 8-CTA clusters)
    int nbX, nbE;             // blocks of the combine kernel (x rows, e rows)
    int cluster;              // CTAs of the small kernels (global-memory fallback path)
    int cluster2;             // CTAs per cluster of the fast small path
    int fast_small;           // 1: k_qr_append + k_stacked_solve; 0: k_append_solve (fallback)
    int sketch_kind;
    double sketch_scale;      // 1/sqrt(zeta) for sparse-sign, 1 for Gaussian
    uint64_t keyA, keyL;
    double lam;
    int cgs_passes;
    int has_xtrue;
    int max_iters;
};

// S_A (A W[:, d]) and S_L t from the column d of A W and the scratch t = L w
template <typename T>
cudaError_t launch_sketch_gather_col(const Dims& D, const Bulk<T>& B, const Small& S, const SketchCSR& SK, cudaStream_t st);
// part and cnt elements of the DenseWork of an s x m and an s x p sketch
void dense_work_size(int64_t m, int64_t p, int s, size_t* part, size_t* cnt);
template <typename TA, typename TL>
cudaError_t launch_dense_pair(const Dims& D, const TA* AW, const TL* lw, const Small& S, const double* SA, const double* SL,
                              const DenseWork& K, cudaStream_t st);
cudaError_t launch_sketch_vec(const int32_t* ptr, const uint32_t* idx, const void* v, int vdt, bool acc_f32, int s,
                              double* out, cudaStream_t st);
cudaError_t launch_dense_sketch(const double* SG, const void* v, int vdt, int64_t len, int s, const DenseWork& K,
                                double* out, cudaStream_t st);
cudaError_t build_sketch_csr(uint64_t key, int64_t h, int s, int zeta, int32_t* ptr, uint32_t* idx, int* err,
                             cudaStream_t st);
cudaError_t launchx_sketch_gather_col(const Dims& D, const float2* AW, const double* lw, const SketchCSR& SK,
                                      const Small& S, cudaStream_t st);
template <typename T, typename V>
cudaError_t launch_gradient(const Dims& D, const DevA<T, V>& A, const DevL& L, const Bulk<T>& B,
                            const Small& S, bool refine, cudaStream_t st);
// Register-blocked convolution and fused refinement kernels (k_conv.cu); *done = false when the
// operator or the sizes are outside their scope (the caller then launches the generic kernel).
template <typename T, typename V>
cudaError_t launch_gradient_append_conv(const Dims& D, const DevA<T, V>& A, const DevL& L, const Bulk<T>& B,
                                        const Small& S, cudaStream_t st, bool* done);
template <typename T, typename V>
cudaError_t launch_apply_column_conv(const Dims& D, const DevA<T, V>& A, const DevL& L, const Bulk<T>& B,
                                     const Small& S, cudaStream_t st, bool* done);
template <typename T, typename V>
cudaError_t launch_gradient_refine2(const Dims& D, const DevA<T, V>& A, const DevL& L, const Bulk<T>& B,
                                    const Small& S, cudaStream_t st, bool* done);
template <typename T>
cudaError_t launch_combine(const Dims& D, const Bulk<T>& B, const Small& S, int mode, cudaStream_t st);
cudaError_t launch_append_solve(const Dims& D, const Small& S, cudaStream_t st);
cudaError_t launch_refine_solve(const Dims& D, const Small& S, cudaStream_t st);
// Sarr (device, ninst entries) selects per-instance state for batched handles; null = S only.
cudaError_t launch_qr_append(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr = nullptr,
                             int ninst = 1);
cudaError_t launch_stacked_solve(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr = nullptr,
                                 int ninst = 1);
cudaError_t launch_refine_solve2(const Dims& D, const Small& S, cudaStream_t st, const Small* Sarr = nullptr,
                                 int ninst = 1, int npart = -1);
cudaError_t configure_small_fast(int* cluster_out, int s, int dm);
cudaError_t launch_reduce_rows(const double* part, int nb, int len, double scale, double* out, cudaStream_t st);
cudaError_t configure_cluster_kernels(int* cluster_out, int s, int dmax);

// fp32x form (k_fp32x.cu)
cudaError_t launchx_sketch_column(const Dims& D, const DevA<float, float>& A, const DevL& L, const BulkX& B,
                                  const Small& S, const SketchCSR& SK, cudaStream_t st);
cudaError_t launchx_combine(const Dims& D, const BulkX& B, const Small& S, int mode, cudaStream_t st);
cudaError_t launchx_gradient(const Dims& D, const DevA<float, float>& A, const DevL& L, const BulkX& B,
                             const Small& S, bool refine, cudaStream_t st);
cudaError_t launchx_to_float(const float2* in, float* out, int64_t n, cudaStream_t st);
cudaError_t launchx_gaussian_sketch(const Dims& D, const DevA<float, float>& A, const DevL& L, const BulkX& B,
                                    const Small& S, const double* SA, const double* SL, const DenseWork& K,
                                    cudaStream_t st);

// setup helpers (sgks_setup.cu)
template <typename T, typename V>
cudaError_t launch_apply(const Dims& D, const DevA<T, V>& A, const DevL& L, int which, const T* in, T* out,
                         cudaStream_t st);
template <typename T>
cudaError_t launch_dots(const T* V0, int64_t n, int k, const T* w, double* part, int nb, cudaStream_t st);
template <typename T>
cudaError_t launch_orth_update(T* w, const T* V0, int64_t n, int k, const double* part, int nb,
                               cudaStream_t st);
template <typename T>
cudaError_t launch_normalize(T* w, int64_t n, const double* part, int nb, cudaStream_t st);
template <typename T>
cudaError_t launch_sqnorm(const T* w, int64_t n, double* part, int nb, cudaStream_t st);

// transpose and sketch rows (sgks_util.cu)
cudaError_t csr_transpose_device(int64_t m, int64_t n, int64_t nnz, const int32_t* rp, const int32_t* ci,
                                 const void* val, int vdt, int32_t* trp, int32_t* tci, void* tval, cudaStream_t st,
                                 int* err = nullptr);
// interleaved 32-row slices of a CSR with `rows` rows (DevA::sl_*): the slice sizes w[g], then,
// with off = their exclusive prefix sums, the row lengths and the interleaved entries
cudaError_t slice_width_device(const int32_t* rp, int64_t rows, int64_t* w, cudaStream_t st);
cudaError_t slice_fill_device(const int32_t* rp, const int32_t* ci, const void* val, int vdt, int64_t rows,
                              const int64_t* off, int32_t* len, int32_t* sci, void* sval, cudaStream_t st);
// ------------------------------------------------------------------- batched form
// B instances of one problem shape (same A and L; their own b_i, lambda_i, x_true_i), all n-,
// m- and p-vectors instance-interleaved: v[q * B + i].  B is a power of two, 1 <= B <= 256.
constexpr int kMaxBatch = 256;

struct BDims {
    int64_t n, m, p;
    int B;
    int s, dmax, ell, max_iters;
    int nb_combine;           // CTAs of the combine kernel
    int tma;                  // 1: combine streams W through shared memory by bulk copies
    int slice_kb;             // bulk-copy combine: column slice of 8 or 16 KB (tuned)
    int nl_a, nl_t;           // CSR rows: lanes per row of A and of A^T (powers of two <= 32, tuned)
    int nb_refine;            // CTAs of kb_wtr (each leaves one partial per instance)
    int nb_setup;             // CTAs of the setup reductions
    bool alone;               // the batch's only group
    int tile_ic;              // tiled forward pass: instances per CTA (0: kTileInst; tuned)
    int wait_tries;           // bounded waits of the bulk-copy combine's ring (kWaitTries; 0 in the
                              // timeout test of SGKS_TEST_TIMEOUT_GROUP, see sgks_batch.cu)
    double sketch_scale;      // 1/sqrt(zeta)
};

template <typename T>
struct BBulk {
    T *W, *AW;                // [dmax][n][B], [dmax][m][B]
    T *x, *xs, *e;            // [n][B] current x, x of the last full iteration, [m][B] A x - b
    T* b;                     // [m][B]
    T* xtrue;                 // [n][B] or nullptr
    T *tp, *tm;               // [p][B] L w of the newest column; [m][B] setup temporary
    T* r;                     // [n][B] gradient r(y) inside the refinement
};

// Batched compensated forms (k_batchx.cu): the basis W in TW (float for the FP32 form, float2
// for the float-float form), every other vector as float-float pairs (hi, lo).
template <typename TW>
struct BBulkX {
    TW* W;                    // [dmax][n][B]
    float2* AW;               // [dmax][m][B]
    float2 *x, *xs;           // [n][B]
    float2* e;                // [m][B] A x - b
    float2* b;                // [m][B]
    float2* xtrue;            // [n][B] or nullptr
    float2* tp;               // [p][B] L w of the newest column
    float2* r;                // [n][B] gradient r(y) inside the refinement
    const float2* lam2;       // [B] lambda_i split into (hi, lo)
    float2* y2;               // [dmax][B] y_i split into (hi, lo) for the combine: y2[j * B + i]
};

struct BSmall {
    double *partA, *partL;    // [B][s] sketched newest column (one partial)
    double* Sb;               // [B][s] S_A b_i
    double* gpart;            // [B][nb_refine][dmax] refinement partials
    double* kapart;           // [nb_combine][B][3] norm partials
    double* y;                // [B][dmax]
    double* lam;              // [B]
    double *rc_hist, *rre_hist;   // [B][max_iters]
    double *setup_part, *setup_coef;   // [nb_setup][ell][B], [ell][B]
    DevScalars* sc;           // [B]
    int* ka_done;             // block counter of kb_combine
};

// Input / output pointers of the B instances (kernel parameter, 2 KB).
struct PtrPack {
    const void* p[kMaxBatch];
};

// Lanes that share a ray of n instance lanes in the sums over segments, within a warp: a ray of a CT image crosses
// some 20 to 60 tiles, and eight lanes leave each one round or two of loads.  512^2, FP64, one vector: 45 -> 20 us;
// a batch of one, float-float, 301^2: 17 -> 11 us.  The lanes set the order of a ray's sum, so they follow from n
// alone: a batch of several groups, which run next to each other and fill the chip without, would be a little faster
// with one lane (7.61 against 7.72 ms per solve of 11 slices of 243^2), but an instance's result would
// then depend on what else is in the batch.
inline int seg_lanes(int n) { return n >= 32 ? 1 : std::min(8, 32 / n); }

template <typename T, typename V>
cudaError_t launchb_apply_column(const BDims& D, const DevA<T, V>& A, const DevL& L, const BBulk<T>& X,
                                 const BSmall& S, cudaStream_t st, bool a_rows = true);
template <typename T>
cudaError_t launchb_sketch_gather(const BDims& D, const BBulk<T>& X, const SketchCSR& SK, const BSmall& S,
                                  const T* vec, double* out_vec, cudaStream_t st);
template <typename T>
cudaError_t launchb_combine(const BDims& D, const BBulk<T>& X, const BSmall& S, int mode, cudaStream_t st);
// out == nullptr: append the gradient as column d_i of W_i; else write it to out ([n][B])
template <typename T, typename V>
cudaError_t launchb_gradient(const BDims& D, const DevA<T, V>& A, const DevL& L, const BBulk<T>& X, const BSmall& S,
                             T* out, cudaStream_t st);
// refinement partials g_i = W_i^T r_i into S.gpart
template <typename T>
cudaError_t launchb_wtr(const BDims& D, const BBulk<T>& X, const BSmall& S, const T* r, cudaStream_t st);
template <typename T, typename V>
cudaError_t launchb_apply(const BDims& D, const DevA<T, V>& A, const DevL& L, int which, const T* in, T* out,
                          cudaStream_t st);
template <typename T>
cudaError_t launchb_dots(const BDims& D, const T* V0, int k, const T* w, const BSmall& S, cudaStream_t st);
template <typename T>
cudaError_t launchb_vec_update(const BDims& D, T* w, const T* V0, int k, const BSmall& S, int mode, cudaStream_t st);
template <typename T>
cudaError_t launchb_gather_in(const PtrPack& P, T* out, int64_t len, int B, cudaStream_t st);
template <typename T>
cudaError_t launchb_scatter_out(const T* in, const PtrPack& P, int64_t len, int B, cudaStream_t st);
// A CSR operator re-blocked by pixel tiles for the batched passes (k_tiles.cu, k_tile_build.cu): the
// image (nt frames of ny x nx) cut into TX x TY tiles.  Entries come in groups of four rows: pair k of
// a group is four (slot, slot, value, value), one per row, at ent[4 (goff[g] + k)].
// Forward: a segment is the run of one row's entries in one tile; the segments of tile t, longest
// first, are the positions [4 tile_grp[t], 4 tile_grp[t+1]) (the last group filled up with empty ones);
// row r's are ray_seg[ray_ptr[r] .. ray_ptr[r+1]), in the order of the row's entries.
struct TiledA {
    int TX, TY, nx, ny, nt, ntx, nty, ntiles;
    int64_t npart;             // segment positions: rows of the partial sums
    int64_t nseg;              // segments, without the filling
    const int32_t* order;      // tiles by descending work, so that the last CTAs are the short ones
    const int32_t* tile_grp;   // [ntiles + 1]
    const int32_t* goff;       // [npart / 4 + 1]
    const int32_t* ray_ptr;    // [m + 1]
    const int32_t* ray_seg;
    const uint4* ent;          // slots: tile_slot of the pixel; TX TY holds 0
};
// Transposed: the rows of A that cross tile t are ray[tile_ray[t] .. tile_ray[t+1]), taken `stage` at a
// time; stage tile_stage[t] + i has a group per four neighbouring pixels of the tile.
struct TiledT {
    int TX, TY, nx, ny, nt, ntx, nty, ntiles;   // ntiles = 0: not built
    const int32_t* order;        // tiles by descending work
    const int32_t* tile_stage;   // [ntiles + 1]
    const int32_t* tile_ray;     // [ntiles + 1]
    const int32_t* ray;
    const int32_t* goff;         // [stages * TX TY / 4 + 1]
    int stage;
    const uint4* ent;            // slots: the row's place in its stage; `stage` holds 0
};
constexpr int kTileInst = 16;    // instances per CTA of the tiled passes
constexpr int kTileAhead = 4;    // entry pairs behind the last group that may be read (and are not used)
// rows of A staged at a time for a largest group of B instances: 64 KB of float-float values, 32 KB for
// less than 8 (fewer stages, hence fewer barriers and less filling, while two CTAs still share an SM)
inline int tile_stage(int B) { return B >= kTileInst ? 512 : (B >= 8 ? 1024 : (B >= 4 ? 1024 : (B >= 2 ? 2048 : 4096))); }
// tiles of the transposed pass: 16 x 8 pixels for groups of 16 instances and more (a thread's
// accumulators then leave registers for the loads: 2.4 -> 2.0 ms, 512^2 at 64), else 16 x 16
constexpr int kTileTX = 16;
inline int tile_ty(int B) { return B >= kTileInst ? 8 : 16; }
// Shared-memory slot of local pixel q (row-major in a tile of width TX, TX even): neighbouring slots
// swap on odd pixel rows.  With fewer than 128 bytes per pixel a load phase serves pixels of
// neighbouring rays, which on rays along x lie one pixel row apart; the swap puts them in different
// parts of a bank line, as pixels one column apart are.
__host__ __device__ inline int tile_slot(int q, int TX) { return q ^ ((q / TX) & 1); }
// The layouts are an option: where device memory is short, or positions would not fit in 32 bits, the builders
// return SGKS_OK with ntiles = 0 and leave nothing in allocs.  They run after everything that a handle cannot do
// without.  tile_memory adds an array to allocs (the partial sums); both it and tile_room free all of allocs and
// return false when memory is short, that is, when less than kTileRoom is left for graphs and modules
// loaded later.
constexpr size_t kTileRoom = (size_t)128 << 20;
bool tile_room(std::vector<void*>& allocs);
bool tile_memory(std::vector<void*>& allocs, void** p, size_t bytes);
void drop_tile_memory(std::vector<void*>& allocs);
int build_tiles(const int32_t* rp, const int32_t* ci, const float* val, int64_t m, int64_t n, int64_t nnz, int nx, int ny,
                int nt, int TX, int TY, TiledA& T, std::vector<void*>& allocs, cudaStream_t st, std::string* why);
int build_tiles_t(const int32_t* trp, const int32_t* tci, const float* tval, int64_t m, int64_t n, int64_t nnz, int nx,
                  int ny, int nt, int TY, int stage, TiledT& T, std::vector<void*>& allocs, cudaStream_t st, std::string* why);
// Vectors of B interleaved instances for the FP64 tiled passes (k_tiles64.cu): p[q B + b], or, with
// scalars, column sc[b].d of p (columns of `col` values).
struct TileVec64 {
    const double* p;
    int64_t col;
    const DevScalars* sc;   // null: a plain vector
    int dmax, B;
    // instance b's vector (element q at [q B]); null when the instance has stopped or its basis is full
    __device__ __forceinline__ const double* column(int b) const {
        if (!sc) return p + b;
        return !sc[b].stop && sc[b].d < dmax ? p + (size_t)sc[b].d * col + b : nullptr;
    }
};
// U = A W through the tiles (part: npart x B doubles); lw (single handle): L w too, else null
cudaError_t launch64_tile_apply(const TiledA& T, const TileVec64& W, const TileVec64& U, int64_t m, bool alone, double* part,
                                const DevL& L, double* lw, cudaStream_t st);
// O = A^T E + lambda L^T L x (x null: A^T E); lambda per instance (lam) or one (lam1).  O without scalars but
// sc given: instances that have stopped are left out.
cudaError_t launch64_tile_gradient(const TiledT& T, const TileVec64& E, const TileVec64& O, DevScalars* sc, const DevL& L,
                                   const double* x, const double* lam, double lam1, cudaStream_t st);
// Both layouts for FP64 vectors where they pay: a CSR operator with finite FP32 values and 2^20 entries or more (1.26
// to 1.47 times the row kernels at 1.3 M entries; smaller ones were not measured) on an image (the regularizer's)
// of enough tiles, whose rows share tiles; else T.ntiles = Tt.ntiles = 0.  B: largest group.
int build_tiles64(const sgks_reg* reg, const int32_t* rp, const int32_t* ci, const float* val, const int32_t* trp,
                  const int32_t* tci, const float* tval, int64_t m, int64_t n, int64_t nnz, int B, TiledA& T, TiledT& Tt,
                  std::vector<void*>& allocs, cudaStream_t st, std::string* why);
int tile_instances(const BDims& D);   // instances per CTA of the forward pass
// u_i = A w_i into column d_i of AW through the tiles (partials in part, npart x B float-float)
template <typename TW>
cudaError_t launchbx_tile_apply(const BDims& D, const TiledA& T, const BBulkX<TW>& X, const BSmall& S, float2* part,
                                cudaStream_t st);
// as launchbx_gradient
template <typename TW>
cudaError_t launchbx_tile_gradient(const BDims& D, const TiledT& T, const DevL& L, const BBulkX<TW>& X, const BSmall& S,
                                   float2* out, cudaStream_t st);

// compensated batched kernels (k_batchx.cu); TW = float or float2
// a_rows = false: no A rows (they come from launchbx_tile_apply); l_rows = false: no t = L w
// column (S_L L w comes from launchbx_sketch_chunks)
template <typename TW>
cudaError_t launchbx_apply_column(const BDims& D, const DevA<float, float>& A, const DevL& L, const BBulkX<TW>& X,
                                  const BSmall& S, cudaStream_t st, bool a_rows = true, bool l_rows = true);
// partial sums part[nA + nL][s][B] of S_A u_i and S_L L w_i for the newest column of every live instance
// (L w is formed on the way, not stored), then their sums into S.partA and S.partL
template <typename TW>
cudaError_t launchbx_sketch_chunks(const BDims& D, const DevL& L, const BBulkX<TW>& X, const SketchChunks& K,
                                   const BSmall& S, float2* part, cudaStream_t st);
cudaError_t launchbx_sketch_reduce(const BDims& D, const SketchChunks& K, const BSmall& S, const float2* part,
                                   cudaStream_t st);
// S_A v_i, scaled, for an m-vector v [m][B], to out [B][s] (at the setup, while S.sc is zero)
template <typename TW>
cudaError_t launchbx_sketch_vec(const BDims& D, const DevL& L, const BBulkX<TW>& X, const SketchChunks& K,
                                const BSmall& S, const float2* vec, float2* part, double* out, cudaStream_t st);
// chunks for a largest group of B instances (device arrays to allocs)
int build_sketch_chunks(const SketchCSR& SK, int64_t m, int64_t p, int s, int B, SketchChunks& K,
                        std::vector<void*>& allocs, cudaStream_t st, std::string* why);
template <typename TW>
cudaError_t launchbx_combine(const BDims& D, const BBulkX<TW>& X, const BSmall& S, int mode, cudaStream_t st);
template <typename TW>
cudaError_t launchbx_gradient(const BDims& D, const DevA<float, float>& A, const DevL& L, const BBulkX<TW>& X,
                              const BSmall& S, float2* out, cudaStream_t st);
template <typename TW>
cudaError_t launchbx_wtr(const BDims& D, const BBulkX<TW>& X, const BSmall& S, const float2* r, cudaStream_t st);
// in: float (in_dt SGKS_F32) or double values per instance -> float-float [len][B]
cudaError_t launchbx_gather_in(const PtrPack& P, int in_dt, float2* out, int64_t len, int B, cudaStream_t st);
// float-float [len][B] -> float (rounded) or double per instance (null pointers skipped)
cudaError_t launchbx_scatter_out(const float2* in, const PtrPack& P, int out_dt, int64_t len, int B, cudaStream_t st);
// out[i] = in[i] rounded to TW (float: nearest float; float2: split)
template <typename TW>
cudaError_t launchbx_from_double(const double* in, TW* out, int64_t len, cudaStream_t st);
// double copy of a float-float vector
cudaError_t launchbx_to_double(const float2* in, double* out, int64_t len, cudaStream_t st);
size_t batchx_combine_smem(size_t welem, int slice_kb);
int batchx_combine_grid(const BDims& D, size_t welem);
cudaError_t launchb_set_xt2(const BSmall& S, int B, cudaStream_t st);
cudaError_t launchb_set_tol(DevScalars* sc, int B, double tol, cudaStream_t st);
size_t batch_refine_smem(int dmax, int B, size_t elem);
size_t batch_combine_tma_smem(size_t elem, int slice_kb);
int batch_combine_tiles(int64_t n, int64_t m, int B, bool tma, size_t elem, int slice_kb);
// CTAs of the combine for a configuration (residency from its shared memory)
int batch_combine_grid(const BDims& D, size_t elem);

// ------------------------------------------------------------------- reverse sweep (k_adjoint.cu)
cudaError_t launchd_record_y(const DevScalars* sc, const double* y, double* yhist, int dmax, int offset, int rows,
                             int sub, int nsub, cudaStream_t st);
template <typename T>
cudaError_t launchd_gemv_n(const T* W, int64_t n, int d, const double* c, T* out, cudaStream_t st);
template <typename T>
cudaError_t launchd_rank2(T* Wb, int64_t n, int d, const T* a, const double* p, const T* q, const double* r,
                          cudaStream_t st);
template <typename T>
cudaError_t launchd_axpby(T* out, const T* x, double alpha, const T* y, double beta, int64_t n, cudaStream_t st);
// x scaled by the power of two that brings its largest element to [1, 2), kept in *bits; and the scale taken off
// another vector and off *acc again
cudaError_t launchd_scale_down(double* x, int64_t n, unsigned long long* bits, cudaStream_t st);
cudaError_t launchd_scale_back(double* x, int64_t n, const unsigned long long* bits, double* acc, cudaStream_t st);
cudaError_t launchd_axpby_d(double* out, const double* x, double alpha, const double* y, double beta, int n,
                            cudaStream_t st);
cudaError_t launchd_dot_acc(const double* a, const double* b, int len, double sign, double* acc, cudaStream_t st);
cudaError_t launchd_acc_parts(const double* part, int nb, double sign, double* acc, cudaStream_t st);
template <typename T>
cudaError_t launchd_sketch_adj(uint64_t key, const double* gauss, int64_t h, int s, int zeta, double scale,
                               const double* u, T* out, int* err, cudaStream_t st);
cudaError_t launchd_solve_G(const double* X, const double* Xr, int dm, int d, const double* v, double* z,
                            cudaStream_t st);
cudaError_t launchd_qr_products(const Small& S, int s, int dm, int d, const double* y, const double* z, double* uy,
                                double* uz, double* vy, double* vz, cudaStream_t st);
cudaError_t launchd_small_inverse(const double* R, int ell, double* Rinv, cudaStream_t st);
template <typename T>
cudaError_t launchd_kbar(const T* Wb0, int64_t n, int ell, const double* Rinv, T* Kbar, cudaStream_t st);

// ------------------------------------------------------------------------ GKS (k_gks.cu)
template <typename T, typename V>
cudaError_t launch_apply_new_column(const Dims& D, const DevA<T, V>& A, const DevL& L, const Bulk<T>& B,
                                    const Small& S, cudaStream_t st);
// One factor that a column is appended to or projected against: column d of Q (h rows), its coefficients.
template <typename T>
struct GJob {
    T* Q;                // [.][h]
    int64_t h;
    const T* src;        // the new column is copied from here first (+ d h when src_col); null: it is in Q
    int src_col;
    const T* b;          // the partials of the updated column's product with b are wanted; or null
    double* part;        // [gks_blocks(h)][dm + 1]: products with the columns before it, squared norm
    double* npart;       // [gks_vec_blocks(h)][2]: squared norm and product with b after an update
    double *c1, *c2;     // [dm + 1] sums of part in the first and the second pass
    double* Rm;          // R, column d is written
    double* out;         // rho, breakdown, finite, d_A entry (layout of S.qr_out)
    double* scale;       // 1 / norm of the new column
};
template <typename T>
struct GJobs {
    GJob<T> j[2];
    int n;
};
int gks_blocks(int64_t h);
int gks_vec_blocks(int64_t h);
// pass 0: copy the new column (src), part; then c1.  pass 1: part, then c2.
template <typename T>
cudaError_t launchg_coef(const GJobs<T>& J, const DevScalars* sc, int dm, int pass, cudaStream_t st);
// column d -= Q[:, :d] c (c1 for pass 0, c2 for pass 1; skipped when flag is given and 0); npart for pass 1
template <typename T>
cudaError_t launchg_update(const GJobs<T>& J, const DevScalars* sc, int dm, int pass, const int* flag, cudaStream_t st);
// column d of R, out and scale from c1, c2 and npart
template <typename T>
cudaError_t launchg_qr_finish(const GJobs<T>& J, const DevScalars* sc, int dm, cudaStream_t st);
template <typename T>
cudaError_t launchg_scale(const GJobs<T>& J, const DevScalars* sc, cudaStream_t st);
// flag = ||c2[:d]|| >= tau sqrt(c2[d]) (eq. loss_criterion; c2[d]: squared norm of the projected column)
cudaError_t launchg_loss(const double* c2, const DevScalars* sc, double tau, int* flag, cudaStream_t st);
// scale = 1 / norm from npart (nb entries); a zero or non-finite norm stops the solve
cudaError_t launchg_inv_norm(const double* npart, int nb, double* scale, DevScalars* sc, cudaStream_t st);

// Host-side preparation shared by the single and the batched handles (sgks_api.cu): the L
// descriptor, the operator in the solver precision (CSR validation, value conversion, device
// transpose) and the sparse-sign sketches by rows.  Device memory goes to `allocs`; the int
// returned is an SGKS_* status with the reason in *why.
void add_launches(int64_t k);
int validate_problem(const sgks_op* A, const sgks_reg* L, const void* b, double lambda, int s, const sgks_options& o,
                     std::string* why);
DevL make_devl(const sgks_reg* reg);
template <typename T, typename V>
int prepare_operator(const sgks_op* op, DevA<T, V>& A, std::vector<void*>& allocs, int* d_err, cudaStream_t st,
                     std::string* why, bool slices = true);
int prepare_sparse_sign(uint64_t keyA, uint64_t keyL, int64_t m, int64_t p, int s, int zeta, SketchCSR& SK,
                        std::vector<void*>& allocs, int* d_err, cudaStream_t st, std::string* why);

// Scratch size of the allocation-free CSR transpose and the bytes a given size needs of it.
constexpr size_t kNoAllocScratchBytes = (size_t)16 << 20;
size_t transpose_noalloc_need(int64_t n, int64_t nnz, int vdt);
// *err receives the device address of the call's malformed-input flag (read it after the stream)
cudaError_t csr_transpose_noalloc_device(int64_t m, int64_t n, int64_t nnz, const int32_t* rp, const int32_t* ci,
                                         const void* val, int vdt, int32_t* trp, int32_t* tci, void* tval,
                                         cudaStream_t st, int** err);
cudaError_t sparse_sign_rows_device(uint64_t key, int64_t h, int s, int zeta, int32_t* rows, uint8_t* neg,
                                    int* err, cudaStream_t st);
cudaError_t convert_values(const void* in, int in_dt, void* out, int out_dt, int64_t count, cudaStream_t st);
cudaError_t launch_srtt_fill(const int8_t* signs, const int32_t* rows, int64_t h, int s, double* out, cudaStream_t st);
cudaError_t launch_set_tol(DevScalars* sc, double tol, cudaStream_t st);
cudaError_t validate_csr_device(const int32_t* rp, const int32_t* ci, int64_t m, int64_t n, int64_t nnz, int* err,
                                cudaStream_t st);

// Host-side count of kernel launches enqueued by the library (graph replays add the number of
// kernel nodes of the step graph).
int64_t launches_total();
void launches_add(int64_t k);

}  // namespace sgks
