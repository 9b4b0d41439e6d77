// Dense sketches (Gaussian, SRTT): S u and S t as matrix-vector products with FP64 matrices.
//
// The matrices are streamed once per column and every entry costs one FP64 multiply-add, so a
// product is bound by HBM (8 bytes per entry) or by the FP64 pipe (2 lanes per clock and SM),
// whichever is slower: on 400 x 196,096 entries (256^2 deblurring, both sketches) 93 us at 6.8 TB/s
// and 125 us at 0.63 T FMA/s.  A warp per row (100 CTAs, one 8-byte load in flight per lane) left most of
// the chip idle: 1,790 us per column with the operator's own pass, 240 us in the form below.  Here a CTA takes R rows and a chunk of the columns: a thread loads one value
// of the vector and the R matrix entries of its column (R independent loads, R independent sums),
// the warp's R sums are reduced together (9 instead of 40 FP64 adds per lane for R = 8: on GB300 an
// FP64 warp instruction holds the pipe for 16 clocks), and the CTA leaves one partial per row.  The
// last CTA of a row group to arrive adds the group's partials in chunk order, so that the result
// does not depend on the order in which the CTAs ran.
#include <algorithm>

#include "sgks_internal.cuh"

namespace sgks {

namespace {

__device__ __forceinline__ double dense_val(double v) { return v; }
__device__ __forceinline__ double dense_val(float v) { return (double)v; }
__device__ __forceinline__ double dense_val(float2 v) { return (double)v.x + (double)v.y; }

// Rows [g R, g R + R) of SG (s x len) times v over the columns [c C, c C + C); nc chunks a row.
template <int R, typename TV>
__device__ void dense_rows(const double* __restrict__ SG, const TV* __restrict__ v, int64_t len, int s, int64_t C, int nc,
                           int g, int c, double* __restrict__ part, int* __restrict__ cnt, double* __restrict__ out) {
    __shared__ double red[kWarps][R];
    __shared__ bool last;
    const int r0 = g * R;
    const double* row[R];
#pragma unroll
    for (int r = 0; r < R; ++r) row[r] = SG + (size_t)min(r0 + r, s - 1) * len;   // past the end: a row again, not stored
    const int64_t j1 = min(len, (int64_t)(c + 1) * C);
    double a[R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = 0.0;
#pragma unroll 2
    for (int64_t j = (int64_t)c * C + threadIdx.x; j < j1; j += kThreads) {
        const double x = dense_val(v[j]);
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] += __ldcs(row[r] + j) * x;
    }
    const double t = warp_sum_rows<R>(a);
    constexpr int W = 32 / R;
    if (lane_id() % W == 0) red[warp_id()][lane_id() / W] = t;
    __syncthreads();
    const bool mine = threadIdx.x < R && r0 + (int)threadIdx.x < s;
    const double sum = mine ? tree_sumd<kWarps>(&red[0][threadIdx.x], R) : 0.0;
    if (nc == 1) {
        if (mine) out[r0 + threadIdx.x] = sum;
        return;
    }
    if (mine) part[((size_t)g * nc + c) * R + threadIdx.x] = sum;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(cnt + g, 1) == nc - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int r = warp_id(); r < R && r0 + r < s; r += kWarps) {   // a warp per row, lanes over the chunks
        double b = 0.0;
        for (int k = lane_id(); k < nc; k += 32) b += __ldcg(part + ((size_t)g * nc + k) * R + r);
        b = warp_sum(b);
        if (lane_id() == 0) out[r0 + r] = b;
    }
    if (threadIdx.x == 0) cnt[g] = 0;
}

// S_A u and S_L t for the newest column (d read on the device): CTAs [0, gA ncA) take S_A
template <int R, typename TA, typename TL>
__global__ void __launch_bounds__(kThreads) k_dense_pair(Dims D, const TA* __restrict__ AW, const TL* __restrict__ lw,
                                                         Small S, const double* __restrict__ SA,
                                                         const double* __restrict__ SL, DensePlan PA, DensePlan PL,
                                                         DenseWork K) {
    pdl_wait();
    pdl_trigger();   // the QR append loads its earlier columns meanwhile
    if (S.sc->stop) return;
    const int d = S.sc->d;
    if (d >= D.dmax) return;
    const int nA = PA.groups * PA.nc, bid = (int)blockIdx.x;
    if (bid < nA)
        dense_rows<R>(SA, AW + (size_t)d * D.m, D.m, D.s, PA.C, PA.nc, bid / PA.nc, bid % PA.nc, K.part, K.cnt, S.partA);
    else
        dense_rows<R>(SL, lw, D.p, D.s, PL.C, PL.nc, (bid - nA) / PL.nc, (bid - nA) % PL.nc, K.part + (size_t)nA * R,
                      K.cnt + PA.groups, S.partL);
}

// S v for one vector (S_A b at the setup, sgks_apply)
template <int R, typename TV>
__global__ void __launch_bounds__(kThreads) k_dense_vec(const double* __restrict__ SG, const TV* __restrict__ v, int64_t len,
                                                        int s, DensePlan P, DenseWork K, double* __restrict__ out) {
    dense_rows<R>(SG, v, len, s, P.C, P.nc, (int)blockIdx.x / P.nc, (int)blockIdx.x % P.nc, K.part, K.cnt, out);
}

// Rows per CTA: 8 reads the vector once per eight matrix rows; a matrix pair of less than 2^20
// entries (1-D problems: 240 x 256) does not fill the chip that way and takes 2.
int dense_r(int64_t entries) { return entries >= (1 << 20) ? 8 : 2; }

// Chunks so that the launch has about eight CTAs per SM, of at least 1,024 columns (four per
// thread) so that the CTA's reduction stays small against its products.
DensePlan dense_plan(int64_t len, int s, int64_t entries, int R) {
    int64_t C = entries / ((int64_t)152 * 8 * R);
    C = std::max<int64_t>(1024, (C + kThreads - 1) / kThreads * kThreads);
    DensePlan P;
    P.C = C;
    P.nc = (int)((len + C - 1) / C);
    P.groups = (s + R - 1) / R;
    return P;
}

}  // namespace

void dense_work_size(int64_t m, int64_t p, int s, size_t* part, size_t* cnt) {
    *part = *cnt = 0;
    // the pair, and each matrix on its own (a smaller number of entries gives more chunks)
    const int64_t pairs[3] = {s * (m + p), s * m, s * p};
    for (int k = 0; k < 3; ++k) {
        const int R = dense_r(pairs[k]);
        const DensePlan PA = dense_plan(m, s, pairs[k], R), PL = dense_plan(p, s, pairs[k], R);
        const size_t a = k != 2 ? (size_t)PA.groups * PA.nc * R : 0, l = k != 1 ? (size_t)PL.groups * PL.nc * R : 0;
        *part = std::max(*part, a + l);
        *cnt = std::max(*cnt, (size_t)2 * PA.groups);
    }
}

template <typename TA, typename TL>
cudaError_t launch_dense_pair(const Dims& D, const TA* AW, const TL* lw, const Small& S, const double* SA, const double* SL,
                              const DenseWork& K, cudaStream_t st) {
    const int64_t entries = (int64_t)D.s * (D.m + D.p);
    const int R = dense_r(entries);
    const DensePlan PA = dense_plan(D.m, D.s, entries, R), PL = dense_plan(D.p, D.s, entries, R);
    const unsigned grid = (unsigned)(PA.groups * PA.nc + PL.groups * PL.nc);
    if (R == 8) k_dense_pair<8, TA, TL><<<grid, kThreads, 0, st>>>(D, AW, lw, S, SA, SL, PA, PL, K);
    else k_dense_pair<2, TA, TL><<<grid, kThreads, 0, st>>>(D, AW, lw, S, SA, SL, PA, PL, K);
    return cudaGetLastError();
}

template <typename TV>
static cudaError_t dense_vec(const double* SG, const TV* v, int64_t len, int s, const DenseWork& K, double* out,
                             cudaStream_t st) {
    const int R = dense_r(s * len);
    const DensePlan P = dense_plan(len, s, s * len, R);
    const unsigned grid = (unsigned)(P.groups * P.nc);
    if (R == 8) k_dense_vec<8, TV><<<grid, kThreads, 0, st>>>(SG, v, len, s, P, K, out);
    else k_dense_vec<2, TV><<<grid, kThreads, 0, st>>>(SG, v, len, s, P, K, out);
    return cudaGetLastError();
}

cudaError_t launch_dense_sketch(const double* SG, const void* v, int vdt, int64_t len, int s, const DenseWork& K,
                                double* out, cudaStream_t st) {
    return vdt == SGKS_F32 ? dense_vec(SG, (const float*)v, len, s, K, out, st)
                           : dense_vec(SG, (const double*)v, len, s, K, out, st);
}

template cudaError_t launch_dense_pair<double, double>(const Dims&, const double*, const double*, const Small&,
                                                       const double*, const double*, const DenseWork&, cudaStream_t);
template cudaError_t launch_dense_pair<float, float>(const Dims&, const float*, const float*, const Small&, const double*,
                                                     const double*, const DenseWork&, cudaStream_t);
template cudaError_t launch_dense_pair<float2, double>(const Dims&, const float2*, const double*, const Small&,
                                                       const double*, const double*, const DenseWork&, cudaStream_t);

}  // namespace sgks
