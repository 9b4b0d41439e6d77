// GKS (Algorithm 1) on the GPU: the building blocks that sGKS does not need.
//
// GKS keeps an orthonormal basis V_k.  The new gradient column is orthogonalised against V_k,
// and once more when the loss ratio ||V^T v|| / ||v|| of eq. loss_criterion is at least tau.  It
// keeps full-size thin QR factors A V_k = Q_A R_A and L V_k = Q_L R_L, updated by one column
// per iteration (eq. updqr with S = I), and solves the projected problem of eq.
// projected_withQR.  Those updates are the tall-and-skinny products Q^T u and u - Q c over
// the m-, p- and n-row factors, done here with FP64 reductions in a fixed order; one launch serves
// both factors.  The small
// stacked solve is the one sGKS uses (k_small2.cu); it is fed with the R columns, the flags and
// the d_A entry written here.  Every kernel takes the subspace size d from the device scalars
// (u is column d of its factor) and does nothing once the solve has stopped, so one captured
// graph serves every iteration, as for sGKS.
//
// Cost on GB300 (201 x 157 deblurring, d around 20): the products take 3 us of FP64 per pass, the rest is
// launches and latency.  So the column is copied, its norm taken and its products formed in one kernel, norms
// and the d_A entry ride on the updates, sums over CTAs run on a warp per column, and a tile is 256 rows
// (16 to 31 CTAs of 2,048 rows and a serial sum over CTAs took 197 us per append of both factors).
#include <math.h>

#include "sgks_internal.cuh"

namespace sgks {

constexpr int kGTile = 256;     // rows of the new column staged per CTA step of kg_dots
constexpr int kGMaxD = 1024;    // largest subspace

// blockIdx.x is split over the jobs: nb(h) CTAs each
template <typename T, typename NB>
__device__ __forceinline__ const GJob<T>& my_job(const GJobs<T>& J, NB nb, int* b, int* n) {
    const int n0 = nb(J.j[0].h);
    const int k = (int)blockIdx.x < n0 ? 0 : 1;
    *b = (int)blockIdx.x - (k ? n0 : 0);
    *n = k ? nb(J.j[1].h) : n0;
    return J.j[k];
}

__host__ __device__ inline int ggrid(int64_t h) {
    const int64_t b = (h + kGTile - 1) / kGTile;
    return (int)(b > 4 * 152 ? 4 * 152 : (b < 1 ? 1 : b));
}

__host__ __device__ inline int vgrid(int64_t h) {
    const int64_t b = (h + kThreads - 1) / kThreads;
    return (int)(b > 4 * 152 ? 4 * 152 : (b < 1 ? 1 : b));
}

// part[b][j] = sum over the rows of CTA b of Q[j h + i] u[i], j < d; part[b][d] that of u[i]^2; u = column
// d, copied from src first when that is given.
template <typename T>
__global__ void __launch_bounds__(kThreads) kg_dots(GJobs<T> J, const DevScalars* sc, int dm, int pass) {
    extern __shared__ double acc[];   // [dm + 1]
    __shared__ T us[kGTile];
    __shared__ double red[kWarps];
    if (sc->stop) return;
    int b, nb;
    const GJob<T>& G = my_job(J, ggrid, &b, &nb);
    const int d = sc->d;
    const int64_t h = G.h;
    T* u = G.Q + (size_t)d * h;
    const T* src = pass == 0 && G.src ? G.src + (G.src_col ? (size_t)d * h : 0) : nullptr;
    for (int j = threadIdx.x; j < d; j += kThreads) acc[j] = 0.0;
    double nn = 0.0;
    for (int64_t i0 = (int64_t)b * kGTile; i0 < h; i0 += (int64_t)nb * kGTile) {
        const int rows = (int)min((int64_t)kGTile, h - i0);
        __syncthreads();
        for (int q = threadIdx.x; q < rows; q += kThreads) {
            const T v = src ? src[i0 + q] : u[i0 + q];
            if (src) u[i0 + q] = v;
            us[q] = v;
            nn += (double)v * (double)v;
        }
        __syncthreads();
        tile_dots<T>(G.Q + i0, (size_t)h, us, rows, d, acc);
    }
    nn = warp_sum(nn);
    if (lane_id() == 0) red[warp_id()] = nn;
    __syncthreads();
    double* o = G.part + (size_t)b * (dm + 1);
    for (int j = threadIdx.x; j < d; j += kThreads) o[j] = acc[j];
    if (threadIdx.x == 0) o[d] = tree_sumd<kWarps>(red);
}

// c[j] = sum_b part[b][j], j <= d: a warp per column, lanes over the CTAs' partials; blockIdx.y: job
template <typename T>
__global__ void __launch_bounds__(kThreads) kg_reduce(GJobs<T> J, const DevScalars* sc, int dm, int pass) {
    if (sc->stop) return;
    const GJob<T>& G = J.j[blockIdx.y];
    const int j = (int)blockIdx.x * kWarps + warp_id();
    if (j > sc->d) return;
    const double v = warp_sum_parts(G.part + j, ggrid(G.h), dm + 1);
    if (lane_id() == 0) (pass ? G.c2 : G.c1)[j] = v;
}

// u -= Q[:, :d] c with u = column d of Q (left as it is when flag is given and *flag == 0); LAST: the
// partials of u.u and u.b afterwards
template <typename T, bool LAST>
__global__ void __launch_bounds__(kThreads) kg_update(GJobs<T> J, const DevScalars* sc, const int* flag) {
    __shared__ T cs[kGMaxD];
    __shared__ double red[2][kWarps];
    if (sc->stop) return;
    const bool on = !flag || *flag != 0;
    if (!LAST && !on) return;
    int b, nb;
    const GJob<T>& G = my_job(J, vgrid, &b, &nb);
    const int d = on ? sc->d : 0;
    const int64_t h = G.h;
    const T* Q = G.Q;
    T* u = G.Q + (size_t)sc->d * h;
    const double* c = LAST ? G.c2 : G.c1;
    for (int j = threadIdx.x; j < d; j += kThreads) cs[j] = (T)c[j];
    __syncthreads();
    double nn = 0.0, ub = 0.0;
    for (int64_t i = (int64_t)b * kThreads + threadIdx.x; i < h; i += (int64_t)nb * kThreads) {
        T a = T(0);
#pragma unroll 8
        for (int j = 0; j < d; ++j) a += Q[(size_t)j * h + i] * cs[j];
        const T v = u[i] - a;
        u[i] = v;
        if (LAST) {
            nn += (double)v * (double)v;
            if (G.b) ub += (double)v * (double)G.b[i];
        }
    }
    if (!LAST) return;
    double s[2] = {nn, ub};
    const double v = warp_sum_rows<2>(s);
    if ((lane_id() & 15) == 0) red[lane_id() >> 4][warp_id()] = v;
    __syncthreads();
    if (threadIdx.x < 2) G.npart[(size_t)b * 2 + threadIdx.x] = tree_sumd<kWarps>(red[threadIdx.x]);
}

// Loss ratio of eq. loss_criterion after the first projection: flag = ||c2|| >= tau sqrt(nv2), nv2 = c2[d]
__global__ void kg_loss(const double* __restrict__ c2, const DevScalars* sc, double tau, int* flag) {
    if (sc->stop) return;
    const int d = sc->d;
    double s = 0.0;
    for (int j = lane_id(); j < d; j += 32) s += c2[j] * c2[j];
    s = warp_sum(s);
    if (lane_id() == 0) *flag = sqrt(s) >= tau * sqrt(c2[d]) ? 1 : 0;
}

// the new basis vector is normalised: scale = 1 / sqrt(sum of npart's norms); a zero or non-finite
// norm stops the solve (breakdown / non-finite)
__global__ void kg_inv_norm(const double* __restrict__ npart, int nb, double* scale, DevScalars* sc) {
    if (sc->stop) return;
    const double v = warp_sum_parts(npart, nb, 2);
    if (lane_id() != 0) return;
    if (!(v > 0.0) || !isfinite(v)) {
        *scale = 0.0;
        sc->status = v == 0.0 ? ST_BREAKDOWN : ST_NONFINITE;
        sc->stop = 1;
        return;
    }
    *scale = 1.0 / sqrt(v);
}

// column d of Q *= *scale
template <typename T>
__global__ void kg_scale(GJobs<T> J, const DevScalars* sc) {
    if (sc->stop) return;
    int b, nb;
    const GJob<T>& G = my_job(J, vgrid, &b, &nb);
    T* u = G.Q + (size_t)sc->d * G.h;
    const T s = (T)*G.scale;
    for (int64_t i = (int64_t)b * blockDim.x + threadIdx.x; i < G.h; i += (int64_t)nb * blockDim.x) u[i] *= s;
}

// End of a column append to a thin QR factor (a CTA per job): R[:, d] = [c1 + c2; rho] with rho = ||u||
// after the two projections; breakdown when rho <= 1e-13 ||u before||; out = {rho, broke, finite, d_A
// entry} (the layout the stacked solve reads) and scale = 1 / rho for the new column of Q.
template <typename T>
__global__ void __launch_bounds__(kThreads) kg_qr_finish(GJobs<T> J, const DevScalars* sc, int dm) {
    __shared__ double sums[2];
    if (sc->stop) return;
    const GJob<T>& G = J.j[blockIdx.x];
    const int d = sc->d;
    if (warp_id() < 2) {   // u.u and u.b
        const double v = warp_sum_parts(G.npart + warp_id(), vgrid(G.h), 2);
        if (lane_id() == 0) sums[warp_id()] = v;
    }
    double* R = G.Rm + (size_t)d * dm;
    for (int j = threadIdx.x; j < d; j += kThreads) R[j] = G.c1[j] + G.c2[j];
    __syncthreads();
    if (threadIdx.x) return;
    const double un2 = G.c1[d], r2 = sums[0];
    double rho = sqrt(r2);
    const bool fin = isfinite(un2) && isfinite(r2);
    const bool brk = !(rho > 1e-13 * sqrt(un2));
    if (brk) rho = 0.0;
    const double inv = rho > 0.0 ? 1.0 / rho : 0.0;
    R[d] = rho;
    G.out[0] = rho;
    G.out[1] = brk ? 1.0 : 0.0;
    G.out[2] = fin ? 1.0 : 0.0;
    if (G.b) G.out[3] = sums[1] * inv;
    *G.scale = inv;
}

// ------------------------------------------------------------------------------ launchers
int gks_blocks(int64_t h) { return ggrid(h); }
int gks_vec_blocks(int64_t h) { return vgrid(h); }

template <typename T, typename NB>
static int grid_of(const GJobs<T>& J, NB nb) {
    return nb(J.j[0].h) + (J.n > 1 ? nb(J.j[1].h) : 0);
}

template <typename T>
cudaError_t launchg_coef(const GJobs<T>& J, const DevScalars* sc, int dm, int pass, cudaStream_t st) {
    kg_dots<T><<<grid_of(J, ggrid), kThreads, sizeof(double) * (size_t)(dm + 1), st>>>(J, sc, dm, pass);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    kg_reduce<T><<<dim3((dm + 1 + kWarps - 1) / kWarps, J.n), kThreads, 0, st>>>(J, sc, dm, pass);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launchg_update(const GJobs<T>& J, const DevScalars* sc, int dm, int pass, const int* flag, cudaStream_t st) {
    if (dm > kGMaxD) return cudaErrorInvalidValue;
    if (pass) kg_update<T, true><<<grid_of(J, vgrid), kThreads, 0, st>>>(J, sc, flag);
    else kg_update<T, false><<<grid_of(J, vgrid), kThreads, 0, st>>>(J, sc, flag);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launchg_qr_finish(const GJobs<T>& J, const DevScalars* sc, int dm, cudaStream_t st) {
    kg_qr_finish<T><<<J.n, kThreads, 0, st>>>(J, sc, dm);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launchg_scale(const GJobs<T>& J, const DevScalars* sc, cudaStream_t st) {
    kg_scale<T><<<grid_of(J, vgrid), kThreads, 0, st>>>(J, sc);
    return cudaGetLastError();
}

cudaError_t launchg_loss(const double* c2, const DevScalars* sc, double tau, int* flag, cudaStream_t st) {
    kg_loss<<<1, 32, 0, st>>>(c2, sc, tau, flag);
    return cudaGetLastError();
}

cudaError_t launchg_inv_norm(const double* npart, int nb, double* scale, DevScalars* sc, cudaStream_t st) {
    kg_inv_norm<<<1, 32, 0, st>>>(npart, nb, scale, sc);
    return cudaGetLastError();
}

#define SGKS_INST_G(T)                                                                                          \
    template cudaError_t launchg_coef<T>(const GJobs<T>&, const DevScalars*, int, int, cudaStream_t);             \
    template cudaError_t launchg_update<T>(const GJobs<T>&, const DevScalars*, int, int, const int*, cudaStream_t); \
    template cudaError_t launchg_qr_finish<T>(const GJobs<T>&, const DevScalars*, int, cudaStream_t);             \
    template cudaError_t launchg_scale<T>(const GJobs<T>&, const DevScalars*, cudaStream_t);
SGKS_INST_G(float)
SGKS_INST_G(double)

}  // namespace sgks
