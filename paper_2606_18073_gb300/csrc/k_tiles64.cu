// Pixel-tiled passes of a CSR operator with FP32 values, FP64 vectors: u = A w and r = A^T e + lambda L^T L x,
// for a single handle and for batches, on the layouts of k_tile_build.cu (see k_tiles.cu).
//
// Bound: an FP64 warp instruction takes its quarter of the SM for 64 clocks on GB300, 0.63 T FMA/s for the
// chip: 95 us per pass of the 512^2 CT operator (60 M entries), 71 us for its bytes.  The row kernels took 302
// and 285 us there for a single vector (a scattered L2 load per entry), 171 and 413 us for 16 instances of the
// 256^2 tomography problem (floor 60).  Now 147 (127 + 20 for the partials' sums; the FP64 pipe of the first
// kernel is 90 % busy) and 151 us, 119 and 180 us for the 16 instances.  Here the gathered side lies in shared
// memory, entries come in order, and the FP64 pipe does nothing but the multiply-adds:
// - segments of a tile are sorted by length, so that the lanes of a warp run equally long;
// - a conversion from FP32 costs as much as a multiply-add, so a value's bits are only moved into place: as
//   a double they are a 2^-896 exactly (FP32 subnormals included).  Staged values are multiplied by 2^448
//   and sums by 2^448 once each, which leaves products between 2^-574 and 2^576 exact; outside of
//   that the solver's squared norms have under- or overflowed before, and the reverse sweep, which takes no such
//   norms, scales its cotangent and keeps its Krylov vectors on the row kernels (sgks_api.cu).  An operator with infinite or NaN values
//   keeps the row kernels (build_tiles64), and so does one with fewer than 2^20 entries;
// - with several instances a lane takes up to four of them, for one entry load and one set of bit moves.
#include <algorithm>

#include "sgks_internal.cuh"

namespace sgks {

namespace {

constexpr double kHalfScale = 0x1p448;

__device__ __forceinline__ double tiny_bits(uint32_t f) {   // the FP32 value with bits f, times 2^-896
    return __hiloint2double((int)(((f >> 3) & 0x0fffffffu) | (f & 0x80000000u)), (int)(f << 29));
}

// v 2^448 for the shared memory, for a vector that comes from the caller (b at the setup): what would overflow, finite
// values from 2^575 on, stays finite at 2^1023.  The squared norm is infinite in any case, and the solver then
// ends as it does with the row kernels, in a breakdown (infinite elements would make its first column NaN).
// Elsewhere such values end a solve either way; all staged values that way cost 1.6 % of a solve (16 instances, 256^2).
__device__ __forceinline__ double to_stage(double v) {
    const int hi = __double2hiint(v), field = (hi >> 20) & 0x7ff;
    const double r = v * kHalfScale;
    return field >= 1023 + 575 && field != 0x7ff ? __hiloint2double((hi & 0x80000000) | 0x7fe00000, 0) : r;
}

template <int IC>
struct Lanes64 {
    static constexpr int VV = IC >= 4 ? 4 : IC, G = IC / VV, rows = kThreads / G;
};

template <int VV>
__device__ __forceinline__ void load_staged(const double* p, double (&v)[VV]) {
    if constexpr (VV == 1) {
        v[0] = *p;
    } else {
#pragma unroll
        for (int k = 0; k < VV; k += 2) {
            const double2 q = *reinterpret_cast<const double2*>(p + k);
            v[k] = q.x;
            v[k + 1] = q.y;
        }
    }
}

// entry pairs [beg, end) of row `pos` of its group into acc (scaled by 2^-448)
template <int IC>
__device__ __forceinline__ void add_entries64(double (&acc)[Lanes64<IC>::VV], const uint4* __restrict__ ent, int beg, int end,
                                              const double* st) {
    constexpr int VV = Lanes64<IC>::VV;
#pragma unroll 4
    for (int k = beg; k < end; ++k) {
        const uint4 e = __ldg(ent + (size_t)k * 4);
        double a[VV], b[VV];
        load_staged<VV>(st + e.x * IC, a);
        load_staged<VV>(st + e.y * IC, b);
        const double c0 = tiny_bits(e.z), c1 = tiny_bits(e.w);
#pragma unroll
        for (int v = 0; v < VV; ++v) acc[v] = fma(c0, a[v], acc[v]);
#pragma unroll
        for (int v = 0; v < VV; ++v) acc[v] = fma(c1, b[v], acc[v]);
    }
}

}  // namespace

// CTA (tile, IC instances, one of `split` shares of the segments): partials of the segments
template <int IC>
__global__ void __launch_bounds__(kThreads, 4) kd_tile_apply(TiledA T, TileVec64 X, int split, double* __restrict__ part) {
    pdl_wait();
    extern __shared__ __align__(16) double ws[];   // [TX TY + 1][IC]
    using LN = Lanes64<IC>;
    const int B = X.B, nch = B / IC;
    const int bid = (int)blockIdx.x / split, sp = (int)blockIdx.x - bid * split;
    const int t = T.order[bid / nch], row = threadIdx.x / LN::G, b0 = (bid % nch) * IC + (threadIdx.x % LN::G) * LN::VV;
    const double* w[LN::VV];
    bool any = false;
#pragma unroll
    for (int v = 0; v < LN::VV; ++v) {
        w[v] = X.column(b0 + v);
        any = any || w[v];
    }
    if (!__syncthreads_or(any)) return;
    const int tpf = T.ntx * T.nty;
    const int f = t / tpf, rt = t - f * tpf, ty = rt / T.ntx, tx = rt - ty * T.ntx;
    const int npx = T.TX * T.TY, lane0 = (threadIdx.x % LN::G) * LN::VV;
    const int64_t fbase = (int64_t)f * T.nx * T.ny;
    for (int q = row; q <= npx; q += LN::rows) {   // slot npx holds 0
        const int py = q / T.TX, px = q - py * T.TX;
        const int iy = ty * T.TY + py, ix = tx * T.TX + px;
        const bool in = q < npx && iy < T.ny && ix < T.nx;
        const int64_t off = (fbase + (int64_t)iy * T.nx + ix) * B;
        double* dst = ws + (q < npx ? tile_slot(q, T.TX) : npx) * IC + lane0;
#pragma unroll
        for (int v = 0; v < LN::VV; ++v) dst[v] = (in && w[v]) ? __ldcg(w[v] + off) * kHalfScale : 0.0;
    }
    __syncthreads();
    const int s1 = T.tile_grp[t + 1] * 4;
    for (int s = T.tile_grp[t] * 4 + sp * LN::rows + row; s < s1; s += LN::rows * split) {
        const int g = s >> 2;
        double a[LN::VV] = {};
        add_entries64<IC>(a, T.ent + (s & 3), T.goff[g], T.goff[g + 1], ws + lane0);
#pragma unroll
        for (int v = 0; v < LN::VV; ++v) part[(size_t)s * B + b0 + v] = a[v];
    }
}

// u_i = 2^448 sum over the ray's segments; then, where lw is given (single handle), t = L w, a row per
// thread.  Latency: a lane waits for the segment's number, then for its partial, so `lanes` (seg_lanes)
// neighbouring ones share a ray.
__global__ void __launch_bounds__(kThreads) kd_seg_reduce(TiledA T, TileVec64 U, int64_t m, const double* __restrict__ part,
                                                          int lanes, int nbu, DevL L, TileVec64 W, double* lw) {
    pdl_wait();
    if ((int)blockIdx.x >= nbu) {
        const double* w = W.column(0);
        if (!w) return;
        const int64_t step = (int64_t)((int)gridDim.x - nbu) * kThreads;
        for (int64_t j = (int64_t)((int)blockIdx.x - nbu) * kThreads + threadIdx.x; j < L.p; j += step)
            lw[j] = l_row<double>(L, j, w);
        return;
    }
    const int B = U.B, b = threadIdx.x & (B - 1), G = B * lanes;
    double* u = const_cast<double*>(U.column(b));
    if (!__any_sync(0xffffffffu, u != nullptr)) return;
    const int s = (threadIdx.x & (G - 1)) / B;
    const int64_t tot = m * G;
    for (int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x; t - lane_id() < tot; t += (int64_t)nbu * kThreads) {
        const int64_t r = qdiv(t, G);
        const bool in = t < tot && u;
        double a = 0.0;
        const int k1 = in ? T.ray_ptr[r + 1] : 0;
#pragma unroll 4
        for (int k = in ? T.ray_ptr[r] + s : 0; k < k1; k += lanes) a += __ldcs(part + (size_t)T.ray_seg[k] * B + b);
        for (int off = B; off < G; off <<= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (in && s == 0) u[r * B] = a * kHalfScale;
    }
}

// CTA (tile of 16 x TY pixels, IC instances): out = A^T e + lambda L^T L x (x null: A^T e).  O with scalars:
// column d of the basis; a full basis is reported as by the row kernels.
template <int IC, int TY>
__global__ void __launch_bounds__(kThreads, 3) kd_tile_gradient(TiledT T, TileVec64 E, TileVec64 O, DevScalars* sc, DevL L,
                                                                const double* __restrict__ x, const double* lam,
                                                                double lam1) {
    pdl_wait();
    extern __shared__ __align__(16) double es[];   // [stage + 1][IC]
    using LN = Lanes64<IC>;
    constexpr int px = kTileTX * TY, rows = LN::rows < px ? LN::rows : px, PP = px / rows;
    const int B = E.B, nch = B / IC;
    const int t = T.order[blockIdx.x / nch], row = threadIdx.x / LN::G, lane0 = (threadIdx.x % LN::G) * LN::VV;
    const int b0 = (int)(blockIdx.x % nch) * IC + lane0;
    double* out[LN::VV];
    bool any = false;
#pragma unroll
    for (int v = 0; v < LN::VV; ++v) {
        out[v] = const_cast<double*>(O.column(b0 + v));
        if (!out[v] && O.sc && !sc[b0 + v].stop && t == 0 && row == 0) {   // sc[b0 + v].d >= dmax
            sc[b0 + v].status = ST_FULL;
            sc[b0 + v].stop = 1;
        }
        if (sc && !O.sc && sc[b0 + v].stop) out[v] = nullptr;
        any = any || out[v];
    }
    if (!__syncthreads_or(any)) return;
    const bool idle = rows < LN::rows && row >= rows;   // more threads than pixels: they stage only
    double acc[PP][LN::VV] = {};
    const int ray1 = T.tile_ray[t + 1];
    int g = T.tile_stage[t] * (px / 4) + (row >> 2);
    for (int r0 = T.tile_ray[t]; r0 < ray1; r0 += T.stage) {
        const int nr = min(T.stage, ray1 - r0);
        __syncthreads();   // the stage before has been read
#pragma unroll 4
        for (int q = row; q <= nr; q += LN::rows) {
            const double* src = E.p + (size_t)(q < nr ? T.ray[r0 + q] : 0) * B + b0;
            double* dst = es + (q < nr ? q : T.stage) * IC + lane0;   // slot T.stage holds 0
#pragma unroll
            for (int v = 0; v < LN::VV; ++v) {
                const double ev = q < nr ? __ldcg(src + v) : 0.0;
                dst[v] = sc ? ev * kHalfScale : to_stage(ev);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PP; ++u, g += rows / 4)
            if (!idle) add_entries64<IC>(acc[u], T.ent + (row & 3), T.goff[g], T.goff[g + 1], es + lane0);
    }
    if (idle) return;
    const int tpf = T.ntx * T.nty;
    const int f = t / tpf, rt = t - f * tpf, ty = rt / T.ntx, tx = rt - ty * T.ntx;
#pragma unroll
    for (int u = 0; u < PP; ++u) {
        const int loc = u * rows + row;
        const int iy = ty * TY + loc / kTileTX, ix = tx * kTileTX + loc % kTileTX;
        if (iy >= T.ny || ix >= T.nx) continue;
        const int64_t i = ((int64_t)f * T.ny + iy) * T.nx + ix;
#pragma unroll
        for (int v = 0; v < LN::VV; ++v) {
            if (!out[v]) continue;
            const int b = b0 + v;
            double r = acc[u][v] * kHalfScale;
            if (x) r = fma(lam ? lam[b] : lam1, ltl_row_x<double>(L, i, Strided<double>{x + b, B}), r);
            out[v][i * B] = r;
        }
    }
}

// ------------------------------------------------------------------------------ launchers
template <int IC>
static cudaError_t apply64_ic(const TiledA& T, const TileVec64& W, double* part, cudaStream_t st) {
    const size_t smem = (size_t)(T.TX * T.TY + 1) * IC * sizeof(double);
    auto k = kd_tile_apply<IC>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    // shares of a tile's segments until there are four rounds of CTAs, with four segments or more per lane
    const int64_t ctas = (int64_t)T.ntiles * (W.B / IC);
    const int64_t want = std::min<int64_t>(8, (4 * 152 * 4 + ctas - 1) / ctas), most = T.npart / ((int64_t)T.ntiles * Lanes64<IC>::rows * 4);
    const int split = (int)std::max<int64_t>(1, std::min(want, most));
    return launch_pdl(k, (unsigned)(ctas * split), kThreads, smem, st, T, W, split, part);
}

cudaError_t launch64_tile_apply(const TiledA& T, const TileVec64& W, const TileVec64& U, int64_t m, bool alone, double* part,
                                const DevL& L, double* lw, cudaStream_t st) {
    cudaError_t e;
    // Four instances per CTA give every lane a segment of its own, and a warp waits for one staged tile less
    // often; the entries, read once per CTA, stay cheap next to the multiply-adds: 16 instances of 256^2
    // take 147 us with 16 per CTA, 142 with 8, 119 with 4.  Several groups side by side hide those waits
    // themselves and gain from fewer reads (groups of 8, 2 and 1, 243^2: 8.2 against 8.6 ms per solve).
    switch (std::min(W.B, alone ? 4 : kTileInst)) {
        case 1: e = apply64_ic<1>(T, W, part, st); break;
        case 2: e = apply64_ic<2>(T, W, part, st); break;
        case 4: e = apply64_ic<4>(T, W, part, st); break;
        case 8: e = apply64_ic<8>(T, W, part, st); break;
        default: e = apply64_ic<16>(T, W, part, st); break;
    }
    if (e != cudaSuccess) return e;
    const int lanes = seg_lanes(W.B);
    const int nbu = (int)std::max<int64_t>(1, std::min<int64_t>((m * W.B * lanes + kThreads - 1) / kThreads, 8 * 152));
    const int nbl = lw ? (int)std::max<int64_t>(1, std::min<int64_t>((L.p + kThreads - 1) / kThreads, 8 * 152)) : 0;
    return launch_pdl(kd_seg_reduce, nbu + nbl, kThreads, 0, st, T, U, m, part, lanes, nbu, L, W, lw);
}

template <int IC, int TY>
static cudaError_t gradient64_ty(const TiledT& T, const TileVec64& E, const TileVec64& O, DevScalars* sc, const DevL& L,
                                 const double* x, const double* lam, double lam1, cudaStream_t st) {
    const size_t smem = (size_t)(T.stage + 1) * IC * sizeof(double);
    auto k = kd_tile_gradient<IC, TY>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(k, (unsigned)((int64_t)T.ntiles * (E.B / IC)), kThreads, smem, st, T, E, O, sc, L, x, lam, lam1);
}

template <int IC>
static cudaError_t gradient64_ic(const TiledT& T, const TileVec64& E, const TileVec64& O, DevScalars* sc, const DevL& L,
                                 const double* x, const double* lam, double lam1, cudaStream_t st) {
    return T.TY == 8 ? gradient64_ty<IC, 8>(T, E, O, sc, L, x, lam, lam1, st)
                     : gradient64_ty<IC, 16>(T, E, O, sc, L, x, lam, lam1, st);
}

cudaError_t launch64_tile_gradient(const TiledT& T, const TileVec64& E, const TileVec64& O, DevScalars* sc, const DevL& L,
                                   const double* x, const double* lam, double lam1, cudaStream_t st) {
    // at most eight instances per CTA: 16 instances of 256^2 take 189 us with 16 per CTA (512 rays a stage),
    // 180 with 8 (1024 rays), 196 with 4 (2048)
    switch (std::min(E.B, 8)) {
        case 1: return gradient64_ic<1>(T, E, O, sc, L, x, lam, lam1, st);
        case 2: return gradient64_ic<2>(T, E, O, sc, L, x, lam, lam1, st);
        case 4: return gradient64_ic<4>(T, E, O, sc, L, x, lam, lam1, st);
        default: return gradient64_ic<8>(T, E, O, sc, L, x, lam, lam1, st);
    }
}

}  // namespace sgks
