// The sparse-sign sketches S_A A w and S_L L w of the newest column, batched compensated forms.
//
// Every value of u = A w and t = L w goes into zeta rows of its sketch.  A CTA per sketch row that
// gathers its entries reads each value zeta = 8 times from L2 in 512-byte pieces (64 instances), and L w
// would have to be stored first.  Here a CTA holds a chunk of C values of u or t for IC instances in
// shared memory, L w formed there from the basis column (the stencil of eq. reg_matrix /
// eq. spacetime_tik, exact in float-float), and adds up every sketch row's entries in the chunk; it leaves
// one partial per (chunk, row, instance), and kbx_sketch_reduce adds those in a fixed order.
//
// Bound: reading the basis column and u once, and the partials: (m + p) / C x s x B x 8 bytes written
// and read, 262 MB on the 512^2 CT batch (m + p = 653,764, s = 600, 64 instances), about 90 us together
// with the two vectors; the additions (5.2 M entries x 64 x 8 operations) take 80 us of the FP32 pipe.
// Measured there 330 + 60 us (before: 607 us for S_L L w with four instances a CTA and 177 us for a CTA per
// row of S_A); one instance of 301^2 pixels 51 -> 26 us.
// Values lie as in the tiled passes (batchx_common.cuh): pairs of instances for the .f32x2 instructions,
// rows of 128 bytes at 16 instances.  Entries (slot, sign in bit 31) come four at a time for groups of
// four sketch rows; the rows of a chunk are sorted by their number of entries, so that the rows of a
// group run equally long; shorter ones are filled with a slot that holds 0.
#include <algorithm>
#include <string>
#include <vector>

#include "batchx_common.cuh"

namespace sgks {

namespace {

// The points and weights of row k of L, decoded once for all instances of a lane.
struct LPoints {
    int64_t q[5];
    float w[5];
    int n;
    __device__ __forceinline__ LPoints(const DevL& L, int64_t k) : n(2) {
        const int nx = L.nx, ny = L.ny;
        int64_t lo = 0, step = 1;
        if (L.kind == SGKS_REG_FD1) {
            lo = k;
        } else if (L.kind == SGKS_REG_LAPLACE2D) {
            const int iy = (int)qdiv(k, nx), ix = (int)(k - (int64_t)iy * nx);
            n = 1;
            q[0] = k;
            w[0] = 4.f;
            if (ix > 0) { q[n] = k - 1; w[n++] = -1.f; }
            if (ix < nx - 1) { q[n] = k + 1; w[n++] = -1.f; }
            if (iy > 0) { q[n] = k - nx; w[n++] = -1.f; }
            if (iy < ny - 1) { q[n] = k + nx; w[n++] = -1.f; }
            return;
        } else {   // differences in x, then in y, then in time
            const int nt = L.kind == SGKS_REG_SPACETIME ? L.nt : 1;
            const int64_t per = (int64_t)ny * (nx - 1), per2 = (int64_t)(ny - 1) * nx, fr = (int64_t)nx * ny;
            if (k < per * nt) {
                const int64_t line = qdiv(k, nx - 1);
                lo = k + line;
            } else if (k < (per + per2) * nt) {
                const int64_t kk = k - per * nt, t = qdiv(kk, per2);
                lo = t * fr + (kk - t * per2);
                step = nx;
            } else {
                lo = k - (per + per2) * nt;
                step = fr;
            }
        }
        q[0] = lo + step;
        w[0] = 1.f;
        q[1] = lo;
        w[1] = -1.f;
    }
};

template <int IC>
constexpr int kSketchThreads = IC >= 16 ? 512 : 256;

}  // namespace

// CTA (chunk, IC instances); chunks [0, nA) of u = column d of AW, then those of t = L w
template <typename TW, int IC>
__global__ void __launch_bounds__(kSketchThreads<IC>, IC >= 16 ? 2 : 4)
    kbx_sketch_chunks(BDims D, DevL L, BBulkX<TW> X, SketchChunks K, BSmall S, float2* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using LN = Lanes<IC>;
    constexpr int rows = kSketchThreads<IC> / LN::G;
    const int B = D.B, nch = B / IC, c = (int)(blockIdx.x / nch), b0 = (int)(blockIdx.x % nch) * IC;
    const bool isA = c < K.nA;
    const int row = threadIdx.x / LN::G;
    const Staged<float2, IC> st(smem_raw, threadIdx.x % LN::G, row);
    const int64_t q0 = (int64_t)(isA ? c : c - K.nA) * K.C;
    const int nq = (int)min((int64_t)K.C, (isA ? D.m : D.p) - q0);
    int d[LN::VV];   // -1: the instance has stopped
    bool any = false;
#pragma unroll
    for (int v = 0; v < LN::VV; ++v) {
        const DevScalars& sc = S.sc[b0 + st.inst(v)];
        d[v] = !sc.stop && sc.d < D.dmax ? sc.d : -1;
        any = any || d[v] >= 0;
    }
    if (!__syncthreads_or(any)) return;
    if (isA) {
#pragma unroll 2
        for (int q = row; q < nq; q += rows) {
            float2 v[LN::VV];
#pragma unroll
            for (int k = 0; k < LN::VV; ++k)
                v[k] = d[k] >= 0 ? __ldcg(X.AW + ((size_t)d[k] * D.m + q0 + q) * B + b0 + st.inst(k)) : ff_zero();
            st.put(smem_raw, q, v);
        }
    } else {
        for (int q = row; q < nq; q += rows) {
            const LPoints P(L, q0 + q);
            Dot2 a[LN::VV];
            for (int i = 0; i < P.n; ++i) {
                TW w[LN::VV];
#pragma unroll
                for (int k = 0; k < LN::VV; ++k)
                    w[k] = d[k] >= 0 ? __ldcg(X.W + ((size_t)d[k] * D.n + P.q[i]) * B + b0 + st.inst(k)) : TW{};
#pragma unroll
                for (int k = 0; k < LN::VV; ++k) acc_add(a[k], P.w[i], w[k]);   // times 1, -1 or 4: exact
            }
            float2 v[LN::VV];
#pragma unroll
            for (int k = 0; k < LN::VV; ++k) v[k] = a[k].value();
            st.put(smem_raw, q, v);
        }
    }
    if (row == 0) {   // slot C holds 0
        const float2 z[LN::VV] = {};
        st.put(smem_raw, K.C, z);
    }
    __syncthreads();
    const int pos = row & 3;
    for (int gi = row >> 2; gi < K.groups; gi += rows / 4) {
        const size_t id = (size_t)c * K.groups + gi;
        const int beg = K.goff[id], end = K.goff[id + 1], r = K.row[id * 4 + pos];
        Dot2x2 a[LN::NP];
        uint4 cur = beg < end ? __ldg(K.ent + (size_t)beg * 4 + pos) : make_uint4(0u, 0u, 0u, 0u);
        for (int kb = beg; kb < end; kb += kDot2Block / 4) {   // blocked Dot2 (ff.cuh)
            const int ke = min(end, kb + kDot2Block / 4);
            Dot2x2 blk[LN::NP];
            for (int k = kb; k < ke; ++k) {
                const uint4 e = cur;
                if (k + 1 < end) cur = __ldg(K.ent + (size_t)(k + 1) * 4 + pos);
                constexpr uint32_t slot = 0x7fffffffu, sign = 0x80000000u;
                if constexpr (LN::VV == 1) {
                    st.add_both_signed(blk[0], e.x & slot, e.y & slot, e.x & sign, e.y & sign);
                    st.add_both_signed(blk[0], e.z & slot, e.w & slot, e.z & sign, e.w & sign);
                } else {
                    st.add_signed(blk, e.x & slot, e.x & sign);
                    st.add_signed(blk, e.y & slot, e.y & sign);
                    st.add_signed(blk, e.z & slot, e.z & sign);
                    st.add_signed(blk, e.w & slot, e.w & sign);
                }
            }
#pragma unroll
            for (int i = 0; i < LN::NP; ++i) a[i].merge(blk[i]);
        }
        if (r < 0) continue;   // filling behind the last row
        float2* dst = part + ((size_t)c * D.s + r) * B + b0;
        if constexpr (LN::VV == 1) {
            dst[0] = both_halves(a[0]).value();
        } else {
#pragma unroll
            for (int i = 0; i < LN::NP; ++i) {
                ulonglong2 o;
                a[i].value(o.x, o.y);
                *reinterpret_cast<ulonglong2*>(dst + st.inst(2 * i)) = o;
            }
        }
    }
}

// CTA r < s: row r of S_A, the others row r - s of S_L: the chunks' partials by kThreads / (B / NB)
// strands per instance (pair), chunk by chunk with Dot2, the strands in FP64 by a fixed pairwise tree.
// vec_out: S_A rows only, scaled, to vec_out[i][r].
template <int NB>
__global__ void __launch_bounds__(kThreads) kbx_sketch_reduce(BDims D, SketchChunks K, BSmall S,
                                                              const float2* __restrict__ part, double* vec_out) {
    pdl_wait();
    pdl_trigger();   // the QR append loads its earlier columns meanwhile
    __shared__ double red[NB][kThreads];
    const int B = D.B, H = B / NB, strands = kThreads / H;
    const int h = threadIdx.x & (H - 1), strand = threadIdx.x / H;
    const bool isA = (int)blockIdx.x < D.s;
    const int r = isA ? (int)blockIdx.x : (int)blockIdx.x - D.s;
    const int c1 = isA ? K.nA : K.nA + K.nL;
    const float2* p = part + (size_t)r * B + h * NB;
    const size_t stride = (size_t)D.s * B;
    if constexpr (NB == 2) {
        Dot2x2 a;
        int n = 0;
#pragma unroll 4
        for (int c = (isA ? 0 : K.nA) + strand; c < c1; c += strands) {
            const float4 f = __ldcs(reinterpret_cast<const float4*>(p + c * stride));
            a.accumulate(pack2(f.x, f.y), pack2(f.z, f.w));
            if (++n % 4 == 0) a.renorm();
        }
        red[0][threadIdx.x] = a.half(0).to_double();
        red[NB - 1][threadIdx.x] = a.half(1).to_double();
    } else {
        Dot2 a;
        int n = 0;
#pragma unroll 4
        for (int c = (isA ? 0 : K.nA) + strand; c < c1; c += strands) {
            const float2 f = __ldcs(p + c * stride);
            a.add2(f.x, f.y);
            if (++n % 4 == 0) a.renorm();
        }
        red[0][threadIdx.x] = a.to_double();
    }
    __syncthreads();
    for (int w = strands / 2; w > 0; w >>= 1) {
        if (strand < w)
#pragma unroll
            for (int v = 0; v < NB; ++v) red[v][threadIdx.x] += red[v][threadIdx.x + w * H];
        __syncthreads();
    }
    if (strand) return;
#pragma unroll
    for (int v = 0; v < NB; ++v) {
        const int b = h * NB + v;
        const DevScalars& sc = S.sc[b];
        if (sc.stop || sc.d >= D.dmax) continue;
        if (vec_out) vec_out[(size_t)b * D.s + r] = D.sketch_scale * red[v][h];
        else (isA ? S.partA : S.partL)[(size_t)b * D.s + r] = red[v][h];
    }
}

// ------------------------------------------------------------------------------ launchers
// a_only: the chunks of u alone
template <typename TW, int IC>
static cudaError_t sketch_chunks_ic(const BDims& D, const DevL& L, const BBulkX<TW>& X, const SketchChunks& K,
                                    const BSmall& S, float2* part, bool a_only, cudaStream_t st) {
    const size_t smem = (size_t)(K.C + 1) * IC * sizeof(float2);
    auto k = kbx_sketch_chunks<TW, IC>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    const int64_t chunks = a_only ? K.nA : K.nA + K.nL;
    k<<<(unsigned)(chunks * (D.B / IC)), kSketchThreads<IC>, smem, st>>>(D, L, X, K, S, part);
    return cudaGetLastError();
}

template <typename TW>
static cudaError_t sketch_chunks(const BDims& D, const DevL& L, const BBulkX<TW>& X, const SketchChunks& K,
                                 const BSmall& S, float2* part, bool a_only, cudaStream_t st) {
    switch (std::min(D.B, kTileInst)) {
        case 1: return sketch_chunks_ic<TW, 1>(D, L, X, K, S, part, a_only, st);
        case 2: return sketch_chunks_ic<TW, 2>(D, L, X, K, S, part, a_only, st);
        case 4: return sketch_chunks_ic<TW, 4>(D, L, X, K, S, part, a_only, st);
        case 8: return sketch_chunks_ic<TW, 8>(D, L, X, K, S, part, a_only, st);
        default: return sketch_chunks_ic<TW, 16>(D, L, X, K, S, part, a_only, st);
    }
}

static cudaError_t sketch_reduce(const BDims& D, const SketchChunks& K, const BSmall& S, const float2* part,
                                 double* vec_out, cudaStream_t st) {
    const int grid = vec_out ? D.s : 2 * D.s;
    if (D.B == 1) kbx_sketch_reduce<1><<<grid, kThreads, 0, st>>>(D, K, S, part, vec_out);
    else kbx_sketch_reduce<2><<<grid, kThreads, 0, st>>>(D, K, S, part, vec_out);
    return cudaGetLastError();
}

template <typename TW>
cudaError_t launchbx_sketch_chunks(const BDims& D, const DevL& L, const BBulkX<TW>& X, const SketchChunks& K,
                                   const BSmall& S, float2* part, cudaStream_t st) {
    return sketch_chunks<TW>(D, L, X, K, S, part, false, st);
}

cudaError_t launchbx_sketch_reduce(const BDims& D, const SketchChunks& K, const BSmall& S, const float2* part,
                                   cudaStream_t st) {
    return sketch_reduce(D, K, S, part, nullptr, st);
}

template <typename TW>
cudaError_t launchbx_sketch_vec(const BDims& D, const DevL& L, const BBulkX<TW>& X, const SketchChunks& K,
                                const BSmall& S, const float2* vec, float2* part, double* out, cudaStream_t st) {
    BBulkX<TW> Xv = X;
    Xv.AW = const_cast<float2*>(vec);   // "column 0 of A W": S.sc is zero when this is called
    const cudaError_t e = sketch_chunks<TW>(D, L, Xv, K, S, part, true, st);
    return e == cudaSuccess ? sketch_reduce(D, K, S, part, out, st) : e;
}

#define SGKS_INST_SKX(TW)                                                                                             \
    template cudaError_t launchbx_sketch_chunks<TW>(const BDims&, const DevL&, const BBulkX<TW>&, const SketchChunks&, \
                                                    const BSmall&, float2*, cudaStream_t);                            \
    template cudaError_t launchbx_sketch_vec<TW>(const BDims&, const DevL&, const BBulkX<TW>&, const SketchChunks&,    \
                                                 const BSmall&, const float2*, float2*, double*, cudaStream_t);
SGKS_INST_SKX(float)
SGKS_INST_SKX(float2)

// ---------------------------------------------------------------------------- chunk layout
// Largest chunk: 96 KB at 16 instances (two CTAs per SM), 64 KB at 8, then 32 KB and less.  A longer chunk
// leaves fewer partials, a shorter one more CTAs: chunks are cut down to two CTAs per SM where the vectors
// are short, but not below 256 columns.
static int chunk_columns(int64_t mp, int B) {
    const int64_t most = B >= 16 ? 768 : 1024, ctas = 2 * 152;
    const int64_t fit = (mp * std::max(1, B / kTileInst) + ctas - 1) / ctas;
    return (int)std::min(most, std::max<int64_t>(256, (fit + 63) / 64 * 64));
}

int build_sketch_chunks(const SketchCSR& SK, int64_t m, int64_t p, int s, int B, SketchChunks& K,
                        std::vector<void*>& allocs, cudaStream_t st, std::string* why) {
    const int C = chunk_columns(m + p, B), groups = (s + 3) / 4;
    const int nA = (int)((m + C - 1) / C), nL = (int)((p + C - 1) / C);
    std::vector<int32_t> ptr((size_t)s + 1), goff((size_t)(nA + nL) * groups + 1, 0), row((size_t)(nA + nL) * groups * 4, -1);
    std::vector<uint32_t> idx, ent;
    auto cuda = [&](cudaError_t e) {
        if (e == cudaSuccess) return false;
        *why = std::string("sketch chunks: ") + cudaGetErrorString(e);
        return true;
    };
    size_t quads = 0;   // of all groups so far
    for (int which = 0; which < 2; ++which) {
        const int32_t* dptr = which ? SK.ptrL : SK.ptrA;
        const uint32_t* didx = which ? SK.idxL : SK.idxA;
        const int64_t h = which ? p : m;
        const int nch = which ? nL : nA, c0 = which ? nA : 0;
        if (cuda(cudaMemcpyAsync(ptr.data(), dptr, sizeof(int32_t) * (s + 1), cudaMemcpyDeviceToHost, st)) ||
            cuda(cudaStreamSynchronize(st)))
            return SGKS_ERR_CUDA;
        idx.resize((size_t)ptr[s]);
        if (ptr[s] && (cuda(cudaMemcpyAsync(idx.data(), didx, sizeof(uint32_t) * ptr[s], cudaMemcpyDeviceToHost, st)) ||
                       cuda(cudaStreamSynchronize(st))))
            return SGKS_ERR_CUDA;
        // a row lists its columns in ascending order, so its entries of a chunk are a run
        std::vector<int32_t> at(ptr.begin(), ptr.end() - 1), cnt((size_t)s), order((size_t)s);
        for (int c = 0; c < nch; ++c) {
            const uint32_t lim = (uint32_t)std::min<int64_t>(h, (int64_t)(c + 1) * C), base = (uint32_t)((int64_t)c * C);
            int most = 0;
            for (int r = 0; r < s; ++r) {
                int32_t k = at[r];
                while (k < ptr[r + 1] && (idx[k] & 0x7fffffffu) < lim) ++k;
                cnt[r] = k - at[r];
                most = std::max(most, cnt[r]);
            }
            // rows by descending count (stable)
            std::vector<int32_t> first((size_t)most + 2, 0);
            for (int r = 0; r < s; ++r) ++first[most - cnt[r] + 1];
            for (int i = 1; i <= most + 1; ++i) first[i] += first[i - 1];
            for (int r = 0; r < s; ++r) order[first[most - cnt[r]]++] = r;
            for (int g = 0; g < groups; ++g) {
                const size_t id = (size_t)(c0 + c) * groups + g;
                const int len = (cnt[order[4 * g]] + 3) / 4;
                goff[id] = (int32_t)quads;
                ent.resize((quads + len) * 16, (uint32_t)C);
                for (int i = 0; i < 4 && 4 * g + i < s; ++i) {
                    const int r = order[4 * g + i];
                    row[id * 4 + i] = r;
                    for (int k = 0; k < cnt[r]; ++k) {
                        const uint32_t u = idx[at[r] + k];
                        ent[((quads + k / 4) * 4 + i) * 4 + k % 4] = ((u & 0x7fffffffu) - base) | (u & 0x80000000u);
                    }
                    at[r] += cnt[r];
                }
                quads += len;
                if (quads >= ((size_t)1 << 29)) {
                    *why = "sketch chunks: too many entries";
                    return SGKS_ERR_INVALID;
                }
            }
        }
        for (int r = 0; r < s; ++r)
            if (at[r] != ptr[r + 1]) {
                *why = "sketch chunks: a column index outside the operator's rows";
                return SGKS_ERR_STATE;
            }
    }
    goff.back() = (int32_t)quads;
    cudaError_t e = cudaSuccess;
    auto up = [&](const void* host, size_t bytes) -> void* {
        void* q = nullptr;
        if (e == cudaSuccess) e = cudaMalloc(&q, bytes + 16);
        if (e != cudaSuccess) return nullptr;
        allocs.push_back(q);
        e = cudaMemcpyAsync(q, host, bytes, cudaMemcpyHostToDevice, st);
        return q;
    };
    K.C = C;
    K.nA = nA;
    K.nL = nL;
    K.groups = groups;
    K.goff = (const int32_t*)up(goff.data(), sizeof(int32_t) * goff.size());
    K.row = (const int32_t*)up(row.data(), sizeof(int32_t) * row.size());
    K.ent = (const uint4*)up(ent.data(), sizeof(uint32_t) * ent.size());
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // the host vectors die on return
    if (e != cudaSuccess) {
        cuda(e);
        return e == cudaErrorMemoryAllocation ? SGKS_ERR_NOMEM : SGKS_ERR_CUDA;
    }
    return SGKS_OK;
}

}  // namespace sgks
