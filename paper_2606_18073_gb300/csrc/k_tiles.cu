// Pixel-tiled passes of a CSR operator on an image geometry, batched compensated forms: u = A w and
// r = A^T e + lambda L^T L x.
//
// A ray operator (CT, travel-time tomography) has rows that are long lines through the image, so a
// CSR pass gathers one whole instance vector per nonzero: 512 bytes each for 64 float-float
// instances, 30 GB per pass on the 512^2 CT operator.  Here the image is cut into pixel tiles and a
// CTA keeps the gathered side in shared memory:
//   forward    a tile of w (IC instances); the CTA walks the (ray, tile) segments that cross the tile
//              and leaves one float-float partial per segment and instance, which kbx_seg_reduce adds
//              up ray by ray;
//   transposed the rays that cross a tile are staged in shared memory a few hundred at a time (rays of a
//              tile in ascending order) and every pixel of the tile adds its entries of the stage to
//              accumulators that stay in registers; the stencil and lambda finish the row, so the
//              gradient is written once and e is read once per crossing (ray, tile) pair.
//
// What bounds both is the FP32 pipe: 11 operations per entry and instance of Dot2 (ff.cuh) are
// 42.3 G on the CT batch (60 M entries, 64 instances), 1.05 ms at 40.3 T/s; Dot2 alone, on registers,
// reaches 33 T/s.  Measured there (float-float): A w 2.82 -> 1.93 ms with kbx_seg_reduce's 0.25, A^T e
// 3.07 -> 2.18 ms against the row kernel's 512-byte gathers.  A batch of one on a 301^2 image: 105 -> 62
// and 92 -> 43 us.  Therefore
// - a lane works on two instances at once with the .f32x2 instructions, 11 per entry, which leaves half
//   of the issue slots for the loads and addresses; with 16 instances it takes two such pairs, so that
//   an entry's load (which the lanes of a row repeat) serves twice as many products;
// - staged values lie as pairs (hi0, hi1, lo0, lo1), so that one 16-byte load gives two operands;
// - 16 instances per CTA make a staged float-float row 128 bytes, all banks once: the eight lanes of a
//   load phase read half of one row and the other half of another, without bank conflicts;
// - entries are stored for groups of four rows (segments, or pixels), interleaved: entries k and
//   k + 1 of a row side by side (slot, slot, value, value), the four rows next to each other, so a
//   warp's entry load is one contiguous line.  Segments of a tile are sorted by length, so that the
//   four of a group run equally long; shorter rows are filled with entries of value 0 on a slot
//   that holds 0.
// A batch of one takes the two entries of a pair in the two halves instead of two instances.
// The layouts are built on the device, once per operator (k_tile_build.cu).
#include <algorithm>

#include "batchx_common.cuh"

namespace sgks {

namespace {

// A row's entry pairs are read as one stream with those of the rows that the lane takes after it: two
// pairs (four entries) at a time, the next two on their way while the present ones are added, also
// from one row to the next.  The loads run two pairs past a row's last ones at most, into the next group
// or into the filling behind the last one (kTileAhead).
struct Entries {
    uint4 a, b;
    __device__ __forceinline__ void load(const uint4* __restrict__ ent, int pair) {
        const uint4* q = ent + (size_t)pair * 4;
        a = __ldg(q);
        b = __ldg(q + 4);
    }
};

// The next row's entries (pairs [beg, end) of its group) into L2, a line per lane: the first CTA that
// comes to a tile would otherwise wait for HBM at every row (2.04 -> 2.01 ms per pass, 512^2 at 64).
__device__ __forceinline__ void entries_to_l2(const uint4* ent, int beg, int end, int k) {
    if (beg + 2 * k < end) asm volatile("prefetch.global.L2 [%0];" ::"l"(ent + (size_t)(beg + 2 * k) * 4));
}

template <typename TW, int IC>
__device__ __forceinline__ void add_pair(Dot2x2 (&d)[Lanes<IC>::NP], const Staged<TW, IC>& st, const uint4& e) {
    if constexpr (Lanes<IC>::VV == 1) {
        st.add_both(d[0], e.x, e.y, __uint_as_float(e.z), __uint_as_float(e.w));
    } else {
        st.add(d, e.x, __uint_as_float(e.z));
        st.add(d, e.y, __uint_as_float(e.w));
    }
}

// Pairs [beg, end) of a row into acc, in blocks of kDot2Block terms (ff.cuh); cur holds the pairs beg
// and beg + 1 and leaves with those of the next row, from `next` on.
template <typename TW, int IC>
__device__ __forceinline__ void add_row(Dot2x2 (&acc)[Lanes<IC>::NP], const Staged<TW, IC>& st, Entries& cur,
                                        const uint4* __restrict__ ent, int beg, int end, int next) {
    constexpr int NP = Lanes<IC>::NP, PB = kDot2Block / 2;
    static_assert(PB % 4 == 0, "blocks of whole double steps");
    if (beg == end) {
        cur.load(ent, next);
        return;
    }
    for (int kb = beg; kb < end; kb += PB) {
        const int ke = min(end, kb + PB);
        Dot2x2 blk[NP];
        for (int k = kb; k < ke; k += 4) {
            Entries nxt;
            nxt.load(ent, k + 2 < end ? k + 2 : next);
            add_pair<TW, IC>(blk, st, cur.a);
            if (k + 1 < ke) add_pair<TW, IC>(blk, st, cur.b);
            if (k + 2 < ke) {
                cur.load(ent, k + 4 < end ? k + 4 : next);
                add_pair<TW, IC>(blk, st, nxt.a);
                if (k + 3 < ke) add_pair<TW, IC>(blk, st, nxt.b);
            } else {
                cur = nxt;
            }
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            if (kb == beg) acc[i] = blk[i];
            else acc[i].merge(blk[i]);
        }
    }
}

// The same for the transposed pass, whose rows go on through the stages of a tile.  Added one block after the other
// (as above, 16 terms each) such a row's error was 1.3 to 1.8 times that of the row kernel's eight lanes: every
// merge into a sum of full size rounds its low part.  So the terms form a tree, blocks of eight, up to 32 terms of
// them in a sum of their own, and that into acc: 0.9 to 1.1 times the row kernel's (rms of x after one iteration,
// float-float, 97^2 with 100, 181^2 with 180 and 256^2 with 30 views).  With 16 instances a stage brings a pixel
// of a ray operator about 30 terms, so one sum takes them all; HALVES (float-float, fewer instances): each block is
// two chains of four.  512^2 at 64: 2.00 -> 2.18 ms per pass; with fewer instances the same time as before.
template <bool HALVES, int IC>
__device__ __forceinline__ void add_row_tree(Dot2x2 (&acc)[Lanes<IC>::NP], const Staged<float2, IC>& st, Entries& cur,
                                             const uint4* __restrict__ ent, int beg, int end, int next) {
    constexpr int NP = Lanes<IC>::NP, part = IC >= 16 ? 1 << 28 : 16;   // entry pairs in a sum of their own
    if (beg == end) {
        cur.load(ent, next);
        return;
    }
    for (int pb = beg; pb < end; pb += part) {
        const int pe = min(end, pb + part);
        Dot2x2 sum[NP];
        for (int k = pb; k < pe; k += 4) {
            Dot2x2 blk[NP], alt[NP];
            auto& odd = HALVES ? alt : blk;
            Entries nxt;
            nxt.load(ent, k + 2 < end ? k + 2 : next);
            add_pair<float2, IC>(blk, st, cur.a);
            if (k + 1 < pe) add_pair<float2, IC>(odd, st, cur.b);
            if (k + 2 < pe) {
                cur.load(ent, k + 4 < end ? k + 4 : next);
                add_pair<float2, IC>(blk, st, nxt.a);
                if (k + 3 < pe) add_pair<float2, IC>(odd, st, nxt.b);
            } else {
                cur = nxt;
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                if (HALVES) blk[i].merge(alt[i]);
                sum[i].merge(blk[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            acc[i].merge(sum[i]);
            acc[i].renorm();
        }
    }
}

}  // namespace

// ------------------------------------------------------------------------------- u = A w
// CTA (tile, IC instances)
template <typename TW, int IC>
__global__ void __launch_bounds__(Lanes<IC>::threads, IC >= 16 ? 3 : 2) kbx_tile_apply(BDims D, TiledA T, BBulkX<TW> X, BSmall S,
                                                              int split, float2* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using LN = Lanes<IC>;
    constexpr int rows = LN::threads / LN::G;   // segments that the CTA walks at a time
    const int B = D.B, nch = B / IC;
    const int bid = (int)blockIdx.x / split, sp = (int)blockIdx.x - bid * split;
    const int t = T.order[bid / nch], c = bid % nch;
    const int row = threadIdx.x / LN::G;
    const Staged<TW, IC> st(smem_raw, threadIdx.x % LN::G, row);
    const TW* wb[LN::VV];
    bool any = false;
#pragma unroll
    for (int v = 0; v < LN::VV; ++v) {
        const int b = c * IC + st.inst(v);
        const DevScalars& sc = S.sc[b];
        wb[v] = (!sc.stop && sc.d < D.dmax) ? X.W + (size_t)sc.d * D.n * B + b : nullptr;
        any = any || wb[v];
    }
    if (!__syncthreads_or(any)) return;
    const int tpf = T.ntx * T.nty;
    const int f = t / tpf, rt = t - f * tpf, ty = rt / T.ntx, tx = rt - ty * T.ntx;
    const int npx = T.TX * T.TY;
    const int64_t fbase = (int64_t)f * T.nx * T.ny;
    for (int q = row; q <= npx; q += rows) {   // slot npx holds 0
        const int py = q / T.TX, px = q - py * T.TX;
        const int iy = ty * T.TY + py, ix = tx * T.TX + px;
        const bool in = q < npx && iy < T.ny && ix < T.nx;
        const int64_t off = (fbase + (int64_t)iy * T.nx + ix) * B;
        TW v[LN::VV];
#pragma unroll
        for (int k = 0; k < LN::VV; ++k) v[k] = (in && wb[k]) ? __ldcg(wb[k] + off) : TW{};
        st.put(smem_raw, q < npx ? tile_slot(q, T.TX) : npx, v);
    }
    __syncthreads();
    // segments s, s + step, ... of the tile: (beg, end) of the present one and of the next
    const int s1 = T.tile_grp[t + 1] * 4, step = rows * split;
    int s = T.tile_grp[t] * 4 + sp * rows + row;
    if (s >= s1) return;
    const uint4* ent = T.ent + (s & 3);
    auto group = [&](int q, int& beg, int& end) {
        const int g = min(q, s1 - 1) >> 2;
        beg = T.goff[g];
        end = T.goff[g + 1];
    };
    int beg, end, nbeg, nend;
    group(s, beg, end);
    group(s + step, nbeg, nend);
    Entries cur;
    cur.load(ent, beg);
    for (; s < s1; s += step) {
        int fbeg, fend;
        group(s + 2 * step, fbeg, fend);
        if constexpr (IC == 16) entries_to_l2(T.ent, nbeg, nend, threadIdx.x & 15);
        Dot2x2 a[LN::NP];
        add_row<TW, IC>(a, st, cur, ent, beg, end, nbeg);
        beg = nbeg;
        end = nend;
        nbeg = fbeg;
        nend = fend;
        float2* dst = part + (size_t)s * B + c * IC;
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

// u_i = sum over the ray's segments of the partials -> column d_i of AW.  NB = 2: a thread takes two
// instances, partials as (hi0, hi1, lo0, lo1).  `lanes` neighbouring lanes share a ray (seg_lanes), each
// with its own accumulator, merged in a fixed tree.
template <typename TW, int NB>
__global__ void __launch_bounds__(kThreads) kbx_seg_reduce(BDims D, TiledA T, BBulkX<TW> X, BSmall S,
                                                           const float2* __restrict__ part, int lanes) {
    const int B = D.B, H = B / NB, G = H * lanes;
    const int b = (threadIdx.x & (H - 1)) * NB, s = (threadIdx.x & (G - 1)) / H;
    float2* out[NB];
    bool any = false;
#pragma unroll
    for (int v = 0; v < NB; ++v) {
        const DevScalars& sc = S.sc[b + v];
        out[v] = (!sc.stop && sc.d < D.dmax) ? X.AW + (size_t)sc.d * D.m * B + b + v : nullptr;
        any = any || out[v];
    }
    if (!__any_sync(0xffffffffu, any)) return;
    const int64_t tot = D.m * G;
    for (int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x; t - lane_id() < tot; t += gstride()) {
        const int64_t r = qdiv(t, G);
        const bool in = t < tot && any;
        const int k0 = in ? T.ray_ptr[r] + s : 0, k1 = in ? T.ray_ptr[r + 1] : 0;
        int c = 0;
        Dot2 a[NB];
        if constexpr (NB == 2) {
            Dot2x2 q;
#pragma unroll 8
            for (int k = k0; k < k1; k += lanes) {
                const float4 f = __ldcs(reinterpret_cast<const float4*>(part + (size_t)T.ray_seg[k] * B + b));
                q.accumulate(pack2(f.x, f.y), pack2(f.z, f.w));
                if (++c % 4 == 0) q.renorm();   // ff.cuh: free, the loads set the pace
            }
            a[0] = q.half(0);
            a[1] = q.half(1);
        } else {
#pragma unroll 8
            for (int k = k0; k < k1; k += lanes) {
                const float2 v = __ldcs(part + (size_t)T.ray_seg[k] * B + b);
                a[0].add2(v.x, v.y);
                if (++c % 4 == 0) a[0].renorm();
            }
        }
#pragma unroll
        for (int v = 0; v < NB; ++v) {
            for (int off = H; off < G; off <<= 1) dot2_xor_merge(a[v], off);
            if (out[v] && in && s == 0) out[v][r * B] = a[v].value();
        }
    }
}

// --------------------------------------------------------- r = A^T e + lambda L^T L x
// CTA (tile of 16 x TY pixels, IC instances); a thread holds PP pixels (u rows + its row) of the tile.
// out == nullptr: appended as column d_i of W_i (rounded to TW); otherwise written to out.
template <int IC, int TY>
struct GradShape {
    static constexpr int px = kTileTX * TY, threads = std::min(Lanes<IC>::threads, px * Lanes<IC>::G);
    static constexpr int rows = threads / Lanes<IC>::G, PP = px / rows;
};

template <typename TW, int IC, int TY>
__global__ void __launch_bounds__(GradShape<IC, TY>::threads, IC >= 16 ? 3 : 1024 / GradShape<IC, TY>::threads)
    kbx_tile_gradient(BDims D, TiledT T, DevL L, BBulkX<TW> X, BSmall S, float2* out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using LN = Lanes<IC>;
    constexpr int rows = GradShape<IC, TY>::rows, PP = GradShape<IC, TY>::PP;
    const int B = D.B, nch = B / IC;
    const int t = T.order[blockIdx.x / nch], c = (int)(blockIdx.x % nch);
    const int row = threadIdx.x / LN::G;
    const Staged<float2, IC> st(smem_raw, threadIdx.x % LN::G, row);
    bool any = false;
#pragma unroll
    for (int v = 0; v < LN::VV; ++v) {
        DevScalars& sc = S.sc[c * IC + st.inst(v)];
        if (sc.stop) continue;
        if (!out && sc.d >= D.dmax) {
            if (t == 0 && row == 0) {
                sc.status = ST_FULL;
                sc.stop = 1;
            }
            continue;
        }
        any = true;
    }
    if (!__syncthreads_or(any)) return;
    Dot2x2 acc[PP][LN::NP];
    // Rows of entries of this lane: pixel u of stage k is group g0 + (k PP + u) rows / 4
    const int ray1 = T.tile_ray[t + 1], stages = T.tile_stage[t + 1] - T.tile_stage[t];
    const uint4* ent = T.ent + (row & 3);
    int g = T.tile_stage[t] * (kTileTX * TY / 4) + (row >> 2);
    const int glast = g + (stages * PP - 1) * (rows / 4);
    int beg = 0, end = 0, nbeg = 0, nend = 0;
    Entries cur{};
    if (stages) {
        beg = T.goff[g];
        end = T.goff[g + 1];
        g = min(g + rows / 4, glast);
        nbeg = T.goff[g];
        nend = T.goff[g + 1];
        cur.load(ent, beg);
    }
    for (int r0 = T.tile_ray[t]; r0 < ray1; r0 += T.stage) {
        const int nr = min(T.stage, ray1 - r0);
        __syncthreads();   // the stage before has been read
#pragma unroll 4
        for (int q = row; q <= nr; q += rows) {
            float2 v[LN::VV] = {};
            if (q < nr) {
                const float2* src = X.e + (size_t)T.ray[r0 + q] * B + c * IC;
                if constexpr (LN::VV == 1) {
                    v[0] = __ldcg(src);
                } else {
#pragma unroll
                    for (int i = 0; i < LN::NP; ++i) {
                        const float4 f = __ldcg(reinterpret_cast<const float4*>(src + st.inst(2 * i)));
                        v[2 * i] = make_float2(f.x, f.y);
                        v[2 * i + 1] = make_float2(f.z, f.w);
                    }
                }
            }
            st.put(smem_raw, q < nr ? q : T.stage, v);   // slot T.stage holds 0
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PP; ++u) {
            g = min(g + rows / 4, glast);
            const int fbeg = T.goff[g], fend = T.goff[g + 1];
            if constexpr (IC == 16) entries_to_l2(T.ent, nbeg, nend, threadIdx.x & 15);
            add_row_tree<(IC < 16 && sizeof(TW) == sizeof(float2)), IC>(acc[u], st, cur, ent, beg, end, nbeg);
            beg = nbeg;
            end = nend;
            nbeg = fbeg;
            nend = fend;
        }
    }
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
            const int b = c * IC + st.inst(v);
            const DevScalars& sc = S.sc[b];
            const int d = sc.d;
            if (sc.stop || (!out && d >= D.dmax)) continue;
            Dot2 a = LN::VV == 1 ? both_halves(acc[u][0]) : acc[u][v / 2].half(v & 1);
            Dot2 lt;
            ff_ltl_row(lt, L, i, StridedW<float2>{X.x + b, B});
            const float2 ltv = lt.value(), lam = X.lam2[b];
            a.add_prod22(lam.x, lam.y, ltv.x, ltv.y);
            if (out) out[i * B + b] = a.value();
            else store_w(X.W + ((size_t)d * D.n + i) * B + b, a);
        }
    }
}

// ------------------------------------------------------------------------------ launchers
int tile_instances(const BDims& D) { return std::min(D.B, D.tile_ic > 0 ? D.tile_ic : kTileInst); }

template <typename TW, int IC>
static cudaError_t tile_apply_ic(const BDims& D, const TiledA& T, const BBulkX<TW>& X, const BSmall& S, float2* part,
                                 cudaStream_t st) {
    const size_t smem = (size_t)(T.TX * T.TY + 1) * IC * sizeof(TW);
    auto k = kbx_tile_apply<TW, IC>;
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    // A tile's segments go to `split` CTAs (each stages the tile) until there are eight rounds of CTAs:
    // with 4.5 rounds, 512^2 at 64 instances, the last one leaves a tenth of the chip's time unused.
    // Eight segments or more remain for every lane, against the staging.
    const int64_t ctas = (int64_t)T.ntiles * (D.B / IC), rows = Lanes<IC>::threads / Lanes<IC>::G;
    const int64_t want = std::min<int64_t>(4, (8 * 152 * 3 + ctas - 1) / ctas), most = T.npart / (T.ntiles * rows * 8);
    const int split = (int)std::max<int64_t>(1, std::min(want, most));
    k<<<(unsigned)(ctas * split), Lanes<IC>::threads, smem, st>>>(D, T, X, S, split, part);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    constexpr int NB = IC == 1 ? 1 : 2;
    const int lanes = seg_lanes(D.B / NB);
    const int64_t rb = (D.m * (D.B / NB) * lanes + kThreads - 1) / kThreads;
    kbx_seg_reduce<TW, NB><<<(int)std::max<int64_t>(1, std::min<int64_t>(rb, 8 * 152)), kThreads, 0, st>>>(D, T, X, S, part, lanes);
    return cudaGetLastError();
}

template <typename TW>
cudaError_t launchbx_tile_apply(const BDims& D, const TiledA& T, const BBulkX<TW>& X, const BSmall& S, float2* part,
                                cudaStream_t st) {
    switch (tile_instances(D)) {
        case 1: return tile_apply_ic<TW, 1>(D, T, X, S, part, st);
        case 2: return tile_apply_ic<TW, 2>(D, T, X, S, part, st);
        case 4: return tile_apply_ic<TW, 4>(D, T, X, S, part, st);
        case 8: return tile_apply_ic<TW, 8>(D, T, X, S, part, st);
        default: return tile_apply_ic<TW, 16>(D, T, X, S, part, st);
    }
}

template <typename TW, int IC, int TY>
static cudaError_t tile_gradient_ty(const BDims& D, const TiledT& T, const DevL& L, const BBulkX<TW>& X, const BSmall& S,
                                    float2* out, cudaStream_t st) {
    const size_t smem = (size_t)(T.stage + 1) * IC * sizeof(float2);
    auto k = kbx_tile_gradient<TW, IC, TY>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)((int64_t)T.ntiles * (D.B / IC)), GradShape<IC, TY>::threads, smem, st>>>(D, T, L, X, S, out);
    return cudaGetLastError();
}

template <typename TW, int IC>
static cudaError_t tile_gradient_ic(const BDims& D, const TiledT& T, const DevL& L, const BBulkX<TW>& X, const BSmall& S,
                                    float2* out, cudaStream_t st) {
    return T.TY == 8 ? tile_gradient_ty<TW, IC, 8>(D, T, L, X, S, out, st)
                     : tile_gradient_ty<TW, IC, 16>(D, T, L, X, S, out, st);
}

template <typename TW>
cudaError_t launchbx_tile_gradient(const BDims& D, const TiledT& T, const DevL& L, const BBulkX<TW>& X, const BSmall& S,
                                   float2* out, cudaStream_t st) {
    switch (std::min(D.B, kTileInst)) {
        case 1: return tile_gradient_ic<TW, 1>(D, T, L, X, S, out, st);
        case 2: return tile_gradient_ic<TW, 2>(D, T, L, X, S, out, st);
        case 4: return tile_gradient_ic<TW, 4>(D, T, L, X, S, out, st);
        case 8: return tile_gradient_ic<TW, 8>(D, T, L, X, S, out, st);
        default: return tile_gradient_ty<TW, 16, 8>(D, T, L, X, S, out, st);   // T is built for the largest group
    }
}

#define SGKS_INST_TILES(TW)                                                                                         \
    template cudaError_t launchbx_tile_apply<TW>(const BDims&, const TiledA&, const BBulkX<TW>&, const BSmall&,     \
                                                 float2*, cudaStream_t);                                            \
    template cudaError_t launchbx_tile_gradient<TW>(const BDims&, const TiledT&, const DevL&, const BBulkX<TW>&,    \
                                                    const BSmall&, float2*, cudaStream_t);
SGKS_INST_TILES(float)
SGKS_INST_TILES(float2)

}  // namespace sgks
