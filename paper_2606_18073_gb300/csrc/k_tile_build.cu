// Builds the tiled layouts of k_tiles.cu from a CSR operator, on the device.
//
// Both sides start from one bit per (tile, row of A): set when the row has an entry in the tile.  A tile has
// bits for the range of rows that reach its frame (frames of a block-diagonal operator share no rows: bits for
// all of them would grow with the square of the number of frames).  The
// running bit count of a tile numbers its rows in ascending order ("local index").  Forward: the
// (row, tile) segments are counted, sorted by length within the tile (stable), cut into groups of four
// and filled by one warp per row, which walks the row's entries in order.  Transposed: the rows of a
// tile are cut into stages; one thread per pixel walks its entries and files each under
// its row's stage.  Every position follows from the order of the entries alone, so the layouts (and the
// sums that run through them) are the same on every run.  Small prefix sums (tiles, groups, rows) are
// taken on the host.
#include <algorithm>
#include <string>
#include <vector>

#include "sgks_internal.cuh"

namespace sgks {

namespace {

// Bits of the tiles of one frame: nw words a tile, tile by tile from word `base`, for the rows from 32 w0 on.
struct FrameBits {
    int64_t base;
    int32_t w0, nw;
};

struct Geo {
    int nx, ny, TX, TY, ntx, nty, ntiles, nt;
    int64_t n, m;
    const FrameBits* fb;   // [nt]
    int64_t words;         // of all tiles
    // first word of a tile; its first row (a multiple of 32) and its number of words
    __device__ __forceinline__ size_t bits_of(int tile, int64_t* row0, int* nw) const {
        const int tpf = ntx * nty, f = tile / tpf;
        const FrameBits b = fb[f];
        *row0 = (int64_t)b.w0 * 32;
        *nw = b.nw;
        return (size_t)b.base + (size_t)(tile - f * tpf) * b.nw;
    }
    __device__ __forceinline__ size_t word(int tile, int64_t row) const {
        int64_t row0;
        int nw;
        const size_t w = bits_of(tile, &row0, &nw);
        return w + (size_t)((row - row0) >> 5);
    }
    __device__ __forceinline__ void locate(int64_t col, int* tile, int* loc) const {
        const int64_t fr = (int64_t)nx * ny, f = qdiv(col, fr), r = col - f * fr;
        const int iy = (int)qdiv(r, nx), ix = (int)(r - (int64_t)iy * nx);
        *tile = (int)(f * ((int64_t)ntx * nty)) + (iy / TY) * ntx + ix / TX;
        *loc = (iy % TY) * TX + ix % TX;
    }
};

__device__ __forceinline__ void mark(uint32_t* bits, const Geo& g, int tile, int64_t row) {
    uint32_t* w = bits + g.word(tile, row);
    const uint32_t b = 1u << (row & 31);
    if (!(*(volatile uint32_t*)w & b)) atomicOr(w, b);
}

// Rows of A with an entry in frame f: lo[f] .. hi[f] (0x7f7f7f7f .. -1 without one), from the rows of A (by_row,
// a warp per row) or from those of A^T (a warp per pixel).  Indices out of range are skipped.
__global__ void k_frame_rows(Geo g, bool by_row, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int64_t nnz,
                             int32_t* lo, int32_t* hi) {
    const int64_t GW = (int64_t)gridDim.x * kWarps, fr = (int64_t)g.nx * g.ny, rows = by_row ? g.m : g.n;
    for (int64_t r = (int64_t)blockIdx.x * kWarps + warp_id(); r < rows; r += GW) {
        const int32_t a = rp[r], z = rp[r + 1];
        if (a < 0 || z < a || z > nnz) continue;
        for (int32_t k = a + lane_id(); k < z; k += 32) {
            const int32_t c = ci[k];
            if (c < 0 || c >= (by_row ? g.n : g.m)) continue;
            const int f = (int)qdiv(by_row ? c : r, fr), row = by_row ? (int)r : c;
            if (row < *(volatile int32_t*)(lo + f)) atomicMin(lo + f, row);
            if (row > *(volatile int32_t*)(hi + f)) atomicMax(hi + f, row);
        }
    }
}

// rows of A: a warp per row.  Column indices and row pointers out of range set err and are skipped.
__global__ void k_tile_mark_rows(Geo g, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int64_t nnz,
                                 uint32_t* bits, int* err) {
    const int64_t GW = (int64_t)gridDim.x * kWarps;
    for (int64_t r = (int64_t)blockIdx.x * kWarps + warp_id(); r < g.m; r += GW) {
        const int32_t a = rp[r], z = rp[r + 1];
        if (a < 0 || z < a || z > nnz) {
            if (lane_id() == 0) *err = 1;
            continue;
        }
        for (int32_t k = a + lane_id(); k < z; k += 32) {
            const int64_t col = ci[k];
            if (col < 0 || col >= g.n) {
                *err = 1;
                continue;
            }
            int tile, loc;
            g.locate(col, &tile, &loc);
            mark(bits, g, tile, r);
        }
    }
}

// rows of A^T: a warp per pixel
__global__ void k_tile_mark_cols(Geo g, const int32_t* __restrict__ trp, const int32_t* __restrict__ tci, int64_t nnz,
                                 uint32_t* bits, int* err) {
    const int64_t GW = (int64_t)gridDim.x * kWarps;
    for (int64_t c = (int64_t)blockIdx.x * kWarps + warp_id(); c < g.n; c += GW) {
        const int32_t a = trp[c], z = trp[c + 1];
        if (a < 0 || z < a || z > nnz) {
            if (lane_id() == 0) *err = 1;
            continue;
        }
        int tile, loc;
        g.locate(c, &tile, &loc);
        for (int32_t k = a + lane_id(); k < z; k += 32) {
            const int64_t r = tci[k];
            if (r < 0 || r >= g.m) *err = 1;
            else mark(bits, g, tile, r);
        }
    }
}

// before[t][w] = set bits of tile t in words < w; cnt[t] their number; rows[r] += 1 per tile of row r
__global__ void __launch_bounds__(kThreads) k_tile_count(Geo g, const uint32_t* __restrict__ bits, int32_t* before,
                                                         int32_t* cnt, int32_t* rows) {
    __shared__ int32_t part[kWarps];
    int64_t row0;
    int nw;
    const size_t first = g.bits_of(blockIdx.x, &row0, &nw);
    const uint32_t* b = bits + first;
    int32_t* o = before + first;
    int32_t base = 0;
    for (int w0 = 0; w0 < nw; w0 += kThreads) {
        const int w = w0 + (int)threadIdx.x;
        const uint32_t v = w < nw ? b[w] : 0u;
        int32_t inc = __popc(v);
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t up = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane_id() >= off) inc += up;
        }
        if (lane_id() == 31) part[warp_id()] = inc;
        __syncthreads();
        int32_t pre = 0, tot = 0;
#pragma unroll
        for (int i = 0; i < kWarps; ++i) {
            if (i < warp_id()) pre += part[i];
            tot += part[i];
        }
        if (w < nw) o[w] = base + pre + inc - __popc(v);
        if (rows)
            for (uint32_t x = v; x; x &= x - 1) atomicAdd(rows + row0 + w * 32 + (__ffs(x) - 1), 1);
        base += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) cnt[blockIdx.x] = base;
}

__device__ __forceinline__ int32_t local_index(const Geo& g, const uint32_t* __restrict__ bits,
                                               const int32_t* __restrict__ before, int tile, int64_t row) {
    const size_t w = g.word(tile, row);
    return before[w] + __popc(bits[w] & ((1u << (row & 31)) - 1u));
}

// entries per segment, segment id = 4 tile_grp[t] + local index
__global__ void k_seg_len(Geo g, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                          const uint32_t* __restrict__ bits, const int32_t* __restrict__ before,
                          const int32_t* __restrict__ tile_grp, int32_t* len) {
    const int64_t GW = (int64_t)gridDim.x * kWarps;
    for (int64_t r = (int64_t)blockIdx.x * kWarps + warp_id(); r < g.m; r += GW)
        for (int32_t k = rp[r] + lane_id(); k < rp[r + 1]; k += 32) {
            int tile, loc;
            g.locate(ci[k], &tile, &loc);
            atomicAdd(len + 4 * tile_grp[tile] + local_index(g, bits, before, tile, r), 1);
        }
}

// Segments of a tile by descending length (lengths from kLenBuckets - 1 on share a bucket), stable:
// pos[id] = the sorted position; pairs[grp] = entry pairs of the longest of a group's four segments.
constexpr int kLenBuckets = 128;
__global__ void __launch_bounds__(32) k_seg_sort(const int32_t* __restrict__ tile_grp, const int32_t* __restrict__ cnt,
                                                 const int32_t* __restrict__ len, int32_t* pos, int32_t* pairs) {
    __shared__ int32_t at[kLenBuckets];
    const int lane = threadIdx.x, t = blockIdx.x;
    const int32_t id0 = 4 * tile_grp[t], ns = cnt[t];
    for (int i = lane; i < kLenBuckets; i += 32) at[i] = 0;
    __syncwarp();
    for (int32_t i = lane; i < ns; i += 32) atomicAdd(at + min(len[id0 + i], kLenBuckets - 1), 1);
    __syncwarp();
    if (lane == 0) {   // first position of each bucket, the longest first
        int32_t run = 0;
        for (int i = kLenBuckets - 1; i >= 0; --i) {
            const int32_t c = at[i];
            at[i] = run;
            run += c;
        }
    }
    __syncwarp();
    for (int32_t i0 = 0; i0 < ns; i0 += 32) {
        const int32_t i = i0 + lane;
        const int32_t l = i < ns ? len[id0 + i] : 0;
        const int bk = i < ns ? min(l, kLenBuckets - 1) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, bk);
        if (bk >= 0) {
            const int32_t p = id0 + at[bk] + __popc(peers & ((1u << lane) - 1u));
            pos[id0 + i] = p;
            atomicMax(pairs + (p >> 2), (l + 1) / 2);
        }
        __syncwarp();
        if (bk >= 0 && lane == 31 - __clz(peers)) at[bk] += __popc(peers);
        __syncwarp();
    }
}

// entry e of row `pos` of a group whose pairs start at `off`: (slot, slot, value, value) per pair
__device__ __forceinline__ void put_entry(uint32_t* ent, int32_t off, int32_t e, int pos, uint32_t slot, float val) {
    uint32_t* q = ent + (((size_t)off + (e >> 1)) * 4 + pos) * 4 + (e & 1);
    q[0] = slot;
    q[2] = __float_as_uint(val);
}

__global__ void k_tile_pad(uint4* ent, int64_t count, uint32_t slot) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        ent[i] = make_uint4(slot, slot, 0u, 0u);
}

// a warp per row, 32 entries at a time in their order; used[id]: entries placed so far
__global__ void k_seg_fill(Geo g, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                           const float* __restrict__ val, const uint32_t* __restrict__ bits,
                           const int32_t* __restrict__ before, const int32_t* __restrict__ tile_grp,
                           const int32_t* __restrict__ pos, const int32_t* __restrict__ goff,
                           const int32_t* __restrict__ ray_ptr, int32_t* used, uint32_t* ent, int32_t* ray_seg) {
    const int64_t GW = (int64_t)gridDim.x * kWarps;
    const int lane = lane_id();
    for (int64_t r = (int64_t)blockIdx.x * kWarps + warp_id(); r < g.m; r += GW) {
        const int32_t a = rp[r], z = rp[r + 1];
        int32_t out = ray_ptr[r];
        for (int32_t k0 = a; k0 < z; k0 += 32) {
            const int32_t k = k0 + lane;
            const bool act = k < z;
            int32_t id = -1, p = 0, have = 0;
            int tile = 0, loc = 0;
            if (act) {
                g.locate(ci[k], &tile, &loc);
                id = 4 * tile_grp[tile] + local_index(g, bits, before, tile, r);
                p = pos[id];
                have = *(volatile int32_t*)(used + id);
            }
            const unsigned peers = __match_any_sync(0xffffffffu, id);
            const int32_t e = have + __popc(peers & ((1u << lane) - 1u));
            const bool first = act && e == 0;
            const unsigned firsts = __ballot_sync(0xffffffffu, first);
            if (first) ray_seg[out + __popc(firsts & ((1u << lane) - 1u))] = p;
            out += __popc(firsts);
            if (act) {
                put_entry(ent, goff[p >> 2], e, p & 3, (uint32_t)tile_slot(loc, g.TX), val[k]);
                if (lane == 31 - __clz(peers)) *(volatile int32_t*)(used + id) = have + __popc(peers);
            }
            __syncwarp();
        }
    }
}

// the rows of each tile in ascending order
__global__ void k_tile_rays(Geo g, const uint32_t* __restrict__ bits, const int32_t* __restrict__ before,
                            const int32_t* __restrict__ tile_ray, int32_t* ray) {
    int64_t row0;
    int nw;
    const size_t first = g.bits_of(blockIdx.x, &row0, &nw);
    const uint32_t* b = bits + first;
    const int32_t* o = before + first;
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
        int32_t p = tile_ray[blockIdx.x] + o[w];
        for (uint32_t x = b[w]; x; x &= x - 1) ray[p++] = (int32_t)(row0 + w * 32 + (__ffs(x) - 1));
    }
}

// Entries of a pixel per stage (fill = false), or placed (fill = true): one thread per pixel, in order.
template <bool FILL>
__global__ void k_pixel_entries(Geo g, const int32_t* __restrict__ trp, const int32_t* __restrict__ tci,
                                const float* __restrict__ tval, const uint32_t* __restrict__ bits,
                                const int32_t* __restrict__ before, const int32_t* __restrict__ tile_stage, int stage,
                                int32_t* used,
                                const int32_t* __restrict__ goff, uint32_t* ent) {
    const int npx = g.TX * g.TY;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < g.n; c += (int64_t)gridDim.x * blockDim.x) {
        int tile, loc;
        g.locate(c, &tile, &loc);
        for (int32_t k = trp[c]; k < trp[c + 1]; ++k) {
            const int32_t li = local_index(g, bits, before, tile, tci[k]);
            const int64_t st = tile_stage[tile] + li / stage;
            const int32_t e = used[st * npx + loc]++;
            if (FILL) put_entry(ent, goff[st * (npx / 4) + (loc >> 2)], e, loc & 3, (uint32_t)(li % stage), tval[k]);
        }
    }
}

__global__ void k_group_pairs(const int32_t* __restrict__ used, int64_t groups, int32_t* pairs) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < groups; i += (int64_t)gridDim.x * blockDim.x) {
        const int4 u = reinterpret_cast<const int4*>(used)[i];
        pairs[i] = (max(max(u.x, u.y), max(u.z, u.w)) + 1) / 2;
    }
}

unsigned grid_for(int64_t work) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>(work, 16 * 152)); }

// Device memory of one build on its stream; what is not handed over (keep) is freed at the end.
struct Build {
    cudaStream_t st;
    cudaError_t e = cudaSuccess;
    std::vector<void*> tmp, own;
    explicit Build(cudaStream_t s) : st(s) {}
    template <typename P>
    P* temp(size_t count) {
        void* q = nullptr;
        if (e == cudaSuccess) e = cudaMallocAsync(&q, count * sizeof(P) + 16, st);
        if (e == cudaSuccess) tmp.push_back(q);
        return e == cudaSuccess ? (P*)q : nullptr;
    }
    template <typename P>
    P* held(size_t count) {
        void* q = nullptr;
        if (e == cudaSuccess) e = cudaMalloc(&q, count * sizeof(P) + 16);
        if (e == cudaSuccess) own.push_back(q);
        return e == cudaSuccess ? (P*)q : nullptr;
    }
    void keep(std::vector<void*>& allocs) {
        allocs.insert(allocs.end(), own.begin(), own.end());
        own.clear();
    }
    void zero(void* p, size_t bytes) {
        if (e == cudaSuccess && bytes) e = cudaMemsetAsync(p, 0, bytes, st);
    }
    void ran() {
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    std::vector<int32_t> down(const int32_t* p, size_t count) {
        std::vector<int32_t> h(count);
        if (e == cudaSuccess && count) e = cudaMemcpyAsync(h.data(), p, sizeof(int32_t) * count, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        return h;
    }
    int32_t* up(const std::vector<int32_t>& h) {
        int32_t* p = held<int32_t>(h.size());
        if (e == cudaSuccess) e = cudaMemcpyAsync(p, h.data(), sizeof(int32_t) * h.size(), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // the host vector may die
        return p;
    }
    ~Build() {
        for (void* q : tmp) cudaFreeAsync(q, st);
        for (void* q : own) cudaFree(q);   // waits for the kernels that use it
    }
};

// Bit rows of all tiles, with their counts 8 bytes a word: 32 GB at most, for a while.  Rays through the whole image
// with fewer than 2^31 entries stay below it up to 16384^2 pixels; beyond, and where that memory is not
// there, the row kernels remain.
constexpr size_t kMaxWords = (size_t)1 << 32;

// exclusive prefix sums with the total at the end; false when they do not fit
bool prefix(const std::vector<int32_t>& v, std::vector<int32_t>* out) {
    out->resize(v.size() + 1);
    int64_t run = 0;
    for (size_t i = 0; i < v.size(); ++i) {
        (*out)[i] = (int32_t)run;
        run += v[i];
        if (run >= ((int64_t)1 << 31)) return false;
    }
    (*out)[v.size()] = (int32_t)run;
    return true;
}

// tiles by descending number of entry pairs (equal ones in their own order)
std::vector<int32_t> heavy_first(const std::vector<int32_t>& off, const std::vector<int32_t>& tile0, int per) {
    std::vector<int32_t> o(tile0.size() - 1);
    for (size_t i = 0; i < o.size(); ++i) o[i] = (int32_t)i;
    auto work = [&](int32_t t) { return off[(size_t)tile0[t + 1] * per] - off[(size_t)tile0[t] * per]; };
    std::stable_sort(o.begin(), o.end(), [&](int32_t a, int32_t b) { return work(a) > work(b); });
    return o;
}

bool geometry(int64_t m, int64_t n, int nx, int ny, int nt, int TX, int TY, Geo* g) {
    if ((int64_t)nx * ny * nt != n) return false;
    *g = Geo{nx, ny, TX, TY, (nx + TX - 1) / TX, (ny + TY - 1) / TY, 0, nt, n, m, nullptr, 0};
    const int64_t tiles = (int64_t)g->ntx * g->nty * nt;
    g->ntiles = (int)tiles;
    return tiles < ((int64_t)1 << 31);
}

// g.fb and g.words; one frame takes bits for all rows without looking at the entries
void frame_bits(Build& b, Geo& g, bool by_row, const int32_t* rp, const int32_t* ci, int64_t nnz) {
    std::vector<int32_t> lo((size_t)g.nt, 0), hi((size_t)g.nt, (int32_t)(g.m - 1));
    if (g.nt > 1) {
        int32_t *dlo = b.temp<int32_t>(g.nt), *dhi = b.temp<int32_t>(g.nt);
        if (b.e == cudaSuccess) b.e = cudaMemsetAsync(dlo, 0x7f, 4 * (size_t)g.nt, b.st);
        if (b.e == cudaSuccess) b.e = cudaMemsetAsync(dhi, 0xff, 4 * (size_t)g.nt, b.st);
        if (b.e != cudaSuccess) return;
        const int64_t rows = by_row ? g.m : g.n;
        k_frame_rows<<<grid_for((rows + kWarps - 1) / kWarps), kThreads, 0, b.st>>>(g, by_row, rp, ci, nnz, dlo, dhi);
        b.ran();
        lo = b.down(dlo, g.nt);
        hi = b.down(dhi, g.nt);
    }
    std::vector<FrameBits> h((size_t)g.nt);
    for (int f = 0; f < g.nt; ++f) {
        const int32_t w0 = hi[f] < 0 ? 0 : lo[f] / 32, nw = hi[f] < 0 ? 0 : hi[f] / 32 - w0 + 1;
        h[f] = FrameBits{g.words, w0, nw};
        g.words += (int64_t)nw * g.ntx * g.nty;
    }
    FrameBits* d = b.temp<FrameBits>(g.nt);
    if (b.e == cudaSuccess) b.e = cudaMemcpyAsync(d, h.data(), sizeof(FrameBits) * h.size(), cudaMemcpyHostToDevice, b.st);
    if (b.e == cudaSuccess) b.e = cudaStreamSynchronize(b.st);   // the host vector dies
    g.fb = d;
}

// Without the memory for a layout the row kernels remain, which need none of it: no error.
int failed(const Build& b, std::string* why) {
    if (b.e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return SGKS_OK;
    }
    *why = std::string("tiled operator: ") + cudaGetErrorString(b.e);
    return SGKS_ERR_CUDA;
}

int refused(std::string* why, const char* what) {
    *why = std::string("tiled operator: ") + what;
    return SGKS_ERR_INVALID;
}

}  // namespace

bool tile_room(std::vector<void*>& allocs) {
    size_t room = 0, total = 0;
    if (cudaMemGetInfo(&room, &total) == cudaSuccess && room >= kTileRoom) return true;
    cudaGetLastError();
    drop_tile_memory(allocs);
    return false;
}

bool tile_memory(std::vector<void*>& allocs, void** p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        drop_tile_memory(allocs);
        return false;
    }
    allocs.push_back(*p);
    return tile_room(allocs);
}

void drop_tile_memory(std::vector<void*>& allocs) {
    for (void* q : allocs) cudaFree(q);
    allocs.clear();
}

int build_tiles(const int32_t* rp, const int32_t* ci, const float* val, int64_t m, int64_t n, int64_t nnz, int nx, int ny,
                int nt, int TX, int TY, TiledA& T, std::vector<void*>& allocs, cudaStream_t st, std::string* why) {
    Geo g;
    if (TX % 2 != 0 || nnz >= ((int64_t)1 << 31) || !geometry(m, n, nx, ny, nt, TX, TY, &g))
        return refused(why, "geometry does not match the unknowns");
    Build b(st);
    frame_bits(b, g, true, rp, ci, nnz);
    const size_t nw = (size_t)g.words, row_words = (size_t)(m + 31) / 32 * 32;
    if (nw > kMaxWords) return SGKS_OK;
    uint32_t* bits = b.temp<uint32_t>(nw);
    int32_t *before = b.temp<int32_t>(nw), *cnt = b.temp<int32_t>(g.ntiles), *rows = b.temp<int32_t>(row_words);
    int32_t* err = b.temp<int32_t>(1);
    b.zero(bits, nw * 4);
    b.zero(rows, row_words * 4);
    b.zero(err, 4);
    if (b.e != cudaSuccess) return failed(b, why);
    const unsigned gr = grid_for((m + kWarps - 1) / kWarps);
    k_tile_mark_rows<<<gr, kThreads, 0, st>>>(g, rp, ci, nnz, bits, err);
    k_tile_count<<<g.ntiles, kThreads, 0, st>>>(g, bits, before, cnt, rows);
    b.ran();
    const std::vector<int32_t> herr = b.down(err, 1), hcnt = b.down(cnt, g.ntiles);
    if (b.e != cudaSuccess) return failed(b, why);
    if (herr[0]) return refused(why, "a row pointer or column index out of range");
    std::vector<int32_t> grp(hcnt), grp0, off;
    for (int32_t& v : grp) v = (v + 3) / 4;
    if (!prefix(grp, &grp0) || grp0.back() >= (1 << 29)) return SGKS_OK;
    const int64_t ngrp = grp0.back();
    int32_t* tile_grp = b.up(grp0);
    int32_t *len = b.temp<int32_t>(4 * ngrp), *pos = b.temp<int32_t>(4 * ngrp), *pairs = b.temp<int32_t>(ngrp);
    b.zero(len, 16 * ngrp);
    b.zero(pairs, 4 * ngrp);
    if (b.e != cudaSuccess) return failed(b, why);
    k_seg_len<<<gr, kThreads, 0, st>>>(g, rp, ci, bits, before, tile_grp, len);
    k_seg_sort<<<g.ntiles, 32, 0, st>>>(tile_grp, cnt, len, pos, pairs);
    b.ran();
    if (!prefix(b.down(pairs, ngrp), &off)) return SGKS_OK;   // too many for 32-bit positions
    const int64_t npairs = (int64_t)off.back() + kTileAhead;
    int32_t *goff = b.up(off), *order = b.up(heavy_first(off, grp0, 1));
    if (!prefix(b.down(rows, m), &off)) return SGKS_OK;
    const int64_t nseg = off.back();
    int32_t *ray_ptr = b.up(off), *ray_seg = b.held<int32_t>(nseg);
    uint4* ent = b.held<uint4>(4 * npairs);
    b.zero(len, 16 * ngrp);   // from here on: entries placed
    if (b.e != cudaSuccess) return failed(b, why);
    k_tile_pad<<<grid_for((4 * npairs + 255) / 256), 256, 0, st>>>(ent, 4 * npairs, (uint32_t)(TX * TY));
    k_seg_fill<<<gr, kThreads, 0, st>>>(g, rp, ci, val, bits, before, tile_grp, pos, goff, ray_ptr, len, (uint32_t*)ent,
                                        ray_seg);
    b.ran();
    if (b.e != cudaSuccess) return failed(b, why);
    b.keep(allocs);
    T = TiledA{TX, TY, nx, ny, nt, g.ntx, g.nty, g.ntiles, 4 * ngrp, nseg, order, tile_grp, goff, ray_ptr, ray_seg, ent};
    return SGKS_OK;
}

int build_tiles_t(const int32_t* trp, const int32_t* tci, const float* tval, int64_t m, int64_t n, int64_t nnz, int nx,
                  int ny, int nt, int TY, int stage, TiledT& T, std::vector<void*>& allocs, cudaStream_t st, std::string* why) {
    constexpr int TX = kTileTX;
    const int npx = TX * TY;
    Geo g;
    if (nnz >= ((int64_t)1 << 31) || !geometry(m, n, nx, ny, nt, TX, TY, &g))
        return refused(why, "geometry does not match the unknowns");
    Build b(st);
    frame_bits(b, g, false, trp, tci, nnz);
    const size_t nw = (size_t)g.words;
    if (nw > kMaxWords) return SGKS_OK;
    uint32_t* bits = b.temp<uint32_t>(nw);
    int32_t *before = b.temp<int32_t>(nw), *cnt = b.temp<int32_t>(g.ntiles), *err = b.temp<int32_t>(1);
    b.zero(bits, nw * 4);
    b.zero(err, 4);
    if (b.e != cudaSuccess) return failed(b, why);
    k_tile_mark_cols<<<grid_for((n + kWarps - 1) / kWarps), kThreads, 0, st>>>(g, trp, tci, nnz, bits, err);
    k_tile_count<<<g.ntiles, kThreads, 0, st>>>(g, bits, before, cnt, nullptr);
    b.ran();
    const std::vector<int32_t> herr = b.down(err, 1), hcnt = b.down(cnt, g.ntiles);
    if (b.e != cudaSuccess) return failed(b, why);
    if (herr[0]) return refused(why, "a row pointer or row index of A^T out of range");
    std::vector<int32_t> rays, stages(hcnt), stage0;
    for (int32_t& v : stages) v = (v + stage - 1) / stage;
    if (!prefix(hcnt, &rays) || !prefix(stages, &stage0) || (int64_t)stage0.back() * npx >= ((int64_t)1 << 31)) return SGKS_OK;
    // A pixel has to find a staged ray several times over for the staging to pay (a ray crosses 16-odd
    // pixels of a tile; 4 is where the staged rows cost as much as a quarter of the row kernel's gathers),
    // and its entries have to fill the groups of four: otherwise the row kernel stays (T.ntiles = 0).
    if ((int64_t)rays.back() * 4 > nnz) return SGKS_OK;
    const int64_t groups = (int64_t)stage0.back() * (npx / 4);
    int32_t *used = b.temp<int32_t>(4 * groups), *pairs = b.temp<int32_t>(groups);
    int32_t* tile_stage = b.up(stage0);
    b.zero(used, 16 * groups);
    if (b.e != cudaSuccess) return failed(b, why);
    const unsigned gc = grid_for((n + kThreads - 1) / kThreads);
    k_pixel_entries<false><<<gc, kThreads, 0, st>>>(g, trp, tci, tval, bits, before, tile_stage, stage, used, nullptr, nullptr);
    k_group_pairs<<<grid_for((groups + 255) / 256), 256, 0, st>>>(used, groups, pairs);
    b.ran();
    std::vector<int32_t> off;
    if (!prefix(b.down(pairs, groups), &off)) return SGKS_OK;
    const int64_t npairs = (int64_t)off.back() + kTileAhead;
    if (b.e != cudaSuccess) return failed(b, why);
    if ((npairs - kTileAhead) * 8 > 2 * nnz) return SGKS_OK;
    int32_t *goff = b.up(off), *order = b.up(heavy_first(off, stage0, npx / 4)), *tile_ray = b.up(rays), *ray = b.held<int32_t>(rays.back());
    uint4* ent = b.held<uint4>(4 * npairs);
    b.zero(used, 16 * groups);
    if (b.e != cudaSuccess) return failed(b, why);
    k_tile_rays<<<g.ntiles, kThreads, 0, st>>>(g, bits, before, tile_ray, ray);
    k_tile_pad<<<grid_for((4 * npairs + 255) / 256), 256, 0, st>>>(ent, 4 * npairs, (uint32_t)stage);
    k_pixel_entries<true><<<gc, kThreads, 0, st>>>(g, trp, tci, tval, bits, before, tile_stage, stage, used, goff, (uint32_t*)ent);
    b.ran();
    if (b.e != cudaSuccess) return failed(b, why);
    b.keep(allocs);
    T = TiledT{TX, TY, nx, ny, nt, g.ntx, g.nty, g.ntiles, order, tile_stage, tile_ray, ray, goff, stage, ent};
    return SGKS_OK;
}

__global__ void k_tile_finite(const float* __restrict__ val, int64_t nnz, int* bad) {
    bool b = false;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nnz; k += (int64_t)gridDim.x * blockDim.x)
        b = b || !isfinite(val[k]);
    if (b) *bad = 1;
}

int build_tiles64(const sgks_reg* reg, const int32_t* rp, const int32_t* ci, const float* val, const int32_t* trp,
                  const int32_t* tci, const float* tval, int64_t m, int64_t n, int64_t nnz, int B, TiledA& T, TiledT& Tt,
                  std::vector<void*>& allocs, cudaStream_t st, std::string* why) {
    if (reg->kind == SGKS_REG_FD1 || nnz < (1 << 20)) return SGKS_OK;
    const int nt = reg->kind == SGKS_REG_SPACETIME ? reg->nt : 1;
    if ((int64_t)reg->nx * reg->ny * nt != n) return SGKS_OK;
    // A CTA of the transposed pass holds a tile, for eight instances at most, so a small image with many rays leaves
    // most of the chip idle, where the row kernels fill it.  Solves of 12 iterations against the row kernels
    // (CT, 90 and 300 views; CTAs): one vector 0.90 (16), 1.01 (25), 1.10-1.17 (49); groups of 2 to 8, also
    // 8 + 2 + 1, 0.55-1.0 (49), 0.87-1.1 (64), 0.86-1.16 (81), 0.96-1.23 (100), 1.02-1.3 (144); of 16 and more, also
    // 16 + 1, 0.88-1.1 (64), 0.95-1.2 (182), 0.98-1.27 (196), 1.1-1.36 (256).
    const int64_t grad_ctas = (int64_t)((reg->nx + kTileTX - 1) / kTileTX) * ((reg->ny + tile_ty(B) - 1) / tile_ty(B)) * nt *
                              std::max(1, B / 8);
    if (grad_ctas < (B == 1 ? 24 : (B < kTileInst ? 128 : 224))) return SGKS_OK;
    {
        Build b(st);
        int32_t* bad = b.temp<int32_t>(1);
        b.zero(bad, 4);
        if (b.e != cudaSuccess) return failed(b, why);
        for (const float* v : {val, tval}) k_tile_finite<<<grid_for((nnz + 255) / 256), 256, 0, st>>>(v, nnz, bad);
        b.ran();
        const std::vector<int32_t> h = b.down(bad, 1);
        if (b.e != cudaSuccess) return failed(b, why);
        if (h[0]) return SGKS_OK;
    }
    TiledA a{};
    TiledT t{};
    Build both(st);   // holds the one layout until the other is there too
    int rc = build_tiles_t(trp, tci, tval, m, n, nnz, reg->nx, reg->ny, nt, tile_ty(B), tile_stage(std::min(B, 8)), t, both.own, st, why);
    if (rc != SGKS_OK || !t.ntiles) return rc;
    // 32 x 16 pixels for the forward pass where the same count of tiles as for the compensated batches allows it: that
    // pass has up to four times as many CTAs, of four instances, but its tiles are the ones that were measured.
    const int64_t ctas = (int64_t)((reg->nx + 31) / 32) * ((reg->ny + 15) / 16) * nt * std::max(1, B / kTileInst);
    rc = build_tiles(rp, ci, val, m, n, nnz, reg->nx, reg->ny, nt, ctas < 4 * 152 ? 16 : 32, 16, a, both.own, st, why);
    if (rc != SGKS_OK || !a.ntiles || a.nseg * 4 > nnz) return rc;
    both.keep(allocs);
    T = a;
    Tt = t;
    return SGKS_OK;
}

}  // namespace sgks
