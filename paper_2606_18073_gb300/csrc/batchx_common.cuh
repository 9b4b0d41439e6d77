// Pieces shared by the compensated batched kernels (k_batchx.cu, k_tiles.cu): basis values in TW
// (float or float2) into Dot2 accumulators, the rows of L and L^T L in float-float, and vectors staged in
// shared memory row by row.
#pragma once

#include "batch_common.cuh"
#include "ff.cuh"

namespace sgks {

__device__ __forceinline__ float2 ff_zero() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ float2 ff_neg(float2 v) { return make_float2(-v.x, -v.y); }

// coef * w into the accumulator, w in the basis storage type
__device__ __forceinline__ void acc_w(Dot2& a, float coef, float w) { a.add_prod(coef, w); }
__device__ __forceinline__ void acc_w(Dot2& a, float coef, float2 w) { a.add_prod2(coef, w.x, w.y); }
// w * (yh + yl)
__device__ __forceinline__ void acc_wy(Dot2& a, float w, float yh, float yl) { a.add_prod2(w, yh, yl); }
__device__ __forceinline__ void acc_wy(Dot2& a, float2 w, float yh, float yl) { a.add_prod22(w.x, w.y, yh, yl); }
// +- v into the accumulator (sign = +-1, exact)
__device__ __forceinline__ void acc_add(Dot2& a, float sign, float v) { a.add(sign * v); }
__device__ __forceinline__ void acc_add(Dot2& a, float sign, float2 v) { a.add2(sign * v.x, sign * v.y); }
// store an accumulated value in the basis type (float: nearest float of p + s)
__device__ __forceinline__ void store_w(float* p, const Dot2& a) { *p = a.rounded(); }
__device__ __forceinline__ void store_w(float2* p, const Dot2& a) { *p = a.value(); }

template <typename TW>
__device__ __forceinline__ TW wzero() { return TW{}; }

// VV consecutive basis values with one 16-byte load (VV * sizeof(TW) == 16), or VV loads
template <typename TW, int VV>
__device__ __forceinline__ void ldw(const TW* __restrict__ p, TW (&o)[VV]) {
    if constexpr (VV * sizeof(TW) == 16) {
        const float4 f = __ldcg(reinterpret_cast<const float4*>(p));
        if constexpr (sizeof(TW) == 4) {
            o[0] = f.x; o[1] = f.y; o[2] = f.z; o[3] = f.w;
        } else {
            o[0] = make_float2(f.x, f.y);
            o[1] = make_float2(f.z, f.w);
        }
    } else {
#pragma unroll
        for (int v = 0; v < VV; ++v) o[v] = __ldcg(p + v);
    }
}

// ------------------------------------------------------------------ stencils in float-float
// (L w)_k as float-float (a difference of two values, or the 5-point Laplacian).
template <typename TW, typename X>
__device__ __forceinline__ float2 ff_l_row(const DevL& L, int64_t k, const X& w) {
    const int nx = L.nx, ny = L.ny;
    Dot2 a;
    switch (L.kind) {
        case SGKS_REG_FD1:
            acc_add(a, 1.f, w(k + 1));
            acc_add(a, -1.f, w(k));
            break;
        case SGKS_REG_GRAD2D: {
            const int64_t nh = (int64_t)ny * (nx - 1);
            if (k < nh) {
                const int64_t iy = qdiv(k, nx - 1), ix = k - iy * (nx - 1), q = iy * nx + ix;
                acc_add(a, 1.f, w(q + 1));
                acc_add(a, -1.f, w(q));
            } else {
                const int64_t q = k - nh;
                acc_add(a, 1.f, w(q + nx));
                acc_add(a, -1.f, w(q));
            }
            break;
        }
        case SGKS_REG_LAPLACE2D: {
            const int iy = (int)qdiv(k, nx), ix = (int)(k - (int64_t)iy * nx);
            acc_w(a, 4.f, w(k));
            if (ix > 0) acc_add(a, -1.f, w(k - 1));
            if (ix < nx - 1) acc_add(a, -1.f, w(k + 1));
            if (iy > 0) acc_add(a, -1.f, w(k - nx));
            if (iy < ny - 1) acc_add(a, -1.f, w(k + nx));
            break;
        }
        default: {   // SPACETIME
            const int64_t per = (int64_t)ny * (nx - 1), per2 = (int64_t)(ny - 1) * nx;
            const int64_t n1 = per * L.nt, n2 = per2 * L.nt, fr = (int64_t)nx * ny;
            int64_t q, st;
            if (k < n1) {
                const int64_t t = qdiv(k, per), r = k - t * per, iy = qdiv(r, nx - 1), ix = r - iy * (nx - 1);
                q = t * fr + iy * nx + ix;
                st = 1;
            } else if (k < n1 + n2) {
                const int64_t kk = k - n1, t = qdiv(kk, per2);
                q = t * fr + (kk - t * per2);
                st = nx;
            } else {
                q = k - n1 - n2;
                st = fr;
            }
            acc_add(a, 1.f, w(q + st));
            acc_add(a, -1.f, w(q));
            break;
        }
    }
    return a.value();
}

// coef * (x_i - x_{i+stride}) and coef * (x_i - x_{i-stride}) where the neighbours exist
template <typename X>
__device__ __forceinline__ void ff_fd_pair(Dot2& a, const X& x, int64_t i, int64_t stride, int pos, int len) {
    const float2 xi = x(i);
    if (pos < len - 1) {
        acc_add(a, 1.f, xi);
        acc_add(a, -1.f, x(i + stride));
    }
    if (pos > 0) {
        acc_add(a, 1.f, xi);
        acc_add(a, -1.f, x(i - stride));
    }
}

template <typename X>
__device__ __forceinline__ void ff_lap5(Dot2& a, float coef, const X& x, int iy, int ix, int nx, int ny) {
    const int64_t q = (int64_t)iy * nx + ix;
    acc_w(a, 4.f * coef, x(q));
    if (ix > 0) acc_w(a, -coef, x(q - 1));
    if (ix < nx - 1) acc_w(a, -coef, x(q + 1));
    if (iy > 0) acc_w(a, -coef, x(q - nx));
    if (iy < ny - 1) acc_w(a, -coef, x(q + nx));
}

// (L^T L x)_i accumulated into a (x float-float)
template <typename X>
__device__ __forceinline__ void ff_ltl_row(Dot2& a, const DevL& L, int64_t i, const X& x) {
    const int nx = L.nx, ny = L.ny;
    switch (L.kind) {
        case SGKS_REG_FD1:
            ff_fd_pair(a, x, i, 1, (int)i, nx);
            break;
        case SGKS_REG_GRAD2D: {
            const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
            ff_fd_pair(a, x, i, 1, ix, nx);
            ff_fd_pair(a, x, i, nx, iy, ny);
            break;
        }
        case SGKS_REG_LAPLACE2D: {   // L symmetric: L^T L = L^2
            const int iy = (int)qdiv(i, nx), ix = (int)(i - (int64_t)iy * nx);
            ff_lap5(a, 4.f, x, iy, ix, nx, ny);
            if (ix > 0) ff_lap5(a, -1.f, x, iy, ix - 1, nx, ny);
            if (ix < nx - 1) ff_lap5(a, -1.f, x, iy, ix + 1, nx, ny);
            if (iy > 0) ff_lap5(a, -1.f, x, iy - 1, ix, nx, ny);
            if (iy < ny - 1) ff_lap5(a, -1.f, x, iy + 1, ix, nx, ny);
            break;
        }
        default: {   // SPACETIME
            const int64_t fr = (int64_t)nx * ny;
            const int t = (int)qdiv(i, fr);
            const int64_t r = i - (int64_t)t * fr;
            const int iy = (int)qdiv(r, nx), ix = (int)(r - (int64_t)iy * nx);
            ff_fd_pair(a, x, i, 1, ix, nx);
            ff_fd_pair(a, x, i, nx, iy, ny);
            ff_fd_pair(a, x, i, fr, t, L.nt);
            break;
        }
    }
}

template <typename TW>
struct StridedW {
    const TW* __restrict__ p;
    int64_t st;
    __device__ __forceinline__ TW operator()(int64_t q) const { return p[q * st]; }
};

// -------------------------------------------------- values staged in shared memory (k_tiles.cu, k_sketchx.cu)
// Lane layout for IC staged instances: a lane takes VV of them (VV = 1: IC = 1, the halves of an
// .f32x2 operand are then the two entries of a pair), G = IC / VV lanes per row.
template <int IC>
struct Lanes {
    static constexpr int VV = IC >= 16 ? 4 : (IC >= 2 ? 2 : 1);
    static constexpr int NP = VV == 4 ? 2 : 1;   // .f32x2 accumulators of a lane
    static constexpr int G = IC / VV;
    // Threads: two such pairs per lane take 80 registers, 256 threads then fill an SM three times over;
    // with fewer instances a tile's CTA is small work and takes 512.
    static constexpr int threads = IC >= 16 ? 256 : 512;
};

// A staged row in shared memory and a lane's part of it.
template <typename TW, int IC>
struct Staged;

// float-float: pairs of instances as (hi0, hi1, lo0, lo1).  With 16 instances a row fills all banks; the
// eight lanes of a load phase belong to two rows, and those of the odd one take the row's upper half
// first, so that the phase touches every bank once.
template <int IC>
struct Staged<float2, IC> {
    using LN = Lanes<IC>;
    static constexpr int kRow = IC * 8;
    int first;    // instance of accumulator 0
    int second;   // of accumulator 1 (VV = 4)
    const unsigned char *p0, *p1;
    __device__ __forceinline__ Staged(const unsigned char* base, int j, int row) {
        if constexpr (LN::VV == 4) {
            const int c0 = j + ((row & 1) ? LN::G : 0), c1 = j + ((row & 1) ? 0 : LN::G);
            first = 2 * c0;
            second = 2 * c1;
        } else {
            first = second = LN::VV * j;
        }
        p0 = base + first * 8;
        p1 = base + second * 8;
    }
    __device__ __forceinline__ int inst(int v) const { return (v < 2 ? first : second) + (v & 1); }
    __device__ __forceinline__ void add(Dot2x2 (&d)[LN::NP], uint32_t slot, float c) const {
        const f32x2 cc = pack2(c, c);
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p0 + slot * kRow);
        d[0].add_prod2(cc, v.x, v.y);
        if constexpr (LN::NP == 2) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(p1 + slot * kRow);
            d[1].add_prod2(cc, w.x, w.y);
        }
    }
    __device__ __forceinline__ void add_both(Dot2x2& d, uint32_t s0, uint32_t s1, float c0, float c1) const {
        const float2 a = *reinterpret_cast<const float2*>(p0 + s0 * kRow), b = *reinterpret_cast<const float2*>(p0 + s1 * kRow);
        d.add_prod2(pack2(c0, c1), pack2(a.x, b.x), pack2(a.y, b.y));
    }
    // values with the sign bits of m (0 or 0x80000000) turned over, exactly
    static __device__ __forceinline__ f32x2 turned(f32x2 v, uint32_t m) { return v ^ (((f32x2)m << 32) | m); }
    __device__ __forceinline__ void add_signed(Dot2x2 (&d)[LN::NP], uint32_t slot, uint32_t m) const {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p0 + slot * kRow);
        d[0].accumulate(turned(v.x, m), turned(v.y, m));
        if constexpr (LN::NP == 2) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(p1 + slot * kRow);
            d[1].accumulate(turned(w.x, m), turned(w.y, m));
        }
    }
    __device__ __forceinline__ void add_both_signed(Dot2x2& d, uint32_t s0, uint32_t s1, uint32_t m0, uint32_t m1) const {
        const float2 a = *reinterpret_cast<const float2*>(p0 + s0 * kRow), b = *reinterpret_cast<const float2*>(p0 + s1 * kRow);
        const f32x2 m = ((f32x2)m1 << 32) | m0;
        d.accumulate(pack2(a.x, b.x) ^ m, pack2(a.y, b.y) ^ m);
    }
    // the lane's instances of row `slot`, v[k] instance inst(k)
    __device__ __forceinline__ void put(unsigned char* base, int slot, const float2 (&v)[LN::VV]) const {
        if constexpr (LN::VV == 1) {
            *reinterpret_cast<float2*>(base + slot * kRow) = v[0];
        } else {
            *reinterpret_cast<float4*>(base + slot * kRow + first * 8) = make_float4(v[0].x, v[1].x, v[0].y, v[1].y);
            if constexpr (LN::VV == 4)
                *reinterpret_cast<float4*>(base + slot * kRow + second * 8) = make_float4(v[2].x, v[3].x, v[2].y, v[3].y);
        }
    }
};

// FP32 basis: plain values, a lane's VV next to each other
template <int IC>
struct Staged<float, IC> {
    using LN = Lanes<IC>;
    static constexpr int kRow = IC * 4;
    int first;
    const unsigned char* p0;
    __device__ __forceinline__ Staged(const unsigned char* base, int j, int) : first(LN::VV * j), p0(base + LN::VV * j * 4) {}
    __device__ __forceinline__ int inst(int v) const { return first + v; }
    __device__ __forceinline__ void add(Dot2x2 (&d)[LN::NP], uint32_t slot, float c) const {
        const f32x2 cc = pack2(c, c);
        if constexpr (LN::NP == 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p0 + slot * kRow);
            d[0].add_prod(cc, v.x);
            d[1].add_prod(cc, v.y);
        } else {
            d[0].add_prod(cc, *reinterpret_cast<const f32x2*>(p0 + slot * kRow));
        }
    }
    __device__ __forceinline__ void add_both(Dot2x2& d, uint32_t s0, uint32_t s1, float c0, float c1) const {
        d.add_prod(pack2(c0, c1), pack2(*reinterpret_cast<const float*>(p0 + s0 * kRow), *reinterpret_cast<const float*>(p0 + s1 * kRow)));
    }
    __device__ __forceinline__ void put(unsigned char* base, int slot, const float (&v)[LN::VV]) const {
#pragma unroll
        for (int k = 0; k < LN::VV; ++k) *reinterpret_cast<float*>(base + slot * kRow + (first + k) * 4) = v[k];
    }
};

// A batch of one: the sums of the first and of the second entries
__device__ __forceinline__ Dot2 both_halves(const Dot2x2& a) {
    Dot2 d = a.half(0);
    d.merge(a.half(1));
    return d;
}

}  // namespace sgks
