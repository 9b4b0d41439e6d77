// Pieces shared by the compensated batched kernels (k_batchx.cu, k_tiles.cu): basis values in TW
// (float or float2) into Dot2 accumulators, and the rows of L and L^T L in float-float.
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

}  // namespace sgks
