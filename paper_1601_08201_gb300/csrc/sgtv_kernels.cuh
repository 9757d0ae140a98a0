// sgtv_kernels.cuh -- sm_103a kernels of one ADMM iteration of spectrally
// grouped TV reconstruction (Sec. III, Eqs. 5-7) and its FP64 reductions.
//
// Three launches per iteration:
//   k_forward      ybar_i = sum_j a_ij f_j + r_i, ratio_i = y_i / ybar_i   (Eq. 1; CSR)
//   k_back_update  e_j = sum_i a_ij ratio_i (CSC) and, in the same warp, the
//                  closed-form hyper-voxel update of Eq. 5 (EM surrogate +
//                  De Pierro split), writing f^{k+1} to a second buffer
//   k_shrink       v = w.G f^{k+1} + c^k, group soft-threshold per spatial bin
//                  (Eq. 6, grouping of Eq. 2), c^{k+1} = v - d^{k+1} (Eq. 7)
//
// Both sparse products are warp-per-row (warp-per-column) streams with
// coalesced, lane-strided index and value loads (see seg_dot) and gathers of
// the dense operand (f or ratio, both L2-resident) through the read-only path.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

#include <type_traits>

#include "sgtv_internal.h"

namespace sgtv {

// ---------------------------------------------------------------------------------------
// loads

__device__ __forceinline__ double to_f64(float v) { return double(v); }
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(__nv_bfloat16 v) { return double(__bfloat162float(v)); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Dot product of the sparse segment [start, end) of (idx, val) with the dense
// vector x, accumulated in T by one warp; every lane returns its partial.
// Lane k takes elements start + k, start + k + 32, ...: every index and value
// load is one fully coalesced 128-byte (64-byte for BF16) warp access, and one
// gather instruction touches the few cache lines that 32 consecutive nonzeros
// of a row (or column) fall in, instead of one line per lane. U loads of each
// array are issued before the first gather, so a warp keeps 32 * U indices
// and values in flight.
__device__ __forceinline__ int32_t ld_idx(const int32_t *p) { return __ldcs(p); }
__device__ __forceinline__ int32_t ld_idx(const uint16_t *p)
{
    return int32_t(__ldcs(reinterpret_cast<const unsigned short *>(p)));
}

// The dense operand: global memory through the read-only path, or a
// shared-memory tile (SX = true) staged by the tiled kernels.
template <bool SX, typename T>
__device__ __forceinline__ T ld_x(const T *x, int32_t c)
{
    if (SX) return x[c];
    return __ldg(x + c);
}
__device__ __forceinline__ float ld_val(const float *p) { return __ldcs(p); }
__device__ __forceinline__ double ld_val(const double *p) { return __ldcs(p); }
__device__ __forceinline__ float ld_val(const __nv_bfloat16 *p)
{
    return __uint_as_float(uint32_t(__ldcs(reinterpret_cast<const unsigned short *>(p))) << 16);
}

template <int U, typename T, typename V, typename IdxT = int32_t, bool SX = false>
__device__ __forceinline__ T seg_dot(int64_t start, int64_t end, const IdxT *__restrict__ idx,
                                     const V *__restrict__ val, const T *__restrict__ x, int lane)
{
    T acc = T(0);
    for (int64_t p = start + lane; p < end; p += 32 * U) {
        int32_t c[U];
        T v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t q = p + 32 * u;
            c[u] = 0;
            v[u] = T(0);
            if (q < end) {
                c[u] = ld_idx(idx + q);
                v[u] = T(ld_val(val + q));
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (p + 32 * u < end) acc = fma(v[u], ld_x<SX>(x, c[u]), acc);
    }
    return acc;
}

// Vector form of seg_dot for 16-bit local indices and a shared-memory dense
// operand: lane k loads 4 consecutive indices (8 bytes) and 4 consecutive
// values (16 bytes for FP32) from a 4-aligned position and masks the elements
// outside the segment; UV such 4-element chunks (128 elements per warp each)
// are in flight before the first gather. Each lane still adds its elements
// in increasing position order, but the partition of elements among lanes
// differs from seg_dot's, so the two forms round differently (both are
// deterministic).
__device__ __forceinline__ void ld_idx4(const uint16_t *p, int32_t (&c)[4])
{
    const uint2 u = __ldcs(reinterpret_cast<const uint2 *>(p));
    c[0] = int32_t(u.x & 0xFFFFu);
    c[1] = int32_t(u.x >> 16);
    c[2] = int32_t(u.y & 0xFFFFu);
    c[3] = int32_t(u.y >> 16);
}

__device__ __forceinline__ void ld_val4(const float *p, float (&v)[4])
{
    const float4 a = __ldcs(reinterpret_cast<const float4 *>(p));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}

__device__ __forceinline__ void ld_val4(const double *p, double (&v)[4])
{
    const double2 a = __ldcs(reinterpret_cast<const double2 *>(p));
    const double2 b = __ldcs(reinterpret_cast<const double2 *>(p + 2));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

__device__ __forceinline__ void ld_val4(const __nv_bfloat16 *p, float (&v)[4])
{
    const uint2 u = __ldcs(reinterpret_cast<const uint2 *>(p));
    v[0] = __uint_as_float(u.x << 16);
    v[1] = __uint_as_float(u.x & 0xFFFF0000u);
    v[2] = __uint_as_float(u.y << 16);
    v[3] = __uint_as_float(u.y & 0xFFFF0000u);
}

template <int UV, typename T, typename V>
__device__ __forceinline__ T seg_dot_v4(int64_t start, int64_t end, const uint16_t *__restrict__ idx,
                                        const V *__restrict__ val, const T *xs, int lane)
{
    T acc = T(0);
    for (int64_t p = (start & ~int64_t(3)) + 4 * lane; p < end; p += 128 * UV) {
        int32_t c[UV][4];
        T v[UV][4];
#pragma unroll
        for (int u = 0; u < UV; u++) {
            const int64_t q = p + 128 * u;
            if (q < end) {
                ld_idx4(idx + q, c[u]);
                ld_val4(val + q, v[u]);
            } else {
#pragma unroll
                for (int k = 0; k < 4; k++) { c[u][k] = 0; v[u][k] = T(0); }
            }
        }
#pragma unroll
        for (int u = 0; u < UV; u++)
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int64_t q = p + 128 * u + k;
                if (q >= start && q < end) acc = fma(v[u][k], xs[c[u][k]], acc);
            }
    }
    return acc;
}

template <int UV, typename T, typename V>
__device__ __forceinline__ T warp_segments_v4(const int64_t *__restrict__ ptr, int64_t seg0, int nseg,
                                              const uint16_t *__restrict__ idx, const V *__restrict__ val,
                                              const T *xs, int lane)
{
    const int64_t bound = (lane <= nseg) ? ptr[seg0 + lane] : 0;
    T mine = T(0);
#pragma unroll 1
    for (int k = 0; k < nseg; k++) {
        const int64_t s = __shfl_sync(0xffffffffu, bound, k);
        const int64_t e = __shfl_sync(0xffffffffu, bound, k + 1);
        const T acc = warp_sum(seg_dot_v4<UV, T, V>(s, e, idx, val, xs, lane));
        if (lane == k) mine = acc;
    }
    return mine;
}

// One warp reduces nseg (<= 31) consecutive segments (rows or columns)
// seg0 .. seg0+nseg-1 and lane k returns segment k's dot product. The segment
// bounds are loaded once, lane-parallel. With PIPE the first 32 * U indices and
// values of segment k+1 are loaded before segment k's gathers, so the warp has
// the next segment's stream in flight while it waits on the current gathers
// and reduction.
template <int U, typename T, typename V, typename IdxT>
__device__ __forceinline__ void load_chunk(int64_t p, int64_t end, const IdxT *__restrict__ idx,
                                           const V *__restrict__ val, int32_t (&c)[U], T (&v)[U])
{
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int64_t q = p + 32 * u;
        c[u] = 0;
        v[u] = T(0);
        if (q < end) {
            c[u] = ld_idx(idx + q);
            v[u] = T(ld_val(val + q));
        }
    }
}

template <int U, typename T, typename V, bool PIPE, typename IdxT = int32_t, bool SX = false>
__device__ __forceinline__ T warp_segments(const int64_t *__restrict__ ptr, int64_t seg0, int nseg,
                                           const IdxT *__restrict__ idx, const V *__restrict__ val,
                                           const T *__restrict__ x, int lane)
{
    const int64_t bound = (lane <= nseg) ? ptr[seg0 + lane] : 0;
    if (!PIPE) {  // one segment at a time, no prefetch
        T mine = T(0);
#pragma unroll 1
        for (int k = 0; k < nseg; k++) {
            const int64_t s = __shfl_sync(0xffffffffu, bound, k);
            const int64_t e = __shfl_sync(0xffffffffu, bound, k + 1);
            const T acc = warp_sum(seg_dot<U, T, V, IdxT, SX>(s, e, idx, val, x, lane));
            if (lane == k) mine = acc;
        }
        return mine;
    }
    int64_t s = __shfl_sync(0xffffffffu, bound, 0);
    int64_t e = __shfl_sync(0xffffffffu, bound, 1);
    int32_t c0[U];
    T v0[U];
    load_chunk<U, T, V, IdxT>(s + lane, e, idx, val, c0, v0);
    T mine = T(0);
#pragma unroll 1
    for (int k = 0; k < nseg; k++) {
        int32_t c1[U];
        T v1[U];
        int64_t s1 = 0, e1 = 0;
        if (k + 1 < nseg) {
            s1 = __shfl_sync(0xffffffffu, bound, k + 1);
            e1 = __shfl_sync(0xffffffffu, bound, k + 2);
            load_chunk<U, T, V, IdxT>(s1 + lane, e1, idx, val, c1, v1);
        } else {
#pragma unroll
            for (int u = 0; u < U; u++) { c1[u] = 0; v1[u] = T(0); }
        }
        T acc = T(0);
        const int64_t p0 = s + lane;
#pragma unroll
        for (int u = 0; u < U; u++)
            if (p0 + 32 * u < e) acc = fma(v0[u], ld_x<SX>(x, c0[u]), acc);
        if (s + 32 * U < e) acc += seg_dot<U, T, V, IdxT, SX>(s + 32 * U, e, idx, val, x, lane);
        acc = warp_sum(acc);
        if (lane == k) mine = acc;
#pragma unroll
        for (int u = 0; u < U; u++) { c0[u] = c1[u]; v0[u] = v1[u]; }
        s = s1;
        e = e1;
    }
    return mine;
}

// Same stream, summing the values only (column sums s = A^T 1).
template <typename T, typename V>
__device__ __forceinline__ T seg_sum(int64_t start, int64_t end, const V *__restrict__ val, int lane)
{
    T acc = T(0);
    for (int64_t p = start + lane; p < end; p += 32) acc += T(ld_val(val + p));
    return acc;
}

// ---------------------------------------------------------------------------------------
// a1: forward projection with the ratio epilogue (Eq. 1; EM surrogate input)

template <typename T, typename V, int RPW, int U, bool PIPE, int MINB>
__global__ void __launch_bounds__(256, MINB)
k_forward(int64_t I, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col,
          const V *__restrict__ val, const T *__restrict__ f, const T *__restrict__ r,
          int r_scalar, const T *__restrict__ y, T *__restrict__ ratio)
{
    const int lane = threadIdx.x & 31;
    const int64_t ntask = (I + RPW - 1) / RPW;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t t = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; t < ntask; t += nwarps) {
        const int64_t i0 = t * RPW;
        const int n = int(I - i0 < RPW ? I - i0 : RPW);
        const T acc = warp_segments<U, T, V, PIPE>(rowptr, i0, n, col, val, f, lane);
        const int64_t i = i0 + lane;
        if (lane < n) {
            const T yb = acc + (r_scalar ? r[0] : r[i]);
            const T yi = y[i];
            ratio[i] = (yi == T(0)) ? T(0) : yi / yb;
        }
    }
}

// ---------------------------------------------------------------------------------------
// a4: the closed-form hyper-voxel update (Eq. 5)
//
// Separable surrogate of Eq. 5's objective at f (all sums over directions p):
//   EM part (De Pierro's EM surrogate of the Poisson NLL): s_j t - f_j e_j log t
//   quadratic part: each term (a, p) of rho/2 (u_{a,p} - w_p (t_a - t_b))^2 with
//     b = nbr_p(a) inside the domain is split 1/2-1/2 around f, adding rho w^2 to
//     the t^2 coefficient alpha of both a and b and rho w (w (f_a + f_b) +- u)
//     (+ for a, - for b) to the -t coefficient gamma; a ghost term (b outside)
//     adds rho w^2 / 2 to alpha_a and rho w u to gamma_a.
// Voxel j meets the terms (j, p) and the terms (a, p) with a = j - step_p.
// Minimiser on t >= 0: the root of 2 alpha t^2 + (s - gamma) t - f e = 0.
template <typename T>
__device__ __forceinline__ T sgtv_root(T alpha, T B, T E, T s)
{
    if (alpha == T(0)) return (s > T(0)) ? E / s : T(0);
    T disc = sqrt(B * B + T(8) * alpha * E);
    if (B >= T(0)) {
        T den = B + disc;
        return (den > T(0)) ? T(2) * E / den : T(0);
    }
    return (-B + disc) / (T(4) * alpha);
}

// Scan holding hyper-voxel (or site) v: the last k with off[k] <= v.
__device__ __forceinline__ int scan_of(const int64_t *__restrict__ off, int nscans, int64_t v)
{
    int lo = 0, hi = nscans - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= v) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Position of hyper-voxel j inside its scan.
struct Loc {
    int32_t Nx, Nz, Nq, x, z;
    double rho, tau, beta;
    float rhof, tauf;
};

// The stencil weight w_p, the penalty rho and the threshold tau as operands
// of type T: FP32 values rounded once on the host (no per-element FP64-to-FP32
// conversion), FP64 values as given.
template <typename T> __device__ __forceinline__ T wgt(const Geom &g, int p);
template <> __device__ __forceinline__ float wgt<float>(const Geom &g, int p) { return g.wf[p]; }
template <> __device__ __forceinline__ double wgt<double>(const Geom &g, int p) { return g.w[p]; }
template <typename T> __device__ __forceinline__ T lrho(const Loc &L);
template <> __device__ __forceinline__ float lrho<float>(const Loc &L) { return L.rhof; }
template <> __device__ __forceinline__ double lrho<double>(const Loc &L) { return L.rho; }
template <typename T> __device__ __forceinline__ T ltau(const Loc &L);
template <> __device__ __forceinline__ float ltau<float>(const Loc &L) { return L.tauf; }
template <> __device__ __forceinline__ double ltau<double>(const Loc &L) { return L.tau; }

__device__ __forceinline__ Loc locate_voxel(const Geom &g, int64_t j)
{
    const Scan &sc = g.scans[scan_of(g.vox_off, g.nscans, j)];
    Loc L;
    L.Nx = sc.Nx;
    L.Nz = sc.Nz;
    L.Nq = sc.Nq;
    // J < 2^31 (checked at set-up): 32-bit unsigned divisions are exact
    const uint32_t site = uint32_t(j - sc.vox0) / uint32_t(sc.Nq);
    L.x = int32_t(site / uint32_t(sc.Nz));
    L.z = int32_t(site - uint32_t(L.x) * uint32_t(sc.Nz));
    L.rho = sc.rho;
    L.tau = sc.tau;
    L.beta = sc.beta;
    L.rhof = sc.rhof;
    L.tauf = sc.tauf;
    return L;
}

__device__ __forceinline__ bool inside(const Loc &L, int32_t x, int32_t z)
{
    return x >= 0 && x < L.Nx && z >= 0 && z < L.Nz;
}

__device__ __forceinline__ int64_t step_of(const Geom &g, const Loc &L, int p)
{
    return (int64_t(g.dx[p]) * L.Nz + g.dz[p]) * L.Nq;
}

// Each direction's neighbour loads sit behind its inside test (inside the fused
// backprojection faster than all loads first).
template <typename T>
__device__ __forceinline__ T voxel_update_at(const Geom &g, const Loc &L, int64_t j, T e, const T *__restrict__ s,
                                             const T *__restrict__ f, const T *__restrict__ d,
                                             const T *__restrict__ c)
{
    const T fj = f[j];
    T alpha = T(0), gamma = T(0);
#pragma unroll
    for (int p = 0; p < 4; p++) {
        if (p >= g.n_dirs) break;
        const int dx = g.dx[p], dz = g.dz[p];
        const T w = wgt<T>(g, p);
        const T w2 = w * w;
        const int64_t step = step_of(g, L, p);
        const int64_t pj = int64_t(p) * g.J + j;
        const T u_jp = d[pj] - c[pj];
        if (inside(L, L.x + dx, L.z + dz)) {
            alpha += w2;
            gamma += w * (w * (fj + f[j + step]) + u_jp);
        } else {
            alpha += T(0.5) * w2;
            gamma += w * u_jp;
        }
        if (inside(L, L.x - dx, L.z - dz)) {
            const T u_ap = d[pj - step] - c[pj - step];
            alpha += w2;
            gamma += w * (w * (f[j - step] + fj) - u_ap);
        }
    }
    const T rho = lrho<T>(L);
    alpha *= rho;
    gamma *= rho;
    const T sj = s[j];
    return sgtv_root<T>(alpha, sj - gamma, fj * e, sj);
}

template <typename T>
__device__ __forceinline__ T voxel_update(const Geom &g, int64_t j, T e, const T *__restrict__ s,
                                          const T *__restrict__ f, const T *__restrict__ d,
                                          const T *__restrict__ c)
{
    return voxel_update_at<T>(g, locate_voxel(g, j), j, e, s, f, d, c);
}

// a2 + a4: backprojection fused with the f-update. One warp owns CPW
// consecutive columns: it reduces each column's dot product in turn (lane k
// keeps column k's e, see warp_segments), then CPW lanes update their
// hyper-voxels side by side, so the epilogue's loads are coalesced across
// neighbouring q-bins.
template <typename T, typename V, int CPW, int U, bool PIPE, int MINB>
__global__ void __launch_bounds__(256, MINB)
k_back_update(Geom g, const int64_t *__restrict__ colptr, const int32_t *__restrict__ row,
              const V *__restrict__ val, const T *__restrict__ ratio, const T *__restrict__ s,
              const T *__restrict__ f, const T *__restrict__ d, const T *__restrict__ c,
              T *__restrict__ f_new)
{
    const int lane = threadIdx.x & 31;
    const int64_t ntask = (g.J + CPW - 1) / CPW;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t t = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; t < ntask; t += nwarps) {
        const int64_t j0 = t * CPW;
        const int n = int(g.J - j0 < CPW ? g.J - j0 : CPW);
        const T my_e = warp_segments<U, T, V, PIPE>(colptr, j0, n, row, val, ratio, lane);
        const int64_t j = j0 + lane;
        if (lane < n) f_new[j] = voxel_update<T>(g, j, my_e, s, f, d, c);
    }
}

// FP64 forms of both products with eight lanes per segment, so four segments
// side by side in a warp. The FP64 unit takes two lanes per clock, so what
// counts is FP64 warp instructions, and in a warp per segment the shuffle tree
// is five of them for as few as two multiply-adds. Here it is three for four
// segments. The tasks are small and each is one pass through its loads, so
// that a scan of a few thousand measurements reaches every multiprocessor.
// 13 x 7 x 37, 3001 measurements (1.7e5 nonzeros): forward 9.7 (the best of the
// tiled forms) -> 6.0 us, backprojection with f-update 14.3 -> 5.5 us; 64^3,
// 65,536 measurements (3.4e7 nonzeros) 120 -> 108 and 348 -> 239 us. The
// set-up's timing chooses among these and the tiled forms.
constexpr int kG8Threads = 64;  // eight segments a block

__device__ __forceinline__ double g8_sum(double v)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// This lane's part of a segment's dot product: every eighth nonzero, two sums
// in turn (a shorter chain), eight loads in flight.
template <typename V>
__device__ __forceinline__ double g8_dot(int64_t start, int64_t end, const int32_t *__restrict__ idx,
                                         const V *__restrict__ val, const double *__restrict__ x, int l)
{
    double a0 = 0.0, a1 = 0.0;
    for (int64_t p = start + l; p < end; p += 64) {
        int32_t c[8];
        double v[8], xv[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const bool in = p + 8 * u < end;
            c[u] = in ? ld_idx(idx + p + 8 * u) : 0;
            v[u] = in ? double(ld_val(val + p + 8 * u)) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; u++) xv[u] = p + 8 * u < end ? x[c[u]] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            if (p + 8 * u < end) a0 = fma(v[u], xv[u], a0);
            if (p + 8 * u + 8 < end) a1 = fma(v[u + 1], xv[u + 1], a1);
        }
    }
    return a0 + a1;
}

template <typename V>
__global__ void __launch_bounds__(kG8Threads)
k_forward_g8(int64_t I, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col,
             const V *__restrict__ val, const double *__restrict__ f, const double *__restrict__ r, int r_scalar,
             const double *__restrict__ y, double *__restrict__ ratio)
{
    const int l = threadIdx.x & 7;
    const int64_t i = int64_t(blockIdx.x) * (kG8Threads / 8) + (threadIdx.x >> 3);
    const bool in = i < I;
    const int64_t a = in ? rowptr[i] : 0, b = in ? rowptr[i + 1] : 0;
    const double yi = in ? y[i] : 0.0, ri = in ? (r_scalar ? r[0] : r[i]) : 1.0;
    const double yb = g8_sum(g8_dot<V>(a, b, col, val, f, l)) + ri;
    if (in && l == 0) ratio[i] = yi == 0.0 ? 0.0 : yi / yb;
}

// The f-update's four directions are dealt to the lanes too: lane l adds the
// forward (l even) or backward (l odd) term of direction l / 2 of Eq. 5, whose
// operands it loads before the dot product.
template <typename V>
__global__ void __launch_bounds__(kG8Threads)
k_back_update_g8(Geom g, const int64_t *__restrict__ colptr, const int32_t *__restrict__ row,
                 const V *__restrict__ val, const double *__restrict__ ratio, const double *__restrict__ s,
                 const double *__restrict__ f, const double *__restrict__ d, const double *__restrict__ c,
                 double *__restrict__ f_new)
{
    const int l = threadIdx.x & 7, p = l >> 1;
    const bool back = l & 1;
    const int64_t j = int64_t(blockIdx.x) * (kG8Threads / 8) + (threadIdx.x >> 3);
    const bool in = j < g.J;
    double fj = 0.0, sj = 0.0, rho = 0.0, fn = 0.0, up = 0.0, w = 0.0;
    bool inner = false;
    int64_t a = 0, b = 0;
    if (in) {
        a = colptr[j];
        b = colptr[j + 1];
        fj = f[j];
        sj = s[j];
        const Scan &sc = g.scans[g.nscans == 1 ? 0 : scan_of(g.vox_off, g.nscans, j)];
        const uint32_t v = uint32_t(j - sc.vox0);  // J < 2^31
        const uint32_t site = (__umulhi(sc.q_mul, v) + v) >> sc.q_shift;
        const int32_t x = int32_t((__umulhi(sc.z_mul, site) + site) >> sc.z_shift);
        const int32_t z = int32_t(site) - x * sc.Nz;
        rho = sc.rho;
        if (p < g.n_dirs) {
            const int32_t dx = back ? -g.dx[p] : g.dx[p], dz = back ? -g.dz[p] : g.dz[p];
            inner = x + dx >= 0 && x + dx < sc.Nx && z + dz >= 0 && z + dz < sc.Nz;
            const int64_t step = (int64_t(dx) * sc.Nz + dz) * sc.Nq;
            w = g.w[p];
            if (inner) fn = f[j + step];
            if (inner || !back) {
                const int64_t pj = int64_t(p) * g.J + j + (back ? step : 0);
                up = d[pj] - c[pj];
            }
        }
    }
    const double e = g8_sum(g8_dot<V>(a, b, row, val, ratio, l));
    const double w2 = w * w;
    const double alpha = rho * g8_sum(inner ? w2 : (back ? 0.0 : 0.5 * w2));
    const double gamma = rho * g8_sum(inner ? w * (w * (fj + fn) + (back ? -up : up)) : w * up);
    if (in && l == 0) f_new[j] = sgtv_root<double>(alpha, sj - gamma, fj * e, sj);
}

// Backprojection alone: out = A^T v (used by the KKT measure).
template <typename T, typename V>
__global__ void __launch_bounds__(256)
k_backproject(int64_t J, const int64_t *__restrict__ colptr, const int32_t *__restrict__ row,
              const V *__restrict__ val, const T *__restrict__ v, T *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t j = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; j < J; j += nwarps) {
        T acc = warp_sum(seg_dot<8, T, V>(colptr[j], colptr[j + 1], row, val, v, lane));
        if (lane == 0) out[j] = acc;
    }
}

// s_j = sum_i a_ij.
template <typename T, typename V>
__global__ void __launch_bounds__(256)
k_colsum(int64_t J, const int64_t *__restrict__ colptr, const V *__restrict__ val, T *__restrict__ s)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t j = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; j < J; j += nwarps) {
        T acc = warp_sum(seg_sum<T, V>(colptr[j], colptr[j + 1], val, lane));
        if (lane == 0) s[j] = acc;
    }
}

// ---------------------------------------------------------------------------------------
// a5 + a6: group shrink (Eq. 6) and dual update (Eq. 7), one warp per spatial bin.

template <typename T>
__device__ __forceinline__ T wgrad_at(const Geom &g, const Loc &L, const T *__restrict__ f, int64_t j, int p)
{
    const bool in = inside(L, L.x + g.dx[p], L.z + g.dz[p]);
    return wgt<T>(g, p) * (f[j] - (in ? f[j + step_of(g, L, p)] : T(0)));
}

// Site `site` (global) of its scan: geometry plus its first hyper-voxel.
__device__ __forceinline__ Loc locate_site(const Geom &g, int64_t site, int64_t &vox)
{
    const Scan &sc = g.scans[scan_of(g.site_off, g.nscans, site)];
    const int64_t ls = site - sc.site0;
    Loc L;
    L.Nx = sc.Nx;
    L.Nz = sc.Nz;
    L.Nq = sc.Nq;
    L.x = int32_t(uint32_t(ls) / uint32_t(sc.Nz));  // S < 2^31: exact in 32 bits
    L.z = int32_t(uint32_t(ls) - uint32_t(L.x) * uint32_t(sc.Nz));
    L.rho = sc.rho;
    L.tau = sc.tau;
    L.beta = sc.beta;
    L.rhof = sc.rhof;
    L.tauf = sc.tauf;
    vox = sc.vox0 + ls * sc.Nq;
    return L;
}

// Eqs. 6-7 for one spatial site, by one warp. QPL > 0: a site of at most
// 32 QPL q-bins keeps v = w.G f + c in registers between the group norm and
// the writes of d and c (the same arithmetic in the same order as the
// two-sweep form that recomputes v).
template <typename T, int QPL = 0>
__device__ __forceinline__ void shrink_site(const Geom &g, const T *__restrict__ f, T *__restrict__ d,
                                            T *__restrict__ c, int64_t site, int lane, int *__restrict__ flag,
                                            T *__restrict__ u = nullptr)
{
    int64_t v0;
    const Loc L = locate_site(g, site, v0);
    const T tau = ltau<T>(L);
    if (g.per_bin) {  // standard TV: each lane shrinks its own (site, q) groups over p
        for (int q = lane; q < L.Nq; q += 32) {
            const int64_t j = v0 + q;
            T v[4];
            T m2 = T(0);
#pragma unroll
            for (int p = 0; p < 4; p++) {
                v[p] = T(0);
                if (p < g.n_dirs) {
                    v[p] = wgrad_at(g, L, f, j, p) + c[int64_t(p) * g.J + j];
                    m2 = fma(v[p], v[p], m2);
                }
            }
            const T m = sqrt(m2);
            if (!isfinite(m)) atomicOr(flag, 1);
            T sc = (m > T(0)) ? T(1) - tau / m : T(0);
            sc = sc > T(0) ? sc : T(0);
#pragma unroll
            for (int p = 0; p < 4; p++) {
                if (p >= g.n_dirs) break;
                const int64_t pj = int64_t(p) * g.J + j;
                const T dv = sc * v[p];
                const T cv = v[p] - dv;
                d[pj] = dv;
                c[pj] = cv;
                if (u) u[pj] = dv - cv;
            }
        }
        return;
    }
    if (QPL > 0 && L.Nq <= 32 * QPL) {  // v stays in registers between the norm and the writes
        constexpr int QR = QPL > 0 ? QPL : 1;
        T v[QR][4];
        T n2 = T(0);
#pragma unroll
        for (int qq = 0; qq < QR; qq++) {
            const int q = lane + 32 * qq;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                v[qq][p] = T(0);
                if (q < L.Nq && p < g.n_dirs) {
                    const int64_t j = v0 + q;
                    v[qq][p] = wgrad_at(g, L, f, j, p) + c[int64_t(p) * g.J + j];
                    n2 = fma(v[qq][p], v[qq][p], n2);
                }
            }
        }
        n2 = warp_sum(n2);
        const T n = sqrt(n2);
        if (!isfinite(n)) {
            if (lane == 0) atomicOr(flag, 1);
        }
        T scale = (n > T(0)) ? T(1) - tau / n : T(0);
        scale = scale > T(0) ? scale : T(0);
#pragma unroll
        for (int qq = 0; qq < QR; qq++) {
            const int q = lane + 32 * qq;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                if (q < L.Nq && p < g.n_dirs) {
                    const int64_t pj = int64_t(p) * g.J + v0 + q;
                    const T dv = scale * v[qq][p];
                    const T cv = v[qq][p] - dv;
                    d[pj] = dv;
                    c[pj] = cv;
                    if (u) u[pj] = dv - cv;
                }
            }
        }
        return;
    }
    T n2 = T(0);
    for (int q = lane; q < L.Nq; q += 32) {
        const int64_t j = v0 + q;
#pragma unroll
        for (int p = 0; p < 4; p++) {
            if (p >= g.n_dirs) break;
            T v = wgrad_at(g, L, f, j, p) + c[int64_t(p) * g.J + j];
            n2 = fma(v, v, n2);
        }
    }
    n2 = warp_sum(n2);
    const T n = sqrt(n2);
    if (!isfinite(n)) {
        if (lane == 0) atomicOr(flag, 1);
    }
    T scale = (n > T(0)) ? T(1) - tau / n : T(0);
    scale = scale > T(0) ? scale : T(0);
    for (int q = lane; q < L.Nq; q += 32) {
        const int64_t j = v0 + q;
#pragma unroll
        for (int p = 0; p < 4; p++) {
            if (p >= g.n_dirs) break;
            const int64_t pj = int64_t(p) * g.J + j;
            T v = wgrad_at(g, L, f, j, p) + c[pj];
            T dv = scale * v;
            const T cv = v - dv;
            d[pj] = dv;
            c[pj] = cv;
            if (u) u[pj] = dv - cv;
        }
    }
}

// d is double-buffered: the shrink writes d^{k+1} into d_out (the buffer that
// held d^{k-1}) and leaves d^k in place for the dual residual.
template <typename T, int QPL>
__global__ void __launch_bounds__(256)
k_shrink(Geom g, const T *__restrict__ f, T *__restrict__ d_out, T *__restrict__ c, int *__restrict__ flag,
         T *__restrict__ u)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t site = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; site < g.S; site += nwarps)
        shrink_site<T, QPL>(g, f, d_out, c, site, lane, flag, u);
}

// Eqs. 6-7 under the group TV (Nq <= 32 QPL): the arithmetic of
// shrink_site's register form in the same order, hence the same bits, with
// less around it. ONE (a one-scan problem): the scan's shape, the direction
// offsets and the threshold are read once per thread, with no scan-table
// lookup. Otherwise (a batch) each site looks up its scan once. Either way a
// site's neighbour tests are made once per site, not per q-bin, and every
// operand of the site (f, its in-scan neighbours, c) is loaded before the
// first product, so each warp has all of them in flight together.
template <typename T, int QPL, bool ONE>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? (QPL >= 4 ? 3 : 4) : 1)  // FP32: 80 / 64 registers
k_shrink_lean(Geom g, const T *__restrict__ f, T *__restrict__ d_out, T *__restrict__ c, int *__restrict__ flag,
              T *__restrict__ u)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    const int64_t J = g.J;
    struct Shape {
        int32_t Nx, Nz, Nq;
        int64_t vox0, site0;
        T tau;
        int32_t step[4];
    };
    auto shape_of = [&](int sidx) {
        const Scan &sc = g.scans[sidx];
        Shape sh;
        sh.Nx = sc.Nx;
        sh.Nz = sc.Nz;
        sh.Nq = sc.Nq;
        sh.vox0 = sc.vox0;
        sh.site0 = sc.site0;
        Loc L0;
        L0.tau = sc.tau;
        L0.tauf = sc.tauf;
        sh.tau = ltau<T>(L0);
#pragma unroll
        for (int p = 0; p < 4; p++) sh.step[p] = (g.dx[p] * sh.Nz + g.dz[p]) * sh.Nq;  // |step| < J < 2^31
        return sh;
    };
    Shape one;
    if (ONE) one = shape_of(0);
    for (int64_t site = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; site < g.S; site += nwarps) {
        const Shape sh = ONE ? one : shape_of(scan_of(g.site_off, g.nscans, site));
        // S < 2^31 (checked at set-up): 32-bit unsigned divisions are exact
        const uint32_t ls = uint32_t(site - sh.site0);
        const int32_t x = int32_t(ls / uint32_t(sh.Nz));
        const int32_t z = int32_t(ls - uint32_t(x) * uint32_t(sh.Nz));
        const int64_t v0 = sh.vox0 + int64_t(ls) * sh.Nq;
        bool in[4];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int32_t xn = x + g.dx[p], zn = z + g.dz[p];
            in[p] = p < g.n_dirs && xn >= 0 && xn < sh.Nx && zn >= 0 && zn < sh.Nz;
        }
        T fj[QPL], fn[QPL][4], cj[QPL][4];
#pragma unroll
        for (int qq = 0; qq < QPL; qq++) {
            const int q = lane + 32 * qq;
            const int64_t j = v0 + q;
            if (q < sh.Nq) {
                fj[qq] = f[j];
#pragma unroll
                for (int p = 0; p < 4; p++) {
                    if (p < g.n_dirs) {
                        fn[qq][p] = in[p] ? f[j + sh.step[p]] : T(0);
                        cj[qq][p] = c[int64_t(p) * J + j];
                    }
                }
            }
        }
        T v[QPL][4];
        T n2 = T(0);
#pragma unroll
        for (int qq = 0; qq < QPL; qq++) {
            const int q = lane + 32 * qq;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                v[qq][p] = T(0);
                if (q < sh.Nq && p < g.n_dirs) {
                    v[qq][p] = wgt<T>(g, p) * (fj[qq] - fn[qq][p]) + cj[qq][p];
                    n2 = fma(v[qq][p], v[qq][p], n2);
                }
            }
        }
        n2 = warp_sum(n2);
        const T n = sqrt(n2);
        if (!isfinite(n)) {
            if (lane == 0) atomicOr(flag, 1);
        }
        T scale = (n > T(0)) ? T(1) - sh.tau / n : T(0);
        scale = scale > T(0) ? scale : T(0);
#pragma unroll
        for (int qq = 0; qq < QPL; qq++) {
            const int q = lane + 32 * qq;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                if (q < sh.Nq && p < g.n_dirs) {
                    const int64_t pj = int64_t(p) * J + v0 + q;
                    const T dv = scale * v[qq][p];
                    const T cv = v[qq][p] - dv;
                    d_out[pj] = dv;
                    c[pj] = cv;
                    if (u) u[pj] = dv - cv;
                }
            }
        }
    }
}

// out = a - b elementwise (u = d - c after a state set from outside).
template <typename T>
__global__ void k_sub(int64_t n, const T *__restrict__ a, const T *__restrict__ b, T *__restrict__ out)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x)
        out[k] = a[k] - b[k];
}

// Scaled dual consistent with the group shrink (Eq. 6) at a fixed point of
// Eqs. 6-7: there d = w.G f, and v = d + c must shrink back to d, which for a
// group with d_s != 0 forces c_s = tau * d_s / |d_s|; a group with d_s = 0 only
// needs |c_s| <= tau and gets 0. `theta` in [0, 1] scales the rule (0: c = 0).
template <typename T>
__global__ void __launch_bounds__(256)
k_dual_rule(Geom g, const T *__restrict__ d, T *__restrict__ c, double theta)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t site = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; site < g.S; site += nwarps) {
        int64_t v0;
        const Loc L = locate_site(g, site, v0);
        if (g.per_bin) {  // standard TV: groups (site, q)
            for (int q = lane; q < L.Nq; q += 32) {
                double m2 = 0.0;
                for (int p = 0; p < g.n_dirs; p++) {
                    const double v = double(d[int64_t(p) * g.J + v0 + q]);
                    m2 = fma(v, v, m2);
                }
                const double m = sqrt(m2);
                const double k = m > 0.0 ? theta * L.tau / m : 0.0;
                for (int p = 0; p < g.n_dirs; p++) {
                    const int64_t pj = int64_t(p) * g.J + v0 + q;
                    c[pj] = T(k * double(d[pj]));
                }
            }
            continue;
        }
        double n2 = 0.0;
        for (int q = lane; q < L.Nq; q += 32)
            for (int p = 0; p < g.n_dirs; p++) {
                const double v = double(d[int64_t(p) * g.J + v0 + q]);
                n2 = fma(v, v, n2);
            }
        n2 = warp_sum(n2);
        const double n = sqrt(n2);
        const double k = n > 0.0 ? theta * L.tau / n : 0.0;
        for (int q = lane; q < L.Nq; q += 32)
            for (int p = 0; p < g.n_dirs; p++) {
                const int64_t pj = int64_t(p) * g.J + v0 + q;
                c[pj] = T(k * double(d[pj]));
            }
    }
}

// d = w.G f (initial split variable).
template <typename T>
__global__ void k_wgrad(Geom g, const T *__restrict__ f, T *__restrict__ out)
{
    const int64_t n = g.J * g.n_dirs;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const int p = int(k / g.J);
        const int64_t j = k - int64_t(p) * g.J;
        const Loc L = locate_voxel(g, j);
        out[k] = wgrad_at(g, L, f, j, p);
    }
}

// out = num / den elementwise (0 where den = 0), as FP32: the normalised
// backprojection A^T y / A^T 1.
template <typename T>
__global__ void k_ratio_out(int64_t n, const T *__restrict__ num, const T *__restrict__ den, float *__restrict__ out)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const T dv = den[k];
        out[k] = dv > T(0) ? float(num[k] / dv) : 0.0f;
    }
}

// f = max(src, 0) from an FP32 image; flags a non-finite value (bit 0).
template <typename T>
__global__ void k_load_image(int64_t n, const float *__restrict__ src, T *__restrict__ f, int *__restrict__ flag)
{
    bool bad = false;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const float v = src[k];
        bad |= !isfinite(v);
        f[k] = T(v > 0.0f ? v : 0.0f);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

// a = src converted to T; a non-finite value sets flag bit 0.
template <typename T>
__global__ void k_load_vec(int64_t n, const float *__restrict__ src, T *__restrict__ a, int *__restrict__ flag)
{
    bool bad = false;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const float v = src[k];
        bad |= !isfinite(v);
        a[k] = T(v);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

template <typename T>
__global__ void k_fill(int64_t n, T *__restrict__ a, double val)
{
    const T v = T(val);
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x)
        a[k] = v;
}

// ---------------------------------------------------------------------------------------
// Tiled local-index (TLI) forms of the two sparse products.
//
// At set-up every tile of 64 consecutive rows (columns) gets 16-bit local
// indices into a per-tile staging buffer (see sgtv_tli.cu), in one of two
// forms chosen per tile:
//   window (wlen[t] > 0): the tile's index window [wbase[t], wbase[t] + wlen[t]),
//                  16-byte aligned; staged by one TMA bulk copy
//                  (cp.async.bulk, completion on an mbarrier)
//   list (wlen[t] == 0): the tile's sorted unique global indices
//                  uidx[uoff[t] .. uoff[t+1]); staged by a gather,
//                  x_s[k] = x[uidx[uoff[t] + k]]
// The stream then carries 2-byte indices instead of 4, and the gathers hit
// shared memory instead of the L1 data pipe.

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return uint32_t(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bulk prefetch into L2 of the bytes [a, b) of an array, widened to 16-byte
// bounds (the arrays are padded past their last element, so the widened
// range stays inside them). A hint only: no register or shared memory holds
// the data, and the later loads of the range hit L2 instead of waiting on
// HBM. One thread issues it for the whole block's tile at the block's start.
__device__ __forceinline__ void prefetch_l2(const void *base, int64_t a, int64_t b)
{
    a &= ~int64_t(15);
    b = (b + 15) & ~int64_t(15);
    if (b <= a) return;
    const char *p = static_cast<const char *>(base) + a;
    // evict-first: the stream is read once, and should not push the
    // iteration's resident vectors (f, d, c, s, e) out of L2
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    while (b > a) {  // one bulk prefetch moves at most 2^31 bytes here
        const int64_t n = (b - a) < (int64_t(1) << 31) ? (b - a) : (int64_t(1) << 31);
        asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(p), "r"(uint32_t(n)),
                     "l"(pol)
                     : "memory");
        p += n;
        a += n;
    }
}

// The index and value streams of segments [s0, s1) (positions ptr[s0] ..
// ptr[s1]) into L2.
template <typename IdxT, typename V>
__device__ __forceinline__ void prefetch_segments_l2(const int64_t *__restrict__ ptr, int64_t s0, int64_t s1,
                                                     const IdxT *idx, const V *val)
{
    const int64_t p0 = ptr[s0], p1 = ptr[s1];
    prefetch_l2(idx, p0 * int64_t(sizeof(IdxT)), p1 * int64_t(sizeof(IdxT)));
    prefetch_l2(val, p0 * int64_t(sizeof(V)), p1 * int64_t(sizeof(V)));
}

// Stage x[base .. base + n) into xs with one bulk copy; every thread returns
// true once the bytes have landed, false if the wait gave up (about 1 s),
// after a second bounded wait for the copy still in flight.
template <typename T>
__device__ __forceinline__ bool stage_window(T *xs, const T *x, int64_t base, int n, uint64_t *mbar)
{
    const uint32_t bar = smem_u32(mbar);
    const uint32_t bytes = uint32_t(n) * uint32_t(sizeof(T));
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (bytes == 0) return true;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(xs)), "l"(x + base), "r"(bytes), "r"(bar) : "memory");
    }
    const uint64_t t0 = global_ns();
    for (int pass = 0; pass < 2; pass++) {
        for (;;) {
            uint32_t done;
            asm volatile("{\n\t.reg .pred p;\n\t"
                         "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(bar) : "memory");
            if (done) return pass == 0;
            if (global_ns() - t0 > (pass == 0 ? 1000000000ull : 2000000000ull)) break;
        }
    }
    return false;
}

template <typename T>
__device__ __forceinline__ bool stage_tile(T *xs, const T *x, int64_t t, const int64_t *__restrict__ uoff,
                                           const int32_t *__restrict__ uidx, const int32_t *__restrict__ wbase,
                                           const int32_t *__restrict__ wlen, uint64_t *mbar)
{
    const int n = wlen[t];
    if (n == 0) {  // list form (block-uniform branch)
        const int64_t u0 = uoff[t];
        const int nu = int(uoff[t + 1] - u0);
        for (int k = threadIdx.x; k < nu; k += blockDim.x) xs[k] = __ldg(x + uidx[u0 + k]);
        __syncthreads();
        return true;
    }
    return stage_window<T>(xs, x, wbase[t], n, mbar);
}

struct TliTiles {
    const uint16_t *lidx;
    const int64_t *uoff;
    const int32_t *uidx;
    const int32_t *wbase;
    const int32_t *wlen;
};

template <typename T, typename V, int RPW, int U, bool PIPE, int UV = 0, int MINB = 1, bool L2PF = false>
__global__ void __launch_bounds__(256, MINB)
k_forward_tli(int64_t I, const int64_t *__restrict__ rowptr, TliTiles tl, const V *__restrict__ val,
              const T *__restrict__ f, const T *__restrict__ r, int r_scalar, const T *__restrict__ y,
              T *__restrict__ ratio, int *__restrict__ flag)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t mbar;
    T *xs = reinterpret_cast<T *>(smem_raw);
    const int64_t t = blockIdx.x;
    if (L2PF && threadIdx.x == 0)
        prefetch_segments_l2(rowptr, t * (8 * RPW), (t + 1) * (8 * RPW) < I ? (t + 1) * (8 * RPW) : I, tl.lidx, val);
    if (!stage_tile<T>(xs, f, t, tl.uoff, tl.uidx, tl.wbase, tl.wlen, &mbar)) {
        if (threadIdx.x == 0) atomicOr(flag, 2);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = t * (8 * RPW) + int64_t(warp) * RPW;
    if (i0 >= I) return;
    const int n = int(I - i0 < RPW ? I - i0 : RPW);
    const T acc = UV > 0 ? warp_segments_v4<(UV > 0 ? UV : 1), T, V>(rowptr, i0, n, tl.lidx, val, xs, lane)
                         : warp_segments<U, T, V, PIPE, uint16_t, true>(rowptr, i0, n, tl.lidx, val, xs, lane);
    const int64_t i = i0 + lane;
    if (lane < n) {
        const T yb = acc + (r_scalar ? r[0] : r[i]);
        const T yi = y[i];
        ratio[i] = (yi == T(0)) ? T(0) : yi / yb;
    }
}

template <typename T, typename V, int CPW, int U, bool PIPE, int UV = 0, int MINB = 1, bool L2PF = false>
__global__ void __launch_bounds__(256, MINB)
k_back_update_tli(Geom g, const int64_t *__restrict__ colptr, TliTiles tl, const V *__restrict__ val,
                  const T *__restrict__ ratio, const T *__restrict__ s, const T *__restrict__ f,
                  const T *__restrict__ d, const T *__restrict__ c, T *__restrict__ f_new,
                  int *__restrict__ flag)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t mbar;
    T *xs = reinterpret_cast<T *>(smem_raw);
    const int64_t t = blockIdx.x;
    if (L2PF && threadIdx.x == 0)
        prefetch_segments_l2(colptr, t * (8 * CPW), (t + 1) * (8 * CPW) < g.J ? (t + 1) * (8 * CPW) : g.J, tl.lidx,
                             val);
    if (!stage_tile<T>(xs, ratio, t, tl.uoff, tl.uidx, tl.wbase, tl.wlen, &mbar)) {
        if (threadIdx.x == 0) atomicOr(flag, 2);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = t * (8 * CPW) + int64_t(warp) * CPW;
    if (j0 >= g.J) return;
    const int n = int(g.J - j0 < CPW ? g.J - j0 : CPW);
    const T my_e = UV > 0 ? warp_segments_v4<(UV > 0 ? UV : 1), T, V>(colptr, j0, n, tl.lidx, val, xs, lane)
                          : warp_segments<U, T, V, PIPE, uint16_t, true>(colptr, j0, n, tl.lidx, val, xs, lane);
    const int64_t j = j0 + lane;
    if (lane < n) f_new[j] = voxel_update<T>(g, j, my_e, s, f, d, c);
}

// ---------------------------------------------------------------------------------------
// Single-pass form of a1 + a2: A is streamed once per surrogate step, by rows.
//
// e = A^T ratio needs ratio_i = y_i / (A f + r)_i, which is complete as soon as
// row i has been reduced; the row's nonzeros are then still in the warp's
// registers, so the warp scatters a_ij * ratio_i at once. The scatter goes to a
// shared-memory accumulator over the tile's staged columns (indexed by the
// same 16-bit local indices as the gather), and the block adds each touched
// column's partial to e with one global atomic add. The f-update then runs as
// an elementwise pass over e. Each lane adds its elements of a row in
// increasing position, as the lane-strided two-pass forward does, so ratio
// is bit-identical to it; e's sums are formed in an order set by the atomics,
// so this form is deterministic only up to rounding.

template <bool PRIV, typename T>
__device__ __forceinline__ void scatter_add(T *acc, int32_t c, T v)
{
    if (PRIV) acc[c] += v;
    else atomicAdd(acc + c, v);
}

// PRIV = false: one accumulator per block, shared-memory atomic adds.
// PRIV = true: one accumulator per warp (8 x the staging buffer), plain
// read-add-write (a row's columns are distinct, and a __syncwarp orders one
// row's updates before the next row's), summed over the warps in a fixed
// order before the global add; only the order of the global adds varies.
// KEEP = true: the first 32 U elements of a row stay in registers between the
// product and the scatter (longer rows are read again); KEEP = false: the
// scatter reads the row again (from L2, where the product's read left it),
// which keeps far fewer registers live and more warps resident.
template <typename T, typename V, int RPW, int U, bool PRIV, bool KEEP, int MINB>
__global__ void __launch_bounds__(256, MINB)
k_project_scatter_tli(int64_t I, int64_t J, const int64_t *__restrict__ rowptr, TliTiles tl,
                      const V *__restrict__ val, const T *__restrict__ f, const T *__restrict__ r, int r_scalar,
                      const T *__restrict__ y, int cap, T *__restrict__ e, int *__restrict__ flag)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t mbar;
    T *xs = reinterpret_cast<T *>(smem_raw);
    T *acc = xs + cap;
    const int64_t t = blockIdx.x;
    const int wl = tl.wlen[t];
    const int nstage = wl > 0 ? wl : int(tl.uoff[t + 1] - tl.uoff[t]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T *accw = PRIV ? acc + warp * cap : acc;
    if (PRIV) {
        for (int k = lane; k < nstage; k += 32) accw[k] = T(0);
    } else {
        for (int k = threadIdx.x; k < nstage; k += blockDim.x) acc[k] = T(0);
    }
    const bool staged = stage_tile<T>(xs, f, t, tl.uoff, tl.uidx, tl.wbase, tl.wlen, &mbar);
    if (!__syncthreads_and(staged)) {  // block-uniform exit
        if (threadIdx.x == 0) atomicOr(flag, 2);
        return;
    }
    const int64_t i0 = t * (8 * RPW) + int64_t(warp) * RPW;
    if (i0 < I) {
        const int n = int(I - i0 < RPW ? I - i0 : RPW);
        // the warp's rows: positions relative to their first nonzero (set-up
        // checks that RPW consecutive rows hold fewer than 2^31), counts and
        // backgrounds loaded lane-parallel up front so that no row waits on a
        // dependent global load
        const int64_t base = rowptr[i0];
        const uint16_t *__restrict__ li = tl.lidx + base;
        const V *__restrict__ va = val + base;
        const int bound = (lane <= n) ? int(rowptr[i0 + lane] - base) : 0;
        const T ylane = (lane < n) ? y[i0 + lane] : T(0);
        const T rlane = (lane < n) ? (r_scalar ? r[0] : r[i0 + lane]) : T(0);
#pragma unroll 1
        for (int k = 0; k < n; k++) {
            const int s0 = __shfl_sync(0xffffffffu, bound, k);
            const int s1 = __shfl_sync(0xffffffffu, bound, k + 1);
            const T yi = __shfl_sync(0xffffffffu, ylane, k);
            const T ri = __shfl_sync(0xffffffffu, rlane, k);
            if (KEEP) {
                int32_t c[U];
                T v[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int q = s0 + lane + 32 * u;
                    c[u] = 0;
                    v[u] = T(0);
                    if (q < s1) {
                        c[u] = ld_idx(li + q);
                        v[u] = T(ld_val(va + q));
                    }
                }
                T dot = T(0);
#pragma unroll
                for (int u = 0; u < U; u++)
                    if (s0 + lane + 32 * u < s1) dot = fma(v[u], xs[c[u]], dot);
                for (int p = s0 + lane + 32 * U; p < s1; p += 32)  // rows longer than 32 U
                    dot = fma(T(ld_val(va + p)), xs[ld_idx(li + p)], dot);
                dot = warp_sum(dot);
                if (yi != T(0)) {  // warp-uniform; a zero count scatters nothing
                    const T qr = yi / (dot + ri);
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (s0 + lane + 32 * u < s1) scatter_add<PRIV>(accw, c[u], v[u] * qr);
                    for (int p = s0 + lane + 32 * U; p < s1; p += 32)
                        scatter_add<PRIV>(accw, ld_idx(li + p), T(ld_val(va + p)) * qr);
                }
            } else {
                T dot = T(0);
                for (int p0 = s0 + lane; p0 < s1; p0 += 32 * U) {
                    int32_t c[U];
                    T v[U];
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const int q = p0 + 32 * u;
                        c[u] = 0;
                        v[u] = T(0);
                        if (q < s1) {
                            c[u] = ld_idx(li + q);
                            v[u] = T(ld_val(va + q));
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (p0 + 32 * u < s1) dot = fma(v[u], xs[c[u]], dot);
                }
                dot = warp_sum(dot);
                if (yi != T(0)) {
                    const T qr = yi / (dot + ri);
                    for (int p0 = s0 + lane; p0 < s1; p0 += 32 * U) {
                        int32_t c[U];
                        T v[U];
#pragma unroll
                        for (int u = 0; u < U; u++) {
                            const int q = p0 + 32 * u;
                            c[u] = 0;
                            v[u] = T(0);
                            if (q < s1) {
                                c[u] = int32_t(li[q]);
                                v[u] = T(va[q]);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; u++)
                            if (p0 + 32 * u < s1) scatter_add<PRIV>(accw, c[u], v[u] * qr);
                    }
                }
            }
            if (PRIV) __syncwarp();
        }
    }
    __syncthreads();
    const int64_t u0 = wl > 0 ? 0 : tl.uoff[t];
    const int64_t wb = wl > 0 ? tl.wbase[t] : 0;
    for (int k = threadIdx.x; k < nstage; k += blockDim.x) {
        T a = acc[k];
        if (PRIV) {
#pragma unroll
            for (int w = 1; w < 8; w++) a += acc[w * cap + k];
        }
        if (a != T(0)) {
            const int64_t col = wl > 0 ? wb + k : int64_t(tl.uidx[u0 + k]);
            if (col < J) atomicAdd(e + col, a);
        }
    }
}

// 4-wide form of the single-pass scatter: each lane loads 4 consecutive
// (16-bit index, value) pairs of a row from a 4-aligned position (8-byte and
// 16-byte loads, masked at the row's ends), UV such chunks (128 elements per
// warp each) in flight; the first UV chunks of a row stay in registers for
// the scatter, longer rows read the rest again. The product's element order
// is that of the 4-wide two-pass forward with the same UV, so ratio matches it
// bit for bit. PRIV as in k_project_scatter_tli.
template <typename T, typename V, int RPW, int UV, bool PRIV, int MINB, bool L2PF = false>
__global__ void __launch_bounds__(256, MINB)
k_project_scatter_tli_v4(int64_t I, int64_t J, const int64_t *__restrict__ rowptr, TliTiles tl,
                         const V *__restrict__ val, const T *__restrict__ f, const T *__restrict__ r,
                         int r_scalar, const T *__restrict__ y, int cap, T *__restrict__ e, int *__restrict__ flag)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t mbar;
    T *xs = reinterpret_cast<T *>(smem_raw);
    T *acc = xs + cap;
    const int64_t t = blockIdx.x;
    if (L2PF && threadIdx.x == 0)
        prefetch_segments_l2(rowptr, t * (8 * RPW), (t + 1) * (8 * RPW) < I ? (t + 1) * (8 * RPW) : I, tl.lidx, val);
    const int wl = tl.wlen[t];
    const int nstage = wl > 0 ? wl : int(tl.uoff[t + 1] - tl.uoff[t]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T *accw = PRIV ? acc + warp * cap : acc;
    if (PRIV) {
        for (int k = lane; k < nstage; k += 32) accw[k] = T(0);
    } else {
        for (int k = threadIdx.x; k < nstage; k += blockDim.x) acc[k] = T(0);
    }
    const bool staged = stage_tile<T>(xs, f, t, tl.uoff, tl.uidx, tl.wbase, tl.wlen, &mbar);
    if (!__syncthreads_and(staged)) {  // block-uniform exit
        if (threadIdx.x == 0) atomicOr(flag, 2);
        return;
    }
    const int64_t i0 = t * (8 * RPW) + int64_t(warp) * RPW;
    if (i0 < I) {
        const int n = int(I - i0 < RPW ? I - i0 : RPW);
        // positions relative to a 4-aligned base, so that aligned relative
        // positions are aligned addresses (set-up checks that RPW consecutive
        // rows hold fewer than 2^31 nonzeros)
        const int64_t base = rowptr[i0] & ~int64_t(3);
        const uint16_t *__restrict__ li = tl.lidx + base;
        const V *__restrict__ va = val + base;
        const int bound = (lane <= n) ? int(rowptr[i0 + lane] - base) : 0;
        const T ylane = (lane < n) ? y[i0 + lane] : T(0);
        const T rlane = (lane < n) ? (r_scalar ? r[0] : r[i0 + lane]) : T(0);
#pragma unroll 1
        for (int k = 0; k < n; k++) {
            const int s0 = __shfl_sync(0xffffffffu, bound, k);
            const int s1 = __shfl_sync(0xffffffffu, bound, k + 1);
            const T yi = __shfl_sync(0xffffffffu, ylane, k);
            const T ri = __shfl_sync(0xffffffffu, rlane, k);
            const int p0 = (s0 & ~3) + 4 * lane;
            int32_t c[UV][4];
            T v[UV][4];
#pragma unroll
            for (int u = 0; u < UV; u++) {
                const int q = p0 + 128 * u;
                if (q < s1) {
                    ld_idx4(li + q, c[u]);
                    ld_val4(va + q, v[u]);
                } else {
#pragma unroll
                    for (int m = 0; m < 4; m++) { c[u][m] = 0; v[u][m] = T(0); }
                }
            }
            T dot = T(0);
#pragma unroll
            for (int u = 0; u < UV; u++)
#pragma unroll
                for (int m = 0; m < 4; m++) {
                    const int q = p0 + 128 * u + m;
                    if (q >= s0 && q < s1) dot = fma(v[u][m], xs[c[u][m]], dot);
                }
            for (int p = p0 + 128 * UV; p < s1; p += 128 * UV) {  // rows longer than the kept chunks
#pragma unroll
                for (int u = 0; u < UV; u++) {
                    const int q = p + 128 * u;
                    if (q < s1) {
                        int32_t c2[4];
                        T v2[4];
                        ld_idx4(li + q, c2);
                        ld_val4(va + q, v2);
#pragma unroll
                        for (int m = 0; m < 4; m++)
                            if (q + m < s1) dot = fma(v2[m], xs[c2[m]], dot);
                    }
                }
            }
            dot = warp_sum(dot);
            if (yi != T(0)) {  // warp-uniform; a zero count scatters nothing
                const T qr = yi / (dot + ri);
#pragma unroll
                for (int u = 0; u < UV; u++)
#pragma unroll
                    for (int m = 0; m < 4; m++) {
                        const int q = p0 + 128 * u + m;
                        if (q >= s0 && q < s1) scatter_add<PRIV>(accw, c[u][m], v[u][m] * qr);
                    }
                for (int p = p0 + 128 * UV; p < s1; p += 128 * UV) {
#pragma unroll
                    for (int u = 0; u < UV; u++) {
                        const int q = p + 128 * u;
                        if (q < s1) {
                            int32_t c2[4];
                            T v2[4];
                            ld_idx4(li + q, c2);
                            ld_val4(va + q, v2);
#pragma unroll
                            for (int m = 0; m < 4; m++)
                                if (q + m < s1) scatter_add<PRIV>(accw, c2[m], v2[m] * qr);
                        }
                    }
                }
            }
            if (PRIV) __syncwarp();
        }
    }
    __syncthreads();
    const int64_t u0 = wl > 0 ? 0 : tl.uoff[t];
    const int64_t wb = wl > 0 ? tl.wbase[t] : 0;
    for (int k = threadIdx.x; k < nstage; k += blockDim.x) {
        T a = acc[k];
        if (PRIV) {
#pragma unroll
            for (int w = 1; w < 8; w++) a += acc[w * cap + k];
        }
        if (a != T(0)) {
            const int64_t col = wl > 0 ? wb + k : int64_t(tl.uidx[u0 + k]);
            if (col < J) atomicAdd(e + col, a);
        }
    }
}

// Single-pass scatter over the bank-dealt row stream (SpStream, built at
// set-up in sgtv_sp.cu): rows padded to multiples of 4 and 4-aligned, each
// lane holding whole 4-element chunks (position rp[i] + 128 u + 4 lane), so
// no element needs a position mask, and the elements of one access
// instruction spread over the shared-memory banks. The UV chunks of the next
// row are loaded into registers before the current row's gathers (PF), so a
// warp always has a row of the stream in flight while it reduces, divides and
// scatters the previous one. Rows longer than 128 UV elements read their
// further chunks in place. One accumulator per warp, as in the PRIV forms
// above; the padding slots gather the zeroed dummy entry xs[nstage] and add 0
// to the unflushed accumulator slot acc[nstage].
template <int UV, typename T>
struct SpRow {
    uint2 c[UV];    // 4 16-bit local indices per chunk
    T v[UV][4];
};

// ZERO = false leaves the chunks past the row's end unset: every use of a
// chunk is guarded by the same position test, so they are never read.
template <int UV, typename T, typename V, bool ZERO = true>
__device__ __forceinline__ void sp_load(SpRow<UV, T> &b, const uint16_t *__restrict__ li, const V *__restrict__ va,
                                        int s0, int n4, int lane)
{
    const uint16_t *__restrict__ lr = li + s0 + 4 * lane;
    const V *__restrict__ vr = va + s0 + 4 * lane;
#pragma unroll
    for (int u = 0; u < UV; u++) {
        if (128 * u + 4 * lane < n4) {
            b.c[u] = __ldcs(reinterpret_cast<const uint2 *>(lr + 128 * u));
            ld_val4(vr + 128 * u, b.v[u]);
        } else if (ZERO) {
            b.c[u] = make_uint2(0u, 0u);
#pragma unroll
            for (int m = 0; m < 4; m++) b.v[u][m] = T(0);
        }
    }
}

__device__ __forceinline__ int sp_idx(const uint2 &c, int m)
{
    const uint32_t w = (m < 2) ? c.x : c.y;
    return int((m & 1) ? (w >> 16) : (w & 0xFFFFu));
}

// Options of the row-stream scatter without register prefetch (bit flags):
// kSpBatch4: each 4-element chunk's accumulator entries are read before any
//   of them is written back (acc + a * ratio as one fused multiply-add).
//   Valid because a row's columns are distinct (only padding shares the
//   dummy slot, and adds 0); it keeps the compiler from ordering each
//   read-add-write behind the previous write, which it must assume may alias.
// kSpLean: the row's chunks past its end are not zero-filled.
constexpr int kSpBatch4 = 1, kSpLean = 2;

// One row: the dot product with the staged f (warp-reduced), then the ratio
// and the scatter into the warp's accumulator (PRIV) or the block's
// (shared-memory atomic adds).
template <int UV, typename T, typename V>
__device__ __forceinline__ T sp_dot(const SpRow<UV, T> &b, const uint16_t *__restrict__ li,
                                    const V *__restrict__ va, int s0, int n4, const T *xs, int lane)
{
    T dot = T(0);
#pragma unroll
    for (int u = 0; u < UV; u++)
        if (128 * u + 4 * lane < n4) {
#pragma unroll
            for (int m = 0; m < 4; m++) dot = fma(b.v[u][m], xs[sp_idx(b.c[u], m)], dot);
        }
    for (int p = 128 * UV + 4 * lane; p < n4; p += 128) {  // rows longer than the kept chunks
        int32_t c2[4];
        T v2[4];
        ld_idx4(li + s0 + p, c2);
        ld_val4(va + s0 + p, v2);
#pragma unroll
        for (int m = 0; m < 4; m++) dot = fma(v2[m], xs[c2[m]], dot);
    }
    return warp_sum(dot);
}

template <int UV, typename T, typename V, bool PRIV, int OPT = 0>
__device__ __forceinline__ void sp_scatter(const SpRow<UV, T> &b, const uint16_t *__restrict__ li,
                                           const V *__restrict__ va, int s0, int n4, T yi, T ri, T dot, T *accw,
                                           int lane)
{
    if (yi != T(0)) {  // warp-uniform; a zero count scatters nothing
        const T qr = yi / (dot + ri);
#pragma unroll
        for (int u = 0; u < UV; u++)
            if (128 * u + 4 * lane < n4) {
                if constexpr (PRIV && (OPT & kSpBatch4)) {
                    T a[4];
#pragma unroll
                    for (int m = 0; m < 4; m++) a[m] = accw[sp_idx(b.c[u], m)];
#pragma unroll
                    for (int m = 0; m < 4; m++) accw[sp_idx(b.c[u], m)] = fma(b.v[u][m], qr, a[m]);
                } else {
#pragma unroll
                    for (int m = 0; m < 4; m++) scatter_add<PRIV>(accw, sp_idx(b.c[u], m), b.v[u][m] * qr);
                }
            }
        for (int p = 128 * UV + 4 * lane; p < n4; p += 128) {
            int32_t c2[4];
            T v2[4];
            ld_idx4(li + s0 + p, c2);
            ld_val4(va + s0 + p, v2);
#pragma unroll
            for (int m = 0; m < 4; m++) scatter_add<PRIV>(accw, c2[m], v2[m] * qr);
        }
    }
    if (PRIV) __syncwarp();
}

template <int UV, typename T, typename V, bool PRIV>
__device__ __forceinline__ void sp_row(const SpRow<UV, T> &b, const uint16_t *__restrict__ li,
                                       const V *__restrict__ va, int s0, int n4, T yi, T ri, const T *xs, T *accw,
                                       int lane)
{
    const T dot = sp_dot<UV, T, V>(b, li, va, s0, n4, xs, lane);
    sp_scatter<UV, T, V, PRIV>(b, li, va, s0, n4, yi, ri, dot, accw, lane);
}

template <typename T, typename V, int UV, int MINB, bool L2PF = false, bool PRIV = true, bool PF = true,
          int OPT = 0>
__global__ void __launch_bounds__(256, MINB)
k_scatter_sp(int64_t I, int64_t J, const int64_t *__restrict__ rp, const uint16_t *__restrict__ li,
             const V *__restrict__ va, TliTiles tl, const T *__restrict__ f, const T *__restrict__ r, int r_scalar,
             const T *__restrict__ y, int cap, T *__restrict__ e, int *__restrict__ flag)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t mbar;
    T *xs = reinterpret_cast<T *>(smem_raw);
    T *acc = xs + cap;
    const int64_t t = blockIdx.x;
    if (L2PF && threadIdx.x == 0)
        prefetch_segments_l2(rp, t * kTliTile, (t + 1) * kTliTile < I ? (t + 1) * kTliTile : I, li, va);
    const int wl = tl.wlen[t];
    const int nstage = wl > 0 ? wl : int(tl.uoff[t + 1] - tl.uoff[t]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T *accw = PRIV ? acc + warp * cap : acc;
    // this thread's entries of a list tile's unique list (k = threadIdx.x + 256 m):
    // loaded once, for the staging gather and for the flush of the sums into e
    constexpr int kU = 3;
    const int64_t u0 = wl > 0 ? 0 : tl.uoff[t];
    int32_t ucol[kU];
#pragma unroll
    for (int m = 0; m < kU; m++) {
        const int k = threadIdx.x + 256 * m;
        ucol[m] = (wl == 0 && k < nstage) ? tl.uidx[u0 + k] : 0;
    }
    // the warp's rows, relative to their first slot (set-up checks that
    // kTliTile / 8 consecutive padded rows hold fewer than 2^31 slots); the
    // first row's chunks are loaded before the staging so that they overlap it
    const int64_t i0 = t * kTliTile + int64_t(warp) * (kTliTile / 8);
    const int n = i0 < I ? int(I - i0 < kTliTile / 8 ? I - i0 : kTliTile / 8) : 0;
    const int64_t base = n > 0 ? rp[i0] : 0;
    const uint16_t *__restrict__ lw = li + base;
    const V *__restrict__ vw = va + base;
    const int bound = (lane <= n && n > 0) ? int(rp[i0 + lane] - base) : 0;
    const T ylane = (lane < n) ? y[i0 + lane] : T(0);
    const T rlane = (lane < n) ? (r_scalar ? r[0] : r[i0 + lane]) : T(0);
    SpRow<UV, T> A, B;
    int a0 = __shfl_sync(0xffffffffu, bound, 0), a1 = __shfl_sync(0xffffffffu, bound, 1);
    if (n > 0) sp_load<UV, T, V, !(OPT & kSpLean)>(A, lw, vw, a0, a1 - a0, lane);
    if (PRIV) {
        for (int k = lane; k <= nstage; k += 32) accw[k] = T(0);  // with the dummy slot
    } else {
        for (int k = threadIdx.x; k <= nstage; k += blockDim.x) acc[k] = T(0);
    }
    bool staged = true;
    if (wl > 0) {  // window tile: one bulk copy (block-uniform branch)
        staged = stage_window<T>(xs, f, tl.wbase[t], wl, &mbar);
    } else {
#pragma unroll
        for (int m = 0; m < kU; m++) {
            const int k = threadIdx.x + 256 * m;
            if (k < nstage) xs[k] = __ldg(f + ucol[m]);
        }
        for (int k = threadIdx.x + 256 * kU; k < nstage; k += blockDim.x) xs[k] = __ldg(f + tl.uidx[u0 + k]);
    }
    if (threadIdx.x == 0) xs[nstage] = T(0);  // the padding slots' operand (outside the staged range)
    if (!__syncthreads_and(staged)) {  // block-uniform exit
        if (threadIdx.x == 0) atomicOr(flag, 2);
        return;
    }
    if (n > 0) {
        if (!PF) {  // one row at a time: the row's chunks loaded, then reduced and scattered
#pragma unroll 1
            for (int k = 0; k < n; k++) {
                const int s0 = __shfl_sync(0xffffffffu, bound, k), s1 = __shfl_sync(0xffffffffu, bound, k + 1);
                if (k > 0) sp_load<UV, T, V, !(OPT & kSpLean)>(A, lw, vw, s0, s1 - s0, lane);
                const T dot = sp_dot<UV, T, V>(A, lw, vw, s0, s1 - s0, xs, lane);
                sp_scatter<UV, T, V, PRIV, OPT>(A, lw, vw, s0, s1 - s0, __shfl_sync(0xffffffffu, ylane, k),
                                                __shfl_sync(0xffffffffu, rlane, k), dot, accw, lane);
            }
        }
#pragma unroll 1
        for (int k = 0; PF && k < n; k += 2) {
            // row k from A while row k + 1 streams into B
            const int b0 = a1, b1 = __shfl_sync(0xffffffffu, bound, (k + 2 <= n) ? k + 2 : n);
            if (k + 1 < n) sp_load<UV, T, V>(B, lw, vw, b0, b1 - b0, lane);
            sp_row<UV, T, V, PRIV>(A, lw, vw, a0, a1 - a0, __shfl_sync(0xffffffffu, ylane, k),
                                   __shfl_sync(0xffffffffu, rlane, k), xs, accw, lane);
            if (k + 1 >= n) break;
            // row k + 1 from B while row k + 2 streams into A
            a0 = b1;
            a1 = __shfl_sync(0xffffffffu, bound, (k + 3 <= n) ? k + 3 : n);
            if (k + 2 < n) sp_load<UV, T, V>(A, lw, vw, a0, a1 - a0, lane);
            sp_row<UV, T, V, PRIV>(B, lw, vw, b0, b1 - b0, __shfl_sync(0xffffffffu, ylane, k + 1),
                                   __shfl_sync(0xffffffffu, rlane, k + 1), xs, accw, lane);
        }
    }
    __syncthreads();
    const int64_t wb = wl > 0 ? tl.wbase[t] : 0;
    auto flush = [&](int k, int32_t ucolk) {
        T a = acc[k];
        if (PRIV) {
#pragma unroll
            for (int w = 1; w < 8; w++) a += acc[w * cap + k];
        }
        if (a != T(0)) {
            const int64_t col = wl > 0 ? wb + k : int64_t(ucolk);
            if (col < J) atomicAdd(e + col, a);
        }
    };
#pragma unroll
    for (int m = 0; m < kU; m++) {
        const int k = threadIdx.x + 256 * m;
        if (k < nstage) flush(k, ucol[m]);
    }
    for (int k = threadIdx.x + 256 * kU; k < nstage; k += blockDim.x) flush(k, wl > 0 ? 0 : tl.uidx[u0 + k]);
}

// The f-update (Eq. 5 closed form) from e and u = d - c as the shrink left it:
// a thread per hyper-voxel, B of them 256 apart, every load before any
// arithmetic, which is that of voxel_update_at in the same order. Voxels in
// storage order fill the lanes for any number of q-bins (a warp per site left
// half of them idle at 16 and went through its sites one after the other: 22 us
// at 16384 sites of 16 or 32 q-bins), and the place in the image costs two
// multiplications with the scan's precomputed divisors. The four neighbours'
// f serve both the forward and the backward terms: the directions are the
// library's own (+x, -x, +z, -z or +x, +z). Bound: the loads, from L2 as the
// shrink left them. A warp per site -> this form, us: 128 x 128 x 32 22.4 ->
// 6.5, 128 x 128 x 64 13.5 -> 10.2, 64^3 11.1 -> 7.0, 41 x 9 x 54 3.5 -> 2.1; a
// batch of uneven scans (5.3M voxels) 20.6 -> 14.2.
//
// PART = false: e is the accumulated vector, cleared here. PART = true: e holds
// partial sums (k_rows_stack), those of hyper-voxel j at poff[j] .. poff[j+1],
// added up in that order.
template <typename T>
__device__ __forceinline__ T sum_parts(const T *__restrict__ part, const int32_t *__restrict__ poff, int64_t j)
{
    T a = T(0);
    int k = poff[j];
    const int k1 = poff[j + 1];
    for (; k + 4 <= k1; k += 4) {  // four loads in flight, added in order
        const T v0 = part[k], v1 = part[k + 1], v2 = part[k + 2], v3 = part[k + 3];
        a = (((a + v0) + v1) + v2) + v3;
    }
    for (; k < k1; k++) a += part[k];
    return a;
}

template <typename T, int ND, int B, bool ONE, bool PART>
__global__ void __launch_bounds__(256)
k_fupdate(Geom g, T *__restrict__ e, const T *__restrict__ s, const T *__restrict__ f, const T *__restrict__ u,
          T *__restrict__ f_new, const int32_t *__restrict__ poff)
{
    const int64_t j0 = int64_t(blockIdx.x) * (256 * B) + threadIdx.x;
    T ej[B], fj[B], sj[B], fp[B], fm[B], fu[B], fd[B], uF[B][ND], uB[B][ND], rho[B];
    bool xp[B], xm[B], zp[B], zm[B];
#pragma unroll
    for (int b = 0; b < B; b++) {
        const int64_t j = j0 + 256 * b < g.J ? j0 + 256 * b : g.J - 1;  // past the end: the last voxel, not written
        const Scan &sc = g.scans[ONE ? 0 : scan_of(g.vox_off, g.nscans, j)];
        const uint32_t v = uint32_t(j - sc.vox0);  // J < 2^31
        const uint32_t site = (__umulhi(sc.q_mul, v) + v) >> sc.q_shift;
        const int32_t x = int32_t((__umulhi(sc.z_mul, site) + site) >> sc.z_shift);
        const int32_t z = int32_t(site) - x * sc.Nz;
        Loc L;
        L.rho = sc.rho;
        L.rhof = sc.rhof;
        rho[b] = lrho<T>(L);
        xp[b] = x + 1 < sc.Nx;
        xm[b] = x > 0;
        zp[b] = z + 1 < sc.Nz;
        zm[b] = z > 0;
        const int64_t sx = int64_t(sc.Nz) * sc.Nq, sz = sc.Nq;
        const int64_t up = xp[b] ? sx : 0, um = xm[b] ? sx : 0, vp = zp[b] ? sz : 0, vm = zm[b] ? sz : 0;
        ej[b] = PART ? sum_parts<T>(e, poff, j) : e[j];
        fj[b] = f[j];
        sj[b] = s[j];
        fp[b] = f[j + up];  // a ghost's operand is not used
        fm[b] = f[j - um];
        fu[b] = f[j + vp];
        fd[b] = f[j - vm];
#pragma unroll
        for (int p = 0; p < ND; p++) uF[b][p] = u[int64_t(p) * g.J + j];
        if (ND == 4) {
            uB[b][0] = u[j - um];
            uB[b][1] = u[g.J + j + up];
            uB[b][2] = u[2 * g.J + j - vm];
            uB[b][ND - 1] = u[3 * g.J + j + vp];
        } else {
            uB[b][0] = u[j - um];
            uB[b][1] = u[g.J + j - vm];
        }
    }
#pragma unroll
    for (int b = 0; b < B; b++) {
        const int64_t j = j0 + 256 * b;
        if (j >= g.J) break;
        if (!PART) e[j] = T(0);
        T alpha = T(0), gamma = T(0);
#pragma unroll
        for (int p = 0; p < ND; p++) {
            const T w = wgt<T>(g, p);
            const T w2 = w * w;
            const int d = ND == 4 ? p : 2 * p;  // direction: +x, -x, +z, -z
            const bool inF = d == 0 ? xp[b] : (d == 1 ? xm[b] : (d == 2 ? zp[b] : zm[b]));
            const bool inB = d == 0 ? xm[b] : (d == 1 ? xp[b] : (d == 2 ? zm[b] : zp[b]));
            const T fF = d == 0 ? fp[b] : (d == 1 ? fm[b] : (d == 2 ? fu[b] : fd[b]));
            const T fB = d == 0 ? fm[b] : (d == 1 ? fp[b] : (d == 2 ? fd[b] : fu[b]));
            if (inF) {
                alpha += w2;
                gamma += w * (w * (fj[b] + fF) + uF[b][p]);
            } else {
                alpha += T(0.5) * w2;
                gamma += w * uF[b][p];
            }
            if (inB) {
                alpha += w2;
                gamma += w * (w * (fB + fj[b]) - uB[b][p]);
            }
        }
        alpha *= rho[b];
        gamma *= rho[b];
        f_new[j] = sgtv_root<T>(alpha, sj[b] - gamma, fj[b] * ej[b], sj[b]);
    }
}

// ---------------------------------------------------------------------------------------
// TMA-streamed persistent forms of the two sparse products.
//
// One CTA per SM walks the tiles t = blockIdx.x, blockIdx.x + gridDim.x, ...
// through an NS-deep ring of shared-memory stages, with one producer warp and
// NW consumer warps. Filling a stage is one mbarrier phase of bulk copies
// (cp.async.bulk) issued by the producer: the tile's kTliTile + 2 segment
// pointers, its 16-bit local indices, its values, and either its index window
// of the dense operand or its unique-index list. A list tile then needs a
// gather of the dense operand into the stage, which the producer issues one
// tile behind its bulk copies as 4/8-byte cp.async copies completing on the
// stage's full barrier. Consumers compute from shared memory only and release
// the stage on its empty barrier; no block-wide barrier is taken in the loop,
// so warps drift freely and the HBM stream never waits on a computing warp.

struct TmaMat {
    const int64_t *ptr;      // segment pointers, padded to ntiles * kTliTile + 2 entries
    const uint16_t *lidx;    // local indices (padded past nnz)
    const int32_t *wbase, *wlen;
    const int64_t *uoff;
    const int32_t *uidx;     // padded past the last entry
    int64_t nseg, ntiles;
};

// Byte offsets of the regions of one stage (each 128-byte aligned).
struct TmaLayout {
    int off_lidx, off_val, off_uidx, off_xs, stage_bytes;
};

struct TileDesc {
    int64_t p0, p1, u0, u1;
    int32_t wb, wl;
};

__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *b, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *b)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(b)) : "memory");
}

// Bounded wait for the phase with the given parity: false once timeout_ns
// have passed since the first unsuccessful try.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, uint64_t timeout_ns)
{
    uint64_t t0 = 0;
    for (;;) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(smem_u32(b)), "r"(parity) : "memory");
        if (done) return true;
        const uint64_t now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > timeout_ns) return false;
    }
}

template <int BYTES>
__device__ __forceinline__ void cp_async_small(void *dst, const void *src)
{
    if (BYTES == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_arrive_noinc(uint64_t *b)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ uint32_t round16(int64_t bytes) { return uint32_t((bytes + 15) & ~int64_t(15)); }

template <typename T, typename V, int TS, int NS, int NW>
struct TmaPipe {
    static_assert(NS >= 3, "a tile's bulk copies need an iteration to land before its gathers");
    static_assert(TS % NW == 0, "whole segments per warp");
    static constexpr int VA = 16 / int(sizeof(V));   // value elements per 16 bytes
    static constexpr int SPW = TS / NW;              // segments per warp

    __device__ static TileDesc desc(const TmaMat &m, int64_t t)
    {
        TileDesc D;
        D.p0 = m.ptr[t * TS];
        D.p1 = m.ptr[t * TS + TS];
        D.u0 = m.uoff[t];
        D.u1 = m.uoff[t + 1];
        D.wb = m.wbase[t];
        D.wl = m.wlen[t];
        return D;
    }

    // Thread 0: one mbarrier phase of bulk copies filling stage sb with tile t.
    __device__ static void fill(const TmaMat &m, const TmaLayout &L, const V *val, const T *x, int64_t t,
                                const TileDesc &D, unsigned char *sb, uint64_t *tmab)
    {
        const uint32_t b_ptr = (TS + 2) * 8;
        const int64_t a0 = D.p0 & ~int64_t(7);
        const int64_t v0 = D.p0 & ~int64_t(VA - 1);
        const uint32_t b_lidx = D.p1 > D.p0 ? round16((D.p1 - a0) * 2) : 0u;
        const uint32_t b_val = D.p1 > D.p0 ? round16((D.p1 - v0) * int64_t(sizeof(V))) : 0u;
        const int64_t c0 = D.u0 & ~int64_t(3);
        const uint32_t b_u = (D.wl == 0 && D.u1 > D.u0) ? round16((D.u1 - c0) * 4) : 0u;
        const uint32_t b_w = D.wl > 0 ? uint32_t(D.wl) * uint32_t(sizeof(T)) : 0u;
        mbar_arrive_expect_tx(tmab, b_ptr + b_lidx + b_val + b_u + b_w);
        bulk_g2s(sb, m.ptr + t * TS, b_ptr, tmab);
        if (b_lidx) bulk_g2s(sb + L.off_lidx, m.lidx + a0, b_lidx, tmab);
        if (b_val) bulk_g2s(sb + L.off_val, val + v0, b_val, tmab);
        if (b_u) bulk_g2s(sb + L.off_uidx, m.uidx + c0, b_u, tmab);
        if (b_w) bulk_g2s(sb + L.off_xs, x + D.wb, b_w, tmab);
    }

    // Producer warp, after the stage's bulk copies landed: gather a list
    // tile's dense values with async copies, then every lane arrives on fullb
    // once its own copies complete.
    __device__ static void gather(const TileDesc &D, const T *x, unsigned char *sb, const TmaLayout &L,
                                  uint64_t *fullb, int lane)
    {
        if (D.wl == 0 && D.u1 > D.u0) {
            const int32_t *us = reinterpret_cast<const int32_t *>(sb + L.off_uidx) + (D.u0 & 3);
            T *xs = reinterpret_cast<T *>(sb + L.off_xs);
            const int n = int(D.u1 - D.u0);
            for (int k = lane; k < n; k += 32) cp_async_small<sizeof(T)>(xs + k, x + us[k]);
        }
        cp_async_arrive_noinc(fullb);
    }

    // Consumer warp: its SPW segments of the tile from shared memory; lane k
    // returns segment warp * SPW + k's dot product.
    __device__ static T compute(const TileDesc &D, const unsigned char *sb, const TmaLayout &L, int warp, int lane)
    {
        const int64_t *ps = reinterpret_cast<const int64_t *>(sb);
        const uint16_t *ls = reinterpret_cast<const uint16_t *>(sb + L.off_lidx);
        const V *vs = reinterpret_cast<const V *>(sb + L.off_val);
        const T *xs = reinterpret_cast<const T *>(sb + L.off_xs);
        const int64_t a0 = D.p0 & ~int64_t(7);
        const int64_t v0 = D.p0 & ~int64_t(VA - 1);
        T mine = T(0);
#pragma unroll
        for (int k = 0; k < SPW; k++) {
            const int sidx = warp * SPW + k;
            const int64_t st = ps[sidx], en = ps[sidx + 1];
            T acc = T(0);
            int64_t q = st + lane;
            for (; q + 96 < en; q += 128) {
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int64_t qq = q + 32 * u;
                    acc = fma(T(vs[qq - v0]), xs[ls[qq - a0]], acc);
                }
            }
            for (; q < en; q += 32) acc = fma(T(vs[q - v0]), xs[ls[q - a0]], acc);
            acc = warp_sum(acc);
            if (lane == k) mine = acc;
        }
        return mine;
    }

    // Warp-specialised persistent loop: warp NW is the producer (bulk copies of
    // tile k into stage k % NS once the consumers released it, then the list
    // gathers of tile k - 1), warps 0 .. NW-1 consume tiles in order and
    // release each stage on its empty barrier. epi(seg, value) runs on lane
    // k < SPW of each consumer warp for segment tile * TS + warp * SPW + k.
    template <typename Epi>
    __device__ static void run(const TmaMat &m, const TmaLayout &L, const V *val, const T *x, int *flag, Epi epi)
    {
        extern __shared__ __align__(128) unsigned char smem_raw[];
        __shared__ uint64_t tmab[NS], fullb[NS], emptyb[NS];
        __shared__ TileDesc sdesc[NS];
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        if (tid == 0) {
            for (int k = 0; k < NS; k++) {
                mbar_init(&tmab[k], 1);
                mbar_init(&fullb[k], 32);
                mbar_init(&emptyb[k], NW);
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncthreads();
        const int64_t t0 = blockIdx.x, step = gridDim.x;
        const int64_t n = m.ntiles > t0 ? (m.ntiles - t0 + step - 1) / step : 0;  // tiles of this CTA
        auto stage = [&](int64_t k) { return smem_raw + size_t(k % NS) * L.stage_bytes; };
        const uint64_t limit = 1000000000ull;  // 1 s per wait: far beyond any healthy copy
        bool bad = false;
        if (warp == NW) {
            TileDesc Dn{};
            if (lane == 0 && n > 0) Dn = desc(m, t0);
            int64_t filled = -1;
            for (int64_t k = 0; k <= n && !bad; k++) {
                if (k < n) {
                    const int s = int(k % NS);
                    if (k >= NS) bad |= !mbar_wait(&emptyb[s], uint32_t((k / NS - 1) & 1), limit);
                    if (!bad && lane == 0) {
                        sdesc[s] = Dn;
                        fill(m, L, val, x, t0 + k * step, Dn, stage(k), &tmab[s]);
                        if (k + 1 < n) Dn = desc(m, t0 + (k + 1) * step);
                    }
                    if (!bad) filled = k;
                    __syncwarp();
                }
                if (k >= 1 && !bad) {
                    const int s1 = int((k - 1) % NS);
                    bad |= !mbar_wait(&tmab[s1], uint32_t(((k - 1) / NS) & 1), limit);
                    if (!bad) gather(sdesc[s1], x, stage(k - 1), L, &fullb[s1], lane);
                }
                bad = __any_sync(0xffffffffu, bad);
            }
            cp_async_wait_all();
            if (bad) {
                if (lane == 0) {
                    atomicOr(flag, 2);
                    // the last fill may still be landing: one more bounded wait
                    if (filled >= 0) mbar_wait(&tmab[filled % NS], uint32_t((filled / NS) & 1), limit);
                }
            }
        } else {
            for (int64_t i = 0; i < n; i++) {
                const int s = int(i % NS);
                if (!mbar_wait(&fullb[s], uint32_t((i / NS) & 1), limit)) {
                    if (lane == 0) atomicOr(flag, 2);
                    break;
                }
                const TileDesc D = sdesc[s];
                const T v = compute(D, stage(i), L, warp, lane);
                const int64_t seg = (t0 + i * step) * TS + int64_t(warp) * SPW + lane;
                if (lane < SPW && seg < m.nseg) epi(seg, v);
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&emptyb[s])) : "memory");
            }
        }
    }
};

template <typename T, typename V, int NS, int NW>
__global__ void __launch_bounds__(32 * (NW + 1), 1)
k_forward_tma(TmaMat m, TmaLayout L, const V *__restrict__ val, const T *__restrict__ f,
              const T *__restrict__ r, int r_scalar, const T *__restrict__ y, T *__restrict__ ratio,
              int *__restrict__ flag)
{
    TmaPipe<T, V, kTliTile, NS, NW>::run(m, L, val, f, flag, [&](int64_t i, T acc) {
        const T yb = acc + (r_scalar ? r[0] : r[i]);
        const T yi = y[i];
        ratio[i] = (yi == T(0)) ? T(0) : yi / yb;
    });
}

template <typename T, typename V, int NS, int NW>
__global__ void __launch_bounds__(32 * (NW + 1), 1)
k_back_update_tma(TmaMat m, TmaLayout L, Geom g, const V *__restrict__ val, const T *__restrict__ ratio,
                  const T *__restrict__ s, const T *__restrict__ f, const T *__restrict__ d,
                  const T *__restrict__ c, T *__restrict__ f_new, int *__restrict__ flag)
{
    TmaPipe<T, V, kTliTile, NS, NW>::run(m, L, val, ratio, flag, [&](int64_t j, T e) {
        f_new[j] = voxel_update<T>(g, j, e, s, f, d, c);
    });
}

// ---------------------------------------------------------------------------------------
// The row pass over the stacked form (sgtv_stack.cu): a1 and a2 in one read
// of A, by one warp per tile.
//
// Each lane keeps its columns' f and sums of a_ij ratio_i in registers, so a
// nonzero costs neither a gather nor a scatter: per row and word a lane tests
// its bit, reads the next value of its stack from the ring if it is set, and
// two packed FP32 multiply-adds (one per word pair in the product, one in the
// sums) take two words at once; words without a nonzero add 0 times the image
// in the product and 0 times the ratio in the sums. That is 0 only for finite
// factors: an infinite ratio (a count where A f + r is 0, or y / ybar past FP32)
// or image value has to reach the row's own columns and no other. The loop does
// not look: a ratio that is not finite, which an image value that is not finite
// makes of every row of the tile with a count, leaves every sum of the tile
// infinite or NaN, so one sum a lane is looked at when the tile is done, and such
// a tile is done again over its nonzeros alone (stk_redo).
//
// The row stream it replaces as the first choice (k_scatter_sp) is bound by
// instruction issue: 12.4 warp instructions per 32 nonzeros for the gather,
// the accumulator's read and write and the index, and 134 per row. Here a row
// takes about 4.5 per word (32 columns) and about 45, and A is 4.1 + 0.5
// bytes per nonzero on the 2^28-nonzero problem (256 a row, 19 words) instead
// of 6. The measured times stand at the launcher (RowsStack).
//
// Ring: level l of the tile sits at place l mod ring; the first levels are
// repeated behind the end, so a lane's pointer is wrapped once per 8 words. One
// copy and one mbarrier phase per pair of rows, kStkAhead pairs ahead.
//
// PART = false: the sums go to e by global adds (single-pass form, order set
// by the adds). PART = true: ratio is written and each sum goes to its place
// among its column's partial sums, ordered by tile, which the f-update adds
// up in that order (two-pass form: deterministic).

// d = a * b + c on two packed FP32 lanes, each rounded as fmaf rounds.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t pack2(float x, float y)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &x, float &y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}

// If bit `bit` of mk is set: v = the value at the shared-memory address ptr, and
// ptr moves up one level; else v = 0 (what the load found there is dropped).
template <typename V>
__device__ __forceinline__ void stk_pop(float &v, uint32_t &ptr, uint32_t mk, uint32_t bit)
{
    if constexpr (sizeof(V) == 4) {
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t.reg .f32 x;\n\t"
                     "ld.shared.f32 x, [%1];\n\t"
                     "and.b32 t, %2, %3;\n\tsetp.ne.u32 p, t, 0;\n\t"
                     "@p add.u32 %1, %1, 128;\n\tselp.f32 %0, x, 0f00000000, p;\n\t}"
                     : "=f"(v), "+r"(ptr) : "r"(mk), "r"(bit));
    } else {
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t, x;\n\t.reg .b16 h;\n\t"
                     "ld.shared.b16 h, [%1];\n\t"
                     "and.b32 t, %2, %3;\n\tsetp.ne.u32 p, t, 0;\n\t"
                     "@p add.u32 %1, %1, 64;\n\tcvt.u32.u16 x, h;\n\tshl.b32 x, x, 16;\n\t"
                     "selp.b32 %0, x, 0, p;\n\t}"
                     : "=f"(v), "+r"(ptr) : "r"(mk), "r"(bit));
    }
}

// A lane's record of a pair of rows: both rows' bits and the first value's
// place in the ring (sgtv_stack.cu).
__device__ __forceinline__ void stk_split(uint32_t v, uint32_t &a, uint32_t &b, uint32_t &at)
{
    a = v;  // bits past the words are not looked at
    b = v >> 10;
    at = v >> 20;
}
__device__ __forceinline__ void stk_split(uint64_t v, uint32_t &a, uint32_t &b, uint32_t &at)
{
    a = uint32_t(v);
    b = uint32_t(v >> 24);
    at = uint32_t(v >> 48);
}

// One lane issues: the predicate keeps the warp converged.
__device__ __forceinline__ void mbar_expect_if(bool p, uint32_t bar, uint32_t bytes)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
                 "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}"
                 ::"r"(bar), "r"(bytes), "r"(int(p)) : "memory");
}
__device__ __forceinline__ void bulk_g2s_if(bool p, uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                 "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "r"(int(p)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}

// Tile t again, nonzero by nonzero from global memory, its sums in the ring's
// place (at least 2 W + kStkMirror levels of 32 V: room for W of 32 floats). Bound
// by the latency of its loads, kRedo words of them in flight, some
// 1.3 us a row of 20 words: a pass over 2^26 nonzeros takes 80 us, 164 where one
// tile is done again, 565 where all are.
template <typename V, typename M, int W, bool PART>
__device__ __forceinline__ void stk_redo(int64_t I, int64_t t, const StackMat &m, float *sum,
                                         const float *__restrict__ f, const float *__restrict__ r, int r_scalar,
                                         const float *__restrict__ y, float *__restrict__ out,
                                         float *__restrict__ ratio)
{
    static_assert((2 * W + kStkMirror) * sizeof(V) >= W * sizeof(float), "the sums are kept in the ring's place");
    static_assert(kStkMaxRows <= 64, "a lane per pair of rows");
    constexpr int kRedo = W % 5 == 0 ? 5 : (W % 6 == 0 ? 6 : (W % 4 == 0 ? 4 : 2));
    const int lane = threadIdx.x;
    const int64_t r0 = t * m.tr;
    const int n = int(I - r0 < m.tr ? I - r0 : m.tr);
    const V *__restrict__ val = static_cast<const V *>(m.val) + m.lvl[t] * 32;
    const M *__restrict__ rec = static_cast<const M *>(m.rec) + (r0 >> 1) * 32 + lane;
    const int32_t *__restrict__ cols = m.uidx + (t * W) * 32 + lane;
    const int32_t *__restrict__ dst = PART ? m.ppos + (t * W) * 32 + lane : cols;
    int top = 2 * lane < n ? int((m.ctl[(r0 >> 1) + lane] >> 7) & 63u) : 0;  // of pair `lane`: levels up to its last
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int below = __shfl_up_sync(0xffffffffu, top, o);
        if (lane >= o) top += below;
    }
    __syncwarp();
#pragma unroll 1
    for (int w = 0; w < W; w++) sum[32 * w + lane] = 0.f;
    M next = rec[0];
#pragma unroll 1
    for (int k = 0; k < n; k++) {
        const int first = __shfl_sync(0xffffffffu, top, k >> 1) - m.ring;  // the pair's values lie from here on
        const M now = next;
        if (k + 1 < n) next = rec[((k + 1) >> 1) * 32];
        const float yi = y[r0 + k], ri = r[r_scalar ? 0 : r0 + k];
        uint32_t a, b, at;
        stk_split(now, a, b, at);
        const uint32_t all = (1u << W) - 1u, mk = (k & 1 ? b : a) & all;
        const int place = int(at >> 5);
        const int level = first + ((place - first) % m.ring + m.ring) % m.ring + (k & 1 ? __popc(a & all) : 0);
        // a lane without values in the row reads the tile's first ones and drops them
        const V *__restrict__ v = val + (mk != 0u ? int64_t(level) * 32 + (at & 31u) : 0);
        float s = 0.f;
#pragma unroll 1
        for (int w0 = 0; w0 < W; w0 += kRedo) {
            float x[kRedo], z[kRedo];
#pragma unroll
            for (int u = 0; u < kRedo; u++) {
                const bool in = (mk >> (w0 + u)) & 1u;
                x[u] = float(v[in ? 32 * __popc(mk & ((1u << (w0 + u)) - 1u)) : 0]);
                z[u] = f[in ? cols[32 * (w0 + u)] : 0];
            }
#pragma unroll
            for (int u = 0; u < kRedo; u++)
                if ((mk >> (w0 + u)) & 1u) s = fmaf(x[u], z[u], s);
        }
        const float q = yi != 0.f ? yi / (warp_sum(s) + ri) : 0.f;
        if (PART && lane == 0) ratio[r0 + k] = q;
#pragma unroll 1
        for (int w0 = 0; w0 < W && q != 0.f; w0 += kRedo) {  // warp-uniform
            float x[kRedo], z[kRedo];
#pragma unroll
            for (int u = 0; u < kRedo; u++) {
                x[u] = float(v[(mk >> (w0 + u)) & 1u ? 32 * __popc(mk & ((1u << (w0 + u)) - 1u)) : 0]);
                z[u] = sum[32 * (w0 + u) + lane];
            }
#pragma unroll
            for (int u = 0; u < kRedo; u++)
                if ((mk >> (w0 + u)) & 1u) sum[32 * (w0 + u) + lane] = fmaf(x[u], q, z[u]);
        }
    }
#pragma unroll 1
    for (int w = 0; w < W; w++) {
        const int32_t to = dst[32 * w];
        const float a = sum[32 * w + lane];
        if (to < 0) continue;
        if (PART) out[to] = a;
        else if (a != 0.f) atomicAdd(out + to, a);
    }
}

template <typename V, int W, bool PART>
__global__ void __launch_bounds__(32, stk_resident(W, PART))
k_rows_stack(int64_t I, StackMat m, const float *__restrict__ f, const float *__restrict__ r, int r_scalar,
             const float *__restrict__ y, float *__restrict__ out, float *__restrict__ ratio, int *__restrict__ flag)
{
    using M = typename std::conditional<(W <= kStkShortWords), uint32_t, uint64_t>::type;
    constexpr uint32_t kLevel = 32 * uint32_t(sizeof(V));  // bytes of one level
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar[kStkAhead];
    const int lane = threadIdx.x;
    const int64_t t = blockIdx.x, r0 = t * m.tr;
    const int n = int(I - r0 < m.tr ? I - r0 : m.tr);
    const int np = (n + 1) >> 1;
    const uint32_t ring0 = smem_u32(smem_raw), ring_bytes = uint32_t(m.ring) * kLevel;
    const uint32_t ring_end = ring0 + ring_bytes, bar0 = smem_u32(bar);
    const uint32_t *__restrict__ cp = m.ctl + (r0 >> 1);
    const unsigned char *src = static_cast<const unsigned char *>(m.val) + m.lvl[t] * int64_t(kLevel);
    // the copy of one pair's levels (copy_code in sgtv_stack.cu), completing on `b`
    auto issue = [&](uint32_t c, uint32_t b) {
        const uint32_t a = (c & 127u) * kLevel, n1 = ((c >> 13) & 127u) * kLevel, n2 = ((c >> 20) & 63u) * kLevel;
        const bool over = (c >> 26) != 0u;
        mbar_expect_if(lane == 0, b, n1 + n2);
        bulk_g2s_if(lane == 0 && n1 != 0u, ring0 + a, src, n1, b);
        if (n2 != 0u)  // warp-uniform; every third pair or so
            bulk_g2s_if(lane == 0, over ? ring0 : ring_end + a, src + (over ? ring_bytes - a : 0u), n2, b);
        src += ((c >> 7) & 63u) * kLevel;
    };
    if (lane == 0) {
        for (int k = 0; k < kStkAhead; k++) mbar_init(&bar[k], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    for (int k = 0; k < kStkAhead && k < np; k++) issue(__ldg(cp + k), bar0 + 8 * k);

    const int32_t *__restrict__ cols = m.uidx + (t * W) * 32 + lane;
    uint64_t fv[W / 2], acc[W / 2];
#pragma unroll
    for (int w = 0; w < W / 2; w++) {
        const int32_t a = __ldg(cols + 64 * w), b = __ldg(cols + 64 * w + 32);
        fv[w] = pack2(a >= 0 ? __ldg(f + a) : 0.f, b >= 0 ? __ldg(f + b) : 0.f);
        acc[w] = 0;
    }
    const M *__restrict__ rp = static_cast<const M *>(m.rec) + (r0 >> 1) * 32 + lane;
    const float rs = r_scalar ? r[0] : 0.f;
    M rec = __ldcs(rp);
    uint32_t slot = 0, phase = 0;
    bool bad = false;
    auto landed = [&](uint32_t b, uint32_t ph) {  // false: not within 1 s, far beyond any healthy copy
        bool ok = mbar_try(b, ph);
        if (!ok) {
            const uint64_t t0 = global_ns();
            while (!(ok = mbar_try(b, ph)) && global_ns() - t0 < 1000000000ull) {}
        }
        return ok;
    };
#pragma unroll 1
    for (int g0 = 0; g0 < n && !bad; g0 += 32) {
        const int gn = n - g0 < 32 ? n - g0 : 32;
        const int64_t row = r0 + g0 + lane;
        const float yl = lane < gn ? y[row] : 0.f;
        const float rl = (!r_scalar && lane < gn) ? r[row] : 0.f;
        const int pc = (g0 >> 1) + kStkAhead + lane;  // the copies to issue in this group of rows
        const uint32_t cl = pc < np ? __ldcs(cp + pc) : 0u;
        float rat = 0.f;
#pragma unroll 1
        for (int k = 0; k < gn; k += 2) {  // two rows at a time (the second may be past the tile: no bits)
            uint32_t mka, mkb, ptr;
            stk_split(rec, mka, mkb, ptr);
            ptr = ring0 + ptr * uint32_t(sizeof(V));
            rp += 32;
            if (g0 + k + 2 < n) rec = __ldcs(rp);  // the next pair's, in flight
            if (!__all_sync(0xffffffffu, landed(bar0 + 8 * slot, phase))) {
                bad = true;
                break;
            }
            uint64_t va[W / 2], vb[W / 2], da0 = 0, da1 = 0, db0 = 0, db1 = 0;
#pragma unroll
            for (int w = 0; w < W; w += 2) {
                if ((w & 7) == 0) ptr = ptr >= ring_end ? ptr - ring_bytes : ptr;
                float x, z;
                stk_pop<V>(x, ptr, mka, 1u << w);
                stk_pop<V>(z, ptr, mka, 2u << w);
                va[w / 2] = pack2(x, z);
                if (w & 2) da1 = fma2(va[w / 2], fv[w / 2], da1);
                else da0 = fma2(va[w / 2], fv[w / 2], da0);
            }
#pragma unroll
            for (int w = 0; w < W; w += 2) {
                if ((w & 7) == 0) ptr = ptr >= ring_end ? ptr - ring_bytes : ptr;
                float x, z;
                stk_pop<V>(x, ptr, mkb, 1u << w);
                stk_pop<V>(z, ptr, mkb, 2u << w);
                vb[w / 2] = pack2(x, z);
                if (w & 2) db1 = fma2(vb[w / 2], fv[w / 2], db1);
                else db0 = fma2(vb[w / 2], fv[w / 2], db0);
            }
            // both products in one tree: the lower half-warp ends with row k's, the upper with row k + 1's
            float s0, s1, s2, s3;
            unpack2(da0, s0, s1);
            unpack2(da1, s2, s3);
            const float pa = (s0 + s1) + (s2 + s3);
            unpack2(db0, s0, s1);
            unpack2(db1, s2, s3);
            const float pb = (s0 + s1) + (s2 + s3);
            const bool up = lane >= 16;
            float dot = (up ? pb : pa) + __shfl_xor_sync(0xffffffffu, up ? pa : pb, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            const int kk = k + (up ? 1 : 0);
            const float yi = __shfl_sync(0xffffffffu, yl, kk);
            const float ri = r_scalar ? rs : __shfl_sync(0xffffffffu, rl, kk);
            const float q = yi != 0.f ? yi / (dot + ri) : 0.f;
            const float qa = __shfl_sync(0xffffffffu, q, 0), qb = __shfl_sync(0xffffffffu, q, 16);
            if (qa != 0.f) {  // warp-uniform; a zero count adds nothing
                const uint64_t q2 = pack2(qa, qa);
#pragma unroll
                for (int w = 0; w < W / 2; w++) acc[w] = fma2(va[w], q2, acc[w]);
            }
            if (qb != 0.f) {
                const uint64_t q2 = pack2(qb, qb);
#pragma unroll
                for (int w = 0; w < W / 2; w++) acc[w] = fma2(vb[w], q2, acc[w]);
            }
            if (PART) {
                if (lane == k) rat = qa;
                if (lane == k + 1) rat = qb;
            }
            // every lane has read its values (the sums needed them): the pair's barrier and the room
            // below are free for the copy kStkAhead pairs on
            const uint32_t c = __shfl_sync(0xffffffffu, cl, k >> 1);
            if ((g0 + k) / 2 + kStkAhead < np) issue(c, bar0 + 8 * slot);
            if (++slot == kStkAhead) {
                slot = 0;
                phase ^= 1;
            }
        }
        if (PART && lane < gn) ratio[row] = rat;
    }
    if (bad) {  // a copy never landed: record it, wait (bounded) for the ones in flight, leave
        if (lane == 0) atomicOr(flag, 2);
        for (int k = 0; k < kStkAhead; k++) {
            landed(bar0 + 8 * slot, phase);
            if (++slot == kStkAhead) {
                slot = 0;
                phase ^= 1;
            }
        }
        return;
    }
    uint32_t tile;  // read anew: no address is kept through the loop for what follows
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(tile));
    float sum0, sum1;
    unpack2(acc[0], sum0, sum1);
    if (__builtin_expect(__all_sync(0xffffffffu, sum0 <= FLT_MAX), 1)) {  // the sums are >= 0 or NaN
        const int32_t *__restrict__ dst = (PART ? m.ppos : m.uidx) + (int64_t(tile) * W) * 32 + lane;
#pragma unroll
        for (int w = 0; w < W / 2; w++) {
            float a, b;
            unpack2(acc[w], a, b);
            const int32_t ia = __ldg(dst + 64 * w), ib = __ldg(dst + 64 * w + 32);
            if (PART) {
                if (ia >= 0) out[ia] = a;
                if (ib >= 0) out[ib] = b;
            } else {
                if (ia >= 0 && a != 0.f) atomicAdd(out + ia, a);
                if (ib >= 0 && b != 0.f) atomicAdd(out + ib, b);
            }
        }
    } else {
        stk_redo<V, M, W, PART>(I, tile, m, reinterpret_cast<float *>(smem_raw), f, r, r_scalar, y, out, ratio);
    }
}

// ---------------------------------------------------------------------------------------
// One persistent (cooperative) launch per ADMM iteration: the three phases
// of sgtv_iterate -- tiled forward projection, tiled backprojection with the
// f-update, group shrink with the dual update -- separated by grid-wide
// barriers. Every block walks the tiles (then the sites) of each phase with a
// grid stride. Per segment the arithmetic is that of the tiled kernels, so
// results are identical to the three-launch path with the same tile forms.

// Grid-wide barrier (all blocks co-resident: cooperative launch). The last
// block to arrive resets the count and advances the generation; the others
// spin on the generation for at most bar->limit_ns (1 s unless the host set
// another bound; 0 gives up at the first unsuccessful look), then record a
// timeout and report false (the whole block learns it). No bulk copy of the
// block is in flight at a barrier, so a block that gives up may exit.
__device__ __forceinline__ bool grid_sync(GridBar *bar, int *flag)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned int *vgen = &bar->gen;
        const unsigned int gen = *vgen;
        const uint64_t limit = bar->limit_ns;
        __threadfence();
        if (atomicAdd(&bar->count, 1u) == gridDim.x - 1) {
            atomicExch(&bar->count, 0u);
            __threadfence();
            atomicAdd(&bar->gen, 1u);
        } else {
            const uint64_t t0 = global_ns();
            while (*vgen == gen) {
                if (global_ns() - t0 >= limit) {
                    ok = 0;
                    atomicOr(flag, 2);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

template <typename T, typename V, int UVF, int UVB, int MINB>
__global__ void __launch_bounds__(256, MINB)
k_iteration(int64_t I, const int64_t *__restrict__ rowptr, TliTiles tr, int64_t ntr, const V *__restrict__ rval,
            const T *__restrict__ r, int r_scalar, const T *__restrict__ y, T *__restrict__ ratio, Geom g,
            const int64_t *__restrict__ colptr, TliTiles tc, int64_t ntc, const V *__restrict__ cval,
            const T *__restrict__ s, const T *__restrict__ f, T *__restrict__ f_new, const T *__restrict__ d,
            T *__restrict__ d_out, T *__restrict__ c, int do_shrink, GridBar *bar, int *__restrict__ flag)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t mbar;
    T *xs = reinterpret_cast<T *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // phase 1: ybar, ratio (Eq. 1)
    for (int64_t t = blockIdx.x; t < ntr; t += gridDim.x) {
        __syncthreads();  // the previous tile's staging is no longer read
        if (!stage_tile<T>(xs, f, t, tr.uoff, tr.uidx, tr.wbase, tr.wlen, &mbar)) {
            if (threadIdx.x == 0) atomicOr(flag, 2);
            continue;
        }
        const int64_t i0 = t * kTliTile + int64_t(warp) * (kTliTile / 8);
        if (i0 < I) {
            const int n = int(I - i0 < kTliTile / 8 ? I - i0 : kTliTile / 8);
            const T acc = UVF > 0 ? warp_segments_v4<(UVF > 0 ? UVF : 1), T, V>(rowptr, i0, n, tr.lidx, rval, xs, lane)
                                  : warp_segments<8, T, V, false, uint16_t, true>(rowptr, i0, n, tr.lidx, rval, xs, lane);
            const int64_t i = i0 + lane;
            if (lane < n) {
                const T yb = acc + (r_scalar ? r[0] : r[i]);
                const T yi = y[i];
                ratio[i] = (yi == T(0)) ? T(0) : yi / yb;
            }
        }
    }
    if (!grid_sync(bar, flag)) return;
    // phase 2: e = A^T ratio and the closed-form f-update (Eq. 5)
    for (int64_t t = blockIdx.x; t < ntc; t += gridDim.x) {
        __syncthreads();
        if (!stage_tile<T>(xs, ratio, t, tc.uoff, tc.uidx, tc.wbase, tc.wlen, &mbar)) {
            if (threadIdx.x == 0) atomicOr(flag, 2);
            continue;
        }
        const int64_t j0 = t * kTliTile + int64_t(warp) * (kTliTile / 8);
        if (j0 < g.J) {
            const int n = int(g.J - j0 < kTliTile / 8 ? g.J - j0 : kTliTile / 8);
            const T e = UVB > 0 ? warp_segments_v4<(UVB > 0 ? UVB : 1), T, V>(colptr, j0, n, tc.lidx, cval, xs, lane)
                                : warp_segments<8, T, V, false, uint16_t, true>(colptr, j0, n, tc.lidx, cval, xs, lane);
            const int64_t j = j0 + lane;
            if (lane < n) f_new[j] = voxel_update<T>(g, j, e, s, f, d, c);
        }
    }
    if (!do_shrink) return;
    if (!grid_sync(bar, flag)) return;
    // phase 3: group shrink and dual update (Eqs. 6-7)
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t site = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; site < g.S; site += nwarps)
        shrink_site(g, f_new, d_out, c, site, lane, flag);
}

// ---------------------------------------------------------------------------------------
// FP64 reductions. Each block writes one partial per field to `part`
// (field-major: part[field * nblocks + block]); k_finalize then reduces the
// partials of every field in a fixed order, so results do not depend on timing.

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sum (or max) over the block of one value per thread; result valid in thread 0.
template <bool MAX>
__device__ __forceinline__ double block_reduce(double v, double *sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = MAX ? warp_max_d(v) : warp_sum_d(v);
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (lane < nw) ? sh[lane] : (MAX ? -1.0 : 0.0);
        v = MAX ? warp_max_d(v) : warp_sum_d(v);
    }
    return v;
}

// One measurement's deviance term, yb - y + y log(y / yb) with 0 log 0 = 0.
__device__ __forceinline__ double dev_term(double yb, double yi)
{
    double t = yb - yi;
    if (yi > 0.0) t += yi * log(yi / yb);
    return t;
}

// acc += N of a lane's products, 32 nonzeros apart from p on.
template <int N, typename T, typename V>
__device__ __forceinline__ void dev_chunk(const V *__restrict__ val, const T *__restrict__ f,
                                          const int32_t *__restrict__ col, int64_t p, double &acc)
{
    V v[N];
    T x[N];
#pragma unroll
    for (int u = 0; u < N; u++) {
        v[u] = val[p + 32 * u];
        x[u] = f[col[p + 32 * u]];
    }
#pragma unroll
    for (int u = 0; u < N; u++) acc = fma(to_f64(v[u]), double(x[u]), acc);
}

// Deviance partials over the measurements [i0, i1), from the plain CSR form
// (matrices without tiles, tiles whose staging would fill an SM, few rows): ybar
// accumulated in FP64 from the stored A values and f. A warp takes R rows (at
// most 32) in turn, lane k keeps row k's ybar, and their terms (a
// division and a logarithm in FP64, which cost a warp the same for one lane as
// for 32) are formed side by side.
template <typename T, typename V>
__global__ void __launch_bounds__(256)
k_dev_partials(int64_t i0, int64_t i1, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col,
               const V *__restrict__ val, const T *__restrict__ f, const T *__restrict__ r,
               int r_scalar, const T *__restrict__ y, int R, double *__restrict__ part)
{
    __shared__ double sh[32];
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    double mine = 0.0;
    // tasks are dealt to the blocks in turn, so that few rows have an FP64 unit each
    for (int64_t k0 = i0 + R * (int64_t(threadIdx.x >> 5) * gridDim.x + blockIdx.x); k0 < i1; k0 += R * nwarps) {
        const int n = int(i1 - k0 < R ? i1 - k0 : R);
        double yb = 0.0;
        for (int k = 0; k < n; k++) {
            double acc = 0.0;
            const int64_t start = rowptr[k0 + k], end = rowptr[k0 + k + 1];
            int64_t p = start + lane;
            // loads ahead, eight of them in the long rows; added in order
            for (; p + 224 < end; p += 256) dev_chunk<8>(val, f, col, p, acc);
            for (; p + 96 < end; p += 128) dev_chunk<4>(val, f, col, p, acc);
            for (; p < end; p += 32) dev_chunk<1>(val, f, col, p, acc);
            acc = warp_sum_d(acc);
            if (lane == k) yb = acc;
        }
        if (lane < n) mine += dev_term(yb + double(r_scalar ? r[0] : r[k0 + lane]), double(y[k0 + lane]));
    }
    double tot = block_reduce<false>(mine, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// The same from the tiled form (16-bit local indices), T = double: a block takes
// tiles blockIdx.x, + gridDim.x, ... that meet [i0, i1), stages the tile's f in
// shared memory, and each warp forms 8 rows' products with one FP64
// multiply-add per nonzero and no other FP64 work in the loop. The lanes' sums
// are folded by all 256 threads (a warp-wide tree would take 5 FP64 additions
// per row and lane, as much again as 5/8 of the products), and the 64 terms
// are formed by 64 threads side by side. The lanes take consecutive elements
// because an FP64 instruction costs a warp the same for any number of active
// lanes. Bound: the FP64 unit, about 2 lanes per clock and SM.
template <typename T>
__global__ void __launch_bounds__(256, 4)
k_dev_partials_tli(int64_t i0, int64_t i1, int64_t ntiles, const int64_t *__restrict__ rowptr, TliTiles tl,
                   const T *__restrict__ val, const T *__restrict__ f, const T *__restrict__ r, int r_scalar,
                   const T *__restrict__ y, double *__restrict__ part)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double rows[kTliTile][33];
    __shared__ double sh[32];
    T *xs = reinterpret_cast<T *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int R = kTliTile / 8;
    double mine = 0.0;
    for (int64_t t = i0 / kTliTile + blockIdx.x; t < ntiles && t * kTliTile < i1; t += gridDim.x) {
        const int64_t t0 = t * kTliTile, t1 = t0 + kTliTile < i1 ? t0 + kTliTile : i1;
        if (threadIdx.x == 0) prefetch_segments_l2(rowptr, t0, t1, tl.lidx, val);
        const int wl = tl.wlen[t];
        const int64_t u0 = tl.uoff[t];
        const int nstage = wl > 0 ? wl : int(tl.uoff[t + 1] - u0);
        const int64_t wb = tl.wbase[t];
        for (int k = threadIdx.x; k < nstage; k += blockDim.x)
            xs[k] = f[wl > 0 ? wb + k : int64_t(tl.uidx[u0 + k])];
        __syncthreads();
        const int64_t w0 = t0 + warp * R;
        const int n = w0 < t1 ? int(t1 - w0 < R ? t1 - w0 : R) : 0;
        const int64_t bound = lane <= n && n > 0 ? rowptr[w0 + lane] : 0;
#pragma unroll 1
        for (int k = 0; k < n; k++) {
            const int64_t s = __shfl_sync(0xffffffffu, bound, k), e = __shfl_sync(0xffffffffu, bound, k + 1);
            double a0 = 0.0, a1 = 0.0;
            const int n_el = int(e - s);  // a row holds at most J < 2^31 nonzeros
            const uint16_t *__restrict__ li = tl.lidx + s;
            const T *__restrict__ va = val + s;
            for (int p = 0; p < n_el; p += 256) {
                int32_t c[8];
                T v[8];
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    c[u] = 0;
                    v[u] = 0.0;
                    if (p + 32 * u + lane < n_el) {
                        c[u] = ld_idx(li + p + 32 * u + lane);
                        v[u] = ld_val(va + p + 32 * u + lane);
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; u++)
                    if (p + 32 * u < n_el) {  // warp-uniform: no FP64 instruction past the row's end
                        double &a = (u & 1) ? a1 : a0;
                        if (p + 32 * u + lane < n_el) a = fma(v[u], xs[c[u]], a);
                    }
            }
            rows[warp * R + k][lane] = a0 + a1;
        }
        __syncthreads();
        // 4 threads per row: 8 lanes' sums each, then the quad's total in every thread of it
        const int rr = threadIdx.x >> 2, qd = threadIdx.x & 3;
        double yb = 0.0;
#pragma unroll
        for (int m = 0; m < 8; m++) yb += rows[rr][qd + 4 * m];
        yb += __shfl_xor_sync(0xffffffffu, yb, 1);
        yb += __shfl_xor_sync(0xffffffffu, yb, 2);
        __syncthreads();
        if (qd == 0) rows[rr][0] = yb;
        __syncthreads();
        const int64_t i = t0 + threadIdx.x;
        if (threadIdx.x < kTliTile && i >= i0 && i < t1)
            mine += dev_term(rows[threadIdx.x][0] + double(r_scalar ? r[0] : r[i]), double(y[i]));
        __syncthreads();  // rows and xs are rewritten by the next tile
    }
    double tot = block_reduce<false>(mine, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// Packed FP32 sums with their rounding errors (Knuth's two-sum): hi + lo is the
// exact sum, on each half.
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b)
{
    return fma2(b, pack2(-1.f, -1.f), a);  // exact product: rounds as a - b
}
__device__ __forceinline__ uint64_t two_sum2(uint64_t a, uint64_t b, uint64_t &lo)
{
    const uint64_t t = add2(a, b), bb = sub2(t, a);
    lo = add2(sub2(a, sub2(t, bb)), sub2(b, bb));
    return t;
}
__device__ __forceinline__ float two_sum(float a, float b, float &lo)
{
    const float t = __fadd_rn(a, b), bb = __fsub_rn(t, a);
    lo = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bb)), __fsub_rn(b, bb));
    return t;
}

// The same for FP32 images, without the FP64 unit in the loop: a product is
// the exact sum of two FP32 numbers (a multiplication and a multiply-add), and
// a row's sum three FP32 numbers, each taking the rounding errors of the one
// before; what is lost is about 2^-70 of it, where a chain of FP64 sums loses
// 2^-53 per step. Two rows at a time, one in each half of the packed
// instructions: 23 of them for two products, at 64 times the FP64 unit's rate.
// A row for which that may not be so (a product that overflows FP32, or may have
// underflowed next to a ybar as small) is summed again in FP64. Bound:
// issue in the loop (2^28 nonzeros: 0.2 ms) and the 64 divisions and logarithms
// a tile, which are FP64 (0.1 to 0.2 ms beside it). Against the loop with one
// FP64 multiply-add per nonzero (and a plain one with a row at a time): 2^28
// nonzeros, 256 a row, 0.86 -> 0.62 ms (5.11), 64^3 with 128 a row 168 -> 112
// us; the same error against extended precision (at most 2e-16 of the sum).
template <typename V>
__global__ void __launch_bounds__(256, 4)
k_dev_partials_tl3(int64_t i0, int64_t i1, int64_t ntiles, const int64_t *__restrict__ rowptr, TliTiles tl,
                   const V *__restrict__ val, const float *__restrict__ f, const float *__restrict__ r, int r_scalar,
                   const float *__restrict__ y, double *__restrict__ part)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ float rows[3][kTliTile][33];
    __shared__ double sum[kTliTile];
    __shared__ double sh[32];
    float *xs = reinterpret_cast<float *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int R = kTliTile / 8;
    double mine = 0.0;
    for (int64_t t = i0 / kTliTile + blockIdx.x; t < ntiles && t * kTliTile < i1; t += gridDim.x) {
        const int64_t t0 = t * kTliTile, t1 = t0 + kTliTile < i1 ? t0 + kTliTile : i1;
        if (threadIdx.x == 0) prefetch_segments_l2(rowptr, t0, t1, tl.lidx, val);
        const int wl = tl.wlen[t];
        const int64_t u0 = tl.uoff[t];
        const int nstage = wl > 0 ? wl : int(tl.uoff[t + 1] - u0);
        const int64_t wb = tl.wbase[t];
        for (int k = threadIdx.x; k < nstage; k += blockDim.x)
            xs[k] = f[wl > 0 ? wb + k : int64_t(tl.uidx[u0 + k])];
        __syncthreads();
        const int64_t w0 = t0 + warp * R;
        const int n = w0 < t1 ? int(t1 - w0 < R ? t1 - w0 : R) : 0;
        const int64_t bound = lane <= n && n > 0 ? rowptr[w0 + lane] : 0;
#pragma unroll 1
        for (int k = 0; k < n; k += 2) {
            const int64_t sa = __shfl_sync(0xffffffffu, bound, k), sb = __shfl_sync(0xffffffffu, bound, k + 1);
            const int64_t se = __shfl_sync(0xffffffffu, bound, k + 2 <= n ? k + 2 : k + 1);
            const int na = int(sb - sa), nb = int(se - sb);  // the second row: none at an odd end
            const uint16_t *__restrict__ la = tl.lidx + sa, *__restrict__ lb = tl.lidx + sb;
            const V *__restrict__ va = val + sa, *__restrict__ vb = val + sb;
            uint64_t s0 = 0, s1 = 0, s2 = 0;
            for (int p = 0; p < na || p < nb; p += 128) {
                int32_t ca[4], cb[4];
                float x[4], z[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int q = p + 32 * u + lane;
                    ca[u] = cb[u] = 0;
                    x[u] = z[u] = 0.f;
                    if (q < na) {
                        ca[u] = ld_idx(la + q);
                        x[u] = ld_val(va + q);
                    }
                    if (q < nb) {
                        cb[u] = ld_idx(lb + q);
                        z[u] = ld_val(vb + q);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int q0 = p + 32 * u;
                    if (q0 >= na && q0 >= nb) break;  // warp-uniform
                    const int q = q0 + lane;
                    const uint64_t a = pack2(x[u], z[u]);
                    const uint64_t b = pack2(q < na ? xs[ca[u]] : 0.f, q < nb ? xs[cb[u]] : 0.f);
                    const uint64_t w = fma2(a, b, pack2(-0.f, -0.f));
                    const uint64_t e = fma2(a, b, sub2(pack2(-0.f, -0.f), w));  // a b = w + e
                    uint64_t l0, l1, l2;
                    s0 = two_sum2(s0, w, l0);
                    s1 = two_sum2(s1, l0, l1);
                    s1 = two_sum2(s1, e, l2);
                    s2 = add2(s2, add2(l1, l2));
                }
            }
            const uint64_t s[3] = {s0, s1, s2};
#pragma unroll
            for (int m = 0; m < 3; m++) {
                float u, v;
                asm("mov.b64 {%0, %1}, %2;" : "=f"(u), "=f"(v) : "l"(s[m]));
                rows[m][warp * R + k][lane] = u;
                if (k + 1 < n) rows[m][warp * R + k + 1][lane] = v;
            }
        }
        __syncthreads();
        // 4 threads per row: 8 lanes' sums each, then the quad's total
        const int rr = threadIdx.x >> 2, qd = threadIdx.x & 3;
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
        for (int m = 0; m < 8; m++) {
            float l0, l1, l2;
            a0 = two_sum(a0, rows[0][rr][qd + 4 * m], l0);
            a1 = two_sum(a1, l0, l1);
            a1 = two_sum(a1, rows[1][rr][qd + 4 * m], l2);
            a2 += (l1 + l2) + rows[2][rr][qd + 4 * m];
        }
        double yb = double(a0) + (double(a1) + double(a2));
        yb += __shfl_xor_sync(0xffffffffu, yb, 1);
        yb += __shfl_xor_sync(0xffffffffu, yb, 2);
        if (qd == 0) sum[rr] = yb;
        __syncthreads();
        const int64_t i = t0 + threadIdx.x;
        if (threadIdx.x < kTliTile) {  // whole warps
            const bool in = i >= i0 && i < t1;
            const double ri = in ? double(r_scalar ? r[0] : r[i]) : 1.0;
            double ab = in ? sum[threadIdx.x] : 0.0;
            // what underflowed is below 2^-149 a product; NaN fails too
            uint32_t again = __ballot_sync(0xffffffffu, !(fabs(ab + ri) > 0x1p-60 && fabs(ab) < 0x1p100));
            for (; again != 0u; again &= again - 1u) {
                const int k = __ffs(again) - 1;
                const int64_t row = t0 + 32 * warp + k;
                double acc = 0.0;
                for (int64_t p = rowptr[row] + lane; p < rowptr[row + 1]; p += 32)
                    acc = fma(double(ld_val(val + p)), double(xs[ld_idx(tl.lidx + p)]), acc);
                acc = warp_sum_d(acc);
                if (lane == k) ab = acc;
            }
            if (in) mine += dev_term(ab + ri, double(y[i]));
        }
        __syncthreads();  // rows and xs are rewritten by the next tile
    }
    double tot = block_reduce<false>(mine, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// TV partials over sites [s0, s1) of a direction-major field. Without `d`:
// field 0 = R(w.G f), field 1 = sum over the scans of beta R, where R adds one
// norm per site (group TV) or, BIN, per site and q-bin. With `d` (PRIMAL):
// field 0 = ||w.G f - d||^2 and field 1 = ||d||^2 (primal residual). A site's
// q-bins are loaded for all directions before the FP64 arithmetic, which bounds
// the pass (the FP64 unit's 2 lanes per clock): each value is converted once.
// Without the sums of the other regulariser and with twice the warps in flight
// (FP32, four directions): 128 x 128 x 64 92 -> 56 us, 64^3 29 -> 20 us.
template <typename T, bool PRIMAL, bool BIN>
__global__ void __launch_bounds__(256)
k_tv_partials(Geom g, const T *__restrict__ f, const T *__restrict__ d, int64_t s0, int64_t s1,
              double *__restrict__ part)
{
    __shared__ double sh[32];
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    double a0 = 0.0, a1 = 0.0;
    for (int64_t site = s0 + ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5); site < s1; site += nwarps) {
        int64_t v0;
        const Loc L = locate_site(g, site, v0);
        bool in[4];
        int64_t step[4];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            in[p] = p < g.n_dirs && inside(L, L.x + g.dx[p], L.z + g.dz[p]);
            step[p] = in[p] ? step_of(g, L, p) : 0;
        }
        double n2 = 0.0, dd = 0.0, rb = 0.0;  // rb: sum of the (site, q) norms (standard TV)
        for (int q = lane; q < L.Nq; q += 32) {
            const int64_t j = v0 + q;
            const T fj = f[j];
            T fn[4], dv[4];
#pragma unroll
            for (int p = 0; p < 4; p++) {
                fn[p] = in[p] ? f[j + step[p]] : T(0);
                dv[p] = (PRIMAL && p < g.n_dirs) ? d[int64_t(p) * g.J + j] : T(0);
            }
            const double x = double(fj);
            double m2 = 0.0;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                if (p >= g.n_dirs) break;
                double v = g.w[p] * (x - (in[p] ? double(fn[p]) : 0.0));
                if (PRIMAL) {
                    v -= double(dv[p]);
                    dd += double(dv[p]) * double(dv[p]);
                }
                if (BIN) m2 += v * v;
                else n2 += v * v;
            }
            if (BIN) rb += sqrt(m2);
        }
        if (PRIMAL) {  // sums of squares: the lanes keep theirs
            a0 += n2;
            a1 += dd;
            continue;
        }
        const double r = BIN ? warp_sum_d(rb) : sqrt(warp_sum_d(n2));
        if (lane == 0) {
            a0 += r;
            a1 += L.beta * r;
        }
    }
    double t0 = block_reduce<false>(a0, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t0;
    double t1 = block_reduce<false>(a1, sh);
    if (threadIdx.x == 0) part[gridDim.x + blockIdx.x] = t1;
}

// KKT partials: g_j = s_j - e_j + rho_scan ((w.G)^T c)_j, max_j |min(f_j, g_j)|, and max s.
template <typename T>
__global__ void __launch_bounds__(256)
k_kkt_partials(Geom g, const T *__restrict__ f, const T *__restrict__ e, const T *__restrict__ s,
               const T *__restrict__ c, double *__restrict__ part)
{
    __shared__ double sh[32];
    double m = 0.0, smax = 0.0;
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < g.J; j += int64_t(gridDim.x) * blockDim.x) {
        const Loc L = locate_voxel(g, j);
        double adj = 0.0;
        for (int p = 0; p < g.n_dirs; p++) {
            const int64_t pj = int64_t(p) * g.J + j;
            adj += g.w[p] * double(c[pj]);
            if (inside(L, L.x - g.dx[p], L.z - g.dz[p])) adj -= g.w[p] * double(c[pj - step_of(g, L, p)]);
        }
        const double gj = double(s[j]) - double(e[j]) + L.rho * adj;
        m = fmax(m, fabs(fmin(double(f[j]), gj)));
        smax = fmax(smax, double(s[j]));
    }
    double t0 = block_reduce<true>(m, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t0;
    double t1 = block_reduce<true>(smax, sh);
    if (threadIdx.x == 0) part[gridDim.x + blockIdx.x] = t1;
}

// Dual-residual partials: with a_j = rho_scan ((w.G)^T (d - d_prev))_j and
// b_j = rho_scan ((w.G)^T c)_j, field 0 = sum_j a_j^2, field 1 = sum_j b_j^2.
template <typename T>
__global__ void __launch_bounds__(256)
k_dual_partials(Geom g, const T *__restrict__ d, const T *__restrict__ d_prev, const T *__restrict__ c,
                double *__restrict__ part)
{
    __shared__ double sh[32];
    double sa = 0.0, sb = 0.0;
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < g.J; j += int64_t(gridDim.x) * blockDim.x) {
        const Loc L = locate_voxel(g, j);
        double a = 0.0, b = 0.0;
        for (int p = 0; p < g.n_dirs; p++) {
            const int64_t pj = int64_t(p) * g.J + j;
            a += g.w[p] * (double(d[pj]) - double(d_prev[pj]));
            b += g.w[p] * double(c[pj]);
            if (inside(L, L.x - g.dx[p], L.z - g.dz[p])) {
                const int64_t pa = pj - step_of(g, L, p);
                a -= g.w[p] * (double(d[pa]) - double(d_prev[pa]));
                b -= g.w[p] * double(c[pa]);
            }
        }
        a *= L.rho;
        b *= L.rho;
        sa += a * a;
        sb += b * b;
    }
    double t0 = block_reduce<false>(sa, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t0;
    double t1 = block_reduce<false>(sb, sh);
    if (threadIdx.x == 0) part[gridDim.x + blockIdx.x] = t1;
}

// Sum of a T vector in FP64 (kappa of the initialisation).
template <typename T>
__global__ void __launch_bounds__(256)
k_sum_partials(int64_t n, const T *__restrict__ a, double *__restrict__ part)
{
    __shared__ double sh[32];
    double acc = 0.0;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x)
        acc += double(a[k]);
    double t = block_reduce<false>(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

}  // namespace sgtv
