// POINT kernel family: one thread owns one point and runs the whole recursion
// for a compile-time l_max in registers (arXiv 2302.08381, Section 2:
// Eq. iter-sc for c_m/s_m, Eq. iter-q for Q_l^m with the prefactor folded in
// as in Appendix C, Eq. iter-deri for derivatives).
//
// Work decomposition: every warp is independent. It takes tiles of P points
// (P <= 32, lanes >= P idle) from a persistent grid-stride loop. Outputs of a
// tile are contiguous in global memory ([P, K] for sph, [P, 3, K] for dsph), so
// lanes write their rows into a shared-memory image of that range and one lane
// sends it with a bulk (TMA) copy. With K odd (even l_max) the row stride is
// odd and the per-lane stores are bank-conflict free. With K even (odd l_max)
// an image with stride K would put lanes on 4 to 32 times the same bank, so
// rows are padded to an odd stride (K+1, 3K+1) and the warp copies the tile
// out with coalesced plain stores instead. Backward kernels read their [P, K]
// upstream-gradient tile the same way: bulk loads tracked by mbarriers,
// double buffered (odd K), or coalesced plain loads into padded rows (even K).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "sph_core.cuh"
#include "sph_hardcoded.cuh"
#include "sph_internal.h"

namespace sph {

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// Tables passed by value as kernel parameters (constant bank), so every
// coefficient is an immediate constant-bank operand of the FMA that uses it.
template <int L, typename T, bool HESS>
struct PointTabs {
    static constexpr int TRI = (L + 1) * (L + 2) / 2;
    static constexpr int TRIH = HESS ? TRI : 1;
    T qll[L + 1];
    T d[L + 1];
    T a[TRI];
    T b[TRI];
    T e[TRI];
    T fz[TRI];
    T g2[TRIH];
    T g3[TRIH];
    T g4[TRIH];
    T inv_sqrt2;
};

template <int L, typename T, bool HESS>
PointTabs<L, T, HESS> make_point_tabs() {
    const HostTables& h = host_tables();
    PointTabs<L, T, HESS> t;
    std::memset(&t, 0, sizeof(t));
    for (int l = 0; l <= L; ++l) {
        t.qll[l] = static_cast<T>(h.qll[tri(l, l)]);
        t.d[l] = (l >= 1) ? static_cast<T>(h.d[tri(l, l - 1)]) : T(0);
        for (int m = 0; m <= l; ++m) {
            const int i = tri(l, m);
            t.a[i] = static_cast<T>(h.a[i]);
            t.b[i] = static_cast<T>(h.b[i]);
            t.e[i] = static_cast<T>(h.e[i]);
            t.fz[i] = static_cast<T>(h.fz[i]);
            if (HESS) {
                t.g2[i] = static_cast<T>(h.g2[i]);
                t.g3[i] = static_cast<T>(h.g3[i]);
                t.g4[i] = static_cast<T>(h.g4[i]);
            }
        }
    }
    t.inv_sqrt2 = static_cast<T>(h.inv_sqrt2);
    return t;
}

// The unrolled recursion for one point from degree L0 on. (x, y, z, r2) are
// the coordinates the polynomials are evaluated at (already divided by r for
// the normalized form); c, s hold c_m, s_m for m <= L; q1, q2 hold
// Qtilde_{L0-1}^m and Qtilde_{L0-2}^m (zero for m beyond the degree).
// Calls vis.emit(l, k, Deriv) once per output column k = l*l + l + m, l >= L0.
template <int L, int L0, bool GRAD, bool HESS, typename T, typename Tabs, typename Vis>
__device__ __forceinline__ void point_core_from(T x, T y, T z, T r2, const Tabs& tb, Vis& vis, const T (&c)[L + 1],
                                                const T (&s)[L + 1], T (&q1)[L + 1], T (&q2)[L + 1]) {
#pragma unroll
    for (int l = L0; l <= L; ++l) {
        T q[L + 1];
        q[l] = tb.qll[l];
        if (l >= 1) q[l - 1] = tb.d[l] * z * q1[l - 1];
#pragma unroll
        for (int m = 0; m + 2 <= l; ++m) {  // Eq. iter-q, folded
            const int i = tri(l, m);
            q[m] = (tb.a[i] * z) * q1[m] - (tb.b[i] * r2) * q2[m];
        }
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            const int i = tri(l, m);
            QParts<T> qp;
            qp.Q = q[m];
            qp.E1 = (m + 1 <= l - 1) ? tb.e[i] * q1[m + 1] : T(0);
            qp.Qz = (m <= l - 1) ? tb.fz[i] * q1[m] : T(0);
            if constexpr (HESS) {
                qp.G2 = (m + 2 <= l - 2) ? tb.g2[i] * q2[m + 2] : T(0);
                qp.G3 = (m + 1 <= l - 2) ? tb.g3[i] * q2[m + 1] : T(0);
                qp.G4 = (m <= l - 2) ? tb.g4[i] * q2[m] : T(0);
            } else {
                qp.G2 = qp.G3 = qp.G4 = T(0);
            }
            if (m == 0) {
                Deriv<T> d = assemble_m0<GRAD, HESS>(qp, x, y, tb.inv_sqrt2);
                vis.emit(l, l * l + l, d);
            } else {
                Deriv<T> dc, ds;
                const T cm2 = (m >= 2) ? c[m >= 2 ? m - 2 : 0] : T(0);
                const T sm2 = (m >= 2) ? s[m >= 2 ? m - 2 : 0] : T(0);
                assemble_m<GRAD, HESS>(qp, x, y, T(m), T(m - 1), c[m], s[m], c[m - 1], s[m - 1], cm2, sm2, dc,
                                       ds);
                vis.emit(l, l * l + l + m, dc);
                vis.emit(l, l * l + l - m, ds);
            }
        }
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            q2[m] = q1[m];
            q1[m] = q[m];
        }
    }
}

template <int L, typename T>
__device__ __forceinline__ void point_cs(T x, T y, T (&c)[L + 1], T (&s)[L + 1]) {
    c[0] = T(1);
    s[0] = T(0);
#pragma unroll
    for (int m = 1; m <= L; ++m) {  // Eq. iter-sc
        c[m] = x * c[m - 1] - y * s[m - 1];
        s[m] = x * s[m - 1] + y * c[m - 1];
    }
}

// The whole recursion for one point (every degree from 0).
template <int L, bool GRAD, bool HESS, typename T, typename Tabs, typename Vis>
__device__ __forceinline__ void point_core(T x, T y, T z, T r2, const Tabs& tb, Vis& vis) {
    T c[L + 1], s[L + 1];
    point_cs<L>(x, y, c, s);
    T q1[L + 1], q2[L + 1];  // Qtilde_{l-1}^m, Qtilde_{l-2}^m
#pragma unroll
    for (int m = 0; m <= L; ++m) {
        q1[m] = T(0);
        q2[m] = T(0);
    }
    point_core_from<L, 0, GRAD, HESS>(x, y, z, r2, tb, vis, c, s, q1, q2);
}

// Hybrid (Section 3.2: hard-coded low degrees, the general recursion above):
// degrees l <= min(L, 3) from the generated straight-line expressions of
// sph_hardcoded.cuh, which also give Qtilde_LH^m and Qtilde_{LH-1}^m, and
// Eq. iter-q from degree LH + 1. Values and gradients (no Hessians).
template <int L, bool GRAD, typename T, typename Tabs, typename Vis>
__device__ __forceinline__ void point_core_hc(T x, T y, T z, T r2, const Tabs& tb, Vis& vis) {
    constexpr int LH = L < 3 ? L : 3;
    T qa[4] = {T(0), T(0), T(0), T(0)}, qb[4] = {T(0), T(0), T(0), T(0)};
    if constexpr (LH == 0) {
        if constexpr (GRAD) hardcoded_l0_grad(x, y, z, r2, vis, qa, qb); else hardcoded_l0_val(x, y, z, r2, vis, qa, qb);
    } else if constexpr (LH == 1) {
        if constexpr (GRAD) hardcoded_l1_grad(x, y, z, r2, vis, qa, qb); else hardcoded_l1_val(x, y, z, r2, vis, qa, qb);
    } else if constexpr (LH == 2) {
        if constexpr (GRAD) hardcoded_l2_grad(x, y, z, r2, vis, qa, qb); else hardcoded_l2_val(x, y, z, r2, vis, qa, qb);
    } else {
        if constexpr (GRAD) hardcoded_l3_grad(x, y, z, r2, vis, qa, qb); else hardcoded_l3_val(x, y, z, r2, vis, qa, qb);
    }
    if constexpr (L > LH) {
        T c[L + 1], s[L + 1];
        point_cs<L>(x, y, c, s);
        T q1[L + 1], q2[L + 1];
#pragma unroll
        for (int m = 0; m <= L; ++m) {
            q1[m] = m <= LH ? qa[m <= LH ? m : 0] : T(0);
            q2[m] = m <= LH - 1 ? qb[m <= LH - 1 ? m : 0] : T(0);
        }
        point_core_from<L, LH + 1, GRAD, false>(x, y, z, r2, tb, vis, c, s, q1, q2);
    }
}

// ------------------------------------------------------------------ forward
template <typename T, typename TO, bool GRAD, bool HESS, bool NORM, int K>
struct FwdVis {
    TO* rv;  // this lane's sph row in shared memory
    TO* rd;  // this lane's dsph row (3 planes of K)
    TO* rh;  // this lane's ddsph row (9 planes of K, i-major)
    T ux, uy, uz, ir;
    __device__ __forceinline__ void emit(int l, int k, Deriv<T> d) {
        if (GRAD || HESS) {
            if (NORM) normalize_deriv<HESS>(d, l, ux, uy, uz, ir);
            rd[k] = OutConv<TO>::cv(d.gx);
            rd[K + k] = OutConv<TO>::cv(d.gy);
            rd[2 * K + k] = OutConv<TO>::cv(d.gz);
        }
        if (HESS) {
            rh[0 * K + k] = OutConv<TO>::cv(d.hxx);
            rh[1 * K + k] = OutConv<TO>::cv(d.hxy);
            rh[2 * K + k] = OutConv<TO>::cv(d.hxz);
            rh[3 * K + k] = OutConv<TO>::cv(d.hxy);
            rh[4 * K + k] = OutConv<TO>::cv(d.hyy);
            rh[5 * K + k] = OutConv<TO>::cv(d.hyz);
            rh[6 * K + k] = OutConv<TO>::cv(d.hxz);
            rh[7 * K + k] = OutConv<TO>::cv(d.hyz);
            rh[8 * K + k] = OutConv<TO>::cv(d.hzz);
        }
        rv[k] = OutConv<TO>::cv(d.v);
    }
};

// Shared-memory row strides (elements) of a tile: the contiguous image for
// odd K, odd-padded rows for even K.
template <int L>
struct RowStride {
    static constexpr int K = (L + 1) * (L + 1);
    static constexpr bool PAD = (K % 2 == 0);
    static constexpr int V = PAD ? K + 1 : K;          // sph / g rows
    static constexpr int D = PAD ? 3 * K + 1 : 3 * K;  // dsph rows
    static constexpr int H = PAD ? 9 * K + 1 : 9 * K;  // ddsph rows
};

template <int L, bool GRAD, bool HESS, typename TO>
__host__ __device__ constexpr size_t point_fwd_warp_bytes(int P) {
    return align16(size_t(P) * RowStride<L>::V * sizeof(TO)) +
           (GRAD ? align16(size_t(P) * RowStride<L>::D * sizeof(TO)) : 0) +
           (HESS ? align16(size_t(P) * RowStride<L>::H * sizeof(TO)) : 0);
}

// Copies `rows` rows of `cols` elements from a padded shared-memory image
// (row stride `stride`) to a contiguous global range, 32 consecutive
// elements per warp store.
template <int cols, typename TO>
__device__ __forceinline__ void warp_rows_out(TO* __restrict__ gdst, const TO* __restrict__ ssrc, int rows, int stride,
                                              int lane) {
    const int total = rows * cols;
    for (int i = lane; i < total; i += 32) {
        const int r = i / cols;
        gdst[i] = ssrc[r * stride + (i - r * cols)];
    }
}

template <int cols, typename T>
__device__ __forceinline__ void warp_rows_in(T* __restrict__ sdst, const T* __restrict__ gsrc, int rows, int stride,
                                             int lane) {
    const int total = rows * cols;
    for (int i = lane; i < total; i += 32) {
        const int r = i / cols;
        sdst[r * stride + (i - r * cols)] = gsrc[i];
    }
}

// Type of the coordinates: the arithmetic's, but FP32 for FP64 arithmetic on
// FP32 storage.
template <typename T, typename TO>
using PointIn = std::conditional_t<sizeof(T) == 8 && sizeof(TO) != 8, float, T>;

template <int L, bool GRAD, bool HESS, bool NORM, typename T, typename TO, bool HC = false>
__global__ void __launch_bounds__(256) point_fwd_kernel(const PointIn<T, TO>* __restrict__ xyz, int64_t n,
                                                        const __grid_constant__ PointTabs<L, T, HESS> tb,
                                                        TO* __restrict__ sph, TO* __restrict__ dsph,
                                                        TO* __restrict__ ddsph, int P, int bulk) {
    constexpr int K = (L + 1) * (L + 1);
    using RS = RowStride<L>;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    const size_t vbytes = align16(size_t(P) * RS::V * sizeof(TO));
    TO* s_v = reinterpret_cast<TO*>(smem + size_t(warp) * point_fwd_warp_bytes<L, GRAD, HESS, TO>(P));
    TO* s_d = reinterpret_cast<TO*>(reinterpret_cast<unsigned char*>(s_v) + vbytes);
    TO* s_h = reinterpret_cast<TO*>(reinterpret_cast<unsigned char*>(s_d) +
                                    (GRAD ? align16(size_t(P) * RS::D * sizeof(TO)) : 0));

    const int64_t ntiles = (n + P - 1) / P;
    const int64_t stride = int64_t(gridDim.x) * W;
    int64_t tile = int64_t(blockIdx.x) * W + warp;

    // Software-pipelined coordinate loads: the next tile's point is fetched
    // while the current one is computed.
    T nx = T(0), ny = T(0), nz = T(0);
    if (tile < ntiles && lane < P) {
        const int64_t p = tile * P + lane;
        if (p < n) {
            nx = xyz[3 * p];
            ny = xyz[3 * p + 1];
            nz = xyz[3 * p + 2];
        }
    }
    for (; tile < ntiles; tile += stride) {
        T x = nx, y = ny, z = nz;
        const int64_t nt = tile + stride;
        if (nt < ntiles && lane < P) {
            const int64_t p = nt * P + lane;
            if (p < n) {
                nx = xyz[3 * p];
                ny = xyz[3 * p + 1];
                nz = xyz[3 * p + 2];
            }
        }
        const int64_t p0 = tile * P;
        const int cnt = int(min(int64_t(P), n - p0));
        if (lane < cnt) {
            T r2, ir = T(1);
            if (NORM) {
                unit_point(x, y, z, r2, ir);
            } else {
                r2 = x * x + y * y + z * z;
            }
            FwdVis<T, TO, GRAD, HESS, NORM, K> vis{s_v + size_t(lane) * RS::V, s_d + size_t(lane) * RS::D,
                                                   s_h + size_t(lane) * RS::H, x, y, z, ir};
            if constexpr (HC && !HESS)
                point_core_hc<L, GRAD>(x, y, z, r2, tb, vis);
            else
                point_core<L, GRAD, HESS>(x, y, z, r2, tb, vis);
        }
        if constexpr (RS::PAD) {
            __syncwarp();
            warp_rows_out<K>(sph + p0 * K, s_v, cnt, RS::V, lane);
            if (GRAD) warp_rows_out<3 * K>(dsph + p0 * 3 * K, s_d, cnt, RS::D, lane);
            if (HESS) warp_rows_out<9 * K>(ddsph + p0 * 9 * K, s_h, cnt, RS::H, lane);
            __syncwarp();
            continue;
        }
        fence_proxy_async_smem();
        __syncwarp();
        const int64_t ev = int64_t(cnt) * K;  // elements of the sph tile
        int64_t ev_bulk = 0, ed_bulk = 0, eh_bulk = 0;
        if (bulk) {
            ev_bulk = (ev * int64_t(sizeof(TO))) / 16 * 16 / int64_t(sizeof(TO));
            ed_bulk = GRAD ? (3 * ev * int64_t(sizeof(TO))) / 16 * 16 / int64_t(sizeof(TO)) : 0;
            eh_bulk = HESS ? (9 * ev * int64_t(sizeof(TO))) / 16 * 16 / int64_t(sizeof(TO)) : 0;
            if (lane == 0) {
                if (ev_bulk) bulk_store(sph + p0 * K, s_v, uint32_t(ev_bulk * sizeof(TO)));
                if (GRAD && ed_bulk) bulk_store(dsph + p0 * 3 * K, s_d, uint32_t(ed_bulk * sizeof(TO)));
                if (HESS && eh_bulk) bulk_store(ddsph + p0 * 9 * K, s_h, uint32_t(eh_bulk * sizeof(TO)));
                bulk_commit();
            }
        }
        // Ragged remainder (and everything, without bulk copies): plain stores.
        for (int64_t i = ev_bulk + lane; i < ev; i += 32) sph[p0 * K + i] = s_v[i];
        if (GRAD)
            for (int64_t i = ed_bulk + lane; i < 3 * ev; i += 32) dsph[p0 * 3 * K + i] = s_d[i];
        if (HESS)
            for (int64_t i = eh_bulk + lane; i < 9 * ev; i += 32) ddsph[p0 * 9 * K + i] = s_h[i];
        if (bulk && lane == 0) bulk_wait_read_all();
        __syncwarp();
    }
    if (bulk && lane == 0) bulk_wait_all();
}

// -------------------------------------- forward, 4 lanes per point (planes)
// POINT with lanes_per_point = 4 (values and gradients): lane 4j + r of a
// warp owns output plane r (0 the value, 1..3 d/dx, d/dy, d/dz) of the tile's
// point j, so a tile of 8 points keeps all 32 lanes busy where the
// one-lane-per-point tile that fits shared memory at large l_max holds only
// 8 to 16 points. Every lane runs the Q recursion (Eq. iter-q) and Eq.
// iter-sc in full (cheap next to the assembly) and assembles only its plane
// with role weights, the same instruction stream in every lane:
//   plane = A c_m + Qtilde_l^m C'_m,   A = aq Qtilde + ax e Qtilde_{l-1}^{m+1} + a3 f Qtilde_{l-1}^m
// (aq, ax, a3) = (1, 0, 0), (0, x, 0), (0, y, 0), (0, 0, 1) by role, and
// C'_m = m c_{m-1} (d/dx), -m s_{m-1} (d/dy), 0 (value, d/dz); the sin-type column
// takes s_m and S'_m = m s_{m-1}, m c_{m-1}, 0. These are the terms of Eq.
// iter-deri that assemble_m combines for all four planes at once. The
// normalized form, (plane - l u_r Y) / r, has the same terms: 1/r goes into ax,
// a3 and C', S', and -l u_r / r into aq. 13 operations per pair of columns;
// with m and the normalization applied to the assembled columns it was 14, and
// 20 normalized, and bf16 rows and normalized l_max >= 12 are bound by them
// (issue 75 % busy at l_max 10, bf16).
template <int L, bool NORM, typename T, typename TO, typename Tabs>
__device__ __forceinline__ void point4_core(T x, T y, T z, T r2, const Tabs& tb, int r, T ir,
                                            TO* __restrict__ rowp) {
    const T irr = (NORM && r != 0) ? ir : T(1);
    const T a0 = r == 0 ? T(1) : T(0);
    const T ax = irr * (r == 1 ? x : (r == 2 ? y : T(0)));
    const T a3 = r == 3 ? irr : T(0);
    const T nu = NORM ? -irr * (r == 1 ? x : (r == 2 ? y : (r == 3 ? z : T(0)))) : T(0);  // l times: into aq
    T c[L + 1], s[L + 1];
    point_cs<L>(x, y, c, s);
    // The factor m is in (C'_m, S'_m), except in the scaled form to l_max 12, where
    // multiplying Qtilde by it measured 2..3 % faster (bf16; l_max 14, 16: 9 % slower)
    constexpr bool FOLD = NORM || L > 12;
    auto fm = [](int m) { return FOLD ? T(m) : T(1); };
    T c1[L + 1], s1[L + 1];  // (C'_m, S'_m) of this lane's role
    {
        const T k1 = r == 1 ? irr : T(0), k2 = r == 2 ? -irr : T(0);
        const T k3 = r == 2 ? irr : T(0), k4 = r == 1 ? irr : T(0);
        c1[0] = T(0);
        s1[0] = T(0);
#pragma unroll
        for (int m = 1; m <= L; ++m) {
            c1[m] = fm(m) * (k1 * c[m - 1] + k2 * s[m - 1]);
            s1[m] = fm(m) * (k3 * c[m - 1] + k4 * s[m - 1]);
        }
    }
    T q1[L + 1], q2[L + 1];
#pragma unroll
    for (int m = 0; m <= L; ++m) {
        q1[m] = T(0);
        q2[m] = T(0);
    }
#pragma unroll
    for (int l = 0; l <= L; ++l) {
        T q[L + 1];
        q[l] = tb.qll[l];
        if (l >= 1) q[l - 1] = tb.d[l] * z * q1[l - 1];
#pragma unroll
        for (int m = 0; m + 2 <= l; ++m) {  // Eq. iter-q, folded
            const int i = tri(l, m);
            q[m] = (tb.a[i] * z) * q1[m] - (tb.b[i] * r2) * q2[m];
        }
        const T aq = NORM ? fma(nu, T(l), a0) : a0;
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            const int i = tri(l, m);
            const T E1 = (m + 1 <= l - 1) ? tb.e[i] * q1[m + 1] : T(0);
            const T Qz = (m <= l - 1) ? tb.fz[i] * q1[m] : T(0);
            if (m == 0) {
                rowp[l * l + l] = OutConv<TO>::cv((aq * tb.inv_sqrt2) * q[0] + ax * E1 + a3 * Qz);
            } else {
                const T A = aq * q[m] + ax * E1 + a3 * Qz;
                const T mq = FOLD ? q[m] : T(m) * q[m];
                rowp[l * l + l + m] = OutConv<TO>::cv(A * c[m] + mq * c1[m]);
                rowp[l * l + l - m] = OutConv<TO>::cv(A * s[m] + mq * s1[m]);
            }
        }
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            q2[m] = q1[m];
            q1[m] = q[m];
        }
    }
}

// Shared-memory image of a 4-lane tile: P value rows and 3P gradient plane
// rows of stride S (point4_stride): MODE 0 the image of the global ranges
// (one bulk copy per array), 1 rows at 16-byte-aligned strides (one bulk copy
// per row, issued by the lane that wrote it), 2 padded rows copied out by the
// warp with coalesced stores.
template <int L, typename TO>
struct Row4 {
    static constexpr int K = (L + 1) * (L + 1);
    static constexpr int S = point4_stride(L, int(sizeof(TO)));
    static constexpr int MODE = point4_out_mode(L, int(sizeof(TO)));
};

template <int L, typename TO>
__host__ __device__ constexpr size_t point4_warp_bytes(int P) {
    return align16(size_t(P) * Row4<L, TO>::S * sizeof(TO)) + align16(size_t(3 * P) * Row4<L, TO>::S * sizeof(TO));
}

// One tile of a set: points [p0, p0 + cnt), cnt <= P <= 8, lane 4j + r
// computing plane r of point j at (x, y, z); outputs staged at buf
// (point4_warp_bytes<L, TO>(P) bytes) and sent to the set's sph / dsph.
// Warp-collective; returns with the staging buffer free for the next tile.
template <int L, bool NORM, typename T, typename TO, typename Tabs>
__device__ __forceinline__ void point4_tile(TO* __restrict__ sph, TO* __restrict__ dsph, int64_t p0, int cnt, int P,
                                            int bulk, unsigned char* buf, const Tabs& tb, int lane, T x, T y, T z) {
    constexpr int K = (L + 1) * (L + 1);
    constexpr int S = Row4<L, TO>::S;
    constexpr int MODE = Row4<L, TO>::MODE;
    const int pt = lane >> 2, r = lane & 3;
    TO* s_v = reinterpret_cast<TO*>(buf);
    TO* s_d = reinterpret_cast<TO*>(buf + align16(size_t(P) * S * sizeof(TO)));
    TO* rowp = r == 0 ? s_v + size_t(pt) * S : s_d + size_t(3 * pt + r - 1) * S;
    if (pt < cnt) {
        T r2, ir = T(1);
        if (NORM) {
            unit_point(x, y, z, r2, ir);
        } else {
            r2 = x * x + y * y + z * z;
        }
        point4_core<L, NORM>(x, y, z, r2, tb, r, ir, rowp);
    }
    if constexpr (MODE == 1) {
        if (bulk) {  // each lane sends the row it wrote (16-byte aligned at both ends)
            if (pt < cnt) {
                fence_proxy_async_smem();
                TO* g = r == 0 ? sph + (p0 + pt) * K : dsph + ((p0 + pt) * 3 + (r - 1)) * K;
                bulk_store(g, rowp, uint32_t(K * sizeof(TO)));
                bulk_commit();
                bulk_wait_read_all();
            }
            __syncwarp();
            return;
        }
    }
    if constexpr (MODE != 0) {
        __syncwarp();
        warp_rows_out<K>(sph + p0 * K, s_v, cnt, S, lane);
        warp_rows_out<K>(dsph + p0 * 3 * K, s_d, 3 * cnt, S, lane);
        __syncwarp();
        return;
    }
    fence_proxy_async_smem();
    __syncwarp();
    const int64_t ev = int64_t(cnt) * K;
    int64_t ev_bulk = 0, ed_bulk = 0;
    if (bulk) {
        ev_bulk = (ev * int64_t(sizeof(TO))) / 16 * 16 / int64_t(sizeof(TO));
        ed_bulk = (3 * ev * int64_t(sizeof(TO))) / 16 * 16 / int64_t(sizeof(TO));
        if (lane == 0) {
            if (ev_bulk) bulk_store(sph + p0 * K, s_v, uint32_t(ev_bulk * sizeof(TO)));
            if (ed_bulk) bulk_store(dsph + p0 * 3 * K, s_d, uint32_t(ed_bulk * sizeof(TO)));
            bulk_commit();
        }
    }
    for (int64_t i = ev_bulk + lane; i < ev; i += 32) sph[p0 * K + i] = s_v[i];
    for (int64_t i = ed_bulk + lane; i < 3 * ev; i += 32) dsph[p0 * 3 * K + i] = s_d[i];
    if (bulk && lane == 0) bulk_wait_read_all();
    __syncwarp();
}

template <int L, bool NORM, typename T, typename TO>
__global__ void __launch_bounds__(256) point4_fwd_kernel(const T* __restrict__ xyz, int64_t n,
                                                         const __grid_constant__ PointTabs<L, T, false> tb,
                                                         TO* __restrict__ sph, TO* __restrict__ dsph, int P,
                                                         int bulk) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    const int pt = lane >> 2;
    unsigned char* buf = smem + size_t(warp) * point4_warp_bytes<L, TO>(P);

    const int64_t ntiles = (n + P - 1) / P;
    const int64_t stride = int64_t(gridDim.x) * W;
    int64_t tile = int64_t(blockIdx.x) * W + warp;
    T nx = T(0), ny = T(0), nz = T(0);
    if (tile < ntiles && pt < P) {
        const int64_t p = tile * P + pt;
        if (p < n) {
            nx = xyz[3 * p];
            ny = xyz[3 * p + 1];
            nz = xyz[3 * p + 2];
        }
    }
    for (; tile < ntiles; tile += stride) {
        const T x = nx, y = ny, z = nz;
        const int64_t nt = tile + stride;
        if (nt < ntiles && pt < P) {
            const int64_t p = nt * P + pt;
            if (p < n) {
                nx = xyz[3 * p];
                ny = xyz[3 * p + 1];
                nz = xyz[3 * p + 2];
            }
        }
        const int64_t p0 = tile * P;
        const int cnt = int(min(int64_t(P), n - p0));
        point4_tile<L, NORM>(sph, dsph, p0, cnt, P, bulk, buf, tb, lane, x, y, z);
    }
    if (bulk) bulk_wait_all();  // every lane: row copies are issued per lane
}

// ------------------------- forward with Hessians, 16 lanes per point (planes)
// POINT with lanes_per_point = 16 (FP32 values, gradients and Hessians):
// lane 16j + r owns output plane r of point j of the current pair of points
// (0 the value, 1..3 the gradient, 4..12 the Hessian entries (i, k) row-major;
// lanes 13..15 compute plane 12 again and store nothing). Every lane runs the
// recursions in full and assembles its plane from one instance of the terms
// of Eq. iter-deri applied once and twice:
//   plane = A C + m B T1 + m (m - 1) Qtilde_l^m T2
//   A = aQ Qtilde + aE e Qtilde_{l-1}^{m+1} + az f Qtilde_{l-1}^m
//       + a2 g2 Qtilde_{l-2}^{m+2} + a3 g3 Qtilde_{l-2}^{m+1} + a4 g4 Qtilde_{l-2}^m
//   B = bQ Qtilde + bE e Qtilde_{l-1}^{m+1} + bz f Qtilde_{l-1}^m
// with C = c_m (or s_m for the sin-type column), T1 a role combination of
// c_{m-1}, s_{m-1} and T2 of c_{m-2}, s_{m-2} (the derivatives of c_m, s_m),
// role weights from the point's coordinates. The normalized form,
//   sc (plane + wv Y - l u_k g_i - l u_i g_k),  g_i = X_i e Qtilde_{l-1}^{m+1} C + ... + m Qtilde_l^m T_i,
// is linear in the same terms, so it only changes the weights with l (aQ, aE,
// az) and adds l m Qtilde_l^m T3, T3 a role combination of c_{m-1}, s_{m-1}: one
// fma more per column. (Taking Y, g_i and g_k of the column from the lanes that
// own those planes cost six shuffles and eight operations per pair of columns.)
template <int L, bool NORM, bool TWO = false, typename Tabs>
__device__ __forceinline__ void point16_core(float x, float y, float z, float r2, const Tabs& tb, int rr, float ir,
                                             float* __restrict__ rowp, float* __restrict__ rowp2,
                                             bool store) {
    const int hi = rr >= 4 ? (rr - 4) / 3 : 0, hk = rr >= 4 ? (rr - 4) % 3 : 0;
    // the symmetric entry (i, k) with i <= k selects the formula
    const int i0 = hi < hk ? hi : hk, k0 = hi < hk ? hk : hi;
    const bool isv = rr == 0, isgx = rr == 1, isgy = rr == 2, isgz = rr == 3, ish = rr >= 4;
    const bool hxx = ish && i0 == 0 && k0 == 0, hxy = ish && i0 == 0 && k0 == 1, hxz = ish && i0 == 0 && k0 == 2;
    const bool hyy = ish && i0 == 1 && k0 == 1, hyz = ish && i0 == 1 && k0 == 2, hzz = ish && i0 == 2 && k0 == 2;
    const float X = x, Y = y;
    // scale of the plane: 1/r of the gradient, 1/r^2 of the Hessian (normalized)
    const float sc = !NORM || isv ? 1.f : (ish ? ir * ir : ir);
    const float aQ = isv ? 1.f : 0.f;
    const float aE = sc * (isgx ? X : (isgy ? Y : ((hxx || hyy) ? 1.f : 0.f)));
    const float az = sc * (isgz ? 1.f : 0.f);
    const float a2 = sc * (hxx ? X * X : (hyy ? Y * Y : (hxy ? X * Y : 0.f)));
    const float a3 = sc * (hxz ? X : (hyz ? Y : 0.f));
    const float a4 = sc * (hzz ? 1.f : 0.f);
    const float bQ = (isgx || isgy) ? sc : 0.f;
    const float bE = (hxx || hyy || hxy) ? sc : 0.f;
    const float bz = (hxz || hyz) ? sc : 0.f;
    // T1c = k1c c1 + k1s s1, T1s = k2c c1 + k2s s1, T2c = k3c c2 + k3s s2, T2s = k4c c2 + k4s s2
    float k1c = 0.f, k1s = 0.f, k2c = 0.f, k2s = 0.f, k3c = 0.f, k3s = 0.f, k4c = 0.f, k4s = 0.f;
    if (isgx || hxz) {
        k1c = 1.f;
        k2s = 1.f;
    } else if (isgy || hyz) {
        k1s = -1.f;
        k2c = 1.f;
    } else if (hxx) {
        k1c = 2.f * X;
        k2s = 2.f * X;
        k3c = sc;
        k4s = sc;
    } else if (hyy) {
        k1s = -2.f * Y;
        k2c = 2.f * Y;
        k3c = -sc;
        k4s = -sc;
    } else if (hxy) {
        k1c = Y;
        k1s = -X;
        k2c = X;
        k2s = Y;
        k3s = -sc;
        k4c = sc;
    }
    float c[L + 1], s[L + 1];
    point_cs<L>(x, y, c, s);
    // Normalized form, (i0, k0) for both (i, k) and (k, i): the two planes of a
    // symmetric pair run the same operations and come out bit-identical.
    // Weights of l (l (l + 2) for nv2) in aQ, aE and az, and of l m Qtilde in T3
    const float ui = i0 == 0 ? x : (i0 == 1 ? y : z), uk = k0 == 0 ? x : (k0 == 1 ? y : z);
    float nv = 0.f, nv2 = 0.f, nE = 0.f, nz = 0.f, k5 = 0.f, k6 = 0.f;
    if (NORM && ish) {
        const float si = -sc * uk, sk = -sc * ui;
        nv = i0 == k0 ? -sc : 0.f;
        nv2 = sc * ui * uk;
        k5 = (i0 == 0 ? si : 0.f) + (k0 == 0 ? sk : 0.f);  // T3c = k5 c1 - k6 s1, T3s = k5 s1 + k6 c1
        k6 = (i0 == 1 ? si : 0.f) + (k0 == 1 ? sk : 0.f);
        nE = k5 * X + k6 * Y;
        nz = (i0 == 2 ? si : 0.f) + (k0 == 2 ? sk : 0.f);
    } else if (NORM && !isv) {
        nv = -sc * (isgx ? x : (isgy ? y : z));
    }
    // The factors m, m (m - 1) are in the role columns of m alone, except in the scaled
    // form to l_max 9 and at 14 and 15, where multiplying B and Qtilde by them is faster
    // (150k points, in the columns / not, us: 10 178/184, 11 197/213, 12 307/317, 13
    // 347/371, 16 794/809; 9 154/159, but 1k points 5.6/5.0; 8 125/126, 1k 6.5/6.1; 14
    // 553/538, 15 535/519).
    constexpr bool FOLD = NORM || (L >= 10 && L != 14 && L != 15);
    auto fm = [](int m) { return FOLD ? float(m) : 1.f; };
    float q1[L + 1], q2[L + 1];
#pragma unroll
    for (int m = 0; m <= L; ++m) {
        q1[m] = 0.f;
        q2[m] = 0.f;
    }
#pragma unroll
    for (int l = 0; l <= L; ++l) {
        float q[L + 1];
        q[l] = tb.qll[l];
        if (l >= 1) q[l - 1] = tb.d[l] * z * q1[l - 1];
#pragma unroll
        for (int m = 0; m + 2 <= l; ++m) {  // Eq. iter-q, folded
            const int i = tri(l, m);
            q[m] = (tb.a[i] * z) * q1[m] - (tb.b[i] * r2) * q2[m];
        }
        const float aQl = NORM ? fmaf(float(l * (l + 2)), nv2, fmaf(float(l), nv, aQ)) : aQ;
        const float aEl = NORM ? fmaf(float(l), nE, aE) : aE;
        const float azl = NORM ? fmaf(float(l), nz, az) : az;
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            const int i = tri(l, m);
            const float E1 = (m + 1 <= l - 1) ? tb.e[i] * q1[m + 1] : 0.f;
            const float Qz = (m <= l - 1) ? tb.fz[i] * q1[m] : 0.f;
            const float G2 = (m + 2 <= l - 2) ? tb.g2[i] * q2[m + 2] : 0.f;
            const float G3 = (m + 1 <= l - 2) ? tb.g3[i] * q2[m + 1] : 0.f;
            const float G4 = (m <= l - 2) ? tb.g4[i] * q2[m] : 0.f;
            const float A = aEl * E1 + azl * Qz + a2 * G2 + a3 * G3 + a4 * G4;
            if (m == 0) {
                const float out = aQl * tb.inv_sqrt2 * q[0] + A;
                if (store) {
                    rowp[l * l + l] = out;
                    if (TWO) rowp2[l * l + l] = out;
                }
            } else {
                const float Am = aQl * q[m] + A;
                const float B = bQ * q[m] + bE * E1 + bz * Qz;
                const float c1 = c[m - 1], s1 = s[m - 1];
                const float c2 = m >= 2 ? c[m >= 2 ? m - 2 : 0] : 0.f, s2 = m >= 2 ? s[m >= 2 ? m - 2 : 0] : 0.f;
                // role columns of m alone (the same for every l)
                const float t1c = fm(m) * (k1c * c1 + k1s * s1), t1s = fm(m) * (k2c * c1 + k2s * s1);
                const float t2c = fm(m * (m - 1)) * (k3c * c2 + k3s * s2);
                const float t2s = fm(m * (m - 1)) * (k4c * c2 + k4s * s2);
                const float Bm = FOLD ? B : float(m) * B;
                float oc = Am * c[m] + Bm * t1c;
                float os = Am * s[m] + Bm * t1s;
                if (NORM) {
                    const float t3c = float(m) * (k5 * c1 - k6 * s1), t3s = float(m) * (k5 * s1 + k6 * c1);
                    oc += q[m] * (float(l) * t3c + t2c);
                    os += q[m] * (float(l) * t3s + t2s);
                } else if (m >= 2) {
                    const float mq = FOLD ? q[m] : float(m * (m - 1)) * q[m];
                    oc += mq * t2c;
                    os += mq * t2s;
                }
                if (store) {
                    rowp[l * l + l + m] = oc;
                    rowp[l * l + l - m] = os;
                    if (TWO) {
                        rowp2[l * l + l + m] = oc;
                        rowp2[l * l + l - m] = os;
                    }
                }
            }
        }
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            q2[m] = q1[m];
            q1[m] = q[m];
        }
    }
}

// Shared-memory bytes of a 16-lane Hessian tile of P points: value rows,
// gradient rows and Hessian rows, each part 16-byte aligned, stride
// point4_stride (the same rules as the 4-lane tile).
template <int L>
__host__ __device__ constexpr size_t point16_warp_bytes(int P) {
    constexpr size_t S = size_t(point4_stride(L, 4)) * 4;
    return align16(size_t(P) * S) + align16(size_t(3 * P) * S) + align16(size_t(9 * P) * S);
}

constexpr int kPoint16MaxTile = 8;  // points per tile (pairs of points per pass)

// One tile of P <= 8 points (P even): the warp computes two points per pass,
// 16 lanes each, into the staged image; warp-collective.
template <int L, bool NORM, typename Tabs>
__device__ __forceinline__ void point16_tile(const float* __restrict__ xyz, float* __restrict__ sph,
                                             float* __restrict__ dsph, float* __restrict__ ddsph, int64_t p0,
                                             int cnt, int P, int bulk, unsigned char* buf, const Tabs& tb,
                                             int lane) {
    constexpr int K = (L + 1) * (L + 1);
    constexpr int S = point4_stride(L, 4);
    constexpr int MODE = point4_out_mode(L, 4);
    float* s_v = reinterpret_cast<float*>(buf);
    float* s_d = reinterpret_cast<float*>(buf + align16(size_t(P) * S * 4));
    float* s_h = reinterpret_cast<float*>(buf + align16(size_t(P) * S * 4) + align16(size_t(3 * P) * S * 4));
    const int r = lane & 15, half = lane >> 4;
    // coordinates of every pass of the tile, loaded up front
    float cx[kPoint16MaxTile / 2], cy[kPoint16MaxTile / 2], cz[kPoint16MaxTile / 2];
#pragma unroll
    for (int t = 0; t < kPoint16MaxTile / 2; ++t) {
        const int j = 2 * t + half;
        cx[t] = 0.f;
        cy[t] = 0.f;
        cz[t] = 1.f;  // points past the end run on a unit vector and are not sent
        if (2 * t < P && j < cnt) {
            cx[t] = xyz[3 * (p0 + j)];
            cy[t] = xyz[3 * (p0 + j) + 1];
            cz[t] = xyz[3 * (p0 + j) + 2];
        }
    }
#pragma unroll
    for (int t = 0; t < kPoint16MaxTile / 2; ++t) {
        if (2 * t >= P) break;
        const int j = 2 * t + half;
        float x = cx[t], y = cy[t], z = cz[t], r2, ir = 1.f;
        if (NORM) {
            unit_point(x, y, z, r2, ir);
        } else {
            r2 = x * x + y * y + z * z;
        }
        const int rr = r < 13 ? r : 12;
        float* rowp = rr == 0 ? s_v + size_t(j) * S
                              : (rr < 4 ? s_d + size_t(3 * j + rr - 1) * S : s_h + size_t(9 * j + rr - 4) * S);
        point16_core<L, NORM>(x, y, z, r2, tb, rr, ir, rowp, rowp, r < 13);
        if constexpr (MODE == 1) {
            if (bulk && r < 13 && j < cnt) {  // each lane sends the row it wrote
                fence_proxy_async_smem();
                float* g = rr == 0 ? sph + (p0 + j) * K
                                   : (rr < 4 ? dsph + ((p0 + j) * 3 + rr - 1) * K : ddsph + ((p0 + j) * 9 + rr - 4) * K);
                bulk_store(g, rowp, uint32_t(K * 4));
                bulk_commit();
            }
        }
    }
    if constexpr (MODE == 1) {
        if (bulk) {
            bulk_wait_read_all();
            __syncwarp();
            return;
        }
    }
    if (MODE != 0 || !bulk) {
        __syncwarp();
        warp_rows_out<K>(sph + p0 * K, s_v, cnt, S, lane);
        warp_rows_out<K>(dsph + p0 * 3 * K, s_d, 3 * cnt, S, lane);
        warp_rows_out<K>(ddsph + p0 * 9 * K, s_h, 9 * cnt, S, lane);
        __syncwarp();
        return;
    }
    // MODE 0 with bulk copies: the image of the three global ranges; the tile
    // start is 16-byte aligned (P is a multiple of the tile multiple)
    fence_proxy_async_smem();
    __syncwarp();
    const int64_t ev = int64_t(cnt) * K;
    const int64_t ev_b = (ev * 4) / 16 * 4, ed_b = (3 * ev * 4) / 16 * 4, eh_b = (9 * ev * 4) / 16 * 4;
    if (lane == 0) {
        if (ev_b) bulk_store(sph + p0 * K, s_v, uint32_t(ev_b * 4));
        if (ed_b) bulk_store(dsph + p0 * 3 * K, s_d, uint32_t(ed_b * 4));
        if (eh_b) bulk_store(ddsph + p0 * 9 * K, s_h, uint32_t(eh_b * 4));
        bulk_commit();
    }
    for (int64_t i = ev_b + lane; i < ev; i += 32) sph[p0 * K + i] = s_v[i];
    for (int64_t i = ed_b + lane; i < 3 * ev; i += 32) dsph[p0 * 3 * K + i] = s_d[i];
    for (int64_t i = eh_b + lane; i < 9 * ev; i += 32) ddsph[p0 * 9 * K + i] = s_h[i];
    if (lane == 0) bulk_wait_read_all();
    __syncwarp();
}

template <int L, bool NORM>
__global__ void __launch_bounds__(128, 3) point16_fwd_kernel(const float* __restrict__ xyz, int64_t n,
                                                          const __grid_constant__ PointTabs<L, float, true> tb,
                                                          float* __restrict__ sph, float* __restrict__ dsph,
                                                          float* __restrict__ ddsph, int P, int bulk) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    unsigned char* buf = smem + size_t(warp) * point16_warp_bytes<L>(P);
    const int64_t ntiles = (n + P - 1) / P;
    const int64_t stride = int64_t(gridDim.x) * W;
    for (int64_t tile = int64_t(blockIdx.x) * W + warp; tile < ntiles; tile += stride) {
        const int64_t p0 = tile * P;
        const int cnt = int(min(int64_t(P), n - p0));
        point16_tile<L, NORM>(xyz, sph, dsph, ddsph, p0, cnt, P, bulk, buf, tb, lane);
    }
    if (bulk) bulk_wait_all();  // every lane: rows may leave by per-lane copies
}

// ------------------- forward with Hessians, 10 lanes per point (distinct planes)
// POINT with lanes_per_point = 10 (FP32 values, gradients and Hessians): the
// 30 first lanes of a warp compute 3 points per pass, lane 10j + r owning the
// r-th distinct plane of point j (value, 3 gradient components, the Hessian
// entries xx, xy, xz, yy, yz, zz; lanes 30, 31 idle). The lane of an
// off-diagonal entry also writes its mirror, so no lane repeats another's
// work: 1.6x the points per warp instruction of the 16-lane map. The planes
// come from point16_core (the same role weights).
//
// Shared memory, odd K: the image of the tile's three global ranges, each
// placed at its 16-byte phase so that the interior leaves by one bulk copy
// per array (head and tail by plain stores). Even K (K % 4 == 0 in FP32):
// every row is 16-byte aligned at both ends, so each lane keeps only its
// distinct row (10 row slots per point at stride point4_stride) and sends it
// by one bulk copy per global row, the mirror from the same slot.
template <int L>
__host__ __device__ constexpr size_t point10_warp_bytes(int P) {
    constexpr int K = (L + 1) * (L + 1);
    if constexpr (K % 2) {
        const size_t v = (size_t(P) * K + 4 + 3) / 4 * 4, d = (size_t(3 * P) * K + 4 + 3) / 4 * 4,
                     h = (size_t(9 * P) * K + 4 + 3) / 4 * 4;
        return 4 * (v + d + h);
    } else {
        return size_t(4) * 10 * size_t(P) * size_t(point4_stride(L, 4));
    }
}

__host__ __device__ constexpr int point10_plane(int r) {  // distinct plane r -> index among the 13
    return r < 4 ? r : (r == 4 ? 4 : r == 5 ? 5 : r == 6 ? 6 : r == 7 ? 8 : r == 8 ? 9 : 12);
}
__host__ __device__ constexpr int point10_mirror(int q) {  // Hessian plane 4 + 3i + k -> 4 + 3k + i
    return q < 4 ? q : 4 + 3 * ((q - 4) % 3) + (q - 4) / 3;
}
__host__ __device__ constexpr int point10_slot(int q) {  // plane among the 13 -> its distinct row
    return q < 4 ? q : (q == 4 ? 4 : (q == 5 || q == 7) ? 5 : (q == 6 || q == 10) ? 6 : q == 8 ? 7 : (q == 9 || q == 11) ? 8 : 9);
}

// Sends elements [0, E) of a staged range (image element e at img[e], the
// range's global start g; img and g share their 16-byte phase): the
// 16-byte-aligned interior by one bulk copy from lane 0, the rest by plain
// stores of the warp. Returns whether a bulk copy was issued.
__device__ __forceinline__ bool point10_send(float* __restrict__ g, const float* __restrict__ img, int64_t E, int lane) {
    const int64_t h = (4 - int64_t((reinterpret_cast<uintptr_t>(g) / 4) % 4)) % 4;
    const int64_t nb = E > h ? (E - h) / 4 * 4 : 0;
    if (nb > 0 && lane == 0) bulk_store(g + h, img + h, uint32_t(nb * 4));
    for (int64_t i = lane; i < min(h, E); i += 32) g[i] = img[i];
    for (int64_t i = h + nb + lane; i < E; i += 32) g[i] = img[i];
    return nb > 0;
}

// One tile of P points (P a multiple of 3, <= 12): passes of 3 points.
template <int L, bool NORM, typename Tabs>
__device__ __forceinline__ void point10_tile(const float* __restrict__ xyz, float* __restrict__ sph,
                                             float* __restrict__ dsph, float* __restrict__ ddsph, int64_t p0,
                                             int cnt, int P, int bulk, unsigned char* buf, const Tabs& tb,
                                             int lane) {
    constexpr int K = (L + 1) * (L + 1);
    constexpr bool IMG = (K % 2) != 0;
    constexpr int S = IMG ? K : point4_stride(L, 4);
    const int j = min(lane / 10, 2);
    const int r = min(lane - 10 * j, 9);
    const bool on = lane < 30;
    const int rr = point10_plane(r), rm = point10_mirror(rr);
    float *iv = nullptr, *id = nullptr, *ih = nullptr;
    if constexpr (IMG) {
        float* const sv = reinterpret_cast<float*>(buf);
        float* const sd = sv + (size_t(P) * K + 4 + 3) / 4 * 4;
        float* const sh = sd + (size_t(3 * P) * K + 4 + 3) / 4 * 4;
        // each image shares the 16-byte phase of its global range
        iv = sv + (bulk ? (reinterpret_cast<uintptr_t>(sph + p0 * K) / 4) % 4 : 0);
        id = sd + (bulk ? (reinterpret_cast<uintptr_t>(dsph + p0 * 3 * K) / 4) % 4 : 0);
        ih = sh + (bulk ? (reinterpret_cast<uintptr_t>(ddsph + p0 * 9 * K) / 4) % 4 : 0);
    }
    float* const slots = reinterpret_cast<float*>(buf);  // even K: 10 row slots per point
    for (int t = 0; t < P; t += 3) {
        const int pj = t + j;
        const bool live = on && pj < cnt;
        float x = 0.f, y = 0.f, z = 1.f;  // idle lanes run on a unit vector and store nothing
        if (live) {
            x = xyz[3 * (p0 + pj)];
            y = xyz[3 * (p0 + pj) + 1];
            z = xyz[3 * (p0 + pj) + 2];
        }
        float r2, ir = 1.f;
        if (NORM) {
            unit_point(x, y, z, r2, ir);
        } else {
            r2 = x * x + y * y + z * z;
        }
        if constexpr (IMG) {
            float* rowp = rr == 0 ? iv + size_t(pj) * S
                                  : (rr < 4 ? id + size_t(3 * pj + rr - 1) * S : ih + size_t(9 * pj + rr - 4) * S);
            float* rowp2 = rr < 4 ? rowp : ih + size_t(9 * pj + rm - 4) * S;
            point16_core<L, NORM, true>(x, y, z, r2, tb, rr, ir, rowp, rowp2, live);
        } else {
            float* rowp = slots + size_t(10 * pj + r) * S;
            point16_core<L, NORM, false>(x, y, z, r2, tb, rr, ir, rowp, rowp, live);
            if (bulk && live) {  // rows 16-byte aligned at both ends: one copy per global row
                fence_proxy_async_smem();
                const int64_t gp = p0 + pj;
                float* g1 = rr == 0 ? sph + gp * K : (rr < 4 ? dsph + (gp * 3 + rr - 1) * K : ddsph + (gp * 9 + rr - 4) * K);
                bulk_store(g1, rowp, uint32_t(K * 4));
                if (rm != rr) bulk_store(ddsph + (gp * 9 + rm - 4) * K, rowp, uint32_t(K * 4));
                bulk_commit();
            }
        }
    }
    if constexpr (!IMG) {
        if (bulk) {
            bulk_wait_read_all();
            __syncwarp();
            return;
        }
        // outputs not 16-byte aligned: the warp copies the 13 global rows of
        // each point from their slots
        __syncwarp();
        for (int q = 0; q < 13 * cnt; ++q) {
            const int pj = q / 13, pl = q - 13 * pj;
            const int64_t gp = p0 + pj;
            float* g = pl == 0 ? sph + gp * K : (pl < 4 ? dsph + (gp * 3 + pl - 1) * K : ddsph + (gp * 9 + pl - 4) * K);
            const float* src = slots + size_t(10 * pj + point10_slot(pl)) * S;
            for (int c = lane; c < K; c += 32) g[c] = src[c];
        }
        __syncwarp();
        return;
    } else {
        fence_proxy_async_smem();
        __syncwarp();
        if (bulk) {
            bool any = point10_send(sph + p0 * K, iv, int64_t(cnt) * K, lane);
            any = point10_send(dsph + p0 * 3 * K, id, int64_t(3 * cnt) * K, lane) || any;
            any = point10_send(ddsph + p0 * 9 * K, ih, int64_t(9 * cnt) * K, lane) || any;
            if (lane == 0 && any) {
                bulk_commit();
                bulk_wait_read_all();
            }
        } else {
            for (int64_t i = lane; i < int64_t(cnt) * K; i += 32) sph[p0 * K + i] = iv[i];
            for (int64_t i = lane; i < int64_t(3 * cnt) * K; i += 32) dsph[p0 * 3 * K + i] = id[i];
            for (int64_t i = lane; i < int64_t(9 * cnt) * K; i += 32) ddsph[p0 * 9 * K + i] = ih[i];
        }
        __syncwarp();
    }
}

template <int L, bool NORM>
__global__ void __launch_bounds__(128, 3) point10_fwd_kernel(const float* __restrict__ xyz, int64_t n,
                                                             const __grid_constant__ PointTabs<L, float, true> tb,
                                                             float* __restrict__ sph, float* __restrict__ dsph,
                                                             float* __restrict__ ddsph, int P, int bulk) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    unsigned char* buf = smem + size_t(warp) * point10_warp_bytes<L>(P);
    const int64_t ntiles = (n + P - 1) / P;
    const int64_t stride = int64_t(gridDim.x) * W;
    for (int64_t tile = int64_t(blockIdx.x) * W + warp; tile < ntiles; tile += stride) {
        const int64_t p0 = tile * P;
        const int cnt = int(min(int64_t(P), n - p0));
        point10_tile<L, NORM>(xyz, sph, dsph, ddsph, p0, cnt, P, bulk, buf, tb, lane);
    }
    if (bulk) bulk_wait_all();  // every lane: rows may leave by per-lane copies
}

// ----------------------------------------------------------------- backward
// Loads the [cnt, K] tile of `src` at element offset `off` into `dst`: the
// 16-byte-multiple prefix by a bulk copy on `bar` (if `bulk`), the rest with
// plain loads at consumption time. Returns the number of bulk elements.
template <typename T>
__device__ __forceinline__ int64_t issue_tile_load(T* dst, const T* src, int64_t elems, int bulk, uint64_t* bar,
                                                   int lane) {
    int64_t eb = bulk ? (elems * int64_t(sizeof(T))) / 16 * 16 / int64_t(sizeof(T)) : 0;
    if (eb > 0 && lane == 0) {
        mbar_arrive_expect_tx(bar, uint32_t(eb * sizeof(T)));
        bulk_load(dst, src, uint32_t(eb * sizeof(T)), bar);
    }
    return eb;
}

constexpr uint32_t kWaitPolls = 1u << 22;  // bounded mbarrier wait (>> any real load latency)

// Sums over all columns of one point, sum_k g_k dY_k/dx_i, channel by channel.
// The columns +-m of degree l enter only through three combinations of the
// two upstream gradients,
//   A = g+ c_m + g- s_m,  B = g+ c_{m-1} + g- s_{m-1},  C = g- c_{m-1} - g+ s_{m-1},
// and the terms of Eq. iter-deri, summed over (l, m), are
//   P = sum e Q_{l-1}^{m+1} A,  Bq = sum m Q B,  Cq = sum m Q C,  Z = sum f Q_{l-1}^m A
// (Q = Qtilde_l^m, Q_{l-1} = Qtilde_{l-1}): the gradient is (x P + Bq, y P + Cq, Z).
// With DUAL the same sums are differentiated along the direction (dx, dy, dz):
//   dQ_l^m = (x dx + y dy) e Q_{l-1}^{m+1} + dz f Q_{l-1}^m,
//   dA = m (dx B + dy C),  dB, dC from dc_{m-1}, ds_{m-1} likewise,
// and every column's own derivative along that direction, dQ c_m + Q dc_m and
// dQ s_m + Q ds_m, goes to `orow` (which may be `row` itself: a column's upstream
// gradients are read before its outputs are written). That is
// the double backward (grad_xyz is the derivative of the gradient along v,
// grad_g the derivative of Y along v) without any Hessian entry: 37 operations
// per pair of columns (17 without DUAL) where the six Hessian entries of both
// columns and their products with g and v took about 130 (27).
// S = sum l Y g is the term of the normalized form.
template <typename T>
struct ChanSums {
    T P = T(0), Bq = T(0), Cq = T(0), Z = T(0), S = T(0);
    T dP = T(0), dB = T(0), dC = T(0), dZ = T(0), dS = T(0);
};

template <int L, bool NORM, bool DUAL, typename T, typename Tabs>
__device__ __forceinline__ void point_chan_sums(T x, T y, T z, T r2, T dx, T dy, T dz, const Tabs& tb,
                                                const T* row, T* orow, ChanSums<T>& a) {
    T c[L + 1], s[L + 1];
    point_cs<L>(x, y, c, s);
    const T w = DUAL ? x * dx + y * dy : T(0);
    T q1[L + 1], q2[L + 1], p1[L + 1];  // Qtilde_{l-1}^m, Qtilde_{l-2}^m, (DUAL) d Qtilde_{l-1}^m
#pragma unroll
    for (int m = 0; m <= L; ++m) q1[m] = q2[m] = p1[m] = T(0);
#pragma unroll
    for (int l = 0; l <= L; ++l) {
        T q[L + 1], p[L + 1];
        q[l] = tb.qll[l];
        if (l >= 1) q[l - 1] = tb.d[l] * z * q1[l - 1];
#pragma unroll
        for (int m = 0; m + 2 <= l; ++m) {  // Eq. iter-q, folded
            const int i = tri(l, m);
            q[m] = (tb.a[i] * z) * q1[m] - (tb.b[i] * r2) * q2[m];
        }
        T sl = T(0), dsl = T(0);  // sum over the degree of Y g, and its derivative
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            const int i = tri(l, m);
            const T E1 = (m + 1 <= l - 1) ? tb.e[i] * q1[m + 1] : T(0);
            const T Qz = (m <= l - 1) ? tb.fz[i] * q1[m] : T(0);
            // the multipliers of the m = 0 column carry its 1/sqrt2
            T dE1 = T(0), dQz = T(0), dq = T(0);
            if constexpr (DUAL) {
                dE1 = (m + 1 <= l - 1) ? tb.e[i] * p1[m + 1] : T(0);
                dQz = (m <= l - 1) ? tb.fz[i] * p1[m] : T(0);
                dq = w * E1 + dz * Qz;
            }
            const int k = l * l + l;
            if (m == 0) {
                const T g = row[k];
                a.P += E1 * g;
                a.Z += Qz * g;
                if (NORM) sl += (tb.inv_sqrt2 * q[0]) * g;
                if constexpr (DUAL) {
                    orow[k] = dq;
                    a.dP += dE1 * g;
                    a.dZ += dQz * g;
                    if (NORM) dsl += dq * g;
                    p[0] = dq * (T(2) * tb.inv_sqrt2);
                }
            } else {
                const T gp = row[k + m], gn = row[k - m];
                const T c1 = c[m - 1], s1 = s[m - 1];
                const T A = gp * c[m] + gn * s[m];
                const T B = gp * c1 + gn * s1;
                const T C = gn * c1 - gp * s1;
                const T mq = T(m) * q[m];
                a.P += E1 * A;
                a.Z += Qz * A;
                if (NORM || !DUAL) {  // the gradient itself
                    a.Bq += mq * B;
                    a.Cq += mq * C;
                }
                if (NORM) sl += q[m] * A;
                if constexpr (DUAL) {
                    const T mx = T(m) * dx, my = T(m) * dy;
                    const T dcm = mx * c1 - my * s1, dsm = mx * s1 + my * c1;
                    orow[k + m] = dq * c[m] + q[m] * dcm;
                    orow[k - m] = dq * s[m] + q[m] * dsm;
                    const T dA = mx * B + my * C;
                    const T mdq = T(m) * dq;
                    a.dP += dE1 * A + E1 * dA;
                    a.dZ += dQz * A + Qz * dA;
                    a.dB += mdq * B;
                    a.dC += mdq * C;
                    if (m >= 2) {
                        const T c2 = c[m >= 2 ? m - 2 : 0], s2 = s[m >= 2 ? m - 2 : 0];
                        const T nx = T(m - 1) * dx, ny = T(m - 1) * dy;
                        const T dc1 = nx * c2 - ny * s2, ds1 = nx * s2 + ny * c2;
                        a.dB += mq * (gp * dc1 + gn * ds1);
                        a.dC += mq * (gn * dc1 - gp * ds1);
                    }
                    if (NORM) dsl += dq * A + q[m] * dA;
                    p[m] = dq;
                }
            }
        }
        if (NORM) {
            a.S += T(l) * sl;
            if (DUAL) a.dS += T(l) * dsl;
        }
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            q2[m] = q1[m];
            q1[m] = q[m];
            if (DUAL) p1[m] = p[m];
        }
    }
}

// The same with outputs that are known to lie apart from the gradients.
template <int L, bool NORM, bool DUAL, typename T, typename Tabs>
__device__ __forceinline__ void point_chan_sums_apart(T x, T y, T z, T r2, T dx, T dy, T dz, const Tabs& tb,
                                                      const T* __restrict__ row, T* __restrict__ orow,
                                                      ChanSums<T>& a) {
    point_chan_sums<L, NORM, DUAL>(x, y, z, r2, dx, dy, dz, tb, row, orow, a);
}

// Row of the staged upstream-gradient tile. Odd K: the image of the global range
// (one bulk copy; an odd stride is free of bank conflicts). Even K (a multiple
// of 4): rows of K plus 16 bytes, every one 16-byte aligned, filled by 16-byte
// asynchronous copies; 32 lanes reading one column then meet 8 banks. (Padding
// such rows to K + 1 and filling them with plain loads, waited for before each
// tile, ran at 1.65 TB/s at l_max 7 and 0.9 at 11 where l_max 6 and 8 ran at 5.9.)
template <int L, typename T>
struct BwdRow {
    static constexpr int K = (L + 1) * (L + 1);
    static constexpr bool EVEN = K % 2 == 0;
    static constexpr int EL16 = 16 / int(sizeof(T));
    static constexpr int CR = K / EL16;  // 16-byte units of a row (even K)
    // l_max 1 in FP32: a row is one 16-byte unit, which its lane moves itself, in
    // rows of 5 words (4M points: 48 us through the asynchronous copies)
    static constexpr bool ONE = EVEN && CR == 1;
    static constexpr int S = ONE ? K + 1 : (EVEN ? K + EL16 : K);
};

template <int L, typename T>
__host__ __device__ constexpr size_t point_bwd_buf_bytes(int P) {
    return align16(size_t(P) * BwdRow<L, T>::S * sizeof(T));
}

// Tile buffers per warp: two (the next tile's gradients load during the current
// one) while that leaves room for ten warps on an SM; beyond, one, refilled
// after each tile with the next one prefetched into L2: full 32-point tiles
// and twice the warps count for more (the recursion bounds these l_max).
template <int L, typename T>
__host__ __device__ constexpr int point_bwd_bufs() {
    return 2 * point_bwd_buf_bytes<L, T>(32) <= 21 * 1024 ? 2 : 1;
}
// Whether the double backward stages grad_g in a buffer of its own (odd K,
// where three buffers fit the same room): no load waits for its copy out. At
// l_max 6 in place took 269..283 us against 267 (4M points).
template <int L, bool DBW, typename T>
__host__ __device__ constexpr bool point_bwd_apart() {
    return DBW && !BwdRow<L, T>::EVEN && 3 * point_bwd_buf_bytes<L, T>(32) <= 21 * 1024;
}
template <int L, bool DBW, typename T>
__host__ __device__ constexpr size_t point_bwd_warp_bytes(int P) {
    return (point_bwd_bufs<L, T>() + (point_bwd_apart<L, DBW, T>() ? 1 : 0)) * point_bwd_buf_bytes<L, T>(P) + 16;
}

// DBW = false: backward (dxyz). DBW = true: double backward (grad_g, grad_xyz);
// grad_g takes the place of g in the staged rows, or a buffer of its own.
// Shared memory per warp: the tile buffers and two mbarriers.
template <int L, bool NORM, bool DBW, typename T>
__global__ void __launch_bounds__(256) point_bwd_kernel(const T* __restrict__ xyz, const T* __restrict__ g,
                                                        const T* __restrict__ v, int64_t n,
                                                        const __grid_constant__ PointTabs<L, T, false> tb,
                                                        T* __restrict__ dxyz, T* __restrict__ grad_g,
                                                        T* __restrict__ grad_xyz, int P, int bulk_in,
                                                        int bulk_out, uint32_t* __restrict__ status) {
    using BR = BwdRow<L, T>;
    constexpr int K = BR::K;
    constexpr int NB = point_bwd_bufs<L, T>();
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    const size_t buf = point_bwd_buf_bytes<L, T>(P);
    unsigned char* base = smem + size_t(warp) * point_bwd_warp_bytes<L, DBW, T>(P);
    constexpr bool APART = point_bwd_apart<L, DBW, T>();
    T* const so = reinterpret_cast<T*>(base + NB * buf);  // APART: grad_g
    uint64_t* bar = reinterpret_cast<uint64_t*>(base + (NB + (APART ? 1 : 0)) * buf);

    if (lane == 0)
        for (int b = 0; b < NB; ++b) mbar_init(&bar[b], 1);
    fence_proxy_async_smem();
    __syncwarp();

    const int64_t ntiles = (n + P - 1) / P;
    const int64_t stride = int64_t(gridDim.x) * W;
    int64_t tile = int64_t(blockIdx.x) * W + warp;
    uint32_t phase = 0;    // bit b: parity of buffer b's next completion
    uint32_t pending = 0;  // bit b: a bulk load into buffer b is in flight
    bool failed = false;

    // Starts loading a tile into buffer b (free: its readers are past a
    // __syncwarp, bulk stores out of it have been waited for by lane 0).
    auto load = [&](int64_t t, int b) {
        const int64_t p0 = t * P;
        const int64_t cnt = min(int64_t(P), n - p0);
        T* dst = reinterpret_cast<T*>(base + b * buf);
        if constexpr (BR::EVEN && !BR::ONE) {
            if (bulk_in) {
                const T* src = g + p0 * K;
                const uint32_t d0 = smem_u32(dst);
                for (int i = lane; i < int(cnt) * BR::CR; i += 32)
                    cp_async16(d0 + uint32_t((i / BR::CR) * BR::S * int(sizeof(T)) + (i % BR::CR) * 16), src + i * BR::EL16);
            }
        } else if constexpr (!BR::EVEN) {
            if (issue_tile_load(dst, g + p0 * K, cnt * K, bulk_in, &bar[b], lane) > 0) pending |= 1u << b;
        }
    };

    if (tile < ntiles) load(tile, 0);
    cp_async_commit();
    int cur = 0;
    for (; tile < ntiles; tile += stride) {
        const int64_t p0 = tile * P;
        const int cnt = int(min(int64_t(P), n - p0));
        const int64_t nt = tile + stride;
        const int nxt = NB == 2 ? cur ^ 1 : 0;
        if constexpr (NB == 2) {
            if (DBW && !APART && lane == 0) bulk_wait_read_all();  // grad_g of the last tile has left the other buffer
            if (nt < ntiles) load(nt, nxt);
            cp_async_commit();
        } else if (bulk_in && lane == 0 && nt < ntiles) {
            const int64_t bytes = min(int64_t(P), n - nt * P) * K * int64_t(sizeof(T)) / 16 * 16;
            if (bytes > 0) bulk_prefetch_l2(g + nt * P * K, uint32_t(bytes));
        }
        T* const gt = reinterpret_cast<T*>(base + cur * buf);
        if constexpr (BR::EVEN) {
            if (bulk_in && BR::ONE) {
                if (lane < cnt) {
                    const float4 r = *reinterpret_cast<const float4*>(g + (p0 + lane) * K);
                    T* const row = gt + lane * BR::S;
                    row[0] = r.x;
                    row[1] = r.y;
                    row[2] = r.z;
                    row[3] = r.w;
                }
            } else if (bulk_in)
                cp_async_wait<NB - 1>();
            else
                warp_rows_in<K>(gt, g + p0 * K, cnt, BR::S, lane);
        } else {
            // Wait for this tile's bulk part, then load the remainder directly.
            if (pending & (1u << cur)) {
                bool ok = true;
                if (lane == 0) ok = mbar_wait_bounded(&bar[cur], (phase >> cur) & 1u, kWaitPolls);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (ok) {
                    phase ^= (1u << cur);
                    pending &= ~(1u << cur);
                } else {
                    if (lane == 0) atomicOr(status, kStatusLoadTimeout);
                    failed = true;
                }
            }
            if (failed) break;
            const int64_t ev = int64_t(cnt) * K;
            const int64_t eb = bulk_in ? ev * int64_t(sizeof(T)) / 16 * 16 / int64_t(sizeof(T)) : 0;
            for (int64_t i = eb + lane; i < ev; i += 32) gt[i] = g[p0 * K + i];
        }
        if (APART && lane == 0) bulk_wait_read_all();  // grad_g of the last tile has left its buffer
        __syncwarp();
        if (lane < cnt) {
            const int64_t p = p0 + lane;
            T x = xyz[3 * p], y = xyz[3 * p + 1], z = xyz[3 * p + 2];
            T r2, ir = T(1);
            if (NORM) {
                unit_point(x, y, z, r2, ir);
            } else {
                r2 = x * x + y * y + z * z;
            }
            T* const row = gt + size_t(lane) * BR::S;
            ChanSums<T> a;
            if constexpr (!DBW) {
                point_chan_sums<L, NORM, false>(x, y, z, r2, T(0), T(0), T(0), tb, row, row, a);
                T ax = x * a.P + a.Bq, ay = y * a.P + a.Cq, az = a.Z;
                if (NORM) {
                    ax = ir * (ax - x * a.S);
                    ay = ir * (ay - y * a.S);
                    az = ir * (az - z * a.S);
                }
                dxyz[3 * p] = ax;
                dxyz[3 * p + 1] = ay;
                dxyz[3 * p + 2] = az;
            } else {
                // direction of the derivative at the evaluated point: v, or
                // (normalized) that of u = x / r, (v - u (u.v)) / r
                T dx = v[3 * p], dy = v[3 * p + 1], dz = v[3 * p + 2], uv = T(0);
                if (NORM) {
                    uv = x * dx + y * dy + z * dz;
                    dx = ir * (dx - x * uv);
                    dy = ir * (dy - y * uv);
                    dz = ir * (dz - z * uv);
                }
                if constexpr (APART)
                    point_chan_sums_apart<L, NORM, true>(x, y, z, r2, dx, dy, dz, tb, row, so + size_t(lane) * BR::S, a);
                else
                    point_chan_sums<L, NORM, true>(x, y, z, r2, dx, dy, dz, tb, row, row, a);
                if (grad_xyz) {
                    T hx = dx * a.P + x * a.dP + a.dB;
                    T hy = dy * a.P + y * a.dP + a.dC;
                    T hz = a.dZ;
                    if (NORM) {  // of (1/r) (G - u S): d(1/r) = -(u.v) / r^2
                        const T gx = x * a.P + a.Bq - x * a.S;
                        const T gy = y * a.P + a.Cq - y * a.S;
                        const T gz = a.Z - z * a.S;
                        const T iu = ir * uv;
                        hx = ir * (hx - dx * a.S - x * a.dS - iu * gx);
                        hy = ir * (hy - dy * a.S - y * a.dS - iu * gy);
                        hz = ir * (hz - dz * a.S - z * a.dS - iu * gz);
                    }
                    grad_xyz[3 * p] = hx;
                    grad_xyz[3 * p + 1] = hy;
                    grad_xyz[3 * p + 2] = hz;
                }
            }
        }
        if constexpr (DBW) {
            if (grad_g) {
                T* const out = grad_g + p0 * K;
                const T* const src = APART ? so : gt;
                fence_proxy_async_smem();
                __syncwarp();
                if constexpr (BR::EVEN) {
                    if (bulk_out && BR::ONE) {
                        const T* const row = gt + lane * BR::S;
                        if (lane < cnt)
                            *reinterpret_cast<float4*>(out + lane * K) =
                                make_float4(float(row[0]), float(row[1]), float(row[2]), float(row[3]));
                    } else if (bulk_out) {
                        for (int i = lane; i < cnt * BR::CR; i += 32)
                            reinterpret_cast<float4*>(out)[i] = *reinterpret_cast<const float4*>(
                                gt + (i / BR::CR) * BR::S + (i % BR::CR) * BR::EL16);
                    } else {
                        warp_rows_out<K>(out, gt, cnt, BR::S, lane);
                    }
                } else {
                    const int64_t ev = int64_t(cnt) * K;
                    int64_t eo = 0;
                    if (bulk_out) {
                        eo = (ev * int64_t(sizeof(T))) / 16 * 16 / int64_t(sizeof(T));
                        if (lane == 0 && eo > 0) {
                            bulk_store(out, src, uint32_t(eo * sizeof(T)));
                            bulk_commit();
                        }
                    }
                    for (int64_t i = eo + lane; i < ev; i += 32) out[i] = src[i];
                }
            }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if constexpr (NB == 1) {
            if constexpr (DBW) {
                if (lane == 0) bulk_wait_read_all();
                __syncwarp();  // no lane refills the buffer (plain loads, g not 16-byte aligned) before grad_g has left it
            }
            if (nt < ntiles) load(nt, 0);
            cp_async_commit();
        }
        cur = nxt;
    }
    cp_async_wait<0>();
    if (pending && lane == 0) {
        // Loads issued but never observed (after a timeout) may still be in
        // flight: wait for them, bounded, before the shared memory goes away.
        for (int b = 0; b < NB; ++b)
            if (pending & (1u << b)) (void)mbar_wait_bounded(&bar[b], (phase >> b) & 1u, kWaitPolls);
    }
    if (DBW && lane == 0) bulk_wait_all();
    __syncwarp();
}

// ---------------------------------------------------------------- launchers
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Host-side launch cache, keyed by (kernel address, device): the largest
// dynamic shared-memory size already set on the kernel and the occupancy of
// the last (threads, smem) pair queried, so repeated launches skip the
// attribute call and the occupancy query.
struct LaunchEntry {
    int smem_set = 48 * 1024;
    long long occ_key = -1;  // (threads << 32) | smem of `occ`
    int occ = 0;
};

inline std::mutex& launch_cache_mutex() {
    static std::mutex m;
    return m;
}

inline LaunchEntry& launch_entry(const void* kern, int dev) {  // caller holds the mutex
    static std::map<std::pair<const void*, int>, LaunchEntry> cache;
    return cache[std::make_pair(kern, dev)];
}

inline int cache_device() {
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return d;
}

// Raise the dynamic shared-memory limit of `kern` once per device and size.
template <typename K>
inline cudaError_t ensure_smem(K kern, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    const void* f = reinterpret_cast<const void*>(kern);
    const int d = cache_device();
    std::lock_guard<std::mutex> lk(launch_cache_mutex());
    if (d >= 0 && launch_entry(f, d).smem_set >= int(bytes)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e == cudaSuccess && d >= 0) launch_entry(f, d).smem_set = int(bytes);
    return e;
}

template <typename K>
inline int grid_for(K kern, int threads, size_t smem, int64_t work_warps, int blocks_per_sm) {
    int bps = blocks_per_sm;
    if (bps <= 0) {
        const void* f = reinterpret_cast<const void*>(kern);
        const int d = cache_device();
        const long long key = (static_cast<long long>(threads) << 32) | static_cast<long long>(smem);
        int occ = 0;
        std::lock_guard<std::mutex> lk(launch_cache_mutex());
        LaunchEntry* c = d >= 0 ? &launch_entry(f, d) : nullptr;
        if (c && c->occ_key == key) {
            occ = c->occ;
        } else {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, threads, smem) != cudaSuccess) {
                cudaGetLastError();
                occ = 1;
            }
            if (c) {
                c->occ = occ;
                c->occ_key = key;
            }
        }
        bps = std::max(occ, 1);
    }
    const int W = threads / 32;
    int64_t want = ceil_div(work_warps, W);
    int64_t cap = int64_t(bps) * sm_count();
    return int(std::max<int64_t>(1, std::min(want, cap)));
}

template <int L, bool GRAD, bool HESS, bool NORM, typename T, typename TO, bool HC = false>
int launch_point_fwd(const FwdArgs& a) {
    static const PointTabs<L, T, HESS> tb = make_point_tabs<L, T, HESS>();
    const int P = a.launch.points_per_tile, W = a.launch.warps_per_block;
    const size_t smem = size_t(W) * point_fwd_warp_bytes<L, GRAD, HESS, TO>(P);
    auto kern = point_fwd_kernel<L, GRAD, HESS, NORM, T, TO, HC>;
    cudaError_t err = ensure_smem(kern, smem);
    if (err != cudaSuccess) return int(err);
    const int64_t ntiles = ceil_div(a.n, P);
    const int grid = grid_for(kern, 32 * W, smem, ntiles, a.launch.blocks_per_sm);
    const bool bulk = (reinterpret_cast<uintptr_t>(a.sph) % 16 == 0) &&
                      (!GRAD || reinterpret_cast<uintptr_t>(a.dsph) % 16 == 0) &&
                      (!HESS || reinterpret_cast<uintptr_t>(a.ddsph) % 16 == 0);
    kern<<<grid, 32 * W, smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const PointIn<T, TO>*>(a.xyz), a.n, tb, static_cast<TO*>(a.sph), static_cast<TO*>(a.dsph),
        static_cast<TO*>(a.ddsph), P, bulk ? 1 : 0);
    return int(cudaGetLastError());
}

// POINT forward with 4 lanes per point (values and gradients); P <= 8 and W
// resolved by the caller.
template <int L, bool NORM, typename T, typename TO>
int launch_point4_fwd(const FwdArgs& a) {
    static const PointTabs<L, T, false> tb = make_point_tabs<L, T, false>();
    const int P = a.launch.points_per_tile, W = a.launch.warps_per_block;
    const size_t smem = size_t(W) * point4_warp_bytes<L, TO>(P);
    auto kern = point4_fwd_kernel<L, NORM, T, TO>;
    cudaError_t err = ensure_smem(kern, smem);
    if (err != cudaSuccess) return int(err);
    const int64_t ntiles = ceil_div(a.n, P);
    const int grid = grid_for(kern, 32 * W, smem, ntiles, a.launch.blocks_per_sm);
    const bool bulk = (reinterpret_cast<uintptr_t>(a.sph) % 16 == 0) && (reinterpret_cast<uintptr_t>(a.dsph) % 16 == 0);
    kern<<<grid, 32 * W, smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const T*>(a.xyz), a.n, tb, static_cast<TO*>(a.sph), static_cast<TO*>(a.dsph), P, bulk ? 1 : 0);
    return int(cudaGetLastError());
}

// POINT forward with Hessians, 16 lanes per point (FP32); P (even, <= 8) and
// W resolved by the caller.
template <int L, bool NORM>
int launch_point16_fwd(const FwdArgs& a) {
    static const PointTabs<L, float, true> tb = make_point_tabs<L, float, true>();
    const int P = a.launch.points_per_tile, W = a.launch.warps_per_block;
    const size_t smem = size_t(W) * point16_warp_bytes<L>(P);
    auto kern = point16_fwd_kernel<L, NORM>;
    cudaError_t err = ensure_smem(kern, smem);
    if (err != cudaSuccess) return int(err);
    const int64_t ntiles = ceil_div(a.n, P);
    const int grid = grid_for(kern, 32 * W, smem, ntiles, a.launch.blocks_per_sm);
    const bool bulk = reinterpret_cast<uintptr_t>(a.sph) % 16 == 0 && reinterpret_cast<uintptr_t>(a.dsph) % 16 == 0 &&
                      reinterpret_cast<uintptr_t>(a.ddsph) % 16 == 0;
    kern<<<grid, 32 * W, smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const float*>(a.xyz), a.n, tb, static_cast<float*>(a.sph), static_cast<float*>(a.dsph),
        static_cast<float*>(a.ddsph), P, bulk ? 1 : 0);
    return int(cudaGetLastError());
}

// POINT forward with Hessians, 10 lanes per point (FP32); P (a multiple of 3,
// <= 12) and W resolved by the caller.
template <int L, bool NORM>
int launch_point10_fwd(const FwdArgs& a) {
    static const PointTabs<L, float, true> tb = make_point_tabs<L, float, true>();
    const int P = a.launch.points_per_tile, W = a.launch.warps_per_block;
    const size_t smem = size_t(W) * point10_warp_bytes<L>(P);
    auto kern = point10_fwd_kernel<L, NORM>;
    cudaError_t err = ensure_smem(kern, smem);
    if (err != cudaSuccess) return int(err);
    const int64_t ntiles = ceil_div(a.n, P);
    const int grid = grid_for(kern, 32 * W, smem, ntiles, a.launch.blocks_per_sm);
    const bool bulk = reinterpret_cast<uintptr_t>(a.sph) % 16 == 0 && reinterpret_cast<uintptr_t>(a.dsph) % 16 == 0 &&
                      reinterpret_cast<uintptr_t>(a.ddsph) % 16 == 0;
    kern<<<grid, 32 * W, smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const float*>(a.xyz), a.n, tb, static_cast<float*>(a.sph), static_cast<float*>(a.dsph),
        static_cast<float*>(a.ddsph), P, bulk ? 1 : 0);
    return int(cudaGetLastError());
}

template <int L, bool NORM, bool DBW, typename T>
int launch_point_bwd(const BwdArgs& a) {
    static const PointTabs<L, T, false> tb = make_point_tabs<L, T, false>();
    const int P = a.launch.points_per_tile;
    int W = a.launch.warps_per_block;
    const size_t per_warp = point_bwd_warp_bytes<L, DBW, T>(P);
    while (W > 1 && size_t(W) * per_warp > size_t(max_smem_optin())) --W;  // even K: rows wider than the shape's check
    const size_t smem = size_t(W) * per_warp;
    auto kern = point_bwd_kernel<L, NORM, DBW, T>;
    cudaError_t err = ensure_smem(kern, smem);
    if (err != cudaSuccess) return int(err);
    const int64_t ntiles = ceil_div(a.n, P);
    const int grid = grid_for(kern, 32 * W, smem, ntiles, a.launch.blocks_per_sm);
    const bool bulk_in = reinterpret_cast<uintptr_t>(a.g) % 16 == 0;
    const bool bulk_out = reinterpret_cast<uintptr_t>(a.grad_g) % 16 == 0;
    kern<<<grid, 32 * W, smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const T*>(a.xyz), static_cast<const T*>(a.g), static_cast<const T*>(a.v), a.n, tb,
        static_cast<T*>(a.dxyz), static_cast<T*>(a.grad_g), static_cast<T*>(a.grad_xyz), P, bulk_in ? 1 : 0,
        bulk_out ? 1 : 0, a.status);
    return int(cudaGetLastError());
}

}  // namespace sph
