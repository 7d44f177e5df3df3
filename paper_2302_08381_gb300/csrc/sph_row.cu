// ROW kernel family: FP32 forward (values, gradients) for 16 <= l_max <= 63
// whose global writes are long contiguous runs.
//
// On GB300 the write stream reaches the HBM roofline only in contiguous runs
// of about 1 KB or more (measured: scattered 128-byte runs reach ~0.8 TB/s,
// 512-byte runs ~3.2 TB/s, >= 1 KB runs ~6.2 TB/s). A kernel that writes one
// degree (2l+1 columns) of many output rows at a time cannot get there, so
// this family keeps each point's output rows in shared memory in windows of
// whole degrees (about 130..250 columns per plane) and sends every window
// with TMA bulk copies of 32-byte-aligned runs.
//
// Work decomposition (arXiv 2302.08381, Section 2): a group of 8 lanes owns a
// point, a warp owns 4 consecutive points. The degree l is the outer loop and
// is the same for the whole group; lane j owns the m channels m = j (mod 8),
// whose Qtilde_{l-1}^m, Qtilde_{l-2}^m (Eq. iter-q with the prefactors folded
// in, Appendix C) and c_m, s_m, c_{m-1}, s_{m-1} (Eq. iter-sc) stay in
// registers; the derivative identities of Eq. iter-deri need
// Qtilde_{l-1}^{m+1}, which the neighbouring lane holds and passes with a
// shuffle. At every degree the lanes of a group write 8 consecutive columns
// per side, so the shared-memory stores are conflict-free within a group.
//
// The translation unit is compiled twice: SPH_ROW_PART 0 instantiates the
// kernels for 3..5 channels per lane (l_max 16..47), 1 for 6..8 (48..63).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "sph_core.cuh"
#include "sph_internal.h"

#ifndef SPH_ROW_PART
#define SPH_ROW_PART 0
#endif

namespace sph {

namespace {

constexpr int kG = 8;         // lanes per point
constexpr int kPW = 32 / kG;  // points per warp
constexpr int kCap = 256;     // columns buffered before a window is sent (the backward's window size)

// Per output type, channel slots and window policy: elements per 32-byte
// sector, the plane buffer length (SE pre-slots for the row head, then kCap
// columns, or with MINRUN kCap - 1 columns plus one whole degree of at most
// 16 NCH - 1 columns plus a carried partial sector; a multiple of 16 bytes),
// and the distance between the buffers of consecutive points, which is 8
// four-byte words past a multiple of 32 so that the four point groups of a
// warp, each writing 8 consecutive columns, start 8 banks apart.
template <typename TO, int NCH, bool MINRUN>
struct RowGeom {
    static constexpr int SE = 32 / int(sizeof(TO));
    static constexpr int EL16 = 16 / int(sizeof(TO));
    static constexpr int BUF = MINRUN ? (SE + kCap + 16 * NCH + 8 + EL16 - 1) / EL16 * EL16 : SE + kCap;
    template <int NPL>
    __host__ __device__ static constexpr int point_stride() {
        constexpr int words = NPL * BUF * int(sizeof(TO)) / 4;
        constexpr int pad = ((8 - words % 32) + 32) % 32;  // words of padding
        return NPL * BUF + pad * 4 / int(sizeof(TO));
    }
};

template <typename TO, bool GRAD, int NCH, bool MINRUN>
__host__ __device__ constexpr size_t row_warp_bytes() {
    return size_t(kPW) * RowGeom<TO, NCH, MINRUN>::template point_stride<GRAD ? 4 : 1>() * sizeof(TO);
}

struct CSf {
    float c, s;
    __device__ __forceinline__ CSf times(const CSf& w) const {
        return CSf{fmaf(c, w.c, -(s * w.s)), fmaf(c, w.s, s * w.c)};
    }
};

// (x + i y)^e for 0 <= e < 8 from (x + i y)^1, ^2 and ^4: 9 complex products with
// the squares where powers step by step took 30, of the ~1,000 operations a
// tile's prologue and its degrees cost at l_max 20.
__device__ __forceinline__ CSf row_power(const CSf& w1, const CSf& w2, const CSf& w4, int e) {
    CSf r{(e & 1) ? w1.c : 1.f, (e & 1) ? w1.s : 0.f};
    const CSf r2 = r.times(w2);
    if (e & 2) r = r2;
    const CSf r4 = r.times(w4);
    if (e & 4) r = r4;
    return r;
}

// Calls f with the compile-time number of channel slots, kend + 1 <= N, that a
// degree uses: every slot but the last is then full (no lane masked, no
// branch), and the slots of a degree interleave. The backward is 4..10 % faster
// for it (l_max 20, 200k points: 175 -> 162 us; 30, 100k: 179 -> 167); the
// forward, with its eight stores per slot, is not (l_max 40..63 up to 10 % slower).
template <int N, int K = 0, typename F>
__device__ __forceinline__ void row_slots(int kend, F&& f) {
    if constexpr (K + 1 < N) {
        if (kend == K)
            f(std::integral_constant<int, K + 1>{});
        else
            row_slots<N, K + 1>(kend, f);
    } else {
        f(std::integral_constant<int, N>{});
    }
}

// Coefficients in shared memory, once per block: entry (degree, slot, lane) of
// the degrees 0..L and the NCH slots a lane uses, the float4 {A, B, S, e}
// entries first, then the floats f.
template <int NCH>
__host__ __device__ constexpr size_t row_table_bytes(int L) {
    return size_t(L + 1) * NCH * kRowLanes * (sizeof(float4) + sizeof(float));
}

// Starts the copy of the block's table (16-byte asynchronous copies of the
// block's threads); row_table_ready() before the first use.
template <int NCH>
__device__ __forceinline__ void row_table_load(unsigned char* __restrict__ dst, const float4* __restrict__ rowA,
                                               const float* __restrict__ rowF, int L) {
    constexpr int kA = NCH * kRowLanes;      // 16-byte units of one degree: {A, B, S, e}
    constexpr int kF = NCH * kRowLanes / 4;  // and f
    const uint32_t sA = smem_u32(dst), sF = sA + uint32_t((L + 1) * kA * 16);
    for (int i = threadIdx.x; i < (L + 1) * kA; i += blockDim.x)
        cp_async16(sA + 16 * i, rowA + (i / kA) * (kRowSlots * kRowLanes) + i % kA);
    const float4* const f4 = reinterpret_cast<const float4*>(rowF);
    for (int i = threadIdx.x; i < (L + 1) * kF; i += blockDim.x)
        cp_async16(sF + 16 * i, f4 + (i / kF) * (kRowSlots * kRowLanes / 4) + i % kF);
}
__device__ __forceinline__ void row_table_ready() {
    cp_async_wait_all();
    __syncthreads();
}

// Forward kernel. Per degree d and channel slot k (m = j + 8k) a lane runs
// one step of Eq. iter-q, then Eq. real-sh-cartesian and Eq. iter-deri for the
// columns d^2+d+m and d^2+d-m of every plane, stored through per-window plane
// pointers at compile-time offsets. The m = 0 column takes the same path with
// c_0 = 1/sqrt2 and s_0 = 0 (its -m stores land on the same column first and
// are overwritten).
//
// What bounds it: with 8 to 12 warps on an SM (the windows' shared memory), the
// latency and the number of each slot's instructions. So the coefficients
// come from shared memory, one slot ahead (from L1, one degree ahead, they
// cost 1.5 of 5.1 stall cycles per instruction at l_max 50, and the registers
// that held them one warp in five); one block per SM shares the table. And the
// derivatives are assembled on the Q side first,
//   dY/dx = X c_m + q c'_m,  X = x e Q_{d-1}^{m+1} - d u_x q,
// with c'_m = m c_{m-1} (and 1/r) folded into the kept c_{m-1}: 22 floating-point
// operations per slot instead of 30.
constexpr int kRowMaxWarps = 2;  // of an explicit launch shape
// bfloat16 rows take half the shared memory, so the registers are the limit (50k
// points, l_max 20: 79.7 us with 12 warps, 73.9 with 16; l_max 40, 244 with 10, 199 with 14).
template <typename TO>
SPH_HD constexpr int row_block_warps(int NCH) {
    if (sizeof(TO) == 2 && NCH <= 6) return NCH <= 5 ? 16 : 14;
    return NCH <= 5 ? 12 : (NCH == 6 ? 10 : (NCH == 7 ? 9 : 8));
}

template <typename TO, bool GRAD, bool NORM, int NCH, bool MINRUN>
__global__ void __launch_bounds__(32 * row_block_warps<TO>(NCH), 1) row_fwd_kernel(const float* __restrict__ xyz, int64_t n,
                                                      int L, const float4* __restrict__ rowA,
                                                      const float* __restrict__ rowF, float inv_sqrt2,
                                                      TO* __restrict__ sph, TO* __restrict__ dsph) {
    constexpr int NPL = GRAD ? 4 : 1;
    constexpr int SE = RowGeom<TO, NCH, MINRUN>::SE;
    constexpr int BUF = RowGeom<TO, NCH, MINRUN>::BUF;
    constexpr int PSTR = RowGeom<TO, NCH, MINRUN>::template point_stride<NPL>();
    constexpr int kRow = NCH * kRowLanes;  // table entries of one degree
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    const int g = lane / kG;  // point of the warp tile
    const int j = lane % kG;  // channel class m = j (mod 8)
    row_table_load<NCH>(smem, rowA, rowF, L);
    const float4* const tA = reinterpret_cast<const float4*>(smem) + j;
    const float* const tF = reinterpret_cast<const float*>(smem + size_t(L + 1) * kRow * sizeof(float4)) + j;
    TO* const pst = reinterpret_cast<TO*>(smem + row_table_bytes<NCH>(L)) + (size_t(warp) * kPW + g) * PSTR;
    const int64_t K = int64_t(L + 1) * (L + 1);
    const int64_t ntiles = (n + kPW - 1) / kPW;
    const int nb_lane = (lane & ~(kG - 1)) | ((j + 1) & (kG - 1));  // the lane holding channel m+1's class
    row_table_ready();

    for (int64_t tile = int64_t(blockIdx.x) * W + warp; tile < ntiles; tile += int64_t(gridDim.x) * W) {
        const int64_t p = tile * kPW + g;
        const bool live = p < n;
        float x = 0.f, y = 0.f, z = 0.f, ir = 1.f;
        if (live) {
            x = xyz[3 * p];
            y = xyz[3 * p + 1];
            z = xyz[3 * p + 2];
        }
        if (NORM) {
            const float rr = fmaf(x, x, fmaf(y, y, z * z));
            ir = rr > 0.f ? 1.f / sqrtf(rr) : 0.f;
            x *= ir;
            y *= ir;
            z *= ir;
        }
        const float r2 = fmaf(z, z, fmaf(x, x, y * y));

        // c_m + i s_m and m (c_{m-1} + i s_{m-1}) of the lane's channels m = j + 8k
        // (Eq. iter-sc); c_0 carries the 1/sqrt2 of the m = 0 column.
        float cm[NCH], sm[NCH], cm1[NCH], sm1[NCH];
        {
            const CSf xy{x, y};
            const CSf w2 = xy.times(xy), w4 = w2.times(w2), w8 = w4.times(w4);
            CSf a = row_power(xy, w2, w4, j), b = row_power(xy, w2, w4, (j + kG - 1) % kG);
            // (for j = 0, b is (x + i y)^7: channel 8k, k >= 1, needs (x + i y)^(8k-1))
#pragma unroll
            for (int k = 0; k < NCH; ++k) {
                const bool none = (j == 0 && k == 0);  // m = 0: no c_{m-1}
                cm[k] = none ? inv_sqrt2 : a.c;
                sm[k] = none ? 0.f : a.s;
                const float f = NORM ? float(j + kG * k) * ir : float(j + kG * k);
                cm1[k] = none ? 0.f : f * b.c;  // m c_{m-1} (/ r)
                sm1[k] = none ? 0.f : f * b.s;
                a = a.times(w8);
                if (!none) b = b.times(w8);
            }
        }
        float q1[NCH], q2[NCH];  // Qtilde_{l-1}^m, Qtilde_{l-2}^m
#pragma unroll
        for (int k = 0; k < NCH; ++k) q1[k] = q2[k] = 0.f;

        // Output rows of this point: plane 0 = sph row, planes 1..3 = dsph rows.
        // s[i] = first column held in the plane buffer (at slot SE); it is
        // 32-byte aligned in global memory, so every bulk copy starts and
        // (except at the row end) ends on a sector boundary.
        TO* grow[NPL];
        int s[NPL];
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            grow[i] = (i == 0) ? sph + p * K : dsph + p * 3 * K + (i - 1) * K;
            const int phase = int((reinterpret_cast<uintptr_t>(grow[i]) / sizeof(TO)) % SE);
            s[i] = (SE - phase) % SE;
        }

        const float xi = NORM ? x * ir : x, yi = NORM ? y * ir : y;

        int l = 0;
        bool first = true;
        while (l <= L) {
            // A window of whole degrees [l, lw), the same for every point of
            // the warp (the lanes shuffle across point groups): degrees are
            // added while the window fits kCap - SE + 1 new columns, or, with
            // MINRUN, until it holds at least that many (runs of >= kCap - SE
            // columns whatever the degree's width, in larger buffers).
            // Column c of plane i is staged at pst[i * BUF + SE - s[i] + c].
            TO* pp[NPL];  // + j: the +m columns
            TO* pn[NPL];  // - j: the -m columns
#pragma unroll
            for (int i = 0; i < NPL; ++i) {
                pp[i] = pst + (i * BUF + SE - s[i] + j);
                pn[i] = pst + (i * BUF + SE - s[i] - j);
            }
            int d = l;
            while (true) {
                const int ctr = d * d + d;
                const int kend = d / kG;  // channels m = j + 8k <= d need k <= d/8 (same for the whole warp)
                const float4* const dA = tA + d * kRow;
                const float* const dF = tF + d * kRow;
                float ax = 0.f, ay = 0.f, az = 0.f;
                if (NORM && GRAD) {
                    const float lir = float(d) * ir;
                    ax = lir * x;
                    ay = lir * y;
                    az = lir * z;
                }
                TO* qp[NPL];
                TO* qn_[NPL];
#pragma unroll
                for (int i = 0; i < NPL; ++i) {
                    qp[i] = pp[i] + ctr;
                    qn_[i] = pn[i] + ctr;
                }
                // Qtilde_{d-1}^{m+1} of slot k, from the lane that holds channel m + 1
                auto next_q = [&](int k) {
                    const float src = (j == 0) ? (k + 1 < NCH ? q1[k + 1 < NCH ? k + 1 : k] : 0.f) : q1[k];
                    return __shfl_sync(0xffffffffu, src, nb_lane);
                };
                float4 tn = dA[0];  // {A, B, S, e} of the next slot
                float fn = GRAD ? dF[0] : 0.f, qnn = GRAD ? next_q(0) : 0.f;
#pragma unroll
                for (int k = 0; k < NCH; ++k) {
                    if (k > kend) break;
                    const float4 t0 = tn;
                    const float f0 = fn, qnb = qnn;
                    if (k + 1 < NCH) {
                        tn = dA[(k + 1) * kRowLanes];
                        if (GRAD) {
                            fn = dF[(k + 1) * kRowLanes];
                            qnn = next_q(k + 1);
                        }
                    }
                    // zero for m > d: the table holds zeros there
                    const float q = fmaf(t0.x * z, q1[k], fmaf(-(t0.y * r2), q2[k], t0.z));
                    if (j + kG * k <= d) {
                        const float c = cm[k], sn = sm[k];
                        qn_[0][-kG * k] = OutConv<TO>::cv(q * sn);  // -m (sin) and +m (cos) columns
                        qp[0][kG * k] = OutConv<TO>::cv(q * c);
                        if (GRAD) {
                            // Eq. iter-deri (prefactors folded)
                            const float E1 = t0.w * qnb;  // e Qtilde_{l-1}^{m+1}
                            const float Qz = NORM ? (f0 * q1[k]) * ir : f0 * q1[k];
                            const float X = NORM ? fmaf(-ax, q, xi * E1) : xi * E1;
                            const float Y = NORM ? fmaf(-ay, q, yi * E1) : yi * E1;
                            const float Z = NORM ? fmaf(-az, q, Qz) : Qz;
                            const float mc1 = q * cm1[k], ms1 = q * sm1[k];
                            qn_[1 % NPL][-kG * k] = OutConv<TO>::cv(fmaf(X, sn, ms1));
                            qn_[2 % NPL][-kG * k] = OutConv<TO>::cv(fmaf(Y, sn, mc1));
                            qn_[3 % NPL][-kG * k] = OutConv<TO>::cv(Z * sn);
                            qp[1 % NPL][kG * k] = OutConv<TO>::cv(fmaf(X, c, mc1));
                            qp[2 % NPL][kG * k] = OutConv<TO>::cv(fmaf(Y, c, -ms1));
                            qp[3 % NPL][kG * k] = OutConv<TO>::cv(Z * c);
                        }
                    }
                    q2[k] = q1[k];
                    q1[k] = q;
                }
                ++d;
                if (d > L) break;
                if (MINRUN ? (d * d - l * l >= kCap - (SE - 1)) : ((d + 1) * (d + 1) - l * l > kCap - (SE - 1)))
                    break;
            }
            const int lw = d;

            // Send the window: per plane, the sector-aligned run [s, e) by one
            // bulk copy; the row head (first window) and the row tail (last
            // window) with plain stores; the rest (< one sector) is carried.
            const int c_hi = lw * lw;
            const bool last = lw > L;
            fence_proxy_async_smem();
            __syncwarp();
            int e[NPL];
#pragma unroll
            for (int i = 0; i < NPL; ++i) {
                const int run = last ? (c_hi - s[i]) * int(sizeof(TO)) / 16 * 16 / int(sizeof(TO))
                                     : (c_hi - s[i]) / SE * SE;
                e[i] = s[i] + max(run, 0);
            }
            if (live) {
                if (j == 0) {
#pragma unroll
                    for (int i = 0; i < NPL; ++i)
                        if (e[i] > s[i])
                            bulk_store(grow[i] + s[i], pst + i * BUF + SE, uint32_t((e[i] - s[i]) * sizeof(TO)));
                    bulk_commit();
                }
#pragma unroll
                for (int i = 0; i < NPL; ++i) {
                    if (first)
                        for (int c = j; c < s[i]; c += kG) grow[i][c] = pst[i * BUF + c - s[i] + SE];
                    if (last)
                        for (int c = e[i] + j; c < c_hi; c += kG) grow[i][c] = pst[i * BUF + c - s[i] + SE];
                }
                if (j == 0) bulk_wait_read_all();  // the buffers are reused below
            }
            __syncwarp();
            if (!last) {
#pragma unroll
                for (int i = 0; i < NPL; ++i) {
                    for (int c = e[i] + j; c < c_hi; c += kG) pst[i * BUF + c - e[i] + SE] = pst[i * BUF + c - s[i] + SE];
                    s[i] = e[i];
                }
                __syncwarp();
            }
            first = false;
            l = lw;
        }
    }
    if (j == 0) bulk_wait_all();
}

// ------------------------------------------------------------- backward
// Fused recompute-backward with the same decomposition: dxyz_i = sum_k g_k
// dY_k/dx_i (Eq. iter-deri), the recursion recomputed in registers, the
// upstream-gradient row of each point read in the same windows of whole
// degrees by TMA bulk loads (double buffered: the next window is in flight
// while the current one is used), the unaligned window edges by plain loads.
// Lane j accumulates its channels' terms; the 8 lanes of a point reduce with
// shuffles at the end. Every mbarrier wait is bounded; a timeout sets the
// device status word and skips the rest of the launch.
constexpr int kBPad = 4;                  // slots before a window's first 16-byte-aligned column
constexpr int kBBuf = kBPad + kCap + 8;   // floats per window buffer
constexpr uint32_t kRowWaitPolls = 1u << 22;

__host__ __device__ constexpr size_t row_bwd_warp_bytes() {
    return size_t(kPW) * 2 * kBBuf * sizeof(float) + size_t(kPW) * 2 * sizeof(uint64_t);
}

// Window of whole degrees starting at degree l: [l, lw).
__device__ __forceinline__ int row_window_end(int l, int L) {
    int lw = l + 1;
    while (lw <= L && (lw + 1) * (lw + 1) - l * l <= kCap - 7) ++lw;
    return lw;
}

// Starts loading the columns [c0, c1) of the upstream-gradient row `grow` into
// `buf` (column c at buf[c - s + kBPad], s = first 16-byte-aligned column >= c0):
// the aligned middle by one bulk copy completing on `bar` (issued by lane j = 0),
// the edges by plain loads of the group's lanes. Returns whether a bulk copy was issued.
__device__ __forceinline__ bool row_window_load(const float* __restrict__ grow, int c0, int c1, float* buf,
                                                uint64_t* bar, int j) {
    const int phase = int((reinterpret_cast<uintptr_t>(grow + c0) / sizeof(float)) % 4);
    const int s = c0 + (4 - phase) % 4;
    const int e = s + max(0, (c1 - s) / 4 * 4);
    const bool bulk = e > s;
    if (bulk && j == 0) {
        mbar_arrive_expect_tx(bar, uint32_t((e - s) * sizeof(float)));
        bulk_load(buf + kBPad, grow + s, uint32_t((e - s) * sizeof(float)), bar);
    }
    for (int c = c0 + j; c < min(s, c1); c += kG) buf[c - s + kBPad] = grow[c];
    for (int c = max(e, c0) + j; c < c1; c += kG) buf[c - s + kBPad] = grow[c];
    return bulk;
}

// Like the forward it is bound by the latency and number of each slot's
// instructions: coefficients from the block's shared table, one slot ahead,
// and the three sums of point_chan_sums (P = sum e Q_{d-1}^{m+1} A, Bq = sum
// m Q B, Cq = sum m Q C, with m folded into the kept c_{m-1}), 17
// floating-point operations per slot where assembling Qx, Qy, Qz took 26. The
// m = 0 column takes the general path with c_0 = 1/sqrt2, s_0 = 0.
constexpr int kRowBwdWarps = 16;

template <bool NORM, int NCH>
__global__ void __launch_bounds__(32 * kRowBwdWarps, 1) row_bwd_kernel(
    const float* __restrict__ xyz, const float* __restrict__ g, int64_t n, int L, const float4* __restrict__ rowA,
    const float* __restrict__ rowF, float inv_sqrt2, float* __restrict__ dxyz, uint32_t* __restrict__ status) {
    constexpr int kRow = NCH * kRowLanes;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    const int gi = lane / kG;  // point of the warp tile
    const int j = lane % kG;   // channel class m = j (mod 8)
    row_table_load<NCH>(smem, rowA, rowF, L);
    const float4* const tA = reinterpret_cast<const float4*>(smem) + j;
    const float* const tF = reinterpret_cast<const float*>(smem + size_t(L + 1) * kRow * sizeof(float4)) + j;
    unsigned char* wbase = smem + row_table_bytes<NCH>(L) + size_t(warp) * row_bwd_warp_bytes();
    float* const bufs = reinterpret_cast<float*>(wbase) + size_t(gi) * 2 * kBBuf;  // this point's two windows
    uint64_t* const bars =
        reinterpret_cast<uint64_t*>(wbase + size_t(kPW) * 2 * kBBuf * sizeof(float)) + 2 * gi;
    const int64_t K = int64_t(L + 1) * (L + 1);
    const int64_t ntiles = (n + kPW - 1) / kPW;
    const int nb_lane = (lane & ~(kG - 1)) | ((j + 1) & (kG - 1));

    if (j == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
    }
    fence_proxy_async_smem();
    row_table_ready();
    uint32_t parity = 0;   // bit b: phase of buffer b's next completion (same in the 8 lanes of a point)
    uint32_t pending = 0;  // bit b: a bulk load into buffer b is in flight
    bool failed = false;

    for (int64_t tile = int64_t(blockIdx.x) * W + warp; tile < ntiles && !failed; tile += int64_t(gridDim.x) * W) {
        const int64_t p = tile * kPW + gi;
        const bool live = p < n;
        float x = 0.f, y = 0.f, z = 0.f, ir = 1.f;
        if (live) {
            x = xyz[3 * p];
            y = xyz[3 * p + 1];
            z = xyz[3 * p + 2];
        }
        if (NORM) {
            const float rr = fmaf(x, x, fmaf(y, y, z * z));
            ir = rr > 0.f ? 1.f / sqrtf(rr) : 0.f;
            x *= ir;
            y *= ir;
            z *= ir;
        }
        const float r2 = fmaf(z, z, fmaf(x, x, y * y));
        const float* grow = g + (live ? p : 0) * K;

        float cm[NCH], sm[NCH], cm1[NCH], sm1[NCH];
        {
            const CSf xy{x, y};
            const CSf w2 = xy.times(xy), w4 = w2.times(w2), w8 = w4.times(w4);
            CSf a = row_power(xy, w2, w4, j), b = row_power(xy, w2, w4, (j + kG - 1) % kG);
#pragma unroll
            for (int k = 0; k < NCH; ++k) {
                const bool none = (j == 0 && k == 0);
                cm[k] = none ? inv_sqrt2 : a.c;
                sm[k] = none ? 0.f : a.s;
                cm1[k] = none ? 0.f : float(j + kG * k) * b.c;  // m c_{m-1}
                sm1[k] = none ? 0.f : float(j + kG * k) * b.s;
                a = a.times(w8);
                if (!none) b = b.times(w8);
            }
        }
        float q1[NCH], q2[NCH];
#pragma unroll
        for (int k = 0; k < NCH; ++k) q1[k] = q2[k] = 0.f;
        float P = 0.f, Bq = 0.f, Cq = 0.f, Z = 0.f, S = 0.f;

        // window 0 into buffer 0
        int l = 0, lw = row_window_end(0, L), buf = 0;
        if (live && row_window_load(grow, 0, lw * lw, bufs, &bars[0], j)) pending |= 1u;
        while (l <= L) {
            // next window into the other buffer (free: consumed before the last fence + sync)
            const int ln = lw, lwn = ln <= L ? row_window_end(ln, L) : ln;
            if (live && ln <= L && row_window_load(grow, ln * ln, lwn * lwn, bufs + (buf ^ 1) * kBBuf, &bars[buf ^ 1], j))
                pending |= 1u << (buf ^ 1);
            // this window's bulk part
            if (live && (pending & (1u << buf))) {
                if (mbar_wait_bounded(&bars[buf], (parity >> buf) & 1u, kRowWaitPolls)) {
                    parity ^= 1u << buf;
                    pending &= ~(1u << buf);
                } else {
                    if (j == 0) atomicOr(status, kStatusLoadTimeout);
                    failed = true;
                }
            }
            if (__any_sync(0xffffffffu, failed)) {
                failed = true;
                break;
            }
            __syncwarp();  // edge elements loaded by the other lanes
            const float* gb = bufs + buf * kBBuf;
            const int phase = int((reinterpret_cast<uintptr_t>(grow + l * l) / sizeof(float)) % 4);
            const int s0 = l * l + (4 - phase) % 4;  // column at gb[kBPad]
            for (int d = l; d < lw; ++d) {
                const int ctr = d * d + d;
                const int kend = d / kG;
                const float4* const dA = tA + d * kRow;
                const float* const dF = tF + d * kRow;
                const float* const gp0 = gb + (ctr - s0 + kBPad + j);  // + 8k: g of column ctr + m
                const float* const gn0 = gb + (ctr - s0 + kBPad - j);
                float sd = 0.f;
                row_slots<NCH>(kend, [&](auto ks) {
                    constexpr int KS = decltype(ks)::value;
                    float qn[KS];
#pragma unroll
                    for (int k = 0; k < KS; ++k) {
                        const float src = (j == 0) ? (k + 1 < NCH ? q1[k + 1 < NCH ? k + 1 : k] : 0.f) : q1[k];
                        qn[k] = __shfl_sync(0xffffffffu, src, nb_lane);
                    }
#pragma unroll
                    for (int k = 0; k < KS; ++k) {
                        const float4 t0 = dA[k * kRowLanes];
                        // zero for m > d: the table holds zeros there
                        const float q = fmaf(t0.x * z, q1[k], fmaf(-(t0.y * r2), q2[k], t0.z));
                        if (k + 1 < KS || j + kG * k <= d) {
                            const float gp = gp0[kG * k], gn = gn0[-kG * k];
                            const float A = fmaf(gp, cm[k], gn * sm[k]);        // g+ c_m + g- s_m
                            const float B = fmaf(gp, cm1[k], gn * sm1[k]);      // m (g+ c_{m-1} + g- s_{m-1})
                            const float Cc = fmaf(gn, cm1[k], -(gp * sm1[k]));  // m (g- c_{m-1} - g+ s_{m-1})
                            P = fmaf(t0.w * qn[k], A, P);
                            Bq = fmaf(q, B, Bq);
                            Cq = fmaf(q, Cc, Cq);
                            Z = fmaf(dF[k * kRowLanes] * q1[k], A, Z);
                            if (NORM) sd = fmaf(q, A, sd);
                        }
                        q2[k] = q1[k];
                        q1[k] = q;
                    }
                });
                if (NORM) S = fmaf(float(d), sd, S);
            }
            fence_proxy_async_smem();  // this buffer is rewritten by the async proxy two windows on
            __syncwarp();
            l = lw;
            lw = lwn;
            buf ^= 1;
        }
        if (failed) break;
        float ax = fmaf(x, P, Bq), ay = fmaf(y, P, Cq), az = Z;
        // reduce over the 8 lanes of the point
#pragma unroll
        for (int off = kG / 2; off > 0; off >>= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, off, kG);
            ay += __shfl_xor_sync(0xffffffffu, ay, off, kG);
            az += __shfl_xor_sync(0xffffffffu, az, off, kG);
            if (NORM) S += __shfl_xor_sync(0xffffffffu, S, off, kG);
        }
        if (live && j == 0) {
            if (NORM) {
                ax = ir * fmaf(-x, S, ax);
                ay = ir * fmaf(-y, S, ay);
                az = ir * fmaf(-z, S, az);
            }
            dxyz[3 * p] = ax;
            dxyz[3 * p + 1] = ay;
            dxyz[3 * p + 2] = az;
        }
    }
    if (pending && j == 0) {
        // loads issued but not observed (after a timeout) may still be in
        // flight: wait for them, bounded, before the shared memory goes away
        for (int b = 0; b < 2; ++b)
            if (pending & (1u << b)) (void)mbar_wait_bounded(&bars[b], (parity >> b) & 1u, kRowWaitPolls);
    }
    __syncwarp();
}

// Warps of the one block per SM: every one that fits (`fit`), but no more than
// the rounds of tiles need. With the largest block the last round can fall on few
// SMs (10k points, l_max 31, 2,500 tiles: 12 warps on each SM, then 57 SMs with 12
// more, 49.1 us; two rounds of 9 39.8; before the blocks of many warps 45.6).
int row_even_warps(int64_t tiles, int64_t fit) {
    const int64_t spread = (tiles + sm_count() - 1) / sm_count(), rounds = (spread + fit - 1) / fit;
    return int(std::max<int64_t>(1, (spread + rounds - 1) / std::max<int64_t>(rounds, 1)));
}

// The default: one such block per SM. An explicit shape of warps_per_block x
// blocks_per_sm runs as many warps on an SM, in one block that shares the table as
// long as they fit: a table for each of the caller's one- or two-warp blocks
// leaves room for few of them (50k points, normalized, 1 x 0, us: l_max 50 1048, in
// one block 405; 63 1679, 608).
struct RowShape {
    int W, grid;
    size_t smem;
};

int row_shape(const void* kern, int64_t n, int cap, size_t per_warp, size_t table, const sph_launch& s, RowShape* r) {
    const int64_t tiles = (n + kPW - 1) / kPW;
    const int64_t fit = std::min<int64_t>(cap, (size_t(max_smem_optin()) - table) / per_warp);
    const int64_t asked = int64_t(s.warps_per_block) * s.blocks_per_sm;  // 0: as many as fit
    r->W = row_even_warps(tiles, asked > 0 ? std::min(asked, fit) : fit);
    r->smem = table + size_t(r->W) * per_warp;
    if (r->smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(r->smem));
        if (e != cudaSuccess) return int(e);
    }
    int64_t bps = asked > 0 ? std::max<int64_t>(1, asked / r->W) : 0;
    if (bps == 0) {
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 32 * r->W, r->smem) != cudaSuccess) {
            cudaGetLastError();
            occ = 1;
        }
        bps = std::max(occ, 1);
    }
    r->grid = int(std::max<int64_t>(1, std::min<int64_t>((tiles + r->W - 1) / r->W, bps * sm_count())));
    return int(cudaSuccess);
}

template <typename TO, bool GRAD, bool NORM, int NCH, bool MINRUN>
int launch_row(const FwdArgs& a) {
    const float* rt = static_cast<const float*>(device_row_tables());
    if (!rt) return int(cudaErrorMemoryAllocation);
    auto kern = row_fwd_kernel<TO, GRAD, NORM, NCH, MINRUN>;
    const size_t per_warp = row_warp_bytes<TO, GRAD, NCH, MINRUN>(), table = row_table_bytes<NCH>(a.l_max);
    if (a.launch.warps_per_block > kRowMaxWarps) return int(cudaErrorInvalidConfiguration);
    RowShape r;
    const int e = row_shape(reinterpret_cast<const void*>(kern), a.n, row_block_warps<TO>(NCH), per_warp, table,
                            a.launch, &r);
    if (e != int(cudaSuccess)) return e;
    constexpr int kEntries = kRowLanes * kRowDegrees * kRowSlots;
    kern<<<r.grid, 32 * r.W, r.smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const float*>(a.xyz), a.n, a.l_max, reinterpret_cast<const float4*>(rt), rt + 4 * kEntries,
        float(host_tables().inv_sqrt2), static_cast<TO*>(a.sph), static_cast<TO*>(a.dsph));
    return int(cudaGetLastError());
}

template <bool NORM, int NCH>
int launch_row_bwd(const BwdArgs& a) {
    const float* rt = static_cast<const float*>(device_row_tables());
    if (!rt) return int(cudaErrorMemoryAllocation);
    auto kern = row_bwd_kernel<NORM, NCH>;
    const size_t per_warp = row_bwd_warp_bytes(), table = row_table_bytes<NCH>(a.l_max);
    RowShape r;
    const int e =
        row_shape(reinterpret_cast<const void*>(kern), a.n, kRowBwdWarps, per_warp, table, a.launch, &r);
    if (e != int(cudaSuccess)) return e;
    constexpr int kEntries = kRowLanes * kRowDegrees * kRowSlots;
    kern<<<r.grid, 32 * r.W, r.smem, static_cast<cudaStream_t>(a.stream)>>>(
        static_cast<const float*>(a.xyz), static_cast<const float*>(a.g), a.n, a.l_max,
        reinterpret_cast<const float4*>(rt), rt + 4 * kEntries, float(host_tables().inv_sqrt2), static_cast<float*>(a.dxyz), a.status);
    return int(cudaGetLastError());
}

template <int NCH>
int launch_row_bwd_flags(const BwdArgs& a) {
    return a.normalized ? launch_row_bwd<true, NCH>(a) : launch_row_bwd<false, NCH>(a);
}

// Window policy: launch.lanes_per_point 1 = windows that fit the buffer,
// 2 = windows of at least kCap - SE columns (MINRUN, larger buffers), 0 = by
// measurement on GB300 (60,000..300,000 points): FP32 rows with gradients
// keep the smaller buffers (more warps per SM), 4..13 % faster, except at l_max
// 40..52, where windows that fit hold two degrees (l_max 40: 4.92 -> 5.54 TB/s,
// 46: 4.90 -> 5.34, 50: 5.00 -> 5.18, 54: 4.87 -> 4.59); bf16 rows, half the
// shared memory, take the longer runs (up to +13 % at l_max 63).
inline bool row_minrun_default(int L, bool bf16) { return bf16 || (L >= 40 && L <= 52); }

template <typename TO, int NCH, bool MINRUN>
int launch_row_policy(const FwdArgs& a) {
    const bool grad = a.dsph != nullptr, norm = a.normalized != 0;
    if (grad)
        return norm ? launch_row<TO, true, true, NCH, MINRUN>(a) : launch_row<TO, true, false, NCH, MINRUN>(a);
    return norm ? launch_row<TO, false, true, NCH, MINRUN>(a) : launch_row<TO, false, false, NCH, MINRUN>(a);
}

template <typename TO, int NCH>
int launch_row_flags(const FwdArgs& a) {
    const int pol = a.launch.lanes_per_point;
    const bool minrun = pol == 2 || (pol == 0 && row_minrun_default(a.l_max, sizeof(TO) == 2));
    return minrun ? launch_row_policy<TO, NCH, true>(a) : launch_row_policy<TO, NCH, false>(a);
}

template <int NCH>
int launch_row_out(const FwdArgs& a) {
    if (a.out == SPH_OUT_BF16) return launch_row_flags<__nv_bfloat16, NCH>(a);
    return launch_row_flags<float, NCH>(a);
}

}  // namespace

#if SPH_ROW_PART == 0
int row_bwd_part0(const BwdArgs& a) {
    switch ((a.l_max + 1 + kG - 1) / kG) {
        case 3:
            return launch_row_bwd_flags<3>(a);
        case 4:
            return launch_row_bwd_flags<4>(a);
        default:
            return launch_row_bwd_flags<5>(a);
    }
}

int row_fwd_part0(const FwdArgs& a) {
    switch ((a.l_max + 1 + kG - 1) / kG) {
        case 3:
            return launch_row_out<3>(a);
        case 4:
            return launch_row_out<4>(a);
        default:
            return launch_row_out<5>(a);
    }
}
#else
int row_bwd_part1(const BwdArgs& a) {
    switch ((a.l_max + 1 + kG - 1) / kG) {
        case 6:
            return launch_row_bwd_flags<6>(a);
        case 7:
            return launch_row_bwd_flags<7>(a);
        default:
            return launch_row_bwd_flags<8>(a);
    }
}

int row_fwd_part1(const FwdArgs& a) {
    switch ((a.l_max + 1 + kG - 1) / kG) {
        case 6:
            return launch_row_out<6>(a);
        case 7:
            return launch_row_out<7>(a);
        default:
            return launch_row_out<8>(a);
    }
}
#endif

}  // namespace sph
