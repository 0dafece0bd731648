// RMSNorm QK-normalisation with a tangent, the step in front of the attention of the paper's transformer
// (Sec. 4 "semi-Lipschitz control": RMSNorm as QK-norm with a learnable scale; App. "Lipschitzness of
// RMSNorm" for the definition and the Jacobian), and its backward pass.  Per row x in R^d:
//     r = sqrt(mean(x^2) + eps),  u = x / r,  y = g u,  ty = g (tx / r - u (u . tx) / (d r))
// One launch normalises Q and K, primal and tangent.  Pure streaming work (each tensor is read or written
// once), bound by HBM once enough bytes are in flight.  A row of cpr 16-byte chunks is shared by P lanes with
// C chunks each (rms_split: d = 72 is 3 x 3, d = 64 is 4 x 2, d = 128 is 4 x 4 or 8 x 2): with one chunk per lane
// (nine lanes a row at d = 72) every row sum cost nine shuffles for three rows of a warp and a thread had 32 or 64
// bytes in flight; with three it costs three for ten rows and 96 or 192 bytes.  Chunk k of lane c is c + P k, so that
// one instruction still touches P * 16 contiguous bytes of a row.
// Measured on B200 (B 16, H 16, N 1024, d 72: 302 and 453 MB): forward 87 -> 55 us (5.5 TB/s), backward with its
// reduction 241 -> 98 us (4.6 TB/s); d = 64, N = 1024, B 64: 221 -> 175 and 496 -> 263 us (6.1 TB/s).  Staging the rows
// through shared memory by bulk copies instead measured 65 and 116 us at d = 72 (1440 bytes a copy).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "geometry.cuh"
#include "sm100_ptx.cuh"

namespace tvm_attn {

constexpr int RMS_THREADS = 256;
constexpr int RMS_BWD_THREADS = 128;
// Blocks of a launch at most, both sides together: what B200's 148 SMs hold at the kernels' register counts, so that every
// block walks over its rows from the start to the end of the launch.  The backward's number is fixed for one more reason: the
// partial sums of dg, a row per block, have a size and a summation order that do not depend on the device.
constexpr int RMS_FWD_BLOCKS = 148 * 3;
constexpr int RMS_BWD_BLOCKS = 148 * 5;
constexpr int RMS_PARTIAL_ROWS = 2 * 592;   // rows of d floats in the workspace (more than RMS_BWD_BLOCKS)

template <typename T> struct RmsVec;
template <> struct RmsVec<float> { static constexpr int N = 4; };
template <> struct RmsVec<__nv_bfloat16> { static constexpr int N = 8; };

// A 16-byte chunk as pairs of floats in 64-bit registers, the operands of the two-wide fp32 instructions: the kernels
// spend half of the issue slots there are at full bandwidth on conversions and FMAs, one element at a time.
__device__ __forceinline__ void rms_unpack(const uint4& q, uint64_t (&v)[2]) {
    v[0] = ptx::pack2u(q.x, q.y);
    v[1] = ptx::pack2u(q.z, q.w);
}
__device__ __forceinline__ void rms_unpack(const uint4& q, uint64_t (&v)[4]) {   // a bf16 is the upper half of its float
    v[0] = ptx::pack2u(q.x << 16, q.x & 0xffff0000u);
    v[1] = ptx::pack2u(q.y << 16, q.y & 0xffff0000u);
    v[2] = ptx::pack2u(q.z << 16, q.z & 0xffff0000u);
    v[3] = ptx::pack2u(q.w << 16, q.w & 0xffff0000u);
}
// A 16-byte chunk as loaded.
template <typename T>
struct RmsRaw {
    uint4 q;
    __device__ __forceinline__ void load(const T* p) { q = __ldg(reinterpret_cast<const uint4*>(p)); }
    __device__ __forceinline__ void zero() { q = make_uint4(0, 0, 0, 0); }
    __device__ __forceinline__ void get(uint64_t (&v)[RmsVec<T>::N / 2]) const { rms_unpack(q, v); }
    // Ends the reuse of an earlier unpacking: the next get() unpacks again (one instruction an element) instead of
    // holding twice the registers across the row sums.
    __device__ __forceinline__ void repack() { asm volatile("" : "+r"(q.x), "+r"(q.y), "+r"(q.z), "+r"(q.w)); }
};
__device__ __forceinline__ void rms_store(float* p, const uint64_t (&v)[2]) {
    float4 q;
    ptx::unpack2(v[0], q.x, q.y);
    ptx::unpack2(v[1], q.z, q.w);
    *reinterpret_cast<float4*>(p) = q;
}
__device__ __forceinline__ void rms_store(__nv_bfloat16* p, const uint64_t (&v)[4]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float lo, hi;
        ptx::unpack2(v[i], lo, hi);
        w[i] = ptx::pack_bf16(lo, hi);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
template <int N>
__device__ __forceinline__ void rms_scale(const float* g, uint64_t (&v)[N]) {   // g: 16-byte aligned, shared memory
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(g + 2 * i);
        v[i] = q.x; v[i + 1] = q.y;
    }
}
__device__ __forceinline__ float rms_hsum(uint64_t v) {
    float lo, hi;
    ptx::unpack2(v, lo, hi);
    return lo + hi;
}

// How the cpr 16-byte chunks of a row are split: C chunks on each of P lanes.  The largest C <= cmax that divides cpr and
// leaves three lanes or more (48 contiguous bytes per row and instruction), or two with up to three chunks each of rows of whole
// 32-byte sectors; if none does (bf16 d = 40, 56, 88, 104), the largest whose last lane has one chunk less: a row's sums and
// scalars cost a warp as much for one chunk a lane as for three.  Measured with bf16 (16, 16, 1024), us: one chunk a lane / as
// here: backward d = 32 49.4 / 40.0, 40 67.9 / 60.8, 56 106.7 / 74.4, 88 231 / 115; forward d = 32 26.7 / 24.6, 40 36.7 / 36.3,
// 56 51.3 / 44.8, 88 97 / 73.  Two lanes instead of three or four: d = 48 forward 38.4 -> 36.9, backward 63.1 -> 59.5; with
// four chunks each, d = 64 forward 45.3 -> 53.2.
struct RmsSplit { int C, P; };
constexpr RmsSplit rms_split(int cpr, int cmax) {
    for (int waste = 0; waste < 2; ++waste)
        for (int c = cmax; c > 1; --c) {
            const int p = (cpr + c - 1) / c;
            if (c * p - cpr == waste && (p >= 3 || (p == 2 && c <= 3 && cpr % 2 == 0))) return {c, p};
        }
    return {1, cpr};
}

// Whether some head dim has its rows split into C chunks a lane, a last lane with one less among them or not.
template <typename T>
constexpr bool rms_split_exists(int cmax, int C, bool ragged) {
    for (int d = 8; d <= 128; d += 8) {
        const int cpr = d * (int)sizeof(T) / 16;
        const RmsSplit s = rms_split(cpr, cmax);
        if (s.C == C && (s.C * s.P > cpr) == ragged) return true;
    }
    return false;
}

// Row groups of a warp in flight in the forward: with one chunk per lane (d = 8, 16, 24) a thread would have two 16-byte loads in
// flight.  Four groups against one, (16, 16, 1024): d = 24 20.5 us against 23.9, d = 8 and 16 equal (9.1 and 12.3).
__host__ __device__ constexpr int rms_fwd_groups(int C) { return C == 1 ? 4 : 1; }

// Sum of v over the P consecutive lanes that share a row, returned to all of them, the same bits on each.
__device__ __forceinline__ float rms_group_sum(float v, int P, int lane, int first) {
    if ((P & (P - 1)) == 0) {
        for (int off = P >> 1; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        return v;
    }
    float acc = __shfl_sync(0xffffffffu, v, first);
    for (int k = 1; k < P; ++k) acc += __shfl_sync(0xffffffffu, v, first + k);
    return acc;
}

// The rows of one side in the order they lie in memory: index i -> element offset, for at most three dimensions
// (n0 innermost).  Dense tensors, packed or (B, rows, H, d), are one dimension of B * H * rows rows.
struct RmsRows {
    unsigned n0, n1;
    long long s0, s1, s2;
    unsigned total;   // B * H * rows per head
    __device__ __forceinline__ size_t offset(unsigned i) const {
        if (n0 == total) return (size_t)i * (size_t)s0;
        const unsigned a = i / n0, i0 = i - a * n0, b = a / n1, i1 = a - b * n1;
        return (size_t)i0 * (size_t)s0 + (size_t)i1 * (size_t)s1 + (size_t)b * (size_t)s2;
    }
};

// The chunks of a lane; the last one reads as zero where there is none.
template <typename T, int C>
__device__ __forceinline__ void rms_load(RmsRaw<T> (&r)[C], const T* p, int P, bool full) {
#pragma unroll
    for (int i = 0; i < C; ++i) {
        if (i == C - 1 && !full) r[i].zero();
        else r[i].load(p + P * i * RmsVec<T>::N);
    }
}

template <typename T>
struct RmsFwdSide {
    const T* x; const T* tx; const float* g; T* y; T* ty;
    RmsRows rows;
};

// Forward for both sides: blocks 0 .. nbq - 1 walk over the rows of Q, the others over those of K.  P = lanes per row;
// a warp has U groups of 32 / P rows in flight (few chunks per lane: more groups).
template <typename T, int C, bool RAGGED>
__global__ void __launch_bounds__(RMS_THREADS, 3)
qk_rmsnorm_jvp_fwd_kernel(const RmsFwdSide<T> q, const RmsFwdSide<T> k, int nbq, int d, int P, float eps) {
    constexpr int V = RmsVec<T>::N, U = rms_fwd_groups(C);
    __shared__ __align__(16) float scale[144];   // (16 more: where a lane has no last chunk) in shared memory: its 8 C registers a thread are worth a third of the warps
    const bool is_q = (int)blockIdx.x < nbq;
    const RmsFwdSide<T>& a = is_q ? q : k;
    const unsigned block = is_q ? blockIdx.x : blockIdx.x - nbq, nblocks = is_q ? nbq : gridDim.x - nbq;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rpw = 32 / P;
    const int sub = lane / P, c = lane - sub * P, first = sub * P;
    const bool full = !RAGGED || (c + P * (C - 1)) * V < d;   // the lane has C chunks of its row (else C - 1)
    for (int j = threadIdx.x; j < 144; j += RMS_THREADS) scale[j] = j < d ? a.g[j] : 0.f;
    __syncthreads();
    const float inv_d = 1.0f / (float)d;
    const unsigned rows_per_block = (RMS_THREADS / 32) * U * rpw, total = a.rows.total;
    for (unsigned base = block * rows_per_block; base < total; base += nblocks * rows_per_block) {
        RmsRaw<T> xr[U][C], tr[U][C];
        size_t off[U];
        bool act[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned row = base + (warp * U + u) * rpw + sub;
            act[u] = sub < rpw && row < total;
            off[u] = act[u] ? a.rows.offset(row) + (size_t)c * V : 0;
            rms_load(xr[u], a.x + off[u], P, full);
            rms_load(tr[u], a.tx + off[u], P, full);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint64_t ss2 = 0ull, s2 = 0ull;
#pragma unroll
            for (int i = 0; i < C; ++i) {
                uint64_t x[V / 2], t[V / 2];
                xr[u][i].get(x); tr[u][i].get(t);
#pragma unroll
                for (int e = 0; e < V / 2; ++e) { ss2 = ptx::fma2(x[e], x[e], ss2); s2 = ptx::fma2(x[e], t[e], s2); }
            }
            const float ss = rms_group_sum(rms_hsum(ss2), P, lane, first);
            const float s = rms_group_sum(rms_hsum(s2), P, lane, first);
            const float inv = 1.0f / sqrtf(ss / (float)d + eps);
            const float m = s * inv * inv * inv_d;   // (u . tx) / (d r)
            const uint64_t inv2 = ptx::pack2(inv, inv), nm2 = ptx::pack2(-m, -m);
            if (act[u]) {
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    uint64_t x[V / 2], t[V / 2], g[V / 2], y[V / 2], ty[V / 2];
                    xr[u][i].repack(); tr[u][i].repack();
                    xr[u][i].get(x); tr[u][i].get(t);
                    if (i == C - 1 && !full) continue;
                    rms_scale(scale + (c + P * i) * V, g);
#pragma unroll
                    for (int e = 0; e < V / 2; ++e) {
                        const uint64_t w = ptx::mul2(x[e], inv2);
                        y[e] = ptx::mul2(g[e], w);
                        ty[e] = ptx::mul2(g[e], ptx::fma2(w, nm2, ptx::mul2(t[e], inv2)));
                    }
                    rms_store(a.y + off[u] + P * i * V, y);
                    rms_store(a.ty + off[u] + P * i * V, ty);
                }
            }
        }
    }
}

template <typename T>
struct RmsBwdSide {
    const T* x; const T* tx; const float* g; const T* dy; const T* dty; T* dx; T* dtx;
    float* partial;   // [blocks of this side][d] partial sums of dg
    RmsRows rows;
};

// Backward for both sides.  With a = g dy, b = g dty and the row sums ss = x.x, s = x.tx, ax = a.x, bx = b.x,
// bt = b.tx:
//     dtx = (b - u (b.u)/d) / r
//     dx  = (a - u (a.u)/d) / r - (bt x + s b + bx tx) / (d r^3) + 3 bx s x / (d^2 r^5)
//     dg += dy u + dty (tx / r - u s / (d r^2))
// Each block walks over its rows with a fixed stride, every thread keeping the dg terms of its own columns; the
// block then adds them up in a fixed order and writes one partial row; a second kernel adds the partial rows, again
// in a fixed order, so dg is bit-reproducible.
template <typename T, int C, bool RAGGED>
__global__ void __launch_bounds__(RMS_BWD_THREADS, 5)
qk_rmsnorm_jvp_bwd_kernel(const RmsBwdSide<T> q, const RmsBwdSide<T> k, int nbq, int d, int P, float eps) {
    constexpr int V = RmsVec<T>::N;
    __shared__ __align__(16) float part[(RMS_BWD_THREADS / 32) * 32 * C * V];   // [warp][row in warp][column]; rows per warp * d <= 32 * C * V
    const bool is_q = (int)blockIdx.x < nbq;
    const RmsBwdSide<T>& a = is_q ? q : k;
    const unsigned block = is_q ? blockIdx.x : blockIdx.x - nbq, nblocks = is_q ? nbq : gridDim.x - nbq;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rpw = 32 / P;
    const int sub = lane / P, c = lane - sub * P, first = sub * P;
    const bool full = !RAGGED || (c + P * (C - 1)) * V < d;   // the lane has C chunks of its row (else C - 1)
    __shared__ __align__(16) float scale[144];   // (16 more: where a lane has no last chunk)
    for (int j = threadIdx.x; j < 144; j += RMS_BWD_THREADS) scale[j] = j < d ? a.g[j] : 0.f;
    __syncthreads();
    uint64_t dg[C][V / 2];
#pragma unroll
    for (int i = 0; i < C; ++i)
#pragma unroll
        for (int e = 0; e < V / 2; ++e) dg[i][e] = 0ull;
    const float fd = (float)d, inv_d = 1.0f / fd;
    const unsigned rows_per_block = (RMS_BWD_THREADS / 32) * rpw, total = a.rows.total;
    for (unsigned base = block * rows_per_block; base < total; base += nblocks * rows_per_block) {
        const unsigned row = base + warp * rpw + sub;
        const bool act = sub < rpw && row < total;
        const size_t off = act ? a.rows.offset(row) + (size_t)c * V : 0;
        RmsRaw<T> xr[C], tr[C], yr[C], zr[C];   // kept as loaded: a quarter of a thread's registers, not half
        rms_load(xr, a.x + off, P, full);
        rms_load(tr, a.tx + off, P, full);
        rms_load(yr, a.dy + off, P, full);
        rms_load(zr, a.dty + off, P, full);
        uint64_t ss2 = 0ull, s2 = 0ull, ax2 = 0ull, bx2 = 0ull, bt2 = 0ull;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            uint64_t x[V / 2], t[V / 2], gy[V / 2], gt[V / 2], g[V / 2];
            xr[i].get(x); tr[i].get(t); yr[i].get(gy); zr[i].get(gt);
            rms_scale(scale + (c + P * i) * V, g);
#pragma unroll
            for (int e = 0; e < V / 2; ++e) {
                const uint64_t ai = ptx::mul2(g[e], gy[e]), bi = ptx::mul2(g[e], gt[e]);
                ss2 = ptx::fma2(x[e], x[e], ss2);
                s2 = ptx::fma2(x[e], t[e], s2);
                ax2 = ptx::fma2(ai, x[e], ax2);
                bx2 = ptx::fma2(bi, x[e], bx2);
                bt2 = ptx::fma2(bi, t[e], bt2);
            }
        }
        const float ss = rms_group_sum(rms_hsum(ss2), P, lane, first);
        const float s = rms_group_sum(rms_hsum(s2), P, lane, first);
        const float ax = rms_group_sum(rms_hsum(ax2), P, lane, first);
        const float bx = rms_group_sum(rms_hsum(bx2), P, lane, first);
        const float bt = rms_group_sum(rms_hsum(bt2), P, lane, first);
        const float inv = 1.0f / sqrtf(ss / fd + eps);
        const float inv2 = inv * inv, k3 = inv2 * inv * inv_d;
        const float m = s * inv2 * inv_d;
        const float kx = 3.0f * k3 * bx * s * inv2 * inv_d - k3 * bt;  // coefficient of x in the terms that differentiate J
        // dtx = inv b - (inv^2 (b.u)/d) x;  dx = inv a + (kx - inv^2 (a.u)/d) x - k3 s b - k3 bx tx
        const float xdt = -bx * inv * inv_d * inv2, xdx = kx - ax * inv * inv_d * inv2;
        const uint64_t I2 = ptx::pack2(inv, inv), M2 = ptx::pack2(-m * inv, -m * inv), A2 = ptx::pack2(xdt, xdt), B2 = ptx::pack2(xdx, xdx);
        const uint64_t S2 = ptx::pack2(-k3 * s, -k3 * s), T2 = ptx::pack2(-k3 * bx, -k3 * bx);
        if (act) {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                uint64_t x[V / 2], t[V / 2], gy[V / 2], gt[V / 2], g[V / 2], dx[V / 2], dtx[V / 2];
                if (i == C - 1 && !full) continue;
                xr[i].repack(); tr[i].repack(); yr[i].repack(); zr[i].repack();
                xr[i].get(x); tr[i].get(t); yr[i].get(gy); zr[i].get(gt);
                rms_scale(scale + (c + P * i) * V, g);
#pragma unroll
                for (int e = 0; e < V / 2; ++e) {
                    const uint64_t ai = ptx::mul2(g[e], gy[e]), bi = ptx::mul2(g[e], gt[e]);
                    dtx[e] = ptx::fma2(bi, I2, ptx::mul2(x[e], A2));
                    dx[e] = ptx::fma2(ai, I2, ptx::fma2(x[e], B2, ptx::fma2(bi, S2, ptx::mul2(t[e], T2))));
                    // dy u + dty (tx / r - u m), u = x / r
                    const uint64_t jt = ptx::fma2(x[e], M2, ptx::mul2(t[e], I2));
                    dg[i][e] = ptx::add2(dg[i][e], ptx::fma2(gt[e], jt, ptx::mul2(gy[e], ptx::mul2(x[e], I2))));
                }
                rms_store(a.dx + off + P * i * V, dx);
                rms_store(a.dtx + off + P * i * V, dtx);
            }
        }
    }
    // the reduction may be launched: its blocks wait for this grid's end before they read anything
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // ---- dg of the block, in a fixed order
    if (sub < rpw) {
#pragma unroll
        for (int i = 0; i < C; ++i) {
            if (i == C - 1 && !full) continue;
            uint64_t* mine = reinterpret_cast<uint64_t*>(part + (warp * rpw + sub) * d + (c + P * i) * V);
#pragma unroll
            for (int e = 0; e < V / 2; ++e) mine[e] = dg[i][e];
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < d; j += RMS_BWD_THREADS) {
        float acc = 0.f;
        for (int r = 0; r < (RMS_BWD_THREADS / 32) * rpw; ++r) acc += part[r * d + j];
        a.partial[(size_t)block * d + j] = acc;
    }
}

// dg[side][4 j .. 4 j + 3] = sum over that side's partial rows in a fixed order; block (j, side).  Launched as a
// programmatic dependent of the kernel above, so that its launch is over when that one's last block is.
constexpr int RMS_REDUCE_THREADS = 128;
__global__ void __launch_bounds__(RMS_REDUCE_THREADS)
qk_rmsnorm_dg_reduce_kernel(const float* __restrict__ partial_q, const float* __restrict__ partial_k, float* __restrict__ dg_q,
                            float* __restrict__ dg_k, int nbq, int nbk, int d) {
    __shared__ float4 acc[RMS_REDUCE_THREADS];
    const float* part = blockIdx.y == 0 ? partial_q : partial_k;
    const int n = blockIdx.y == 0 ? nbq : nbk, j = 4 * blockIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int b = threadIdx.x; b < n; b += RMS_REDUCE_THREADS) {
        const float4 w = *reinterpret_cast<const float4*>(part + (size_t)b * d + j);
        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    acc[threadIdx.x] = v;
    for (int h = RMS_REDUCE_THREADS / 2; h > 0; h >>= 1) {
        __syncthreads();
        if ((int)threadIdx.x < h) {
            const float4 w = acc[threadIdx.x + h];
            v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            acc[threadIdx.x] = v;
        }
    }
    if (threadIdx.x == 0) *reinterpret_cast<float4*>((blockIdx.y == 0 ? dg_q : dg_k) + j) = v;
}

}  // namespace tvm_attn
