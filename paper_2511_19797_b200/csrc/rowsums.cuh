// Backward pre-pass (App. C "Step 1", reduced by the identities Sigma_1 = rowsum(dtO*O), Sigma_2 = rowsum(dtO*tO) and the
// standard-attention row term rowsum(dO*O)):
//   sig1[row] = sum_c Hc*O        cvec[row] = sum_c G*O + Hc*tO        lse2[row] = lse[row] * log2(e)
// Pure streaming work, four tensors read once, bound by HBM once enough bytes are in flight: like the normalisation kernels
// it splits a row over few lanes with several 16-byte chunks each (rms_split: d = 72 is 3 x 3), so that a thread has 192
// bytes in flight and a row sum costs three shuffles, and sums with two-wide FMAs.
// Measured on B200 (B 16, H 16, N 1024, d 72: 151 MB) against one chunk per lane, nine lanes a row: 51 -> 37 us,
// without dtO (75 MB) 47 -> 25 us, taken as the library's timing aid takes them, between two events in the backward's stream:
// that counts the gaps to the launches around it.  The kernel itself takes 28.8 us (5.3 TB/s; the profiler's duration, and
// that of 50 launches one behind another), without dtO 16.5 us (4.6 TB/s).
#pragma once
#include "qk_rmsnorm.cuh"

namespace tvm_attn {

constexpr int ROWSUM_THREADS = 256;
constexpr int ROWSUM_BLOCKS = 148 * 3;   // of a launch at most, what the 148 SMs hold: each block walks over its rows

// P = lanes per row, C = chunks per lane; the rows of a warp are consecutive.
template <typename T, int C, bool RAGGED>
__global__ void __launch_bounds__(ROWSUM_THREADS, 3)
bwd_rowsums_kernel(const T* __restrict__ G, const T* __restrict__ Hc, const T* __restrict__ O, const T* __restrict__ tO,
                   const float* __restrict__ lse, float* __restrict__ sig1, float* __restrict__ cvec, float* __restrict__ lse2,
                   unsigned rows, Geom qg, int H, int d, int P, float sign) {
    constexpr int V = RmsVec<T>::N;
    const int lane = threadIdx.x & 31, rpw = 32 / P;
    const int sub = lane / P, c = lane - sub * P, first = sub * P;
    const unsigned warps = gridDim.x * (ROWSUM_THREADS / 32);
    const unsigned groups = (rows + rpw - 1) / rpw;
    for (unsigned g = blockIdx.x * (ROWSUM_THREADS / 32) + (threadIdx.x >> 5); g < groups; g += warps) {
        const unsigned row = g * rpw + sub;
        const bool act = sub < rpw && row < rows;
        RmsRaw<T> o[C], t[C], x[C], y[C];
#pragma unroll
        for (int k = 0; k < C; ++k) o[k].q = t[k].q = x[k].q = y[k].q = make_uint4(0, 0, 0, 0);   // a null G or Hc (absent cotangent) counts as zeros
        float l = 0.f;
        if (act) {
            // the statistics are packed (B, H, M); the tensors have strides (H == 0 marks the packed layout: no division)
            size_t off = (size_t)row * d;
            if (H > 0) {
                const unsigned bh = row / (unsigned)qg.rows;
                off = qg.head_off((int)bh, H) + (size_t)(row - bh * (unsigned)qg.rows) * (size_t)qg.rs;
            }
            off += c * V;
#pragma unroll
            for (int k = 0; k < C; ++k) {
                if (RAGGED && k == C - 1 && (c + P * k) * V >= d) continue;   // the lane has a chunk less
                o[k].load(O + off + k * P * V);
                if (G) x[k].load(G + off + k * P * V);
                if (Hc) { y[k].load(Hc + off + k * P * V); t[k].load(tO + off + k * P * V); }
            }
            if (c == 0) l = __ldg(lse + row);
        }
        uint64_t s2 = 0ull, c2 = 0ull, ov[V / 2], xv[V / 2], yv[V / 2], tv[V / 2];
#pragma unroll
        for (int k = 0; k < C; ++k) {
            o[k].get(ov); x[k].get(xv); y[k].get(yv); t[k].get(tv);
#pragma unroll
            for (int i = 0; i < V / 2; ++i) {
                s2 = ptx::fma2(yv[i], ov[i], s2);
                c2 = ptx::fma2(xv[i], ov[i], c2);
                c2 = ptx::fma2(yv[i], tv[i], c2);
            }
        }
        const float s1 = rms_group_sum(rms_hsum(s2), P, lane, first), cc = rms_group_sum(rms_hsum(c2), P, lane, first);
        if (act && c == 0) { sig1[row] = sign * s1; cvec[row] = sign * cc; lse2[row] = sign * (l * 1.4426950408889634f); }
    }
}

}  // namespace tvm_attn
