// Attention with a Jacobian-vector product on sm_100a (tcgen05 + TMEM + TMA): the forward and the three passes of the
// backward (App. C Eq. "sdpa", the definitions under "Step 1", and "Multi-step backward pass" with the standard
// attention backward for dO summed in) on one skeleton.
//
// Carrying a tangent next to a primal is dual-number arithmetic, (a + eps b)(c + eps d) = ac + eps (bc + ad), so every
// product of the method has the same shape:
//
//   pass  owner rows  stream rows  score accumulators (128 x 64 fp32)                    bf16 operands A0, A1    acc0, acc1 (128 x d)
//   FWD   queries     keys         S = Q K^T, Sd = tQ K^T + Q tK^T                        P~, P~ (T - c)          O~, R
//   DV    keys        queries      S^T, Sd^T                                              P^T, (P Nn)^T           dtV, dV          (step 6)
//   DK    keys        queries      S^T, Sd^T, D^T = V Hc^T, X^T = tV Hc^T + V G^T        W^T, dA^T               dtK/alpha, dK/alpha   (steps 2, 4)
//   DKV   keys        queries      as DK                                                  as DV; as DK            as DV; as DK (acc2, acc3)
//   DQ    queries     keys         S, Sd, D = Hc V^T, X = G V^T + Hc tV^T                 W, dA                   dtQ/alpha, dQ/alpha   (steps 3, 5)
//   DKV_G keys        queries      S^T, X^T = V G^T                                       P^T, dA^T               dV, dK/alpha
//   DQ_G  queries     keys         S, X = G V^T                                           (none), dA              (none), dQ/alpha
//
//   score pair:  S = X0 Y0^T,  Sd = X1 Y0^T + X0 Y1^T        outputs:  acc0 += A0 B0,  acc1 += A1 B0 + A0 B1
//
// with P = 2^(c2 S - lse2), T = alpha Sd, Nn = T - mu, W = P (D - Sigma1), dA = P (X - c) + W Nn; in the forward
// P~ = 2^(c2 S - m) with a lazily updated row reference m, and O = O~/l, tO = R/l - (mu - c) O.
//
// DKV does DV's and DK's work with one computation of the scores, and one exponential, instead of two.  Its four accumulators
// leave tensor memory for four score blocks of 64 columns at d <= 64 and of 48 at d <= 80; above that DV and DK run on their own.
//
// DKV_G and DQ_G are the backward without Hc = dtO (the "detach JVP" setting), where everything that only feeds the tangent path
// is zero and what remains is the standard attention backward, dA = P (X - c).
//
// A work item is 128 owner rows of one head, against which the other side streams in tiles of 64 rows (48).  The grid has
// one CTA per SM (a CTA needs the whole tensor memory of one); the items go round-robin over the CTAs, and the rings,
// the score buffers and all barrier phases run on through the items.
//
// 16 warps in four warpgroups:
//   warp 0    loads the owner tiles and the E ring (stream tensors that only the score MMAs read; none in DKV_G, DQ_G)
//   warp 1    issues the MMAs
//   warp 2    loads the L ring (stream tensors the output MMAs read)
//   warp 3    DKV, DKV_G: puts the per-query statistics into the tiles (FOLD below)
//   warps 4-11   element-wise work, two groups of four warps
//   warps 12-15  epilogue: normalise, convert and store an item's accumulators while the next item is under way
//
// Why this split.  What bounds a tile is not one unit but the chain scores -> element-wise work -> outputs: passing an
// mbarrier costs a warp 100 to 250 cycles even when the phase has completed, reading tensor memory 180, whether it has 16
// columns to work on or 64, and the warps of a scheduler take issue slots from the one that issues the MMAs: eight
// element-wise warps with many columns each, the accumulators' way out on warps of its own.
//
// Score MMAs: the two tensors of a stage are interleaved so that they form one K-major operand of 128 rows, and
// [S | X0 Y1^T] = X0 [Y0 | Y1]^T is one N = 128 MMA per k-step, Sd += X1 Y0^T one N = 64 MMA.
//
// Measured on B200 at d = 128 (B 2, H 24, N 4096; one CTA per item, 32-key tiles with all four accumulators in two buffers
// before): forward 1.40 -> 1.08 ms, DV / DK / DQ 1.33 / 2.82 / 2.92 -> 1.06 / 1.48 / 1.42 ms.  At d <= 80 (two
// element-wise groups on alternate tiles, which also wrote the outputs, before): d = 64 (8, 16, 4096) forward 1.94 -> 1.75 ms,
// backward 7.37 -> 6.12 ms, with DV and DK in one pass 5.45 ms; d = 72 (16, 16, 1024) forward 321 -> 313 us, backward
// 1.22 -> 1.08 -> 1.01 ms; with the waits as one small loop and items that run on into one another (both at the power cap)
// 284 us and 0.89 ms.
//
// Every wait on an mbarrier is bounded; when one gives up the block records a time-out status and all roles leave their
// loops.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>
#include <type_traits>

#include "geometry.cuh"
#include "sm100_ptx.cuh"

namespace tvm_attn {

enum : int { PASS_FWD = 0, PASS_DV = 1, PASS_DK = 2, PASS_DQ = 3, PASS_DKV = 4, PASS_DKV_G = 5, PASS_DQ_G = 6 };

constexpr int JVP_THREADS = 512;
constexpr int JVP_ROWS = 128;   // owner rows per item
constexpr int JVP_BC = 64;      // stream rows per tile (DKV at padded head dim 80: 48)
// Forward, how far the row reference m may lag behind the running maximum (log2 units), and for WIDE head dims how far the
// centre c of the tangent weights may be from T at the arg-max key before it moves.
constexpr float JVP_LAZY_LOG2 = 3.0f, JVP_LAZY_LOG2_WIDE = 8.0f, JVP_CENTRE_WIDE = 3.0f;
// How long a wait may take: for what is due within a few tiles, and what every tile of an item adds to it where an item's end
// is waited for (the epilogue).  The slowest tile measured takes 2 us (DKV, 2950 cycles at 1.5 GHz); an item of 400 thousand
// tiles, 128 queries against 25.6 million keys at d = 8, takes 0.24 s.  A tile that hangs is reported after the first limit
// all the same, by the roles that work on it.
constexpr uint64_t JVP_WAIT_LIMIT_NS = 200ull * 1000ull * 1000ull, JVP_TILE_LIMIT_NS = 20ull * 1000ull;
// Registers per thread at launch; setmaxnreg moves them between the four warpgroups (JvpCfg::REGS_*) within what the block
// was launched with: the host refuses to launch a build whose kernels have fewer.
constexpr int JVP_REGS = 128;
// DKV_G, DQ_G: what the epilogue does in front of an item's stores, in steps of the issuing warp (a tile each) from the item's end on.
// Owner operands that are due later than that would hold the stores back.  Nothing in front of them / two steps, us: (64, 16, N)
// d = 72 N = 192 149 / 138, N = 200 165 / 138, d = 64 N = 192 116 / 110; d = 56 N = 256 117 / 121.
constexpr int JVP_AHEAD = 2;

struct JvpParams {
    int d, H;
    int items, row_tiles, T;   // work items (128 owner rows of a head), items per head, stream tiles per item
    Geom o, s;    // owner side and stream side of this pass (FWD, DQ: queries own, keys stream; DV, DK, DKV: the other way round)
    float alpha;      // softmax scale
    float c2;         // alpha * log2(e)
    float out_scale;  // factor applied to acc0 / acc1 of the backward passes
    const __nv_bfloat16* own[4];   // owner tensors X0..X3 (X2, X3: DK, DKV, DQ)
    const __nv_bfloat16* strm[4];  // streamed tensors: E ring (0, 1), L ring (2, 3)
    __nv_bfloat16* out0;           // acc0 destination: O | dtV | dtK | dtQ
    __nv_bfloat16* out1;           // acc1 destination: tO | dV | dK | dQ
    __nv_bfloat16* out2;           // DKV: dtK
    __nv_bfloat16* out3;           //      dK
    float* lse;                    // FWD: statistics written, packed (B, H, M)
    float* mu_out;
    // backward: statistics read, packed (B, H, M); the pre-pass writes the negated ones
    const float* nlse2;  // -lse * log2(e)
    const float* mu;
    const float* nsig1;  // -rowsum(dtO * O)
    const float* ncvec;  // -rowsum(dO * O) - rowsum(dtO * tO)
    int* status;         // device status word; non-zero makes the kernel a no-op
    // G (dO) is absent: null means zero.  It is never loaded; where an MMA still reads its tile, the tile is zeroed once, and the
    // MMAs whose result would be exactly zero are not issued.
    int no_g;
    uint64_t item_wait_ns;     // how long the end of an item may be waited for
};

template <int MODE, int DP>
struct JvpCfg {
    static_assert(DP % 16 == 0 && DP >= 16 && DP <= 128, "padded head dim must be 16..128");
    static constexpr bool DKV = MODE == PASS_DKV;
    static constexpr bool GONLY = MODE == PASS_DKV_G || MODE == PASS_DQ_G;     // one ring (L) of two tensors, two products instead of pairs
    static constexpr int NPAIR = MODE == PASS_DK || MODE == PASS_DQ || DKV ? 2 : 1;  // score pairs
    static constexpr bool TRANSPOSED = MODE != PASS_FWD && MODE != PASS_DQ && MODE != PASS_DQ_G;    // owner rows are keys
    // Stream rows per tile.  Four accumulators of DP columns and four of BC have to fit into 512.
    static constexpr int BC = DKV && DP > 64 ? 48 : JVP_BC, KS = DP / 16;
    static constexpr int NA = DP > 64 ? 2 : 1;             // 64-column swizzle atoms per row
    // How the columns from 64 on arrive.  Up to 16 of them (DP = 80): 16-byte asynchronous copies, because a 64-column
    // box hanging over the end of a 144-byte row reads the next row from L2 for nothing; tiles that are only read
    // K-major (owners, E ring) keep them in an unswizzled block [chunk][row][16 bytes] behind the first atom.  More
    // than 16 (WIDE): a second box and a second swizzle atom everywhere.
    static constexpr bool WIDE = DP > 80;
    static constexpr bool TAIL = NA == 2 && !WIDE;
    static_assert(WIDE || (MODE != PASS_DV && MODE != PASS_DK), "DV and DK on their own: only where DKV does not fit");
    static_assert(!WIDE || (!DKV && !GONLY), "DKV: four accumulators do not fit; head dims above 80 take both cotangents");
    static constexpr bool E_MN = DKV;                      // the E ring is read MN-major too: swizzled atoms like the L ring's
    // Owner operands.  The pair of the score MMAs on the tile's critical chain (FWD: the only pair; DQ: the second; DKV_G, DQ_G: both tensors) lies in
    // tensor memory as bf16 A operands: an MMA with A in shared memory moves 4 KB of A per k-step through the
    // shared-memory port.  WIDE, DKV: tensor memory has no room, everything is in shared memory.
    static constexpr bool XT = !WIDE && !DKV;
    // DKV_G, DQ_G (XS): they come to tensor memory by way of shared memory, where warp 0 puts an item's rows as soon as those of the
    // item before have left it; loaded by the epilogue, uncoalesced and behind its stores, they are the chain of a short item.
    // (Without dtO, (64, 16, N), us: d = 64 N = 192 144 -> 110, N = 64 42 -> 41, d = 72 N = 192 171 -> 138, d = 80 N = 192 193 ->
    // 157, (16, 16, 1024, 72) 370 -> 360.  Rows that do not begin on 32 bytes take the TMA longer: d = 40 N = 64 37 -> 41, d = 56
    // 39 -> 41.  With 16-byte copies instead, by warp 0 or by the epilogue: N = 64 at d = 64 53.)
    static constexpr bool XS = GONLY;
    static constexpr int NOWN = XS ? 2 : 2 * NPAIR - (XT ? 2 : 0);   // owner tensors in shared memory
    // FOLD (DKV, DKV_G): the per-query statistics belong to the columns of the tile, the same for every thread; read from
    // shared memory they would cost 512 bytes a warp and column.  Instead they are an extra piece of the score MMAs: each
    // is split into three bf16 parts in columns of its own behind the stream row, against ones behind the owner row, so
    // that the accumulators arrive as S - lse/alpha, Sd - mu/alpha, D - Sigma1, X - c.  At d = 72 these columns are the
    // padding up to 80; other head dims take one more k-step.
    static constexpr bool FOLD = DKV || MODE == PASS_DKV_G;
    static constexpr int OWN_ATOM = JVP_ROWS * 128, ATOM = BC * 128;
    // One owner tensor.  (XS: the columns from 64 on lie in the L ring, whose second atoms have room, so that the ring keeps its six
    // stages: with five, DQ_G at d = 72 (16, 16, 1024) takes 160 us instead of 142.)
    static constexpr int OWN_BYTES = OWN_ATOM * (WIDE ? 2 : 1) + (TAIL && !XS ? JVP_ROWS * 32 : 0);
    static constexpr int EST_BYTES = E_MN ? ATOM * NA : ATOM * (WIDE ? 2 : 1) + (TAIL ? BC * 32 : 0);   // one E-ring tile
    static constexpr int LST_BYTES = ATOM * NA;                                                // one L-ring tile
    static constexpr int SE = GONLY ? 0 : WIDE ? (NPAIR == 2 ? 1 : 2) : DKV ? (TAIL ? 2 : 3) : TAIL ? 3 : 4;
    static constexpr int SL = GONLY ? 6 : WIDE ? 2 : DKV ? (TAIL ? 3 : 4) : TAIL && NPAIR == 2 ? 3 : 4;
    static constexpr int TILE_BYTES = NOWN * OWN_BYTES + SE * 2 * EST_BYTES + SL * 2 * LST_BYTES;
    // FOLD: statistics of a stage, [Y0 rows, Y1 rows][16 bytes], for the rings the score MMAs read; ones and zeros
    static constexpr int FOLD_BYTES = 2 * BC * 16;
    // (DKV_G with a tail: columns 80 to 95 of the L tiles and of the owner operands instead).
    static constexpr bool FOLD_TAIL = FOLD && XS && TAIL;
    static constexpr int FOLD_E = FOLD ? SE : 0, FOLD_L = FOLD && !FOLD_TAIL ? SL : 0;
    static constexpr int ONES_BYTES = FOLD && !FOLD_TAIL ? JVP_ROWS * 32 : 0;
    static constexpr int EFULL_COUNT = 1 + (TAIL ? 32 : 0) + (FOLD_E ? 1 : 0);   // TMA issuer, each lane's own copies, warp 3
    static constexpr int LFULL_COUNT = 1 + (TAIL || (TRANSPOSED && !FOLD) ? 32 : 0) + (FOLD ? 1 : 0);
    // TMEM columns: accumulators, the owner operands in the gaps behind them,
    // score accumulators (FWD, DV: two buffers of S | Sd; DKV_G, DQ_G: of S | X; DK, DQ: one of S | Sd | D | X).
    static constexpr int NACC = DKV ? 4 : 2;
    static constexpr bool HAS_ACC0 = MODE != PASS_DQ_G;
    static constexpr int COL_ACC0 = 0, COL_ACC1 = XT ? 128 : DP, COL_SCORE = NACC * COL_ACC1;
    static constexpr int COL_X0 = DP, COL_X1 = COL_ACC1 + DP;
    static_assert(!XT || DP + DP / 2 <= 128, "operands do not fit behind their accumulators");
    static_assert(COL_SCORE + 4 * BC <= 512, "TMEM over-subscribed");
    // Registers per thread: warpgroup 0, element-wise warps (FWD, DKV_G, DQ_G: 64 columns a thread), epilogue warps (which hold an owner
    // row, 4 registers a chunk, or the columns they have read).  Shares with which no pass spills; DKV with 96, 152 and 112 spills at
    // d <= 48 and takes 1 to 3 % longer there ((64, 16, 256, 32), the backward: 163 us, 158 as here), above it makes no difference.
    static constexpr int REGS_LOAD = MODE == PASS_FWD ? 56 : GONLY ? 80 : DKV ? 112 : 96, REGS_ELEM = MODE == PASS_FWD ? 168 : DKV ? 144 : 152, REGS_EPI = MODE == PASS_FWD ? 120 : GONLY ? 128 : 112;
    static_assert(REGS_LOAD + 2 * REGS_ELEM + REGS_EPI <= 4 * JVP_REGS, "more registers than the block has");
    // barriers
    static constexpr int B_EFULL = 0;
    static constexpr int B_LFULL = B_EFULL + SE;
    static constexpr int OWN_SETS = DKV || XS ? 2 : 1;                 // owner tiles with barriers of their own (DKV: K, tK | V, tV; XS: one tensor each)
    static constexpr int B_OWN = B_LFULL + SL;                         // owner tiles in shared memory loaded
    static constexpr int B_OWNFREE = B_OWN + OWN_SETS;                 // ... free: the score MMAs of the item are complete (XS: read by the epilogue)
    static constexpr int B_XRDY = B_OWNFREE + OWN_SETS;                       // owner operands in tensor memory written
    static constexpr int XSETS = GONLY ? 2 : 1;                        // with barriers of their own
    static constexpr int B_XFREE = B_XRDY + XSETS;                     // ... free
    // MMAs of tile g complete: + (g & 3), phase g >> 2.  The element-wise groups meet every other tile only and the
    // producers run up to four tiles ahead of or behind the others (six in DKV_G, DQ_G), so that a parity wait on one barrier, or on a pair,
    // could take another tile's completion for its own.  They also tell the producers that a ring stage is free: a commit
    // costs the issuing warp 60 cycles, and a barrier of its own per ring would be one more per tile.
    static constexpr int B_SFULL = B_XFREE + XSETS;                        // S (and Sd, except in FWD) written
    static constexpr int B_XFULL = B_SFULL + 4;                        // FWD: Sd written; DK, DQ: D, X written; DKV_G, DQ_G: X written
    static constexpr int B_OUTDONE = B_XFULL + 4;                      // output MMAs complete
    // The stage of a tile is free.  DKV: its output MMAs are in front of the next tile's scores, whose completion implies theirs.
    static constexpr int B_EDONE = DKV || MODE == PASS_DV ? B_SFULL : B_XFULL, EDONE_NEXT = DKV ? 1 : 0;
    static constexpr int B_LDONE = DKV ? B_XFULL : B_OUTDONE, LDONE_NEXT = EDONE_NEXT;
    static constexpr int NOUTDONE = GONLY ? 8 : 4;                     // (DKV_G, DQ_G: the L ring is deeper)
    static_assert(SE <= 4 && SL <= NOUTDONE, "a ring deeper than the completion barriers");
    // operands written: + half of the tile (DK, DQ), + 2 (g & 1) + half (FWD, DV), + pair (DKV),
    // + 2 (g & 1): P written (DKV_G) or S read (DQ_G), + 1: dA written
    static constexpr int B_PREADY = B_OUTDONE + NOUTDONE;
    static constexpr int B_SREAD = B_PREADY + 4;                       // DK, DQ: S, Sd read
    static constexpr int B_FINAL = B_SREAD + 1;                        // + pair of accumulators: the item's last output MMAs complete
    static constexpr int B_ACCFREE = B_FINAL + NACC / 2;               // the epilogue has read the accumulators
    static constexpr int B_TURN = B_ACCFREE + NACC / 2;                       // FWD: + lane quadrant: row state of the tile decided
    static constexpr int B_ROWSTAT = B_TURN + 4;                       // FWD: the item's row sums written
    static constexpr int B_DRAIN = B_ROWSTAT + 1;                      // used once, while winding down after a time-out
    static constexpr int NBARS = B_DRAIN + 1;
    static_assert(NBARS <= 56, "barrier table too small");
    static constexpr int NSTAT = 2 * NPAIR;                            // statistics per query: lse2, mu (, Sigma1, c)
    static constexpr int STATS_FLOATS = TRANSPOSED && !FOLD ? SL * NSTAT * BC : 0;
    static constexpr int FWD_FLOATS = MODE == PASS_FWD ? 4 * JVP_ROWS + 2 * 4 * JVP_ROWS : 0;   // row state; row sums per group
    static constexpr int MISC_BYTES = 56 * 8 + 64 + (STATS_FLOATS + FWD_FLOATS) * 4 + (FOLD_E + FOLD_L) * FOLD_BYTES + ONES_BYTES;
    static constexpr int SMEM_BYTES = TILE_BYTES + MISC_BYTES;         // from a 1024-byte boundary
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory over-subscribed");
};

// A value that is to stay in a register (kernel parameters are otherwise read from constant memory wherever they are used,
// which costs a dependent instruction 30 cycles more).
__device__ __forceinline__ int jvp_pin(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

// Items of this block.
__device__ __forceinline__ int jvp_item_count(const JvpParams& p) {
    return (int)blockIdx.x < p.items ? (p.items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
}

// The value is computed here and not behind the next wait: the compiler moves arithmetic down to where its result is used,
// past the waits that it is meant to run under.  Only an instruction that may have an effect stops it, hence one that never
// runs (for the sake of a NaN whose bits the arithmetic does not make, and harmless if it did).
__device__ __forceinline__ void jvp_force(uint64_t v) {
    const uint32_t w = (uint32_t)v ^ (uint32_t)(v >> 32);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %0, 0x7fc12345;\n\t@p nanosleep.u32 0;\n\t}" ::"r"(w) : "memory");
}

// What the roles of a block share: addresses, all of them the base of its shared memory plus constants (the element-wise
// warps have no registers to spare for more), and waits.
template <int MODE, int DP>
struct JvpBlock {
    using C = JvpCfg<MODE, DP>;
    uint32_t base;
    const JvpParams& p;
    static constexpr uint32_t E = C::NOWN * C::OWN_BYTES, L = E + C::SE * 2 * C::EST_BYTES, MISC = C::TILE_BYTES, SLOT = MISC + 56 * 8, ABORT = SLOT + 16;
    static constexpr uint32_t STATS = SLOT + 64;                              // DV, DK, WIDE: [stage][NSTAT][64] floats
    static constexpr uint32_t ROW_STATE = STATS + C::STATS_FLOATS * 4;        // FWD: float4 (m, c, running maximum) of each row
    static constexpr uint32_t ROW_SUMS = ROW_STATE + 16 * JVP_ROWS;           // FWD: [group][row] float4 (l, sum P~ (T - c), m, c)
    static constexpr uint32_t FOLD_E = ROW_STATE + C::FWD_FLOATS * 4;         // FOLD: statistics of the E and the L stages,
    static constexpr uint32_t FOLD_L = FOLD_E + C::FOLD_E * C::FOLD_BYTES;    // ones and zeros, 128 rows of 16 bytes
    static constexpr uint32_t ONES = FOLD_L + C::FOLD_L * C::FOLD_BYTES, ZEROS = ONES + JVP_ROWS * 16;

    // A copy for a role with registers to spare: the base stays in one.
    __device__ __forceinline__ JvpBlock pinned() const {
        JvpBlock r = *this;
        asm volatile("" : "+r"(r.base));
        return r;
    }
    // FOLD: the statistics have a k-step of their own (else they are the padding columns of the last one)
    __device__ __forceinline__ bool fold_step() const { return C::FOLD && (C::NA == 1 || p.d == DP); }
    __device__ __forceinline__ uint32_t bar(int i) const { return base + MISC + 8u * static_cast<uint32_t>(i); }
    __device__ __forceinline__ bool wait(int i, int phase) const {
        return ptx::mbar_wait_warp_s(bar(i), phase & 1, base + ABORT, JVP_WAIT_LIMIT_NS);
    }
    // For what comes at the end of an item the caller has just begun to wait for.
    __device__ __forceinline__ bool wait_item(int i, int phase) const {
        return ptx::mbar_wait_warp_s(bar(i), phase & 1, base + ABORT, p.item_wait_ns);
    }
    __device__ __forceinline__ bool wait2(int i, int pi, int j, int pj) const {
        if (ptx::mbar_test2_warp(bar(i), pi & 1, bar(j), pj & 1)) return true;
        return wait(i, pi) && wait(j, pj);
    }
    // After the waits for a tile: what other warps copied to it (tails) is ordered before the MMAs that read it.
    __device__ __forceinline__ void tile_fence() const {
        if (C::TAIL) ptx::fence_proxy_async_smem();
        ptx::tc_fence_after_sync();
    }
    __device__ __forceinline__ bool done(int i, int g) const { return wait(i + (g & 3), g >> 2); }   // i: B_SFULL, B_XFULL, B_OUTDONE
    // Ring R's stage of tile g - S is free.
    template <int R>
    __device__ __forceinline__ bool stage_free(int g) const {
        if (R == 0) return done(C::B_EDONE, g - C::SE + C::EDONE_NEXT);
        const int t = g - C::SL + C::LDONE_NEXT;
        return wait(C::B_LDONE + (t & (C::NOUTDONE - 1)), t / C::NOUTDONE);
    }
    __device__ __forceinline__ uint32_t own_tile(int t) const { return base + t * C::OWN_BYTES; }
    // TAIL: 16-byte chunk c behind column 64 of owner row r: compact blocks behind the tile; XS: chunks of the second atoms of the L
    // ring's first stage, which have 64 columns where the stream's tail, with the statistics, has 32.
    __device__ __forceinline__ uint32_t own_tail(int t, int r, int c) const {
        static_assert(!C::XS || C::ATOM == 64 * 128, "rows 64 on: in the second tensor's atom");
        if (C::XS) return base + L + 2 * C::ATOM + r * 128 + (((4 + 2 * t + c) ^ (r & 7)) << 4);
        return own_tile(t) + C::OWN_ATOM + (c * JVP_ROWS + r) * 16;
    }
    __device__ __forceinline__ const float* stats(int s) const { return static_cast<const float*>(__cvta_shared_to_generic(base + STATS + s * C::NSTAT * C::BC * 4)); }
    __device__ __forceinline__ float4& row_state(int r) const { return *static_cast<float4*>(__cvta_shared_to_generic(base + ROW_STATE + 16 * r)); }
    __device__ __forceinline__ float4& row_sums(int r) const { return *static_cast<float4*>(__cvta_shared_to_generic(base + ROW_SUMS + 16 * r)); }
    // one arrival per warp, after its tensor-memory accesses
    __device__ __forceinline__ void arrive(int i, int lane) const {
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar(i));
    }
};

// ------------------------------------------------------------------------------------------------ producers
// A set of owner tiles of an item (by the E ring's warp): two boxes of 64 rows per tensor and atom, like those of the stream tiles,
// so that one tensor map serves both.
template <int MODE, int DP, int SET>
__device__ __forceinline__ void jvp_load_owners(const JvpParams& p, const JvpBlock<MODE, DP>& k, const CUtensorMap* const (&maps)[4], int item, int lane) {
    using C = JvpCfg<MODE, DP>;
    constexpr int T0 = SET * (C::NOWN / C::OWN_SETS), T1 = T0 + C::NOWN / C::OWN_SETS;
    constexpr int KT = C::TAIL ? (DP - 64) / 8 : 1, H64 = 64 * 128;
    const int bh = item / p.row_tiles, row0 = (item - bh * p.row_tiles) * JVP_ROWS;
    const int cb = bh / p.H, ch = bh - cb * p.H;
    const bool upper = !C::XS || p.o.rows - row0 > 64;   // (XS: rows beyond the tensor are not read)
    if (lane == 0) {
        const uint32_t full = k.bar(C::B_OWN + SET);
        uint32_t tx = 0;
#pragma unroll
        for (int t = T0; t < T1; ++t) tx += upper ? C::OWN_ATOM * (C::WIDE ? 2 : 1) : C::OWN_ATOM / 2;
        ptx::mbar_arrive_expect_tx(full, tx);
#pragma unroll
        for (int t = T0; t < T1; ++t) {
            const uint32_t dst = k.own_tile(t);
            ptx::tma_load_4d(dst, maps[t], full, 0, row0, ch, cb);
            if (upper) ptx::tma_load_4d(dst + H64, maps[t], full, 0, row0 + 64, ch, cb);
            if (C::WIDE) {
                ptx::tma_load_4d(dst + C::OWN_ATOM, maps[t], full, 64, row0, ch, cb);
                ptx::tma_load_4d(dst + C::OWN_ATOM + H64, maps[t], full, 64, row0 + 64, ch, cb);
            }
        }
    }
    if constexpr (C::TAIL) {
        const int ntail = (p.d - 64) >> 3, rows_left = p.o.rows - row0;
        const size_t d32 = 32 * (size_t)p.o.rs, lane_row = p.o.head_off(bh, p.H) + (size_t)(row0 + lane) * (size_t)p.o.rs + 64;
#pragma unroll
        for (int t = T0; t < T1; ++t) {
            const __nv_bfloat16* x = p.own[t];
#pragma unroll
            for (int c = 0; c < KT; ++c) {
                if (c < ntail) {
#pragma unroll
                    for (int rp = 0; rp < JVP_ROWS / 32; ++rp) {
                        const bool v = lane + 32 * rp < rows_left;
                        ptx::cp_async_16(k.own_tail(t, lane + 32 * rp, c), v ? x + lane_row + rp * d32 + 8 * c : x, v ? 16u : 0u);
                    }
                }
            }
        }
        ptx::cp_async_arrive(k.bar(C::B_OWN + SET));
    }
}

// One warp per ring; the E ring's loads the owner tiles too.  One lane issues the TMA boxes; with a tail (DP = 80) or
// statistics copied as they are (WIDE) all lanes copy those, 16 bytes each, and each lane's arrival on the stage's barrier
// is left to its copies (a warp that waits for them itself loads no more than one tile per memory latency).  These loops
// run next to element-wise warps that leave them few issue slots, and a ring is refilled no faster than they run: what does
// not depend on the tile is set up before them, and tiles whose rows all exist take a path without predicates.
template <int MODE, int DP, int RING>
__device__ __forceinline__ void jvp_load_ring(const JvpParams& p, const JvpBlock<MODE, DP>& shared, const CUtensorMap* map0, const CUtensorMap* map1,
                                              const CUtensorMap* const (&own_maps)[4], int lane) {
    using C = JvpCfg<MODE, DP>;
    const JvpBlock<MODE, DP> k = shared.pinned();
    const int T = jvp_pin(p.T), rows = jvp_pin(p.s.rows);
    constexpr int BC = C::BC, S = RING == 0 ? C::SE : C::SL, ATOM = C::ATOM;
    constexpr int b_full = RING == 0 ? C::B_EFULL : C::B_LFULL;
    constexpr uint32_t TB = RING == 0 ? C::EST_BYTES : C::LST_BYTES;
    constexpr bool STATS = RING == 1 && C::TRANSPOSED && !C::FOLD;   // this ring carries the statistics as they are
    constexpr bool OWNERS = RING == 0 && C::NOWN > 0;
    constexpr bool HAS_CP = C::TAIL || STATS;           // the warp has asynchronous copies of its own
    constexpr int KT = C::TAIL ? (DP - 64) / 8 : 1;     // 16-byte chunks per row behind column 64, at most
    [[maybe_unused]] const int ntail = C::TAIL ? (p.d - 64) >> 3 : 0;
    [[maybe_unused]] const size_t d32 = 32 * (size_t)p.s.rs;   // 32 rows further down, in elements
    [[maybe_unused]] const size_t tile_elems = (size_t)BC * (size_t)p.s.rs;
    const uint32_t ring_base = k.base + (RING == 0 ? k.E : k.L);
    const __nv_bfloat16* base0 = p.strm[2 * RING];
    const __nv_bfloat16* base1 = p.strm[2 * RING + 1];
    // DKV streams the cotangents (Hc, G) in its E ring: G may be absent (null) and is not loaded then.
    const bool has1 = C::DKV && RING == 0 ? base1 != nullptr : true;
    const uint32_t tx_bytes = (has1 ? 2 : 1) * ATOM * (C::WIDE ? 2 : 1);
    // Chunk 0 of row `lane` behind the first atoms: compact blocks in the E ring, a second swizzled atom in the L ring.
    [[maybe_unused]] const uint32_t sw = lane & 7;  // rows 32 apart share it
    constexpr bool FLAT = RING == 0 && !C::E_MN;
    [[maybe_unused]] const uint32_t dst_lane = 2 * ATOM + (FLAT ? lane * 16 : lane * 128);
    // statistics as they are: 16-byte chunks when the rows of the (B, H, M) arrays are 16-byte aligned, else floats
    [[maybe_unused]] const bool st16 = (p.s.rows & 3) == 0;
    [[maybe_unused]] const uint32_t st_base = k.base + k.STATS;
    bool ok = true;
    int s = 0, ph = 0;
    int g = 0, owners = 0;           // tiles, and items whose owner tiles, have been asked for
    [[maybe_unused]] int owners0 = 0;   // one more item's first set has
    uint32_t stage = ring_base, full = k.bar(b_full);
    // In an item's tiles the owner tiles have their turn where what they wait for is about to happen: behind as many of the
    // item's E tiles as the ring holds.
    [[maybe_unused]] const int owners_at = min(S, T) - 1;
    for (int item = blockIdx.x; ok && item < p.items; item += gridDim.x) {
        const int bh = item / p.row_tiles;
        const int cb = bh / p.H, ch = bh - cb * p.H;   // batch and head: coordinates of the 4-D tensor maps
        // element offset of (row `lane`, column 64) in the stream tensors
        [[maybe_unused]] const size_t lane_row = p.s.head_off(bh, p.H) + (size_t)lane * (size_t)p.s.rs + 64;
        [[maybe_unused]] const __nv_bfloat16* src0 = base0 + lane_row;  // advance by one tile per iteration
        [[maybe_unused]] const __nv_bfloat16* src1 = base1 + lane_row;
        [[maybe_unused]] const size_t srow = (size_t)bh * p.s.rows;
        [[maybe_unused]] const float* st_src0 = nullptr;
        [[maybe_unused]] const float* st_src1 = nullptr;
        if constexpr (STATS) {
            st_src0 = (lane < 16 ? p.nlse2 : p.mu) + srow + 4 * (lane & 15);
            if (C::NSTAT == 4) st_src1 = (lane < 16 ? p.nsig1 : p.ncvec) + srow + 4 * (lane & 15);
        }
        for (int j = 0; j < T; ++j) {
            if (OWNERS && j == owners_at) {   // once the score MMAs of the item before are complete
                ok = owners == 0 || k.wait(C::B_OWNFREE, owners - 1);
                if (!ok) break;
                jvp_load_owners<MODE, DP, 0>(p, k, own_maps, item, lane);
                if constexpr (C::OWN_SETS == 2) {
                    ok = owners == 0 || k.wait(C::B_OWNFREE + 1, owners - 1);
                    if (!ok) { owners0 = 1; break; }
                    jvp_load_owners<MODE, DP, 1>(p, k, own_maps, item, lane);
                }
                ++owners;
            }
            if (g >= S) ok = k.template stage_free<RING>(g);   // the MMAs that read the stage's last tile
            if (!ok) break;
            ++g;
            [[maybe_unused]] const int rows_left = rows - j * BC;  // rows of this tile that exist
            if (ptx::elect_one()) {
                ptx::mbar_arrive_expect_tx(full, tx_bytes);
                ptx::tma_load_4d(stage, map0, full, 0, j * BC, ch, cb);
                if (C::WIDE) ptx::tma_load_4d(stage + 2 * ATOM, map0, full, 64, j * BC, ch, cb);
                if (has1) {
                    ptx::tma_load_4d(stage + ATOM, map1, full, 0, j * BC, ch, cb);
                    if (C::WIDE) ptx::tma_load_4d(stage + 3 * ATOM, map1, full, 64, j * BC, ch, cb);
                }
            }
            __syncwarp();
            if constexpr (STATS) {
                // queries beyond M read as zero: their rows of the B operands are zero too
                const uint32_t slot = st_base + s * (C::NSTAT * BC * 4);
                if (st16) {
                    const bool v = 4 * (lane & 15) < rows_left;
                    const uint32_t dst = slot + (lane >> 4) * 256 + (lane & 15) * 16;
                    ptx::cp_async_16(dst, v ? st_src0 + j * BC : p.nlse2, v ? 16u : 0u);
                    if (C::NSTAT == 4) ptx::cp_async_16(dst + 512, v ? st_src1 + j * BC : p.nlse2, v ? 16u : 0u);
                } else {
                    for (int c = lane; c < C::NSTAT * BC; c += 32) {
                        const int stat = c >> 6, r = c & 63;
                        const float* src = (stat == 0 ? p.nlse2 : stat == 1 ? p.mu : stat == 2 ? p.nsig1 : p.ncvec) + srow + j * BC + r;
                        const bool v = r < rows_left;
                        ptx::cp_async_4(slot + c * 4, v ? src : p.nlse2, v ? 4u : 0u);
                    }
                }
            }
            if constexpr (C::TAIL) {
                const uint32_t d0 = stage + dst_lane;
                constexpr uint32_t T1 = FLAT ? BC * 16 : ATOM, R1 = FLAT ? 32 * 16 : 32 * 128;   // second tensor, second 32 rows
                const bool hi = BC == 64 || lane < BC - 32;   // the lane has a second row
#pragma unroll
                for (int c = 0; c < KT; ++c) {
                    if (c < ntail) {
                        const uint32_t dst = d0 + (FLAT ? c * 2 * BC * 16 : (c ^ sw) << 4);
                        if (__builtin_expect(rows_left >= BC, 1)) {
                            ptx::cp_async_16(dst, src0 + 8 * c);
                            if (hi) ptx::cp_async_16(dst + R1, src0 + d32 + 8 * c);
                            if (has1) { ptx::cp_async_16(dst + T1, src1 + 8 * c); if (hi) ptx::cp_async_16(dst + T1 + R1, src1 + d32 + 8 * c); }
                        } else {
#pragma unroll
                            for (int rp = 0; rp < 2; ++rp) {
                                const bool v = lane + 32 * rp < rows_left;
                                if (rp == 1 && !hi) continue;
                                ptx::cp_async_16(dst + rp * R1, v ? src0 + rp * d32 + 8 * c : base0, v ? 16u : 0u);
                                if (has1) ptx::cp_async_16(dst + rp * R1 + T1, v ? src1 + rp * d32 + 8 * c : base1, v ? 16u : 0u);
                            }
                        }
                    }
                }
                src0 += tile_elems;
                src1 += tile_elems;
            }
            if (HAS_CP) ptx::cp_async_arrive(full);
            stage += 2 * TB;
            full += 8;
            if (++s == S) { s = 0; ph ^= 1; stage = ring_base; full = k.bar(b_full); }
        }
    }
    if (HAS_CP) ptx::cp_async_wait_all();  // nothing of ours stays in flight
    if (!ok) {
        // Winding down after a time-out: the TMA loads this warp started write into this block's shared memory and must
        // have landed before the block exits.  Stages below s carry the phase of this pass over the ring, the others
        // the one before.
        for (int i = 0; i < S; ++i) {
            const bool cur = i < s;
            if (!cur && g < S) continue;  // never filled
            ptx::mbar_wait_drain(k.bar(b_full + i), (cur ? ph : ph ^ 1) & 1, ptx::DRAIN_LIMIT_NS);
        }
        if (OWNERS && owners + owners0 > 0) ptx::mbar_wait_drain(k.bar(C::B_OWN), (owners + owners0 - 1) & 1, ptx::DRAIN_LIMIT_NS);
        if (OWNERS && C::OWN_SETS == 2 && owners > 0) ptx::mbar_wait_drain(k.bar(C::B_OWN + 1), (owners - 1) & 1, ptx::DRAIN_LIMIT_NS);
    }
}

// XS: warp 0 loads the owner tiles of one item after the other, one tensor at a time.
template <int MODE, int DP>
__device__ __forceinline__ void jvp_stage_owners(const JvpParams& p, const JvpBlock<MODE, DP>& shared, const CUtensorMap* const (&maps)[4], int lane) {
    using C = JvpCfg<MODE, DP>;
    const JvpBlock<MODE, DP> k = shared.pinned();
    int n0 = 0, n1 = 0;   // items whose first, second tensor has been asked for
    bool ok = true;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x) {
        ok = n0 == 0 || k.wait_item(C::B_OWNFREE, n0 - 1);
        if (!ok) break;
        jvp_load_owners<MODE, DP, 0>(p, k, maps, item, lane);
        ++n0;
        ok = n1 == 0 || k.wait_item(C::B_OWNFREE + 1, n1 - 1);
        if (!ok) break;
        jvp_load_owners<MODE, DP, 1>(p, k, maps, item, lane);
        ++n1;
    }
    if (C::TAIL) ptx::cp_async_wait_all();   // nothing of ours stays in flight
    if (!ok) {                               // nor, after a time-out, a TMA load
        ptx::mbar_wait_drain(k.bar(C::B_OWN), (n0 - 1) & 1, ptx::DRAIN_LIMIT_NS);
        if (n1 > 0) ptx::mbar_wait_drain(k.bar(C::B_OWN + 1), (n1 - 1) & 1, ptx::DRAIN_LIMIT_NS);
    }
}

// FOLD.  Each statistic is stored as three bf16 parts whose sum is its 24 bits, in the first three of eight columns, against
// ones in the owner operand.
constexpr uint32_t JVP_ONES0 = 0x3F803F80u, JVP_ONES1 = 0x00003F80u;   // 1, 1, 1, 0 in bf16
__device__ __forceinline__ void jvp_split3(float a, float b, uint2& pa, uint2& pb) {   // two values at once
    const uint32_t h = ptx::pack_bf16(a, b);
    a -= __uint_as_float(h << 16); b -= __uint_as_float(h & 0xffff0000u);
    const uint32_t m = ptx::pack_bf16(a, b);
    a -= __uint_as_float(m << 16); b -= __uint_as_float(m & 0xffff0000u);
    const uint32_t l = ptx::pack_bf16(a, b);
    pa = make_uint2(__byte_perm(h, m, 0x5410), l & 0xffffu);
    pb = make_uint2(__byte_perm(h, m, 0x7632), l >> 16);
}

// Warp 3: the statistics of the stream rows lane and lane + 32 of a tile, for the L ring (lse, mu) and the E ring (Sigma1, c) (DKV_G: lse, c for the L ring),
// loaded one tile ahead.
template <int MODE, int DP>
__device__ __forceinline__ void jvp_fold(const JvpParams& p, const JvpBlock<MODE, DP>& shared, int lane) {
    using C = JvpCfg<MODE, DP>;
    const JvpBlock<MODE, DP> k = shared.pinned();
    const int T = jvp_pin(p.T);
    constexpr int BC = C::BC;
    // where the parts of (tensor t, row lane + 32 r) of a stage go: base + stage * step + t * t_step + r * r_step
    struct Dst { uint32_t base, step, t_step, r_step; };
    const uint32_t sw = lane & 7;
    const bool own = k.fold_step();
    const Dst de = own ? Dst{k.base + k.FOLD_E + lane * 16, (uint32_t)C::FOLD_BYTES, BC * 16, 32 * 16}
                       : Dst{k.base + k.E + 2 * C::ATOM + lane * 128 + ((1 ^ sw) << 4), 2u * C::EST_BYTES, C::ATOM, 32 * 128};
    const Dst dl = own && !C::FOLD_TAIL ? Dst{k.base + k.FOLD_L + lane * 16, (uint32_t)C::FOLD_BYTES, BC * 16, 32 * 16}
                                        : Dst{k.base + k.L + 2 * C::ATOM + lane * 128 + (((own ? 2 : 1) ^ sw) << 4), 2u * C::LST_BYTES, C::ATOM, 32 * 128};
    const float f_lse = 1.0f / p.c2, f_mu = -1.0f / p.alpha;   // to the scale of S and Sd
    float a[4];                        // (statistic of tensor 0, of tensor 1) of the two rows: lse, mu (DKV_G: lse, c)
    [[maybe_unused]] float b[4];       // DKV: Sigma1, c
    auto load = [&](int bh, int j) {
        const int left = p.s.rows - j * BC - lane;   // queries beyond M: zero, like their rows of the operands
        const size_t at = (size_t)bh * p.s.rows + (size_t)j * BC + lane;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const bool v = left > 32 * r;
            a[2 * r] = v ? __ldg(p.nlse2 + at + 32 * r) : 0.f;
            a[2 * r + 1] = v ? __ldg((C::DKV ? p.mu : p.ncvec) + at + 32 * r) : 0.f;
            if constexpr (C::DKV) {
                b[2 * r] = v ? __ldg(p.nsig1 + at + 32 * r) : 0.f;
                b[2 * r + 1] = v ? __ldg(p.ncvec + at + 32 * r) : 0.f;
            }
        }
    };
    auto put = [&](const Dst& d, int stage, int full, float x0, float x1, float y0, float y1) {
        const uint32_t at = d.base + stage * d.step;
        uint2 u, v;
        jvp_split3(x0, x1, u, v);
        ptx::st_shared_v4(at, u.x, u.y, 0u, 0u);
        ptx::st_shared_v4(at + d.t_step, v.x, v.y, 0u, 0u);
        if (BC == 64 || lane < BC - 32) {   // the lane has a second row
            jvp_split3(y0, y1, u, v);
            ptx::st_shared_v4(at + d.r_step, u.x, u.y, 0u, 0u);
            ptx::st_shared_v4(at + d.t_step + d.r_step, v.x, v.y, 0u, 0u);
        }
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(k.bar(full + stage));
    };
    if ((int)blockIdx.x < p.items) load(blockIdx.x / p.row_tiles, 0);
    int g = 0, se = 0, sl = 0;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x) {
        const int bh = item / p.row_tiles, next = item + (int)gridDim.x;
        for (int j = 0; j < T; ++j, ++g) {
            if (g >= C::SL && !k.template stage_free<1>(g)) return;
            const float f1 = C::DKV ? f_mu : 1.0f;
            put(dl, sl, C::B_LFULL, a[0] * f_lse, a[1] * f1, a[2] * f_lse, a[3] * f1);
            if (++sl == C::SL) sl = 0;
            if constexpr (C::DKV) {
                if (g >= C::SE && !k.template stage_free<0>(g)) return;
                put(de, se, C::B_EFULL, b[0], b[1], b[2], b[3]);
                if (++se == C::SE) se = 0;
            }
            const bool more = j + 1 < T;
            if (more || next < p.items) load(more ? bh : next / p.row_tiles, more ? j + 1 : 0);
        }
    }
}

// ------------------------------------------------------------------------------------------------ MMA issue
// The whole warp runs this in converged control flow; one elected lane issues (one election per batch of MMAs,
// descriptors as 32-bit halves: see mma_ts_acc).  Tensor memory starts at column 0, because the block owns all of it.
//
// The tensor pipe takes about four MMAs ahead, 130 to 250 cycles of work; whatever the issuing warp does between two
// batches beyond that leaves the pipe idle.  A wait for a barrier that has completed costs it 85 cycles, a commit 60, a
// dependent scalar instruction ten, and an MMA 70 instead of 25 where the lane that issues it was elected in front of a branch
// or a wait: each batch elects its own.  So: ring positions are carried along as descriptors (every descriptor of a batch is
// the carried one plus a constant), barriers of the rings are tested ahead, in front of the batch before, what depends on
// the item stays out of the tile's path, and whether G is absent (NO_G) is a template parameter.
struct JvpSlot {   // a ring's next tile: stage, phase, low descriptor halves of the stage and of its statistics
    uint32_t lo, fold, lo0, fold0;
    int s = 0, ph = 0;
    __device__ __forceinline__ JvpSlot(uint32_t lo_, uint32_t fold_) : lo(lo_), fold(fold_), lo0(lo_), fold0(fold_) {}
    template <int S, uint32_t STEP, uint32_t FSTEP>
    __device__ __forceinline__ void next() {
        lo += STEP;
        fold += FSTEP;
        if (++s == S) { s = 0; ph ^= 1; lo = lo0; fold = fold0; }
    }
};

template <int MODE, int DP>
struct JvpIssue {
    using C = JvpCfg<MODE, DP>;
    using Block = JvpBlock<MODE, DP>;
    static constexpr int BC = C::BC, KS = C::KS, ATOM = C::ATOM;
    static constexpr uint32_t HI_SW = ptx::desc_hi_sw128(1024), HI_TAIL = ptx::desc_hi_nosw(128);
    static constexpr uint32_t I_S = ptx::idesc_bf16_f32(128, BC, 0, 0), I_S2 = ptx::idesc_bf16_f32(128, 2 * BC, 0, 0);
    static constexpr uint32_t I_O = ptx::idesc_bf16_f32(128, DP, 0, 1);
    // Low descriptor half of an address with leading offset 16 (K-major, swizzled); other operands are that plus constants.
    static constexpr uint32_t LBO16 = 1u << 16;
    static __host__ __device__ constexpr uint32_t lbo(uint32_t bytes) { return ((bytes >> 4) << 16) - LBO16; }
    static constexpr uint32_t E_STEP = (2 * C::EST_BYTES) >> 4, L_STEP = (2 * C::LST_BYTES) >> 4;
    static constexpr uint32_t F_STEP = (C::FOLD_BYTES >> 4) - ((C::FOLD_BYTES >> 4) << 16);   // the zeros behind come nearer
    static __device__ __forceinline__ JvpSlot e_slot(const Block& k) { return JvpSlot(ptx::desc_lo(k.base + k.E, 16), ptx::desc_lo(k.base + k.FOLD_E, k.ZEROS - k.FOLD_E)); }
    static __device__ __forceinline__ JvpSlot l_slot(const Block& k) { return JvpSlot(ptx::desc_lo(k.base + k.L, 16), ptx::desc_lo(k.base + k.FOLD_L, k.ZEROS - k.FOLD_L)); }

    static __host__ __device__ constexpr bool is_tail(int kk) { return C::TAIL && kk >= 4; }
    static __host__ __device__ constexpr bool flat(bool from_l, int kk) { return is_tail(kk) && !from_l && !C::E_MN; }   // an unswizzled tail
    // k-step kk of a K-major operand, relative to its tile or stage: owner tile | E stage (rows of Y0, then Y1) | L stage
    static __host__ __device__ constexpr uint32_t own_k(int kk) {
        return kk < 4 ? 2u * kk : C::WIDE ? ((uint32_t)C::OWN_ATOM >> 4) + 2u * (kk - 4) : ((uint32_t)C::OWN_ATOM >> 4) + lbo(JVP_ROWS * 16);
    }
    static __host__ __device__ constexpr uint32_t e_k(int kk) {
        return C::E_MN ? l_k(kk) : kk < 4 ? 2u * kk : C::WIDE ? (2u * ATOM >> 4) + 2u * (kk - 4) : (2u * ATOM >> 4) + lbo(2 * BC * 16);
    }
    static __host__ __device__ constexpr uint32_t l_k(int kk) { return (uint32_t)((kk >> 2) * 2 * ATOM >> 4) + 2u * (kk & 3); }
    // L stage read MN-major by the output MMAs (tensor t): atoms of 64 d-columns are 2 * ATOM bytes apart, 8-row groups
    // 1024 bytes, a k-step of 16 stream rows 2048
    static __host__ __device__ constexpr uint32_t l_n(int t, int u) { return (uint32_t)(t * ATOM + u * 2048) / 16 + lbo(2 * ATOM); }

    // Long batches are loops: their code, run once a tile by one warp, else pushes the element-wise loops out of the instruction
    // cache (head dims above 64: 4 to 8 % of a pass; DKV 3 %).  Short ones (d <= 64, DKV_G and DQ_G) pay more for the loops.
    static constexpr int UNROLL = !C::GONLY && (DP > 64 || C::DKV) ? 1 : 8;
    // One k-step with A in tensor memory (ATM: a = its columns) or in shared memory (a = the tile's descriptor).
    template <bool ATM>
    static __device__ __forceinline__ void step(uint32_t el, uint32_t col, uint32_t a, uint32_t ahi, uint32_t b, uint32_t bhi, uint32_t idesc, uint32_t acc) {
        if (ATM) ptx::mma_ts_acc(el, col, a, b, bhi, idesc, acc);
        else ptx::mma_ss_acc(el, col, a, ahi, b, bhi, idesc, acc);
    }
    // The k-steps of a K-major product: f(a offset, a hi, b offset, b hi, first ? 0 : 1).
    template <bool FROM_L, bool ATM, class F>
    static __device__ __forceinline__ void ksteps(F f) {
        constexpr int K0 = KS < 4 ? KS : 4;
#pragma unroll UNROLL
        for (int kk = 0; kk < K0; ++kk) f(ATM ? 8u * kk : 2u * kk, HI_SW, 2u * kk, HI_SW, kk ? 1u : 0u);
        if constexpr (KS > 4) {
            constexpr uint32_t b4 = FROM_L ? l_k(4) : e_k(4);
#pragma unroll UNROLL
            for (int kk = 0; kk < KS - 4; ++kk)
                f(ATM ? 32u + 8u * kk : own_k(4) + 2u * kk, is_tail(4) ? HI_TAIL : HI_SW, b4 + 2u * kk, flat(FROM_L, 4) ? HI_TAIL : HI_SW, 1u);
        }
    }
    // The statistics' own k-step (FOLD, where the padding columns do not hold them), tensor t0 on.
    static __device__ __forceinline__ void fold_step(uint32_t el, uint32_t col, const Block& k, uint32_t fold, int t0, uint32_t idesc) {
        const uint32_t b = fold + (uint32_t)(t0 * BC * 16 >> 4) - ((uint32_t)(t0 * BC * 16 >> 4) << 16);
        ptx::mma_ss_p<1>(el, col, ptx::desc_lo(k.base + k.ONES, JVP_ROWS * 16), HI_TAIL, b, HI_TAIL, idesc);
    }
    // [S | X0 Y1^T] = X0 [Y0 | Y1]^T, Sd += X1 Y0^T at column col; FROM_L: the stage is one of the L ring.
    template <bool FROM_L, bool ATM, bool SECOND>
    static __device__ __forceinline__ void pair(uint32_t el, uint32_t col, const Block& k, uint32_t a0, uint32_t a1, uint32_t lo, uint32_t fold, uint32_t mid_bar) {
        ksteps<FROM_L, ATM>([&](uint32_t ao, uint32_t ahi, uint32_t bo, uint32_t bhi, uint32_t acc) {
            step<ATM>(el, col, a0 + ao, ahi, lo + bo, bhi, I_S2, acc);
            if (SECOND && MODE != PASS_FWD) step<ATM>(el, col + BC, a1 + ao, ahi, lo + bo, bhi, I_S, 1u);
        });
        if (k.fold_step()) fold_step(el, col, k, fold, 0, I_S2);
        if (MODE == PASS_FWD) {
            ptx::mma_commit_p(el, mid_bar);   // S is complete before Sd
            ksteps<FROM_L, ATM>([&](uint32_t ao, uint32_t ahi, uint32_t bo, uint32_t bhi, uint32_t) {
                step<ATM>(el, col + BC, a1 + ao, ahi, lo + bo, bhi, I_S, 1u);
            });
        }
    }
    // One product X Y^T with Y the T-th tensor of the stage.
    template <bool FROM_L, bool ATM, int T>
    static __device__ __forceinline__ void single(uint32_t el, uint32_t col, const Block& k, uint32_t a, uint32_t lo, uint32_t fold) {
        ksteps<FROM_L, ATM>([&](uint32_t ao, uint32_t ahi, uint32_t bo, uint32_t bhi, uint32_t acc) {
            step<ATM>(el, col, a + ao, ahi, lo + bo + ((uint32_t)(bhi == HI_TAIL ? T * BC * 16 : T * ATOM) >> 4), bhi, I_S, acc);
        });
        if constexpr (C::FOLD_TAIL) {
            if (k.fold_step()) step<ATM>(el, col, a + 8u * KS, HI_SW, lo + l_k(KS) + ((uint32_t)(T * ATOM) >> 4), HI_SW, I_S, 1u);
        } else if (k.fold_step()) {
            fold_step(el, col, k, fold, T, I_S);
        }
    }
    // Half of acc0 += A0 B0, acc1 += A1 B0 + A0 B1 (k-steps U0, U0 + 1 of four; the operand of a k-step lies at the columns of
    // the scores it replaces); acc = 0: the accumulators are overwritten.
    template <int U0>
    static __device__ __forceinline__ void outputs(uint32_t el, uint32_t a0, uint32_t a1, uint32_t lo, uint32_t acc) {
        constexpr uint32_t c0 = C::COL_ACC0, c1 = C::COL_ACC1;
#pragma unroll UNROLL
        for (int u = U0; u < U0 + 2; ++u) {
            const uint32_t b0 = lo + l_n(0, 0) + 128u * u, b1 = lo + l_n(1, 0) + 128u * u, o = 16u * u, first = U0 > 0 || u > 0 ? 1u : acc;
            ptx::mma_ts_acc(el, c0, a0 + o, b0, HI_SW, I_O, first);
            ptx::mma_ts_acc(el, c1, a1 + o, b0, HI_SW, I_O, first);
            ptx::mma_ts_acc(el, c1, a0 + o, b1, HI_SW, I_O, 1u);
        }
    }
    // DKV: acc[C] += A0 B0, acc[C + 1] += A1 B0 + A0 B1 (T2: the last of them; without G it is zero).
    template <bool T2, int ACC>
    static __device__ __forceinline__ void dkv_outputs(uint32_t el, uint32_t a0, uint32_t a1, uint32_t lo, uint32_t acc) {
        constexpr uint32_t c0 = ACC * DP, c1 = c0 + DP;
#pragma unroll UNROLL
        for (int u = 0; u < BC / 16; ++u) {
            const uint32_t b0 = lo + l_n(0, 0) + 128u * u, b1 = lo + l_n(1, 0) + 128u * u, o = 16u * u, first = u > 0 ? 1u : acc;
            ptx::mma_ts_acc(el, c0, a0 + o, b0, HI_SW, I_O, first);
            ptx::mma_ts_acc(el, c1, a1 + o, b0, HI_SW, I_O, first);
            if (T2) ptx::mma_ts_acc(el, c1, a0 + o, b1, HI_SW, I_O, 1u);
        }
    }
    // DKV_G: acc0 += P^T G (ACC 0), acc1 += dA^T Q (ACC 1); DQ_G: acc1 += dA K.
    template <int ACC>
    static __device__ __forceinline__ void g_outputs(uint32_t el, uint32_t a, uint32_t lo, uint32_t acc) {
#pragma unroll
        for (int u = 0; u < BC / 16; ++u)
            ptx::mma_ts_acc(el, ACC ? C::COL_ACC1 : C::COL_ACC0, a + 16u * u, lo + l_n(1 - ACC, 0) + 128u * u, HI_SW, I_O, u > 0 ? 1u : acc);
    }
};

// DKV: one buffer of (S, Sd | D, X), operands written over the scores.  Pipe order: outputs of the first pair (P, P Nn)(n - 1) |
// (S, Sd)(n) | outputs of the second pair (W, dA)(n - 1) | (D, X)(n): what the element-wise warps do to one pair runs under
// the MMAs of the other, so that no unit waits for the whole chain of a tile.  (d = 64, per 64 queries: MMAs of 1860 cycles
// instead of 2250 in two passes, half the exponentials and loads.)  The element-wise warps are done 400 to 800 cycles before
// their operands' turn, so this warp waits and commits twice per tile and no more: for the operands as a whole, together with
// the next stage of the ring, and one completion for outputs and scores.  (Operands handed over in halves, a wait per barrier
// and four commits: d = 72 (16, 16, 1024) 1034 -> 994 us for the backward.)  What bounds a tile now
// is the pipe with two operands in shared memory, whose port the loads share: 2950 cycles, 2490 with nothing to load or compute.
// The tiles run on through the items: the next item's first scores go in front of this one's last outputs, and each pair of
// accumulators is handed to and from the epilogue on its own.  (d = 72, DKV and DQ, (64, 16, 256): the backward 345 -> 334 us.)
template <int MODE, int DP, bool NO_G>
__device__ __forceinline__ void jvp_issue_dkv(const JvpParams& p, const JvpBlock<MODE, DP>& shared) {
    using C = JvpCfg<MODE, DP>;
    using I = JvpIssue<MODE, DP>;
    constexpr int BC = C::BC;
    const JvpBlock<MODE, DP> k = shared.pinned();
    const int T = jvp_pin(p.T);
    const uint32_t x0 = ptx::desc_lo(k.own_tile(0), 16), x1 = ptx::desc_lo(k.own_tile(1), 16);
    const uint32_t x2 = ptx::desc_lo(k.own_tile(2), 16), x3 = ptx::desc_lo(k.own_tile(3), 16);
    constexpr uint32_t cS = C::COL_SCORE, cT = cS + BC, cD = cS + 2 * BC, cX = cS + 3 * BC;
    JvpSlot e = I::e_slot(k), l = I::l_slot(k);   // next tile of the scores
    uint32_t elo = e.lo, llo = l.lo;              // stages of the outputs' tile
    const int last = jvp_item_count(p) * T;
    int sj = 0, si = 0, oj = -1, oi = 0;          // tile within its item and item: of the scores, of the outputs (one tile behind)
    bool ready = false;                           // what the next batch waits for was seen complete
    for (int n = 0; n <= last; ++n) {
        const bool out = n > 0, score = n < last;
        const uint32_t acc = oj > 0 ? 1u : 0u;
        // dtV += P^T Hc, dV += (P Nn)^T Hc + P^T G | (S, Sd) of the next tile
        if (!ready && !(score ? k.wait2(C::B_PREADY, n - 1, C::B_LFULL + l.s, l.ph) : k.wait(C::B_PREADY, n - 1))) return;
        if (oj == 0 && oi > 0 && !k.wait(C::B_ACCFREE, oi - 1)) return;    // the first tile overwrites the accumulators
        k.tile_fence();
        if (out) {
            const uint32_t el = ptx::elect_one();
            I::template dkv_outputs<!NO_G, 0>(el, cS, cT, elo, acc);
            if (oj == T - 1) ptx::mma_commit_p(el, k.bar(C::B_FINAL));
        }
        if (score) {
            if (sj == 0) {
                if (!k.wait(C::B_OWN, si)) return;
                k.tile_fence();
            }
            ready = ptx::mbar_test2_warp(k.bar(C::B_PREADY + 1), (n - 1) & 1, k.bar(C::B_EFULL + e.s), e.ph);
            const uint32_t el = ptx::elect_one();
            I::template pair<true, false, true>(el, cS, k, x0, x1, l.lo, l.fold, 0);
            ptx::mma_commit_p(el, k.bar(C::B_SFULL + (n & 3)));
            if (sj == T - 1) ptx::mma_commit_p(el, k.bar(C::B_OWNFREE));
            l.template next<C::SL, I::L_STEP, I::F_STEP>();
        } else {
            ready = false;
        }
        // dtK += W^T Q, dK += dA^T Q + W^T tQ | (D, X) of the next tile
        if (!ready && !(score ? k.wait2(C::B_PREADY + 1, n - 1, C::B_EFULL + e.s, e.ph) : k.wait(C::B_PREADY + 1, n - 1))) return;
        if (oj == 0 && oi > 0 && !k.wait(C::B_ACCFREE + 1, oi - 1)) return;
        k.tile_fence();
        if (out) {
            const uint32_t el = ptx::elect_one();
            I::template dkv_outputs<true, 2>(el, cD, cX, llo, acc);
            elo = elo + I::E_STEP == e.lo0 + C::SE * I::E_STEP ? e.lo0 : elo + I::E_STEP;
            llo = llo + I::L_STEP == l.lo0 + C::SL * I::L_STEP ? l.lo0 : llo + I::L_STEP;
            if (oj == T - 1) {
                ptx::mma_commit_p(el, k.bar(C::B_FINAL + 1));
                oj = -1;
                ++oi;
            }
        }
        ++oj;
        if (score) {
            if (sj == 0) {
                if (!k.wait(C::B_OWN + 1, si)) return;
                k.tile_fence();
            }
            // (the stage of the tile after the next one, where there is one)
            ready = n + 1 < last && ptx::mbar_test2_warp(k.bar(C::B_PREADY), n & 1, k.bar(C::B_LFULL + l.s), l.ph);
            const uint32_t el = ptx::elect_one();
            I::template pair<false, false, true>(el, cD, k, x2, x3, e.lo, e.fold, 0);
            ptx::mma_commit_p(el, k.bar(C::B_XFULL + (n & 3)));
            if (sj == T - 1) {
                ptx::mma_commit_p(el, k.bar(C::B_OWNFREE + 1));
                sj = -1;
                ++si;
            }
            ++sj;
            e.template next<C::SE, I::E_STEP, I::F_STEP>();
        }
    }
}

// FWD, DV: two score buffers taken in turn, operands written over the scores; pipe order S(0), S(1), out(0), S(2), out(1), ...:
// S(n + 1) overwrites what out(n - 1) reads, and the pipe keeps the order.
template <int MODE, int DP>
__device__ __forceinline__ void jvp_issue_one_pair(const JvpParams& p, const JvpBlock<MODE, DP>& shared) {
    using C = JvpCfg<MODE, DP>;
    using I = JvpIssue<MODE, DP>;
    constexpr int RDY = C::XT ? C::B_XRDY : C::B_OWN, FREE = C::XT ? C::B_XFREE : C::B_OWNFREE;
    const JvpBlock<MODE, DP> k = shared.pinned();
    const int T = jvp_pin(p.T), items = jvp_pin(p.items);
    const uint32_t x0 = C::XT ? C::COL_X0 : ptx::desc_lo(k.own_tile(0), 16), x1 = C::XT ? C::COL_X1 : ptx::desc_lo(k.own_tile(1), 16);
    JvpSlot e = I::e_slot(k), l = I::l_slot(k);
    int n = 0;                 // next tile whose scores are issued
    bool e_ready = false;      // its E stage was seen full
    int g = 0, it = 0;
    bool opened = false;       // the first scores of the item have been issued
    for (int item = blockIdx.x; item < items; item += gridDim.x, ++it) {
        const bool more = item + (int)gridDim.x < items;
        if (!opened && !k.wait(RDY, it)) return;
        for (int j = opened ? 0 : -1; j < T; ++j) {
            // The scores of the next tile go in front of this tile's outputs.  Where they open an item they do if its owner
            // operands are there already, else they follow when the loop gets there.
            bool go = j + 1 < T;
            if (!go) go = opened = more && ptx::mbar_test_warp(k.bar(RDY), (it + 1) & 1);
            if (go) {
                if (!e_ready && !k.wait(C::B_EFULL + e.s, e.ph)) return;
                k.tile_fence();
                const uint32_t el = ptx::elect_one();
                const uint32_t col = C::COL_SCORE + (n & 1) * 2 * C::BC;
                I::template pair<false, C::XT, true>(el, col, k, x0, x1, e.lo, e.fold, k.bar(C::B_SFULL + (n & 3)));
                ptx::mma_commit_p(el, k.bar(C::B_EDONE + (n & 3)));
                if (j + 2 == T || (T == 1 && j == 0)) ptx::mma_commit_p(el, k.bar(FREE));   // the item's last scores
                e.template next<C::SE, I::E_STEP, I::F_STEP>();
                ++n;
            }
            e_ready = ptx::mbar_test_warp(k.bar(C::B_EFULL + e.s), e.ph);
            if (j < 0) continue;
            const int b = g & 1;
            if (!k.wait2(C::B_PREADY + 2 * b, g >> 1, C::B_LFULL + l.s, l.ph)) return;
            // The first tile overwrites the accumulators.  (Waited for here and not before the item's first scores, and operands loaded
            // ahead: an item's end costs 2000 cycles instead of 5500.  d = 72: (64, 16, 256) 111 -> 106 us.)
            if (j == 0 && it > 0 && !k.wait(C::B_ACCFREE, it - 1)) return;
            k.tile_fence();
            const uint32_t a0 = C::COL_SCORE + b * 2 * C::BC;
            I::template outputs<0>(ptx::elect_one(), a0, a0 + C::BC, l.lo, j > 0 ? 1u : 0u);
            if (!k.wait(C::B_PREADY + 2 * b + 1, g >> 1)) return;
            ptx::tc_fence_after_sync();
            const uint32_t el = ptx::elect_one();
            I::template outputs<2>(el, a0, a0 + C::BC, l.lo, 1u);
            ptx::mma_commit_p(el, k.bar(C::B_OUTDONE + (g & 3)));
            if (j == T - 1) ptx::mma_commit_p(el, k.bar(C::B_FINAL));
            l.template next<C::SL, I::L_STEP, 0>();
            ++g;
        }
    }
}

// DK, DQ: one buffer of (S, Sd | D, X), the operands W, dA over D, X.  Pipe order: (S, Sd)(n) once (S, Sd)(n - 1) has been read |
// outputs(n - 1), half by half, as W, dA are written | (D, X)(n), which overwrites them.
template <int MODE, int DP, bool NO_G>
__device__ __forceinline__ void jvp_issue_two_pairs(const JvpParams& p, const JvpBlock<MODE, DP>& shared) {
    using C = JvpCfg<MODE, DP>;
    using I = JvpIssue<MODE, DP>;
    const JvpBlock<MODE, DP> k = shared.pinned();
    const int T = jvp_pin(p.T);
    const uint32_t x0 = ptx::desc_lo(k.own_tile(0), 16), x1 = ptx::desc_lo(k.own_tile(1), 16);
    const uint32_t x2 = C::XT ? C::COL_X0 : ptx::desc_lo(k.own_tile(2), 16), x3 = C::XT ? C::COL_X1 : ptx::desc_lo(k.own_tile(3), 16);
    constexpr uint32_t cS = C::COL_SCORE, cD = C::COL_SCORE + 2 * C::BC, cX = C::COL_SCORE + 3 * C::BC;
    constexpr bool X3 = !NO_G;   // DQ: X3 Y2^T = G V^T is zero with G absent
    JvpSlot e = I::e_slot(k), l = I::l_slot(k);
    uint32_t lo = l.lo;        // L stage of the outputs' tile
    const int last = jvp_item_count(p) * T;
    int sj = 0, si = 0, oj = -1, oi = 0;   // tile within its item and item: of the scores, of the outputs (one tile behind)
    for (int n = 0; n <= last; ++n) {
        const bool score = n < last;
        auto scores = [&]() {   // (S, Sd) of the next tile
            if (!k.wait2(C::B_SREAD, n - 1, C::B_LFULL + l.s, l.ph)) return false;   // (a fresh barrier passes for n = 0)
            if (sj == 0 && !k.wait(C::B_OWN, si)) return false;
            k.tile_fence();
            const uint32_t el = ptx::elect_one();
            I::template pair<true, false, true>(el, cS, k, x0, x1, l.lo, l.fold, 0);
            ptx::mma_commit_p(el, k.bar(C::B_SFULL + (n & 3)));
            if (C::XT && sj == T - 1) ptx::mma_commit_p(el, k.bar(C::B_OWNFREE));
            l.template next<C::SL, I::L_STEP, I::F_STEP>();
            return true;
        };
        // Where an item opens with owner tiles that the item before has used to its end (WIDE), its outputs go first.
        const bool first = C::XT || sj > 0;
        if (score && first && !scores()) return;
        const bool e_ready = ptx::mbar_test_warp(k.bar(C::B_EFULL + e.s), e.ph);
        if (n > 0) {       // outputs
            if (!k.wait(C::B_PREADY, n - 1)) return;
            if (oj == 0 && oi > 0 && !k.wait(C::B_ACCFREE, oi - 1)) return;    // the first tile overwrites the accumulators
            ptx::tc_fence_after_sync();
            I::template outputs<0>(ptx::elect_one(), cD, cX, lo, oj > 0 ? 1u : 0u);
            if (!k.wait(C::B_PREADY + 1, n - 1)) return;
            ptx::tc_fence_after_sync();
            const uint32_t el = ptx::elect_one();
            I::template outputs<2>(el, cD, cX, lo, 1u);
            ptx::mma_commit_p(el, k.bar(C::B_OUTDONE + ((n - 1) & 3)));
            if (oj == T - 1) {
                ptx::mma_commit_p(el, k.bar(C::B_FINAL));
                oj = -1;
                ++oi;
            }
            lo = lo + I::L_STEP == l.lo0 + C::SL * I::L_STEP ? l.lo0 : lo + I::L_STEP;
        }
        ++oj;
        if (score && !first && !scores()) return;
        if (score) {       // (D, X) of the next tile
            if (!e_ready && !k.wait(C::B_EFULL + e.s, e.ph)) return;
            if (C::XT && sj == 0 && !k.wait(C::B_XRDY, si)) return;
            k.tile_fence();
            const uint32_t el = ptx::elect_one();
            I::template pair<false, C::XT, X3>(el, cD, k, x2, x3, e.lo, e.fold, 0);
            ptx::mma_commit_p(el, k.bar(C::B_XFULL + (n & 3)));
            if (sj == T - 1) {
                ptx::mma_commit_p(el, k.bar(C::XT ? C::B_XFREE : C::B_OWNFREE));
                sj = -1;
                ++si;
            }
            ++sj;
            e.template next<C::SE, I::E_STEP, I::F_STEP>();
        }
    }
}

// DKV_G, DQ_G: two score buffers taken in turn, operands written over the scores.  Pipe order: dV(n - 2) | S(n) | dK(n - 3) | X(n - 1)
// (DQ_G: S(n) | dQ(n - 3) | X(n - 1)): while a group works on tile n - 2 the other's n - 3 is complete, and the scores of what
// either takes next are there before it asks for them.  (d = 72 (16, 16, 1024), events around each kernel, below the power cap: 314 +
// 202 us for the two passes as specialisations of DKV and DQ, whose layout has room for tiles of 48, one buffer and owners in
// shared memory; 163 + 136 now.)  One wait a tile, for everything that the tile's batch needs (P(n - 2)
// written, or S(n - 2) read; dA(n - 3) written; stage n full): with a wait in front of every product this warp was what bounded a
// tile (DQ_G, d = 72: 1240 cycles, MMAs of 480).
template <int MODE, int DP>
__device__ __forceinline__ void jvp_issue_g(const JvpParams& p, const JvpBlock<MODE, DP>& shared) {
    using C = JvpCfg<MODE, DP>;
    using I = JvpIssue<MODE, DP>;
    constexpr bool KEYS = MODE == PASS_DKV_G;
    const JvpBlock<MODE, DP> k = shared.pinned();
    const int T = jvp_pin(p.T), last = jvp_item_count(p) * T;
    JvpSlot l = I::l_slot(k);
    uint32_t xlo = 0, xfold = 0, vlo = 0, klo = 0;   // stages of the tiles n - 1, n - 2, n - 3
    uint32_t first = 0, end = 0;                     // bit i: tile n - i is the first, the last of its item
    int sj = 0, si = 0, xi = 0, oi = 0;              // tile within its item; items opened by S, by X, by the outputs
    for (int n = 0; n < last + 3; ++n) {
        const bool score = n < last, x = n >= 1 && n <= last, v_out = n >= 2 && n < last + 2, k_out = n >= 3;
        const int ba = C::B_PREADY + 2 * (n & 1), bb = C::B_PREADY + 2 * ((n - 1) & 1) + 1, pa = ((n - 2) >> 1) & 1, pb = ((n - 3) >> 1) & 1;
        if (!(k_out && score && ptx::mbar_test3_warp(k.bar(ba), pa, k.bar(bb), pb, k.bar(C::B_LFULL + l.s), l.ph))) {
            if (v_out && !k.wait(ba, pa)) return;
            if (k_out && !k.wait(bb, pb)) return;
            if (score && !k.wait(C::B_LFULL + l.s, l.ph)) return;
        }
        first = first << 1 | (score && sj == 0 ? 1u : 0u);
        end = end << 1 | (score && sj == T - 1 ? 1u : 0u);
        const uint32_t col = C::COL_SCORE + (n & 1) * 2 * C::BC, colx = C::COL_SCORE + ((n - 1) & 1) * 2 * C::BC + C::BC;
        // first output MMAs of an item: they overwrite the accumulators
        auto acc_free = [&]() { return oi++ == 0 || k.wait(C::B_ACCFREE, oi - 2); };
        auto part_x = [&]() {
            if (!KEYS && (first & 8u) && !acc_free()) return false;
            if ((first & 2u) && !k.wait(C::B_XRDY + 1, xi++)) return false;
            ptx::tc_fence_after_sync();
            const uint32_t el = ptx::elect_one();
            if (k_out) {
                I::template g_outputs<1>(el, colx, klo, first & 8u ? 0u : 1u);
                ptx::mma_commit_p(el, k.bar(C::B_OUTDONE + ((n - 3) & (C::NOUTDONE - 1))));
                if (end & 8u) ptx::mma_commit_p(el, k.bar(C::B_FINAL));
            }
            if (x) {
                const uint32_t el2 = ptx::elect_one();
                I::template single<true, true, 1>(el2, colx, k, C::COL_X1, xlo, xfold);
                ptx::mma_commit_p(el2, k.bar(C::B_XFULL + ((n - 1) & 3)));
                if (end & 2u) ptx::mma_commit_p(el2, k.bar(C::B_XFREE + 1));
            }
            return true;
        };
        // the item before is still to be ended
        const bool swap = KEYS && (first & 4u);
        if (swap && !part_x()) return;
        if (KEYS && (first & 4u) && !acc_free()) return;
        if ((first & 1u) && !k.wait(C::B_XRDY, si++)) return;
        k.tile_fence();
        if (KEYS && v_out) I::template g_outputs<0>(ptx::elect_one(), col, vlo, first & 4u ? 0u : 1u);
        if (score) {
            const uint32_t el = ptx::elect_one();
            I::template single<true, true, 0>(el, col, k, C::COL_X0, l.lo, l.fold);
            ptx::mma_commit_p(el, k.bar(C::B_SFULL + (n & 3)));
            if (end & 1u) ptx::mma_commit_p(el, k.bar(C::B_XFREE));
        }
        if (!swap && !part_x()) return;
        klo = vlo;
        vlo = xlo;
        xlo = l.lo;
        xfold = l.fold;
        if (score) {
            l.template next<C::SL, I::L_STEP, I::F_STEP>();
            if (++sj == T) sj = 0;
        }
    }
}

// Whether G is absent is decided here, once (WIDE head dims take both cotangents; without Hc the passes are DKV_G and DQ_G).
template <int MODE, int DP, bool NO_G>
__device__ __forceinline__ void jvp_issue_abs(const JvpParams& p, const JvpBlock<MODE, DP>& k) {
    if constexpr (JvpCfg<MODE, DP>::GONLY) jvp_issue_g<MODE, DP>(p, k);
    else if constexpr (MODE == PASS_DKV) jvp_issue_dkv<MODE, DP, NO_G>(p, k);
    else if constexpr (JvpCfg<MODE, DP>::NPAIR == 1) jvp_issue_one_pair<MODE, DP>(p, k);
    else jvp_issue_two_pairs<MODE, DP, NO_G>(p, k);
}
template <int MODE, int DP>
__device__ __forceinline__ void jvp_issue(const JvpParams& p, const JvpBlock<MODE, DP>& k) {
    if constexpr (JvpCfg<MODE, DP>::NPAIR == 1 || JvpCfg<MODE, DP>::WIDE) jvp_issue_abs<MODE, DP, false>(p, k);
    else if (!p.no_g) jvp_issue_abs<MODE, DP, false>(p, k);
    else jvp_issue_abs<MODE, DP, true>(p, k);
}

// ------------------------------------------------------------------------------------------------ element-wise warps
// Forward, DKV_G, DQ_G: the two groups take the tiles in turn; a thread has owner row `row` and the 64 columns of the tile.  The
// other passes: all eight warps work on every tile; a thread has the 32 columns of its group's half (DKV: of half the rows, all
// columns).  (With one score buffer, or in the shorter DV tile, the tensor pipe waits for how long a tile takes; the forward, with
// two, measured 8 % slower that way, with the row maxima to exchange.)  Reads of tensor memory are issued for many columns at once
// (a read costs 180 cycles whatever its width) and released with one arrival per warp; the operands are handed over half by half
// (DKV, DKV_G, DQ_G: whole).

// Forward.  The reference m of a row and the centre c of its tangent weights are shared by the two groups: the warp that
// has a row's tile g decides whether to move them and hands the row state on to the warp that has tile g + 1 (B_TURN), long
// before that one needs it.  m follows the running maximum only when a tile maximum exceeds it by more than JVP_LAZY_LOG2
// (rare after the first tile): then m moves to the new maximum, c to T at the new arg-max key (WIDE: c on its own, whenever
// it is too far off), and the accumulators are rescaled, R += (c_old - c_new) O~ keeping them consistent.  Centring T keeps the bf16 rounding of P~ (T - c) small where
// P~ is large, so that tO = R/l - (mu - c) O does not cancel badly on rows with a peaked softmax.
template <int DP>
__device__ __forceinline__ void jvp_elem_fwd(const JvpParams& p, const JvpBlock<PASS_FWD, DP>& k, int grp, int q, int lane) {
    using C = JvpCfg<PASS_FWD, DP>;
    constexpr int BC = C::BC;
    const int row = q * 32 + lane;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    const uint64_t c2c2 = ptx::pack2(p.c2, p.c2), aa = ptx::pack2(p.alpha, p.alpha);
    bool ok = true;
    int it = 0;
    for (int item = blockIdx.x; ok && item < p.items; item += gridDim.x, ++it) {
        const int g0 = it * p.T;
        float m_own = -CUDART_INF_F, c_own = 0.f;   // reference and centre of this thread's sums
        uint64_t l2 = 0ull, mt2 = 0ull;             // two partial sums each of P~ and of P~ (T - c) over this group's tiles
        for (int j = (grp ^ g0) & 1; j < p.T; j += 2) {
            const int g = g0 + j, b = g & 1;
            const uint32_t sb = lanes + C::COL_SCORE + b * 2 * BC;
            uint32_t s[64], t[64];
            ok = k.done(C::B_SFULL, g);   // S is complete before Sd
            if (!ok) break;
            ptx::tc_fence_after_sync();
            ptx::tmem_ld32(sb, s);
            ptx::tmem_ld32(sb + 32, s + 32);
            ptx::tmem_wait_ld();
            const int nvalid = p.s.rows - j * BC;  // columns that are real keys
            if (__builtin_expect(nvalid < BC, 0)) {
#pragma unroll
                for (int c = 0; c < BC; ++c)
                    if (c >= nvalid) s[c] = __float_as_uint(-CUDART_INF_F);
            }
            float mx[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                mx[i] = __uint_as_float(s[16 * i]);
#pragma unroll
                for (int c = 1; c < 15; c += 2) mx[i] = ptx::max3(mx[i], __uint_as_float(s[16 * i + c]), __uint_as_float(s[16 * i + c + 1]));
                mx[i] = fmaxf(mx[i], __uint_as_float(s[16 * i + 15]));
            }
            const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            const float mrow = top * p.c2;         // tile maximum of the row, log2 units
            ok = k.done(C::B_XFULL, g);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (g > 0) ok = k.wait(C::B_TURN + q, g - 1);
            if (!ok) break;
            float m_ref = -CUDART_INF_F, cen = 0.f, m_max = -CUDART_INF_F;
            if (j > 0) { const float4 st = k.row_state(row); m_ref = st.x; cen = st.y; m_max = st.z; }
            bool scaling = mrow > m_ref + (C::WIDE ? JVP_LAZY_LOG2_WIDE : JVP_LAZY_LOG2), centring = C::WIDE ? mrow > m_max : scaling;
            if (__builtin_expect(__any_sync(0xffffffffu, centring), 0)) {
                ptx::tmem_ld32(sb + BC, t);
                ptx::tmem_ld32(sb + BC + 32, t + 32);
                ptx::tmem_wait_ld();
                float lt = 0.f;                    // Sd at the arg-max key (the first one)
#pragma unroll
                for (int c = BC - 1; c >= 0; --c) lt = __uint_as_float(s[c]) == top ? __uint_as_float(t[c]) : lt;
                const float tw = lt * p.alpha;
                if (C::WIDE) {
                    centring = centring && (j == 0 || fabsf(tw - cen) > JVP_CENTRE_WIDE);
                    m_max = fmaxf(m_max, mrow);
                }
                const float scale = scaling ? ptx::ex2(m_ref - mrow) : 1.0f;
                const float fix = centring ? cen - tw : 0.f;
                if (scaling) m_ref = mrow;
                if (centring) cen = tw;
                if (j > 0 && (!C::WIDE || __any_sync(0xffffffffu, scaling || centring))) {
                    // accumulators must be at rest: the value MMAs of tile g - 1 have completed
                    ok = k.done(C::B_OUTDONE, g - 1);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    // Many columns at a time (s and t are read again below): a round trip through tensor memory takes 250
                    // cycles whatever its width, and the next tile of the row waits.  (Peaked inputs, d = 128 (2, 24, 4096): 1321 -> 1245 us
                    // against eight columns.)
                    constexpr int NC = DP % 32 == 0 ? 32 : 16;
#pragma unroll 1
                    for (int c0 = 0; c0 < DP; c0 += NC) {
                        uint32_t o[NC], r[NC];
                        if constexpr (NC == 32) {
                            ptx::tmem_ld32(lanes + C::COL_ACC0 + c0, o);
                            ptx::tmem_ld32(lanes + C::COL_ACC1 + c0, r);
                        } else {
                            ptx::tmem_ld16(lanes + C::COL_ACC0 + c0, o);
                            ptx::tmem_ld16(lanes + C::COL_ACC1 + c0, r);
                        }
                        ptx::tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const float ov = __uint_as_float(o[c]);
                            r[c] = __float_as_uint(scale * fmaf(fix, ov, __uint_as_float(r[c])));
                            o[c] = __float_as_uint(scale * ov);
                        }
#pragma unroll
                        for (int c = 0; c < NC; c += 8) {
                            ptx::tmem_st8(lanes + C::COL_ACC0 + c0 + c, o + c);
                            ptx::tmem_st8(lanes + C::COL_ACC1 + c0 + c, r + c);
                        }
                    }
                    ptx::tmem_wait_st();
                }
                k.row_state(row) = make_float4(m_ref, cen, m_max, 0.f);
            }
            k.arrive(C::B_TURN + q, lane);
            if (__builtin_expect(__any_sync(0xffffffffu, m_ref != m_own || (C::WIDE && cen != c_own)), 0)) {   // the reference has moved since this group's last tile
                const float scale = ptx::ex2(m_own - m_ref), fix = c_own - cen;
                float l0, l1, t0, t1;
                ptx::unpack2(l2, l0, l1);
                ptx::unpack2(mt2, t0, t1);
                l2 = ptx::pack2(l0 * scale, l1 * scale);
                mt2 = ptx::pack2(scale * fmaf(fix, l0, t0), scale * fmaf(fix, l1, t1));
                m_own = m_ref;
                c_own = cen;
            }
            // ---- P~ = 2^(c2 s - m), P~ (T - c): operands of a k-step (16 keys) at the columns of the scores they replace
            const uint64_t nm = ptx::pack2(-m_ref, -m_ref), nc = ptx::pack2(-cen, -cen);
#pragma unroll 1
            for (int h = 0; h < BC; h += 32) {   // rolled: half the code (the roles of a scheduler share its instruction cache)
                ptx::tmem_ld32(sb + h, s);
                ptx::tmem_ld32(sb + BC + h, t);
                ptx::tmem_wait_ld();
                if (__builtin_expect(nvalid < BC, 0)) {
#pragma unroll
                    for (int c = 0; c < 32; ++c)
                        if (h + c >= nvalid) s[c] = __float_as_uint(-CUDART_INF_F);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    uint32_t pp[8], ppt[8];
#pragma unroll
                    for (int c = 0; c < 16; c += 2) {
                        const uint64_t x2 = ptx::fma2(ptx::pack2u(s[16 * u + c], s[16 * u + c + 1]), c2c2, nm);
                        float x0, x1;
                        ptx::unpack2(x2, x0, x1);
                        const float p0 = ptx::ex2(x0), p1 = ptx::ex2(x1);
                        const uint64_t p2 = ptx::pack2(p0, p1);
                        const uint64_t pt2 = ptx::mul2(p2, ptx::fma2(ptx::pack2u(t[16 * u + c], t[16 * u + c + 1]), aa, nc));
                        l2 = ptx::add2(l2, p2);
                        mt2 = ptx::add2(mt2, pt2);
                        float q0, q1;
                        ptx::unpack2(pt2, q0, q1);
                        pp[c >> 1] = ptx::pack_bf16(p0, p1);
                        ppt[c >> 1] = ptx::pack_bf16(q0, q1);
                    }
                    ptx::tmem_st8(sb + h + 16 * u, pp);
                    ptx::tmem_st8(sb + BC + h + 16 * u, ppt);
                }
                ptx::tmem_wait_st();
                k.arrive(C::B_PREADY + 2 * b + (h >> 5), lane);   // half of the output MMAs may go
            }
        }
        if (!ok) break;
        // the item's sums of this group, for the epilogue (which has read those of the item before)
        if (it > 0) ok = k.wait(C::B_ACCFREE, it - 1);
        float l0, l1, t0, t1;
        ptx::unpack2(l2, l0, l1);
        ptx::unpack2(mt2, t0, t1);
        k.row_sums(grp * JVP_ROWS + row) = make_float4(l0 + l1, t0 + t1, m_own, c_own);
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(k.bar(C::B_ROWSTAT));
    }
}

// DV: P, P Nn from (S, Sd), written over them.
template <int DP>
__device__ __forceinline__ void jvp_elem_dv(const JvpParams& p, const JvpBlock<PASS_DV, DP>& k, int grp, int q, int lane) {
    using C = JvpCfg<PASS_DV, DP>;
    constexpr int BC = C::BC, HC = BC / 2;
    const uint32_t sb0 = (static_cast<uint32_t>(q * 32) << 16) + C::COL_SCORE + grp * HC;
    const uint64_t c2c2 = ptx::pack2(p.c2, p.c2), aa = ptx::pack2(p.alpha, p.alpha);
    const int tiles = jvp_item_count(p) * p.T;
    for (int g = 0; g < tiles; ++g) {
        const int b = g & 1;
        const uint32_t sb = sb0 + b * 2 * BC;
        if (!k.done(C::B_SFULL, g)) return;
        if (!k.wait(C::B_LFULL + g % C::SL, g / C::SL)) return;   // the tile's statistics
        ptx::tc_fence_after_sync();
        uint32_t s[HC], t[HC];
        ptx::tmem_ld32(sb, s);
        ptx::tmem_ld32(sb + BC, t);
        ptx::tmem_wait_ld();
        const float* st = k.stats(g % C::SL) + grp * HC;
#pragma unroll
        for (int u = 0; u < HC / 16; ++u) {
            uint32_t pa0[8], pa1[8];
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
                const int cc = 16 * u + c;
                const ulonglong2 l4 = *reinterpret_cast<const ulonglong2*>(st + cc);
                const ulonglong2 m4 = *reinterpret_cast<const ulonglong2*>(st + BC + cc);
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                    const uint64_t s2 = ptx::pack2u(s[cc + e], s[cc + e + 1]);
                    float x0, x1;
                    ptx::unpack2(ptx::fma2(s2, c2c2, e ? l4.y : l4.x), x0, x1);
                    const float p0 = ptx::ex2(x0), p1 = ptx::ex2(x1);
                    pa0[(c + e) >> 1] = ptx::pack_bf16(p0, p1);
                    const uint64_t t2 = ptx::pack2u(t[cc + e], t[cc + e + 1]);
                    const uint64_t n2 = ptx::fma2(t2, aa, ptx::neg2(e ? m4.y : m4.x));
                    float q0, q1;
                    ptx::unpack2(ptx::mul2(ptx::pack2(p0, p1), n2), q0, q1);
                    pa1[(c + e) >> 1] = ptx::pack_bf16(q0, q1);
                }
            }
            ptx::tmem_st8(sb + 16 * u, pa0);
            ptx::tmem_st8(sb + BC + 16 * u, pa1);
        }
        ptx::tmem_wait_st();
        k.arrive(C::B_PREADY + 2 * b + grp, lane);
    }
}

// DK, DQ.  Phase A: P and Nn from (S, Sd), kept in registers; phase B: W = P (D - Sigma1), dA = P (X - c) + W Nn, written over
// D and X.  The statistics belong to the columns (DK) or to this thread's row (DQ).
template <int MODE, int DP>
__device__ __forceinline__ void jvp_elem_two_pairs(const JvpParams& p, const JvpBlock<MODE, DP>& k, int grp, int q, int lane) {
    using C = JvpCfg<MODE, DP>;
    constexpr int BC = C::BC, HC = BC / 2;
    constexpr bool COL = C::TRANSPOSED, ROW = !COL;
    const int row = q * 32 + lane;
    const uint32_t sb = (static_cast<uint32_t>(q * 32) << 16) + C::COL_SCORE + grp * HC;
    const uint64_t c2c2 = ptx::pack2(p.c2, p.c2), aa = ptx::pack2(p.alpha, p.alpha);
    // DQ: the statistics of this thread's row in the next item, loaded one item ahead
    [[maybe_unused]] float n_lse2 = -CUDART_INF_F, n_mu = 0.f, n_s1 = 0.f, n_cv = 0.f;
    [[maybe_unused]] auto load_stats = [&](int item) {
        const int bh = item / p.row_tiles, r = (item - bh * p.row_tiles) * JVP_ROWS + row;
        n_lse2 = -CUDART_INF_F; n_mu = n_s1 = n_cv = 0.f;
        if (item < p.items && r < p.o.rows) {
            const size_t at = (size_t)bh * p.o.rows + r;
            n_lse2 = p.nlse2[at]; n_mu = p.mu[at]; n_s1 = p.nsig1[at]; n_cv = p.ncvec[at];
        }
    };
    if (ROW) load_stats(blockIdx.x);
    int g = 0;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x) {
        [[maybe_unused]] const uint64_t r_l = ptx::pack2(n_lse2, n_lse2), r_nm = ptx::pack2(-n_mu, -n_mu), r_s = ptx::pack2(n_s1, n_s1), r_c = ptx::pack2(n_cv, n_cv);
        if (ROW) load_stats(item + gridDim.x);
        for (int j = 0; j < p.T; ++j, ++g) {
            [[maybe_unused]] const float* st = COL ? k.stats(g % C::SL) + grp * HC : nullptr;
            uint64_t P2[HC / 2], N2[HC / 2];
            // ---- phase A
            if (!k.done(C::B_SFULL, g)) return;
            if (COL && !k.wait(C::B_LFULL + g % C::SL, g / C::SL)) return;   // (complete: those MMAs read the tile's L stage)
            ptx::tc_fence_after_sync();
            {
                uint32_t s[HC], t[HC];
                ptx::tmem_ld32(sb, s);
                ptx::tmem_ld32(sb + BC, t);
                ptx::tmem_wait_ld();
                k.arrive(C::B_SREAD, lane);
                const int nvalid = p.s.rows - j * BC - grp * HC;
                if (ROW && __builtin_expect(nvalid < HC, 0)) {   // keys beyond N: P = 0
#pragma unroll
                    for (int c = 0; c < HC; ++c)
                        if (c >= nvalid) s[c] = __float_as_uint(-CUDART_INF_F);   // c2 s = -inf (c2 > 0)
                }
#pragma unroll
                for (int c = 0; c < HC; c += 4) {
                    [[maybe_unused]] ulonglong2 l4, m4;
                    if (COL) l4 = *reinterpret_cast<const ulonglong2*>(st + c);
                    if (COL) m4 = *reinterpret_cast<const ulonglong2*>(st + BC + c);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int i = c / 2 + e;
                        const uint64_t s2 = ptx::pack2u(s[2 * i], s[2 * i + 1]);
                        float x0, x1;
                        ptx::unpack2(ptx::fma2(s2, c2c2, COL ? (e ? l4.y : l4.x) : r_l), x0, x1);
                        P2[i] = ptx::pack2(ptx::ex2(x0), ptx::ex2(x1));
                        const uint64_t ts = ptx::pack2u(t[2 * i], t[2 * i + 1]);
                        N2[i] = ptx::fma2(ts, aa, COL ? ptx::neg2(e ? m4.y : m4.x) : r_nm);
                    }
                }
            }
            // The exponentials run while (D, X) are on their way (DQ, B 8, H 16, N 4096, d 64: 1720 cycles a tile; 2110 where the
            // compiler puts them behind the wait).
            uint64_t all = 0ull;
#pragma unroll
            for (int i = 0; i < HC / 2; ++i) all ^= P2[i];
            jvp_force(all);
            // ---- phase B
            if (!k.done(C::B_XFULL, g)) return;
            ptx::tc_fence_after_sync();
            uint32_t dd[HC], xx[HC];
            ptx::tmem_ld32(sb + 2 * BC, dd);
            ptx::tmem_ld32(sb + 3 * BC, xx);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < HC / 16; ++u) {
                uint32_t pa0[8], pa1[8];
#pragma unroll
                for (int c = 0; c < 16; c += 4) {
                    [[maybe_unused]] ulonglong2 s4, c4;
                    if (COL) s4 = *reinterpret_cast<const ulonglong2*>(st + 2 * BC + 16 * u + c);
                    if (COL) c4 = *reinterpret_cast<const ulonglong2*>(st + 3 * BC + 16 * u + c);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int i = c / 2 + e, gi = 8 * u + i;
                        uint64_t x2 = ptx::pack2u(xx[2 * gi], xx[2 * gi + 1]);
                        x2 = ptx::add2(x2, COL ? (e ? c4.y : c4.x) : r_c);
                        const uint64_t t2 = ptx::mul2(P2[gi], x2);
                        float d0, d1, w0, w1;
                        uint64_t y2 = ptx::pack2u(dd[2 * gi], dd[2 * gi + 1]);
                        y2 = ptx::add2(y2, COL ? (e ? s4.y : s4.x) : r_s);
                        const uint64_t w2 = ptx::mul2(P2[gi], y2);
                        ptx::unpack2(w2, w0, w1);
                        ptx::unpack2(ptx::fma2(w2, N2[gi], t2), d0, d1);
                        pa0[i] = ptx::pack_bf16(w0, w1);
                        pa1[i] = ptx::pack_bf16(d0, d1);
                    }
                }
                ptx::tmem_st8(sb + 2 * BC + 16 * u, pa0);
                ptx::tmem_st8(sb + 3 * BC + 16 * u, pa1);
            }
            ptx::tmem_wait_st();
            k.arrive(C::B_PREADY + grp, lane);
        }
    }
}

// DKV.  Both halves of a tile's work in place: P, P Nn over S, Sd, then W, dA over D, X.  A warp has 16 rows of its lane
// quadrant (the two groups share the 32) and all columns, so that the operand of a k-step, which replaces 16 columns, is never
// put together by two warps, whatever the width of the tile.  The statistics are in the scores already, so it does not
// matter which element of a row a thread holds: 16 lanes x 256 bits are read, and two neighbouring values packed make
// 16 lanes x 128 bits.
template <int DP>
__device__ __forceinline__ void jvp_elem_dkv(const JvpParams& p, const JvpBlock<PASS_DKV, DP>& k, int grp, int q, int lane) {
    using C = JvpCfg<PASS_DKV, DP>;
    constexpr int BC = C::BC, NU = BC / 16;
    const uint32_t sb = (static_cast<uint32_t>(q * 32 + grp * 16) << 16) + C::COL_SCORE;
    const uint64_t c2c2 = ptx::pack2(p.c2, p.c2), aa = ptx::pack2(p.alpha, p.alpha);
    const int tiles = jvp_item_count(p) * p.T;
    for (int g = 0; g < tiles; ++g) {
        uint64_t P2[4 * NU], N2[4 * NU];
        uint32_t y[8 * NU], x[8 * NU];   // S, Sd, then D, X
        if (!k.done(C::B_SFULL, g)) return;
        ptx::tc_fence_after_sync();
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            ptx::tmem_ld16_256x2(sb + 16 * u, y + 8 * u);
            ptx::tmem_ld16_256x2(sb + BC + 16 * u, x + 8 * u);
        }
        ptx::tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            uint32_t a0[4], a1[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = 4 * u + i;
                float x0, x1;
                ptx::unpack2(ptx::mul2(ptx::pack2u(y[2 * c], y[2 * c + 1]), c2c2), x0, x1);
                x0 = ptx::ex2(x0); x1 = ptx::ex2(x1);
                P2[c] = ptx::pack2(x0, x1);
                a0[i] = ptx::pack_bf16(x0, x1);
                N2[c] = ptx::mul2(ptx::pack2u(x[2 * c], x[2 * c + 1]), aa);
                ptx::unpack2(ptx::mul2(P2[c], N2[c]), x0, x1);
                a1[i] = ptx::pack_bf16(x0, x1);
            }
            ptx::tmem_st16_128x2(sb + 16 * u, a0);
            ptx::tmem_st16_128x2(sb + BC + 16 * u, a1);
        }
        ptx::tmem_wait_st();
        k.arrive(C::B_PREADY, lane);
        if (!k.done(C::B_XFULL, g)) return;
        ptx::tc_fence_after_sync();
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            ptx::tmem_ld16_256x2(sb + 2 * BC + 16 * u, y + 8 * u);
            ptx::tmem_ld16_256x2(sb + 3 * BC + 16 * u, x + 8 * u);
        }
        ptx::tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            uint32_t a0[4], a1[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = 4 * u + i;
                uint64_t t2 = ptx::mul2(P2[c], ptx::pack2u(x[2 * c], x[2 * c + 1]));
                float x0, x1;
                const uint64_t w2 = ptx::mul2(P2[c], ptx::pack2u(y[2 * c], y[2 * c + 1]));
                ptx::unpack2(w2, x0, x1);
                a0[i] = ptx::pack_bf16(x0, x1);
                t2 = ptx::fma2(w2, N2[c], t2);
                ptx::unpack2(t2, x0, x1);
                a1[i] = ptx::pack_bf16(x0, x1);
            }
            ptx::tmem_st16_128x2(sb + 2 * BC + 16 * u, a0);
            ptx::tmem_st16_128x2(sb + 3 * BC + 16 * u, a1);
        }
        ptx::tmem_wait_st();
        k.arrive(C::B_PREADY + 1, lane);
    }
}

// DKV_G, DQ_G.  The groups take tiles in turn, a row per thread.  DKV_G: P over S, dA = P X over X (the statistics are in the
// scores); DQ_G: dA = P (X - c) over X, statistics of this thread's row.
template <int MODE, int DP>
__device__ __forceinline__ void jvp_elem_g(const JvpParams& p, const JvpBlock<MODE, DP>& k, int grp, int q, int lane) {
    using C = JvpCfg<MODE, DP>;
    constexpr int BC = C::BC;
    constexpr bool ROW = MODE == PASS_DQ_G;
    const int row = q * 32 + lane, T = p.T, grid = gridDim.x;
    const uint32_t sb0 = (static_cast<uint32_t>(q * 32) << 16) + C::COL_SCORE + grp * 2 * BC;
    const uint64_t c2c2 = ptx::pack2(p.c2, p.c2);
    [[maybe_unused]] float n_lse2 = -CUDART_INF_F, n_cv = 0.f;
    [[maybe_unused]] auto load_stats = [&](int item) {
        const int bh = item / p.row_tiles, r = (item - bh * p.row_tiles) * JVP_ROWS + row;
        n_lse2 = -CUDART_INF_F; n_cv = 0.f;
        if (item < p.items && r < p.o.rows) {
            const size_t at = (size_t)bh * p.o.rows + r;
            n_lse2 = p.nlse2[at]; n_cv = p.ncvec[at];
        }
    };
    // item and tile within it: of this tile, and of the group's next one, whose row's statistics are loaded ahead
    int item = blockIdx.x, j = grp;
    for (; j >= T && item < p.items; j -= T) item += grid;
    if (ROW) load_stats(item);
    [[maybe_unused]] uint64_t r_l = ptx::pack2(n_lse2, n_lse2), r_c = ptx::pack2(n_cv, n_cv);
    for (int g = grp; item < p.items; g += 2) {
        int item1 = item, j1 = j + 2;
        for (; j1 >= T && item1 < p.items; j1 -= T) item1 += grid;
        if (ROW && item1 != item) load_stats(item1);
        uint64_t P2[BC / 2];
        if (!k.done(C::B_SFULL, g)) return;
        ptx::tc_fence_after_sync();
        {
            uint32_t s[BC];
            ptx::tmem_ld32(sb0, s);
            ptx::tmem_ld32(sb0 + 32, s + 32);
            ptx::tmem_wait_ld();
            if (ROW) k.arrive(C::B_PREADY + 2 * grp, lane);
            const int nvalid = p.s.rows - j * BC;
            if (ROW && __builtin_expect(nvalid < BC, 0)) {   // keys beyond N: P = 0
#pragma unroll
                for (int c = 0; c < BC; ++c)
                    if (c >= nvalid) s[c] = __float_as_uint(-CUDART_INF_F);   // c2 s = -inf (c2 > 0)
            }
#pragma unroll
            for (int i = 0; i < BC / 2; ++i) {
                const uint64_t s2 = ptx::pack2u(s[2 * i], s[2 * i + 1]);
                float x0, x1;
                ptx::unpack2(ROW ? ptx::fma2(s2, c2c2, r_l) : ptx::mul2(s2, c2c2), x0, x1);
                P2[i] = ptx::pack2(ptx::ex2(x0), ptx::ex2(x1));
            }
        }
        if (!ROW) {
#pragma unroll
            for (int u = 0; u < BC / 16; ++u) {
                uint32_t pa[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float x0, x1;
                    ptx::unpack2(P2[8 * u + i], x0, x1);
                    pa[i] = ptx::pack_bf16(x0, x1);
                }
                ptx::tmem_st8(sb0 + 16 * u, pa);
            }
            ptx::tmem_wait_st();
            k.arrive(C::B_PREADY + 2 * grp, lane);
        } else {   // the exponentials run while X is on its way
            uint64_t all = 0ull;
#pragma unroll
            for (int i = 0; i < BC / 2; ++i) all ^= P2[i];
            jvp_force(all);
        }
        if (!k.done(C::B_XFULL, g)) return;
        ptx::tc_fence_after_sync();
        uint32_t x[BC];
        ptx::tmem_ld32(sb0 + BC, x);
        ptx::tmem_ld32(sb0 + BC + 32, x + 32);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < BC / 16; ++u) {
            uint32_t pa[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int c = 8 * u + i;
                uint64_t x2 = ptx::pack2u(x[2 * c], x[2 * c + 1]);
                if (ROW) x2 = ptx::add2(x2, r_c);
                float d0, d1;
                ptx::unpack2(ptx::mul2(P2[c], x2), d0, d1);
                pa[i] = ptx::pack_bf16(d0, d1);
            }
            ptx::tmem_st8(sb0 + BC + 16 * u, pa);
        }
        ptx::tmem_wait_st();
        k.arrive(C::B_PREADY + 2 * grp + 1, lane);
        if (ROW && item1 != item) {
            r_l = ptx::pack2(n_lse2, n_lse2);
            r_c = ptx::pack2(n_cv, n_cv);
        }
        item = item1;
        j = j1;
    }
}

// ------------------------------------------------------------------------------------------------ epilogue warps
// A thread has one owner row.  Per item: the owner operands of the next item go to tensor memory as soon as the item's last
// score MMAs are done with the present ones (XT), then the accumulators are normalised, converted and stored; they are free
// for the next item once all four warps have read them.
template <int MODE, int DP>
__device__ __forceinline__ void jvp_epilogue(const JvpParams& p, const JvpBlock<MODE, DP>& k, int q, int lane) {
    using C = JvpCfg<MODE, DP>;
    constexpr int NCH = DP / 8;                    // 16-byte chunks of a row
    constexpr int XT0 = C::NPAIR == 2 ? 2 : 0;     // p.own[XT0], p.own[XT0 + 1] -> tensor memory
    const int row = q * 32 + lane;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    // Row of tensor t in an item; what is beyond the head dim or the tensor, and an absent cotangent, reads as zero.
    [[maybe_unused]] auto load_x = [&](int item, int t, uint4 (&v)[NCH]) {
        const int bh = item / p.row_tiles, row0 = (item - bh * p.row_tiles) * JVP_ROWS;
        const __nv_bfloat16* x = p.own[XT0 + t];
        const bool valid = x && row0 + row < p.o.rows;
        const __nv_bfloat16* src = x + (p.o.head_off(bh, p.H) + (size_t)(row0 + row) * (size_t)p.o.rs);
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            v[c] = make_uint4(0, 0, 0, 0);
            if (valid && 8 * c < p.d) v[c] = __ldg(reinterpret_cast<const uint4*>(src + 8 * c));
        }
    };
    [[maybe_unused]] auto store_x = [&](int t, const uint4 (&v)[NCH]) {
#pragma unroll
        for (int c = 0; c < NCH; c += 2) {
            const uint32_t r[8] = {v[c].x, v[c].y, v[c].z, v[c].w, v[c + 1].x, v[c + 1].y, v[c + 1].z, v[c + 1].w};
            ptx::tmem_st8(lanes + (t ? C::COL_X1 : C::COL_X0) + 4 * c, r);
        }
    };
    [[maybe_unused]] uint4 v0[NCH], v1[NCH];
    if (C::XT && !C::XS && (int)blockIdx.x < p.items) {
        load_x(blockIdx.x, 0, v0);
        store_x(0, v0);
        load_x(blockIdx.x, 1, v0);
        store_x(1, v0);
        ptx::tmem_wait_st();
        k.arrive(C::B_XRDY, lane);
    }
    // XS.  Tensor t of the block's item i, from shared memory.
    [[maybe_unused]] const int n_it = jvp_item_count(p);
    [[maybe_unused]] auto stage_x = [&](int t, int i) {
        const bool valid = ((int)blockIdx.x + i * (int)gridDim.x) % p.row_tiles * JVP_ROWS + row < p.o.rows;
        if (!k.wait_item(C::B_OWN + t, i) || (i > 0 && !k.wait_item(C::B_XFREE + t, i - 1))) return false;
        ptx::tc_fence_after_sync();
        const uint32_t tile = k.own_tile(t) + row * 128;
#pragma unroll
        for (int c = 0; c < NCH; c += 2) {
            uint4 v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                // (FOLD: the columns that pad d to DP are ones against the statistics, where those lie there)
                v[e] = C::FOLD && C::TAIL && 8 * (c + e) >= p.d ? make_uint4(JVP_ONES0, JVP_ONES1, 0, 0) : make_uint4(0, 0, 0, 0);
                const uint32_t at = c < 8 ? tile + (((c + e) ^ (row & 7)) << 4) : k.own_tail(t, row, c + e - 8);
                if (valid && 8 * (c + e) < p.d) v[e] = *static_cast<const uint4*>(__cvta_shared_to_generic(at));
            }
            const uint32_t r[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
            ptx::tmem_st8(lanes + (t ? C::COL_X1 : C::COL_X0) + 4 * c, r);
        }
        ptx::tmem_wait_st();
        k.arrive(C::B_XRDY + t, lane);
        if (lane == 0) ptx::mbar_arrive(k.bar(C::B_OWNFREE + t));
        return true;
    };
    // What the issuing warp completes is waited for in the order in which it does: an item's last scores S in its step of that tile,
    // the last X one step later, the last outputs three later.  (Short items: several are opened before one ends.)  Here: the
    // operands whose predecessors are free before step `step`.
    [[maybe_unused]] int staged = 0;   // tensors taken to tensor memory, the first and the second in turn
    [[maybe_unused]] auto stage_until = [&](int step) {
        while (staged < 2 * n_it && (staged >> 1) * p.T - 1 + (staged & 1) < step) {
            if (!stage_x(staged & 1, staged >> 1)) return false;
            ++staged;
        }
        return true;
    };
    if (C::FOLD_TAIL && k.fold_step()) {   // ones against the statistics, for good
        const uint32_t ones[8] = {JVP_ONES0, JVP_ONES1, 0, 0, 0, 0, 0, 0};
        ptx::tmem_st8(lanes + C::COL_X0 + 8 * C::KS, ones);
        ptx::tmem_st8(lanes + C::COL_X1 + 8 * C::KS, ones);
    }
    int it = 0;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x, ++it) {
        if constexpr (C::XS) {
            if (!stage_until((it + 1) * p.T + 2)) return;
        } else if (C::XT && item + (int)gridDim.x < p.items) {
            load_x(item + gridDim.x, 0, v0);                       // in flight during the wait
            load_x(item + gridDim.x, 1, v1);
            if (!k.wait_item(C::B_XFREE, it)) return;
            ptx::tc_fence_after_sync();
            store_x(0, v0);
            store_x(1, v1);
            ptx::tmem_wait_st();
            k.arrive(C::B_XRDY, lane);
        }
        const int bh = item / p.row_tiles, row0 = (item - bh * p.row_tiles) * JVP_ROWS;
        const size_t off = p.o.head_off(bh, p.H) + (size_t)(row0 + row) * (size_t)p.o.rs;
        // lane pairs write the two rows of the pair one after the other, each as complete 32-byte sectors
        const bool ok_even = row0 + (row & ~1) < p.o.rows, ok_odd = row0 + (row | 1) < p.o.rows;
        float f0 = MODE == PASS_DKV_G ? 1.0f : p.out_scale, mun = 0.f;   // (DKV_G: dV is not scaled)
        if constexpr (MODE == PASS_FWD) {   // O = O~/l, tO = R/l - (mu - c) O
            if (!k.wait_item(C::B_ROWSTAT, it)) return;
            const int last = (it * p.T + p.T - 1) & 1;   // the group whose reference is the accumulators'
            const float4 f = k.row_sums(last * JVP_ROWS + row), o = k.row_sums((last ^ 1) * JVP_ROWS + row);
            const float scale = ptx::ex2(o.z - f.z);     // (a group without a tile: m = -inf, factor 0)
            const float l = fmaf(o.x, scale, f.x), mt = f.y + scale * fmaf(o.w - f.w, o.x, o.y);
            f0 = 1.0f / l;
            mun = mt * f0;
            if (row0 + row < p.o.rows) {
                const size_t at = (size_t)bh * p.o.rows + row0 + row;
                p.lse[at] = (f.z + log2f(l)) * 0.6931471805599453f;
                p.mu_out[at] = f.w + mun;
            }
        }
#pragma unroll 1
        for (int pair = 0; pair < C::NACC / 2; ++pair) {
            const uint32_t at = lanes + 2 * pair * C::COL_ACC1;
            __nv_bfloat16* const out0 = pair ? p.out2 : p.out0;
            __nv_bfloat16* const out1 = pair ? p.out3 : p.out1;
            if (C::DKV) f0 = pair ? p.out_scale : 1.0f;
            auto read = [&](int ch, uint32_t (&q0)[8], uint32_t (&q1)[8]) {   // 16 columns of both accumulators, as bf16
                uint32_t x0[16], x1[16];
                if (C::HAS_ACC0) ptx::tmem_ld16(at + 16 * ch + C::COL_ACC0, x0);
                ptx::tmem_ld16(at + 16 * ch + C::COL_ACC1, x1);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 16; c += 2) {
                    const float f1 = MODE == PASS_DKV_G ? p.out_scale : f0;
                    float a0 = 0.f, a1 = 0.f;
                    if (C::HAS_ACC0) { a0 = __uint_as_float(x0[c]) * f0; a1 = __uint_as_float(x0[c + 1]) * f0; }
                    float b0 = __uint_as_float(x1[c]) * f1, b1 = __uint_as_float(x1[c + 1]) * f1;
                    if (MODE == PASS_FWD) { b0 = fmaf(-mun, a0, b0); b1 = fmaf(-mun, a1, b1); }
                    q0[c >> 1] = ptx::pack_bf16(a0, a1);
                    q1[c >> 1] = ptx::pack_bf16(b0, b1);
                }
            };
            auto store = [&](int ch, const uint32_t (&q0)[8], const uint32_t (&q1)[8]) {
                if (16 * ch >= p.d) return;
                const bool has_hi = 16 * ch + 8 < p.d;
                store_row_pairs(out1 + off + 16 * ch, p.o.rs, lane, ok_even, ok_odd, has_hi, make_uint4(q1[0], q1[1], q1[2], q1[3]), make_uint4(q1[4], q1[5], q1[6], q1[7]));
                if (C::HAS_ACC0)
                    store_row_pairs(out0 + off + 16 * ch, p.o.rs, lane, ok_even, ok_odd, has_hi, make_uint4(q0[0], q0[1], q0[2], q0[3]), make_uint4(q0[4], q0[5], q0[6], q0[7]));
            };
            if (!k.wait_item(C::B_FINAL + pair, it)) return;
            ptx::tc_fence_after_sync();
            // The next item's first output MMAs wait for the accumulators: up to d = 80 all of them are read and converted first and
            // stored behind the arrival (reads and stores in turn held them for 3200 cycles at d = 72).  WIDE: there are not the
            // registers, and the items are long.  Forward at d > 48 with one or two tiles an item: the stores are what bounds it, and
            // spread over the reads they get by faster ((64, 16, 256 x 64), both layouts, us: d = 64 62, 63 -> 58, 59, d = 72 78, 84 ->
            // 68, 71; 256 x 128 72, 90 -> 69, 85; equal at d = 32; three tiles, 256 x 192, d = 72: 81 -> 84).
            auto put_out = [&](auto hold) {
                constexpr int HOLD = decltype(hold)::value;
#pragma unroll 1
                for (int ch = 0; ch < C::KS - HOLD; ++ch) {
                    uint32_t q0[8], q1[8];
                    read(ch, q0, q1);
                    store(ch, q0, q1);
                }
                uint32_t q0[HOLD][8], q1[HOLD][8];
#pragma unroll
                for (int i = 0; i < HOLD; ++i) read(C::KS - HOLD + i, q0[i], q1[i]);
                k.arrive(C::B_ACCFREE + pair, lane);
                // (what the next two steps wait for goes in front of the stores)
                if constexpr (C::XS)
                    if (!stage_until((it + 1) * p.T + 2 + min(p.T, JVP_AHEAD))) return false;
#pragma unroll
                for (int i = 0; i < HOLD; ++i) store(C::KS - HOLD + i, q0[i], q1[i]);
                return true;
            };
            constexpr bool SPREAD = MODE == PASS_FWD && DP > 48 && !C::WIDE;
            if (SPREAD && p.T <= 2) put_out(std::integral_constant<int, 1>());
            else if (!put_out(std::integral_constant<int, C::WIDE ? 1 : C::KS>())) return;
        }
    }
}

// ------------------------------------------------------------------------------------------------ the kernel
template <int MODE, int DP>
__global__ void __launch_bounds__(JVP_THREADS, 1)
jvp_kernel(const __grid_constant__ CUtensorMap s0, const __grid_constant__ CUtensorMap s1, const __grid_constant__ CUtensorMap s2,
           const __grid_constant__ CUtensorMap s3, const __grid_constant__ CUtensorMap o0, const __grid_constant__ CUtensorMap o1,
           const __grid_constant__ CUtensorMap o2, const __grid_constant__ CUtensorMap o3, const __grid_constant__ JvpParams p) {
    using C = JvpCfg<MODE, DP>;
    constexpr int BC = C::BC;
    constexpr bool DEPENDENT = MODE == PASS_DK || MODE == PASS_DQ || MODE == PASS_DQ_G;   // launched as a programmatic dependent of the pass before
    // the next backward pass in the stream, if launched as a programmatic dependent, may start as SMs free up
    if (MODE != PASS_FWD) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*reinterpret_cast<volatile int*>(p.status) != 0) {  // an earlier kernel timed out
        if (DEPENDENT && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    extern __shared__ __align__(1024) uint8_t jvp_smem[];
    const JvpBlock<MODE, DP> k{ptx::smem_u32(jvp_smem), p};
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(jvp_smem + k.SLOT);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(jvp_smem + k.ABORT);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        auto init = [&](int b, int n, int count) { for (int i = 0; i < n; ++i) ptx::mbar_init(k.bar(b + i), count); };
        init(C::B_EFULL, C::SE, C::EFULL_COUNT);
        init(C::B_LFULL, C::SL, C::LFULL_COUNT);
        init(C::B_OWN, C::OWN_SETS, C::TAIL ? 33 : 1);
        init(C::B_OWNFREE, C::OWN_SETS, C::XS ? 4 : 1);
        init(C::B_XRDY, C::XSETS, 4);
        init(C::B_XFREE, C::XSETS, 1);
        init(C::B_SFULL, 8 + C::NOUTDONE, 1);   // SFULL, XFULL, OUTDONE
        init(C::B_PREADY, 4, C::DKV ? 8 : 4);   // (of four: the warps of a group)
        init(C::B_SREAD, 1, 8);
        init(C::B_FINAL, C::NACC / 2, 1);
        init(C::B_ACCFREE, C::NACC / 2, 4);
        init(C::B_TURN, 4, 1);
        init(C::B_ROWSTAT, 1, 8);
        init(C::B_DRAIN, 1, 1);
        ptx::fence_mbar_init();
    }
    const uint4 zero = make_uint4(0, 0, 0, 0);
    if (C::TAIL && ((p.d - 64) >> 3) < 2) {
        // The 16-byte chunk behind the copied columns (d = 72) pads the head dim to a multiple of 16: zeroed once, never
        // written again.  Owners and E ring: the second chunk block; L ring: chunk 1 of the second atom, which lies at
        // physical chunk 1 ^ (r & 7) of row r.  FOLD: the stages have the statistics there, the first owner tensor of a pair
        // the ones.
        for (int i = threadIdx.x; i < (C::XS ? 0 : C::NOWN) * JVP_ROWS; i += JVP_THREADS)   // (XS: the epilogue puts them in)
            *reinterpret_cast<uint4*>(jvp_smem + (i / JVP_ROWS) * C::OWN_BYTES + C::OWN_ATOM + (JVP_ROWS + i % JVP_ROWS) * 16) =
                C::FOLD && !(i / JVP_ROWS & 1) ? make_uint4(JVP_ONES0, JVP_ONES1, 0, 0) : zero;
        if (!C::FOLD) {
            uint8_t* e = jvp_smem + C::NOWN * C::OWN_BYTES;
            for (int i = threadIdx.x; i < C::SE * 2 * BC; i += JVP_THREADS)
                *reinterpret_cast<uint4*>(e + (i / (2 * BC)) * 2 * C::EST_BYTES + 2 * C::ATOM + (2 * BC + i % (2 * BC)) * 16) = zero;
            uint8_t* l = e + C::SE * 2 * C::EST_BYTES;
            for (int i = threadIdx.x; i < C::SL * 2 * BC; i += JVP_THREADS) {
                const int t = i / BC, r = i - t * BC;
                *reinterpret_cast<uint4*>(l + (t >> 1) * 2 * C::LST_BYTES + (2 + (t & 1)) * C::ATOM + r * 128 + ((1 ^ (r & 7)) << 4)) = zero;
            }
        }
    }
    if (C::FOLD_TAIL && k.fold_step()) {   // the other half of the statistics' k-step
        uint8_t* l = jvp_smem + k.L;
        for (int i = threadIdx.x; i < C::SL * 2 * BC; i += JVP_THREADS) {
            const int t = i / BC, r = i - t * BC;
            *reinterpret_cast<uint4*>(l + (t >> 1) * 2 * C::LST_BYTES + (2 + (t & 1)) * C::ATOM + r * 128 + ((3 ^ (r & 7)) << 4)) = zero;
        }
    }
    if (C::DKV && p.no_g) {
        // both cotangent tiles of an E stage are read by one MMA: the never-loaded one must read as zero
        constexpr int t = 1;
        uint8_t* e = jvp_smem + C::NOWN * C::OWN_BYTES;
        for (int st = 0; st < C::SE; ++st) {
            uint8_t* stage = e + st * 2 * C::EST_BYTES;
            for (int i = threadIdx.x; i < BC * 8; i += JVP_THREADS) {
                *reinterpret_cast<uint4*>(stage + t * C::ATOM + i * 16) = zero;
                if (C::NA == 2) *reinterpret_cast<uint4*>(stage + (2 + t) * C::ATOM + i * 16) = zero;
            }
        }
    }
    if (C::ONES_BYTES)
        for (int i = threadIdx.x; i < 2 * JVP_ROWS; i += JVP_THREADS)
            *reinterpret_cast<uint4*>(jvp_smem + k.ONES + i * 16) = i < JVP_ROWS ? make_uint4(JVP_ONES0, JVP_ONES1, 0, 0) : zero;
    ptx::fence_proxy_async_smem();
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    // The whole tensor memory starts at 0 and the shared memory of a kernel without static arrays at a 1024-byte boundary:
    // the roles take both for granted.
    const bool placed = *tmem_slot == 0 && (k.base & 1023) == 0;
    if (!placed && threadIdx.x == 0) *abort_flag = 1;

    // warpgroup 0: loads and MMA issue; 1, 2: element-wise; 3: epilogue
    if (warp < 4) {
        ptx::setmaxnreg_dec<C::REGS_LOAD>();
        if (placed) {
            const CUtensorMap* const maps[4] = {&o0, &o1, &o2, &o3};
            if (warp == 1) jvp_issue<MODE, DP>(p, k);
            else if (warp == 2) jvp_load_ring<MODE, DP, 1>(p, k, &s2, &s3, maps, lane);
            else if (warp == 0) {
                if constexpr (C::XS) jvp_stage_owners<MODE, DP>(p, k, maps, lane);
                else jvp_load_ring<MODE, DP, 0>(p, k, &s0, &s1, maps, lane);
            }
            else if constexpr (C::FOLD) jvp_fold<MODE, DP>(p, k, lane);
        }
        if (warp == 1 && *abort_flag && placed) {
            // after a time-out: the queued MMAs must be done before the tensor memory is given back
            ptx::mma_commit_elect(k.bar(C::B_DRAIN));
            ptx::mbar_wait_drain(k.bar(C::B_DRAIN), 0, ptx::DRAIN_LIMIT_NS);
        }
    } else if (warp < 12) {
        ptx::setmaxnreg_inc<C::REGS_ELEM>();
        if (placed) {
            const int grp = (warp - 4) >> 2, q = warp & 3;
            if constexpr (MODE == PASS_FWD) jvp_elem_fwd<DP>(p, k, grp, q, lane);
            else if constexpr (C::GONLY) jvp_elem_g<MODE, DP>(p, k, grp, q, lane);
            else if constexpr (MODE == PASS_DKV) jvp_elem_dkv<DP>(p, k, grp, q, lane);
            else if constexpr (MODE == PASS_DV) jvp_elem_dv<DP>(p, k, grp, q, lane);
            else jvp_elem_two_pairs<MODE, DP>(p, k, grp, q, lane);
        }
    } else {
        ptx::setmaxnreg_dec<C::REGS_EPI>();
        if (placed) jvp_epilogue(p, k, warp & 3, lane);
    }

    // ---------------------------------------------------------------------- teardown
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(*tmem_slot, 512);
    }
    if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, 1);
    // DK and DQ start while the pass before them still runs and read nothing it writes; they must still not complete
    // before it, or completion of the last pass would not imply that the gradients of the earlier ones are written.
    // (No effect on a launch without the attribute.)
    if (DEPENDENT && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace tvm_attn
