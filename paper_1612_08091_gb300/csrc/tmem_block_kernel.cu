// tmem_block_kernel.cu -- a fused 5- or 6-qubit block applied on the tensor
// cores (tcgen05) with the state operand in tensor memory; complex64
// amplitudes, BF16x3 split products.
//
// The paper's simulator gains its speed from lazily buffering gates and
// executing them together (ProjectQ paper, Sec. 4.3.2, Fig. 7 caption).
// Here a run of gates on the K qubits S = {s0 < ... < s(K-1)} (K = 5 or 6)
// has been multiplied into one 2^K x 2^K complex matrix U, and the pass
// computes Psi' = U Psi with Psi viewed as a 2^K x 2^(n-K) matrix (row = the
// bits of S).  A 6-qubit block takes more gates per pass over the state (a
// depth-40 brickwork on 32 qubits needs 69 passes with 6-qubit blocks
// against 106 with 5-qubit ones) for twice the tensor work per amplitude:
// 1536 flop per 16 bytes moved, still well below the bf16 ridge of this part
// (about 286 flop per byte).
//
// Real form.  With interleaved (re, im) amplitudes, the real vector x of a
// column (x[2r] = Re psi_r, x[2r+1] = Im psi_r) maps to y = R x with
// R[2r+a][2r'+b] the 2x2 real block of U[r][r'].  A tile of 128 columns is
// the GEMM D(128 x N) = X(128 x N) R^T(N x N), N = 2^(K+1): M = 128 tile
// columns (the 7 lowest qubits F outside S), N = K_mma = the real form of
// the 2^K rows.  A tile is the 2^(K+7) amplitudes whose bits outside
// V = S u F are fixed.
//
// BF16x3.  X = X1 + X2 and R = R1 + R2 (+ R3) are split into bfloat16 parts;
// the products X1 R1 + X2 R1 + X1 R2 (or five with X2 R2 + X1 R3) accumulate
// in FP32 in tensor memory.  The state split loses about 2^-17 relatively
// per element and pass; the gate split is computed in FP64 (k_build_operand).
//
// Where the operands live.  R's bf16 parts are operand B in shared memory:
// K-major, 128-byte swizzle, in 64-element K halves of N x 128 bytes.  The
// state tile X is operand A and lives in tensor memory: thread t owns tile
// column t, which is TMEM lane t; it loads that column's 2^K amplitudes,
// splits each into bf16 hi and lo words (re in the low half: K elements 2r,
// 2r+1) and writes them with tcgen05.st to TMEM columns [0, 2^K) (hi) and
// [2^K, 2^(K+1)) (lo); the accumulator takes the next N columns.  So the
// state is never staged in shared memory and needs no swizzle arithmetic.
// Per CTA: 2^(K+2) TMEM columns (128 or 256) and 17 or 66 KB of shared
// memory; three (K = 5) or two (K = 6) CTAs per SM.
//
// Per CTA, over its tiles t of a persistent grid:
//   wait for MMA(t-1) -> read D(t-1) from TMEM, scale, store it -> split tile
//   t into TMEM -> thread 0 issues N/16 tcgen05.mma M128 N K16 per product
//   and commits them to an mbarrier -> issue the loads of tile t+1 (2^K
//   amplitudes per thread held in registers: 96 or 128 KB in flight per SM).
// The other CTAs on the SM fill this CTA's waits.  Every wait is bounded; on
// time-out the kernel raises an error flag in the workspace, frees its
// tensor memory and returns.
//
// Norm control.  The bf16 split and the FP32 accumulation shrink the norm by
// a few 1e-7 per pass, and the shrink is systematic on structured states
// (Grover's search repeats the same blocks on a state whose amplitudes are
// mostly equal), so uncorrected it adds up over 1e5 passes.  Each pass is a
// step of the norm chain of norm_chain.cuh: from the previous pass's input
// and output sums it scales its outputs so that the norm returns to the
// chain's target.  Errors therefore do not accumulate: what remains is one
// pass's change of shrink ratio and the drift of the passes outside the
// chain since the previous one, both corrected by the pass after.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "internal.h"
#include "norm_chain.cuh"
#include "tc_common.cuh"

using namespace qsim_dev;
using namespace qsim_tc;

namespace {

constexpr int kTmThreads = 128;
constexpr int kTmExtra = 128;  // barriers, TMEM slot, scale, reduction

template <int K>
struct TmShape {
    static constexpr int kRows = 1 << K;          // block rows
    static constexpr int kTileBits = K + 7;       // + 7 column bits
    static constexpr int kN = 2 * kRows;          // real outputs = real inputs
    static constexpr int kBHalf = kN * 128;       // one 64-element K half of one part: N rows x 128 B
    static constexpr int kBPart = (kN / 64) * kBHalf;
    static constexpr uint32_t kColAHi = 0, kColALo = kRows, kColD = 2 * kRows;
    static constexpr uint32_t kCols = 4 * kRows;  // tensor-memory columns per CTA
    static constexpr uint32_t kIdesc = idesc_bf16(128, kN);
    static constexpr int kCtasPerSm = 512 / kCols < 3 ? 512 / kCols : 3;
};

struct TmArgs {
    float2 *psi;
    const unsigned char *rec;  // nsplit x kBPart: pre-split, pre-swizzled R (16-B aligned)
    uint32_t rec_bytes;
    int nsplit;                // bf16 parts of R: 2 (BF16x3) or 3 (five products)
    uint64_t ntiles;           // 2^(n - K - 7)
    InsertSpec vspec;          // the K + 7 positions of V = S u F, ascending
    unsigned int *err;         // error flag
    qsim_chain::ChainArgs chain;  // norm control (norm_chain.cuh)
    int fpos[7];               // tile column bit j <-> qubit fpos[j]
    uint64_t rdep[64];         // address bits of block row r
    uint64_t qoff[4];          // W = 16: address bits of column 4q + i relative to column 4q
};

// 32-byte global accesses (one whole sector per thread): four adjacent
// amplitudes as two float4 (the address is 32-byte aligned)
__device__ __forceinline__ void ld_v8(const float2 *p, float4 &a, float4 &b) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                 : "l"(p));
}
__device__ __forceinline__ void st_v8(float2 *p, const float4 &a, const float4 &b) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// D(tmem) (+)= A(tmem) * B(smem)^T, M = 128, K = 16
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// W: amplitudes per global access.  W = 2: qubit 0 is in S, so rows r and
// r+1 (r even) are adjacent amplitudes and move as one 16-byte access.  W = 4:
// qubits 0 and 1 are in S, rows 4j..4j+3 are adjacent and move as one
// 32-byte access; the tile columns are then at least 4 amplitudes apart, and
// narrower accesses would use half a sector per instruction.  W = 1: 8-byte
// accesses, the columns being adjacent amplitudes.  W = 16: qubits 0..3 are
// in S, so each 16-row line of a column is 128 contiguous bytes, but the
// lanes' columns lie 512 (K = 6) or 256 (K = 5) bytes apart and a warp
// access with one column per lane touches 32 lines.  Instead the four lanes
// of a quad read one column's line together (32 bytes each: 8 lines per
// warp access) and move it to and from tensor memory with the 16x256b
// shape, in which a quad shares a TMEM lane and each of its threads holds
// two adjacent 32-bit columns per 8.  Thread k of a quad holds rows 4k..4k+3
// of each 16-row line; the host orders the gate operand's K (input rows)
// and N (output rows) to match: A column 16G + 8h + 2k + e holds row
// 16G + 4k + 2h + e, and D columns 2j, 2j + 1 with j = 16G + 4h + k hold
// output row 16G + 4k + h.  Tile column 32w + q + 8i (warp w, quad q) is
// TMEM lane 32w + q + 8i as in the other widths.
template <int K, int W>
__global__ void __launch_bounds__(kTmThreads, TmShape<K>::kCtasPerSm) k_block_tmem(const TmArgs args) {
    using Sh = TmShape<K>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *B = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = (uint64_t *)(B + args.nsplit * Sh::kBPart);  // [0] operand copy, [1] MMA done
    uint32_t *tmem_slot = (uint32_t *)(bars + 2);
    float *s_scale = (float *)(tmem_slot + 1);
    double *s_red = (double *)(bars + 4);  // [4 warps][2]

    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        bulk_load(B, args.rec, args.rec_bytes, &bars[0]);
    }
    if (warp == 1) {
        // output scale from the previous pass's sums, and record
        const float sc = qsim_chain::chain_scale(args.chain);
        if ((tid & 31) == 0) *s_scale = sc;
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(Sh::kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);  // this warp's 32 TMEM lanes

    // (this wait after the tile addresses below, with the first tile's loads
    // before it or after, took the tile loop five more registers and a 32-qubit
    // pass 2 % longer: 6.49 instead of 6.62 TB/s)
    bool failed = !mbar_wait(&bars[0], 0);
    if (failed) atomicOr(args.err, 1u);
    const bool abort0 = __syncthreads_or(failed) != 0;

    double nrm_in = 0.0, nrm_out = 0.0;
    const float scale = *s_scale;
    if (!abort0) {
        uint64_t coff = 0;  // address bits of this thread's tile column
#pragma unroll
        for (int j = 0; j < 7; ++j)
            if ((tid >> j) & 1) coff |= 1ull << args.fpos[j];
        // W = 16: this lane's place k4 in its quad q4; the address bits of
        // the quad's first column 32 warp + q4 (the others: + qoff[i])
        const unsigned lane = (unsigned)tid & 31u, k4 = lane & 3u, q4 = lane >> 2;
        uint64_t coffq = 0;
#pragma unroll
        for (int j = 0; j < 7; ++j)
            if ((((tid & ~31) | (int)q4) >> j) & 1) coffq |= 1ull << args.fpos[j];
        const int nterms = args.nsplit == 3 ? 5 : 3;

        float4 v[Sh::kRows / 2];  // rows 2j, 2j+1 of this column: (re, im, re, im)
        auto load_tile = [&](uint64_t tt) {
            const float2 *p = args.psi + insert_zeros(tt, args.vspec) + coff;
            if constexpr (W == 16) {
                // quad layout: v[8m + 2i + h] = half h of rows 16m + 4k4 ..
                // 16m + 4k4 + 3 of tile column 32 warp + q4 + 8i
                const float2 *pq = args.psi + insert_zeros(tt, args.vspec) + coffq + 4 * k4;
#pragma unroll
                for (int m = 0; m < Sh::kRows / 16; ++m)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        ld_v8(pq + args.qoff[i] + args.rdep[16 * m], v[8 * m + 2 * i], v[8 * m + 2 * i + 1]);
            } else if constexpr (W == 4) {
#pragma unroll
                for (int j = 0; j < Sh::kRows / 4; ++j) ld_v8(p + args.rdep[4 * j], v[2 * j], v[2 * j + 1]);
            } else {
#pragma unroll
                for (int j = 0; j < Sh::kRows / 2; ++j) {
                    if constexpr (W == 2) {
                        v[j] = *(const float4 *)(p + args.rdep[2 * j]);
                    } else {
                        const float2 a = p[args.rdep[2 * j]], b = p[args.rdep[2 * j + 1]];
                        v[j] = make_float4(a.x, a.y, b.x, b.y);
                    }
                }
            }
        };
        auto epilogue = [&](uint64_t tt) {
            float2 *const pb = args.psi + insert_zeros(tt, args.vspec);
            float2 *p = pb + coff;
            // four FP32 partial sums (chains of 2^K / 2 terms): the rounding
            // of a long chain is systematic when many amplitudes are equal;
            // FP64 across tiles (an FP64 add per 16 rows measured 1.2 %
            // slower)
            float ssq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int chunk = 0; chunk < Sh::kN / 32; ++chunk) {
                if constexpr (W == 16) {
                    // output rows 16 chunk + 4k4 .. + 3 of tile columns
                    // 32 warp + q4 + 8i: 32-byte stores, four lanes per line
                    float2 *pq = pb + coffq + 4 * k4 + args.rdep[16 * chunk];
#pragma unroll
                    for (int b2 = 0; b2 < 2; ++b2) {
                        float d[16];  // d[4 rho + 2c + a]: row 16 chunk + 4k4 + rho of column i = 2 b2 + c
                        tmem_ld16x256b_x4(lanes + ((uint32_t)(16 * b2) << 16) + Sh::kColD + chunk * 32, d);
#pragma unroll
                        for (int q = 0; q < 16; ++q) ssq[q & 3] = fmaf(d[q], d[q], ssq[q & 3]);
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            st_v8(pq + args.qoff[2 * b2 + c],
                                  make_float4(d[2 * c] * scale, d[2 * c + 1] * scale, d[4 + 2 * c] * scale,
                                              d[5 + 2 * c] * scale),
                                  make_float4(d[8 + 2 * c] * scale, d[9 + 2 * c] * scale, d[12 + 2 * c] * scale,
                                              d[13 + 2 * c] * scale));
                    }
                } else {
                float d[32];  // rows 16 chunk .. 16 chunk + 15, (re, im) interleaved
                tmem_ld32(lanes + Sh::kColD + chunk * 32, d);
#pragma unroll
                for (int q = 0; q < 32; ++q) ssq[q & 3] = fmaf(d[q], d[q], ssq[q & 3]);
#pragma unroll
                for (int q = 0; q < 16; q += 2) {
                    const int r = chunk * 16 + q;
                    const float4 o = make_float4(d[2 * q] * scale, d[2 * q + 1] * scale, d[2 * q + 2] * scale,
                                                 d[2 * q + 3] * scale);
                    if constexpr (W == 4) {
                        if (q % 4 == 0) {
                            const float4 o2 = make_float4(d[2 * q + 4] * scale, d[2 * q + 5] * scale,
                                                          d[2 * q + 6] * scale, d[2 * q + 7] * scale);
                            st_v8(p + args.rdep[r], o, o2);
                        }
                    } else if constexpr (W == 2) {
                        *(float4 *)(p + args.rdep[r]) = o;
                    } else {
                        p[args.rdep[r]] = make_float2(o.x, o.y);
                        p[args.rdep[r + 1]] = make_float2(o.z, o.w);
                    }
                }
                }
            }
            nrm_out += (double)((ssq[0] + ssq[1]) + (ssq[2] + ssq[3]));
        };

        uint64_t t = blockIdx.x;
        int it = 0;
        bool stop = false;
        if (t < args.ntiles) load_tile(t);
        for (; t < args.ntiles; t += gridDim.x, ++it) {
            if (it >= 1) {
                // MMA(it-1) done: the A columns are free and D holds the
                // previous tile
                if (mbar_wait(&bars[1], (uint32_t)((it - 1) & 1))) {
                    tc_fence_after();
                    epilogue(t - gridDim.x);
                } else {
                    failed = true;
                    atomicOr(args.err, 2u);
                }
            }
            float xsq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int chunk = 0; chunk < Sh::kRows / 16; ++chunk) {
                if constexpr (W == 16) {
                    // lanes 32 warp + 16 b2 + q4 + 8c (tile column i = 2 b2 + c),
                    // A columns 16 chunk + 8h + 2k4 + e = rows 16 chunk + 4k4 + 2h + e
#pragma unroll
                    for (int b2 = 0; b2 < 2; ++b2) {
                        uint32_t hw[8], lw[8];
#pragma unroll
                        for (int c = 0; c < 2; ++c)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const float4 x = v[8 * chunk + 2 * (2 * b2 + c) + h];
                                xsq[0] = fmaf(x.x, x.x, xsq[0]);
                                xsq[1] = fmaf(x.y, x.y, xsq[1]);
                                xsq[2] = fmaf(x.z, x.z, xsq[2]);
                                xsq[3] = fmaf(x.w, x.w, xsq[3]);
                                split_pair(x.x, x.y, hw[4 * h + 2 * c], lw[4 * h + 2 * c]);
                                split_pair(x.z, x.w, hw[4 * h + 2 * c + 1], lw[4 * h + 2 * c + 1]);
                            }
                        const uint32_t l16 = lanes + ((uint32_t)(16 * b2) << 16) + chunk * 16;
                        tmem_st16x256b_x2(l16 + Sh::kColAHi, hw);
                        tmem_st16x256b_x2(l16 + Sh::kColALo, lw);
                    }
                } else {
                    // this lane's own column: A columns 16 chunk + j = rows
                    uint32_t hw[16], lw[16];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 x = v[chunk * 8 + j];
                        xsq[0] = fmaf(x.x, x.x, xsq[0]);
                        xsq[1] = fmaf(x.y, x.y, xsq[1]);
                        xsq[2] = fmaf(x.z, x.z, xsq[2]);
                        xsq[3] = fmaf(x.w, x.w, xsq[3]);
                        split_pair(x.x, x.y, hw[2 * j], lw[2 * j]);
                        split_pair(x.z, x.w, hw[2 * j + 1], lw[2 * j + 1]);
                    }
                    tmem_st16(lanes + Sh::kColAHi + chunk * 16, hw);
                    tmem_st16(lanes + Sh::kColALo + chunk * 16, lw);
                }
            }
            nrm_in += (double)((xsq[0] + xsq[1]) + (xsq[2] + xsq[3]));
            tcgen05_wait_st();
            tc_fence_before();
            if (__syncthreads_or(failed)) {
                stop = true;
                break;
            }
            if (tid == 0) {
                tc_fence_after();
                const uint32_t b0 = smem_u32(B);
                uint32_t acc = 0;
                for (int term = 0; term < nterms; ++term) {
                    // (A part, B part): X1R1, X2R1, X1R2, X2R2, X1R3.  (Issuing
                    // the small products first measured a 3x larger coherent
                    // error on Grover's search, the same on random circuits.)
                    const uint32_t a = tmem + ((term == 1 || term == 3) ? Sh::kColALo : Sh::kColAHi);
                    const uint32_t b = b0 + (uint32_t)(term < 2 ? 0 : (term < 4 ? 1 : 2)) * Sh::kBPart;
#pragma unroll
                    for (int kk = 0; kk < Sh::kN / 16; ++kk) {
                        mma_ts(tmem + Sh::kColD, a + kk * 8, sw128_desc(b + (kk >> 2) * Sh::kBHalf + (kk & 3) * 32),
                               Sh::kIdesc, acc);
                        acc = 1;
                    }
                }
                mma_commit(&bars[1]);
            }
            const uint64_t tn = t + gridDim.x;
            if (tn < args.ntiles) load_tile(tn);
        }
        if (it >= 1 && !stop) {
            if (mbar_wait(&bars[1], (uint32_t)((it - 1) & 1))) {
                tc_fence_after();
                epilogue(t - gridDim.x);
            } else {
                atomicOr(args.err, 2u);
            }
        }
    }
    // per-CTA norm sums, fixed reduction order
    nrm_in = warp_sum(nrm_in);
    nrm_out = warp_sum(nrm_out);
    if ((tid & 31) == 0) {
        s_red[2 * warp] = nrm_in;
        s_red[2 * warp + 1] = nrm_out;
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0)
        qsim_chain::chain_sums(args.chain, s_red[0] + s_red[2] + s_red[4] + s_red[6],
                               s_red[1] + s_red[3] + s_red[5] + s_red[7]);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Sh::kCols) : "memory");
    }
}

// The B operand image: the nsplit bf16 parts of R = real form of U (D = 2^K
// rows), each N rows (output index 2j+a) x N K elements (input index 2j'+b)
// in K halves of 64 elements; within a half, row `row` is 128 bytes at
// row * 128 with its 16-byte chunks XOR-swizzled by row & 7.  Output j is
// block row orow(j) and input j' block row irow(j'): the identity, or for
// the quad fragments of W = 16 (see k_block_tmem) orow(16G + 4h + k) =
// 16G + 4k + h and irow(16G + 8h + 2k + e) = 16G + 4k + 2h + e.  Here the
// inverse of both: block row r is output quad_out(r) and input quad_in(r).
__device__ __forceinline__ int quad_out(int r) { return (r & ~15) | ((r & 3) << 2) | ((r >> 2) & 3); }
__device__ __forceinline__ int quad_in(int r) {
    return (r & ~15) | (((r >> 1) & 1) << 3) | (((r >> 2) & 3) << 1) | (r & 1);
}

// Building the images on the device.  U is the ordered product of the
// block's gates; column c of U is the gates applied to the basis vector
// e_c, so the columns are independent and a warp (a CTA of its own) takes
// one: 2^K amplitudes in shared memory in FP64, two or one per lane, each
// lane forming its outputs' 2^t-term sums.  Then it splits its column into
// bf16 parts and writes them at their swizzled places.  One launch builds
// the images of many blocks (blockIdx.y).  On the host the same took 200 us
// per 6-qubit block (the product of some 28 gates and 16,384 elements
// split), longer than a pass over a register of 26 qubits or fewer.  Here a
// launch is bound by the FP64 units' latency and rate (8 FMAs per output,
// gate and column, two a cycle on an SM): 29 us for one block of 36 gates,
// 35 us for eight blocks (20-qubit circuit of 21 blocks: 7.66 -> 0.62 ms with
// the gates queued in one call).
struct BlockGate {      // one gate of a block, in block-local bits
    uint32_t cmask;     // controls
    uint32_t tmask;     // targets
    uint16_t type;      // 0 dense, 1 diagonal, 2 X
    uint16_t t;         // targets
    uint8_t tpos[8];    // target j <-> block bit tpos[j]
    uint32_t off;       // its matrix (dense: 4^t, diagonal: 2^t entries), bytes from the record's start
    uint32_t pad[2];
};
static_assert(sizeof(cd) == 16 && sizeof(BlockGate) == 32, "records are made of 16-byte units");
struct BlockJob {       // one block
    unsigned char *out; // operand image
    const unsigned char *rec;
    uint32_t rec_bytes;
    uint16_t K, quad;
    uint16_t nsplit, init;  // init: the record is U itself (row-major), no gates
    uint32_t ngates;
};
constexpr int kJobStage = 6144;  // bytes of a record kept in shared memory

__global__ void __launch_bounds__(32) k_build_operand(const BlockJob *__restrict__ jobs) {
    __shared__ double2 x[64];
    __shared__ __align__(16) unsigned char stage[kJobStage];
    const BlockJob J = jobs[blockIdx.y];
    const int D = 1 << J.K, c = blockIdx.x, lane = threadIdx.x;
    if (c >= D) return;
    const unsigned char *rec = J.rec;
    if (J.rec_bytes <= (uint32_t)kJobStage && !J.init) {
        const int units = (int)J.rec_bytes / 16;
#pragma unroll 4
        for (int i = lane; i < units; i += 32) ((float4 *)stage)[i] = ((const float4 *)J.rec)[i];
        rec = stage;
    }
    const int per = D >> 5;  // outputs per lane: 2 or 1
    for (int u = 0; u < per; ++u) {
        const int i = lane + 32 * u;
        x[i] = J.init ? ((const double2 *)J.rec)[i * D + c] : make_double2(i == c ? 1.0 : 0.0, 0.0);
    }
    __syncwarp();
    for (uint32_t g = 0; g < J.ngates; ++g) {
        const BlockGate G = ((const BlockGate *)rec)[g];
        const double2 *m = (const double2 *)(rec + G.off);
        if (G.t == 1) {
            // a pair per lane, in place
            const int b = G.tpos[0], i0 = ((lane >> b) << (b + 1)) | (lane & ((1 << b) - 1)), i1 = i0 | (1 << b);
            if (lane < D / 2 && ((uint32_t)i0 & G.cmask) == G.cmask) {
                const double2 v0 = x[i0], v1 = x[i1];
                double2 y0 = v1, y1 = v0;
                if (G.type == 0) {
                    const double2 a = m[0], e = m[1], f = m[2], h = m[3];
                    y0.x = fma(a.x, v0.x, -a.y * v0.y) + fma(e.x, v1.x, -e.y * v1.y);
                    y0.y = fma(a.x, v0.y, a.y * v0.x) + fma(e.x, v1.y, e.y * v1.x);
                    y1.x = fma(f.x, v0.x, -f.y * v0.y) + fma(h.x, v1.x, -h.y * v1.y);
                    y1.y = fma(f.x, v0.y, f.y * v0.x) + fma(h.x, v1.y, h.y * v1.x);
                } else if (G.type == 1) {
                    const double2 a = m[0], h = m[1];
                    y0 = make_double2(fma(a.x, v0.x, -a.y * v0.y), fma(a.x, v0.y, a.y * v0.x));
                    y1 = make_double2(fma(h.x, v1.x, -h.y * v1.y), fma(h.x, v1.y, h.y * v1.x));
                }
                x[i0] = y0;
                x[i1] = y1;
            }
            __syncwarp();
            continue;
        }
        double2 y[2];
        for (int u = 0; u < per; ++u) {
            const int i = lane + 32 * u;
            y[u] = x[i];
            if (((uint32_t)i & G.cmask) != G.cmask) continue;
            int r = 0;
            for (int j = 0; j < G.t; ++j) r |= ((i >> G.tpos[j]) & 1) << j;
            if (G.type == 1) {
                const double2 z = m[r], v = y[u];
                y[u] = make_double2(fma(z.x, v.x, -z.y * v.y), fma(z.x, v.y, z.y * v.x));
                continue;
            }
            const int base = i & ~(int)G.tmask, T = 1 << G.t;
            y[u] = make_double2(0.0, 0.0);
            for (int k = 0; k < T; ++k) {
                int s = base;
                for (int j = 0; j < G.t; ++j) s |= ((k >> j) & 1) << G.tpos[j];
                const double2 w = m[r * T + k], v = x[s];
                y[u].x += fma(w.x, v.x, -w.y * v.y);
                y[u].y += fma(w.x, v.y, w.y * v.x);
            }
        }
        __syncwarp();
        for (int u = 0; u < per; ++u) x[lane + 32 * u] = y[u];
        __syncwarp();
    }
    // column c of U is input j' = 2^-1 k: elements k = 2j', 2j'+1 of rows 2j, 2j+1
    const int N = 2 * D, half = N * 128, part = (N / 64) * half;
    const int k = 2 * (J.quad ? quad_in(c) : c), kb = (k & 63) * 2;
    for (int u = 0; u < per; ++u) {
        const int i = lane + 32 * u;
        const double2 z = x[i];
        const int j = J.quad ? quad_out(i) : i;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int row = 2 * j + a;
            double r0 = a ? z.y : z.x, r1 = a ? z.x : -z.y;
            unsigned char *dst =
                J.out + (size_t)(k >> 6) * half + (size_t)row * 128 + ((((kb >> 4) ^ (row & 7)) << 4)) + (kb & 15);
            for (int sp = 0; sp < J.nsplit; ++sp) {
                const uint32_t h0 = f32_to_bf16_bits((float)r0), h1 = f32_to_bf16_bits((float)r1);
                r0 -= (double)__uint_as_float(h0 << 16);
                r1 -= (double)__uint_as_float(h1 << 16);
                *(uint32_t *)(dst + (size_t)sp * part) = h0 | (h1 << 16);
            }
        }
    }
}

// amplitudes per global access (see k_block_tmem)
int access_width(const int *q) {
    const bool low4 = q[0] == 0 && q[1] == 1 && q[2] == 2 && q[3] == 3;
    return low4 ? 16 : (q[0] == 0 && q[1] == 1) ? 4 : (q[0] == 0 ? 2 : 1);
}

template <int K>
int launch_tmem(qsim *s, const int *qubits, const unsigned char *dev_rec) {
    using Sh = TmShape<K>;
    const int n = s->n;
    const int nsplit = s->tc_terms == 5 ? 3 : 2;
    TmArgs a{};
    uint64_t Smask = 0;
    for (int j = 0; j < K; ++j) Smask |= 1ull << qubits[j];
    uint64_t Vmask = Smask;
    for (int b = 0, nf = 0; b < n && nf < 7; ++b)
        if (!((Smask >> b) & 1ull)) {
            a.fpos[nf++] = b;
            Vmask |= 1ull << b;
        }
    a.vspec.m = Sh::kTileBits;
    for (int b = 0, k = 0; b < n; ++b)
        if ((Vmask >> b) & 1ull) a.vspec.pos[k++] = b;
    for (int r = 0; r < Sh::kRows; ++r) {
        uint64_t d = 0;
        for (int j = 0; j < K; ++j)
            if ((r >> j) & 1) d |= 1ull << qubits[j];
        a.rdep[r] = d;
    }
    // W = 16: tile columns 32w + q + 8i lie qoff[i] from 32w + q
    for (int i = 0; i < 4; ++i)
        a.qoff[i] = ((i & 1) ? 1ull << a.fpos[3] : 0ull) + ((i & 2) ? 1ull << a.fpos[4] : 0ull);
    const int W = access_width(qubits);
    const int wi = W == 16 ? 3 : W == 4 ? 2 : W - 1;

    auto kernel = W == 16 ? k_block_tmem<K, 16>
                          : W == 4 ? k_block_tmem<K, 4> : (W == 2 ? k_block_tmem<K, 2> : k_block_tmem<K, 1>);
    const int dev = s->device;
    if (dev < 0 || dev >= 64) return QSIM_ENOTSUP;
    static int smem_for[4][64][4] = {{{0}}};  // [access width][device][nsplit]: dynamic shared memory to request
    static int smem_attr[4][64] = {{0}};      // [access width][device]: the kernel's shared-memory limit set so far
    int &smem = smem_for[wi][dev][nsplit];
    if (!smem) {
        // At most kCtasPerSm CTAs per SM, as many as the tensor memory holds
        // (512 columns).  If registers and shared memory would let another
        // CTA in, request more shared memory so that it stays out: its
        // allocation would wait for one of the others to finish and
        // unbalance the persistent grid.
        cudaFuncAttributes fa;
        int regs_sm = 65536, smem_sm = 233472;
        cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        if (e != cudaSuccess) return cuda_err(s, e, "tmem block kernel attributes");
        int bytes = 1024 + nsplit * Sh::kBPart + kTmExtra;
        const int cap = Sh::kCtasPerSm;
        const int by_regs = regs_sm / (fa.numRegs * kTmThreads);
        if (by_regs > cap && smem_sm / (bytes + 1024) > cap) bytes = smem_sm / (cap + 1) - 1024 + 64;
        // the limit is per kernel, shared by both operand sizes: only raise it
        if (bytes > smem_attr[wi][dev]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            if (e != cudaSuccess) return cuda_err(s, e, "tmem block kernel attribute");
            smem_attr[wi][dev] = bytes;
        }
        if (getenv("QSIM_DEBUG"))
            fprintf(stderr, "qsim: k_block_tmem<%d,%d> regs %d smem %d (registers allow %d CTAs/SM, cap %d)\n", K, W,
                    fa.numRegs, bytes, by_regs, cap);
        smem = bytes;
    }
    a.psi = (float2 *)s->state;
    a.rec = dev_rec;
    a.rec_bytes = (uint32_t)(nsplit * Sh::kBPart);
    a.nsplit = nsplit;
    a.ntiles = 1ull << (n - Sh::kTileBits);
    a.err = (unsigned int *)((char *)s->ws + kWsErr);
    uint64_t cap = (uint64_t)s->sms * Sh::kCtasPerSm;
    if (cap > (uint64_t)kMaxTcGrid) cap = kMaxTcGrid;
    const uint64_t grid = a.ntiles < cap ? a.ntiles : cap;
    a.chain = qsim_chain::chain_next(s);
    kernel<<<(unsigned)grid, kTmThreads, smem, s->stream>>>(a);
    s->stats.launches++;
    qsim_chain::chain_advance(s, (int)grid);
    return cuda_err(s, cudaGetLastError(), "tmem block launch");
}

// A block's record: its gates in block-local bits and their matrices, or,
// where that would be longer than U itself, U (block_matrix).
void block_record(const std::vector<GateRec> &q, const PlanItem &it, const int *S, int K, std::vector<unsigned char> &rec,
                  BlockJob &job) {
    const size_t start = rec.size(), D = (size_t)1 << K;
    size_t bytes = sizeof(BlockGate) * it.members.size();
    for (int gi : it.members) {
        const GateRec &g = q[gi];
        const size_t T = (size_t)1 << g.t;
        bytes += g.kind == GK_X ? 0 : sizeof(cd) * (g.diag ? T : T * T);
    }
    if (bytes > sizeof(cd) * D * D) {
        PlanItem whole = it;
        whole.k = K;
        for (int j = 0; j < K; ++j) whole.qubits[j] = S[j];
        block_matrix(q, whole);
        rec.resize(start + sizeof(cd) * D * D);
        std::memcpy(&rec[start], whole.m.data(), sizeof(cd) * D * D);
        job.init = 1;
        job.ngates = 0;
        job.rec_bytes = (uint32_t)(sizeof(cd) * D * D);
        return;
    }
    rec.resize(start + bytes);
    BlockGate *gates = (BlockGate *)&rec[start];
    size_t off = sizeof(BlockGate) * it.members.size();
    for (size_t i = 0; i < it.members.size(); ++i) {
        const GateRec &g = q[it.members[i]];
        BlockGate &b = gates[i];
        b = BlockGate{};
        auto bit = [&](int qubit) {
            int j = 0;
            while (S[j] != qubit) ++j;
            return j;
        };
        for (int c : g.controls) b.cmask |= 1u << bit(c);
        for (int j = 0; j < g.t; ++j) {
            b.tpos[j] = (uint8_t)bit(g.targets[j]);
            b.tmask |= 1u << b.tpos[j];
        }
        b.t = (uint16_t)g.t;
        b.type = g.kind == GK_X ? 2 : g.diag ? 1 : 0;
        b.off = (uint32_t)off;
        const int T = 1 << g.t;
        cd *m = (cd *)&rec[start + off];
        if (b.type == 0) {
            std::memcpy((void *)m, g.m.data(), sizeof(cd) * T * T);
            off += sizeof(cd) * T * T;
        } else if (b.type == 1) {
            for (int r = 0; r < T; ++r) m[r] = g.m[(size_t)r * T + r];
            off += sizeof(cd) * T;
        }
    }
    job.init = 0;
    job.ngates = (uint32_t)it.members.size();
    job.rec_bytes = (uint32_t)bytes;
}

}  // namespace

int tmem_block_qubits(const qsim *s, const PlanItem &it, int *q) {
    if (!it.fused || it.diag_block || it.prod_block || it.perm_block || s->prec != QSIM_C64 || !s->tc_enabled) return 0;
    if (it.k < 4 || it.k > 6 || s->n < (it.k == 6 ? 13 : 12)) return 0;
    uint64_t S = 0;
    for (int j = 0; j < it.k; ++j) S |= 1ull << it.qubits[j];
    // a 4-qubit block runs as the 5-qubit block on its qubits and the lowest
    // other one
    for (int b = 0; b < s->n && __builtin_popcountll(S) < 5; ++b) S |= 1ull << b;
    int K = 0;
    for (int b = 0; b < s->n; ++b)
        if ((S >> b) & 1ull) q[K++] = b;
    return K;
}

int build_operands(qsim *s, PlanItem *const *items, int count) {
    if (count < 1) return QSIM_OK;
    const uint32_t nsplit = s->tc_terms == 5 ? 3 : 2;
    // the jobs, then the records; offsets turn into addresses once the place
    // in the device ring is known
    std::vector<unsigned char> rec(sizeof(BlockJob) * count);
    std::vector<size_t> at(count), image(count);
    size_t images = 0;
    int kmax = 5;
    for (int i = 0; i < count; ++i) {
        int q[6];
        const int K = tmem_block_qubits(s, *items[i], q);
        BlockJob job{};
        job.K = (uint16_t)K;
        job.nsplit = (uint16_t)nsplit;
        job.quad = access_width(q) == 16;
        at[i] = rec.size();
        block_record(s->queue, *items[i], q, K, rec, job);
        std::memcpy(&rec[sizeof(BlockJob) * i], &job, sizeof(job));
        image[i] = images;
        images += (size_t)nsplit * (K == 6 ? TmShape<6>::kBPart : TmShape<5>::kBPart);
        if (K > kmax) kmax = K;
    }
    unsigned char *out = nullptr, *dev = nullptr;
    int rc = ring_reserve(s, images + rec.size() + 512, &out);  // both in one piece of the ring
    if (rc) return rc;
    dev = out + ((images + 255) & ~(size_t)255);
    for (int i = 0; i < count; ++i) {
        BlockJob *job = (BlockJob *)&rec[sizeof(BlockJob) * i];
        job->out = out + image[i];
        job->rec = dev + at[i];
        items[i]->operand = job->out;
    }
    if ((rc = stage_to(s, dev, rec.data(), rec.size()))) return rc;
    k_build_operand<<<dim3(1u << kmax, (unsigned)count), 32, 0, s->stream>>>((const BlockJob *)dev);
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "block operand launch");
}

int launch_block_tmem(qsim *s, const PlanItem &it) {
    int q[6];
    const int K = tmem_block_qubits(s, it, q);
    if (K == 0 || !it.operand) return QSIM_ENOTSUP;
    return K == 6 ? launch_tmem<6>(s, q, it.operand) : launch_tmem<5>(s, q, it.operand);
}
