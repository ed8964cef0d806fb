// product_kernel.cu -- a layer of Hadamard-like one-qubit gates on many
// qubits, applied twelve qubits per pass over a complex64 state.
//
// The simulator executes buffered gates together (ProjectQ paper, Sec.
// 4.3.2).  Between gates too wide for any block (Grover's many-controlled Z,
// Appendix A) a layer of one-qubit gates on m qubits has nothing to fuse
// with; as dense 6-qubit blocks it costs ceil(m / 6) passes.  Grover's
// layers are products of H and X on each wire, c [[s00, s01], [s10, s11]]
// with c = 2^(-1/2), signs s = +-1 and orthogonal rows (s00 s11 = -s01
// s10), which the planner recognises ("butterfly" matrices).  For such a
// gate
//     x0' = c s00 (x0 + p x1),   x1' = c s10 (x0 - p x1),   p = s00 s01:
// two FMAs per amplitude, the factors c s00 / c s10 left for the end.  A
// pass takes tiles of 2^12 amplitudes whose bits V are the pass's qubits
// plus the lowest address bits (runs of at least 16 amplitudes, 128 bytes),
// applies the butterflies of all its qubits and multiplies each output once
// by C sigma (-1)^popc(e & F), C = prod c_j, sigma = prod s00_j, F = the
// tile bits whose s10 differs from s00: one read and one write of the
// state, about 40 instructions per amplitude.  (General complex 2x2 factors
// would cost 8 FMAs per amplitude and qubit, 96 for a 12-qubit pass, more
// than the issue rate allows at HBM speed; those layers stay with the
// tensor-core blocks.)
//
// A tile is 32 KB of shared memory.  256 threads hold 16 amplitudes each in
// three layouts (tile index e, bits 0..11), so that every butterfly finds
// both amplitudes in one thread's registers:
//   1  registers = tile bits 0, 1, 10, 11, thread = bits 2..9: loaded from
//      global memory as whole 32-byte sectors, 1 KB per warp access;
//   2  registers = tile bits 2..5, read and written back in place;
//   3  registers = tile bits 6..9, thread = bits 0..5, 10, 11: stored, the
//      lanes on consecutive amplitudes.
// A tile crosses shared memory four times; four CTAs per SM cover one
// another's loads and barriers (three a tile).  Element e sits at position
// p = e ^ (bits 6..8 of e) << 2, then bit 1 XOR bit 4 of p: the 16-byte
// writes of eight lanes meet eight different slots, the 8-byte accesses of a
// warp 32 different places.  The global addresses of a thread's accesses step
// through the register bits in Gray-code order, one 64-bit add each.
// Per 28-qubit pass: 0.718 ms (5.98 TB/s, 89 % of HBM); 0.778 ms with the
// passes' qubits in ascending order (launch_product), then 0.805 ms with
// tiles copied in asynchronously ahead (double-buffered, 24 instead of 32
// warps per SM, six crossings of shared memory).  With 64 amplitudes a thread
// and two layouts (two crossings, 12 warps per SM) a pass took 1.18 ms: too
// few warps to cover the latencies.
//
// Norm control.  A product pass is one step of the same norm chain as the
// tensor-core block passes (norm_chain.cuh): its inputs' and outputs' sums
// of |x|^2 per CTA in FP64 and the scale from the previous pass's record.
// C is rounded to FP32 (2^(-k/2) for k gates, exact only for even k) and the
// FP32 additions round; the control returns the norm to its target after
// every pass.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "common.cuh"
#include "internal.h"
#include "norm_chain.cuh"

using namespace qsim_dev;

namespace {

constexpr int kPBits = 12;                           // tile bits
constexpr int kPThreads = 256;
constexpr int kPPer = (1 << kPBits) / kPThreads;     // amplitudes per thread: 16
constexpr int kPCtasPerSm = 4;
constexpr int kPMinRun = 4;                          // runs of at least 2^4 amplitudes (128 B)
constexpr int kPTile = 1 << kPBits;                  // amplitudes per tile
constexpr int kPSmem = kPTile * 8;                   // 32 KB

struct ProdArgs {
    float2 *psi;
    uint64_t ntiles;          // 2^(n - 12)
    InsertSpec vspec;         // the 12 tile bits V as address bits, ascending
    int nruns;                // V as runs of consecutive address bits: [run_pos, run_pos + run_len)
    int run_pos[kPBits];
    int run_len[kPBits];
    uint32_t gmask;           // tile bits that carry a gate
    uint32_t fmask;           // F: tile bits whose s10 differs from s00
    float p[kPBits];          // p = s00 s01 of tile bit j
    uint64_t step[kPBits];    // address bit of tile bit j
    uint32_t flip[kPBits];    // the sign bit where F holds tile bit j
    float cs;                 // C sigma
    qsim_chain::ChainArgs chain;  // norm control (norm_chain.cuh)
};

// shared-memory position of tile element e (linear over GF(2))
__host__ __device__ constexpr uint32_t swz(uint32_t e) {
    const uint32_t p = e ^ (((e >> 6) & 7u) << 2);
    return p ^ (((p >> 4) & 1u) << 1);
}

// Gray code of step k and the bit it changes from step k - 1
__host__ __device__ constexpr int gray(int k) { return k ^ (k >> 1); }
__host__ __device__ constexpr int gray_bit(int k) {
    if (k == 0) return -1;
    int b = 0;
    while (!((k >> b) & 1)) ++b;
    return b;
}

// First address of tile t: the bits of t spread around the runs of V
__device__ __forceinline__ uint64_t tile_base(uint64_t t, const ProdArgs &A) {
    for (int j = 0; j < A.nruns; ++j) {
        const int p = A.run_pos[j];
        t = ((t >> p) << (p + A.run_len[j])) | (t & ((1ull << p) - 1ull));
    }
    return t;
}

__device__ __forceinline__ void bfly(float2 &v0, float2 &v1, float p) {
    const float2 a = v0, b = v1;
    v0 = make_float2(fmaf(p, b.x, a.x), fmaf(p, b.y, a.y));
    v1 = make_float2(fmaf(-p, b.x, a.x), fmaf(-p, b.y, a.y));
}

// Butterfly of register bit r (a tile bit's p)
template <int R>
__device__ __forceinline__ void stage(float2 (&v)[kPPer], float p) {
#pragma unroll
    for (int i = 0; i < kPPer; ++i)
        if (!((i >> R) & 1)) bfly(v[i], v[i | (1 << R)], p);
}

// whole-sector load: four adjacent amplitudes (32-byte aligned)
__device__ __forceinline__ void ld_sector(const float2 *p, float2 &a, float2 &b, float2 &c, float2 &d) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(b.x), "=f"(b.y), "=f"(c.x), "=f"(c.y), "=f"(d.x), "=f"(d.y)
                 : "l"(p));
}

__global__ void __launch_bounds__(kPThreads, kPCtasPerSm) k_product(const ProdArgs A) {
    extern __shared__ __align__(16) float2 x[];  // a tile of 2^12 amplitudes (positions swz(e))
    __shared__ float s_scale;
    __shared__ double s_red[kPThreads / 32][2];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // address bits of tile index e
    auto addr = [&](uint32_t e) {
        uint64_t a = 0;
#pragma unroll
        for (int j = 0; j < kPBits; ++j)
            if ((e >> j) & 1u) a |= A.step[j];
        return a;
    };
    if (warp == 0) {
        const float sc = qsim_chain::chain_scale(A.chain);  // and the record
        if (lane == 0) s_scale = sc;
    }
    __syncthreads();
    const float out_scale = s_scale * A.cs;  // every output, before its sign
    // this thread's tile bits in the three layouts
    const uint32_t e1 = tid << 2, e2 = (tid & 3u) | ((tid >> 2) << 6), e3 = (tid & 63u) | ((tid >> 6) << 10);
    const uint64_t off1 = addr(e1), off3 = addr(e3);
    // the sign of this thread's first output; the others follow bit by bit
    const float f_tid = (__popc(e3 & A.fmask) & 1) ? -out_scale : out_scale;
    const uint32_t w1 = swz(e1), r2 = swz(e2), r3 = swz(e3);
    double nin = 0.0, nout = 0.0;
    for (uint64_t t = blockIdx.x; t < A.ntiles; t += gridDim.x) {
        const uint64_t base = tile_base(t, A);
        float2 v[kPPer];  // layout 1: register i = tile bits 0, 1 | bits 10, 11 << 2
        {
            const float2 *p = A.psi + base + off1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int g = gray(k), b = gray_bit(k);
                if (b >= 0) p = (gray(k - 1) >> b) & 1 ? p - A.step[10 + b] : p + A.step[10 + b];
                ld_sector(p, v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
            }
        }
        {
            float q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < kPPer; ++i) q[i & 3] = fmaf(v[i].x, v[i].x, fmaf(v[i].y, v[i].y, q[i & 3]));
            nin += (double)((q[0] + q[1]) + (q[2] + q[3]));
        }
        if (A.gmask & 1u) stage<0>(v, A.p[0]);
        if (A.gmask & 2u) stage<1>(v, A.p[1]);
        if (A.gmask & 0x400u) stage<2>(v, A.p[10]);
        if (A.gmask & 0x800u) stage<3>(v, A.p[11]);
        __syncthreads();  // the previous tile has been read
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 a = v[4 * g + 2 * h], b = v[4 * g + 2 * h + 1];
                *(float4 *)(x + (w1 ^ swz(((uint32_t)g << 10) | (2u * h)))) = make_float4(a.x, a.y, b.x, b.y);
            }
        __syncthreads();
        if (A.gmask & 0x3Cu) {
#pragma unroll
            for (int i = 0; i < kPPer; ++i) v[i] = x[r2 ^ swz((uint32_t)i << 2)];
            if (A.gmask & 4u) stage<0>(v, A.p[2]);
            if (A.gmask & 8u) stage<1>(v, A.p[3]);
            if (A.gmask & 0x10u) stage<2>(v, A.p[4]);
            if (A.gmask & 0x20u) stage<3>(v, A.p[5]);
#pragma unroll
            for (int i = 0; i < kPPer; ++i) x[r2 ^ swz((uint32_t)i << 2)] = v[i];
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < kPPer; ++i) v[i] = x[r3 ^ swz((uint32_t)i << 6)];
        if (A.gmask & 0x40u) stage<0>(v, A.p[6]);
        if (A.gmask & 0x80u) stage<1>(v, A.p[7]);
        if (A.gmask & 0x100u) stage<2>(v, A.p[8]);
        if (A.gmask & 0x200u) stage<3>(v, A.p[9]);
        {
            float q[4] = {0.f, 0.f, 0.f, 0.f};
            float2 *p = A.psi + base + off3;
            float f = f_tid;
#pragma unroll
            for (int k = 0; k < kPPer; ++k) {
                const int i = gray(k), b = gray_bit(k);
                if (b >= 0) {
                    p = (gray(k - 1) >> b) & 1 ? p - A.step[6 + b] : p + A.step[6 + b];
                    f = __uint_as_float(__float_as_uint(f) ^ A.flip[6 + b]);
                }
                q[k & 3] = fmaf(v[i].x, v[i].x, fmaf(v[i].y, v[i].y, q[k & 3]));
                *p = make_float2(v[i].x * f, v[i].y * f);
            }
            nout += (double)((q[0] + q[1]) + (q[2] + q[3]));
        }
    }
    // per-CTA sums, fixed order; the outputs' sum before the chain's scale
    nin = warp_sum(nin);
    nout = warp_sum(nout);
    if (lane == 0) {
        s_red[warp][0] = nin;
        s_red[warp][1] = nout;
    }
    __syncthreads();
    if (tid == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < kPThreads / 32; ++w) {
            a += s_red[w][0];
            b += s_red[w][1];
        }
        qsim_chain::chain_sums(A.chain, a, b * (double)A.cs * (double)A.cs);
    }
}

// One pass: the butterfly gates of `qubits` (m of them, ascending, at most
// 12) with tile bits V = qubits plus the lowest address bits outside them.
int launch_pass(qsim *s, const int *qubits, const cd *const *mats, int m) {
    const int n = s->n;
    ProdArgs a{};
    uint64_t V = 0;
    for (int j = 0; j < m; ++j) V |= 1ull << qubits[j];
    for (int b = 0; b < n && __builtin_popcountll(V) < kPBits; ++b) V |= 1ull << b;
    a.vspec.m = kPBits;
    double C = 1.0, sigma = 1.0;
    for (int b = 0, k = 0; b < n; ++b)
        if ((V >> b) & 1ull) {
            for (int j = 0; j < m; ++j)
                if (qubits[j] == b) {
                    const cd *u = mats[j];
                    if (!butterfly2(u)) return set_err(s, QSIM_EINVAL, "product pass: not a butterfly matrix");
                    const double s00 = u[0].real() > 0 ? 1.0 : -1.0, s01 = u[1].real() > 0 ? 1.0 : -1.0,
                                 s10 = u[2].real() > 0 ? 1.0 : -1.0;
                    a.p[k] = (float)(s00 * s01);
                    if (s10 != s00) a.fmask |= 1u << k;
                    a.gmask |= 1u << k;
                    C *= std::abs(u[0]);
                    sigma *= s00;
                }
            a.step[k] = 1ull << b;
            a.flip[k] = (a.fmask >> k) & 1u ? 0x80000000u : 0u;
            a.vspec.pos[k++] = b;
        }
    a.cs = (float)(C * sigma);
    for (int k = 0; k < kPBits;) {
        int l = 1;
        while (k + l < kPBits && a.vspec.pos[k + l] == a.vspec.pos[k] + l) ++l;
        a.run_pos[a.nruns] = a.vspec.pos[k];
        a.run_len[a.nruns++] = l;
        k += l;
    }
    a.psi = (float2 *)s->state;
    a.ntiles = 1ull << (n - kPBits);
    uint64_t cap = (uint64_t)s->sms * kPCtasPerSm;
    if (cap > (uint64_t)kMaxTcGrid) cap = kMaxTcGrid;
    const uint64_t grid = a.ntiles < cap ? a.ntiles : cap;
    a.chain = qsim_chain::chain_next(s);  // the norm chain of the block passes
    static bool attr_set[64] = {false};
    if (s->device < 0 || s->device >= 64) return QSIM_ENOTSUP;
    if (!attr_set[s->device]) {
        const cudaError_t e = cudaFuncSetAttribute(k_product, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmem);
        if (e != cudaSuccess) return cuda_err(s, e, "product pass attribute");
        attr_set[s->device] = true;
    }
    k_product<<<(unsigned)grid, kPThreads, kPSmem, s->stream>>>(a);
    s->stats.launches++;
    qsim_chain::chain_advance(s, (int)grid);
    return cuda_err(s, cudaGetLastError(), "product pass launch");
}

}  // namespace

int product_pass_count(uint64_t qmask) {
    const uint64_t low = qmask & ((1ull << kPBits) - 1ull);
    const int nlo = __builtin_popcountll(low), nhi = __builtin_popcountll(qmask >> kPBits);
    const int per = kPBits - kPMinRun;
    const int npass_hi = (nhi + per - 1) / per;
    const int last = nhi - (npass_hi - 1) * per;
    const int top_lo = low ? 63 - __builtin_clzll(low) : -1;
    const bool fold = npass_hi > 0 && (nlo == 0 || top_lo < kPBits - last);
    return npass_hi + ((nlo > 0 && !fold) ? 1 : 0);
}

int launch_product(qsim *s, uint64_t qmask, const cd *mats, int *npasses) {
    *npasses = 0;
    if (s->prec != QSIM_C64 || s->n < kPBits) return QSIM_ENOTSUP;
    int lo[64], hi[64], nlo = 0, nhi = 0;
    const cd *mlo[64], *mhi[64];
    for (int b = 0, k = 0; b < s->n; ++b)
        if ((qmask >> b) & 1ull) {
            if (b < kPBits) {
                mlo[nlo] = mats + 4 * k;
                lo[nlo++] = b;
            } else {
                mhi[nhi] = mats + 4 * k;
                hi[nhi++] = b;
            }
            ++k;
        }
    // the qubits above the tile, kPBits - kPMinRun per pass; the last (the
    // smallest) pass also takes the low qubits if they lie in its runs
    const int per = kPBits - kPMinRun;
    const int npass_hi = (nhi + per - 1) / per;
    const int last = nhi - (npass_hi - 1) * per;  // qubits of the last high pass
    const bool fold = npass_hi > 0 && (nlo == 0 || lo[nlo - 1] < kPBits - last);
    // Each pass takes half its qubits from the lowest and half from the highest
    // left.  A tile of a pass on the 8 highest qubits of 28 has its 256 runs 8 MB
    // and more apart, each in a page of its own: 0.89 ms, the passes on lower
    // qubits 0.72.  In halves the pages of a tile are at most 64: the two passes
    // 1.39 instead of 1.60 ms (every other qubit: 1.43).
    int of[64];
    for (int p = 0, a = 0, b = nhi - 1; p < npass_hi; ++p) {
        const int k = p < npass_hi - 1 ? per : last;
        for (int i = 0; i < k; ++i) of[i < (k + 1) / 2 ? a++ : b--] = p;
    }
    int rc = QSIM_OK;
    if (nlo > 0 && !fold) {
        rc = launch_pass(s, lo, mlo, nlo);
        ++*npasses;
    }
    for (int p = 0; p < npass_hi && !rc; ++p) {
        int q[kPBits];
        const cd *m[kPBits];
        int k = 0;
        if (p == npass_hi - 1 && fold)
            for (int j = 0; j < nlo; ++j) {
                q[k] = lo[j];
                m[k++] = mlo[j];
            }
        for (int j = 0; j < nhi; ++j)
            if (of[j] == p) {
                q[k] = hi[j];
                m[k++] = mhi[j];
            }
        rc = launch_pass(s, q, m, k);
        ++*npasses;
    }
    return rc;
}
