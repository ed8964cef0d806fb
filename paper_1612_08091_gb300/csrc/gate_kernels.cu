// gate_kernels.cu -- unfused ("plain") gate application, one launch per gate.
//
// The operation is the simulator's per-gate sweep over the 2^n amplitudes
// (ProjectQ paper, Sec. 4.3.2): for every group of amplitudes that differ
// only in the target bits and have every control bit equal to 1 (Sec. 4.1.3,
// Control), replace the 2^t amplitudes of the group by U times them.  Groups
// are enumerated directly by inserting zero bits at the target and control
// positions into a group counter, so a gate with c controls touches only the
// 2^(n-c) amplitudes it changes (a 27-control Z on 28 qubits touches 2).
//
// Each thread owns one group: it gathers 2^t amplitudes, multiplies, and
// scatters.  complex128 uses FP64 arithmetic, complex64 FP32.  Specialised
// kernels avoid arithmetic the gate does not need: a phase on the all-ones
// subspace (Z, S, T, R(phi), CZ, multi-controlled Z), a diagonal one-qubit
// gate (RZ), and the X permutation (X, CNOT, Toffoli).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "df128.cuh"
#include "fx128.cuh"
#include "internal.h"

using namespace qsim_dev;

namespace {

template <typename Amp> struct Mat1 { Amp m[4]; };
template <typename Amp, int K> struct MatK { Amp m[(1 << K) * (1 << K)]; uint64_t off[1 << K]; };

// One-qubit, phase and X kernels: each thread takes kGroups groups, g =
// block * 256 kGroups + u * 256 + thread (u < kGroups), and issues all their
// loads before any arithmetic, so that 4 to 8 amplitudes per thread are in
// flight (one group per thread left too few bytes in flight for HBM).
// A register whose groups would not fill the SMs that way takes one group a
// thread in blocks of 64 (kGroups and kPhaseGroups are then 1): at 12 qubits
// complex128 two CTAs did all the FP64 work, 8 us a dense gate against
// 3.5 us.
constexpr int kWide = 4, kWidePhase = 8;  // the phase kernel loads one amplitude per group
constexpr int kWideFx = 2;                 // k_dense1_fx: 4 groups leave too few warps, 1 too few loads in flight
constexpr int kNarrowThreads = 64;

inline unsigned blocks_for(uint64_t work, int threads) {
    return (unsigned)((work + (uint64_t)threads - 1) / (uint64_t)threads);
}
// fewer than two wide blocks per SM
inline bool narrow(const qsim *s, uint64_t ngroups, int wide) {
    return ngroups < (uint64_t)s->sms * 2 * 256 * (uint64_t)wide;
}

template <typename Amp, int kGroups>
__global__ void __launch_bounds__(256) k_dense1(Amp *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                uint64_t cmask, uint64_t tbit, const Mat1<Amp> M) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kGroups) + threadIdx.x;
    uint64_t i0[kGroups];
    Amp a[kGroups], b[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i0[u] = insert_zeros(g0 + u * blockDim.x, ins) | cmask;
            a[u] = psi[i0[u]];
            b[u] = psi[i0[u] | tbit];
        }
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            Amp na = cmul(M.m[0], a[u]);
            na = cfma(M.m[1], b[u], na);
            Amp nb = cmul(M.m[2], a[u]);
            nb = cfma(M.m[3], b[u], nb);
            psi[i0[u]] = na;
            psi[i0[u] | tbit] = nb;
        }
}

// complex128 one-qubit dense gate in shared-exponent integers (fx128.cuh): 26
// qubits 0.43 ms on a full state (5.0 TB/s, 74 % of HBM; 0.31 ms while most
// groups are zero) against 1.03 ms in FP64 arithmetic; bound by the integer
// multiply-add pipe.
template <int kGroups, bool Apart>
__global__ void __launch_bounds__(256) k_dense1_fx(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                   uint64_t cmask, uint64_t tbit, const qsim_fx::MatFx M) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kGroups) + threadIdx.x;
    // the groups' first indices: a zero bit inserted at p turns i into
    // i + (i & -2^p), two operations (the integer units are the bottleneck)
    uint64_t i0[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u) i0[u] = g0 + u * blockDim.x;
    for (int j = 0; j < ins.m; ++j) {
        const uint64_t high = ~0ull << ins.pos[j];
#pragma unroll
        for (int u = 0; u < kGroups; ++u) i0[u] += i0[u] & high;
    }
    double2 a[kGroups], b[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i0[u] |= cmask;
            a[u] = psi[i0[u]];
            b[u] = psi[i0[u] | tbit];
        }
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        if (g0 + u * blockDim.x >= ngroups) continue;
        double2 na, nb;
        qsim_fx::dense1<Apart>(M, a[u], b[u], na, nb);
        psi[i0[u]] = na;
        psi[i0[u] | tbit] = nb;
    }
}

template <typename Amp, int K>
__global__ void __launch_bounds__(128) k_denseK(Amp *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                uint64_t cmask, const MatK<Amp, K> M) {
    constexpr int D = 1 << K;
    const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (g >= ngroups) return;
    const uint64_t base = insert_zeros(g, ins) | cmask;
    Amp v[D];
#pragma unroll
    for (int r = 0; r < D; ++r) v[r] = psi[base + M.off[r]];
#pragma unroll 1
    for (int r = 0; r < D; ++r) {
        Amp acc = cmul(M.m[r * D], v[0]);
#pragma unroll
        for (int c = 1; c < D; ++c) acc = cfma(M.m[r * D + c], v[c], acc);
        psi[base + M.off[r]] = acc;
    }
}

template <typename Amp, int kPhaseGroups>
__global__ void __launch_bounds__(256) k_phase(Amp *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                               uint64_t mask, Amp z) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kPhaseGroups) + threadIdx.x;
    uint64_t i[kPhaseGroups];
    Amp v[kPhaseGroups];
#pragma unroll
    for (int u = 0; u < kPhaseGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i[u] = insert_zeros(g0 + u * blockDim.x, ins) | mask;
            v[u] = psi[i[u]];
        }
#pragma unroll
    for (int u = 0; u < kPhaseGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) psi[i[u]] = cmul(z, v[u]);
}

template <typename Amp, int kGroups>
__global__ void __launch_bounds__(256) k_diag1(Amp *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                               uint64_t cmask, uint64_t tbit, Amp d0, Amp d1) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kGroups) + threadIdx.x;
    uint64_t i0[kGroups];
    Amp a[kGroups], b[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i0[u] = insert_zeros(g0 + u * blockDim.x, ins) | cmask;
            a[u] = psi[i0[u]];
            b[u] = psi[i0[u] | tbit];
        }
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            psi[i0[u]] = cmul(d0, a[u]);
            psi[i0[u] | tbit] = cmul(d1, b[u]);
        }
}

template <typename Amp, int kGroups>
__global__ void __launch_bounds__(256) k_x(Amp *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                           uint64_t cmask, uint64_t tbit) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kGroups) + threadIdx.x;
    uint64_t i0[kGroups];
    Amp a[kGroups], b[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i0[u] = insert_zeros(g0 + u * blockDim.x, ins) | cmask;
            a[u] = psi[i0[u]];
            b[u] = psi[i0[u] | tbit];
        }
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            psi[i0[u]] = b[u];
            psi[i0[u] | tbit] = a[u];
        }
}

// complex128 with double-float arithmetic (df128.cuh): one-qubit dense,
// diagonal and phase gates, kGroups (kPhaseGroups) groups per thread
struct MatDF {
    qsim_df::C2 m[4];
};

template <int kGroups>
__global__ void __launch_bounds__(256) k_dense1_df(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                   uint64_t cmask, uint64_t tbit, const MatDF M) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kGroups) + threadIdx.x;
    uint64_t i0[kGroups];
    double2 a[kGroups], b[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i0[u] = insert_zeros(g0 + u * blockDim.x, ins) | cmask;
            a[u] = psi[i0[u]];
            b[u] = psi[i0[u] | tbit];
        }
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            const qsim_df::C2 x = qsim_df::split(a[u]), y = qsim_df::split(b[u]);
            psi[i0[u]] = qsim_df::to_double(qsim_df::cdot2(M.m[0], x, M.m[1], y));
            psi[i0[u] | tbit] = qsim_df::to_double(qsim_df::cdot2(M.m[2], x, M.m[3], y));
        }
}

template <int kGroups>
__global__ void __launch_bounds__(256) k_diag1_df(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                  uint64_t cmask, uint64_t tbit, const MatDF M) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kGroups) + threadIdx.x;
    uint64_t i0[kGroups];
    double2 a[kGroups], b[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i0[u] = insert_zeros(g0 + u * blockDim.x, ins) | cmask;
            a[u] = psi[i0[u]];
            b[u] = psi[i0[u] | tbit];
        }
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            psi[i0[u]] = qsim_df::to_double(qsim_df::cmul(M.m[0], qsim_df::split(a[u])));
            psi[i0[u] | tbit] = qsim_df::to_double(qsim_df::cmul(M.m[3], qsim_df::split(b[u])));
        }
}

template <int kPhaseGroups>
__global__ void __launch_bounds__(256) k_phase_df(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                  uint64_t mask, const MatDF M) {
    const uint64_t g0 = blockIdx.x * (uint64_t)(blockDim.x * kPhaseGroups) + threadIdx.x;
    uint64_t i[kPhaseGroups];
    double2 v[kPhaseGroups];
#pragma unroll
    for (int u = 0; u < kPhaseGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) {
            i[u] = insert_zeros(g0 + u * blockDim.x, ins) | mask;
            v[u] = psi[i[u]];
        }
#pragma unroll
    for (int u = 0; u < kPhaseGroups; ++u)
        if (g0 + u * blockDim.x < ngroups) psi[i[u]] = qsim_df::to_double(qsim_df::cmul(M.m[3], qsim_df::split(v[u])));
}

// complex128 5-qubit dense gate or fused block in double-float arithmetic: the
// group's 2^k amplitudes split into FP32 pairs, each output the sum of 2^k exact-product complex MACs
// with two-sum additions, rounded once to double.  About 40 FP32 operations per
// MAC instead of 4 FP64 FMAs (FP64 runs at 1/58 of the FP32 rate here).
template <int K> struct MatKDF { qsim_df::C2 m[(1 << K) * (1 << K)]; uint64_t off[1 << K]; };

template <int K>
__global__ void __launch_bounds__(128) k_denseK_df(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                   uint64_t cmask, const MatKDF<K> M) {
    constexpr int D = 1 << K;
    const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (g >= ngroups) return;
    const uint64_t base = insert_zeros(g, ins) | cmask;
    qsim_df::C2 v[D];
#pragma unroll
    for (int r = 0; r < D; ++r) v[r] = qsim_df::split(psi[base + M.off[r]]);
#pragma unroll 1
    for (int r = 0; r < D; ++r) {
        // four partial sums: each addition rounds the low parts
        qsim_df::C2 acc[4];
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const qsim_df::C2 z = qsim_df::cmul(M.m[r * D + c], v[c]);
            acc[c & 3] = c < 4 ? z : qsim_df::cadd(acc[c & 3], z);
        }
        psi[base + M.off[r]] =
            qsim_df::to_double(qsim_df::cadd(qsim_df::cadd(acc[0], acc[1]), qsim_df::cadd(acc[2], acc[3])));
    }
}

// complex128 gate or fused block on 2 to 4 qubits whose matrix has one element
// in each row and column (CNOTs, SWAPs, phases), double-float option: every
// amplitude goes to its place, times its element in FP64 unless that is 1.  26
// qubits, a block of CNOTs: 0.49 ms (4.4 TB/s; 16 amplitudes a thread, few
// threads) where the integer form below takes 0.98 and rounds.
template <int K> struct MatKMono {
    double2 w[1 << K];
    uint64_t from[1 << K], to[1 << K];
    uint32_t ones;
};

template <int K>
__global__ void __launch_bounds__(128) k_monomial(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                  uint64_t cmask, const MatKMono<K> M) {
    constexpr int D = 1 << K;
    const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (g >= ngroups) return;
    double2 *const p = psi + (insert_zeros(g, ins) | cmask);
    double2 v[D];
#pragma unroll
    for (int c = 0; c < D; ++c) v[c] = p[M.from[c]];
#pragma unroll
    for (int c = 0; c < D; ++c) p[M.to[c]] = (M.ones >> c) & 1u ? v[c] : cmul(M.w[c], v[c]);
}

// complex128 k-qubit dense gate or fused block where the handle allows
// double-float accuracy, in shared-exponent integers and FP32 (fx128.cuh): a
// thread takes a group's 2^k amplitudes; a complex product is 4 integer
// multiply-adds and 8 FP32 ones, on two halves of the FMA pipe, where pairs of
// FP32 took 48 operations; one FP64 conversion per result.
// The error of this form is relative to the group's largest amplitude, that of
// pairs (2^-45) to a result's own products.  So each row's sum of |m| |v| is
// looked at (first a lower bound from the least elements of a quarter's rows for
// all of them, then, in a warp where that is too small, each): from kFxRow of U
// (fx128.cuh) on the error is below 2^-44.6 of it; where it is smaller
// (amplitudes of very different sizes under rows that do not mix them), the
// result is formed again in pairs, from the inputs kept in shared memory.
// 26 qubits, 4-qubit blocks: 0.98 to 1.04 ms a pass on a full state; a circuit of
// 27 passes 21.5 ms, 5.7e-15 from 64 bits, in pairs 43.7 ms and 6.2e-14.  (51 bits
// and no look at the rows: 21.7 ms, 6.0e-14, and amplitudes far below the group's
// largest kept few bits.)  Bound by issue and the integer multiply-adds.
template <int K> struct MatKFx {
    // each element's re and im (hi, hi rounded, lo) for 16- and 8-byte loads
    int4 a[(1 << K) * (1 << K)];    // re hi, im hi, and both as floats
    float2 b[(1 << K) * (1 << K)];  // re lo, im lo
    qsim_df::C2 m[(1 << K) * (1 << K)];
    float w[(1 << K) * (1 << K)];   // |element|, the largest row sum being 1/2 to 1
    float low[4][1 << K];           // the least of a quarter of the rows
    uint64_t off[1 << K];
    int shift;                    // -1027 - S
};
// times the square root of the number of amplitudes that are not 0, as the error
// (fx128.cuh): 2^-8 to 2^-6
constexpr float kFxRow = 0x1p-8f;

// All rows in FP64, from the matrix in pairs.
template <int K>
__device__ __forceinline__ void dense_fp64(double2 *p, const qsim_df::C2 *m, const uint64_t *off) {
    constexpr int D = 1 << K;
    double2 v[D];
#pragma unroll
    for (int r = 0; r < D; ++r) v[r] = p[off[r]];
#pragma unroll 1
    for (int r = 0; r < D; ++r) {
        double2 acc = make_double2(0.0, 0.0);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const qsim_df::C2 w = m[r * D + c];
            acc = cfma(make_double2((double)w.re.hi + w.re.lo, (double)w.im.hi + w.im.lo), v[c], acc);
        }
        p[off[r]] = acc;
    }
}

// One row times the inputs of this thread (E: their exponent; nz: which are not
// 0), in pairs, or FP64 beyond their range.
template <int K>
__device__ __forceinline__ double2 row_apart(const qsim_df::C2 *m, const double2 (*in)[128], uint32_t nz, int E) {
    constexpr int D = 1 << K;
    const int t = threadIdx.x;
    if (E > 1023 - 60 && E < 1023 + 60) {
        qsim_df::C2 acc[4] = {};
#pragma unroll 1
        for (int c = 0; c < D; c += 4) {
            if (!((nz >> c) & 15u)) continue;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[j] = qsim_df::cadd(acc[j], qsim_df::cmul(m[c + j], qsim_df::split(in[c + j][t])));
        }
        return qsim_df::to_double(qsim_df::cadd(qsim_df::cadd(acc[0], acc[1]), qsim_df::cadd(acc[2], acc[3])));
    }
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int c = 0; c < D; ++c)
        acc = cfma(make_double2((double)m[c].re.hi + m[c].re.lo, (double)m[c].im.hi + m[c].im.lo), in[c][t], acc);
    return acc;
}

template <int K>
__global__ void __launch_bounds__(128) k_denseK_fx(double2 *__restrict__ psi, uint64_t ngroups, const InsertSpec ins,
                                                   uint64_t cmask, const MatKFx<K> M) {
    using namespace qsim_fx;
    constexpr int D = 1 << K;
    __shared__ double2 s_in[D][128];
    const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (g >= ngroups) return;
    double2 *const p = psi + (insert_zeros(g, ins) | cmask);
    double2 v[D];
    uint32_t top = 0;
#pragma unroll
    for (int r = 0; r < D; ++r) {
        v[r] = p[M.off[r]];
        top = max(top, mag(v[r]));
    }
    const int E = (int)(top >> 20);
    if (!fx_range(E)) {
        bool zero = top == 0;
#pragma unroll
        for (int r = 0; r < D; ++r) zero = zero && v[r].x == 0.0 && v[r].y == 0.0;
        if (zero) return;
        dense_fp64<K>(p, M.m, M.off);  // amplitudes near the ends of the range
        return;
    }
    FxF xr[D], xi[D];
#pragma unroll
    for (int r = 0; r < D; ++r) {
        xr[r] = to_fxf(v[r].x, E);
        xi[r] = to_fxf(v[r].y, E);
    }
    uint32_t apart = 0, nz = 0;  // rows to be formed apart, amplitudes that are not 0
    {
        float size[D], low = 0x1p30f, count = 0.f;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            size[c] = fmaxf(fabsf(xr[c].fhi), fabsf(xi[c].fhi));
            count += size[c] > 0.f ? 1.f : 0.f;
        }
        const float line = kFxRow * 0x1p30f * sqrtf(count);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float t = 0.f;
#pragma unroll
            for (int c = 0; c < D; ++c) t = fmaf(M.low[q][c], size[c], t);
            low = fminf(low, t);
        }
        if (__any_sync(__activemask(), low < line)) {
#pragma unroll 2
            for (int r = 0; r < D; ++r) {
                float t = 0.f;
#pragma unroll
                for (int c = 0; c < D; ++c) t = fmaf(M.w[r * D + c], size[c], t);
                apart |= (uint32_t)(t < line) << r;
            }
        }
    }
    if (apart) {
        // (read again, one by one: v kept, or all at once, takes 40 registers more)
#pragma unroll 1
        for (int r = 0; r < D; ++r) {
            const double2 z = p[M.off[r]];
            s_in[r][threadIdx.x] = z;
            nz |= (uint32_t)(z.x != 0.0 || z.y != 0.0) << r;
        }
    }
    const int eadd = (E + M.shift) << 20;
#pragma unroll 2
    for (int r = 0; r < D; ++r) {
        long long rr = 0, ii = 0, ri = 0;  // sums of mr xr, mi xi, mr xi + mi xr
        float cr = 0.f, ci = 0.f;          // cross sums of the two results: hi by lo
        float dr = 0.f, di = 0.f;          // and lo by hi
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const int4 w = M.a[r * D + c];
            const float2 l = M.b[r * D + c];
            const float frh = __int_as_float(w.z), fih = __int_as_float(w.w);
            rr = mad_wide(w.x, xr[c].hi, rr);
            ii = mad_wide(w.y, xi[c].hi, ii);
            ri = mad_wide(w.x, xi[c].hi, ri);
            ri = mad_wide(w.y, xr[c].hi, ri);
            cr = fmaf(frh, xr[c].flo, cr);
            dr = fmaf(l.x, xr[c].fhi, dr);
            cr = fmaf(-fih, xi[c].flo, cr);
            dr = fmaf(-l.y, xi[c].fhi, dr);
            ci = fmaf(frh, xi[c].flo, ci);
            di = fmaf(l.x, xi[c].fhi, di);
            ci = fmaf(fih, xr[c].flo, ci);
            di = fmaf(l.y, xr[c].fhi, di);
        }
        p[M.off[r]] = make_double2(to_double_f(rr - ii, cr + dr, eadd), to_double_f(ri, ci + di, eadd));
    }
#pragma unroll 1
    for (; apart; apart &= apart - 1u) {
        const int r = __ffs(apart) - 1;
        p[M.off[r]] = row_apart<K>(M.m + r * D, s_in, nz, E);
    }
}

qsim_df::F2 host_split(double x) {
    qsim_df::F2 r;
    r.hi = (float)x;
    r.lo = (float)(x - (double)r.hi);
    return r;
}

MatDF make_df(const cd *m, int count) {
    MatDF M{};
    for (int i = 0; i < count; ++i) M.m[i] = qsim_df::C2{host_split(m[i].real()), host_split(m[i].imag())};
    return M;
}

// Returns true if the gate was launched on a double-float kernel.
bool gate_df(qsim *s, const GateRec &g) {
    if (g.t != 1) return false;
    double2 *psi = (double2 *)s->state;
    const uint64_t tbit = 1ull << g.targets[0];
    InsertSpec ins{};
    auto spec = [&](uint64_t mask) {
        ins.m = 0;
        for (int b = 0; b < 64; ++b)
            if ((mask >> b) & 1ull) ins.pos[ins.m++] = b;
    };
    const MatDF M = make_df(g.m.data(), 4);
    switch (g.kind) {
    case GK_DENSE: {
        spec(g.tmask | g.cmask);
        const uint64_t ng = 1ull << (s->n - ins.m);
        if (narrow(s, ng, kWide))
            k_dense1_df<1><<<blocks_for(ng, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ng, ins, g.cmask, tbit, M);
        else
            k_dense1_df<kWide><<<blocks_for(ng, 256 * kWide), 256, 0, s->stream>>>(psi, ng, ins, g.cmask, tbit, M);
        return true;
    }
    case GK_DIAG1: {
        spec(g.tmask | g.cmask);
        const uint64_t ng = 1ull << (s->n - ins.m);
        if (narrow(s, ng, kWide))
            k_diag1_df<1><<<blocks_for(ng, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ng, ins, g.cmask, tbit, M);
        else
            k_diag1_df<kWide><<<blocks_for(ng, 256 * kWide), 256, 0, s->stream>>>(psi, ng, ins, g.cmask, tbit, M);
        return true;
    }
    case GK_PHASE: {
        const uint64_t mask = g.tmask | g.cmask;
        spec(mask);
        const uint64_t ng = 1ull << (s->n - ins.m);
        if (narrow(s, ng, kWidePhase))
            k_phase_df<1><<<blocks_for(ng, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ng, ins, mask, M);
        else
            k_phase_df<kWidePhase><<<blocks_for(ng, 256 * kWidePhase), 256, 0, s->stream>>>(psi, ng, ins, mask, M);
        return true;
    }
    default:
        return false;
    }
}

InsertSpec make_spec(uint64_t mask) {
    InsertSpec s{};
    s.m = 0;
    for (int b = 0; b < 64; ++b)
        if ((mask >> b) & 1ull) s.pos[s.m++] = b;
    return s;
}

inline double2 to_amp(cd z, double2 *) { return make_double2(z.real(), z.imag()); }
inline float2 to_amp(cd z, float2 *) { return make_float2((float)z.real(), (float)z.imag()); }
template <typename Amp> Amp amp(cd z) { return to_amp(z, (Amp *)nullptr); }

template <int K>
int dense_k_df(qsim *s, const int *targets, uint64_t cmask, const cd *m) {
    constexpr int D = 1 << K;
    MatKDF<K> M;
    uint64_t tmask = 0;
    for (int j = 0; j < K; ++j) tmask |= 1ull << targets[j];
    for (int r = 0; r < D; ++r) {
        uint64_t o = 0;
        for (int j = 0; j < K; ++j)
            if ((r >> j) & 1) o |= 1ull << targets[j];
        M.off[r] = o;
    }
    for (int i = 0; i < D * D; ++i) M.m[i] = qsim_df::C2{host_split(m[i].real()), host_split(m[i].imag())};
    const InsertSpec ins = make_spec(tmask | cmask);
    const uint64_t ngroups = 1ull << (s->n - ins.m);
    k_denseK_df<K><<<blocks_for(ngroups, 128), 128, 0, s->stream>>>((double2 *)s->state, ngroups, ins, cmask, M);
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "double-float dense gate launch");
}

template <typename Amp, int K>
int dense_k_plain(qsim *s, const int *targets, uint64_t cmask, const cd *m) {
    constexpr int D = 1 << K;
    MatK<Amp, K> M;
    uint64_t tmask = 0;
    for (int j = 0; j < K; ++j) tmask |= 1ull << targets[j];
    for (int r = 0; r < D; ++r) {
        uint64_t o = 0;
        for (int j = 0; j < K; ++j)
            if ((r >> j) & 1) o |= 1ull << targets[j];
        M.off[r] = o;
    }
    for (int i = 0; i < D * D; ++i) M.m[i] = amp<Amp>(m[i]);
    const InsertSpec ins = make_spec(tmask | cmask);
    const uint64_t ngroups = 1ull << (s->n - ins.m);
    k_denseK<Amp, K><<<blocks_for(ngroups, 128), 128, 0, s->stream>>>((Amp *)s->state, ngroups, ins, cmask, M);
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "dense gate launch");
}

template <int K>
int dense_k_fx(qsim *s, const int *targets, uint64_t cmask, const cd *m) {
    constexpr int D = 1 << K;
    MatKFx<K> M;
    uint64_t tmask = 0;
    for (int j = 0; j < K; ++j) tmask |= 1ull << targets[j];
    for (int r = 0; r < D; ++r) {
        uint64_t o = 0;
        for (int j = 0; j < K; ++j)
            if ((r >> j) & 1) o |= 1ull << targets[j];
        M.off[r] = o;
    }
    double rows = 0.0;  // largest sum of |re| + |im| of a row
    int in_row[D] = {0}, in_col[D] = {0}, row_of[D] = {0};
    for (int r = 0; r < D; ++r) {
        double t = 0.0;
        for (int c = 0; c < D; ++c) {
            const cd z = m[r * D + c];
            t += std::abs(z.real()) + std::abs(z.imag());
            if (z != 0.0) ++in_row[r], ++in_col[c], row_of[c] = r;
        }
        rows = std::max(rows, t);
    }
    bool mono = true;
    for (int r = 0; r < D; ++r) mono = mono && in_row[r] == 1 && in_col[r] == 1;
    if (mono) {
        MatKMono<K> P;
        P.ones = 0;
        for (int c = 0; c < D; ++c) {
            const cd z = m[row_of[c] * D + c];
            P.w[c] = amp<double2>(z);
            P.from[c] = M.off[c];
            P.to[c] = M.off[row_of[c]];
            if (z == 1.0) P.ones |= 1u << c;
        }
        const InsertSpec ins = make_spec(tmask | cmask);
        const uint64_t ngroups = 1ull << (s->n - ins.m);
        k_monomial<K><<<blocks_for(ngroups, 128), 128, 0, s->stream>>>((double2 *)s->state, ngroups, ins, cmask, P);
        s->stats.launches++;
        return cuda_err(s, cudaGetLastError(), "monomial gate launch");
    }
    // a zero or an extreme matrix: FP64
    if (!(rows > qsim_fx::kFxMatrixLow) || !(rows < qsim_fx::kFxMatrixTop))
        return dense_k_plain<double2, K>(s, targets, cmask, m);
    int x;
    std::frexp(rows, &x);  // rows < 2^x
    const int S = 55 - x;
    for (int i = 0; i < D * D; ++i) {
        auto part = [&](double v, int &hi, float &fhi, float &flo) {
            const long long w = std::llrint(std::ldexp(v, S));
            hi = (int)((w + (1ll << 24)) >> 25);
            fhi = (float)hi;
            flo = (float)(w - ((long long)hi << 25));
        };
        float fr, fi;
        part(m[i].real(), M.a[i].x, fr, M.b[i].x);
        part(m[i].imag(), M.a[i].y, fi, M.b[i].y);
        std::memcpy(&M.a[i].z, &fr, 4);
        std::memcpy(&M.a[i].w, &fi, 4);
        M.m[i] = qsim_df::C2{host_split(m[i].real()), host_split(m[i].imag())};
        M.w[i] = (float)std::ldexp(std::abs(m[i]), -x);
    }
    // the least elements of a quarter's rows, rows that mix the same columns together
    uint32_t cols[D] = {0};
    int row[D];
    for (int r = 0; r < D; ++r) {
        row[r] = r;
        for (int c = 0; c < D; ++c) cols[r] |= (uint32_t)(M.w[r * D + c] > 0x1p-20f) << c;
    }
    std::stable_sort(row, row + D, [&](int a, int b) { return cols[a] < cols[b]; });
    for (int q = 0; q < 4; ++q)
        for (int c = 0; c < D; ++c) {
            float low = M.w[row[q * (D / 4)] * D + c];
            for (int k = 1; k < D / 4; ++k) low = std::min(low, M.w[row[q * (D / 4) + k] * D + c]);
            M.low[q][c] = low;
        }
    M.shift = -1027 - S;
    const InsertSpec ins = make_spec(tmask | cmask);
    const uint64_t ngroups = 1ull << (s->n - ins.m);
    k_denseK_fx<K><<<blocks_for(ngroups, 128), 128, 0, s->stream>>>((double2 *)s->state, ngroups, ins, cmask, M);
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "integer dense gate launch");
}

template <typename Amp, int K>
int dense_k(qsim *s, const int *targets, uint64_t cmask, const cd *m) {
    if constexpr (sizeof(Amp) == 16) {
        // integers up to 4 qubits; the 32 amplitudes of a 5-qubit group in FP32
        // pairs, whose plans the narrower blocks beat either way (27 qubits,
        // depth 10: 56 ms with 4-qubit blocks, 69 ms with integer 5-qubit ones)
        if (s->c128_df) {
            if constexpr (K <= 4)
                return dense_k_fx<K>(s, targets, cmask, m);
            else
                return dense_k_df<K>(s, targets, cmask, m);
        }
    }
    return dense_k_plain<Amp, K>(s, targets, cmask, m);
}

template <typename Amp>
int gate_plain(qsim *s, const GateRec &g) {
    Amp *psi = (Amp *)s->state;
    const uint64_t tbit = 1ull << g.targets[0];
    switch (g.kind) {
    case GK_PHASE: {
        const uint64_t mask = g.tmask | g.cmask;
        const InsertSpec ins = make_spec(mask);
        const uint64_t ngroups = 1ull << (s->n - ins.m);
        if (narrow(s, ngroups, kWidePhase))
            k_phase<Amp, 1><<<blocks_for(ngroups, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ngroups, ins, mask, amp<Amp>(g.m[3]));
        else
            k_phase<Amp, kWidePhase><<<blocks_for(ngroups, 256 * kWidePhase), 256, 0, s->stream>>>(psi, ngroups, ins, mask, amp<Amp>(g.m[3]));
        break;
    }
    case GK_DIAG1: {
        const InsertSpec ins = make_spec(g.tmask | g.cmask);
        const uint64_t ngroups = 1ull << (s->n - ins.m);
        if (narrow(s, ngroups, kWide))
            k_diag1<Amp, 1><<<blocks_for(ngroups, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ngroups, ins, g.cmask, tbit, amp<Amp>(g.m[0]), amp<Amp>(g.m[3]));
        else
            k_diag1<Amp, kWide><<<blocks_for(ngroups, 256 * kWide), 256, 0, s->stream>>>(psi, ngroups, ins, g.cmask, tbit, amp<Amp>(g.m[0]), amp<Amp>(g.m[3]));
        break;
    }
    case GK_X: {
        const InsertSpec ins = make_spec(g.tmask | g.cmask);
        const uint64_t ngroups = 1ull << (s->n - ins.m);
        if (narrow(s, ngroups, kWide))
            k_x<Amp, 1><<<blocks_for(ngroups, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ngroups, ins, g.cmask, tbit);
        else
            k_x<Amp, kWide><<<blocks_for(ngroups, 256 * kWide), 256, 0, s->stream>>>(psi, ngroups, ins, g.cmask, tbit);
        break;
    }
    default: {
        switch (g.t) {
        case 1: {
            const InsertSpec ins = make_spec(g.tmask | g.cmask);
            const uint64_t ngroups = 1ull << (s->n - ins.m);
            if constexpr (sizeof(Amp) == 16) {
                qsim_fx::MatFx F;
                if (qsim_fx::make_fx(g.m.data(), F)) {
                    const bool nr = narrow(s, ngroups, kWideFx);
                    auto kernel = nr ? (F.apart ? k_dense1_fx<1, true> : k_dense1_fx<1, false>)
                                     : (F.apart ? k_dense1_fx<kWideFx, true> : k_dense1_fx<kWideFx, false>);
                    const int threads = nr ? kNarrowThreads : 256;
                    kernel<<<blocks_for(ngroups, nr ? threads : threads * kWideFx), threads, 0, s->stream>>>(
                        psi, ngroups, ins, g.cmask, tbit, F);
                    break;
                }
            }
            Mat1<Amp> M;
            for (int i = 0; i < 4; ++i) M.m[i] = amp<Amp>(g.m[i]);
            if (narrow(s, ngroups, kWide))
            k_dense1<Amp, 1><<<blocks_for(ngroups, kNarrowThreads), kNarrowThreads, 0, s->stream>>>(psi, ngroups, ins, g.cmask, tbit, M);
        else
            k_dense1<Amp, kWide><<<blocks_for(ngroups, 256 * kWide), 256, 0, s->stream>>>(psi, ngroups, ins, g.cmask, tbit, M);
            break;
        }
        case 2: return dense_k<Amp, 2>(s, g.targets, g.cmask, g.m.data());
        case 3: return dense_k<Amp, 3>(s, g.targets, g.cmask, g.m.data());
        case 4: return dense_k<Amp, 4>(s, g.targets, g.cmask, g.m.data());
        case 5: return dense_k<Amp, 5>(s, g.targets, g.cmask, g.m.data());
        default: return set_err(s, QSIM_EINVAL, "gate with more than 5 targets");
        }
    }
    }
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "gate launch");
}

template <typename Amp>
int block_dense(qsim *s, const int *q, int k, const cd *m) {
    if (k == 1) {
        GateRec g;
        g.t = 1;
        g.targets[0] = q[0];
        g.tmask = 1ull << q[0];
        g.m.assign(m, m + 4);
        g.kind = GK_DENSE;
        return launch_gate_plain(s, g);  // applies the double-float choice
    }
    switch (k) {
    case 2: return dense_k<Amp, 2>(s, q, 0, m);
    case 3: return dense_k<Amp, 3>(s, q, 0, m);
    case 4: return dense_k<Amp, 4>(s, q, 0, m);
    case 5: return dense_k<Amp, 5>(s, q, 0, m);
    }
    return set_err(s, QSIM_EINVAL, "block width outside 1..5");
}

template <typename Amp>
__global__ void k_set_basis(Amp *__restrict__ psi, uint64_t N, uint64_t basis) {
    uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (; i < N; i += stride) {
        Amp z;
        z.x = (i == basis) ? 1 : 0;
        z.y = 0;
        psi[i] = z;
    }
}

}  // namespace

int launch_gate_plain(qsim *s, const GateRec &g) {
    if (s->prec == QSIM_C128 && s->c128_df && gate_df(s, g)) {
        s->stats.launches++;
        return cuda_err(s, cudaGetLastError(), "double-float gate launch");
    }
    return s->prec == QSIM_C128 ? gate_plain<double2>(s, g) : gate_plain<float2>(s, g);
}

int launch_block_dense(qsim *s, const int *qubits, int k, const cd *m) {
    return s->prec == QSIM_C128 ? block_dense<double2>(s, qubits, k, m) : block_dense<float2>(s, qubits, k, m);
}

int launch_set_basis(qsim *s, uint64_t basis) {
    const uint64_t N = 1ull << s->n;
    const unsigned grid = (unsigned)std::min<uint64_t>(blocks_for(N, 256), (uint64_t)s->sms * 16);
    if (s->prec == QSIM_C128)
        k_set_basis<double2><<<grid, 256, 0, s->stream>>>((double2 *)s->state, N, basis);
    else
        k_set_basis<float2><<<grid, 256, 0, s->stream>>>((float2 *)s->state, N, basis);
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "set basis launch");
}
