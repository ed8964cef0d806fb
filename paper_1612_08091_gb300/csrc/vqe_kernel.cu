// vqe_kernel.cu -- a batch of variational circuits in one persistent launch.
//
// Not a method of the paper: the serving pattern of many small
// hardware-efficient-ansatz circuits (different qubit counts and depths)
// evaluated together, each ending in the transverse-field Ising energy
//   E = -sum_{i<n-1} <Z_i Z_{i+1}> - h sum_i <X_i>   (open chain).
// A circuit starts in |0...0> and runs L layers of RY(theta_q) on every
// qubit, RZ(phi_q) on every qubit, then CNOT(q -> q+1) for q = 0..n-2.
//
// Per layer the two rotations on a qubit fuse into U_q = RZ(phi) RY(theta)
// (they commute with the rotations on the other qubits), and the CNOT
// ladder is one permutation: applied in order it maps |b> to |b'> with
// b'_k = b_0 ^ ... ^ b_k, i.e. psi'[y] = psi[y ^ (y << 1) mod 2^n].
//
// Two persistent launches: every CTA, or cluster of CTAs, takes circuit ids
// from an atomic counter (largest circuits first) until its part of the batch
// is done; no CTA waits for one outside its cluster.  A circuit of n <= m qubits (m = 12..14, tuned) lives
// in the CTA's shared memory (k_vqe_batch); a larger one lives in a per-CTA
// global buffer and is processed in tiles of 2^13 amplitudes by window passes
// (k_vqe_window; vqe_window.cuh says which gates a pass applies).  The energy's
// X terms on the qubits above 12 are read in the last pass, the rest in one
// more read of the state.  Amplitudes are complex64 in FP32 arithmetic;
// energies accumulate per thread in FP32 over a few terms and in FP64 beyond.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <new>
#include <numeric>
#include <string>
#include <vector>

#include "../../include/qsim.h"
#include "common.cuh"
#include "vqe_window.cuh"

using namespace qsim_dev;
using namespace qsim_vqe;

namespace {

// amplitudes per thread held in registers for the in-place permutation
template <int T> struct RegAmps { static constexpr int value = T >= 1024 ? 16 : 32; };

struct VqeArgs {
    const int *order;
    const int *nq;
    const int *nl;
    const long long *aoff;
    const double *angles;
    double *energies;
    unsigned int *counter;  // this launch's queue (k_vqe_window: the clusters', then the CTAs')
    unsigned int *err;      // error flag (a bounded wait gave up)
    int begin, end;   // its circuits: order[begin..end)
    int split;        // k_vqe_window: order[begin..split) by clusters
    int m;            // qubits held in shared memory
    float2 *gbuf;     // per-CTA global buffers of gstride amplitudes
    size_t gstride;
    double h;
};

// A layer's rotations factor as (prod_q RZ(phi_q)) (prod_q RY(theta_q)):
// RZ and RY on one qubit keep their order, and gates on different qubits
// commute.  Write theta/2 = theta'/2 + j pi/2 with |theta'/2| <= pi/4; then
//   RY(theta) = RY(j pi) RY(theta'),   RY(pi) = X Z,   RY(2 pi) = -I,
//   RY(theta') = c' [[1, -t], [t, 1]],  c' = cos(theta'/2), t = tan(theta'/2),
// so the rotation proper is two FMAs per amplitude (|t| <= 1) and the rest
// is bookkeeping: c' and the sign (-1)^floor(j/2) join the layer's global
// factor, and for odd j the X Z is moved past the RZ (RZ(phi) X = X RZ(-phi)):
//   RZ(phi) RY(theta) = s c' X diag(e^{i phi/2}, -e^{-i phi/2}) [[1, -t], [t, 1]].
// The diagonal part of all qubits is
//   exp(-i Phi'/2) prod_{q in i} p_q,  p_q = e^{i phi_q} or -e^{-i phi_q} (odd j),
// Phi' = sum_q (+-phi_q), applied as one complex factor per amplitude from
// two small tables (low and high bits) while the amplitudes move anyway, and
// the X of the qubits with odd j (the layer's flip mask F) is an XOR of the
// index where each amplitude is read for writing back.
struct Rot {
    float t;
};

__device__ __forceinline__ void apply_pair(float2 *x, unsigned i0, unsigned i1, const Rot &g) {
    const float2 a = x[i0], b = x[i1];
    x[i0] = make_float2(fmaf(-g.t, b.x, a.x), fmaf(-g.t, b.y, a.y));
    x[i1] = make_float2(fmaf(g.t, a.x, b.x), fmaf(g.t, a.y, b.y));
}

// Rotation pairing the elements i and i ^ mask of a 2^k-amplitude array in
// shared memory (mask's lowest bit, the pivot, is 0 in i).
__device__ __forceinline__ void gate_smem(float2 *x, int k, unsigned mask, const Rot &g) {
    const unsigned half = 1u << (k - 1);
    const unsigned lowmask = (mask & (0u - mask)) - 1u;
    for (unsigned p = threadIdx.x; p < half; p += blockDim.x) {
        const unsigned i0 = ((p & ~lowmask) << 1) | (p & lowmask);
        apply_pair(x, i0, i0 ^ mask, g);
    }
    __syncthreads();
}

__device__ __forceinline__ unsigned ladder_src(unsigned y, unsigned mask) { return (y ^ (y << 1)) & mask; }

// Rotations g[0..nb) on a 2^k-amplitude array in shared memory, applied four
// at a time in registers: each thread loads the 16 amplitudes of a group,
// applies the four rotations there and stores them back, so a layer of k
// one-qubit rotations costs ceil(k/4) passes over shared memory instead of k.
// Rotation j pairs the elements i and i ^ mask[j] (single bits).  The masks'
// bits must differ; a group is a base with zeros at its bits XOR any subset of
// its masks.  A group of fewer than four rotations is padded with identity
// rotations on other bits.
__device__ __forceinline__ void cswap(int &a, int &b) {
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    a = lo;
    b = hi;
}

__device__ void gates_blocked(float2 *x, int k, const unsigned *mask, const Rot *g, int nb) {
    if (k < 4) {
        // fewer than four bits in the array: one pass per gate
        for (int j = 0; j < nb; ++j) gate_smem(x, k, mask[j], g[j]);
        return;
    }
    for (int g0 = 0; g0 < nb; g0 += 4) {
        // the group's four bits (padded with identity gates on the lowest
        // unused bits)
        const bool h1 = g0 + 1 < nb, h2 = g0 + 2 < nb, h3 = g0 + 3 < nb;
        unsigned m0 = mask[g0], m1 = h1 ? mask[g0 + 1] : 0u, m2 = h2 ? mask[g0 + 2] : 0u,
                 m3 = h3 ? mask[g0 + 3] : 0u;
        unsigned used = (m0 & (0u - m0)) | (m1 & (0u - m1)) | (m2 & (0u - m2)) | (m3 & (0u - m3));
        // padding on the lowest unused bit, at bit 4 or above where one is
        // free (a pivot in bits 0..3, the bank bits, costs a bank conflict)
        auto pad = [&]() {
            const unsigned hi = ~used & ((1u << k) - 1u) & ~15u;
            const unsigned m = hi ? (hi & (0u - hi)) : (~used & (used + 1u));
            used |= m;
            return m;
        };
        if (!h1) m1 = pad();
        if (!h2) m2 = pad();
        if (!h3) m3 = pad();
        const float t0 = g[g0].t, t1 = h1 ? g[g0 + 1].t : 0.f, t2 = h2 ? g[g0 + 2].t : 0.f,
                    t3 = h3 ? g[g0 + 3].t : 0.f;
        int s0 = __ffs(m0) - 1, s1 = __ffs(m1) - 1, s2 = __ffs(m2) - 1, s3 = __ffs(m3) - 1;
        cswap(s0, s1);
        cswap(s2, s3);
        cswap(s0, s2);
        cswap(s1, s3);
        cswap(s1, s2);
        const unsigned ngroups = 1u << (k - 4);
        for (unsigned gi = threadIdx.x; gi < ngroups; gi += blockDim.x) {
            unsigned base = gi;
            base = ((base >> s0) << (s0 + 1)) | (base & ((1u << s0) - 1u));
            base = ((base >> s1) << (s1 + 1)) | (base & ((1u << s1) - 1u));
            base = ((base >> s2) << (s2 + 1)) | (base & ((1u << s2) - 1u));
            base = ((base >> s3) << (s3 + 1)) | (base & ((1u << s3) - 1u));
            float2 v[16];
#pragma unroll
            for (int r = 0; r < 16; ++r)
                v[r] = x[base ^ ((r & 1) ? m0 : 0u) ^ ((r & 2) ? m1 : 0u) ^ ((r & 4) ? m2 : 0u) ^ ((r & 8) ? m3 : 0u)];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float t = j == 0 ? t0 : j == 1 ? t1 : j == 2 ? t2 : t3;
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    if ((r >> j) & 1) continue;
                    const int r1 = r | (1 << j);
                    const float2 a = v[r], bb = v[r1];
                    v[r] = make_float2(fmaf(-t, bb.x, a.x), fmaf(-t, bb.y, a.y));
                    v[r1] = make_float2(fmaf(t, a.x, bb.x), fmaf(t, a.y, bb.y));
                }
            }
#pragma unroll
            for (int r = 0; r < 16; ++r)
                x[base ^ ((r & 1) ? m0 : 0u) ^ ((r & 2) ? m1 : 0u) ^ ((r & 4) ? m2 : 0u) ^ ((r & 8) ? m3 : 0u)] = v[r];
        }
        __syncthreads();
    }
}

__device__ double block_sum_d(double v, double *sh) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (warp == 0) {
        r = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
        r = warp_sum(r);
    }
    __syncthreads();
    return r;
}

// ZZ part of a 2^k chunk whose global index bits above k are `hi` (n qubits):
// sum_i |psi_i|^2 * ((n-1) - 2 popc((i ^ i>>1) & (2^(n-1)-1))).
__device__ float zz_chunk(const float2 *x, int k, unsigned long long hi, int n) {
    const unsigned long long m1 = (n >= 2) ? ((1ull << (n - 1)) - 1ull) : 0ull;
    float acc = 0.f;
    for (unsigned i = threadIdx.x; i < (1u << k); i += blockDim.x) {
        const unsigned long long gi = hi | i;
        const float w = norm2(x[i]);
        acc += w * (float)((n - 1) - 2 * __popcll((gi ^ (gi >> 1)) & m1));
    }
    return acc;
}

// sum over pairs on bit `bit` of 2 Re(conj(a) b) inside a 2^k array
__device__ float x_chunk(const float2 *x, int k, int bit) {
    const unsigned half = 1u << (k - 1);
    const unsigned lowmask = (1u << bit) - 1u;
    float acc = 0.f;
    for (unsigned p = threadIdx.x; p < half; p += blockDim.x) {
        const unsigned i0 = ((p & ~lowmask) << 1) | (p & lowmask);
        const float2 a = x[i0], b = x[i0 | (1u << bit)];
        acc += 2.f * (a.x * b.x + a.y * b.y);
    }
    return acc;
}

// t[j] = extra * prod over the set bits i of j (i < kb) of ph[i]
__device__ void build_phase_table(float2 *t, int kb, const float2 *ph, float2 extra) {
    for (unsigned j = threadIdx.x; j < (1u << kb); j += blockDim.x) {
        float2 z = extra;
        for (int i = 0; i < kb; ++i)
            if ((j >> i) & 1u) z = cmul(z, ph[i]);
        t[j] = z;
    }
}

// A qubit's part of a layer (see Rot): t, the phase p_q, its factor
// s c' e^{-i (+-phi) / 2} of the layer's global factor, and its flip.
struct QubitLayer {
    float t;
    float2 ph, f;
    unsigned flip;
};
__device__ __forceinline__ QubitLayer qubit_layer(double theta, double phi) {
    constexpr double kPi = 3.14159265358979323846;
    const double hth = remainder(0.5 * theta, 2.0 * kPi);  // theta/2 (RY has period 4 pi)
    const double j = rint(hth * (2.0 / kPi));               // -2..2
    const int ji = (int)j;
    float sh, ch, sp, cp, s2, c2;
    sincosf((float)(hth - j * (0.5 * kPi)), &sh, &ch);
    sincosf((float)remainder(phi, 2.0 * kPi), &sp, &cp);
    sincosf((float)(0.5 * remainder(phi, 4.0 * kPi)), &s2, &c2);
    QubitLayer r;
    r.flip = (unsigned)ji & 1u;
    const float sc = ((ji >> 1) & 1) ? -ch : ch;  // (-1)^floor(j/2) c'
    r.t = sh / ch;
    r.ph = r.flip ? make_float2(-cp, sp) : make_float2(cp, sp);
    r.f = make_float2(sc * c2, r.flip ? sc * s2 : -sc * s2);
    return r;
}

// Circuits of n <= m qubits, each held in one CTA's shared memory.
template <int T>
__global__ void __launch_bounds__(T, 1) k_vqe_batch(const VqeArgs A) {
    constexpr int kRegAmps = RegAmps<T>::value;
    extern __shared__ float2 sm[];
    __shared__ int s_idx;
    __shared__ double s_red[32];
    __shared__ Rot s_rot[32];       // this layer's RY per qubit
    __shared__ float2 s_ph[32];     // e^{i phi_q}
    __shared__ unsigned s_mask[32]; // XOR mask of each rotation in the current pass
    __shared__ float2 s_tlo[128];   // phases of index bits 0..6 (times the global factor)
    __shared__ float2 s_thi[128];   // phases of the next bits of a chunk or register
    __shared__ float2 s_gph;        // the layer's global factor: prod_q s_q c'_q times e^{-i Phi'/2}
    __shared__ unsigned s_flip;     // the layer's flip mask F
    // the layer's rotations t_q, per-qubit phases p_q, flip mask and global
    // factor (warp 0; n <= 32)
    auto layer_setup = [&](const double *al, int n) {
        if (threadIdx.x < 32) {
            const unsigned q = threadIdx.x;
            unsigned flip = 0;
            float2 f = make_float2(1.f, 0.f);
            if (q < (unsigned)n) {
                const QubitLayer r = qubit_layer(al[q], al[n + q]);
                s_rot[q] = Rot{r.t};
                s_ph[q] = r.ph;
                flip = r.flip;
                f = r.f;
            }
            const unsigned fl = __ballot_sync(0xffffffffu, flip);
#pragma unroll
            for (int o = 16; o; o >>= 1)
                f = cmul(f, make_float2(__shfl_xor_sync(0xffffffffu, f.x, o), __shfl_xor_sync(0xffffffffu, f.y, o)));
            if (q == 0) {
                s_gph = f;
                s_flip = fl;
            }
        }
        __syncthreads();
    };
    for (;;) {
        if (threadIdx.x == 0) s_idx = A.begin + (int)atomicAdd(A.counter, 1u);
        __syncthreads();
        const int idx = s_idx;
        __syncthreads();
        if (idx >= A.end) break;
        const int c = A.order[idx];
        const int n = A.nq[c], L = A.nl[c];
        const double *ang = A.angles + A.aoff[c];
        const unsigned N = 1u << n;
        double zz = 0.0, xx = 0.0;
        {
            // --- shared-memory resident circuit -------------------------------
            for (unsigned i = threadIdx.x; i < N; i += T) sm[i] = make_float2(i == 0 ? 1.f : 0.f, 0.f);
            __syncthreads();
            const int klo = n < 7 ? n : 7;
            for (int l = 0; l < L; ++l) {
                const double *al = ang + 2 * l * n;
                if (threadIdx.x < (unsigned)n) s_mask[threadIdx.x] = 1u << threadIdx.x;
                layer_setup(al, n);
                build_phase_table(s_tlo, klo, s_ph, s_gph);
                build_phase_table(s_thi, n - klo, s_ph + klo, make_float2(1.f, 0.f));
                gates_blocked(sm, n, s_mask, s_rot, n);  // ends with a barrier
                // the RZ phases, the flips and the CNOT ladder as one pass
                // through registers
                const unsigned F = s_flip;
                float2 v[kRegAmps];
#pragma unroll
                for (int j = 0; j < kRegAmps; ++j) {
                    const unsigned y = threadIdx.x + (unsigned)j * T;
                    if (y < N) {
                        const unsigned x = ladder_src(y, N - 1) ^ F;
                        v[j] = cmul(sm[x], cmul(s_tlo[x & 127u], s_thi[x >> 7]));
                    }
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < kRegAmps; ++j) {
                    const unsigned y = threadIdx.x + (unsigned)j * T;
                    if (y < N) sm[y] = v[j];
                }
                __syncthreads();
            }
            zz = (double)zz_chunk(sm, n, 0ull, n);
            for (int q = 0; q < n; ++q) xx += (double)x_chunk(sm, n, q);
        }
        const double zzs = block_sum_d(zz, s_red);
        const double xxs = block_sum_d(xx, s_red);
        if (threadIdx.x == 0) A.energies[c] = -zzs - A.h * xxs;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// larger circuits: window passes over a state in global memory
// ---------------------------------------------------------------------------
// A CTA of 256 threads takes a circuit.  Per pass it works out the gates
// (thread 0), their rotations and phase tables and the groups (a thread each),
// then for every tile: asynchronous 16-byte copies in (zeros where the state
// is still zero), the steps, and 16-byte stores in logical order.  A step's
// rotations go five at a time on 32 amplitudes in registers, one start of the
// group per thread, the lanes on different banks (vqe_window.cuh); the last
// group of a step multiplies in the step's RZ phases, one factor per amplitude
// from two tables.  Two CTAs per SM (registers); on a full chip issue slots and
// shared memory are both half busy, between barriers, DRAM at 2 TB/s.
// (Before: a pair pass and a top-qubit pass over the whole state per layer:
// 4096 circuits of 10..20 qubits 26.3 ms, now 16.7.)
//
// Where few circuits hold much of the work, a circuit is shared by a cluster
// (Joint): each CTA works out the passes for itself and takes every csize-th
// tile, a cluster barrier between passes, the energy's parts added in the order
// of the ranks.  One CTA per circuit left most of the chip idle at the end (a
// circuit of 20 qubits and 8 layers alone 7.7 ms; by 8 CTAs 1.33).  When the
// clusters' circuits are done each CTA goes on alone with the smaller ones.
constexpr int kWinThreads = 256;
constexpr int kWinCtas = 2;
constexpr int kTile = 1 << kTileBits;
static_assert(kWinThreads == 1 << (kTileBits - kGroupBits), "one start of a group per thread");

struct WinShared {
    Progress prog;
    Pass pass;
    Map map[kMaxSteps];      // before each step
    Map end;                 // after the last
    Group group[kMaxGroups];
    float t[kMaxGroups][kGroupBits];
    float ts[kMaxSteps][kTileBits];
    float2 ph[kMaxSteps][kTileBits], f[kMaxSteps][kTileBits];
    unsigned flip[kMaxSteps];
    float2 tlo[kMaxSteps][128], thi[kMaxSteps][64];
    Group xgroup[3];         // X terms
    int nx;
};

// One group on the tile: each thread's 32 amplitudes, position start ^ sums of
// the masks, logical index y ^ the corresponding bits.
template <class F>
__device__ __forceinline__ void with_group(float2 *x, const Group &G, bool store, F f) {
    const unsigned sy = G.lane[threadIdx.x & 31] ^ G.hi[threadIdx.x >> 5];
    unsigned m[kGroupBits];
#pragma unroll
    for (int j = 0; j < kGroupBits; ++j) m[j] = G.m[j];
    float2 v[1 << kGroupBits];
    unsigned p = sy & 0xFFFFu;
#pragma unroll
    for (int k = 0; k < (1 << kGroupBits); ++k) {
        const int g = k ^ (k >> 1);
        if (k) {
            const int b = (k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : (k & 8) ? 3 : 4;
            p ^= m[b];
        }
        v[g] = x[p];
    }
    f(v, sy >> 16);
    if (!store) return;
    p = sy & 0xFFFFu;
#pragma unroll
    for (int k = 0; k < (1 << kGroupBits); ++k) {
        const int g = k ^ (k >> 1);
        if (k) {
            const int b = (k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : (k & 8) ? 3 : 4;
            p ^= m[b];
        }
        x[p] = v[g];
    }
}

// The groups of X terms on the tile bits of `bits`, under the map a (threads 0..2).
__device__ __forceinline__ void x_groups(WinShared &S, const Map &a, unsigned bits) {
    const int c = __popc(bits), ng = (c + kGroupBits - 1) / kGroupBits;
    if (threadIdx.x == 0) S.nx = ng;
    if ((int)threadIdx.x < ng) {
        int q[kGroupBits], k = 0, i = 0;
        for (int t = 0; t < kTileBits; ++t)
            if ((bits >> t) & 1u) {
                if (i % ng == (int)threadIdx.x) q[k++] = t;
                ++i;
            }
        make_group(a, q, k, S.xgroup[threadIdx.x]);
    }
    __syncthreads();
}
// sum over the groups' X terms of 2 Re(conj(a) b) over the pairs
__device__ __forceinline__ float x_terms(float2 *x, const WinShared &S) {
    float acc = 0.f;
    for (int g = 0; g < S.nx; ++g) {
        const int cnt = S.xgroup[g].cnt;
        with_group(x, S.xgroup[g], false, [&](float2(&v)[32], unsigned) {
#pragma unroll
            for (int j = 0; j < kGroupBits; ++j) {
                if (j >= cnt) continue;
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    if (!((k >> j) & 1)) s = fmaf(v[k].x, v[k | (1 << j)].x, fmaf(v[k].y, v[k | (1 << j)].y, s));
                acc = fmaf(2.f, s, acc);
            }
        });
    }
    return acc;
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// 64 bits of another CTA's shared memory, where this CTA has `p`
__device__ __forceinline__ unsigned long long peer_u64(const void *p, unsigned rank) {
    uint32_t a;
    unsigned long long v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}

template <bool Joint>
__global__ void __launch_bounds__(kWinThreads, kWinCtas) k_vqe_window(const VqeArgs A) {
    extern __shared__ __align__(16) float2 x[];  // the tile
    __shared__ WinShared S;
    __shared__ unsigned long long s_idx;
    __shared__ double s_red[32];
    __shared__ double s_part[2];  // this CTA's part of a cluster's energy
    const unsigned tid = threadIdx.x;
    unsigned rank = 0, csize = 1;  // 0 of 1 too once the clusters' circuits are done
    if (Joint) {
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(csize));
    }
    float2 *buf = A.gbuf + (size_t)(blockIdx.x - rank) * A.gstride;  // a cluster's: its first CTA's
    // every thread of the circuit's CTAs; what they wrote is visible after it
    auto sync = [&] {
        if (Joint && csize > 1)
            cluster_barrier();
        else
            __syncthreads();
    };
    // address of unit u (amplitudes 2u, 2u + 1 of the tile) of tile t
    auto tile_fixed = [](unsigned t, int w) {
        return ((t & ((1u << (w - kRunBits)) - 1u)) << kRunBits) | ((t >> (w - kRunBits)) << (w + kWindow));
    };
    auto unit_addr = [](unsigned u, int w) { return ((u & 1u) << 1) | ((u >> 1) << w); };
    constexpr unsigned kUnits = kTile / 2 / kWinThreads;  // 16 per thread
    auto load = [&](unsigned fixed, int w, int nz) {
#pragma unroll 4
        for (unsigned i = 0; i < kUnits; ++i) {
            const unsigned u = tid + i * kWinThreads, at = fixed | unit_addr(u, w);
            if (at >> nz)
                *(float4 *)(x + 2 * u) = make_float4(0.f, 0.f, 0.f, 0.f);
            else
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(x + 2 * u)),
                             "l"(buf + at)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    };
    for (;;) {
        sync();
        if (tid == 0 && rank == 0)
            s_idx = Joint && csize > 1 ? A.begin + atomicAdd(A.counter, 1u) : A.split + atomicAdd(A.counter + 1, 1u);
        sync();
        const int idx = (int)(Joint && csize > 1 ? peer_u64(&s_idx, 0) : s_idx);
        if (Joint && csize > 1 && idx >= A.split) {
            cluster_barrier();  // rank 0's word has been read
            buf = A.gbuf + (size_t)blockIdx.x * A.gstride;
            rank = 0;
            csize = 1;
            continue;
        }
        if (idx >= A.end) break;
        const int c = A.order[idx];
        const int n = A.nq[c], L = A.nl[c];
        const double *ang = A.angles + A.aoff[c];
        if (L == 0) {  // |0...0>
            if (tid == 0 && rank == 0) A.energies[c] = -(double)(n - 1);
            continue;
        }
        if (tid == 0) {
            progress_start(S.prog, n, L);
            if (rank == 0) {
                buf[0] = make_float2(1.f, 0.f);
                buf[1] = make_float2(0.f, 0.f);
            }
        }
        int nz = 1;  // the state is zero from index 2^nz on
        double xx = 0.0, zz = 0.0;
        for (bool last = false; !last;) {
            sync();
            if (tid == 0) make_pass(S.prog, window_start(S.prog), S.pass);
            __syncthreads();
            const int w = S.pass.w, ns = S.pass.nsteps;
            last = lowest_ready(S.prog) >= n;
            if (ns == 0 && S.pass.cn0 == 0) {  // cannot happen: every window holds a ready gate
                if (tid == 0) atomicOr(A.err, 1u);
                break;
            }
            // rotations of every step
            if (tid < kMaxSteps) S.flip[tid] = 0;
            __syncthreads();
            for (int i = tid; i < ns * kTileBits; i += kWinThreads) {
                const int st = i / kTileBits, t = i - st * kTileBits;
                if (!((S.pass.step[st].rot >> t) & 1u)) continue;
                const int q = t < kRunBits ? t : w + t - kRunBits, l = S.pass.step[st].layer[t];
                const QubitLayer r = qubit_layer(ang[2 * l * n + q], ang[2 * l * n + n + q]);
                S.ts[st][t] = r.t;
                S.ph[st][t] = r.ph;
                S.f[st][t] = r.f;
                if (r.flip) atomicOr(&S.flip[st], 1u << t);
            }
            __syncthreads();
            if (tid == 0) {
                Map M;
                map_identity(M);
                auto sweep = [&](unsigned cn) {
                    for (int t = 0; t + 1 < kTileBits; ++t)
                        if ((cn >> t) & 1u) map_cnot(M, t, t + 1);
                };
                sweep(S.pass.cn0);
                for (int st = 0; st < ns; ++st) {
                    S.map[st] = M;
                    M.f ^= S.flip[st];
                    sweep(S.pass.step[st].cn);
                }
                S.end = M;
            }
            // phase tables: index bits 0..6 (times the step's factor) and 7..12
            for (int i = tid; i < ns * 192; i += kWinThreads) {
                const int st = i / 192, e = i - st * 192;
                const unsigned rot = S.pass.step[st].rot;
                float2 z = make_float2(1.f, 0.f);
                if (e < 128) {
                    for (int t = 0; t < kTileBits; ++t)
                        if ((rot >> t) & 1u) z = cmul(z, S.f[st][t]);
                    for (int t = 0; t < 7; ++t)
                        if (((rot & (unsigned)e) >> t) & 1u) z = cmul(z, S.ph[st][t]);
                    S.tlo[st][e] = z;
                } else {
                    for (int t = 7; t < kTileBits; ++t)
                        if ((rot >> t) & ((unsigned)(e - 128) >> (t - 7)) & 1u) z = cmul(z, S.ph[st][t]);
                    S.thi[st][e - 128] = z;
                }
            }
            __syncthreads();
            if (tid < kMaxGroups) {
                for (int st = 0; st < ns; ++st) {
                    const Step &P = S.pass.step[st];
                    if ((int)tid < P.g0 || (int)tid >= P.g1) continue;
                    const int ng = P.g1 - P.g0, g = (int)tid - P.g0;
                    int q[kGroupBits], k = 0, i = 0;
                    for (int t = 0; t < kTileBits; ++t)
                        if ((P.rot >> t) & 1u) {
                            if (i % ng == g) {
                                S.t[tid][k] = S.ts[st][t];
                                q[k++] = t;
                            }
                            ++i;
                        }
                    make_group(S.map[st], q, k, S.group[tid]);
                }
            }
            __syncthreads();
            // the X terms on qubits 13 and above: the last window holds them
            unsigned xbits = 0;
            if (last)
                for (int t = kRunBits; t < kTileBits; ++t)
                    if (w + t - kRunBits >= kTileBits && w + t - kRunBits < n) xbits |= 1u << t;
            if (xbits) x_groups(S, S.end, xbits);
            const int reach = w + kWindow < n ? w + kWindow : n;
            const int nz_out = reach > nz ? reach : nz;
            // where this thread's stores find their amplitudes
            const unsigned p_tid = map_position(S.end, 2 * tid), p_one = S.end.inv[0];
            const unsigned tiles = 1u << (nz_out - kTileBits);
            for (unsigned t = rank; t < tiles; t += csize) {
                const unsigned fixed = tile_fixed(t, w);
                load(fixed, w, nz);
                for (int st = 0; st < ns; ++st) {
                    const int g1 = S.pass.step[st].g1;
                    for (int g = S.pass.step[st].g0; g < g1; ++g) {
                        const Group &G = S.group[g];
                        const bool phases = g == g1 - 1;
                        with_group(x, G, true, [&](float2(&v)[32], unsigned y) {
                            const int cnt = G.cnt;
#pragma unroll
                            for (int j = 0; j < kGroupBits; ++j) {
                                if (j >= cnt) continue;
                                float r = S.t[g][j];
                                if ((y >> G.q[j]) & 1u) r = -r;
#pragma unroll
                                for (int k = 0; k < 32; ++k) {
                                    if ((k >> j) & 1) continue;
                                    const float2 a = v[k], b = v[k | (1 << j)];
                                    v[k] = make_float2(fmaf(-r, b.x, a.x), fmaf(-r, b.y, a.y));
                                    v[k | (1 << j)] = make_float2(fmaf(r, a.x, b.x), fmaf(r, a.y, b.y));
                                }
                            }
                            if (phases) {
#pragma unroll
                                for (int k = 0; k < 32; ++k) {
                                    const int gk = k ^ (k >> 1);
                                    if (k) {
                                        const int b = (k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : (k & 8) ? 3 : 4;
                                        y ^= 1u << G.q[b];
                                    }
                                    v[gk] = cmul(v[gk], cmul(S.tlo[st][y & 127u], S.thi[st][y >> 7]));
                                }
                            }
                        });
                        __syncthreads();
                    }
                }
                if (xbits) xx += (double)x_terms(x, S);
#pragma unroll 4
                for (unsigned i = 0; i < kUnits; ++i) {
                    // unit tid + 256 i: index bits 9..12 are i's
                    unsigned p = p_tid;
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if ((i >> b) & 1u) p ^= S.end.inv[9 + b];
                    const float2 a = x[p], b = x[p ^ p_one];
                    *(float4 *)(buf + (fixed | unit_addr(tid + i * kWinThreads, w))) = make_float4(a.x, a.y, b.x, b.y);
                }
                __syncthreads();
            }
            nz = nz_out;
        }
        // ZZ of all qubits and X of the 13 lowest
        if (tid == 0) map_identity(S.end);
        sync();
        x_groups(S, S.end, n < kTileBits ? (1u << n) - 1u : (unsigned)kTile - 1u);
        const unsigned m1 = (1u << (n - 1)) - 1u;
        for (unsigned t = rank; t < (1u << (n - kTileBits)); t += csize) {
            load(t << kTileBits, kRunBits, n);
            float zf = 0.f;
            for (unsigned i = 0; i < kTile / kWinThreads; ++i) {
                const unsigned e = tid + i * kWinThreads, gi = (t << kTileBits) | e;
                zf = fmaf(norm2(x[e]), (float)((n - 1) - 2 * __popc((gi ^ (gi >> 1)) & m1)), zf);
            }
            const float xf = x_terms(x, S);
            zz += (double)zf;
            xx += (double)xf;
            __syncthreads();
        }
        double zzs = block_sum_d(zz, s_red);
        double xxs = block_sum_d(xx, s_red);
        if (Joint && csize > 1) {
            if (tid == 0) {
                s_part[0] = zzs;
                s_part[1] = xxs;
            }
            cluster_barrier();
            if (tid == 0 && rank == 0)
                for (unsigned r = 1; r < csize; ++r) {
                    zzs += __longlong_as_double((long long)peer_u64(&s_part[0], r));
                    xxs += __longlong_as_double((long long)peer_u64(&s_part[1], r));
                }
        }
        if (tid == 0 && rank == 0) A.energies[c] = -zzs - A.h * xxs;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side: the batch object, its graph and the tile autotuner
// ---------------------------------------------------------------------------
struct qsim_batch {
    int count = 0, nmax = 0;
    long long nangles = 0;
    double h = 0.7;
    std::vector<int> nq, nl, order;
    std::vector<long long> aoff;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int device = 0, sms = 0;
    // device memory
    unsigned char *mem = nullptr;
    size_t mem_bytes = 0;
    bool own_mem = false;
    double *d_angles = nullptr, *d_energies = nullptr;
    int *d_order = nullptr, *d_nq = nullptr, *d_nl = nullptr;
    long long *d_aoff = nullptr;
    unsigned int *d_counter = nullptr;
    float2 *d_gbuf = nullptr;
    size_t gstride = 0;
    int max_grid = 0;
    // pinned staging
    double *h_angles = nullptr, *h_energies = nullptr;
    unsigned int *h_flag = nullptr;  // the device error flag after a run
    // tuned launch configuration and its graph
    int threads = 512, m = 13, grid = 0;
    cudaGraphExec_t graph = nullptr;
    std::string err;
};

namespace {

constexpr int kCandidates[][2] = {{256, 12}, {256, 13}, {512, 12}, {512, 13}, {512, 14}, {1024, 13}, {1024, 14}};

int reg_amps(int threads) { return threads == 256 ? RegAmps<256>::value : threads == 512 ? RegAmps<512>::value
                                                                                       : RegAmps<1024>::value; }

typedef void (*VqeKernel)(const VqeArgs);
VqeKernel kernel_for(int threads) {
    return threads == 256 ? k_vqe_batch<256> : threads == 512 ? k_vqe_batch<512> : k_vqe_batch<1024>;
}

// the top window and the 13 lowest qubits cover all qubits
constexpr int kMaxBatchQubits = kTileBits + kWindow;
static_assert(kMaxBatchQubits == 24 && kMaxBatchQubits <= kMaxQ, "the range the interface states");
constexpr size_t kWinSmem = (size_t)8 << kTileBits;

// circuits with more than m qubits: a prefix of the order (sorted by size)
int count_large(const qsim_batch *b, int m) {
    int k = 0;
    while (k < b->count && b->nq[b->order[k]] > m) ++k;
    return k;
}

bool config_valid(int threads, int m) {
    return (1 << m) <= reg_amps(threads) * threads;  // in-place permutation through registers
}

int occupancy_global(const qsim_batch *b, int *grid) {
    VqeKernel k = k_vqe_window<true>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWinSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_vqe_window<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWinSmem);
    if (e != cudaSuccess) return QSIM_ECUDA;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kWinThreads, kWinSmem);
    if (e != cudaSuccess || per_sm < 1) return QSIM_ENOTSUP;
    *grid = b->sms * std::min(per_sm, kWinCtas);  // a buffer each
    return QSIM_OK;
}

int occupancy(const qsim_batch *b, int threads, int m, int *grid) {
    const size_t smem = (size_t)8 << m;
    VqeKernel k = kernel_for(threads);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return QSIM_ECUDA;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
    if (e != cudaSuccess || per_sm < 1) return QSIM_ENOTSUP;
    *grid = std::min(b->sms * per_sm, b->max_grid);
    return QSIM_OK;
}

int berr(qsim_batch *b, int code, const std::string &msg) {
    b->err = msg;
    return code;
}

int launch(qsim_batch *b, int threads, int m, int grid) {
    const int large = count_large(b, m);
    // the three queues' counters and the error flag
    cudaError_t e = cudaMemsetAsync(b->d_counter, 0, 4 * sizeof(unsigned int), b->stream);
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    VqeArgs a;
    a.order = b->d_order;
    a.nq = b->d_nq;
    a.nl = b->d_nl;
    a.aoff = b->d_aoff;
    a.angles = b->d_angles;
    a.energies = b->d_energies;
    a.err = b->d_counter + 3;
    a.m = m;
    a.gbuf = b->d_gbuf;
    a.gstride = b->gstride;
    a.h = b->h;
    if (large > 0) {
        // the larger circuits first, several CTAs per SM
        int ggrid = 0;
        const int rc = occupancy_global(b, &ggrid);
        if (rc) return berr(b, rc, "occupancy query failed");
        a.counter = b->d_counter;
        a.begin = 0;
        a.end = large;
        const int cl = cluster_size([b](int k) { return b->nq[b->order[k]]; }, large, ggrid, &a.split);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ggrid / cl * cl);
        cfg.blockDim = dim3(kWinThreads);
        cfg.dynamicSmemBytes = kWinSmem;
        cfg.stream = b->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cl;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = cl > 1;
        e = cudaLaunchKernelEx(&cfg, cl > 1 ? k_vqe_window<true> : k_vqe_window<false>, a);
        if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    }
    if (large < b->count) {
        a.counter = b->d_counter + 2;
        a.begin = large;
        a.end = b->count;
        kernel_for(threads)<<<grid, threads, (size_t)8 << m, b->stream>>>(a);
        e = cudaGetLastError();
        if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    }
    return QSIM_OK;
}

// Capture angles H2D -> queue reset -> persistent kernel -> energies D2H.
int build_graph(qsim_batch *b) {
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    int grid = 0;
    int rc = occupancy(b, b->threads, b->m, &grid);
    if (rc) return berr(b, rc, "occupancy query failed");
    b->grid = grid;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    cudaMemcpyAsync(b->d_angles, b->h_angles, sizeof(double) * b->nangles, cudaMemcpyHostToDevice, b->stream);
    rc = launch(b, b->threads, b->m, grid);
    cudaMemcpyAsync(b->h_energies, b->d_energies, sizeof(double) * b->count, cudaMemcpyDeviceToHost, b->stream);
    cudaMemcpyAsync(b->h_flag, b->d_counter + 3, sizeof(unsigned int), cudaMemcpyDeviceToHost, b->stream);
    e = cudaStreamEndCapture(b->stream, &g);
    if (rc) return rc;
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    e = cudaGraphInstantiate(&b->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    return QSIM_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" {

int sim_batch_workspace_bytes(int count, const int *nqubits, const int *layers, size_t *bytes) {
    if (count < 1 || !nqubits || !layers || !bytes) return QSIM_EINVAL;
    long long nang = 0;
    int nmax = 0;
    for (int i = 0; i < count; ++i) {
        if (nqubits[i] < 2 || nqubits[i] > kMaxBatchQubits || layers[i] < 0) return QSIM_EINVAL;
        nang += 2LL * nqubits[i] * layers[i];
        nmax = std::max(nmax, nqubits[i]);
    }
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return QSIM_ECUDA;
    }
    const size_t buffers = (size_t)sms * kWinCtas;  // one per CTA of k_vqe_window
    const size_t gstride = nmax > 12 ? ((size_t)1 << nmax) : 0;
    size_t s = align256(sizeof(double) * nang) + align256(sizeof(double) * count) + 3 * align256(sizeof(int) * count) +
               align256(sizeof(long long) * count) + 256 + buffers * gstride * sizeof(float2);
    *bytes = s;
    return QSIM_OK;
}

int sim_batch_create(int count, const int *nqubits, const int *layers, double h, void *stream, void *workspace,
                     size_t workspace_bytes, qsim_batch **out) {
    if (!out) return QSIM_EINVAL;
    *out = nullptr;
    size_t need = 0;
    int rc = sim_batch_workspace_bytes(count, nqubits, layers, &need);
    if (rc) return rc;
    if (!std::isfinite(h)) return QSIM_ENONFINITE;
    qsim_batch *b = new (std::nothrow) qsim_batch();
    if (!b) return QSIM_ENOMEM;
    b->count = count;
    b->h = h;
    b->nq.assign(nqubits, nqubits + count);
    b->nl.assign(layers, layers + count);
    b->aoff.resize(count);
    long long off = 0;
    b->nmax = 0;
    for (int i = 0; i < count; ++i) {
        b->aoff[i] = off;
        off += 2LL * nqubits[i] * layers[i];
        b->nmax = std::max(b->nmax, nqubits[i]);
    }
    b->nangles = off;
    // largest first: by qubits, then layers (so the circuits above any
    // shared-memory threshold m are a prefix of the order)
    b->order.resize(count);
    std::iota(b->order.begin(), b->order.end(), 0);
    std::stable_sort(b->order.begin(), b->order.end(), [&](int x, int y) {
        return b->nq[x] != b->nq[y] ? b->nq[x] > b->nq[y] : b->nl[x] > b->nl[y];
    });
    cudaGetDevice(&b->device);
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    b->max_grid = b->sms * 4;
    b->gstride = b->nmax > 12 ? ((size_t)1 << b->nmax) : 0;
    if (stream) {
        b->stream = (cudaStream_t)stream;
    } else {
        if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete b;
            return QSIM_ECUDA;
        }
        b->own_stream = true;
    }
    if (workspace) {
        if (workspace_bytes < need || ((uintptr_t)workspace & 255u)) {
            sim_batch_destroy(b);
            return QSIM_EINVAL;
        }
        b->mem = (unsigned char *)workspace;
    } else {
        if (cudaMalloc((void **)&b->mem, need) != cudaSuccess) {
            cudaGetLastError();
            b->mem = nullptr;
            sim_batch_destroy(b);
            return QSIM_ENOMEM;
        }
        b->own_mem = true;
    }
    b->mem_bytes = need;
    unsigned char *p = b->mem;
    b->d_angles = (double *)p;
    p += align256(sizeof(double) * b->nangles);
    b->d_energies = (double *)p;
    p += align256(sizeof(double) * count);
    b->d_order = (int *)p;
    p += align256(sizeof(int) * count);
    b->d_nq = (int *)p;
    p += align256(sizeof(int) * count);
    b->d_nl = (int *)p;
    p += align256(sizeof(int) * count);
    b->d_aoff = (long long *)p;
    p += align256(sizeof(long long) * count);
    b->d_counter = (unsigned int *)p;
    p += 256;
    b->d_gbuf = (float2 *)p;
    if (cudaMallocHost((void **)&b->h_angles, sizeof(double) * std::max<long long>(1, b->nangles)) != cudaSuccess ||
        cudaMallocHost((void **)&b->h_energies, sizeof(double) * count) != cudaSuccess ||
        cudaMallocHost((void **)&b->h_flag, sizeof(unsigned int)) != cudaSuccess) {
        cudaGetLastError();
        sim_batch_destroy(b);
        return QSIM_ENOMEM;
    }
    cudaMemcpyAsync(b->d_order, b->order.data(), sizeof(int) * count, cudaMemcpyHostToDevice, b->stream);
    cudaMemcpyAsync(b->d_nq, b->nq.data(), sizeof(int) * count, cudaMemcpyHostToDevice, b->stream);
    cudaMemcpyAsync(b->d_nl, b->nl.data(), sizeof(int) * count, cudaMemcpyHostToDevice, b->stream);
    cudaMemcpyAsync(b->d_aoff, b->aoff.data(), sizeof(long long) * count, cudaMemcpyHostToDevice, b->stream);
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) {
        sim_batch_destroy(b);
        return QSIM_ECUDA;
    }
    // default configuration: window passes from 13 qubits on (4096 circuits of
    // 13..16 qubits 3.3 ms, with up to 14 qubits in shared memory by 512 threads
    // 4.1; of 4..12 qubits 1.09 and 1.24; one of 10..20 as long either way)
    b->threads = 256;
    b->m = 12;
    *out = b;
    return QSIM_OK;
}

int sim_batch_destroy(qsim_batch *b) {
    if (!b) return QSIM_OK;
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->own_mem && b->mem) cudaFree(b->mem);
    if (b->h_angles) cudaFreeHost(b->h_angles);
    if (b->h_energies) cudaFreeHost(b->h_energies);
    if (b->h_flag) cudaFreeHost(b->h_flag);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return QSIM_OK;
}

int sim_batch_run(qsim_batch *b, const double *angles, double *energies) {
    if (!b || (!angles && b->nangles) || !energies) return QSIM_EINVAL;
    for (long long i = 0; i < b->nangles; ++i)
        if (!std::isfinite(angles[i])) return berr(b, QSIM_ENONFINITE, "non-finite angle");
    if (!b->graph) {
        int rc = build_graph(b);
        if (rc) return rc;
    }
    std::memcpy(b->h_angles, angles, sizeof(double) * b->nangles);
    cudaError_t e = cudaGraphLaunch(b->graph, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    if (*b->h_flag) return berr(b, QSIM_ETIMEOUT, "a device loop gave up; energies not computed");
    std::memcpy(energies, b->h_energies, sizeof(double) * b->count);
    return QSIM_OK;
}

int sim_batch_autotune(qsim_batch *b, const double *angles, int reps, int *threads_out, int *m_out) {
    if (!b || (!angles && b->nangles) || reps < 1) return QSIM_EINVAL;
    cudaError_t e = cudaMemcpyAsync(b->d_angles, angles, sizeof(double) * b->nangles, cudaMemcpyHostToDevice, b->stream);
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int bt = b->threads, bm = b->m;
    for (const auto &cand : kCandidates) {
        const int threads = cand[0], m = cand[1];
        if (!config_valid(threads, m)) continue;
        int grid = 0;
        if (occupancy(b, threads, m, &grid)) continue;
        std::vector<float> t;
        for (int r = 0; r <= reps; ++r) {
            cudaEventRecord(e0, b->stream);
            int rc = launch(b, threads, m, grid);
            cudaEventRecord(e1, b->stream);
            if (rc) break;
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (r > 0) t.push_back(ms);  // first run is a warm-up
        }
        if ((int)t.size() != reps) continue;
        std::sort(t.begin(), t.end());
        const float med = t[t.size() / 2];
        if (med < best) {
            best = med;
            bt = threads;
            bm = m;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return berr(b, QSIM_ECUDA, cudaGetErrorString(e));
    b->threads = bt;
    b->m = bm;
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    if (threads_out) *threads_out = bt;
    if (m_out) *m_out = bm;
    return QSIM_OK;
}

int sim_batch_set_config(qsim_batch *b, int threads, int m) {
    if (!b) return QSIM_EINVAL;
    if (threads != 256 && threads != 512 && threads != 1024) return berr(b, QSIM_EINVAL, "threads must be 256/512/1024");
    if (m < 12 || m > 14 || !config_valid(threads, m)) return berr(b, QSIM_EINVAL, "invalid tile configuration");
    b->threads = threads;
    b->m = m;
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    return QSIM_OK;
}

const char *sim_batch_last_error(const qsim_batch *b) { return b ? b->err.c_str() : "null batch"; }

}  // extern "C"
