// small_kernel.cu -- a queue of plain gates on a small register, executed one
// after the other in one launch.
//
// The simulator's per-gate sweep (ProjectQ paper, Sec. 4.3.2) over a register
// of a few thousand amplitudes is bound by the launch, not by the sweep: at
// 12 qubits a gate is 64 KB of complex128 amplitudes, and a launch with its
// gap took 3 to 8 us.  Here a cluster of 16 CTAs holds the register in its
// shared memory (the top 4 qubits are the CTA's rank) and applies the queued
// gates in order, each with the arithmetic of its plain kernel
// (gate_kernels.cu), so the results are the same bits:
//   - a one-qubit gate on a qubit below the rank bits pairs amplitudes of the
//     same CTA: in place, one block barrier;
//   - a gate on a rank qubit, or on several qubits: every CTA forms its own
//     outputs from the others' amplitudes, read through distributed shared
//     memory, into its second buffer; one cluster barrier before.  A CTA
//     writes the buffer that others may still be reading only after the next
//     such barrier, which they reach when they have read.
// Registers of up to 8 qubits take one CTA.  complex128 runs up to 13 qubits:
// a dense gate costs 8 FP64 FMAs an amplitude, 0.5 us for 12 qubits on 16 SMs
// at two a cycle, so larger registers are better off with all SMs
// (12 qubits, 350 gates: 0.33 ms against 2.46 ms launched one by one);
// complex64 up to 16.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstring>
#include <vector>

#include "common.cuh"
#include "fx128.cuh"
#include "internal.h"

using namespace qsim_dev;
namespace cgrp = cooperative_groups;

namespace {

constexpr int kSmallThreads = 128;
constexpr int kSmallRankBits = 4;
constexpr int kSmallOneCta = 8;           // registers of up to this many qubits take one CTA
constexpr uint32_t kSmallRecord = 81920;  // bytes of gates and matrices per launch

struct SmallGate {
    uint32_t cmask, tmask;  // controls and targets
    uint32_t off;           // its matrix (4^t, or the entries a diagonal kind needs), bytes from the record's start
    uint8_t kind, t;        // GateKind, targets
    uint8_t tpos[6];        // target j <-> qubit tpos[j]
    uint32_t fx;            // its matrix is a qsim_fx::MatFx
    uint32_t pad[2];
};
static_assert(sizeof(SmallGate) == 32, "records are made of 16-byte units");

template <typename Amp, int RB>
__global__ void __launch_bounds__(kSmallThreads) k_small(Amp *__restrict__ psi, int n,
                                                         const unsigned char *__restrict__ rec, int ngates,
                                                         uint32_t rec_bytes) {
    extern __shared__ __align__(16) unsigned char sms[];
    const int nl = n - RB;               // qubits below the rank bits
    const uint32_t L = 1u << nl;         // amplitudes of this CTA
    Amp *buf[2] = {(Amp *)sms, (Amp *)sms + L};
    unsigned char *r = sms + 2 * sizeof(Amp) * (size_t)L;
    const uint32_t tid = threadIdx.x, rank = RB ? blockIdx.x : 0u;
    for (uint32_t i = tid; i < rec_bytes / 16; i += kSmallThreads) ((float4 *)r)[i] = ((const float4 *)rec)[i];
    Amp *x = buf[0], *other = buf[1];
    for (uint32_t i = tid; i < L; i += kSmallThreads) x[i] = psi[((uint64_t)rank << nl) | i];
    __syncthreads();
    const uint32_t base = rank << nl;    // register index of this CTA's amplitude 0
    for (int g = 0; g < ngates; ++g) {
        const SmallGate G = ((const SmallGate *)r)[g];
        const Amp *m = (const Amp *)(r + G.off);
        if (G.kind == GK_PHASE) {
            const uint32_t mask = G.cmask | G.tmask;
            for (uint32_t i = tid; i < L; i += kSmallThreads)
                if (((base | i) & mask) == mask) x[i] = cmul(m[0], x[i]);
            __syncthreads();
        } else if (G.kind == GK_DIAG1) {
            for (uint32_t i = tid; i < L; i += kSmallThreads)
                if (((base | i) & G.cmask) == G.cmask) x[i] = cmul(m[((base | i) & G.tmask) ? 1 : 0], x[i]);
            __syncthreads();
        } else if (G.t == 1 && G.tpos[0] < nl) {
            const int b = G.tpos[0];
            for (uint32_t p = tid; p < L / 2; p += kSmallThreads) {
                const uint32_t i0 = ((p >> b) << (b + 1)) | (p & ((1u << b) - 1u)), i1 = i0 | (1u << b);
                if (((base | i0) & G.cmask) != G.cmask) continue;
                const Amp v0 = x[i0], v1 = x[i1];
                if (G.kind == GK_X) {
                    x[i0] = v1;
                    x[i1] = v0;
                    continue;
                }
                if constexpr (sizeof(Amp) == 16) {
                    if (G.fx) {
                        const qsim_fx::MatFx &F = *(const qsim_fx::MatFx *)m;
                        if (F.apart)
                            qsim_fx::dense1<true>(F, v0, v1, x[i0], x[i1]);
                        else
                            qsim_fx::dense1<false>(F, v0, v1, x[i0], x[i1]);
                        continue;
                    }
                }
                {
                    x[i0] = cfma(m[1], v1, cmul(m[0], v0));
                    x[i1] = cfma(m[3], v1, cmul(m[2], v0));
                }
            }
            __syncthreads();
        } else {
            // outputs from amplitudes of any CTA, into the other buffer
            if (RB)
                cgrp::this_cluster().sync();
            else
                __syncthreads();
            auto at = [&](uint32_t i) {  // amplitude i of the register
                const uint32_t owner = i >> nl;
                const Amp *p = RB && owner != rank ? cgrp::this_cluster().map_shared_rank(x, owner) : x;
                return p[i & (L - 1u)];
            };
            for (uint32_t i = tid; i < L; i += kSmallThreads) {
                const uint32_t gi = base | i;
                Amp y = x[i];
                if ((gi & G.cmask) == G.cmask) {
                    if (G.kind == GK_X) {
                        y = at(gi ^ G.tmask);
                    } else if (sizeof(Amp) == 16 && G.fx) {
                        if constexpr (sizeof(Amp) == 16)
                            y = qsim_fx::dense1_row(*(const qsim_fx::MatFx *)m, (gi & G.tmask) ? 1 : 0,
                                                    at(gi & ~G.tmask), at(gi | G.tmask));
                    } else {
                        const uint32_t rest = gi & ~G.tmask;
                        const int T = 1 << G.t;
                        uint32_t row = 0;
                        for (int j = 0; j < G.t; ++j) row |= ((gi >> G.tpos[j]) & 1u) << j;
                        y = cmul(m[row * T], at(rest));
                        for (int k = 1; k < T; ++k) {
                            uint32_t s = rest;
                            for (int j = 0; j < G.t; ++j) s |= (uint32_t)((k >> j) & 1) << G.tpos[j];
                            y = cfma(m[row * T + k], at(s), y);
                        }
                    }
                }
                other[i] = y;
            }
            Amp *swap = x;
            x = other;
            other = swap;
            __syncthreads();
        }
    }
    for (uint32_t i = tid; i < L; i += kSmallThreads) psi[((uint64_t)rank << nl) | i] = x[i];
    if (RB) cgrp::this_cluster().sync();  // no CTA ends while another reads its amplitudes
}

inline void put(double2 *d, cd z) { *d = make_double2(z.real(), z.imag()); }
inline void put(float2 *d, cd z) { *d = make_float2((float)z.real(), (float)z.imag()); }

// QSIM_ENOTSUP: nothing was launched (the caller runs the gates one by one)
template <typename Amp, int RB>
int launch_small(qsim *s, const unsigned char *dev, int ngates, uint32_t rec_bytes) {
    static signed char usable[64] = {0};  // per device: 1 yes, -1 no
    // at most 2 x 2^9 complex128 or 2 x 2^12 complex64 amplitudes, or those of kSmallOneCta qubits
    constexpr int kMaxSmem = (int)(2 * (sizeof(Amp) == 16 ? 8192 : 32768) + kSmallRecord);
    if (s->device < 0 || s->device >= 64) return QSIM_ENOTSUP;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << RB);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = kMaxSmem;
    cfg.stream = s->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << RB;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = RB ? 1 : 0;
    if (!usable[s->device]) {
        cudaError_t e =
            cudaFuncSetAttribute(k_small<Amp, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        // a cluster of 16 needs a GPC with as many free SMs
        if (e == cudaSuccess && RB)
            e = cudaFuncSetAttribute(k_small<Amp, RB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        int clusters = 1;
        if (e == cudaSuccess && RB) e = cudaOccupancyMaxActiveClusters(&clusters, k_small<Amp, RB>, &cfg);
        if (e != cudaSuccess) cudaGetLastError();
        usable[s->device] = e == cudaSuccess && clusters > 0 ? 1 : -1;
    }
    if (usable[s->device] < 0) return QSIM_ENOTSUP;
    cfg.dynamicSmemBytes = 2 * (sizeof(Amp) << (s->n - RB)) + rec_bytes;
    if (cudaLaunchKernelEx(&cfg, k_small<Amp, RB>, (Amp *)s->state, s->n, dev, ngates, rec_bytes) != cudaSuccess) {
        cudaGetLastError();
        return QSIM_ENOTSUP;
    }
    s->stats.launches++;
    return QSIM_OK;
}

// Gates [*done, end) of the queue.
template <typename Amp>
int small_queue(qsim *s, size_t end, size_t *done) {
    const std::vector<GateRec> &q = s->queue;
    std::vector<unsigned char> mats;
    std::vector<SmallGate> gates;
    for (size_t i = *done; i < end;) {
        gates.clear();
        mats.clear();
        for (; i < end; ++i) {
            const GateRec &g = q[i];
            const size_t T = (size_t)1 << g.t;
            const size_t count = g.kind == GK_X ? 0 : g.kind == GK_PHASE ? 1 : g.kind == GK_DIAG1 ? 2 : T * T;
            qsim_fx::MatFx fx;
            const bool use_fx =
                sizeof(Amp) == 16 && g.t == 1 && g.kind == GK_DENSE && qsim_fx::make_fx(g.m.data(), fx);
            const size_t mb = ((use_fx ? sizeof(fx) : count * sizeof(Amp)) + 15) & ~(size_t)15;
            if (sizeof(SmallGate) * (gates.size() + 1) + mats.size() + mb > kSmallRecord) break;
            SmallGate r{};
            r.cmask = (uint32_t)g.cmask;
            r.tmask = (uint32_t)g.tmask;
            r.off = (uint32_t)mats.size();
            r.kind = (uint8_t)g.kind;
            r.t = (uint8_t)g.t;
            for (int j = 0; j < g.t; ++j) r.tpos[j] = (uint8_t)g.targets[j];
            gates.push_back(r);
            mats.resize(mats.size() + mb);
            Amp *d = (Amp *)(mats.data() + r.off);
            if (use_fx) {
                gates.back().fx = 1;
                std::memcpy((void *)d, &fx, sizeof(fx));
            } else if (g.kind == GK_PHASE) {
                put(d, g.m[3]);
            } else if (g.kind == GK_DIAG1) {
                put(d, g.m[0]);
                put(d + 1, g.m[3]);
            } else {
                for (size_t e = 0; e < count; ++e) put(d + e, g.m[e]);
            }
        }
        const size_t head = sizeof(SmallGate) * gates.size();
        for (SmallGate &g : gates) g.off += (uint32_t)head;
        std::vector<unsigned char> rec(head + mats.size());
        std::memcpy(rec.data(), gates.data(), head);
        std::memcpy(rec.data() + head, mats.data(), mats.size());
        unsigned char *dev = nullptr;
        int rc = stage_operand(s, rec.data(), rec.size(), &dev);
        if (rc) return rc;
        rc = s->n <= kSmallOneCta ? launch_small<Amp, 0>(s, dev, (int)gates.size(), (uint32_t)rec.size())
                                  : launch_small<Amp, kSmallRankBits>(s, dev, (int)gates.size(), (uint32_t)rec.size());
        if (rc) return rc;
        *done = i;
    }
    return QSIM_OK;
}

}  // namespace

bool small_queue_ok(const qsim *s) {
    if (s->fusion != QSIM_FUSE_NONE || s->profiling || s->c128_df || s->queue.size() < (size_t)kSmallMinRun ||
        s->n > (s->prec == QSIM_C128 ? 13 : 16))
        return false;
    // in a stream capture gates are launched one by one, their matrices in the
    // launches: the graph would copy the record again at each replay, from a
    // staging buffer that later calls write to
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s->stream, &st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return st == cudaStreamCaptureStatusNone;
}

// Where a gate's outputs come from amplitudes of other CTAs, 16 SMs read 2^t of
// them each; a launch of its own has the whole chip.  complex64, us a gate here
// and launched: 2 targets 4.2 of 13 qubits, 6.9 of 14 (4.4 launched); 3 targets
// 4.4 of 12 (4.4); 4 targets 6.2 of 8 (4.6); a dense gate on a rank qubit 4.4 of
// 14, 7.6 of 15 (4.4); X there 3.3 of 15, 5.5 of 16 (4.4).  complex128 is bound
// by FP64 either way: 2 to 5 targets of 13 qubits 6.2, 11.5, 22, 47 (6.5, 12.7,
// 42, 156).
size_t small_run(const qsim *s, size_t begin) {
    auto pays = [s](const GateRec &g) {
        if (s->prec == QSIM_C128 || g.kind == GK_PHASE || g.kind == GK_DIAG1) return true;
        if (g.t == 1 && (s->n <= kSmallOneCta || g.targets[0] < s->n - kSmallRankBits)) return true;
        if (g.kind == GK_X) return s->n <= 15;
        return s->n <= (g.t == 1 ? 14 : g.t == 2 ? 13 : g.t == 3 ? 12 : 0);
    };
    size_t i = begin;
    while (i < s->queue.size() && pays(s->queue[i])) ++i;
    return i;
}

int launch_small_queue(qsim *s, size_t begin, size_t end, size_t *done) {
    *done = begin;
    return s->prec == QSIM_C128 ? small_queue<double2>(s, end, done) : small_queue<float2>(s, end, done);
}
