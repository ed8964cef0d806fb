// diag_kernels.cu -- a block of diagonal gates applied in one pass.
//
// Gates whose matrices are diagonal (Z, S, T, R(phi), RZ, CZ, controlled
// phases, multi-controlled Z) only multiply each amplitude by a phase that
// depends on the bits of its index on the gate's qubits, and they commute
// with one another.  A run of them over a qubit set S (|S| <= 12) is one
// table d of 2^|S| factors (the product of the gates' diagonal entries for
// every assignment of S, in FP64), and the pass is
//     psi_i <- d[bits of i on S] * psi_i.
// The phase ladders of the QFT (ProjectQ paper, Sec. 3: the constant adder
// is QFT, phase shifts, inverse QFT) and the controlled z-rotation chain of
// the simulator benchmark (Sec. 4.3.2, Fig. 7) are made of such gates.
//
// Diagonal blocks that follow one another in a plan (a QFT's phases from one
// group of qubits onto each of the others) are applied in one pass, up to
// kMaxDiagRun of them: the pass reads and writes the state once and
// multiplies each amplitude by one entry of each table, in order, the same
// products a pass per table rounds.  The 30-qubit QFT's ten diagonal blocks
// come in runs of 4, 3, 2 and 1: 14 passes instead of 20, 38.3 against
// 54.8 ms, each at 97 % of HBM.
//
// The tables are built on the device (k_build_diag, an entry per thread, its
// gates' factors multiplied in FP64 and rounded once) and copied to shared
// memory per CTA, with one gather table of 5 x 256 entries: entry [c][v]
// holds for every table the byte offset that bits 8c.. of an index equal to v
// contribute, 16 bits each, so two reads give an amplitude's place in all
// tables.  A CTA takes contiguous chunks of up to 2^16 amplitudes, so the
// offsets of index bits 16 and above are gathered once per chunk; each
// thread handles 16 bytes of amplitudes per access (two complex64 or one
// complex128), eight accesses in flight.
// complex128 uses FP64 products, or double-float products when the handle
// runs complex128 gates in double-float arithmetic.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "df128.cuh"
#include "internal.h"

using namespace qsim_dev;

namespace {

struct DiagMasks {
    uint64_t m[kMaxDiagRun];  // qubits of each table
    const unsigned char *tab[kMaxDiagRun];
};

// threads per CTA: one table leaves room for several CTAs per SM, the tables
// of a run for one to three
template <int NT> __host__ __device__ constexpr int diag_threads() { return NT == 1 ? 256 : 512; }

template <typename Amp, int NT>
__global__ void __launch_bounds__(diag_threads<NT>()) k_diag_block(Amp *__restrict__ psi, uint64_t nchunks, int cb,
                                                                  const DiagMasks M, int use_df) {
    constexpr int T = diag_threads<NT>();
    extern __shared__ __align__(16) unsigned char sm_raw[];
    // the gather table, then the tables
    unsigned long long *gather = (unsigned long long *)sm_raw;  // [5][256]
    unsigned char *tab[NT];
    {
        unsigned char *at = sm_raw + 5 * 256 * sizeof(unsigned long long);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            tab[t] = at;
            const int units = (int)((sizeof(Amp) << __popcll(M.m[t])) / 16);
            const float4 *src = (const float4 *)M.tab[t];
#pragma unroll 4
            for (int i = threadIdx.x; i < units; i += T) ((float4 *)at)[i] = src[i];
            at += sizeof(Amp) << __popcll(M.m[t]);
        }
    }
    for (int e = threadIdx.x; e < 5 * 256; e += T) {
        const int c = e >> 8;
        unsigned long long r = 0;
#pragma unroll
        for (int t = 0; t < NT; ++t)
            for (int bit = 0; bit < 8; ++bit) {
                const uint64_t b = 1ull << (8 * c + bit);
                if (((e >> bit) & 1) && (M.m[t] & b))
                    r |= (unsigned long long)(sizeof(Amp) << __popcll(M.m[t] & (b - 1ull))) << (16 * t);
            }
        gather[e] = r;
    }
    __syncthreads();
    constexpr int kU = 8;                      // 16-byte accesses in flight per thread
    constexpr int kPer = 16 / sizeof(Amp);     // amplitudes per access
    const unsigned units = (1u << cb) / kPer;  // accesses per chunk
    const unsigned long long bit0 = gather[1];
    for (uint64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const uint64_t base = ch << cb;
        // offsets of index bits 16.. (constant over the chunk, cb <= 16)
        const unsigned long long hi =
            gather[512 + ((base >> 16) & 255)] | gather[768 + ((base >> 24) & 255)] | gather[1024 + ((base >> 32) & 255)];
        const unsigned lo0 = (unsigned)(base & 0xFFFFu);
        float4 *p4 = (float4 *)(psi + base);
        for (unsigned u0 = threadIdx.x; u0 < units; u0 += kU * T) {
            float4 v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (u0 + u * T < units) v[u] = p4[u0 + u * T];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const unsigned idx = u0 + u * T;
                if (idx >= units) continue;
                const unsigned lo = lo0 | (idx * kPer);
                const unsigned long long off = gather[lo & 255] | gather[256 + (lo >> 8)] | hi;
                if constexpr (sizeof(Amp) == 8) {
                    float2 a = make_float2(v[u].x, v[u].y), b = make_float2(v[u].z, v[u].w);
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        const unsigned o = (unsigned)(off >> (16 * t)) & 0xFFFFu;
                        // the second amplitude adds the offset of index bit 0
                        const unsigned o1 = o | ((unsigned)(bit0 >> (16 * t)) & 0xFFFFu);
                        a = cmul(*(const float2 *)(tab[t] + o), a);
                        b = cmul(*(const float2 *)(tab[t] + o1), b);
                    }
                    p4[idx] = make_float4(a.x, a.y, b.x, b.y);
                } else {
                    double2 a = *(const double2 *)&v[u];
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        const double2 z = *(const double2 *)(tab[t] + ((unsigned)(off >> (16 * t)) & 0xFFFFu));
                        a = use_df ? qsim_df::to_double(qsim_df::cmul(qsim_df::split(z), qsim_df::split(a))) : cmul(z, a);
                    }
                    p4[idx] = *(const float4 *)&a;
                }
            }
        }
    }
}

// Tables of several diagonal blocks (blockIdx.y): entry r is the product, in
// the order of the gates, of their diagonal entries for the assignment r of
// the block's qubits, controls that are not all 1 leaving it alone.  (On the
// host a 12-qubit table of 36 gates took 250 us.)
struct DiagGate {
    uint32_t cmask;    // controls, block-local bits
    uint16_t t, off;   // targets; its 2^t entries at off (in entries) after the gates
    uint8_t tpos[8];
};
static_assert(sizeof(DiagGate) == 16, "records are made of 16-byte units");
struct DiagJob {
    unsigned char *out;
    const unsigned char *rec;
    uint32_t ngates, k;
    uint32_t pad[2];
};
static_assert(sizeof(DiagJob) == 32, "records are made of 16-byte units");

__device__ __forceinline__ void store_amp(double2 *p, double2 z) { *p = z; }
__device__ __forceinline__ void store_amp(float2 *p, double2 z) { *p = make_float2((float)z.x, (float)z.y); }

template <typename Amp>
__global__ void __launch_bounds__(128) k_build_diag(const DiagJob *__restrict__ jobs) {
    const DiagJob J = jobs[blockIdx.y];
    const uint32_t r = blockIdx.x * 128u + threadIdx.x;
    if (r >> J.k) return;
    const DiagGate *gates = (const DiagGate *)J.rec;
    const double2 *ent = (const double2 *)(gates + J.ngates);
    double2 d = make_double2(1.0, 0.0);
    for (uint32_t g = 0; g < J.ngates; ++g) {
        const DiagGate G = gates[g];
        if ((r & G.cmask) != G.cmask) continue;
        uint32_t ti = 0;
        for (int j = 0; j < G.t; ++j) ti |= ((r >> G.tpos[j]) & 1u) << j;
        d = cmul(d, ent[G.off + ti]);
    }
    store_amp((Amp *)J.out + r, d);
}

template <typename Amp, int NT>
int diag_launch(qsim *s, const DiagMasks &M) {
    size_t smem = 5 * 256 * sizeof(unsigned long long);
    for (int t = 0; t < NT; ++t) smem += sizeof(Amp) << __builtin_popcountll(M.m[t]);
    static bool attr[64] = {false};
    if (s->device < 0 || s->device >= 64 || !attr[s->device]) {
        const cudaError_t e = cudaFuncSetAttribute(
            k_diag_block<Amp, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
            (int)(NT * (sizeof(Amp) << kMaxDiagQubits) + 5 * 256 * sizeof(unsigned long long)));
        if (e != cudaSuccess) return cuda_err(s, e, "diagonal kernel attribute");
        if (s->device >= 0 && s->device < 64) attr[s->device] = true;
    }
    // contiguous chunks of 2^cb amplitudes (cb <= 16), at least about four
    // per SM where the register allows
    const int n = s->n;
    const int cb = std::max(std::min(n, 9), std::min(16, n - 10));
    const uint64_t nchunks = 1ull << (n - cb);
    const uint64_t grid = std::min<uint64_t>(nchunks, (uint64_t)s->sms * (NT == 1 ? 8 : 2));
    k_diag_block<Amp, NT><<<(unsigned)grid, diag_threads<NT>(), smem, s->stream>>>((Amp *)s->state, nchunks, cb, M,
                                                                                   s->c128_df ? 1 : 0);
    s->stats.launches++;
    return cuda_err(s, cudaGetLastError(), "diagonal block launch");
}

template <typename Amp>
int diag_run(qsim *s, const DiagMasks &M, int count) {
    switch (count) {
    case 1: return diag_launch<Amp, 1>(s, M);
    case 2: return diag_launch<Amp, 2>(s, M);
    case 3: return diag_launch<Amp, 3>(s, M);
    default: break;
    }
    if constexpr (sizeof(Amp) == 8) return diag_launch<Amp, 4>(s, M);
    return set_err(s, QSIM_EINVAL, "diagonal run too long");
}

}  // namespace

// complex128 tables of 12 qubits are 64 KB: three fit an SM's shared memory
int diag_run_limit(const qsim *s) { return s->prec == QSIM_C128 ? 3 : kMaxDiagRun; }

int build_diag_tables(qsim *s, PlanItem *const *items, int count) {
    if (count < 1) return QSIM_OK;
    const size_t amp = amp_bytes(s);
    std::vector<unsigned char> rec(sizeof(DiagJob) * count);
    std::vector<size_t> at(count), image(count);
    size_t images = 0;
    int kmax = 1;
    for (int i = 0; i < count; ++i) {
        const PlanItem &it = *items[i];
        const int k = __builtin_popcountll(it.dmask);
        if (s->n < 2) return set_err(s, QSIM_ENOTSUP, "diagonal block needs n >= 2");
        if (k < 1 || k > kMaxDiagQubits) return set_err(s, QSIM_EINVAL, "diagonal block width");
        auto bit = [&](int qubit) { return __builtin_popcountll(it.dmask & ((1ull << qubit) - 1ull)); };
        std::vector<DiagGate> gates;
        std::vector<cd> ent;
        auto add = [&](const GateRec &g) {
            DiagGate d{};
            d.t = (uint16_t)g.t;
            d.off = (uint16_t)ent.size();
            for (int c : g.controls) d.cmask |= 1u << bit(c);
            for (int j = 0; j < g.t; ++j) d.tpos[j] = (uint8_t)bit(g.targets[j]);
            const int T = 1 << g.t;
            for (int e = 0; e < T; ++e) ent.push_back(g.m[(size_t)e * T + e]);
            gates.push_back(d);
        };
        bool fits = true;  // 16-bit offsets, records of at most kDiagRecordBytes
        for (size_t m = 0; m < it.members.size() && fits; ++m) {
            add(s->queue[it.members[m]]);
            fits = sizeof(DiagGate) * gates.size() + sizeof(cd) * ent.size() <= kDiagRecordBytes;
        }
        if (!fits) {
            // more gates than a record holds: the table from the host
            PlanItem whole = it;
            block_matrix(s->queue, whole);
            image[i] = images;
            images += (std::max<size_t>(amp << k, 16) + 255) & ~(size_t)255;
            at[i] = SIZE_MAX;
            items[i]->dtab = std::move(whole.dtab);
            continue;
        }
        DiagJob job{};
        job.ngates = (uint32_t)gates.size();
        job.k = (uint32_t)k;
        at[i] = rec.size();
        std::memcpy(&rec[sizeof(DiagJob) * i], &job, sizeof(job));
        rec.resize(at[i] + sizeof(DiagGate) * gates.size() + sizeof(cd) * ent.size());
        std::memcpy(&rec[at[i]], gates.data(), sizeof(DiagGate) * gates.size());
        std::memcpy(&rec[at[i] + sizeof(DiagGate) * gates.size()], (const void *)ent.data(), sizeof(cd) * ent.size());
        image[i] = images;
        images += (std::max<size_t>(amp << k, 16) + 255) & ~(size_t)255;
        kmax = std::max(kmax, k);
    }
    unsigned char *out = nullptr;
    int rc = ring_reserve(s, images + rec.size(), &out);  // both in one piece of the ring
    if (rc) return rc;
    unsigned char *dev = out + images;
    for (int i = 0; i < count; ++i) {
        items[i]->operand = out + image[i];
        DiagJob *job = (DiagJob *)&rec[sizeof(DiagJob) * i];
        job->out = out + image[i];
        job->rec = dev + (at[i] == SIZE_MAX ? 0 : at[i]);
    }
    if ((rc = stage_to(s, dev, rec.data(), rec.size()))) return rc;
    const dim3 grid((1u << kmax) > 128 ? (1u << kmax) / 128 : 1, (unsigned)count);
    if (s->prec == QSIM_C128)
        k_build_diag<double2><<<grid, 128, 0, s->stream>>>((const DiagJob *)dev);
    else
        k_build_diag<float2><<<grid, 128, 0, s->stream>>>((const DiagJob *)dev);
    s->stats.launches++;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_err(s, e, "diagonal table launch");
    // the host's tables, rounded to the amplitude type (their jobs have no
    // gates and k = 0: they wrote entry 0, before this copy)
    for (int i = 0; i < count && !rc; ++i) {
        if (at[i] != SIZE_MAX) continue;
        const std::vector<cd> &d = items[i]->dtab;
        if (s->prec == QSIM_C128) {
            rc = stage_to(s, items[i]->operand, d.data(), sizeof(cd) * d.size());
        } else {
            std::vector<float2> f(d.size());
            for (size_t j = 0; j < d.size(); ++j) f[j] = make_float2((float)d[j].real(), (float)d[j].imag());
            rc = stage_to(s, items[i]->operand, f.data(), sizeof(float2) * f.size());
        }
    }
    return rc;
}

int launch_block_diag(qsim *s, PlanItem *const *items, int count) {
    if (count < 1 || count > diag_run_limit(s)) return set_err(s, QSIM_EINVAL, "diagonal run too long");
    DiagMasks M{};
    for (int i = 0; i < count; ++i) {
        M.m[i] = items[i]->dmask;
        M.tab[i] = items[i]->operand;
    }
    return s->prec == QSIM_C128 ? diag_run<double2>(s, M, count) : diag_run<float2>(s, M, count);
}
