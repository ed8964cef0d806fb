// vqe_window.cuh -- the window passes of the batched variational kernel: which
// gates a pass over a circuit's state can apply, and how its tile holds them.
//
// A layer of the ansatz rotates every qubit (RY then RZ) and then runs the
// ladder CNOT(q -> q+1), q ascending.  A gate needs only the earlier gates on
// its own wires, so a pass whose tile holds the qubits of a window need not
// stop at the end of a layer: on a window [w, w + k) it goes on, layer after
// layer, on the part of the window that the neighbours outside do not hold
// back (one qubit less per layer at the upper edge).  The next pass takes the
// window from the lowest qubit with a gate ready.  From |0...0> the first pass
// touches one tile, and each pass doubles the touched part of the state by no
// more than its window's reach, so most of the work happens on a small part
// of it: 20 qubits and 8 layers take four passes over 2^13, 2^16, 2^19 and 2^20
// amplitudes, where a pass per half layer took sixteen over 2^20.
//
// Inside a tile nothing is moved for a CNOT: the tile's logical index is y =
// A p ^ f of the position p, A a bit matrix (rows a_k, unit lower triangular:
// controls lie below targets), f the bits flipped by the X of the rotations
// (vqe_kernel.cu).  A rotation of logical bit k pairs p and p ^ m_k, m_k the
// k-th column of the inverse; CNOT(k -> k') adds row k to row k' and column
// k' of the inverse to column k.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define VQE_HD __host__ __device__
#else
#define VQE_HD
#endif

namespace qsim_vqe {

constexpr int kTileBits = 13;      // 2^13 amplitudes, 64 KB
constexpr int kRunBits = 2;        // the lowest qubits below a window: runs of 32 bytes
constexpr int kWindow = kTileBits - kRunBits;
constexpr int kMaxQ = 26;
constexpr int kMaxSteps = 8;       // rotation steps per pass
constexpr int kGroupBits = 5;      // rotations applied at a time, on 32 amplitudes in registers
constexpr int kMaxGroups = kMaxSteps * 3;

VQE_HD inline int parity32(uint32_t x) {
#ifdef __CUDA_ARCH__
    return __popc(x) & 1;
#else
    return __builtin_popcount(x) & 1;
#endif
}

// Progress of a circuit: layers whose rotation on q, whose CNOT(q, q + 1) are done.
struct Progress {
    int n, L;
    int rot[kMaxQ], cn[kMaxQ];
};

VQE_HD inline void progress_start(Progress &s, int n, int L) {
    s.n = n;
    s.L = L;
    for (int q = 0; q < n; ++q) s.rot[q] = s.cn[q] = 0;
}
VQE_HD inline bool rot_ready(const Progress &s, int q) {
    const int l = s.rot[q];
    return l < s.L && (q == 0 || s.cn[q - 1] >= l) && (q == s.n - 1 || s.cn[q] >= l);
}
VQE_HD inline bool cn_ready(const Progress &s, int q) {
    const int l = s.cn[q];
    return l < s.L && s.rot[q] > l && s.rot[q + 1] > l && (q == 0 || s.cn[q - 1] > l);
}

// the lowest qubit with a gate that can run now, n if none is left (the
// earliest gate still to come always can)
VQE_HD inline int lowest_ready(const Progress &s) {
    for (int q = 0; q < s.n; ++q)
        if (rot_ready(s, q) || (q < s.n - 1 && cn_ready(s, q))) return q;
    return s.n;
}

// A tile's qubits: tile bit b is qubit b for b < kRunBits, and w + b - kRunBits
// above; w = kRunBits is the contiguous tile of the lowest qubits.
VQE_HD inline int window_start(const Progress &s) {
    const int q = lowest_ready(s), top = s.n - kWindow;
    const int w = q < top ? q : top;
    return w <= kRunBits ? kRunBits : w;
}

// Rotations of a step in groups of up to kGroupBits: masks m (columns of the
// inverse), tile bits q; `cnt` of them rotate, the others complete the group.
// Group member start index gi (8 bits) -> position | logical index << 16, as
// the XOR of lane[gi & 31] and hi[gi >> 5]: a set of 256 positions that with all
// sums of the masks makes up the tile, its first four bits (the lanes of a
// half-warp) on 16 different banks (bits 0..3 of the position).
struct Group {
    uint32_t m[kGroupBits];
    int q[kGroupBits];
    int cnt;
    uint32_t lane[32], hi[8];
};

struct Map {  // y = A p ^ f on tile bits
    uint32_t row[kTileBits], inv[kTileBits], f;
};
VQE_HD inline void map_identity(Map &a) {
    for (int k = 0; k < kTileBits; ++k) a.row[k] = a.inv[k] = 1u << k;
    a.f = 0;
}
// CNOT on tile bits c -> t
VQE_HD inline void map_cnot(Map &a, int c, int t) {
    a.row[t] ^= a.row[c];
    a.inv[c] ^= a.inv[t];
    a.f ^= ((a.f >> c) & 1u) << t;
}
VQE_HD inline uint32_t map_logical(const Map &a, uint32_t p) {
    uint32_t y = a.f;
    for (int k = 0; k < kTileBits; ++k) y ^= (uint32_t)parity32(a.row[k] & p) << k;
    return y;
}
VQE_HD inline uint32_t map_position(const Map &a, uint32_t y) {
    y ^= a.f;
    uint32_t p = 0;
    for (int k = 0; k < kTileBits; ++k)
        if ((y >> k) & 1u) p ^= a.inv[k];
    return p;
}

// The group of the tile bits q[0..cnt) (cnt >= 1).
VQE_HD inline void make_group(const Map &a, const int *q, int cnt, Group &g) {
    uint32_t used = 0;
    for (int j = 0; j < cnt; ++j) {
        g.q[j] = q[j];
        used |= 1u << q[j];
    }
    // complete it from the top, away from the bank bits
    for (int j = cnt, b = kTileBits - 1; j < kGroupBits; --b)
        if (!((used >> b) & 1u)) {
            g.q[j++] = b;
            used |= 1u << b;
        }
    g.cnt = cnt;
    for (int j = 0; j < kGroupBits; ++j) g.m[j] = a.inv[g.q[j]];
    // echelon form of the masks, pivots as high as they go
    uint32_t v[kGroupBits], piv = 0;
    int pb[kGroupBits];
    for (int j = 0; j < kGroupBits; ++j) v[j] = g.m[j];
    for (int j = 0; j < kGroupBits; ++j) {
        int b = kTileBits - 1, src = -1;
        for (; src < 0; --b)
            for (int i = j; i < kGroupBits; ++i)
                if ((v[i] >> b) & 1u) {
                    src = i;
                    break;
                }
        ++b;
        const uint32_t t = v[j];
        v[j] = v[src];
        v[src] = t;
        for (int i = 0; i < kGroupBits; ++i)
            if (i != j && ((v[i] >> b) & 1u)) v[i] ^= v[j];
        pb[j] = b;
        piv |= 1u << b;
    }
    // complement: the unit vectors of the other bits, the bank bits first; a
    // bank bit that is a pivot is brought in by adding its vector to one of
    // the others'
    uint32_t basis[kTileBits - kGroupBits], rest[kTileBits];
    int nb = 0, nr = 0, lost = 0;
    for (int b = 0; b < kTileBits; ++b) {
        if ((piv >> b) & 1u) continue;
        if (b < 4)
            basis[nb++] = 1u << b;
        else
            rest[nr++] = 1u << b;
    }
    for (int j = 0; j < kGroupBits; ++j)
        if (pb[j] < 4) basis[nb++] = rest[lost++] ^ v[j];
    while (nb < kTileBits - kGroupBits) basis[nb++] = rest[lost++];
    uint32_t yb[kTileBits - kGroupBits];
    for (int i = 0; i < kTileBits - kGroupBits; ++i) yb[i] = map_logical(a, basis[i]) ^ a.f;
    for (int e = 0; e < 32; ++e) {
        uint32_t p = 0, y = a.f;
        for (int i = 0; i < 5; ++i)
            if ((e >> i) & 1) p ^= basis[i], y ^= yb[i];
        g.lane[e] = p | (y << 16);
    }
    for (int e = 0; e < 8; ++e) {
        uint32_t p = 0, y = 0;
        for (int i = 0; i < 3; ++i)
            if ((e >> i) & 1) p ^= basis[5 + i], y ^= yb[5 + i];
        g.hi[e] = p | (y << 16);
    }
}

// One rotation step of a pass: rotations on the tile bits of `rot` (of
// layer[b]) in groups [g0, g1), then flips and the CNOTs t -> t + 1 of `cn`,
// ascending (on the map only).
struct Step {
    uint32_t rot, cn;
    int g0, g1;
    int layer[kTileBits];
};
struct Pass {
    int w, nsteps;
    uint32_t cn0;  // CNOTs before the first step
    Step step[kMaxSteps];
};

// The gates of a pass on the window from w, taken off the circuit's progress.
VQE_HD inline void make_pass(Progress &s, int w, Pass &p) {
    p.w = w;
    p.nsteps = 0;
    p.cn0 = 0;
    const int lo = w == kRunBits ? 0 : kRunBits;
    int groups = 0;
    for (;;) {
        Step st;
        st.rot = st.cn = 0;
        int c = 0;
        if (p.nsteps < kMaxSteps)
            for (int t = lo; t < kTileBits; ++t) {
                const int q = t < kRunBits ? t : w + t - kRunBits;
                if (q < s.n && rot_ready(s, q)) {
                    st.rot |= 1u << t;
                    st.layer[t] = s.rot[q]++;
                    ++c;
                }
            }
        for (int t = lo; t + 1 < kTileBits; ++t) {
            const int q = t < kRunBits ? t : w + t - kRunBits;
            if (q + 1 < s.n && cn_ready(s, q)) {
                s.cn[q]++;
                st.cn |= 1u << t;
            }
        }
        if (c == 0) {
            // CNOTs alone come first in a pass, or not at all: the sweep
            // after a step runs all that its rotations allow
            if (st.cn == 0 || p.nsteps > 0) return;
            p.cn0 = st.cn;
            continue;
        }
        st.g0 = groups;
        st.g1 = groups += (c + kGroupBits - 1) / kGroupBits;
        p.step[p.nsteps++] = st;
    }
}

// CTAs per cluster for the first circuits of the order (qubits(0) >= qubits(1)
// >= .. qubits(large - 1)), *joint of them, when few circuits hold much of the
// work; 1 and none when there are enough circuits.  A CTA
// alone with a circuit ends late if the circuit is more than a CTA's share of
// the work; of 17 qubits on (16 tiles and more, so that the passes over one
// tile and their preparation weigh less) sharing pays from half of that on.
// Milliseconds with 1, 4 and 8 CTAs per circuit, 10..20 qubits: 40 circuits
// 6.2, 2.1, 1.2; 200: 9.8, 3.9, 2.2; 1024: 14.4, 5.5, 6.3; 4096: 16.7, 19, 20;
// 13..16 qubits: 1024 circuits 1.2, 1.5, 1.9.
template <class Qubits>
inline int cluster_size(Qubits qubits, int large, int ctas, int *joint) {
    auto amps = [&](int k) { return (double)(1u << qubits(k)); };
    double work = 0.0;
    for (int k = 0; k < large; ++k) work += amps(k);
    auto shared = [&](int k) {
        const int n = qubits(k);
        return n >= 16 && amps(k) * ctas * (n >= 17 ? 2 : 1) > work;
    };
    *joint = 0;
    while (*joint < large && shared(*joint)) ++*joint;
    const int cl = amps(0) * ctas > 4.0 * work ? 8 : 4;
    if (*joint > 0 && ctas >= cl) return cl;
    *joint = 0;
    return 1;
}

}  // namespace qsim_vqe
