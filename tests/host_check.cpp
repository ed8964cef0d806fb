// Host-side checks of the library on a fake CUDA runtime (fake_cudart.h),
// linked with the library's own objects by tests/test_host_cpu.py: what its
// host code hands to the device, and what it does when a call fails.
#include "fake_cudart.h"

#include <cstdio>
#include <vector>

#include "../include/qsim.h"
#include "../paper_1612_08091_gb300/csrc/internal.h"
#include "../paper_1612_08091_gb300/csrc/vqe_window.cuh"

namespace {

int failures = 0;
#define CHECK(c)                                                          \
    do {                                                                  \
        if (!(c)) {                                                       \
            std::printf("line %d: %s is false\n", __LINE__, #c);          \
            ++failures;                                                   \
        }                                                                 \
    } while (0)

// sim_mlp_train: what its copies read lives until they have run, also where it
// returns an error
void check_training_sources() {
    const int n = 10;
    std::vector<float> X(16 * n, 0.5f), T(n, 1.f);
    qsim_mlp *m = nullptr;
    CHECK(sim_mlp_create(64, 1, nullptr, &m) == QSIM_OK);
    float loss = 0.f;
    fake::freed_sources = 0;
    CHECK(sim_mlp_train(m, X.data(), T.data(), n, 2, 4, 1e-3f, &loss) == QSIM_OK);
    CHECK(fake::launched("k_train") == 1);
    CHECK(sim_mlp_train(m, X.data(), T.data(), n, 500, 1, 1e-3f, &loss) == QSIM_OK);  // 5000 steps: two launches
    CHECK(fake::launched("k_train") == 3);
    CHECK(fake::freed_sources == 0);
    fake::fail_launch = "k_train";
    CHECK(sim_mlp_train(m, X.data(), T.data(), n, 2, 4, 1e-3f, &loss) == QSIM_ECUDA);
    fake::fail_launch = nullptr;
    CHECK(fake::npending == 0 && fake::freed_sources == 0);
    fake::fail_attribute = 1;
    CHECK(sim_mlp_train(m, X.data(), T.data(), n, 2, 4, 1e-3f, &loss) == QSIM_ECUDA);
    fake::fail_attribute = 0;
    CHECK(fake::npending == 0 && fake::freed_sources == 0);
    fake::run_copies();
    sim_mlp_destroy(m);
}

const double kHadamard[8] = {0.7, 0, 0.7, 0, 0.7, 0, -0.7, 0};

qsim *register_of(int n, int precision, int fusion = QSIM_FUSE_NONE) {
    qsim_opts o = {};
    o.fusion = fusion;
    o.kmax = 4;
    qsim *s = nullptr;
    CHECK(sim_create(n, precision, &o, &s) == QSIM_OK);
    CHECK(sim_reset(s, 0) == QSIM_OK);
    fake::launches().clear();
    return s;
}

// a queue on a small register where the cluster launch is not possible: the
// gates run one by one (complex128: cannot be placed; complex64: the launch fails)
void check_small_queue_falls_back() {
    for (int precision : {QSIM_C128, QSIM_C64}) {
        qsim *s = register_of(11, precision);
        fake::clusters = precision == QSIM_C128 ? 0 : 1;
        fake::fail_launch = precision == QSIM_C64 ? "k_small" : nullptr;
        for (int k = 0; k < 5; ++k) CHECK(sim_apply(s, kHadamard, &k, 1, nullptr, 0) == QSIM_OK);
        CHECK(sim_flush(s) == QSIM_OK);
        CHECK(fake::launched("k_small") == 0 && fake::launched("k_dense1") == 5);
        fake::clusters = 1;
        fake::fail_launch = nullptr;
        sim_destroy(s);
    }
    qsim *s = register_of(8, QSIM_C128);  // one CTA
    for (int k = 0; k < 5; ++k) CHECK(sim_apply(s, kHadamard, &k, 1, nullptr, 0) == QSIM_OK);
    CHECK(sim_flush(s) == QSIM_OK);
    CHECK(fake::launched("k_small") == 1 && fake::launches().size() == 1);
    sim_destroy(s);
}

// complex64 gates that the one launch makes slower go on their own, those
// between them together
void check_small_queue_runs() {
    const double swap[32] = {1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 1, 0, 0, 0, 0, 0, 1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 1, 0};
    for (int n : {13, 14}) {
        qsim *s = register_of(n, QSIM_C64);
        const int pair[2] = {1, 4};
        for (int k = 0; k < 5; ++k) CHECK(sim_apply(s, kHadamard, &k, 1, nullptr, 0) == QSIM_OK);
        CHECK(sim_apply(s, swap, pair, 2, nullptr, 0) == QSIM_OK);
        for (int k = 0; k < 2; ++k) CHECK(sim_apply(s, kHadamard, &k, 1, nullptr, 0) == QSIM_OK);
        CHECK(sim_apply(s, swap, pair, 2, nullptr, 0) == QSIM_OK);
        for (int k = 0; k < 5; ++k) CHECK(sim_apply(s, kHadamard, &k, 1, nullptr, 0) == QSIM_OK);
        CHECK(sim_flush(s) == QSIM_OK);
        if (n == 13)
            CHECK(fake::launches().size() == 1 && fake::launched("k_small") == 1);
        else
            CHECK(fake::launches().size() == 6 && fake::launched("k_small") == 2 && fake::launched("k_denseK") == 2 &&
                  fake::launched("k_dense1") == 2);
        sim_destroy(s);
    }
}

// plain gates in a stream capture: launches alone, no copy from host memory
// that a replay would repeat
void check_small_queue_under_capture() {
    for (int n : {7, 11}) {
        qsim *s = register_of(n, QSIM_C64);
        for (int k = 0; k < 5; ++k) CHECK(sim_apply(s, kHadamard, &k, 1, nullptr, 0) == QSIM_OK);
        fake::capturing = 1;
        const int copies = fake::copies;
        CHECK(sim_flush(s) == QSIM_OK);
        fake::capturing = 0;
        CHECK(fake::copies == copies && fake::launched("k_dense1") == 5 && fake::launches().size() == 5);
        sim_destroy(s);
    }
}

// which kernel moves a register's values: tiles, or the walk along the cycles,
// whichever was measured to be the faster on the register's qubits and cycles
void check_permutation_choice() {
    enum Kind { SWAPS, ADD, LONG, CADD, EIGHTS, IDENTITY };
    auto kernel = [](int n, int precision, int m, int q0, Kind kind) {
        qsim *s = register_of(n, precision);
        std::vector<uint64_t> f(1u << m);
        std::vector<int> qubits(m);
        const uint64_t D = f.size(), h = D / 2;
        for (int j = 0; j < m; ++j) qubits[j] = q0 + j;
        for (uint64_t v = 0; v < D; ++v) {
            f[v] = v;
            if (kind == SWAPS) f[v] = v ^ (D - 1);
            if (kind == ADD) f[v] = (v + 1) % D;
            if (kind == LONG) f[v] = (5 * v + 3) % D;  // one cycle of D values, far apart
            if (kind == EIGHTS) f[v] = (v + D / 8) % D;  // cycles of 8
            if (kind == CADD && v >= h) f[v] = h + (v - h + 3) % h;
        }
        CHECK(sim_apply_permutation(s, f.data(), qubits.data(), m, nullptr, 0) == QSIM_OK);
        const int walks = fake::launched("k_permute_cycles"), tiles = fake::launched("k_permute") - walks;
        sim_destroy(s);
        return walks ? 'w' : tiles ? 't' : '-';
    };
    for (int precision : {QSIM_C64, QSIM_C128}) {
        const int n = precision == QSIM_C64 ? 28 : 27, low = precision == QSIM_C64 ? 3 : 2;  // pieces of 64 bytes
        for (int m : {5, 6, 7, 8, 10}) {
            CHECK(kernel(n, precision, m, low, SWAPS) == 't');  // 1.2 ms and more against 0.9
            CHECK(kernel(n, precision, m, low, LONG) == 't');
        }
        CHECK(kernel(n, precision, 12, low, LONG) == 't');      // 2.0 to 2.9 ms against 1.0 to 1.5
        CHECK(kernel(n, precision, 12, low + 4, LONG) == 't');  // 2.1 to 2.5 against 1.2 to 1.6
        CHECK(kernel(n, precision, 12, low + 3, SWAPS) == 'w'); // 1.0 against 1.6 (1.2)
        CHECK(kernel(n, precision, 12, low, EIGHTS) == (precision == QSIM_C64 ? 'w' : 't'));  // 1.1 against 1.44 (1.0)
        CHECK(kernel(n, precision, 3, low, ADD) == 'w');        // 0.7 against 0.93
        CHECK(kernel(n, precision, 2, low + 1, SWAPS) == 'w');
        CHECK(kernel(n, precision, 8, low + 1, CADD) == 'w');   // half the values: 0.5 against 0.85
        CHECK(kernel(n, precision, 6, low + 7, LONG) == 'w');   // pieces of 8 KB
        CHECK(kernel(n, precision, 8, low, IDENTITY) == '-');
        CHECK(kernel(n - 6, precision, 12, low + 1, SWAPS) == 't');  // in L2: what the host does per value
        CHECK(kernel(n - 6, precision, 4, low + 1, SWAPS) == 'w');
        CHECK(kernel(n, precision, 4, 0, ADD) == 't');
    }
}

// every circuit of a batch is some CTA's: circuits are set aside for clusters
// only where clusters are launched
void check_batch_clusters() {
    for (int ctas = 1; ctas <= 304; ctas += ctas < 16 ? 1 : 16)
        for (int top = 13; top <= 24; ++top)
            for (int large : {1, 2, 5, 40, 400}) {
                int joint = -1;
                const int cl = qsim_vqe::cluster_size([&](int k) { return top - (k > 0 ? 1 : 0); }, large, ctas, &joint);
                CHECK(cl == 1 ? joint == 0 : joint > 0 && joint <= large && cl <= ctas);
            }
}

// gates queued in many short lists: the queue moves seldom
void check_queue_growth() {
    qsim *s = register_of(20, QSIM_C128);
    int moves = 0;
    for (int i = 0; i < 4096; ++i) {
        const int kind = QSIM_G_H, nt = 1, nc = 0, target = i % 20;
        const size_t before = s->queue.capacity();
        CHECK(sim_apply_gates(s, 1, &kind, &nt, &nc, &target, nullptr, nullptr, nullptr) == QSIM_OK);
        moves += s->queue.capacity() != before;
    }
    CHECK(s->queue.size() == 4096 && moves <= 13);
    sim_destroy(s);
}

// a batch reserves a state for every CTA that works on one, and no more
void check_batch_buffers() {
    const std::vector<int> nq(400, 15), nl(400, 2);
    std::vector<double> angles(400 * 60, 0.1), energies(400);
    for (int per_sm : {1, 2, 4}) {
        fake::ctas_per_sm = per_sm;
        size_t bytes = 0;
        CHECK(sim_batch_workspace_bytes(400, nq.data(), nl.data(), &bytes) == QSIM_OK);
        qsim_batch *b = nullptr;
        CHECK(sim_batch_create(400, nq.data(), nl.data(), 0.7, nullptr, nullptr, 0, &b) == QSIM_OK);
        CHECK(sim_batch_run(b, angles.data(), energies.data()) == QSIM_OK);
        const size_t state = sizeof(float) * 2 << 15, rest = sizeof(double) * angles.size() + 65536;
        CHECK(fake::grid * state < bytes && bytes <= 2 * fake::sms * state + rest);
        sim_batch_destroy(b);
    }
    fake::ctas_per_sm = 2;
}

}  // namespace

int main() {
    check_training_sources();
    check_small_queue_falls_back();
    check_small_queue_runs();
    check_small_queue_under_capture();
    check_permutation_choice();
    check_batch_clusters();
    check_queue_growth();
    check_batch_buffers();
    std::printf(failures ? "%d failures\n" : "ok\n", failures);
    return failures != 0;
}
