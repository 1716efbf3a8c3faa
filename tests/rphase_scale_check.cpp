// Test program (built and run by tests/test_rphase_scale_cpu.py, CPU only): 2x2 matrices of any
// scale and shape through the host rewrites that take rotations apart.  QS_DENSE takes any finite
// matrix, so a rewrite that asks for a rotation or a unitary has to ask it of the matrix itself,
// not of its distance to zero.  Matrices far from unitary, at scales from 1 down to 1e-20 and up
// to 1e8, stand between diagonals on their qubits: split_register_phases and the packed phases
// (pack_register_phases, without and with an account of roundings) must act as the circuit.
// Usage: rphase_scale_check <seed>; prints OK and exits 0 on success.
#include "rphase_pack_helpers.h"  // rphase_pack_check.cpp up to its main, written by the test

namespace {

// The circuit's phases, and the same packed, on one tile; the largest difference relative to the
// largest amplitude.  drift: packed with an account, whose corrections are at most kMaxDriftFix.
double packed_error(std::mt19937_64 &g, const std::vector<Op> &ops, bool account, int trial) {
    const int m = kTileThreadBits + kRpBits;
    int pos[64];
    for (int q = 0; q < 64; q++) pos[q] = q;
    std::vector<double> mats, packed;
    const std::vector<KOp> kops = build_register_phases(ops, pos, m, kTileThreadBits, mats, nullptr, true);
    RoundingDrift drift;
    const std::vector<KOp> pk = pack_register_phases(kops, mats, 10000, packed, account ? &drift : nullptr);
    check(!(std::fabs(drift.fixed) > kMaxDriftFix), "more divided out than allowed", trial);
    std::normal_distribution<double> N;
    State psi((size_t)1 << m);
    for (cd &z : psi) z = cd(N(g), N(g));
    const State want = run(psi, ops);
    for (const KOp &k : pk) {
        if (k.fkind == F_RPHASE) apply_packed(psi, m, k, packed, trial);
        else apply_kop(psi, m, k, packed, 0);
    }
    return rel_err(want, psi);
}

}  // namespace

int main(int argc, char **argv) {
    const int seed = argc > 1 ? std::atoi(argv[1]) : 1;
    const int n = kTileThreadBits + kRpBits;
    const std::vector<std::vector<cd>> shapes = {
        {1.0, 0.3, 0.1, 3.0},                              // real, no rotation
        {1.0, 0.0, 0.0, 1.0001},                           // real diagonal
        {0.6, 0.8, 0.8, -0.5999},                          // almost a reflection
        {0.6, -0.8, 0.8, 0.6},                             // a rotation
        {1.0, cd(0.0, 0.5), 0.5, cd(2.0, 0.3)},            // complex, no unitary
        {0.6, cd(0.0, -0.8), cd(0.0, -0.8), 0.6},          // RX-like
        {cd(0.36, 0.48), cd(0.0, 0.8), cd(0.8, 0.0), cd(0.48, -0.359)},  // almost unitary
    };
    std::mt19937_64 g(7000 + seed);
    std::uniform_real_distribution<double> ang(0.0, 2.0 * M_PI);
    int trial = 0;
    for (const auto &shape : shapes)
        for (double scale : {1.0, 1e-6, 1e-12, 1e-15, 1e-16, 1e-20, 1e8}) {
            // the matrix on one qubit in three (the scales of all would multiply), U3 on the others
            std::vector<Op> ops;
            for (int q = 0; q < n; q++) ops.push_back(gate(QS_P, {q}, ang(g)));
            for (int q = 0; q < n; q++) {
                if ((q + seed) % 3) {
                    ops.push_back(gate(QS_U3, {q}, ang(g), ang(g), ang(g)));
                    continue;
                }
                Op t;
                t.kind = K_DENSE1;
                t.k = 1;
                t.q[0] = q;
                for (const cd &z : shape) t.m.push_back(z * scale);
                ops.push_back(t);
            }
            for (int q = 0; q < n; q++) ops.push_back(gate(QS_P, {q}, ang(g)));
            try {
                std::vector<Op> split = split_register_phases(ops);
                State psi((size_t)1 << n);
                std::normal_distribution<double> N;
                for (cd &z : psi) z = cd(N(g), N(g));
                check(rel_err(run(psi, ops), run(psi, split)) < 1e-12, "split_register_phases", trial);
                check(rel_err(run(psi, ops), run(psi, split_one_qubit_phases(ops))) < 1e-12, "split_one_qubit_phases", trial);
                for (const auto *list : {&ops, &split}) {
                    check(packed_error(g, *list, false, trial) < 1e-12, "packed phases", trial);
                    // an account divides at most kMaxDriftFix out, and a rotation's shears take
                    // over what rounding its reals to FP32 did (2^-24 each)
                    check(packed_error(g, *list, true, trial) < kMaxDriftFix + n * 6e-8, "packed phases with an account", trial);
                }
            } catch (const Error &e) {
                std::printf("FAIL trial %d: error %d %s\n", trial, e.code, e.msg.c_str());
                g_bad++;
            }
            trial++;
        }
    std::printf("%s (%d circuits)\n", g_bad ? "FAIL" : "OK", trial);
    return g_bad ? 1 : 0;
}
