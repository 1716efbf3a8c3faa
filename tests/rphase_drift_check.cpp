// Test program (built and run by tests/test_rphase_drift_cpu.py, CPU only): what the corrections
// of FP32 rounding do to the norm.  Programs have their reals rounded to FP32 as the kernels read
// them and are applied in double precision, so that the rounding of reals is the only error.
//  * correct_drift (phases of one tile, 10 to 12 qubits): what every state suffers alike (equal
//    rotations) is taken back in full; what depends on the state's populations is taken back by at
//    most kMaxDriftFix in a call, so a state that does not suffer it is no further off than that.
//  * pack_register_phases with an account: the account's open part is the logarithm of what the
//    norm of a random state did, and no more than kMaxDriftFix is divided out.
// Usage: rphase_drift_check <seed>; prints OK and exits 0 on success.
#include "rphase_pack_helpers.h"  // rphase_pack_check.cpp up to its main, written by the test

namespace {

constexpr double kUlp = 6e-8;  // 2^-24

std::vector<double> as_fp32(std::vector<double> v) {
    for (double &x : v) x = (double)(float)x;  // codes and offsets are whole numbers below 2^24
    return v;
}

double norm2(const State &s) {
    double r = 0.0;
    for (const cd &z : s) r += std::norm(z);
    return r;
}

// The circuit on one tile of 2^n amplitudes from psi, corrected, reals as FP32.
State run_tile(const std::vector<Op> &ops, int n, State psi, RoundingDrift &account) {
    int pos[64];
    for (int q = 0; q < 64; q++) pos[q] = q;
    std::vector<double> mats;
    std::vector<KOp> kops = build_register_phases(ops, pos, n, n - kRpBits, mats);
    correct_drift(kops, mats, account);
    mats = as_fp32(mats);
    for (const KOp &k : kops) {
        if (k.fkind == F_RPHASE) apply_rphase(psi, n, k, mats);
        else apply_kop(psi, n, k, mats, 0);
    }
    return psi;
}

State zero_state(int n) {
    State psi((size_t)1 << n);
    psi[0] = 1.0;
    return psi;
}

void check_one_tile(int n, std::mt19937_64 &g) {
    std::uniform_real_distribution<double> ang(0.1, 3.0);
    for (double theta : {0.8043, 1.0, ang(g), ang(g)}) {
        // gates that leave |0> alone, thousands of one angle: no state of theirs changes its norm
        for (int type : {QS_CP, QS_P}) {
            std::vector<Op> ops = {gate(QS_RY, {n - 1}, 0.4)};
            for (int i = 0; i < 3600; i++) {
                const int a = i % (n - 1), b = (i + 1 + i / (n - 1)) % (n - 1);
                if (type == QS_CP && a != b) ops.push_back(gate(QS_CP, {a, b}, theta));
                if (type == QS_P) ops.push_back(gate(QS_P, {a}, theta));
            }
            RoundingDrift account;
            const State got = run_tile(ops, n, zero_state(n), account), want = run(zero_state(n), ops);
            check(rel_err(want, got) <= kMaxDriftFix + 4 * kUlp, "gates on |0> scaled the state", n);
            check(std::fabs(account.fixed) <= kMaxDriftFix, "cap of a call", n);
            // a second pass of the same call has only what is left of the cap
            run_tile(ops, n, zero_state(n), account);
            check(std::fabs(account.fixed) <= kMaxDriftFix, "cap of a call over two passes", n);
        }
        // one rotation repeated on a few qubits of |0...0>: every state suffers its rounding, up to
        // 2 * 2000 * 2^-24 of the norm
        for (int type : {QS_RX, QS_RY}) {
            std::vector<Op> ops;
            for (int i = 0; i < 2000; i++) ops.push_back(gate(type, {i % 3}, theta));
            RoundingDrift account;
            check(std::fabs(norm2(run_tile(ops, n, zero_state(n), account)) - 1.0) <= 6 * kUlp, "equal rotations", n);
            check(account.fixed == 0.0, "equal rotations do not use the cap", n);
        }
    }
}

// Packed phases with one account over all of them, applied to a Gaussian state, whose amplitudes
// populate all factors alike.
void check_account(std::mt19937_64 &g, const std::vector<Op> &ops, int trial) {
    const int m = kTileThreadBits + kRpBits;
    int pos[64];
    for (int q = 0; q < 64; q++) pos[q] = q;
    std::normal_distribution<double> N;
    State psi((size_t)1 << m);
    for (cd &z : psi) z = cd(N(g), N(g));
    std::vector<double> mats, packed;
    const std::vector<KOp> kops = build_register_phases(ops, pos, m, kTileThreadBits, mats, nullptr, true);
    RoundingDrift account;
    const std::vector<KOp> pk = pack_register_phases(kops, mats, 1000000, packed, &account);
    check(std::fabs(account.fixed) <= kMaxDriftFix, "more divided out than allowed", trial);
    packed = as_fp32(packed);
    const double before = norm2(psi);
    for (const KOp &k : pk) {
        if (k.fkind == F_RPHASE) apply_packed(psi, m, k, packed, trial);
        else apply_kop(psi, m, k, packed, 0);
    }
    // an amplitude's factor differs from its table's mean by a rounding, and 2^13 random amplitudes
    // average them, weighted by exponentially distributed probabilities (a factor of sqrt 2)
    const double tol = 5.0 * std::sqrt((double)ops.size()) * kUlp * std::sqrt(2.0 / (double)psi.size());
    check(std::fabs(0.5 * std::log(norm2(psi) / before) - account.open) <= tol, "the account's open part", trial);
}

}  // namespace

int main(int argc, char **argv) {
    const int seed = argc > 1 ? std::atoi(argv[1]) : 1;
    std::mt19937_64 g(9000 + seed);
    std::uniform_real_distribution<double> ang(0.0, 2.0 * M_PI);
    try {
        for (int n : {10, 11, 12}) check_one_tile(n, g);
        const int n = kTileThreadBits + kRpBits;
        for (int steps : {4, 30}) {  // the cap is reached in some of the longer ones
            std::vector<Op> trotter, brick;
            const double t = 0.05 + 0.01 * ang(g), h = 0.07 + 0.01 * ang(g);
            for (int s = 0; s < steps; s++) {
                for (int q = 0; q + 1 < n; q++) trotter.push_back(gate(QS_RZZ, {q, q + 1}, t));
                for (int q = 0; q < n; q++) trotter.push_back(gate(QS_RX, {q}, h));
                for (int q = 0; q < n; q++) brick.push_back(gate(QS_U3, {q}, ang(g), ang(g), ang(g)));
                for (int q = s % 2; q + 1 < n; q += 2) brick.push_back(gate(QS_CZ, {q, q + 1}));
            }
            check_account(g, trotter, steps);
            check_account(g, split_register_phases(trotter), steps);
            check_account(g, split_register_phases(brick), steps);  // whole U3 make no tables, and no account
        }
    } catch (const Error &e) {
        std::printf("FAIL: error %d %s\n", e.code, e.msg.c_str());
        g_bad++;
    }
    std::printf("%s\n", g_bad ? "FAIL" : "OK");
    return g_bad ? 1 : 0;
}
