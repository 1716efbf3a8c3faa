// Test program (built and run by tests/test_rphase_plain_cpu.py, CPU only): which ops a plain register
// phase (not in layers) takes.  Plain phases multiply by a diagonal on thread-index positions as by
// one factor per thread, so such a diagonal goes into the first phase that may hold it; only phases
// in layers leave it to the phase whose tables it can join.  And which circuits of 10 to 12 qubits run
// in phases (use_register_phases): not at 10 where exchanges or wide blocks would cut them short.
// Prints OK and exits 0 on success.
#include "rphase_pack_helpers.h"  // rphase_pack_check.cpp up to its main, written by the test

int main() {
    // a phase on every qubit of the lower eight, H on the upper five, then RX on the lower: the upper
    // five fill a phase's registers, the lower eight are thread-index bits there
    const int m = kTileThreadBits + kRpBits;
    std::vector<Op> ops;
    for (int q = 0; q < kTileThreadBits; q++) ops.push_back(gate(QS_T, {q}));
    for (int q = kTileThreadBits; q < m; q++) ops.push_back(gate(QS_H, {q}));
    for (int q = 0; q < kTileThreadBits; q++) ops.push_back(gate(QS_RX, {q}, 0.3));
    int pos[64];
    for (int q = 0; q < 64; q++) pos[q] = q;
    // phases on thread-index positions that the phase with the H members holds
    auto taken = [&](bool layered) {
        std::vector<double> mats;
        const std::vector<KOp> kops = build_register_phases(ops, pos, m, kTileThreadBits, mats, nullptr, layered);
        int phases = 0;
        for (const KOp &k : kops) {
            const double *at = mats.data() + k.mat + 1;
            bool h = false;
            int here = 0;
            for (int i = 0; i < (int)mats[(size_t)k.mat]; i++) {
                const int code = (int)at[0], type = code & 7, slot = (code >> 3) & 7, ea = (code >> 6) & 31;
                h |= type == RP_M1 && ((code >> 11) & 31) == RP_REAL && k.pos[slot] >= kTileThreadBits;
                if (type == RP_PH) here += slot == 1 ? ea : 1;
                at += 1 + ((code >> 16) & 255);
            }
            if (h) phases += here;
        }
        return phases;
    };
    check(taken(false) == kTileThreadBits, "a plain phase leaves diagonals on thread-index positions behind", 0);
    check(taken(true) == 0, "a phase in layers takes diagonals that a later phase's tables hold", 1);
    const qs_options o{};
    for (int n : {9, 10, 11, 12, 13}) {
        std::vector<Op> rotations, mixed, blocks, qft;
        for (int i = 0; i < 96; i++) {
            rotations.push_back(gate(i % 3 ? QS_U3 : QS_CZ, i % 3 ? std::initializer_list<int>{i % n} : std::initializer_list<int>{i % n, (i + 1) % n}, 0.1, 0.2, 0.3));
            mixed.push_back(i % 40 ? rotations.back() : gate(QS_SWAP, {0, 1}));  // 3 of 96
            qft.push_back(i % 2 ? gate(QS_H, {i % n}) : gate(QS_CP, {i % n, (i + 1) % n}, 0.1));
            blocks.push_back(gate(QS_SWAP, {i % n, (i + 1) % n}));
        }
        blocks.push_back(gate(QS_RX, {0}, 0.1));
        check(use_register_phases(rotations, n, o), "rotations in phases", n);
        check(use_register_phases(mixed, n, o) == (n != 10), "gates with exchanges between them", n);
        check(use_register_phases(blocks, n, o), "blocks for the most part", n);
        check(use_register_phases(qft, n, o) == (n < 10 || n > 12), "no rotation", n);
    }
    std::printf("%s\n", g_bad ? "FAIL" : "OK");
    return g_bad ? 1 : 0;
}
