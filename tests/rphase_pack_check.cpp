// Test program (built and run by tests/test_rphase_pack_cpu.py, CPU only): packed register
// phases (pack_register_phases) against the programs they are made from.  Seeded random
// circuits on one tile of 2^13 amplitudes become register phases (build_register_phases);
// every phase is applied as built and as packed to the same random tile, in double
// precision, and both must agree.  A packed program's table members are applied here from the
// layout kops.cuh documents, with the register order (sigma) followed through the exchanges
// before them; its other members go through the interpreter of host_transforms_check.cpp one
// at a time.  Also checked: alignment, class bits, the limit on reals.
// Usage: rphase_pack_check <seed> <trials>; prints OK and exits 0 on success.
#define main host_transforms_main
#include "host_transforms_check.cpp"
#undef main

namespace {

int g_slot_tables = 0, g_thread_tables = 0, g_packed = 0, g_kept = 0, g_shears = 0, g_toggles = 0;

// Factor tables on the tile: per thread and register, entry(r, class).
template <typename F>
void apply_table(State &tile, const KOp &ph, const uint32_t *sig_bits, const bool *sig_one, int nb, uint64_t pos,
                 const F &entry) {
    for (uint32_t tid = 0; tid < (1u << ph.nt); tid++) {
        uint32_t c = 0, sigma = 0, base = 0;
        for (int b = 0; b < nb; b++) c |= ((tid >> ((pos >> (4 * b)) & 15u)) & 1u) << b;
        for (int j = 0; j < kRpBits; j++)
            sigma |= (uint32_t)((__builtin_popcount(sig_bits[j] & tid) & 1) ^ (int)sig_one[j]) << j;
        for (int b = 0; b < ph.nt; b++) base |= ((tid >> b) & 1u) << (uint32_t)((ph.off[0] >> (4 * b)) & 15u);
        for (uint32_t r = 0; r < 32; r++) {
            uint32_t x = base;
            for (int j = 0; j < kRpBits; j++)
                if (((r ^ sigma) >> j) & 1u) x |= 1u << ph.pos[j];
            tile[x] *= entry(r, c);
        }
    }
}

// x += u y, y += l x on the amplitudes that registers with bit j clear and set hold; in threads whose
// bit of sigma is set, those are the amplitudes with that position set and clear, and u, l negated.
void apply_shears(State &tile, const KOp &ph, const uint32_t *sig_bits, const bool *sig_one, int j, double u, double l) {
    for (uint32_t tid = 0; tid < (1u << ph.nt); tid++) {
        const bool s = (__builtin_popcount(sig_bits[j] & tid) & 1) ^ (int)sig_one[j];
        uint64_t base = 0;
        for (int b = 0; b < ph.nt; b++) base |= (uint64_t)((tid >> b) & 1u) << (uint32_t)((ph.off[0] >> (4 * b)) & 15u);
        for (uint32_t r = 0; r < 32; r++) {
            if ((r >> j) & 1u) continue;
            uint64_t x = base;
            for (int i = 0; i < kRpBits; i++)
                if ((r >> i) & 1u) x |= 1ull << ph.pos[i];
            const uint64_t y = x | 1ull << ph.pos[j];
            cd &a = tile[s ? y : x], &b = tile[s ? x : y];
            a += (s ? -u : u) * b;
            b += (s ? -l : l) * a;
        }
    }
}

// One packed phase on the tile.
void apply_packed(State &tile, int m, const KOp &ph, const std::vector<double> &mats, int trial) {
    check(ph.mat % 4 == 0, "packed program not at a multiple of 4 reals", trial);
    const double *prog = mats.data() + ph.mat;
    uint32_t sig_bits[kRpBits] = {0};
    bool sig_one[kRpBits] = {false};
    int nlow = 0;
    for (int j = 0; j < kRpBits; j++) nlow += ph.pos[j] < 4 ? 1 : 0;
    int li = 4 - nlow;
    for (int j = 0; j < kRpBits; j++)
        if (ph.pos[j] < 4) sig_bits[j] = 1u << li++;
    auto member = [&](const double *code, int len) {
        std::vector<double> one = {1.0};
        one.insert(one.end(), code, code + len);
        KOp k = ph;
        k.mat = 0;
        k.nmat = (int)one.size();
        apply_rphase(tile, m, k, one);
    };
    const double *at = prog + 4;
    for (int layer = 0; layer < (int)prog[0]; layer++) {
        const uint32_t h0 = (uint32_t)at[0], h1 = (uint32_t)at[1], h2 = (uint32_t)at[2], h3 = (uint32_t)at[3];
        check((at - prog) % 4 == 0, "layer not at a multiple of 4 reals", trial);
        const int nb = (int)((h0 >> 10) & 7u);
        if (h0 & (1u << 13)) {
            g_slot_tables++;
            check(nb <= kRpMaxClassBits && h1 % 4 == 0 && (int)(h1 + (64u << nb)) <= ph.nmat, "slot table", trial);
            apply_table(tile, ph, sig_bits, sig_one, nb, h2, [&](uint32_t r, uint32_t c) {
                const double *e = prog + h1 + 4 * (((r >> 1) << nb) + c) + 2 * (r & 1u);
                return cd(e[0], e[1]);
            });
        }
        const double *P = at + 4;
        for (int j = 0; j < kRpBits; j++) {
            if (!((h0 >> j) & 1u)) continue;
            check(P[2] == -P[0] && P[3] == -P[1] && std::fabs(P[0]) <= 1.0 && std::fabs(P[1]) <= 1.0, "shears", trial);
            apply_shears(tile, ph, sig_bits, sig_one, j, P[0], P[1]);
            g_shears++;
            P += 4;
        }
        for (int j = 0; j < kRpBits; j++)
            if ((h0 >> (5 + j)) & 1u) {  // an exchange that relabels
                for (uint64_t x = 0; x < tile.size(); x++)
                    if ((x >> ph.pos[j]) & 1u) std::swap(tile[x], tile[x ^ (1ull << ph.pos[j])]);
                sig_one[j] = !sig_one[j];
                g_toggles++;
            }
        const double *mm = P;
        for (int i = 0; i < (int)(h3 & 255u); i++) {
            const int code = (int)mm[0], type = code & 7, J = (code >> 3) & 7, ea = (code >> 6) & 31;
            const int len = (code >> 16) & 255;
            if (type == RP_M1 && ((code >> 11) & 31) == RP_R0)
                check(sig_bits[J] == 0 && !sig_one[J], "RP_R0 on a slot that sigma relabels", trial);
            if (type == RP_DIAG && J != 0) {
                g_thread_tables++;
                const size_t off = (size_t)mm[1];
                check((int)(off + (2u << ea)) <= ph.nmat, "thread table", trial);
                apply_table(tile, ph, sig_bits, sig_one, ea, (uint64_t)mm[2] | (uint64_t)mm[3] << 16,
                            [&](uint32_t, uint32_t c) { return cd(prog[off + 2 * c], prog[off + 2 * c + 1]); });
            } else {
                member(mm, 1 + len);
                if (type == RP_X) {
                    if (ea == kRpAlways) sig_one[J] = !sig_one[J];
                    else if (ea < 16) sig_bits[J] ^= 1u << ea;
                }
            }
            mm += 1 + len;
        }
        at = P + 4 * (h3 >> 8);
    }
}

// The phases themselves against the circuit, then each phase packed against itself.
void check_pack(std::mt19937_64 &g, const std::vector<Op> &ops, size_t max_reals, int trial, bool layered) {
    const int m = kTileThreadBits + kRpBits;
    int pos[64];
    for (int q = 0; q < 64; q++) pos[q] = q;
    std::vector<double> mats, packed;
    const std::vector<KOp> kops = build_register_phases(ops, pos, m, kTileThreadBits, mats, nullptr, layered);
    const std::vector<KOp> pk = pack_register_phases(kops, mats, max_reals, packed);
    check(pk.size() == kops.size(), "number of ops", trial);
    if (mats.size() + 16 * kops.size() <= max_reals) check(packed.size() <= max_reals, "more reals than allowed", trial);
    std::normal_distribution<double> N;
    State psi((size_t)1 << m);
    for (cd &z : psi) z = cd(N(g), N(g));
    const State start = psi;
    State all = psi;
    for (const KOp &k : kops) {
        if (k.fkind == F_RPHASE) apply_rphase(all, m, k, mats);
        else apply_kop(all, m, k, mats, 0);
    }
    check(rel_err(run(start, ops), all) < 1e-11, "phases", trial);
    for (size_t i = 0; i < kops.size(); i++) {
        if (kops[i].fkind != F_RPHASE) {
            check(std::equal(mats.begin() + kops[i].mat, mats.begin() + kops[i].mat + kops[i].nmat,
                             packed.begin() + pk[i].mat), "reals of an ordinary op", trial);
            continue;
        }
        State a = psi, b = psi;
        apply_rphase(a, m, kops[i], mats);
        check(max_reals >= 600 || pk[i].nmat <= kMaxOpReals, "kept phase too long to stage by itself", trial);
        const int tables = g_slot_tables;
        apply_packed(b, m, pk[i], packed, trial);
        (g_slot_tables > tables ? g_packed : g_kept)++;
        check(rel_err(a, b) < 1e-12, "packed phase", trial);
        psi = a;
        double s = 0.0;
        for (const cd &z : psi) s = std::max(s, std::abs(z));
        for (cd &z : psi) z /= s;
    }
}

Op gate(int type, std::initializer_list<int> q, double a = 0.0, double b = 0.0, double c = 0.0) {
    qs_gate r{};
    r.type = type;
    r.nq = (int)q.size();
    std::copy(q.begin(), q.end(), r.q);
    r.p[0] = a; r.p[1] = b; r.p[2] = c;
    return lower_gate(r);
}

}  // namespace

int main(int argc, char **argv) {
    const int seed = argc > 1 ? std::atoi(argv[1]) : 1, trials = argc > 2 ? std::atoi(argv[2]) : 8;
    const int n = kTileThreadBits + kRpBits;
    for (int trial = 0; trial < trials; trial++) {
        std::mt19937_64 g(1000 * seed + trial);
        std::uniform_real_distribution<double> ang(0.0, 2.0 * M_PI);
        try {
            for (int mix = 0; mix < 4; mix++)
                for (bool layered : {false, true}) check_pack(g, random_ops(g, n, 150, 0, mix), 10000, trial, layered);
            std::vector<Op> chain, phases, dense;
            for (int s = 0; s < 5; s++) {  // equal-angle bonds, then one-qubit gates: RX or U3
                const double t = ang(g);
                for (int q = 0; q + 1 < n; q++) chain.push_back(gate(QS_RZZ, {q, q + 1}, t));
                for (int q = 0; q < n; q++)
                    chain.push_back(trial & 1 ? gate(QS_RX, {q}, t) : gate(QS_U3, {q}, ang(g), ang(g), ang(g)));
                for (int q = 0; q < n; q++) phases.push_back(gate(q % 2 ? QS_P : QS_T, {q}, ang(g)));
                for (int q = s % 2; q + 1 < n; q += 2) phases.push_back(gate(QS_CZ, {q, q + 1}));
                for (int q = 0; q < n; q += 3) phases.push_back(gate(QS_CNOT, {q, (q + 5) % n}));
                for (int q = 0; q < n; q++) phases.push_back(gate(QS_RY, {q}, ang(g)));
                for (int q = 0; q < n; q++) phases.push_back(gate(QS_X, {q}));
                for (int a = 0; a < n; a++)  // every pair: more class bits than one table takes
                    for (int b = a + 1; b < n; b++) dense.push_back(gate(s & 1 ? QS_CP : QS_RZZ, {a, b}, ang(g)));
                for (int q = 0; q < n; q++) dense.push_back(gate(QS_H, {q}));
            }
            // rotations and reflections by any angle, at the ends of the shears' range too, with their
            // diagonals before or after them
            for (bool first : {false, true}) {
                std::vector<Op> turns;
                const double edge[6] = {0.0, M_PI / 4, M_PI / 2, M_PI, 1e-9, -M_PI / 4};
                for (int q = 0; q < n; q++) {
                    const double a = (q + trial) % 3 ? ang(g) : edge[(q + trial) / 3 % 6], c = std::cos(a), s = std::sin(a);
                    Op t;
                    t.kind = K_DENSE1;
                    t.k = 1;
                    t.q[0] = q;
                    if (q & 1) t.m = {cd(c), cd(s), cd(s), cd(-c)};
                    else t.m = {cd(c), cd(-s), cd(s), cd(c)};
                    if (first) turns.push_back(t);
                    turns.push_back(gate(QS_P, {q}, ang(g)));
                    if (!first) turns.push_back(t);
                }
                check_pack(g, turns, 10000, trial, true);
            }
            for (const auto *ops : {&chain, &phases, &dense})
                for (size_t limit : {(size_t)10000, (size_t)2500, (size_t)0}) {
                    check_pack(g, *ops, limit, trial, true);
                    check_pack(g, split_register_phases(*ops), limit, trial, limit != 2500);
                }
        } catch (const Error &e) {
            std::printf("FAIL trial %d: error %d %s\n", trial, e.code, e.msg.c_str());
            g_bad++;
        }
    }
    check(g_slot_tables > 0 && g_thread_tables > 0 && g_shears > 0 && g_toggles > 0 && g_packed > 0 && g_kept > 0, "packing not exercised", -1);
    std::printf("%s (%d slot tables, %d thread tables, %d phases packed, %d kept)\n", g_bad ? "FAIL" : "OK",
                g_slot_tables, g_thread_tables, g_packed, g_kept);
    return g_bad ? 1 : 0;
}
