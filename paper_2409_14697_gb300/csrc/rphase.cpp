// Host: packing of complex64 register-phase programs for the device.
//
// build_register_phases (kgeom.cpp) gives each phase a list of members in circuit order:
// one-qubit matrices, controlled matrices and exchanges on register slots, and diagonals on
// any positions.  Applied one by one the diagonals cost the phase more than its matrices
// (every equal-angle RZZ run counts bit patterns per register, every run of one-qubit
// phases builds factor tables per thread).  But which factor register r of thread t takes
// from a run of diagonals depends on the thread only through a few bits of its index: the
// partners of two-qubit diagonals outside the register slots, and the lane bits that permute
// the register order (sigma).  So the run becomes one table of 2^5 factors for every value
// ("class") of those bits, made here in FP64, and one complex multiply per amplitude on
// the device whatever the number of gates.
//
// Members commute unless one changes a position that the other uses, so the list is first
// rescheduled: matrices as early as their slots' diagonals allow, diagonals gathered in as few
// runs as the matrices between them allow.  The result is a list of layers, each a table, then
// shears (rotations) on different slots, then other members as they were: the device reads one
// header per layer, where a member by itself cost about as many instructions to read as a
// real matrix costs to apply.
//
// A real matrix that is a rotation, c [[1, -t], [t, 1]], is D L(k) U(-t) or L(t) U(-k) D with shears
// L (lower) and U (upper), k = t / (1 + t^2) and D = diag(c, c (1 + t^2)).  Where the slot has a table
// after it, or before it, D goes there and the device applies the shears.  D is by register, as the
// shears are: a lane whose bit of sigma is set holds the rotation the other way round, which
// negates t and k and leaves D.  |t| <= 1: a rotation by more is the one by a right angle less, a
// sign for the table and an exchange, which only relabels the registers.  So no value grows by more
// than sqrt(2) before its table, and an amplitude is rounded once where the matrix rounded it twice.
// A reflection (H) is a rotation and a sign.
//
// The device's reals are FP32, and the rounding of an angle that a circuit repeats (Trotter
// steps) changes the norm the same way each time.  What the matrices and the tables so far have
// changed it by is divided out of the next table, whose own rounding then joins the account
// (RoundingDrift).  The 25-qubit Trotter circuit of 16 steps and its <Z> were 1.8e-5 to 2.3e-5 off
// with members alone, now 6.0e-6 to 8.5e-6 (four seeds); one of 23 qubits and 4 steps 4.3e-6, now
// 6.9e-7.  The account takes amplitudes as equally populated.  A call never divides out more than
// kMaxDriftFix, so that a state that is not (thousands of phases on qubits in |0>) is no further off than
// that, and the result stays near to what the plain FP32 matrices of the other execution modes give.
#include <algorithm>
#include <cmath>

#include "kgeom.h"

namespace qs {
namespace {

constexpr int kThreadBits = kTileThreadBits;  // position ids 0..7: thread-index bits, 8..12: slots
constexpr int kRegs = 1 << kRpBits;
constexpr uint32_t kSlotMask = ((1u << kRpBits) - 1u) << kThreadBits;

// One diagonal factor on at most two positions (ids ascending): d[x0 + 2 x1].
struct Term {
    int np = 0;
    int pos[2] = {-1, -1};
    cd d[4] = {1.0, 1.0, 1.0, 1.0};
    bool sign = false;  // only factors 1 and -1, from a sign member
    bool fixed = false; // d by register number, not by position's bit (D of a rotation; one slot)
    int lo = 0, hi = 0, at = -1;
    uint32_t mask() const { return (np > 0 ? 1u << pos[0] : 0u) | (np > 1 ? 1u << pos[1] : 0u); }
};

// A matrix, controlled matrix or exchange, kept as it is encoded.
struct Matrix {
    const double *code;
    int len;
    int slot, ctl;  // ctl: operand encoding of the control, -1 if none
    bool exchange, real;
    int at = 0;
    bool shears = false, toggle = false;  // real: as shears; then an exchange by relabelling
    double upper = 0.0, lower = 0.0;      // x += upper y, y += lower x
};

// sigma bit of a slot as an affine function of the thread index
struct Sigma {
    uint32_t bits = 0;
    bool one = false;
};

constexpr int kNone = -1, kOn = -2, kOff = -3;
// operand encoding -> position id, kOn (bit 1 everywhere) or kOff
int position_of(int enc) {
    if (enc == kRpAlways) return kOn;
    if (enc == kRpNever) return kOff;
    return (enc & 16) ? kThreadBits + (enc & 15) : enc;
}

// Encoding of a position id in a member.
int encode_position(int id) {
    if (id < 0) return kRpAlways;
    return id >= kThreadBits ? 16 + (id - kThreadBits) : id;
}

// A term from a function f(x_a, x_b) of two operand encodings.
template <typename F> Term make_term(int ea, int eb, const F &f) {
    Term t;
    const int a = position_of(ea), b = position_of(eb);
    auto value = [](int p, int id, int x) { return p == kOn ? 1 : p == kOff ? 0 : p == id ? x : 0; };
    if (a >= 0) t.pos[t.np++] = a;
    if (b >= 0 && b != a) t.pos[t.np++] = b;
    if (t.np == 2 && t.pos[0] > t.pos[1]) std::swap(t.pos[0], t.pos[1]);
    for (int x = 0; x < 4; x++) {
        const int x0 = x & 1, x1 = x >> 1;
        const int va = a >= 0 ? (a == t.pos[0] ? x0 : x1) : value(a, a, 0);
        const int vb = b >= 0 ? (b == t.pos[0] ? x0 : x1) : value(b, b, 0);
        t.d[x] = f(va, vb);
    }
    return t;
}

// log(1 + x) / 2 and exp(x) for the small x of roundings (|x| < 1e-5: next terms below 1e-15)
double half_log1p(double x) { return 0.5 * x * (1.0 - 0.5 * x); }
double exp_small(double x) { return 1.0 + x * (1.0 + 0.5 * x); }

// Logarithm of the factor by which rounding the reals of a 2x2 member to FP32 changes the norm.
double rounding_drift(const Matrix &m) {
    if (((int)m.code[0] & 7) != RP_M1) return 0.0;
    double exact = 0.0, rounded = 0.0;
    for (int i = 1; i < m.len; i++) {
        const double v = m.code[i], f = (double)(float)v;
        exact += v * v;
        rounded += f * f;
    }
    return exact > 0.0 && rounded > 0.0 ? half_log1p((rounded - exact) / exact) : 0.0;
}

struct Packer {
    const KOp &ph;
    std::vector<Term> terms;
    std::vector<Matrix> mats;
    std::vector<std::pair<bool, int>> order;  // (is matrix, index) in circuit order
    Sigma sigma[kRpBits];

    explicit Packer(const KOp &p) : ph(p) {
        int nlow = 0;
        for (int j = 0; j < kRpBits; j++) nlow += ph.pos[j] < 4 ? 1 : 0;
        int li = 4 - nlow;  // lane bits of the positions below 4, as rp_geometry assigns them
        for (int j = 0; j < kRpBits; j++)
            if (ph.pos[j] < 4) sigma[j].bits = 1u << li++;
    }

    void add(Term t) {
        order.push_back({false, (int)terms.size()});
        terms.push_back(t);
    }

    // false: a member this packing does not know
    bool decode(const double *prog) {
        const int nmem = (int)prog[0];
        const double *mm = prog + 1;
        for (int i = 0; i < nmem; i++) {
            const int code = (int)mm[0];
            const int type = code & 7, J = (code >> 3) & 7, ea = (code >> 6) & 31, eb = (code >> 11) & 31;
            const int len = (code >> 16) & 255;
            const double *P = mm + 1;
            auto c = [&](int j) { return cd(P[2 * j], P[2 * j + 1]); };
            switch (type) {
            case RP_M1: case RP_C1: case RP_X:
                order.push_back({true, (int)mats.size()});
                mats.push_back({mm, 1 + len, J, type == RP_M1 ? -1 : ea, type == RP_X, type == RP_M1 && eb == RP_REAL});
                break;
            case RP_DIAG:
                if (ea == eb) add(make_term(ea, ea, [&](int a, int) { return c(3 * a); }));
                else add(make_term(ea, eb, [&](int a, int b) { return c(2 * a + b); }));
                break;
            case RP_NEG:
                for (int q = 0; q <= J; q++) {
                    const int e = (int)P[q];
                    add(make_term(e & 31, e >> 5, [&](int a, int b) { return cd(a && b ? -1.0 : 1.0); }));
                    terms.back().sign = true;
                }
                break;
            case RP_PARITY:
                add(make_term(ea, eb, [&](int a, int b) { return c(a ^ b); }));
                break;
            case RP_PARITYN: {
                const int np = (len - 2) / 3;
                const cd t0(P[np], P[np + 1]), t1(P[np + 2], P[np + 3]);
                if (t0 == cd(0.0)) return false;
                Term k;  // the factor of no odd pattern, then the step from one count to the next
                for (cd &z : k.d) z = t0;
                add(k);
                const cd step = t1 / t0;
                for (int q = 0; q < np; q++) {
                    const int e = (int)P[q];
                    add(make_term(e & 31, e >> 5, [&](int a, int b) { return a ^ b ? step : cd(1.0); }));
                }
                break;
            }
            default:  // RP_PH
                if (J == 1) {
                    for (int q = 0; q < ea; q++) {
                        const int e = (int)P[3 * q];
                        const cd z(P[3 * q + 1], P[3 * q + 2]);
                        add(make_term(e, e, [&](int a, int) { return a ? z : cd(1.0); }));
                    }
                    for (int q = 0; q < eb; q++) {
                        const int e = (int)P[3 * ea + q];
                        add(make_term(e & 31, e >> 5, [&](int a, int b) { return cd(a && b ? -1.0 : 1.0); }));
                        terms.back().sign = true;
                    }
                } else {
                    add(make_term(ea, eb, [&](int a, int b) { return a && b ? c(0) : cd(1.0); }));
                }
                break;
            }
            mm += 1 + len;
        }
        return true;
    }

    // Rotations and reflections as shears where a table takes their slot's next diagonal, or its
    // last.  keep_norm: scaled so that the norm changes as by the matrix's reals in FP32, whichever
    // way the shears' are rounded.
    void make_shears(bool keep_norm) {
        const std::vector<std::pair<bool, int>> list = std::move(order);
        order.clear();
        order.reserve(3 * list.size());
        terms.reserve(terms.size() + 2 * mats.size());
        bool diagonal[kRpBits] = {false};  // on the slot until its next matrix, seen from the end
        bool plain[kRpBits] = {false};     // an RP_R0 is still to come: no exchanges on the slot
        std::vector<char> after(list.size(), 0), keep(list.size(), 0);
        auto pass = [&](const Term &t) {
            for (int k = 0; k < t.np; k++)
                if (!t.sign && t.pos[k] >= kThreadBits) diagonal[t.pos[k] - kThreadBits] = true;
        };
        for (size_t i = list.size(); i-- > 0;) {
            if (!list[i].first) {
                pass(terms[list[i].second]);
                continue;
            }
            const Matrix &m = mats[list[i].second];
            const int code = (int)m.code[0];
            after[i] = diagonal[m.slot];
            keep[i] = plain[m.slot];
            diagonal[m.slot] = false;
            if ((code & 7) == RP_M1 && ((code >> 11) & 31) == RP_R0) plain[m.slot] = true;
        }
        std::fill(diagonal, diagonal + kRpBits, false);
        for (size_t i = 0; i < list.size(); i++) {
            if (!list[i].first) {
                pass(terms[list[i].second]);
                order.push_back(list[i]);
                continue;
            }
            Matrix &m = mats[list[i].second];
            const bool before = diagonal[m.slot];
            diagonal[m.slot] = false;
            Term d, z;
            if ((after[i] || before) && shears(m, after[i], !keep[i], keep_norm, d, z)) {
                auto diagonals = [&]() {
                    add(d);
                    if (z.d[0] != cd(1.0) || z.d[1] != cd(1.0)) add(z);
                };
                if (!after[i]) diagonals();
                order.push_back(list[i]);
                if (after[i]) diagonals();
            } else {
                order.push_back(list[i]);
            }
        }
    }

    // m as shears with the diagonal d by register and signs z, both after it or both before it.
    static bool shears(Matrix &m, bool after, bool may_toggle, bool keep_norm, Term &d, Term &z) {
        if (!m.real) return false;
        const double *u = m.code + 1;
        // any matrix may come here (QS_DENSE): equal entries are asked for relative to the largest, and
        // matrices far from unit scale, whose reals FP32 may not hold to 24 bits, stay as they are
        double top = 0.0;
        for (int i = 0; i < 4; i++) top = std::max(top, std::fabs(u[i]));
        if (!(top >= 0.25 && top <= 4.0)) return false;
        const double tol = 1e-15 * top;
        const bool reflection = std::fabs(u[0] + u[3]) <= tol && std::fabs(u[1] - u[2]) <= tol;
        if (!reflection && (std::fabs(u[0] - u[3]) > tol || std::fabs(u[1] + u[2]) > tol)) return false;
        double a = u[0], b = reflection ? -u[2] : u[2];  // [[a, -b], [b, a]], then a sign if a reflection
        const bool toggle = std::fabs(a) < std::fabs(b);
        if (toggle) {  // X Z after [[b, a], [-a, b]]
            std::swap(a, b);
            b = -b;
        }
        if (a == 0.0 || (toggle && !may_toggle)) return false;
        m.shears = true;
        m.toggle = toggle;
        const double t = b / a, g = 1.0 + t * t, k = t / g;
        double s = a;
        if (keep_norm) {
            // squared norm of diag(1, g) L U, rows (1, -t) and (g k, g (1 - k t)), from rounded reals
            // (of U L diag(1, g), the other order, the same with rows and columns exchanged)
            const double tf = (double)(float)t, kf = (double)(float)k, x = 1.0 - kf * tf;
            const double change = (tf * tf - t * t + g * g * (kf * kf - k * k) + (g * x - 1.0) * (g * x + 1.0)) / (2.0 * g);
            s *= exp_small(rounding_drift(m) - half_log1p(change));
        }
        d.np = z.np = 1;
        d.pos[0] = z.pos[0] = kThreadBits + m.slot;
        d.fixed = z.sign = true;
        d.d[0] = s;
        d.d[1] = s * g;
        // D L(k) U(-t) or L(t) U(-k) D
        m.upper = after ? -t : -k;
        m.lower = after ? k : t;
        if (after) {
            z.d[0] = toggle ? -1.0 : 1.0;  // Z or (as X Z X) -Z
            z.d[1] = reflection ? -1.0 : 1.0;
            return true;
        }
        // before: a sign passes the shears and negates them
        if (toggle != reflection) {
            m.upper = -m.upper;
            m.lower = -m.lower;
            z.d[1] = -1.0;
        } else if (toggle) {
            z.d[0] = z.d[1] = -1.0;  // Z X Z = -X
        }
        return true;
    }

    // Times: diagonal runs at even times, matrices at odd ones.  Matrices as early as their
    // operands allow; a term may go to any even time of [lo, hi].
    void schedule() {
        int changed[kThreadBits + kRpBits], read[kThreadBits + kRpBits];  // last time a position was ...
        std::fill(changed, changed + kThreadBits + kRpBits, -1);
        std::fill(read, read + kThreadBits + kRpBits, 0);
        std::vector<int> open[kRpBits];  // terms on a slot since its last matrix
        int last = 0;
        for (const auto &o : order) {
            if (!o.first) {
                Term &t = terms[o.second];
                t.lo = 0;
                for (int k = 0; k < t.np; k++) t.lo = std::max(t.lo, changed[t.pos[k]] + 1);
                t.hi = 1 << 20;
                for (int k = 0; k < t.np; k++) {
                    read[t.pos[k]] = std::max(read[t.pos[k]], t.lo);
                    if (t.pos[k] >= kThreadBits) open[t.pos[k] - kThreadBits].push_back(o.second);
                }
                continue;
            }
            Matrix &m = mats[o.second];
            const int s = kThreadBits + m.slot;
            int t = std::max(changed[s], read[s] + 1);
            const int c = m.ctl >= 0 ? position_of(m.ctl) : kNone;
            if (c >= 0) t = std::max(t, changed[c]);
            if (t % 2 == 0) t++;
            m.at = t;
            changed[s] = t;
            // a control is read at an odd time: a later matrix on it may share that time (order
            // is kept inside a time), a diagonal on it does not change it
            if (c >= kThreadBits) read[c] = std::max(read[c], t - 1);
            for (int i : open[m.slot]) terms[i].hi = std::min(terms[i].hi, t - 1);
            open[m.slot].clear();
            last = std::max(last, t);
        }
        // fewest runs: terms by their last time, each in the latest run already placed inside its
        // interval, else in a new run at its last time
        std::vector<int> by(terms.size());
        const int end = last ? last + 1 : 0;
        for (Term &t : terms) t.hi = std::min(t.hi, end);
        std::vector<int> first((size_t)end + 2, 0);
        for (const Term &t : terms) first[(size_t)t.hi + 1]++;
        for (int i = 0; i <= end; i++) first[(size_t)i + 1] += first[(size_t)i];
        for (size_t i = 0; i < terms.size(); i++) by[(size_t)first[(size_t)terms[i].hi]++] = (int)i;
        std::vector<int> runs;
        for (int i : by) {
            Term &t = terms[i];
            if ((t.mask() & kSlotMask) == 0) continue;
            for (int r : runs)
                if (r >= t.lo && r <= t.hi) t.at = std::max(t.at, r);
            if (t.at < 0) runs.push_back(t.at = t.hi);
        }
        // factors that no register position chooses: with any run
        for (Term &t : terms)
            if (t.at < 0) t.at = runs.empty() ? end : runs.back();
    }
};

// A table under construction: the terms it takes and the thread bits that choose its class.
struct Table {
    std::vector<int> terms;
    uint32_t bits = 0;
};

// Appends the 2^5 factors per class: factor of register r and class c at
// ((r >> 1) 2^b + c) 4 + 2 (r & 1), so that a thread's loads are 16 bytes and threads of a
// quarter-warp, which differ in the lowest thread bits, read neighbouring classes.
// All of them are multiplied by `scale`; returns the sum of their squares as they are and as
// FP32.
std::pair<double, double> emit_table(const Packer &p, const Table &tb, double scale, std::vector<double> &out) {
    int bit[kRpMaxClassBits], nb = 0;
    for (int i = 0; i < kThreadBits; i++)
        if ((tb.bits >> i) & 1u) bit[nb++] = i;
    const size_t at = out.size();
    out.resize(at + ((size_t)64 << nb));
    // A class's factors in logical order (slot bits x) are a number, a pair per slot and, for all
    // classes, a product over pairs of slots.
    struct Factors {
        double re[kRegs], im[kRegs];
    };
    cd number = scale, slot[kRpBits][2];
    for (auto &f : slot) f[0] = f[1] = 1.0;
    double by_register[kRegs], weight[kRegs];
    by_register[0] = weight[0] = 1.0;
    double fixed[kRpBits][2];
    for (auto &f : fixed) f[0] = f[1] = 1.0;
    Factors two;
    bool any_two = false;
    std::vector<const Term *> mixed;
    uint32_t chooses = 0;  // thread bits in terms (the others of the class only permute)
    for (int i : tb.terms) {
        const Term &t = p.terms[i];
        const int a = t.np > 0 ? t.pos[0] - kThreadBits : 0;
        if (t.fixed) {
            for (int h = 0; h < 2; h++) fixed[a][h] *= t.d[h].real();
        } else if (t.np == 0) {
            number *= t.d[0];
        } else if (a < 0) {
            mixed.push_back(&t);
            chooses |= t.mask();
        } else if (t.np == 1) {
            for (int h = 0; h < 2; h++) slot[a][h] *= t.d[h];
        } else {
            const int b = t.pos[1] - kThreadBits;
            for (int x = 0; x < kRegs; x++) {
                const cd z = t.d[((x >> a) & 1) + 2 * ((x >> b) & 1)];
                const double re = any_two ? two.re[x] : 1.0, im = any_two ? two.im[x] : 0.0;
                two.re[x] = re * z.real() - im * z.imag();
                two.im[x] = re * z.imag() + im * z.real();
            }
            any_two = true;
        }
    }
    double inverse[kRpBits][2];  // squares
    for (int j = 0; j < kRpBits; j++)
        for (int h = 0; h < 2; h++) inverse[j][h] = fixed[j][h] == 1.0 ? 1.0 : 1.0 / (fixed[j][h] * fixed[j][h]);
    for (int j = 0; j < kRpBits; j++)
        for (int x = 0; x < (1 << j); x++) {
            by_register[x + (1 << j)] = by_register[x] * fixed[j][1];
            by_register[x] *= fixed[j][0];
            weight[x + (1 << j)] = weight[x] * inverse[j][1];
            weight[x] *= inverse[j][0];
        }
    Factors f;
    double exact = 0.0, rounded = 0.0, exact_f = 0.0, rounded_f = 0.0;
    uint32_t made = ~0u;  // the chosen bits that f was made for
    for (int c = 0; c < (1 << nb); c++) {
        uint32_t tid = 0;
        for (int i = 0; i < nb; i++) tid |= (uint32_t)((c >> i) & 1) << bit[i];
        const bool make = (tid & chooses) != made;
        if (make) {
            made = tid & chooses;
            cd n = number, s[kRpBits][2];
            std::copy(&slot[0][0], &slot[0][0] + 2 * kRpBits, &s[0][0]);
            for (const Term *t : mixed) {
                const int x0 = (tid >> t->pos[0]) & 1;
                if (t->np == 2 && t->pos[1] >= kThreadBits)
                    for (int h = 0; h < 2; h++) s[t->pos[1] - kThreadBits][h] *= t->d[x0 + 2 * h];
                else n *= t->d[x0 + (t->np == 2 ? 2 * ((tid >> t->pos[1]) & 1) : 0)];
            }
            f.re[0] = n.real();
            f.im[0] = n.imag();
            for (int j = 0; j < kRpBits; j++) {
                const double ar = s[j][0].real(), ai = s[j][0].imag(), br = s[j][1].real(), bi = s[j][1].imag();
                for (int x = 0; x < (1 << j); x++) {
                    const double re = f.re[x], im = f.im[x];
                    f.re[x + (1 << j)] = re * br - im * bi;
                    f.im[x + (1 << j)] = re * bi + im * br;
                    f.re[x] = re * ar - im * ai;
                    f.im[x] = re * ai + im * ar;
                }
            }
            if (any_two)
                for (int x = 0; x < kRegs; x++) {
                    const double re = f.re[x];
                    f.re[x] = re * two.re[x] - f.im[x] * two.im[x];
                    f.im[x] = re * two.im[x] + f.im[x] * two.re[x];
                }
        }
        int sg = 0;  // register r holds the amplitude whose slot bits are r ^ sigma
        for (int j = 0; j < kRpBits; j++)
            sg |= (int)((__builtin_popcount(p.sigma[j].bits & tid) & 1) ^ (p.sigma[j].one ? 1 : 0)) << j;
        double *o = out.data() + at + 4 * (size_t)c;
        const size_t step = (size_t)4 << nb;
        for (int r = 0; r < kRegs; r++) {
            double *e = o + (size_t)(r >> 1) * step + 2 * (r & 1);
            e[0] = f.re[r ^ sg] * by_register[r];
            e[1] = f.im[r ^ sg] * by_register[r];
        }
        if (make) {  // for all classes of these factors, whose order differs; an amplitude counts by
                     // what it was before a rotation's D
            exact_f = rounded_f = 0.0;
            for (int r = 0; r < kRegs; r++) {
                const double *e = o + (size_t)(r >> 1) * step + 2 * (r & 1);
                const double a = (double)(float)e[0], b = (double)(float)e[1];
                exact_f += weight[r] * (e[0] * e[0] + e[1] * e[1]);
                rounded_f += weight[r] * (a * a + b * b);
            }
        }
        exact += exact_f;
        rounded += rounded_f;
    }
    return {exact, rounded};
}

// Appends the factor of every class for terms that no slot chooses, 2 reals each.
void emit_thread_table(const Packer &p, const Table &tb, std::vector<double> &out) {
    int at[kThreadBits] = {0}, nb = 0;
    for (int i = 0; i < kThreadBits; i++)
        if ((tb.bits >> i) & 1u) at[i] = nb++;
    for (int c = 0; c < (1 << nb); c++) {
        cd f = 1.0;
        for (int i : tb.terms) {
            const Term &t = p.terms[i];
            const int x0 = t.np > 0 ? (c >> at[t.pos[0]]) & 1 : 0, x1 = t.np > 1 ? (c >> at[t.pos[1]]) & 1 : 0;
            f *= t.d[x0 + 2 * x1];
        }
        out.push_back(f.real());
        out.push_back(f.imag());
    }
    while (out.size() % 4) out.push_back(0.0);
}

// One layer of the packed program, in the device's order of execution.
struct Layer {
    int table = -1;      // index into the tables' offsets, -1: none
    int class_bits = 0;  // number of thread bits that spell a class
    uint32_t class_pos = 0;
    const Matrix *real[kRpBits] = {nullptr};  // as shears
    int members = 0;          // other members, in order
    std::vector<double> raw;
    uint32_t raw_uses = 0;    // slots they change or read
};

// Packs one phase; the program goes to `out` at a multiple of 4 reals.  max_reals: what it may
// take.  False: `out` is as before (no table to gain, an unknown member, or too long).
bool pack_phase(const KOp &ph, const std::vector<double> &in, size_t max_reals, RoundingDrift *drift,
                std::vector<double> &out, KOp &res) {
    Packer p(ph);
    if (ph.nt != kThreadBits || !p.decode(in.data() + ph.mat)) return false;
    if (p.terms.empty()) return false;
    p.make_shears(drift != nullptr);
    p.schedule();
    int last = 0;
    for (const Matrix &m : p.mats) last = std::max(last, m.at);
    for (const Term &t : p.terms) last = std::max(last, t.at);
    RoundingDrift account = drift ? *drift : RoundingDrift{};
    for (const Matrix &m : p.mats) account.open += rounding_drift(m);
    std::vector<Layer> layers;
    std::vector<double> tables;
    std::vector<size_t> table_at;
    auto raw = [&](int type, int slot, int ea, int eb, const std::vector<double> &pay) {
        if (layers.empty()) layers.emplace_back();
        Layer &l = layers.back();
        l.members++;
        l.raw.push_back((double)(type | slot << 3 | ea << 6 | eb << 11 | (int)pay.size() << 16));
        l.raw.insert(l.raw.end(), pay.begin(), pay.end());
        l.raw_uses = kSlotMask;  // a diagonal: nothing later may go before it
    };
    // terms by themselves: sign pairs are collected, other factors as a diagonal of their own
    auto raw_terms = [&](const std::vector<int> &list) {
        std::vector<double> pairs;
        auto flush = [&]() {
            if (!pairs.empty()) raw(RP_NEG, (int)pairs.size() - 1, 0, 0, pairs);
            pairs.clear();
        };
        for (int i : list) {
            const Term &t = p.terms[i];
            const int a = t.np > 0 ? encode_position(t.pos[0]) : kRpAlways;
            const int b = t.np > 1 ? encode_position(t.pos[1]) : a;
            if (t.sign) {
                // a sign member's term is -1 exactly where its one or two positions are 1, or
                // nowhere (paired with a bit that is 0); a rotation's may be -1 where they are 0
                const cd v = t.np == 0 ? t.d[0] : t.d[t.np == 2 ? 3 : 1];
                if (t.np == 1 && t.d[0] == cd(-1.0)) {
                    pairs.push_back((double)(kRpAlways | kRpAlways << 5));
                    if (v == cd(1.0)) pairs.push_back((double)(a | b << 5));
                    if (pairs.size() >= 7) flush();
                    continue;
                }
                if (v != cd(-1.0)) continue;
                pairs.push_back((double)(a | b << 5));
                if (pairs.size() >= 7) flush();
            } else if (t.np < 2) {
                const cd d0 = t.d[0], d1 = t.np ? t.d[1] : t.d[0];
                raw(RP_PARITY, 0, a, kRpNever, {d0.real(), d0.imag(), d1.real(), d1.imag()});
            } else {
                // entry index of the member: 2 x_a + x_b
                raw(RP_DIAG, 0, a, b, {t.d[0].real(), t.d[0].imag(), t.d[2].real(), t.d[2].imag(),
                                       t.d[1].real(), t.d[1].imag(), t.d[3].real(), t.d[3].imag()});
            }
        }
        flush();
    };
    auto matrix = [&](const Matrix &m) {
        const uint32_t slot = 1u << (kThreadBits + m.slot);
        const int c = m.ctl >= 0 ? position_of(m.ctl) : kNone;
        if (layers.empty()) layers.emplace_back();
        if (m.shears) {
            if (layers.back().real[m.slot] || (layers.back().raw_uses & slot)) layers.emplace_back();
            Layer &l = layers.back();
            l.real[m.slot] = &m;
            if (m.toggle) p.sigma[m.slot].one = !p.sigma[m.slot].one;
            return;
        }
        Layer &l = layers.back();
        l.members++;
        l.raw.insert(l.raw.end(), m.code, m.code + m.len);
        l.raw_uses |= slot;
        if (c >= kThreadBits) l.raw_uses |= 1u << c;
        if (!m.exchange) return;
        if (c == kOn) p.sigma[m.slot].one = !p.sigma[m.slot].one;
        else if (c >= 0 && c < kThreadBits) p.sigma[m.slot].bits ^= 1u << c;
    };
    // terms (even times) and matrices (odd ones), each in circuit order
    std::vector<int> begin((size_t)last + 2, 0), list(p.order.size());
    auto time_of = [&](const std::pair<bool, int> &o) { return o.first ? p.mats[o.second].at : p.terms[o.second].at; };
    for (const auto &o : p.order) begin[(size_t)time_of(o) + 1]++;
    for (size_t i = 1; i < begin.size(); i++) begin[i] += begin[i - 1];
    {
        std::vector<int> next(begin);
        for (const auto &o : p.order) list[(size_t)next[(size_t)time_of(o)]++] = o.second;
    }
    for (int time = 0; time <= last; time++) {
        const int *const first = list.data() + begin[(size_t)time], *const end = list.data() + begin[(size_t)time + 1];
        if (time & 1) {
            for (const int *i = first; i < end; i++) matrix(p.mats[*i]);
            continue;
        }
        if (first == end) continue;
        std::vector<Table> tabs;
        Table uniform;  // terms that no slot chooses
        std::vector<int> alone, free_terms;
        bool signs_only = true;
        for (const int *i = first; i < end; i++) signs_only = signs_only && p.terms[*i].sign;
        for (const int *i = first; i < end; i++) {
            const Term &t = p.terms[*i];
            if (signs_only) {  // a sign costs less than a table's complex multiply
                alone.push_back(*i);
                continue;
            }
            if ((t.mask() & kSlotMask) == 0) {
                free_terms.push_back(*i);
                continue;
            }
            uint32_t need = t.mask() & ((1u << kThreadBits) - 1u);
            for (int k = 0; k < t.np; k++)
                if (t.pos[k] >= kThreadBits && !t.fixed) need |= p.sigma[t.pos[k] - kThreadBits].bits;
            if (__builtin_popcount(need) > kRpMaxClassBits) {
                alone.push_back(*i);
                continue;
            }
            Table *to = nullptr;
            for (Table &tb : tabs)
                if (!to && __builtin_popcount(tb.bits | need) <= kRpMaxClassBits) to = &tb;
            if (!to) {
                tabs.emplace_back();
                to = &tabs.back();
            }
            to->bits |= need;
            to->terms.push_back(*i);
        }
        // factors without a register position: in a table that has room for their bits
        for (int i : free_terms) {
            Table *to = &uniform;
            for (Table &tb : tabs)
                if (to == &uniform && __builtin_popcount(tb.bits | p.terms[i].mask()) <= kRpMaxClassBits) to = &tb;
            to->bits |= p.terms[i].mask();
            to->terms.push_back(i);
        }
        for (const Table &tb : tabs) {
            Layer l;
            l.table = (int)table_at.size();
            for (int i = 0; i < kThreadBits; i++)
                if ((tb.bits >> i) & 1u) l.class_pos |= (uint32_t)i << (4 * l.class_bits++);
            layers.push_back(std::move(l));
            table_at.push_back(tables.size());
            double fix = 0.0;
            if (drift && std::fabs(account.open) < kMaxDriftFix)
                fix = std::min(std::max(account.fixed - account.open, -kMaxDriftFix), kMaxDriftFix) - account.fixed;
            const auto sums = emit_table(p, tb, exp_small(fix), tables);
            account.fixed += fix;
            account.open += fix;
            if (sums.first > 0.0) account.open += half_log1p((sums.second - sums.first) / sums.first);
        }
        if (!uniform.terms.empty()) {
            double lo = 0.0, hi = 0.0;
            int nb = 0;
            for (int i = 0; i < kThreadBits; i++)
                if ((uniform.bits >> i) & 1u) {
                    (nb < 4 ? lo : hi) += (double)(i << (4 * (nb & 3)));
                    nb++;
                }
            raw(RP_DIAG, 1, nb, 0, {(double)table_at.size(), lo, hi});
            table_at.push_back(tables.size());
            emit_thread_table(p, uniform, tables);
        }
        raw_terms(alone);
    }
    if (table_at.empty()) return false;
    // lay out: layer count, layers, tables
    size_t size = 4;
    for (Layer &l : layers) {
        while (l.raw.size() % 4) l.raw.push_back(0.0);
        size += 4 + l.raw.size();
        for (const Matrix *m : l.real) size += m ? 4 : 0;
    }
    const size_t pad = (4 - out.size() % 4) % 4;
    if (pad + size + tables.size() > max_reals || layers.size() > 1000) return false;
    out.resize(out.size() + pad, 0.0);
    res = ph;
    res.mat = (int32_t)out.size();
    res.nmat = (int32_t)(size + tables.size());
    out.insert(out.end(), {(double)layers.size(), 0.0, 0.0, 0.0});
    for (Layer &l : layers) {
        uint32_t mask = 0;
        for (int j = 0; j < kRpBits; j++)
            if (const Matrix *m = l.real[j]) mask |= (m->toggle ? 33u : 1u) << j;
        out.push_back((double)(mask | (uint32_t)l.class_bits << 10 | (l.table >= 0 ? 1u << 13 : 0u)));
        out.push_back(l.table >= 0 ? (double)(size + table_at[(size_t)l.table]) : 0.0);
        out.push_back((double)l.class_pos);
        out.push_back((double)(l.members | (uint32_t)(l.raw.size() / 4) << 8));
        for (const Matrix *m : l.real)
            if (m) out.insert(out.end(), {m->upper, m->lower, -m->upper, -m->lower});
        // a thread table's member names its table by number until here
        for (size_t at = 0, k = 0; k < (size_t)l.members; k++) {
            const int code = (int)l.raw[at];
            if ((code & 7) == RP_DIAG && ((code >> 3) & 7) == 1)
                l.raw[at + 1] = (double)(size + table_at[(size_t)l.raw[at + 1]]);
            at += 1 + ((code >> 16) & 255);
        }
        out.insert(out.end(), l.raw.begin(), l.raw.end());
    }
    out.insert(out.end(), tables.begin(), tables.end());
    if (drift) *drift = account;
    return true;
}

// Logarithm of the factor by which rounding a member's reals to FP32 changes the norm of a state:
// for every state by at least `sure` (0 where some states gain and others lose), on average over
// equally populated amplitudes by `mean`.
struct Change {
    double sure = 0.0, mean = 0.0;
};

// of factors that changes lo to hi apply to
Change between(double lo, double hi, double mean) { return {lo > 0.0 ? lo : hi < 0.0 ? hi : 0.0, mean}; }

Change member_drift(const double *code) {
    const int c = (int)code[0], type = c & 7, J = (c >> 3) & 7, ea = (c >> 6) & 31, eb = (c >> 11) & 31;
    const int len = (c >> 16) & 255;
    const double *P = code + 1;
    // of squared moduli; what is no rounding (an underflow, an overflow) is not taken back
    auto change = [](double rounded, double exact) {
        const double x = exact > 0.0 ? (rounded - exact) / exact : 0.0;
        return std::fabs(x) <= 1e-6 ? half_log1p(x) : 0.0;
    };
    auto square = [](double x) { return x * x; };
    auto factor = [&](int i) {  // the complex number at P[i]
        return change(square((float)P[i]) + square((float)P[i + 1]), square(P[i]) + square(P[i + 1]));
    };
    // entries at P[first], P[first + step], ...: unweighted, or by binomial weights of n - 1 patterns
    auto factors = [&](int first, int n, int step, bool binomial) {
        double lo = factor(first), hi = lo, mean = 0.0, w = binomial ? std::ldexp(1.0, 1 - n) : 1.0 / n;
        for (int k = 0; k < n; k++) {
            const double x = factor(first + k * step);
            lo = std::min(lo, x);
            hi = std::max(hi, x);
            mean += w * x;
            if (binomial) w = w * (n - 1 - k) / (k + 1);
        }
        return between(lo, hi, mean);
    };
    switch (type) {
    case RP_M1: {
        cd m[4], r[4];
        for (int i = 0; i < 4; i++) {
            const bool off = i == 1 || i == 2;
            if (eb == RP_REAL) m[i] = P[i];
            else if (eb == RP_RX) m[i] = off ? cd(0.0, P[i]) : cd(P[i]);
            else if (eb == RP_R0) m[i] = i ? cd(P[2 * i - 1], P[2 * i]) : cd(P[0]);
            else m[i] = cd(P[2 * i], P[2 * i + 1]);
            r[i] = cd((float)m[i].real(), (float)m[i].imag());
        }
        // squared norms of the columns and how far they are from orthogonal: the squared norm of a
        // state changes by a factor within x0, x1 and that
        const double e0 = std::norm(m[0]) + std::norm(m[2]), e1 = std::norm(m[1]) + std::norm(m[3]), e = 0.5 * (e0 + e1);
        const double was = std::abs(std::conj(m[0]) * m[1] + std::conj(m[2]) * m[3]);
        if (!(std::fabs(e0 - e1) <= 1e-12 * e && was <= 1e-12 * e)) return {};  // no multiple of a unitary
        const double x0 = change(std::norm(r[0]) + std::norm(r[2]), e0), x1 = change(std::norm(r[1]) + std::norm(r[3]), e1);
        const double off = 0.5 * std::abs(std::conj(r[0]) * r[1] + std::conj(r[2]) * r[3]) / e;
        const double mid = 0.5 * (x0 + x1), spread = std::hypot(0.5 * (x0 - x1), off);
        return between(mid - spread, mid + spread, mid);
    }
    case RP_DIAG: return ea == eb ? factors(0, 2, 6, false) : factors(0, 4, 2, false);
    case RP_PARITY: return factors(0, 2, 2, false);
    case RP_PARITYN: return factors((len - 2) / 3, (len - 2) / 3 + 1, 2, true);
    case RP_PH: {  // amplitudes without the pattern do not change
        Change s;
        if (J != 1) s.mean = (ea == eb ? 0.5 : 0.25) * factor(0);
        for (int q = 0; J == 1 && q < ea; q++) s.mean += 0.5 * factor(3 * q + 1);
        return s;
    }
    default: return {};
    }
}

}  // namespace

void correct_drift(std::vector<KOp> &kops, std::vector<double> &mats, RoundingDrift &account) {
    double sure = 0.0;
    KOp *last = nullptr;
    for (KOp &k : kops) {
        if (k.fkind != F_RPHASE) continue;
        last = &k;
        const double *at = mats.data() + k.mat + 1;
        for (int i = 0; i < (int)mats[(size_t)k.mat]; i++) {
            const Change d = member_drift(at);
            sure += d.sure;
            account.open += d.mean - d.sure;
            at += 1 + (((int)at[0] >> 16) & 255);
        }
    }
    const double fix = std::min(std::max(account.fixed - account.open, -kMaxDriftFix), kMaxDriftFix) - account.fixed;
    // below an FP32 rounding or so there is nothing to gain; one more member has to fit
    if (!last || std::fabs(fix - sure) < 1e-7 || last->nmat + 3 > kMaxOpReals) return;
    account.fixed += fix;
    account.open += fix;
    std::vector<double> prog(mats.begin() + last->mat, mats.begin() + last->mat + last->nmat);
    prog[0] += 1.0;
    prog.insert(prog.end(), {(double)(RP_PH | kRpAlways << 6 | kRpAlways << 11 | 2 << 16), std::exp(fix - sure), 0.0});
    last->mat = (int32_t)mats.size();
    last->nmat = (int32_t)prog.size();
    mats.insert(mats.end(), prog.begin(), prog.end());
}

std::vector<KOp> pack_register_phases(const std::vector<KOp> &kops, const std::vector<double> &mats, size_t max_reals,
                                      std::vector<double> &out, RoundingDrift *drift) {
    std::vector<KOp> res(kops);
    out.reserve(std::max(max_reals, mats.size() + 16 * kops.size()));
    size_t left = 0;  // reals of the ops not packed yet, as they are
    for (const KOp &k : kops) left += (size_t)k.nmat + 16;
    for (KOp &k : res) {
        left -= (size_t)k.nmat + 16;
        KOp packed;
        if (k.fkind == F_RPHASE && out.size() + left < max_reals &&
            pack_phase(k, mats, max_reals - out.size() - left, drift, out, packed)) {
            k = packed;
            continue;
        }
        if (k.fkind == F_RPHASE) {  // its members as they are, in one layer
            while (out.size() % 4) out.push_back(0.0);
            const size_t at = out.size(), reals = (size_t)k.nmat - 1, padded = (reals + 3) / 4 * 4;
            out.insert(out.end(), {1.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0,
                                   (double)((int)mats[(size_t)k.mat] | (int)(padded / 4) << 8)});
            out.insert(out.end(), mats.begin() + k.mat + 1, mats.begin() + k.mat + k.nmat);
            out.resize(at + 8 + padded, 0.0);
            k.mat = (int32_t)at;
            k.nmat = (int32_t)(8 + padded);
            continue;
        }
        const int at = (int)out.size();
        out.insert(out.end(), mats.begin() + k.mat, mats.begin() + k.mat + k.nmat);
        k.mat = at;
    }
    return res;
}

}  // namespace qs
