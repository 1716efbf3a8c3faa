// Host: lowered Op -> KOp (kernel-side op) in a given index space.
#pragma once

#include "kops.cuh"
#include "qs_internal.h"

namespace qs {

// Builds the KOp of `op`; pos[q] is the bit position of qubit q in the target index
// space (identity for the whole state, tile-local position for a chunk pass).  The
// op's matrix entries are appended to `mats` (as re, im doubles; KOp.mat indexes them).
KOp make_kop(const Op &op, const int *pos, std::vector<double> &mats);

// The same for the shared-memory tile kernels: a diagonal on 3 or more qubits whose entries
// are 1 unless some qubits ("controls") are set becomes F_CDIAGK, which touches only the
// elements with every control set.
KOp make_tile_kop(const Op &op, const int *pos, std::vector<double> &mats);

// complex128 FP64 tile programs: an unscaled Hadamard (F_H with scale 1) directly followed
// by an F_CDIAGK whose only control is the Hadamard's position becomes one F_HCDIAGK (the
// block multiplies only the elements the butterfly's difference lands on, so both fit
// one sweep of the tile; a QFT target and its controlled phases).
std::vector<KOp> join_h_cdiag(const std::vector<KOp> &kops, const std::vector<double> &mats);

// complex64 tiles of 2^m amplitudes with 2^thread_bits threads: true if register phases
// apply (m = thread_bits + kRpBits).
bool rphase_applicable(int m, int thread_bits);
// Thread-index bits of the register phases of an n-qubit complex64 state in tiles of 2^m
// amplitudes, 0: none.  All threads on tiles of 2^13; 32 to 128 of them where the whole state is
// one tile of 2^10 to 2^12 (a phase of 32 amplitudes per thread replaces several sweeps and
// barriers: 128 circuits of 12 qubits and 60 layers in one batch 1173 -> 400 us, of 10 qubits
// 543 -> 336).
int rphase_threads(int n, int m);
// Packs the pass's ops (logical qubits, tile position of qubit q = pos[q]) into register
// phases (F_RPHASE KOps; their programs appended to `mats`).  Ops no phase can hold
// (swaps, wider dense or diagonal blocks) become ordinary KOps in their place in the
// order.  n_phases (optional) receives the number of phases.
std::vector<KOp> build_register_phases(const std::vector<Op> &ops, const int *pos, int m, int thread_bits,
                                       std::vector<double> &mats, int *n_phases = nullptr, bool layered = false);

// Passes of 2^kPackTileBits tiles or more run their register phases in layers, with one-qubit
// gates split into rotations and phases; smaller states wait for the host, which takes about
// 60 us longer per pass to build them (20-layer brickwork, 21 qubits: 0.76 ms against 0.60; 22
// qubits: 0.80 against 0.96).
constexpr int kPackTileBits = 9;
// A pass's register phases in layers: layers of a factor table and shears (rphase.cpp).
// Returns the ops with their reals re-laid in `out` (other ops unchanged), which stays within
// max_reals, if it can, by giving later phases one layer of their members as they are; every
// phase starts at a multiple of 4 reals.  drift: the call's account of what rounding to FP32 did
// to the norm; none: tables are not corrected for it.
std::vector<KOp> pack_register_phases(const std::vector<KOp> &kops, const std::vector<double> &mats, size_t max_reals,
                                      std::vector<double> &out, RoundingDrift *drift = nullptr);

// Register phases as they are (not in layers): one member more at the end of the last, a real
// factor that takes back what rounding the others' reals to FP32 does to the norm.  For states of
// one tile, whose gates would otherwise run fused in FP64 and add up less of it.  What every state
// suffers alike (equal rotations) is taken back in full; what only equally populated amplitudes
// do (a phase on some of them) by at most kMaxDriftFix in a call, whose account it is: 3600
// controlled phases on qubits in |0> change nothing, and an uncapped factor was 3.7e-5 off.
void correct_drift(std::vector<KOp> &kops, std::vector<double> &mats, RoundingDrift &account);

// Fraction of the state's bytes one streaming application reads and writes, counting
// whole DRAM sectors of 2^sector_bits elements.
double kop_touched_fraction(const KOp &k, int sector_bits);

}  // namespace qs
