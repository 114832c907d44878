// The unitary step by the sparse Hamiltonian: V = U rho U^+ with U = exp(X), X = -i dt H
// (minus dt/2 diag(d) in the effective step), formed by applying the Taylor series of exp(X)
// to every column of rho and then to every row of the result, without forming U.
//
// Every H of this library couples a basis state to a few others (one term per atom, bond and
// tunnelling digit), so X t costs a few multiply-adds per element where the dense product
// costs D: at dim 512 (at most five couplings a row, seven terms) 1/25 of the multiply-adds.
// The series starts from X' = X - Lambda, Lambda the middle of H's diagonal over each connected
// component of H's graph: X is block diagonal over the components, so exp(X) =
// exp(Lambda) exp(X') exactly, and what is left in X' (couplings and detunings) is small: a
// few terms reach the rounding level.  The phases exp(Lambda) are applied once, at the end.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "model.h"

namespace qed {

// Device tables of X' (rows in ELL form, entry j of row k at [j * D + k]) and the phases.
struct SparseX {
    void *block = nullptr;       // the allocation of every table
    int D = 0;
    int terms = 0;               // Taylor terms of exp(X' / substeps) in a step's pass
    int all_terms = 0;           // in U's, at least 16
    int frechet_terms = 0;       // of the Frechet derivative's series, at least 13
    int substeps = 0;
    double norm = 0.0;           // infinity norm of X'
    bool pays = false;           // a step is faster through it (passes_pay)
    int *len = nullptr;          // [D] couplings of row k
    int *col = nullptr;          // [width][D]
    double *val = nullptr;       // [width][D]  dt H_kl
    double2 *diag = nullptr;     // [D] residual diagonal of X' (real, imaginary), or null if all zero
    double2 *phi = nullptr;      // [D] exp(Lambda_k)
    // Rows sorted by their number of couplings (a warp's rows then end together): entry j of sorted
    // row p at [j * D + p].
    int2 *order = nullptr;       // [D] {row, couplings}
    int *place = nullptr;        // [D] the sorted place of row k
    int4 *entry = nullptr;       // [longest row, at least 1][D] {column's place, 0, dt H_kl}
    double *inv = nullptr;       // [all_terms + 1] 1 / (substeps n)
    double2 *diag_sorted = nullptr;  // [D] diag in sorted order, or null
    // Lambda's distinct values: class of each row, and phi of class a times conj(phi) of b
    int *cls = nullptr;          // [D]
    double2 *pair = nullptr;     // [classes][classes], or null beyond kSparseClasses
    int classes = 0;
};
constexpr int kSparseClasses = 32;

// A pass over all columns: out = (op In)^T, op = exp(X') (adjoint-side false) or its complex
// conjugate (true); two passes give V: A = (U In)^T, then (conj(U) A)^T = U In U^+.  With
// `phases` the result's element (i, j) is multiplied by phi_i conj(phi_j), or by phi_i alone
// (kPhaseRow): what exp(Lambda) adds to both sides or to one.
// kPhaseConj is kPhaseBoth conjugated, for U^+ In U.
enum SparsePhase { kPhaseNone = 0, kPhaseBoth = 1, kPhaseRow = 2, kPhaseConj = 3 };

// Largest dimension a pass takes (three columns in shared memory), and the largest norm of X' that
// the series is used for: eight substeps of 18 terms, where U costs half of a step's passes (below)
// against ten and more dense products and an elimination.
constexpr int kSparseMaxDimF64 = 4800;
constexpr double kSparseMaxNormF64 = 8.0;

// Whether V = U rho U^+ is faster in two passes than in two dense FP64 products, by estimates of a
// step in us (Lindblad update and launches in both), fitted to chains of 65 to 801 states, lattices
// of 73 to 1153 and single cavities with 64 atoms each at norms of 0.001 to 7.9 (6 to 144 terms):
// within 20 %, and on the slower side only where both are equal (96 states).  A pass and term costs
// its longest row's chain and the FP64 instructions of its couplings.  Passes and products, measured:
// dim 96 and norm 0.05 27 and 20 us, dim 129 28 and 41; at norm 1.5 dim 160 96 and 67, dim 257 141
// and 244; at norm 7.9 dim 350 935 and 642, dim 512 1860 and 2170; two cavities of 64 atoms (rows
// of 65 couplings, dim 131, norm 0.05) 123 and 42, nine (dim 586) 183 and 4060.
inline bool passes_pay(double D, double couplings, double longest, double terms) {
    const double passes = 8.6 + 3.2e-5 * D * D + terms * (0.32 + 0.177 * longest + 6.9e-6 * D * (couplings + D));
    return passes < 8.0 + 1.58e-5 * D * D * D;
}

// Builds the tables of m's scheme from its host model into m->sx, which is null before and stays
// null where the series does not apply (the dense products then form the step).
qed_status sparse_prepare(qed_model *m, int scheme);
// The component of each state in H's graph (couplings of strength zero included).
std::vector<int> hamiltonian_components(const HostModel &hm);
void sparse_release(SparseX *x);

void sparse_pass_f64(cudaStream_t s, const SparseX &x, const double2 *in, double2 *out, bool conj_side,
                     SparsePhase phases);
// V = U In U^+, or U^+ In U with `back` (X' = -i H' of the Lie and Strang steps, whose inverse is
// its conjugate); tmp and out D x D, out may not be `in`.
void sparse_conjugate_f64(cudaStream_t s, const SparseX &x, const double2 *in, double2 *tmp, double2 *out, bool back);

// The Hamiltonian gradients' matrix: with N = sum_n rho_n lambda_n, M = N U^+ and
// G = L_exp(X, M), the Frechet derivative, on the blocks of H's components (where dH lies):
//   M' = N exp(-X'),  G = sum_n 1/(n+1)! sum_{j+k=n} X'^j M' X'^k
// (on a component's block the phase that exp(X) has over exp(X') is the one that U^+ takes
// away).  Each term is one sparse product from the left and one from the right.  work: 5 D x D.
void sparse_frechet(cudaStream_t s, const SparseX &x, const double2 *N, double2 *G, double2 *work);

// U = exp(X) by one pass over the columns of the identity.
void sparse_propagator(cudaStream_t s, const SparseX &x, double2 *U);

}  // namespace qed
