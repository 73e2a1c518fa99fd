// Internal device-side definitions of the HFX library (not part of the C ABI).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "boys.cuh"

namespace hfx {

// ---------------------------------------------------------------------------
// Per-class recurrence description (generated tables, see gen_eri_tables.py)
// ---------------------------------------------------------------------------
struct EriClassInfo {
  int la, lb, lc, ld, E, F, Lt;
  int n_acc, work_base, scratch;       // group scratch (doubles): acc | VRR slots
  int n_bra_lv, n_ket_lv;
  int lv_off[8], lv_n[8];              // VRR levels: op offset (in uint4) and count
  int acc_off;                         // into kAccSrc: (acc index | slot << 16) entries
  int n_accl;                          // accumulators added after the levels (others are
                                       // accumulated by the op that makes them)
  int n_post;                          // post-contraction stages
  int post_type[8], post_off[8], post_n[8];  // 0 bra HRR, 1 ket HRR, 2 spherical
  int out_base;                        // final spherical block in group scratch
  int dims[4];                         // final block extents (a, b, c, d)
  int flops_prim, flops_quartet;       // flop model (VRR+acc per primitive quartet;
                                       // HRR+spherical+digest per contracted quartet)
  int flops_digest;                    // the digest part of flops_quartet (always FP64)
};

extern const EriClassInfo* class_info_host();

// Hermite engine (generated tables, see gen_md_tables.py): the steps of a class ...
struct MdClassInfo {
  int Lt;
  int kc, n_kc, bc, n_bc;              // contraction tables (first entry, entries)
  int n_row, nab, ncd;                 // rows of Y, function pairs of bra and ket
  int bra_coef0, bra_coef, bra_set;    // bra pair type: first coefficient, coefficients, sets
  int ket_coef, ket_set;
  int z1_round, z1_n, z1_dst, z2_round, z2_n, z2_dst;  // transformation passes
  int dig, dig_n;                      // digest (first round, rounds)
};
// ... and the sets and coefficients of a pair type (set: power of 1/2p | of u_b << 4 | of u_a << 8)
struct MdPairInfo {
  int coef0, n_coef, n_set;
  int set[14];
};
extern const MdClassInfo* md_class_host();
extern const MdPairInfo* md_pair_host();
// per class: flops per primitive quartet, per run of a bra primitive pair, per quartet, in its digest
extern const int (*md_flops_host())[4];

// ---------------------------------------------------------------------------
// Primitive-pair record (one per surviving primitive pair of a shell pair).
// C = sqrt(2) pi^{5/4} w_a w_b exp(-ab/p |AB|^2) / p so that the primitive
// quartet prefactor 2 pi^{5/2} K_ab K_cd / (p q sqrt(p+q)) = C_ab C_cd / sqrt(p+q).
// For a basis whose Hermite integrals could leave FP64's range (hfx_ctx::hexp, 0 for any other) C is held
// times 2^{hexp/2}; the transformation coefficients T of a pair (PairArrays::md) carry the inverse.
// ---------------------------------------------------------------------------
struct __align__(16) PrimPair {
  double p, inv2p;     // exponent sum and 1/(2p)
  double P[3];         // Gaussian product centre
  double PA[3];        // P - A (A = centre of the pair's first shell)
  double C;            // prefactor (see above)
  double inv2p3;       // 3/(2p)
  double ua, ub;       // a/p and b/p, a and b the exponents of the pair's two shells
  // FP32 copies for the FP32 recurrences
  float pf, inv2pf, PAf[3], Pf[3];
};

// Device arrays describing shell pairs (indexed by candidate-pair id).
struct PairArrays {
  const int* sa;            // first shell (l_a >= l_b)
  const int* sb;            // second shell
  const int* prim_off;      // first PrimPair of the pair
  const int* prim_n;        // number of surviving primitive pairs
  const double* AB;         // 3 per pair: A - B
  const PrimPair* prim;     // primitive-pair records
  const long long* md_off;  // first double of the pair's Hermite data in md: the coefficients T of its
  const double* md;         // type, then the factors W of every surviving primitive pair
};

struct ShellArrays {
  const int* bf_off;        // first function of each shell
  const int* atom;          // atom of each shell
};

// Lattice images (periodic builds): the library holds the home cell's shells repeated in a
// box of cells (the image shells, cell-major, the home cell first); every pair of the pair
// list has one shell in the home cell (list-IJ anchored in the home cell, Sec. 3.1).
struct PerCell;
struct PeriodicInfo {
  const int* shell_cell;            // image shell -> cell index (0 = home cell)
  const int* shell_bf;              // image shell -> first function in the home-cell numbering
  const int* cell_xyz;              // cell index -> integer cell coordinates (3 each)
  const unsigned char* home_first;  // candidate pair -> 1 if its first shell is the home-cell one
  const int* rmap;                  // density block index of cell R (-1: absent), R in [-rb, rb]^3
  int rb;
  const double* P;                  // density blocks P^R, n_R x nbf x nbf
  int nbf;
  const double* pmax;               // max |P^R| per (R, home shell, home shell): n_R x nsh x nsh
  int nsh;                          // shells of the home cell
  const PerCell* cells;             // the launch's passes over the quartet list of the class
  long long n_list;                 // quartets of the list
};

// A pass over the list of a class: quartets (bra | ket + shift) of cell G; reverse = 0: the bra pair
// carries the row function of K^G, 1: the ket pair does (the pass then evaluates (q | p - G L) for
// the quartet (p | q + G L) of a lower bra class)
struct PerCell {
  double shift[3];
  double* KG;  // K^G, nbf x nbf
  int gcell[3];
  int reverse;
};

// Arguments of one class launch (passed by value).
struct EriLaunch {
  EriClassInfo ci;
  PairArrays pa;
  ShellArrays sh;
  const int* sorted;          // sorted pair index -> candidate-pair id
  const long long* qoff;      // exclusive scan of quartets per row (global), + total
  int row_begin, row_end;     // rows of this class pair
  int bra_bin_start, ket_bin_start;
  long long q_begin, q_count; // quartet range of this class pair
  int schedule;               // 0 quartet split, 1 bra-pair split, 2 dynamic chunks
  unsigned long long* work;   // schedule 2: next unclaimed quartet (relative to q_begin)
  int chunk;                  // schedule 2: quartets per claim
  const double* boys;         // Boys and exp tables (boys.cuh)
  double omega, omega2;
  MdClassInfo mc;              // Hermite engine: the steps of this class
  int prec;                    // precision pass (PREC_*)
  const double* P;
  double* K;
  int ld;
  // Schwarz-diagonal mode: quartet (p|p) for candidate pairs [diag_begin, diag_end)
  const int* diag_list;
  int diag_n;
  double* diag_Q;
  unsigned long long* busy;     // optional per-SM globaltimer busy ns (indexed by %smid)
  unsigned long long* counters; // optional: [0] primitive quartets evaluated, [1] quartets, [2] skipped
  const double* pmax;           // optional: max |P| of each shell-pair block (ns x ns)
  int ns;
  int skip_zero;                // skip quartets whose four density blocks are all zero
  int fp32_ok;                  // mixed precision allowed for this class
  double fp32_tau;              // FP32 iff Q_IJ Q_KL Pmax < fp32_tau, Pmax = max|P_blocks| ...
  const double* pglob;          // ... or, when non-NULL, *pglob = max |P| over the matrix
  double dens_tau;              // > 0: drop quartets with Q_IJ Q_KL max|P_blocks| < dens_tau
  double dist_tau;              // > 0: drop quartets with Q_IJ Q_KL exp(-kappa rho R^2) < dist_tau
  const double* dist;           // per sorted pair: most diffuse primitive-pair centre (3), spread,
                                // smallest exponent sum (5 doubles)
  const double* Qs;             // Schwarz factor of each sorted pair
  // batched launch (n_sys > 0): quartets of all systems' lists for this class, concatenated;
  // seg[s] = first index of system s (seg[n_sys] = total = q_count); batch[s] = that
  // system's record for this class (device memory)
  int n_sys;
  const long long* seg;
  const EriLaunch* batch;
  // periodic launch: the list of the class once for each of per.cells (q_count = all of them)
  PeriodicInfo per;
  double unscale;             // 2^-hexp (see PrimPair::C): the thread kernel's factor for its integrals
};


}  // namespace hfx
