// Interface of the pair enumeration (swcs_pairs.cu) and of the density-matrix
// pool gradient built on it (swcs_rdm.cu).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "swcs_kernels.h"

namespace swcs {

// A determinant in grouped order: its string of the grouping spin, the other spin's, the amplitude in the
// spin-blocked convention.
struct __align__(16) PairRec {
  uint32_t own, oth;
  double amp;
};

// String table slot: string, number of determinants - 1, first one's place in the grouped order.
struct __align__(16) PairSlot {
  uint32_t key, cnt, off, pad;
};

struct PairCtl {
  unsigned long long alloc[2];  // per spin: items << 32 | determinants placed
  unsigned next;                // next item of the pair kernel
  unsigned next_row;            // next row of the contraction
};

struct PairArgs {
  HamDev H;
  int m;                 // spatial orbitals
  const uint64_t* keys;  // the state
  const double* amps;
  const long long* n;
  uint32_t cap;          // stride of the two spins' grouped arrays (at least n)
  PairSlot* tab;         // [2 (mask + 1)] string tables, alpha then beta
  uint32_t mask;
  uint32_t* slot_of;     // [2 cap]
  uint32_t* pos_of;      // [2 cap]
  PairRec* rec;          // [2 cap]
  uint32_t* oth;         // [2 cap]
  uint32_t* idx;         // [2 cap] place in the state | sign of the spin-blocked convention << 31 (energy only)
  uint4* items;          // [2 cap] string, first, count, block
  uint32_t blk;          // determinants per item, a power of two up to 32
  PairCtl* ctl;
  double* acc;           // [2] energy numerator, <psi|psi>
  double* sig;           // sigma_D in state order (nullptr: not wanted)
  int* err;
  // three-body density matrices <A+_T A_T'>, A_T annihilating T's orbitals in ascending order: mix[s] over
  // (one orbital of the other spin, pair of spin s), index orbital * m(m-1)/2 + pair; same[s] over triples of
  // spin s.  Pairs and triples in colex order.
  double* mix[2];
  double* same[2];
  size_t ld_mix, ld_same;
};

cudaError_t launch_pairs_energy(const PairArgs& a, int64_t n, int nsm, cudaStream_t st);
cudaError_t launch_pairs_gamma(const PairArgs& a, int64_t n, int nsm, cudaStream_t st);

// Tables of the Hamiltonian for the contraction, laid out once per Hamiltonian (m spatial orbitals, P = m(m-1)/2):
//   vss [2][m][P][m]     g(p s, x s; y s, z s), pair (y < z), at ((s m + x) P + pair) m + p
//   vos [2][m][m][m][m]  g(p s, x o; y o, z s), o = 1 - s, at (((s m + x) m + y) m + z) m + p
//   v2s [2][P][P]        g(p s, q s; y s, z s)
//   v2m [m^2][m^2]       g(p alpha, q beta; y alpha, z beta)
// with g(p, x; y, z) = <px||yz>.
struct RdmTables {
  double *vss, *vos, *v2s, *v2m;
};
size_t rdm_table_doubles(int m);
RdmTables rdm_tables(double* base, int m);
cudaError_t launch_rdm_tables(const double* g_full, int n, const RdmTables& t, cudaStream_t st);

struct RdmArgs {
  PairArgs P;            // the density matrices and the state's counters
  RdmTables V;
  const uint8_t* pool_ops;
  int64_t pool_size;
  double* s_ss;          // [2][P][m][m]    contraction, operator order (rs, q, p)
  double* s_ab;          // [m^2][m][m]     p alpha, q beta
  double* s_ba;          // [m^2][m][m]     p beta, q alpha
  double *g_ss, *g_ab;   // two-body density matrices [2][P][P], [m^2][m^2]
  double *w_ss, *w_ab;   // their contractions with the integrals
  double* gam;           // [2][m][m] one-body density matrix
  double* lam;           // [2][m][m] <a+_r K_p>
  double* g;             // the pool gradient
};
size_t rdm_work_doubles(int m);      // s_ss .. lam in one buffer
size_t rdm_gamma_doubles(int m);     // the four density matrices
void rdm_layout(RdmArgs& a, double* work, double* gamma, int m);
cudaError_t launch_rdm_gradient(const RdmArgs& a, int nsm, cudaStream_t st);

}  // namespace swcs
