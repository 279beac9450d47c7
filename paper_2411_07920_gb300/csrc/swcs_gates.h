// Interface of the in-place gate sequence (swcs_gates.cu) and of the adjoint over its tape.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "swcs_kernels.h"

namespace swcs {

constexpr int kGateThreads = 1024;
constexpr int kGateCtrN = 8;
// Bins around the previous cut, counted while the gate's pass writes the amplitudes; the first band_slots entries
// of each bin are kept with it.  Three sets, one per gate in turn.
constexpr int kBandBins = 8192, kBandGroups = 64;
constexpr int kBandShift = 38;  // a bin is 2^38 units of the bit pattern: 2^-14 to 2^-15 of the cut, the band 12 to 25 % around it
constexpr size_t kBandWords = kBandBins + kBandGroups;
constexpr size_t kGateHistWords = (size_t)12 * 4096;  // digits of the general select
struct __align__(16) BandEntry {
  unsigned long long x, key;  // |c| as bits, bitstring
};

// What a pass recorded of its gate: pairs of the two-determinant blocks it rotated (positions, amplitudes before),
// and the positions dropped by the truncation before it.
struct GateTape {
  uint2* pos;     // lower's position | phase bit << 31, upper's position (all ones: not in the work arrays)
  double2* x;     // amplitudes of lower and upper before the gate (0: not in the state)
  uint32_t* drop;
  unsigned long long* start;  // [2 (n_ops + 1)] first record and first drop of each gate's pass
  unsigned long long cap, drop_cap;
};
constexpr uint32_t kNoPos = 0xFFFFFFFFu;

struct GateArgs {
  const uint64_t* in_keys;  // input state, compact (unless reset_to_hf)
  const double* in_amps;
  uint64_t* out_keys;       // output state, compact (may be the input arrays)
  double* out_amps;
  uint32_t* out_pos;        // optional: position of each output determinant in the work arrays
  uint64_t* keys;           // work arrays of `cap` positions: every determinant keeps its position while it lives
  double* amp[2];
  uint32_t cap;
  uint64_t* tab;            // index slots (16-byte aligned)
  uint64_t tab_mask;
  IdxSlot* plain;           // output index in the plain form
  uint64_t plain_mask;
  uint64_t* low_keys;       // partners too small to be kept, most likely (this gate's, cap_low of them)
  double* low_amps;
  uint32_t* low_rec;
  uint32_t cap_low;
  uint32_t* ring;           // free positions
  uint32_t ring_mask;
  const uint8_t* ops;
  const double* cs;
  int n_ops;
  int64_t n_keep;
  uint64_t min_abs_bits;
  int reset_to_hf;
  uint64_t hf;
  long long* n_state;
  unsigned long long* ctr;  // [3 kGateCtrN + 1]
  unsigned* hist;           // kGateHistWords
  unsigned* band;           // [3 kBandWords]
  BandEntry* band_ent;      // [3 kBandBins band_slots]
  int band_slots;           // at most 32
  GridBar* bar;
  int* err;
  uint64_t timeout_ns;
  int skip_arrive_block;
  long long* stats;
  unsigned long long* probe_ctr;
  GateTape tape;            // pos == nullptr: no tape
};

// CTAs of one cluster that the device can hold (0: none of that size).
int gate_cluster_fits(int ctas);
int gate_blocks_per_sm();
// clustered: nblocks CTAs in one cluster (hardware barrier), else a cooperative grid.
cudaError_t launch_gates(const GateArgs& a, int nblocks, bool clustered, cudaStream_t st);

// nu of the final state at its positions: nu[out_pos[i]] = sigma_i - E c_i (everything else 0 before).
// zeros: counts the exactly zero amplitudes that the projectors kept.
cudaError_t launch_nu_final(const double* amps, const double* sigma, const uint32_t* out_pos, const long long* n,
                            const double* acc, double* nu, unsigned long long* zeros, cudaStream_t st);
// nu at the positions of a replayed segment's end from nu over the checkpoint that follows it.
cudaError_t launch_nu_realign(const uint64_t* keys, const uint32_t* out_pos, const long long* n, const IdxSlot* tab,
                              uint64_t mask, const double* nu_ck, double* nu, cudaStream_t st);
struct BackArgs {
  GateTape tape;
  const double* cs;   // the segment's gates
  int n_ops;
  double* nu;         // [positions]
  double* dtheta;     // [n_ops], zeroed
  GridBar* bar;
  int* err;
  uint64_t timeout_ns;
};
cudaError_t launch_back(const BackArgs& a, int nblocks, bool clustered, cudaStream_t st);
int back_blocks_per_sm();

}  // namespace swcs
