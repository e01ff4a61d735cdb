// FP64 supernode products on the tensor cores in a residue number system
// (rns.cu): device kernels' job description and the host-side schedule of one
// block of panels.
#pragma once

#include <cstdint>

#include "kernels.cuh"

namespace pexsi {

constexpr int kRnsModuli = 15;   // product of the moduli 2^117.8
constexpr int kRnsBlock = 256;   // most columns eliminated together (a block of panels)
constexpr int kRnsFronts = 128;  // fronts per launch (tile prefix sums travel as kernel arguments)
constexpr int kRnsGroup = 4;     // most blocks whose updates are applied together (a power of two)
constexpr int kRnsTile = 128;    // rows of an operand tile, edge of an output tile
constexpr int kRnsOutTile = kRnsTile * kRnsTile * kRnsModuli;  // residue bytes of a real output tile

// Columns of a block: whole panels of width b.
__host__ __device__ inline int rns_block(int b) { return kRnsBlock / b * b; }

// Scratch of the residue path: operand planes (slots of one 128-row tile each)
// and residue output tiles, both reused by every launch.
struct RnsScratch {
  uint8_t* planes = nullptr;
  int64_t plane_bytes = 0;
  uint8_t* out = nullptr;
  int64_t out_bytes = 0;
  int* fail = nullptr;
  uint64_t wait_ns = 0;
  int sms = 152;  // of the plan's device
  int hold = 0;   // fault injection: CTA 0 of every GEMM copies no operands
};

// Bytes of one operand slot: 128 rows x K (rounded up to 32) bf16 residues of
// every modulus (re and im planes for complex operands), and the row exponents.
inline int64_t rns_slot_bytes(int k, bool cplx) {
  return int64_t((k + 31) / 32) * 8192 * (cplx ? 2 : 1) * kRnsModuli + kRnsTile * int64_t(sizeof(int));
}

// Most complex output tiles of a launch. 160 of them (79 MB of residues) stay in
// L2, but launches with a nearly full last wave of items and half as many of
// them gain more: 640 against 160 gives 6.31 instead of 6.62 ms for a chain of
// 500 atoms, 48.0 instead of 49.2 for the counts of 256 in a fluid, 50.7 instead
// of 51.4 for a sheet. Where memory is short, the smaller number.
constexpr int kRnsOutTiles = 640, kRnsOutTilesLeast = 160;

cudaError_t rns_configure();

// Exponents of the symmetric scaling D A D, D = 2^-g, of A = H - z S for every
// shift of a batch: the residue products round each operand row relative to its
// norm, so rows and columns of one size are the premise of their accuracy (a
// power of two is exact, and FP64 multiply-adds do not see it). With a_c half the
// exponent of |A_cc|, and E_rc that of a bound of |A_rc|, max(|H_rc|, |z| |S_rc|),
//   g_c = max(a_c, max over r of min(E_rc - a_r, E_rc / 2)),
// the least for which no scaled entry is above 1 (2 with the rounding of halves)
// when each pair raises the row of the smaller diagonal: a graded matrix keeps
// its diagonal's scale, a diagonal entry far below its row (a level at the shift,
// a zero) does not blow the row up, and a weakly coupled level at the shift is
// scaled by its couplings. From A itself, not from H and S: where S = I and H is
// graded, the shift decides which of the two a row is made of. Within kRnsNear of
// half the exponent of max(|H_cc|, |S_cc|), g_c is that: the operands hold 5 bits
// more than FP64, and the scale then follows neither the shift nor a row's level,
// which made the inverse of ordinary systems 10-20% less accurate (24 atoms at Im
// z = 0.01: 6.9e-14 against 8.2e-14, geometric means of 40).
constexpr int kRnsNear = 5;

// For the n columns of one system (values HS components wide: 1 real, 2
// complex); colptr of its columns, diag of its columns in elimination order from
// c0 on, e0 its first entry; row, col and the exponents (g0, g: the members' of
// column c from c * stride on, a multiple of 8) of all systems in elimination
// order. h: half the exponents of max(|H_cc|, |S_cc|), by which the breakdown
// limit knows a row's own size before H and z S cancel. scaled: whether any
// exponent is not zero (of a group, set from its first system on).
void launch_rns_scales(const double* H, const double* S, int wide, const BatchShifts& sh, const int64_t* colptr,
                       const int64_t* diag, int64_t n, int64_t c0, int64_t e0, const int32_t* row, const int32_t* col,
                       int16_t* h, int16_t* g0, int16_t* g, int64_t stride, int* scaled, bool first, cudaStream_t st);

}  // namespace pexsi
