// FP64 supernode products on the tcgen05 tensor cores in a residue number
// system (the Chinese-remainder form of the Ozaki scheme: Ozaki, Uchino and
// Imamura 2025), FP64 in and out.
//
// Why: an SM issues 2 FP64 multiply-adds per clock (1.26 TFLOP/s on the chip,
// DMMA no faster), its bf16 tensor cores 4096. Each operand row is scaled by a
// power of two above its 2-norm and rounded to integers of 58 bits; the
// integers' residues modulo 15 pairwise coprime moduli p <= 256 are exact in
// bf16 (|r| <= 128), so the product modulo every p is one bf16 GEMM whose FP32
// accumulators hold exact integers (2 x 480 products of at most 2^14 stay
// below 2^24), and the 15 residues give the exact integer product (below
// 2^116, half the product of the moduli is 2^116.4) by the remainder theorem.
// The only errors are the rounding of the operands (2^-59 of the row norms,
// against the 2^-53 of each FP64 multiply-add) and of the result. A complex
// product costs 15 x 4 bf16 multiply-adds per complex multiply-add, against
// 45 x 4 for bf16 slices of the same accuracy (9 slices of 7 bits).
//
// Three kernels per product C = A B^T of rows of A (the N operand of the MMA:
// rows of the front) and rows of B (the M operand: panel columns):
//   k_rns_conv   row norms, integers and residues of an operand (HBM bound:
//                16 B read, 60 B written per complex entry)
//   k_rns_gemm   one bf16 GEMM per modulus, residues of C as bytes (tensor
//                bound)
//   k_rns_recon  the integers of C, their FP64 values and the update of F or Y
//                (integer pipe bound: about 130 operations per real entry)
//
// The fronts are eliminated in blocks of kRnsBlock = 256 columns (against the
// panels of the DFMA path): the 256 x 256 diagonal block B is inverted by
// symmetric sweeps over its panels (launch_diag_inv per panel, the rest as
// residue products), L[S,B] = W[S,B] B^-1 is one product, F[S,S] -= L W^T goes in
// groups of blocks (Update), and Y[S,B] = -Y[S,S] L[S,B] converts Y[S,S] once
// per 256 columns.
#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "plan.hpp"
#include "rns.cuh"
#include "tensor_core.cuh"

namespace pexsi {
namespace {

// ------------------------------------------------------------ moduli
typedef unsigned __int128 u128;
typedef __int128 i128;

// Pairwise coprime, largest first. 255 is left out: the FP32 quotient by it may
// round the other way for accumulators near 2^24, and the residue 128 would not
// fit its byte (256 has an exact reciprocal, and 128 = -128 modulo it).
__host__ __device__ constexpr int modulus(int l) {
  constexpr int t[kRnsModuli] = {256, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};
  return t[l];
}
__host__ __device__ constexpr u128 mod_product() {
  u128 p = 1;
  for (int l = 0; l < kRnsModuli; ++l) p *= u128(modulus(l));
  return p;
}
// P / p_l, and its inverse modulo p_l (folded into one operand's residues)
__host__ __device__ constexpr u128 cofactor(int l) { return mod_product() / u128(modulus(l)); }
__host__ __device__ constexpr int cofactor_inv(int l) {
  const int p = modulus(l), c = int(cofactor(l) % u128(p));
  for (int x = 1; x < p; ++x)
    if (c * x % p == 1) return x;
  return 0;
}
// residue of 2^(15 j) (times the inverse of the cofactor) in [-p/2, p/2]
__host__ __device__ constexpr int piece_coef(int l, int j, bool scaled) {
  const int p = modulus(l);
  long long r = 1;
  for (int q = 0; q < 15 * j; ++q) r = r * 2 % p;
  if (scaled) r = r * cofactor_inv(l) % p;
  return int(r > p / 2 ? r - p : r);
}
// limbs of the cofactors: 20 bits (sums of 15 byte multiples stay below 2^32), then 32, 32 and the rest
__host__ __device__ constexpr uint32_t limb(u128 v, int j) {
  return j == 0 ? uint32_t(v & 0xFFFFF) : j == 1 ? uint32_t(v >> 20) : j == 2 ? uint32_t(v >> 52) : uint32_t(v >> 84);
}
// The residues are stored as r + 128, so the sum of the bytes times the cofactors
// exceeds the integer by 128 times the sum of the cofactors and a multiple of P:
// limbs of what is added to it to leave the integer plus a non-negative multiple.
__host__ __device__ constexpr u128 byte_bias() {
  u128 s = 0;
  for (int l = 0; l < kRnsModuli; ++l) s = (s + 128 * (cofactor(l) % mod_product())) % mod_product();
  return 2 * mod_product() - s;
}

constexpr int kBeta = 58;       // bits of the scaled integers
constexpr int kNanRow = 0x7FFF; // exponent marker of a row holding Inf or NaN
constexpr int kK = 32;          // K per staged tile
constexpr int kPlane = kRnsTile * kK * 2;  // bytes of a 128 x 32 residue tile
constexpr int kChunkTiles = 15;            // 480 of K: 2 x 480 x 2^14 + 2^7 < 2^24
constexpr int kStages = 6;
constexpr int kEpi = 8;                    // epilogue warps: 4 lane quarters x (re, im)
constexpr int kThreads = (kEpi + 2) * 32;
constexpr int kItems = 128;                // most items of a CTA (a table in shared memory); a multiple of 32
constexpr int gemm_smem(bool cplx) { return kStages * 2 * (cplx ? 2 : 1) * kPlane; }
static_assert(mod_product() >> 117 == 1, "the bound on the integer products needs 2^117 <= P < 2^118");
static_assert(2 * kChunkTiles * kK * 128 * 128 + 128 < (1 << 24), "the FP32 accumulators stay exact");

// ------------------------------------------------------------ jobs
// Products (rows of N x rows of M, contraction K) of one block of panels
// [p0, p0 + bw), bw = min(rns_block, s - p0), S = the mp rows below it:
enum Mode {
  kSweepT,  // T = V D^-1: V = B[:,p] of the diagonal block B, D^-1 = its inverted panel block
  kSweepU,  // B[R,R] -= T V^T, R = the block's rows outside the panel p
  kResid,   // R = I - B X, X = the swept inverse, B = the block as it was (kept in Y, which takes R)
  kRefine,  // X += X R
  kPanel,   // L[S,B] = W[S,B] B^-1
  kSchur,   // F[S,C] -= L W^T (lower triangle; C and the columns of L and W: Update)
  kTak,     // Y[S,B] = -Y[S,S] L[S,B] and its mirror
  kDiag,    // Y[B,B] = B^-1 - L[S,B]^T Y[S,B]
  // LDU fronts (gen): whole squares, no mirrors, the block's plain inverse in place of its negative
  // during the sweeps, and the row panels
  kSweepDU, // B[p,R] = D^-1 U, U = B[p,R]
  kPanelU,  // U[B,S] = B^-1 A[B,S]
  kTakU     // Y[B,S] = -U[B,S] Y[S,S]
};
// Operands of k_rns_conv.
enum Operand {
  kOpV, kOpD, kOpT, kOpR, kOpW, kOpB, kOpL, kOpLt, kOpY, kOpYt,
  // LDU fronts: rows of D^-1, B, B^-1, Y[S,S] and U[B,S]; columns of U, R, A[B,S], Y[S,S] and Y[S,B]
  kOpDr, kOpBr, kOpXr, kOpYr, kOpUr, kOpU, kOpRc, kOpA, kOpYc, kOpYtc,
  // W[C,.] and A[.,S] of several blocks, kept in Y
  kOpWs, kOpAs
};

struct Job {
  int mode, gen;             // gen: LDU fronts
  int nf, np, pole0;         // nf fronts of the level's list, poles pole0 .. pole0 + np - 1
  int p0, pc, b;             // block start, panel start inside the block (sweeps), panel width
  int rt0, mt0;              // first tile of N or M (a front whose row tiles are taken in pieces)
  int o0, on;                // output tiles of this launch
  int kt, nkt;               // K tiles of a slot, of every item (0: they differ)
  int g0, k0, width;         // kSchur: first column of the block's group, of its update, columns updated (0: all)
  int64_t slot, n_base, m_base;
  int pref_n[kRnsFronts + 1], pref_m[kRnsFronts + 1], pref_o[kRnsFronts + 1];
  // the fronts' sizes and places: as kernel arguments they cost no chain of global loads per item or block
  int s[kRnsFronts], m[kRnsFronts];
  int64_t off[kRnsFronts], pool;
};

static_assert(sizeof(Job) <= 3968, "kernel arguments hold 4 KiB");

struct Dims {
  int s, m, bw, q0, mp, pb;
};

__host__ __device__ __forceinline__ Dims dims_of(int s, int m, int p0, int pc, int b) {
  Dims d;
  d.s = s;
  d.m = m;
  const int blk = rns_block(b);
  d.bw = s - p0 < blk ? s - p0 : blk;
  d.q0 = p0 + d.bw;
  d.mp = m - d.q0;
  d.pb = d.bw - pc < b ? d.bw - pc : b;
  return d;
}

// The update after the block at p0: which columns it reaches (the first `cols`
// of S, and for LDU fronts the rows alike) and which eliminated ones it applies
// (K of them from k0 on). Blocks come in groups of up to kRnsGroup. After the
// i-th block of a group the last b = i & -i blocks are applied to the next b
// blocks' columns; after the group's last block, or the front's, the group is
// applied to all of S. Each column so gets each block once, and most of the
// front is read, updated and written once per group instead of once per block.
struct Update {
  int k0, k, cols;
};

__host__ __device__ __forceinline__ Update update_of(const Dims& d, int g0, int k0, int width) {
  Update u;
  const bool all = width == 0 || d.q0 == d.s;
  u.k0 = all ? g0 : k0;
  u.k = d.q0 - u.k0;
  u.cols = all ? d.mp : (d.s - d.q0 < width ? d.s - d.q0 : width);
  return u;
}

__host__ __device__ __forceinline__ int tiles128(int n) { return n <= 0 ? 0 : (n + kRnsTile - 1) / kRnsTile; }

// rows of N, rows of M, K of a product; sweeps skip blocks of one panel
__host__ __device__ __forceinline__ void product_dims(const Job& j, const Dims& d, int& rn, int& rm, int& k) {
  const int b = j.b;
  switch (j.mode) {
    case kSweepT: rn = d.bw > b && d.pb > 0 ? d.bw : 0; rm = rn ? d.pb : 0; k = d.pb; break;
    case kSweepU: rn = rm = d.bw > b && d.pb > 0 ? d.bw : 0; k = d.pb; break;
    case kResid: case kRefine: rn = rm = d.bw > b ? d.bw : 0; k = d.bw; break;
    case kPanel: rn = d.mp; rm = d.mp > 0 ? d.bw : 0; k = d.bw; break;
    case kSchur: {
      const Update u = update_of(d, j.g0, j.k0, j.width);
      rn = d.mp;
      rm = j.gen ? d.mp : u.cols;
      k = u.k;
      break;
    }
    case kSweepDU: rm = d.bw > b && d.pb > 0 ? d.bw : 0; rn = rm ? d.pb : 0; k = d.pb; break;
    case kPanelU: rn = d.mp > 0 ? d.bw : 0; rm = d.mp; k = d.bw; break;
    case kTakU: rn = d.mp > 0 ? d.bw : 0; rm = d.mp; k = d.mp; break;
    case kTak: rn = d.mp; rm = d.mp > 0 ? d.bw : 0; k = d.mp; break;
    default: rn = rm = d.bw; k = d.mp; break;
  }
}

__host__ __device__ __forceinline__ bool triangular(int mode, int gen) {
  return !gen && (mode == kSweepU || mode == kRefine || mode == kSchur || mode == kDiag);
}

// whether an operand is the M one of its products, and whether the cofactors' inverses go into its residues
__host__ __device__ __forceinline__ bool m_side(int op) {
  return op == kOpD || op == kOpB || op == kOpLt || op >= kOpU;
}
__host__ __device__ __forceinline__ bool scaled_op(int op) {
  return op == kOpD || op == kOpT || op == kOpB || op == kOpL || op == kOpLt || op == kOpDr || op == kOpXr || op == kOpUr;
}

// largest f with pref[f] <= t
__host__ __device__ __forceinline__ int owner(const int* pref, int n, int t) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pref[mid] <= t) lo = mid;
    else hi = mid;
  }
  return lo;
}

struct OutTile {
  int pole, f, nt, mt;  // pole and front list index of the job, tile of N, tile of M
};

__host__ __device__ __forceinline__ OutTile out_tile(const Job& j, int o) {
  OutTile t;
  const int per = j.pref_o[j.nf];
  t.pole = o / per;
  const int x = o - t.pole * per;
  t.f = owner(j.pref_o, j.nf, x);
  const int y = x - j.pref_o[t.f];
  // the tiles of M that an update reaches: a trapezoid, for LDU fronts the rows beyond them alike
  int tm = j.pref_m[t.f + 1] - j.pref_m[t.f];
  if (j.mode == kSchur) tm = tiles128(update_of(dims_of(j.s[t.f], j.m[t.f], j.p0, j.pc, j.b), j.g0, j.k0, j.width).cols);
  const int tri = tm * (tm + 1) / 2;
  if (triangular(j.mode, j.gen) && (j.mode != kSchur || y < tri)) {
    int i = int((sqrtf(8.0f * float(y) + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > y) --i;
    while ((i + 1) * (i + 2) / 2 <= y) ++i;
    t.nt = i;
    t.mt = y - i * (i + 1) / 2;
  } else if (j.mode == kSchur) {
    const int tn = j.pref_n[t.f + 1] - j.pref_n[t.f], z = j.gen ? y : y - tri;
    if (!j.gen) {
      t.nt = tm + z / tm;
      t.mt = z - (t.nt - tm) * tm;
    } else if (z < tn * tm) {
      t.nt = z / tm;
      t.mt = z - t.nt * tm;
    } else {
      const int w = z - tn * tm, side = tn - tm;
      t.nt = w / side;
      t.mt = tm + w - t.nt * side;
    }
  } else {
    // Y[B,B] of a front without rows below it has no operands, and one tile or two by two
    int mtn = j.pref_m[t.f + 1] - j.pref_m[t.f];
    if (mtn == 0) mtn = j.pref_o[t.f + 1] - j.pref_o[t.f] > 1 ? 2 : 1;
    t.nt = y / mtn;
    t.mt = y - t.nt * mtn;
  }
  return t;
}

// ------------------------------------------------------------ conversion
template <typename F, int... L>
__device__ __forceinline__ void each_modulus(F&& f, std::integer_sequence<int, L...>) {
  (f(std::integral_constant<int, L>{}), ...);
}
template <typename F>
__device__ __forceinline__ void each_modulus(F&& f) {
  each_modulus(f, std::make_integer_sequence<int, kRnsModuli>{});
}

// The integer nearest to x 2^(58 - e) (|x| < 2^e) as four floats: 15-bit
// pieces from the low end, the top one signed (two's complement).
__device__ __forceinline__ void pieces(double x, int e, float (&p)[4]) {
  const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
  const int E = int((hi >> 20) & 0x7FF);
  const uint32_t mh = (hi & 0xFFFFFu) | (E ? 0x100000u : 0u);
  const unsigned long long mant = (static_cast<unsigned long long>(mh) << 32) | lo;
  const int n = 1022 + e - (E ? E : 1);  // >= 0
  const unsigned long long t = n > 63 ? 0ull : (mant << 6) >> n;
  long long X = static_cast<long long>((t + 1) >> 1);
  if (int(hi) < 0) X = -X;
  const uint32_t xl = uint32_t(X), xh = uint32_t(static_cast<unsigned long long>(X) >> 32);
  p[0] = __uint_as_float(0x4B000000u | (xl & 0x7FFFu)) - 8388608.0f;
  p[1] = __uint_as_float(0x4B000000u | ((xl >> 15) & 0x7FFFu)) - 8388608.0f;
  p[2] = __uint_as_float(0x4B000000u | (__funnelshift_r(xl, xh, 30) & 0x7FFFu)) - 8388608.0f;
  p[3] = __int_as_float(0x4B400000 + (int(xh) >> 13)) - 12582912.0f;
}

__device__ __forceinline__ uint32_t bf16x2(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// Coefficients of the four pieces, plain and scaled, the modulus and its reciprocal.
struct PieceTable {
  float c[2][kRnsModuli][6];
};
constexpr PieceTable piece_table() {
  PieceTable t = {};
  for (int s = 0; s < 2; ++s)
    for (int l = 0; l < kRnsModuli; ++l) {
      for (int k = 0; k < 4; ++k) t.c[s][l][k] = float(piece_coef(l, k, s != 0));
      t.c[s][l][4] = float(modulus(l));
      t.c[s][l][5] = 1.0f / float(modulus(l));
    }
  return t;
}
__constant__ PieceTable c_piece = piece_table();

// Residues of 8 consecutive k of one row: one 16-byte word per modulus. The
// sum of pieces times coefficients is an exact integer below 2^24 in FP32, its
// quotient by p is rounded by the add of 1.5 2^23, and the residue is exact. A
// loop over the moduli, since all of them in line, for both kinds and parts, were
// 70 KB of instructions that the warps waited for.
__device__ __forceinline__ void store_residues(const float (&p)[8][4], bool scaled, uint8_t* dst, int64_t step) {
  const float(*tab)[6] = c_piece.c[scaled ? 1 : 0];
#pragma unroll 5
  for (int l = 0; l < kRnsModuli; ++l) {
    const float c0 = tab[l][0], c1 = tab[l][1], c2 = tab[l][2], c3 = tab[l][3], pm = tab[l][4], inv = tab[l][5];
    float r[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float t = p[u][0] * c0;
      t = fmaf(p[u][1], c1, t);
      t = fmaf(p[u][2], c2, t);
      t = fmaf(p[u][3], c3, t);
      const float q = fmaf(t, inv, 12582912.0f) - 12582912.0f;
      r[u] = fmaf(q, -pm, t);
    }
    *reinterpret_cast<uint4*>(dst) =
        make_uint4(bf16x2(r[0], r[1]), bf16x2(r[2], r[3]), bf16x2(r[4], r[5]), bf16x2(r[6], r[7]));
    dst += step;
  }
}

// |x| as a float, rounded down; 0 below the float range, garbage above it
// (rows of such magnitude take the bound by their largest entry).
__device__ __forceinline__ float abs_float(uint32_t hi, uint32_t lo) {
  const uint32_t a = hi & 0x7FFFFFFFu;
  return a < (897u << 20) ? 0.0f : __uint_as_float(((a - (896u << 20)) << 3) | (lo >> 29));
}

// Row exponent: 2^e above the 2-norm of the row, from the FP32 sum of squares
// (2% margin for its rounding), or for magnitudes whose squares leave the FP32
// range from the largest entry and the entry count.
__device__ __forceinline__ int row_exponent(uint32_t mx, float sum, int count) {
  if (mx >= 0x7FF00000u) return kNanRow;
  if (mx == 0) return 0;
  const int e = int(mx >> 20) - 1022;  // 2^e above the largest entry
  if (e > 40 || e < -40) return e + (32 - __clz(count)) / 2 + 1;
  const int e2 = int(__float_as_uint(sum * 1.02f) >> 23) - 126;  // 2^e2 above the sum
  return (e2 + 1) >> 1;
}

// One operand (or two, the second by the blocks from nblk_a on) of a job into
// its slots. A block of 256 threads takes 32 / OC groups of 8 rows: thread (row
// r = tid % 8, octet o of OC) reads entries 8 o .. 8 o + 7 of its row, twice
// when K > 8 OC (norm, then residues).
// Three blocks to an SM where their registers
// fit without spilling (real values, and short rows with the parts in turn:
// a 500-atom chain 6.35 -> 6.23 ms, inertia 48.1 -> 47.4 ms); complex long rows
// keep two (three: 57.5 -> 58.8 ms for 512 atoms).
template <typename T, int OC>
__global__ void __launch_bounds__(256, (sizeof(T) == 16 && OC == 32) ? 2 : 3) k_rns_conv(const T* __restrict__ F, const T* __restrict__ Y,
                                                     const __grid_constant__ Job j,
                                                     uint8_t* __restrict__ planes, int op_a, int nblk_a, int op_b) {
  constexpr bool CPLX = sizeof(T) == 16;
  constexpr int G = 32 / OC;  // row groups per block
  const bool second = int(blockIdx.x) >= nblk_a;
  const int op = second ? op_b : op_a;
  const int blk = second ? int(blockIdx.x) - nblk_a : int(blockIdx.x);
  const bool ms = m_side(op);
  const int* pref = ms ? j.pref_m : j.pref_n;
  const int per = pref[j.nf];
  const int sub = threadIdx.x / (8 * OC);
  const int grp = blk * G + sub;             // 8-row group in the launch
  const int flat = grp >> 4;                 // slot
  const bool in = flat < per * j.np;
  __shared__ float s_sum[8][8];
  __shared__ uint32_t s_max[8][8];
  const int r = threadIdx.x & 7, o0 = (threadIdx.x / 8) % OC;
  const int warp = threadIdx.x >> 5;
  Dims d = {};
  int rows = 0, K = 0, row = 0;
  const T* src = nullptr;
  int64_t sk = 0;
  if (in) {
    const int pole = flat / per, x = flat - pole * per, fi = owner(pref, j.nf, x);
    d = dims_of(j.s[fi], j.m[fi], j.p0, j.pc, j.b);
    const int rt = x - pref[fi] + (ms ? j.mt0 : j.rt0);
    row = rt * kRnsTile + (grp & 15) * 8 + r;
    const int64_t base = int64_t(j.pole0 + pole) * j.pool + j.off[fi], m = d.m;
    int64_t si = 1;
    const Update up = update_of(d, j.g0, j.k0, j.width);
    switch (op) {
      case kOpV: case kOpT: src = F + base + j.p0 + m * (j.p0 + j.pc); rows = d.bw; K = d.pb; sk = m; break;
      case kOpD: src = F + base + (j.p0 + j.pc) + m * (j.p0 + j.pc); rows = K = d.pb; si = m; sk = 1; break;
      case kOpR: case kOpRc: src = Y + base + j.p0 + m * j.p0; rows = K = d.bw; si = m; sk = 1; break;
      case kOpW: src = F + base + d.q0 + m * j.p0; rows = d.mp; K = d.bw; sk = m; break;
      case kOpL: src = F + base + d.q0 + m * up.k0; rows = d.mp; K = up.k; sk = m; break;
      case kOpWs: src = Y + base + d.q0 + m * up.k0; rows = up.cols; K = up.k; sk = m; break;
      case kOpAs: src = Y + base + up.k0 + m * d.q0; rows = d.mp; K = up.k; si = m; sk = 1; break;
      case kOpB: src = F + base + j.p0 + m * j.p0; rows = K = d.bw; si = m; sk = 1; break;
      case kOpLt: src = F + base + d.q0 + m * j.p0; rows = d.bw; K = d.mp; si = m; sk = 1; break;
      case kOpY: case kOpYc: src = Y + base + d.q0 + m * d.q0; rows = K = d.mp; si = m; sk = 1; break;
      case kOpDr: src = F + base + (j.p0 + j.pc) + m * (j.p0 + j.pc); rows = K = d.pb; sk = m; break;
      case kOpBr: src = Y + base + j.p0 + m * j.p0; rows = K = d.bw; sk = m; break;
      case kOpXr: src = F + base + j.p0 + m * j.p0; rows = K = d.bw; sk = m; break;
      case kOpYr: src = Y + base + d.q0 + m * d.q0; rows = K = d.mp; sk = m; break;
      case kOpUr: src = F + base + j.p0 + m * d.q0; rows = d.bw; K = d.mp; sk = m; break;
      case kOpU: src = F + base + (j.p0 + j.pc) + m * j.p0; rows = d.bw; K = d.pb; si = m; sk = 1; break;
      case kOpA: src = F + base + j.p0 + m * d.q0; rows = d.mp; K = d.bw; si = m; sk = 1; break;
      default: src = Y + base + d.q0 + m * j.p0; rows = d.bw; K = d.mp; si = m; sk = 1; break;  // kOpYt, kOpYtc
    }
    src += si * row;
  }
  chain_next();
  chain_begin(src);
  const bool row_in = in && row < rows;
  auto load = [&](int o, double (&re)[8], double (&im)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = o * 8 + u;
      re[u] = im[u] = 0.0;
      if (row_in && k < K) {
        if constexpr (CPLX) {
          const double2 v = src[sk * k];
          re[u] = v.x;
          im[u] = v.y;
        } else {
          re[u] = src[sk * k];
        }
      }
    }
  };
  double re[8], im[8];
  float sum = 0.0f;
  uint32_t mx = 0;
  const int no = (K + 31) / 32 * 4;  // octets of the padded row
  for (int o = o0; o < no; o += OC) {
    load(o, re, im);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t hr = uint32_t(__double2hiint(re[u])), hm = uint32_t(__double2hiint(im[u]));
      mx = max(mx, max(hr & 0x7FFFFFFFu, hm & 0x7FFFFFFFu));
      const float a = abs_float(hr, uint32_t(__double2loint(re[u])));
      sum = fmaf(a, a, sum);
      if (CPLX) {
        const float c = abs_float(hm, uint32_t(__double2loint(im[u])));
        sum = fmaf(c, c, sum);
      }
    }
  }
  // over the octets of a row: lanes 8 and 16 apart, then the group's OC / 4 warps
#pragma unroll
  for (int s = 8; s < 32; s <<= 1) {
    sum += __shfl_xor_sync(0xFFFFFFFFu, sum, s);
    mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, s));
  }
  if ((threadIdx.x & 31) < 8) {
    s_sum[warp][r] = sum;
    s_max[warp][r] = mx;
  }
  __syncthreads();
  if (!row_in && (!in || (row & ~7) >= rows)) return;  // whole groups of rows past the operand
  sum = 0.0f;
  mx = 0;
  const int w0 = sub * (OC / 4);
#pragma unroll
  for (int w = 0; w < OC / 4; ++w) {
    sum += s_sum[w0 + w][r];
    mx = max(mx, s_max[w0 + w][r]);
  }
  const int e = row_exponent(mx, sum, CPLX ? 2 * K : K);
  uint8_t* slot = planes + (ms ? j.m_base : j.n_base) + int64_t(flat) * j.slot;
  if (o0 == 0) reinterpret_cast<int*>(slot + j.slot - kRnsTile * sizeof(int))[row & (kRnsTile - 1)] = e;
  const bool scaled = scaled_op(op);
  const int ex = e == kNanRow ? 4000 : e;  // a row with Inf or NaN gives zeros here and NaN in the results
  const int64_t step = int64_t(j.kt) * (CPLX ? 2 : 1) * kPlane;
  const bool again = no > OC;
  for (int o = o0; o < no; o += OC) {
    if (again) load(o, re, im);
    uint8_t* dst = slot + int64_t(o >> 2) * ((CPLX ? 2 : 1) * kPlane) + ((row & (kRnsTile - 1)) >> 3) * 512 +
                   (o & 3) * 128 + r * 16;
#pragma unroll (CPLX && OC == 8 ? 1 : 2)
    for (int c = 0; c < (CPLX ? 2 : 1); ++c) {
      float p[8][4];
#pragma unroll
      for (int u = 0; u < 8; ++u) pieces(c ? im[u] : re[u], ex, p[u]);
      store_residues(p, scaled, dst + c * kPlane, step);
    }
  }
}

// ------------------------------------------------------------ GEMM
__constant__ float c_mod[kRnsModuli] = {256, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

// Persistent: CTA x walks the (modulus, output tile) items x, x + gridDim.x,
// ... (moduli outermost: the operand planes of one modulus stay in L2). Warp 8
// streams K tiles of both operands (one bulk copy each, 6 stages of 32 KiB),
// warp 9 issues the MMAs, warps 0-7 reduce the accumulators modulo p and store
// them as bytes. Complex: accumulator columns 0-127 hold Re, 128-255 Im of the
// tile (lane = row of M, column = row of N): Mr [Nr Ni] is one MMA of N = 256,
// -Mi Ni and Mi Nr two of N = 128. The two accumulators (2 x 256 of 512 TMEM
// columns) alternate between items, so that an item's reduction overlaps the
// next one's MMAs. Items with K > 480 alternate them between chunks of 480: a
// chunk's accumulator is reduced in place while the other one fills, and
// carries its residue on.
// Items are decoded 32 at a time, a lane each (the producer's into a table, the
// epilogue's into registers): the integer divisions and searches of one item
// after the other let the ring of stages run dry (820 tiles at K = 256: complex
// 1341 -> 1419 TFLOP/s, real 450 -> 498).
template <bool CPLX>
__global__ void __launch_bounds__(kThreads, 1) k_rns_gemm(const __grid_constant__ Job j,
                                                          const uint8_t* __restrict__ planes, uint8_t* __restrict__ out,
                                                          int* __restrict__ gfail, uint64_t wait_ns, int hold) {
  constexpr int C = CPLX ? 2 : 1;
  constexpr int kOp = C * kPlane;  // bytes of one operand's K tile
  extern __shared__ __align__(128) uint8_t sm[];
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], acc_full[2], acc_empty[2], mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int4 s_item[kItems];
  __shared__ int s_fail, s_skip;
  chain_begin();
  if (threadIdx.x == 0) s_skip = *static_cast<volatile int*>(gfail);
  __syncthreads();
  if (s_skip) return;  // an earlier CTA gave up: leave together
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* fail = &s_fail;
  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int i = 0; i < kStages; ++i) {
      bar_init(smem_u32(&full[i]), 1);
      bar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      bar_init(smem_u32(&acc_full[i]), 1);
      bar_init(smem_u32(&acc_empty[i]), kEpi);
    }
    bar_init(smem_u32(&mma_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == kEpi + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  const int items = j.on * kRnsModuli;

  // item -> modulus, output tile, K tiles (0: nothing to do)
  auto decode = [&](int it, int& l, OutTile& t, int& rn, int& rm) -> int {
    l = it / j.on;
    t = out_tile(j, j.o0 + it - l * j.on);
    int k;
    product_dims(j, dims_of(j.s[t.f], j.m[t.f], j.p0, j.pc, j.b), rn, rm, k);
    return k <= 0 ? 0 : (k + kK - 1) / kK;
  };
  // Lane i decodes the CTA's i-th item from `it` on: slots of its operands, K tiles and modulus, rows of N and M.
  auto ahead = [&](int it, int& sn, int& sm_, uint32_t& kl, uint32_t& nm) {
    it += lane * int(gridDim.x);
    if (it < items) {
      int l, rn, rm;
      OutTile t;
      const int nkt = decode(it, l, t, rn, rm);
      sn = t.pole * j.pref_n[j.nf] + j.pref_n[t.f] + t.nt;
      sm_ = t.pole * j.pref_m[j.nf] + j.pref_m[t.f] + t.mt;
      kl = uint32_t(nkt) | uint32_t(l) << 24;
      nm = uint32_t(min(kRnsTile, rn - (j.rt0 + t.nt) * kRnsTile)) |
           uint32_t(min(kRnsTile, rm - (j.mt0 + t.mt) * kRnsTile)) << 16;
    }
    __syncwarp();
  };

  if (warp == kEpi) {
    // the CTA's items, decoded by all lanes
    for (int x = 0; x * int(gridDim.x) + int(blockIdx.x) < items; x += 32) {
      int sn = 0, sm_ = 0;
      uint32_t kl = 0, nm = 0;
      ahead(int(blockIdx.x) + x * int(gridDim.x), sn, sm_, kl, nm);
      s_item[x + lane] = make_int4(sn, sm_, int(kl), int(nm));
    }
    __syncwarp();
    if (lane == 0) {  // ---- producer
      int n = 0;
      bool ok = true;
      // hold (fault injection): CTA 0 copies nothing, and its MMA issuer's wait for operands runs out
      for (int it = hold && blockIdx.x == 0 ? items : int(blockIdx.x), x = 0; it < items && ok && !*fail; it += gridDim.x, ++x) {
        const int4 t = s_item[x];
        const int l = int(uint32_t(t.z) >> 24), nkt = t.z & 0xFFFFFF;
        const int64_t lo = int64_t(l) * j.kt * kOp;
        const uint8_t* gn = planes + j.n_base + int64_t(t.x) * j.slot + lo;
        const uint8_t* gm = planes + j.m_base + int64_t(t.y) * j.slot + lo;
        // bytes of the 8-row groups that the tiles have, of each plane (a whole tile: both planes in one copy)
        const uint32_t bn = uint32_t((t.w & 0xFFFF) + 7) / 8 * 512, bm = uint32_t((t.w >> 16) + 7) / 8 * 512;
        for (int kt = 0; kt < nkt; ++kt, ++n) {
          const int st = n % kStages, u = n / kStages;
          if (u > 0 && !bar_wait(smem_u32(&empty[st]), (u - 1) & 1, fail, wait_ns)) {
            record_fail(&s_fail, 9, kt);
            ok = false;
            break;
          }
          bar_expect(smem_u32(&full[st]), C * (bm + bn));
          const uint32_t dst = smem_u32(sm + st * 2 * kOp), bar = smem_u32(&full[st]);
          const uint8_t *pm = gm + int64_t(kt) * kOp, *pn = gn + int64_t(kt) * kOp;
          bulk_load(dst, pm, bm == kPlane ? kOp : bm, bar);
          if (CPLX && bm != kPlane) bulk_load(dst + kPlane, pm + kPlane, bm, bar);
          bulk_load(dst + kOp, pn, bn == kPlane ? kOp : bn, bar);
          if (CPLX && bn != kPlane) bulk_load(dst + kOp + kPlane, pn + kPlane, bn, bar);
        }
      }
      // every copy issued has landed before the CTA leaves (bounded)
      for (int i = 0; i < kStages; ++i)
        if (n > i && !bar_wait_all(smem_u32(&full[i]), ((n - 1 - i) / kStages) & 1)) record_fail(&s_fail, 3, i);
    }
  } else if (warp == kEpi + 1) {
    if (lane == 0) {  // ---- MMA issuer
      int n = 0, u = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
        int l, rn, rm;
        OutTile t;
        const int nkt = j.nkt > 0 ? j.nkt : decode(it, l, t, rn, rm);
        for (int k0 = 0; k0 < nkt && ok; k0 += kChunkTiles, ++u) {
          const int buf = u & 1;
          if (u > 1 && !bar_wait(smem_u32(&acc_empty[buf]), ((u >> 1) - 1) & 1, fail, wait_ns)) {
            record_fail(&s_fail, 10, k0);
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t acc = tmem + uint32_t(buf * 256);
          const int k1 = min(nkt, k0 + kChunkTiles);
          for (int kt = k0; kt < k1; ++kt, ++n) {
            const int st = n % kStages;
            if (!bar_wait(smem_u32(&full[st]), (n / kStages) & 1, fail, wait_ns)) {
              record_fail(&s_fail, 11, kt);
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t mr = sdesc(smem_u32(sm + st * 2 * kOp)), mi = desc_off(mr, kPlane / 16),
                           nr = desc_off(mr, kOp / 16), ni = desc_off(nr, kPlane / 16);
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
              // the third chunk on continues from the reduced residue
              const uint32_t on = (kt > k0 || ks > 0 || k0 >= 2 * kChunkTiles) ? 1u : 0u;
              mma(acc, desc_off(mr, ks * 16), desc_off(nr, ks * 16), idesc(CPLX ? 4 : 2, false), on);
              if (CPLX) {
                mma(acc, desc_off(mi, ks * 16), desc_off(ni, ks * 16), idesc(2, true), 1u);
                mma(acc + 128u, desc_off(mi, ks * 16), desc_off(nr, ks * 16), idesc(2, false), 1u);
              }
            }
            mma_commit(smem_u32(&empty[st]));
          }
          if (!ok) break;
          mma_commit(smem_u32(&acc_full[buf]));
        }
      }
      // every MMA issued has completed before TMEM is read for the last time or freed
      mma_commit(smem_u32(&mma_done));
      if (!bar_wait_all(smem_u32(&mma_done), 0)) record_fail(&s_fail, 7, 0);
    }
  } else {  // ---- reduction modulo p
    const int q = warp & 3, h = warp >> 2;
    const uint32_t lanes = uint32_t(q * 32) << 16;
    // complex: half h reduces Re (columns 0-127) or Im; real: columns 64 h .. 64 h + 63
    constexpr int NC = CPLX ? 128 : 64;
    const uint32_t col0 = uint32_t(h * NC);
    const int mrow = q * 32 + lane;
    int u = 0;
    bool ok = true;
    auto wait_full = [&](int use) {
      bool got = true;
      if (lane == 0) got = bar_wait(smem_u32(&acc_full[use & 1]), (use >> 1) & 1, fail, wait_ns);
      got = __shfl_sync(0xFFFFFFFFu, got, 0);
      if (!got && lane == 0) record_fail(&s_fail, 12, use);
      asm volatile("tcgen05.fence::after_thread_sync;");
      return got;
    };
    auto release = [&](int use) {
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) bar_arrive(smem_u32(&acc_empty[use & 1]));
    };
    int sn = 0, sm_ = 0;
    uint32_t kl = 0, nm = 0;
    for (int it = blockIdx.x, y = 0; it < items && ok; it += gridDim.x, ++y) {
      if ((y & 31) == 0) ahead(it, sn, sm_, kl, nm);
      const uint32_t k = __shfl_sync(0xFFFFFFFFu, kl, y & 31), rows = __shfl_sync(0xFFFFFFFFu, nm, y & 31);
      const int l = int(k >> 24), nch = (int(k & 0xFFFFFF) + kChunkTiles - 1) / kChunkTiles;
      if (nch == 0) continue;
      const float p = c_mod[l], inv = 1.0f / p;
      for (int c = 0; c + 2 < nch && ok; ++c, ++u) {  // chunks whose accumulator carries on: reduced in place
        if (!(ok = wait_full(u))) break;
        const uint32_t a = tmem + lanes + uint32_t((u & 1) * 256) + col0;
#pragma unroll 1
        for (int x = 0; x < NC; x += 16) {
          uint32_t v[16];
          tmem_ld16_nw(a + x, v);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float f = __uint_as_float(v[i]);
            v[i] = __float_as_uint(fmaf(fmaf(f, inv, 12582912.0f) - 12582912.0f, -p, f));
          }
          tmem_st16(a + x, v);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;");
        release(u);
      }
      if (!ok) break;
      const bool two = nch > 1;
      if (two) {  // the last two chunks' accumulators are added here
        if (!(ok = wait_full(u))) break;
        ++u;
      }
      if (!(ok = wait_full(u))) break;
      const uint32_t a = tmem + lanes + uint32_t((u & 1) * 256) + col0,
                     a2 = tmem + lanes + uint32_t(((u & 1) ^ 1) * 256) + col0;
      const int nn = int(rows & 0xFFFF);  // rows of N in the tile
      const bool m_in = mrow < int(rows >> 16);
      // (re, im) x 128 rows of M x 128 rows of N, one byte each
      uint8_t* o = out + (int64_t(it - l * j.on) * kRnsModuli + l) * (C * kRnsTile * kRnsTile) +
                   (CPLX ? h * kRnsTile * kRnsTile : 0) + mrow * kRnsTile + (CPLX ? 0 : h * NC);
#pragma unroll 1
      for (int x = 0; x < NC; x += 32) {
        if ((CPLX ? 0 : h * NC) + x >= nn) break;
        uint32_t v[32];
        tmem_ld32(a + x, v);
        if (two) {
          uint32_t w[32];
          tmem_ld32(a2 + x, w);
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float g = __uint_as_float(w[i]);
            v[i] = __float_as_uint(__uint_as_float(v[i]) + fmaf(fmaf(g, inv, 12582912.0f) - 12582912.0f, -p, g));
          }
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          // r + 128 in the low byte (r = 128 of p = 256 wraps to its other representative)
          const float f = __uint_as_float(v[i]);
          v[i] = __float_as_uint(fmaf(fmaf(f, inv, 12582912.0f) - 12582912.0f, -p, f) + 12583040.0f);
        }
        if (m_in) {
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            uint32_t bw[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint32_t* z = v + 16 * y + 4 * i;
              bw[i] = __byte_perm(__byte_perm(z[0], z[1], 0x0040), __byte_perm(z[2], z[3], 0x0040), 0x5410);
            }
            *reinterpret_cast<uint4*>(o + x + 16 * y) = make_uint4(bw[0], bw[1], bw[2], bw[3]);
          }
        }
      }
      if (two) release(u - 1);
      release(u);
      ++u;
    }
  }
  __syncthreads();
  if (s_fail && threadIdx.x == 0)
    atomicMax(gfail, 1 + (min(s_fail, 255) << 20) + min(int(blockIdx.x), (1 << 20) - 1));
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == kEpi + 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ------------------------------------------------------------ reconstruction
// X 2^sc, X the integer of magnitude below 2^116 whose residues (plus 128) are
// byte `b` of w: the sum of u_l P / p_l less a multiple of P, exactly, in limbs of
// 20, 32, 32 and 34 bits, rounded to the nearest double from its 64 leading bits.
__device__ __forceinline__ double from_residues(const uint32_t (&w)[kRnsModuli], int b, int sc) {
  constexpr u128 P = mod_product(), B = byte_bias();
  uint32_t a0 = 0;
  unsigned long long a1 = limb(B, 1), a2 = limb(B, 2), a3 = static_cast<unsigned long long>(B >> 84);
  each_modulus([&](auto LC) {
    constexpr int l = decltype(LC)::value;
    constexpr uint32_t l0 = limb(cofactor(l), 0), l1 = limb(cofactor(l), 1), l2 = limb(cofactor(l), 2),
                       l3 = limb(cofactor(l), 3);
    const uint32_t u = __byte_perm(w[l], 0u, 0x4440 + b);
    a0 += u * l0;
    a1 += static_cast<unsigned long long>(u) * l1;
    a2 += static_cast<unsigned long long>(u) * l2;
    a3 += static_cast<unsigned long long>(u) * l3;
  });
  // The multiple of P, from the leading limb alone: |X| <= 2^116 against P / 2 > 2^116.3, and what the lower limbs
  // and the float rounding leave out is below 2^-9 of P. It lies between 0 and 22.
  constexpr float pinv = float(19342813113834066795298816.0 / (double(P >> 60) * double(1ull << 60)));  // 2^84 / P
  const uint32_t k = uint32_t(__float2int_rn(__uint2float_rn(uint32_t(a3 >> 8)) * (256.0f * pinv)));
  constexpr uint32_t p0 = limb(P, 0), p1 = limb(P, 1), p2 = limb(P, 2);
  constexpr unsigned long long p3 = static_cast<unsigned long long>(P >> 84);
  const long long s0 = static_cast<long long>(a0) + static_cast<long long>(limb(B, 0)) - static_cast<long long>(k * p0);
  const long long s1 = static_cast<long long>(a1 - static_cast<unsigned long long>(k) * p1) + (s0 >> 20);
  const long long s2 = static_cast<long long>(a2 - static_cast<unsigned long long>(k) * p2) + (s1 >> 32);
  const long long s3 = static_cast<long long>(a3 - k * p3) + (s2 >> 32);
  // magnitude m3 2^84 + m2 2^52 + low (m3 < 2^32, low < 2^52)
  const bool neg = s3 < 0;
  const uint32_t flip = neg ? 0xFFFFFFFFu : 0u;
  const unsigned long long flip52 = neg ? 0xFFFFFFFFFFFFFull : 0ull;
  unsigned long long low = (static_cast<unsigned long long>(uint32_t(s1)) << 20) | (static_cast<uint32_t>(s0) & 0xFFFFFu);
  low = (low ^ flip52) + (neg ? 1u : 0u);
  const unsigned long long mid = static_cast<unsigned long long>(uint32_t(s2) ^ flip) + (low >> 52);
  uint32_t A = (uint32_t(static_cast<unsigned long long>(s3)) ^ flip) + uint32_t(mid >> 32), Bw = uint32_t(mid),
           Cw = uint32_t(low >> 20), Dw = uint32_t(low) << 12;
  int E = 1023 + 84 + 31 + sc;  // biased exponent of bit 31 of A
#pragma unroll
  for (int t = 0; t < 3; ++t)
    if (A == 0) {
      A = Bw;
      Bw = Cw;
      Cw = Dw;
      Dw = 0;
      E -= 32;
    }
  if (A == 0) return 0.0;
  const int lz = __clz(A);
  const uint32_t hi = __funnelshift_l(Bw, A, lz), lo = __funnelshift_l(Cw, Bw, lz);
  unsigned long long mant = ((static_cast<unsigned long long>(hi) << 32) | lo) >> 11;  // 53 bits
  const uint32_t rest = lo & 0x7FFu;
  mant += rest > 0x400u || (rest == 0x400u && (mant & 1ull)) ? 1u : 0u;
  E -= lz;
  if (E <= 0 || E >= 2046) {
    const double v = ldexp(static_cast<double>(mant), E - 1023 - 52);
    return neg ? -v : v;
  }
  // the leading bit adds 1 to the exponent field, and so does a carry out of the mantissa
  return __longlong_as_double(static_cast<long long>((neg ? 1ull << 63 : 0ull) +
                                                     (static_cast<unsigned long long>(E - 1) << 52) + mant));
}

// One thread per part (re, im) of 4 consecutive front rows of a front column,
// over the rows and columns that the output tile really has (small fronts fill
// a few of its 128 x 128 entries): front columns are rows of M, front rows
// (contiguous in memory) rows of N. Everything a product does to F or Y acts on
// the parts alone. One thread's integers are a serial chain of some 600
// instructions, so the small products of the diagonal blocks want many threads:
// two units of both parts per thread took 17 us for a 256 x 256 block.
constexpr int kReconThreads = 128;

template <typename T>
__global__ void __launch_bounds__(kReconThreads) k_rns_recon(double* __restrict__ F, double* __restrict__ Y,
                                                             const __grid_constant__ Job j,
                                                             const uint8_t* __restrict__ planes,
                                                             const uint8_t* __restrict__ out) {
  constexpr int C = sizeof(T) / sizeof(double);
  const OutTile t = out_tile(j, j.o0 + int(blockIdx.x));
  const Dims d = dims_of(j.s[t.f], j.m[t.f], j.p0, j.pc, j.b);
  int rn, rm, K;
  product_dims(j, d, rn, rm, K);
  const int row0 = (j.rt0 + t.nt) * kRnsTile, col0 = (j.mt0 + t.mt) * kRnsTile;
  const int quads = (min(kRnsTile, rn - row0) + 3) / 4, units = C * quads * min(kRnsTile, rm - col0);
  const int unit = int(blockIdx.y) * kReconThreads + threadIdx.x;
  chain_next();
  chain_begin(F, Y, planes, out);
  if (unit >= units) return;
  const int part = unit % C, x = unit / C, mr = x / quads, q = x - mr * quads, c = col0 + mr, n0 = row0 + q * 4;
  const bool tri = triangular(j.mode, j.gen);
  if (tri && n0 + 3 < c) return;
  // an LDU front's update reaches the rows or the columns below `cols`
  const int cols = j.mode == kSchur && j.gen ? update_of(d, j.g0, j.k0, j.width).cols : 1 << 30;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (K > 0) {
    const int tail = kRnsTile * int(sizeof(int));
    const int* en = reinterpret_cast<const int*>(planes + j.n_base +
                                                 (int64_t(t.pole) * j.pref_n[j.nf] + j.pref_n[t.f] + t.nt + 1) * j.slot - tail);
    const int* em = reinterpret_cast<const int*>(planes + j.m_base +
                                                 (int64_t(t.pole) * j.pref_m[j.nf] + j.pref_m[t.f] + t.mt + 1) * j.slot - tail);
    uint32_t w[kRnsModuli];
    const uint8_t* src = out + int64_t(blockIdx.x) * kRnsModuli * (C * kRnsTile * kRnsTile) + part * kRnsTile * kRnsTile +
                         mr * kRnsTile + q * 4;
#pragma unroll
    for (int l = 0; l < kRnsModuli; ++l)
      w[l] = *reinterpret_cast<const uint32_t*>(src + int64_t(l) * (C * kRnsTile * kRnsTile));
    const int eb = em[mr];
    int ea[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) ea[i] = n0 + i < rn ? en[q * 4 + i] : 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = from_residues(w, i, ea[i] + eb - 2 * kBeta);
      if (ea[i] == kNanRow || eb == kNanRow) v[i] = __longlong_as_double(0x7FF8000000000000LL);
    }
  }
  // this part of the front, of its diagonal block and of the same places in Y; the columns' stride
  const int64_t m = int64_t(C) * d.m, base = C * (int64_t(j.pole0 + t.pole) * j.pool + j.off[t.f]) + part;
  double *fb = F + base + m * j.p0 + C * j.p0, *yb = Y + base + m * j.p0 + C * j.p0;
  const int below = C * d.bw;  // from the diagonal block's rows to the rows below it
  const bool in_c = c >= j.pc && c < j.pc + d.pb, last = j.pc + d.pb == d.bw;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = n0 + i;
    if (r >= rn || (tri && r < c) || (r >= cols && c >= cols)) continue;
    const bool in_r = r >= j.pc && r < j.pc + d.pb;
    double* at = fb + m * c + C * r;   // entry (r, c) of the diagonal block
    double* to = fb + m * r + C * c;   // and (c, r)
    switch (j.mode) {
      case kSweepT: {  // column c of the panel; a symmetric block holds minus the inverse until the last panel's sweep
        double* e = fb + m * (j.pc + c) + C * r;
        if (j.gen) {
          if (!in_r) *e = -v[i];
        } else if (in_r) {
          if (!last) *e = -*e;
        } else {
          const double val = last ? -v[i] : v[i];
          *e = val;
          fb[m * r + C * (j.pc + c)] = val;
        }
        break;
      }
      case kSweepDU: if (!in_c) fb[m * c + C * (j.pc + r)] = v[i]; break;
      case kSweepU: {
        if (in_r || in_c) break;
        if (j.gen) {  // T is stored negated
          *at = *at + v[i];
        } else {      // the last sweep's T is already negated, and so is its result
          const double val = last ? -(*at + v[i]) : *at - v[i];
          *at = val;
          *to = val;
        }
        break;
      }
      case kResid: yb[m * c + C * r] = (r == c && part == 0 ? 1.0 : 0.0) - v[i]; break;
      case kRefine: {
        const double val = *at + v[i];
        *at = val;
        if (!j.gen) *to = val;
        break;
      }
      case kPanel: fb[m * c + below + C * r] = v[i]; break;
      case kPanelU: fb[m * (d.bw + c) + C * r] = v[i]; break;
      case kSchur: {
        double* e = fb + m * (d.bw + c) + below + C * r;
        *e = *e - v[i];
        break;
      }
      case kTak:
        yb[m * c + below + C * r] = -v[i];
        if (!j.gen) yb[m * (d.bw + r) + C * c] = -v[i];
        break;
      case kTakU: yb[m * (d.bw + c) + C * r] = -v[i]; break;
      default: {  // kDiag
        const double val = (j.gen ? *at : 0.5 * (*at + *to)) - v[i];
        yb[m * c + C * r] = val;
        if (!j.gen) yb[m * r + C * c] = val;
        break;
      }
    }
  }
}

// Diagonal blocks of more than one panel before their inversion, both
// triangles (symmetric fronts hold the lower one), into Y (free during the factorisation). One block of threads per
// 16 columns, front and pole.
template <typename T>
__global__ void __launch_bounds__(256) k_rns_save(const T* __restrict__ F, T* __restrict__ Y, DevFronts fr,
                                                  const int32_t* __restrict__ fronts, int p0, int b, int gen) {
  const int f = fronts[blockIdx.y];
  chain_next();
  chain_begin(F, Y);
  const Dims d = dims_of(fr.s[f], fr.m[f], p0, 0, b);
  if (d.bw <= b) return;
  const int64_t base = int64_t(blockIdx.z) * fr.pool + fr.off[f] + p0 + int64_t(d.m) * p0;
  for (int c = blockIdx.x * 16; c < min(d.bw, int(blockIdx.x) * 16 + 16); ++c)
    for (int r = threadIdx.x; r < d.bw; r += 256) {
      const int hi = gen ? r : max(r, c), lo = gen ? c : min(r, c);
      Y[base + int64_t(d.m) * c + r] = F[base + int64_t(d.m) * lo + hi];
    }
}

// W = F[S,B] (and A[B,S] of LDU fronts: ROWS) of the fronts whose groups have
// more than one block, into the same places of Y, for the group's updates. A
// block of threads takes 16 columns of 256 rows.
template <typename T, bool ROWS>
__global__ void __launch_bounds__(256) k_rns_keep(const T* __restrict__ F, T* __restrict__ Y, DevFronts fr,
                                                  const int32_t* __restrict__ fronts, int p0, int b, int g0) {
  const int f = fronts[blockIdx.y];
  chain_next();
  chain_begin(F, Y);
  const Dims d = dims_of(fr.s[f], fr.m[f], p0, 0, b);
  if (d.s <= g0 + rns_block(b)) return;
  const int across = ROWS ? 1 : (rns_block(b) + 15) / 16;
  const int r = int(blockIdx.x) / across * 256 * (ROWS ? 0 : 1) + threadIdx.x;
  const int c0 = (ROWS ? int(blockIdx.x) : int(blockIdx.x) % across) * 16;
  const int nr = ROWS ? d.bw : d.mp, nc = ROWS ? d.mp : d.bw;
  if (r >= nr) return;
  const int64_t at = int64_t(blockIdx.z) * fr.pool + fr.off[f] + (ROWS ? p0 : d.q0) + r +
                     int64_t(d.m) * ((ROWS ? d.q0 : p0) + c0);
#pragma unroll
  for (int c = 0; c < 16; ++c)
    if (c0 + c < nc) Y[at + int64_t(d.m) * c] = F[at + int64_t(d.m) * c];
}

// ------------------------------------------------------------ scaling
constexpr int kNoExp = -20000;  // of zero, subnormal and non-finite values, which do not count

__device__ __forceinline__ uint32_t high_word(double x) { return uint32_t(__double2hiint(x)) & 0x7FFFFFFFu; }
// floor(log2) of a value by its high word
__device__ __forceinline__ int exponent(uint32_t high) {
  const int E = int(high >> 20);
  return E == 0 || E == 0x7FF ? kNoExp : E - 1023;
}

// First guess: half the exponent of the diagonal entry of H - z S. h: of max(|H_cc|, |S_cc|).
template <int W>
__global__ void k_rns_diag_scale(const double* __restrict__ H, const double* __restrict__ S,
                                 const int64_t* __restrict__ diag, int64_t n, int64_t c0, int64_t e0,
                                 const __grid_constant__ BatchShifts sh, int64_t stride, int16_t* __restrict__ h,
                                 int16_t* __restrict__ g0, int* __restrict__ scaled, bool first) {
  const int b = blockIdx.y;
  if (first && b == 0 && blockIdx.x == 0 && threadIdx.x == 0) *scaled = 0;
  for (int64_t c = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; c < n; c += int64_t(gridDim.x) * blockDim.x) {
    const int64_t e = (diag[c] - e0) * W;
    const double Hc = H[e], Sc = S[e];  // of Hermitian H and S: real
    if (b == 0) {
      const int E = exponent(max(high_word(Hc), high_word(Sc)));
      h[c0 + c] = int16_t(E == kNoExp ? 0 : max(-500, min(500, E >> 1)));
    }
    const int E = exponent(max(high_word(fma(-sh.re[b], Sc, Hc)), high_word(sh.im[b] * Sc)));
    g0[(c0 + c) * stride + b] = int16_t(E == kNoExp ? kNoExp : (E + 1) >> 1);
  }
}

// Then raised until no entry of the column is above 1: against a row of a larger
// guess by what is missing, against one of a smaller guess by half of the
// entry's exponent, which that row takes the other half of. The exponents alone
// tell an upper bound of |H - z S|, without an FP64 operation. A warp per column
// and 8 members, whose exponents are one 16-byte word.
template <int W>
__global__ void __launch_bounds__(256) k_rns_scale(const double* __restrict__ H, const double* __restrict__ S,
                                                   const int64_t* __restrict__ colptr, const int32_t* __restrict__ row,
                                                   const int32_t* __restrict__ col, int64_t n, int64_t e0,
                                                   const __grid_constant__ BatchShifts sh, int64_t stride,
                                                   const int16_t* __restrict__ h, const int16_t* __restrict__ g0,
                                                   int16_t* __restrict__ g, int* __restrict__ scaled) {
  union Word {
    uint4 u;
    int16_t x[8];
  };
  const int lane = threadIdx.x & 31, b0 = blockIdx.y * 8;
  int ez[8];  // |z| < 2^(ez + 1)
#pragma unroll
  for (int b = 0; b < 8; ++b) ez[b] = b0 + b < sh.nb ? exponent(max(high_word(sh.re[b0 + b]), high_word(sh.im[b0 + b]))) : 0;
  for (int64_t j = blockIdx.x * 8 + (threadIdx.x >> 5); j < n; j += int64_t(gridDim.x) * 8) {
    const int64_t lo = colptr[j], hi = colptr[j + 1];
    const int c = col[lo], hc = h[c];
    bool any = false;
    Word top;
    top.u = *reinterpret_cast<const uint4*>(g0 + c * stride + b0);
    int t[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) t[b] = top.x[b];
    for (int64_t ea = lo + lane; ea < hi; ea += 32 * 4) {  // four entries in flight
      int r[4], eh[4], es[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t e = min(ea + 32 * u, hi - 1);
        r[u] = row[e];
        if constexpr (W == 1) {
          eh[u] = exponent(high_word(H[e - e0]));
          es[u] = exponent(high_word(S[e - e0]));
        } else {
          const double2 a = reinterpret_cast<const double2*>(H)[e - e0], s = reinterpret_cast<const double2*>(S)[e - e0];
          eh[u] = exponent(max(high_word(a.x), high_word(a.y)));
          es[u] = exponent(max(high_word(s.x), high_word(s.y)));
        }
      }
      Word gr[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) gr[u].u = *reinterpret_cast<const uint4*>(g0 + r[u] * stride + b0);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (r[u] == c) continue;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const int E = max(eh[u], es[u] + ez[b] + 1);
          if (E > kNoExp / 2) t[b] = max(t[b], min(E - int(gr[u].x[b]), (E + 1) >> 1));
        }
      }
    }
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int m = __reduce_max_sync(0xFFFFFFFFu, t[b]);
      const int x = m == kNoExp ? 0 : max(-500, min(500, m));
      const int gc = abs(x - hc) <= kRnsNear ? hc : x;
      top.x[b] = int16_t(gc);
      if (b0 + b < sh.nb && (gc | hc)) any = true;
    }
    if (lane == 0) *reinterpret_cast<uint4*>(g + c * stride + b0) = top.u;
    if (lane == 0 && any) *scaled = 1;
  }
}

// ------------------------------------------------------------ host schedule
// Fronts [f0, f0 + nf) of a level's list for the poles [pole0, pole0 + np), or
// row tiles [rt0, rt0 + rtn) of the one front's N operand (rtn = 0: all).
struct Piece {
  int f0, nf, pole0, np, rt0, rtn;
};

struct Slots {
  int fixed, n;  // operand slots of a front: fixed ones, and those of N row tiles that may be taken in pieces
  int k;         // contraction length: the slot size
};

// The pieces of a launch sequence that fit the scratch, in order. Every front's
// fixed slots and one row tile fit (rns_scratch_range); a front for which they did
// not would be left out without a word, so that is an error.
template <typename Fn>
std::vector<Piece> pieces_of(int nact, int nb, int64_t cap, bool cplx, Fn slots) {
  std::vector<Piece> out;
  for (int f0 = 0; f0 < nact;) {
    int nf = 0, k = 0;
    int64_t sum = 0;
    while (f0 + nf < nact && nf < kRnsFronts) {
      const Slots q = slots(f0 + nf);
      const int kk = std::max(k, q.k);
      if (nf > 0 && (sum + q.fixed + q.n) * rns_slot_bytes(kk, cplx) > cap) break;
      sum += q.fixed + q.n;
      k = kk;
      ++nf;
    }
    const int64_t fit = cap / rns_slot_bytes(k, cplx);
    if (sum > fit) {  // one front, in pieces of its row tiles
      const Slots q = slots(f0);
      const int step = int(fit - q.fixed);
      if (q.n <= 0 || step <= 0) throw CudaError{cudaErrorInvalidValue, "residue scratch below a front's operands"};
      for (int pole = 0; pole < nb; ++pole)
        for (int r = 0; r < q.n; r += step) out.push_back({f0, 1, pole, 1, r, std::min(step, q.n - r)});
    } else if (sum > 0) {
      const int np = int(std::min<int64_t>(nb, fit / sum));
      for (int pole = 0; pole < nb; pole += np) out.push_back({f0, nf, pole, std::min(np, nb - pole), 0, 0});
    } else {
      out.push_back({f0, nf, 0, nb, 0, 0});
    }
    f0 += nf;
  }
  return out;
}

Slots update_slots(const Dims& d, const Update& u) { return {2 * tiles128(d.mp), 0, u.k}; }

template <typename T>
struct Runner {
  static constexpr bool CPLX = sizeof(T) == 16;
  const RnsScratch& sc;
  T *F, *Y;
  const int32_t *s, *m;  // sizes of the level's fronts
  const int64_t* off;    // and their places in a pole's pool
  int64_t pool;
  int b;
  cudaStream_t st;
  int gen = 0;
  int group = 1;  // blocks of a group

  // The update after the block at p0 (Update).
  void update(Job& j, int p0) const {
    const int blk = rns_block(b), i = p0 / blk + 1, low = i & -i;
    j.g0 = (i - 1) / group * group * blk;
    j.k0 = p0 + blk - low * blk;
    j.width = i % group == 0 ? 0 : low * blk;
  }

  // W (and A of LDU fronts) of the block at p0 into Y, where the group's updates read it again.
  void keep(const DevFronts& fr, const int32_t* dfr, int nact, int p0, int np) const {
    Job j;
    update(j, p0);
    int n = 0, rows = 0;
    for (; n < nact && s[n] > j.g0 + rns_block(b); ++n) rows = std::max(rows, dims_of(s[n], m[n], p0, 0, b).mp);
    if (group == 1 || rows == 0) return;
    const int across = (rns_block(b) + 15) / 16;
    launch_chained(k_rns_keep<T, false>, dim3((rows + 255) / 256 * across, n, np), 256, 0, st, F, Y, fr, dfr, p0, b, j.g0);
    if (gen) launch_chained(k_rns_keep<T, true>, dim3((rows + 15) / 16, n, np), 256, 0, st, F, Y, fr, dfr, p0, b, j.g0);
  }
  // The widest update of the block's fronts; one of more than a block applies columns kept in Y.
  int update_k(int nact, int p0) const {
    Job j;
    update(j, p0);
    int k = 0;
    for (int f = 0; f < nact; ++f) {
      const Dims d = dims_of(s[f], m[f], p0, 0, b);
      if (d.mp > 0) k = std::max(k, update_of(d, j.g0, j.k0, j.width).k);
    }
    return k;
  }
  // That update, apart from the block's panel products.
  void apart(int nact, int p0, int nb, Profiler& pf) const {
    Job w;
    update(w, p0);
    auto up = [&](int f) { return update_of(dims_of(s[f], m[f], p0, 0, b), w.g0, w.k0, w.width); };
    auto slots = [&](int f) { return update_slots(dims_of(s[f], m[f], p0, 0, b), up(f)); };
    for (const Piece& q : pieces_of(nact, nb, sc.plane_bytes, CPLX, slots)) {
      int k = 32;
      for (int f = q.f0; f < q.f0 + q.nf; ++f) k = std::max(k, up(f).k);
      Job u;
      const int uo = job(u, kSchur, q, p0, 0, (k + kK - 1) / kK);
      if (uo == 0) continue;
      u.n_base = 0;
      u.m_base = int64_t(n_slots(u)) * u.slot;
      cudaEvent_t a = pf.begin(st);
      conv(u, q, kOpL, gen ? kOpAs : kOpWs);
      pf.end(a, P_SLICE, st, 0.0, slot_bytes(u, kOpL) + slot_bytes(u, kOpWs));
      a = pf.begin(st);
      product(u, q, uo);
      const double fl = pf.on ? update_flops(q, p0) : 0.0;
      pf.end(a, P_SCHUR, st, fl, 0.0, 2, fl * kRnsModuli);
    }
  }
  double update_flops(const Piece& q, int p0) const {
    Job w;
    update(w, p0);
    double fl = 0;
    for (int f = q.f0; f < q.f0 + q.nf; ++f) {
      const Dims d = dims_of(s[f], m[f], p0, 0, b);
      const Update u = update_of(d, w.g0, w.k0, w.width);
      const double rest = d.mp - u.cols, cols = u.cols;
      fl += (CPLX ? 8.0 : 2.0) * q.np * u.k *
            (gen ? double(d.mp) * d.mp - rest * rest : cols * (cols + 1) / 2 + rest * cols);
    }
    return fl;
  }

  // Tile counts of a product over a piece; returns the output tiles.
  int job(Job& j, Mode mode, const Piece& q, int p0, int pc, int kt) const {
    j.mode = mode;
    j.gen = gen;
    j.nf = q.nf;
    j.np = q.np;
    j.pole0 = q.pole0;
    j.p0 = p0;
    j.pc = pc;
    j.b = b;
    update(j, p0);
    j.rt0 = mode == kTak ? q.rt0 : 0;
    j.mt0 = mode == kTakU ? q.rt0 : 0;
    j.kt = kt;
    j.slot = rns_slot_bytes(32 * kt, CPLX);
    j.pool = pool;
    j.pref_n[0] = j.pref_m[0] = j.pref_o[0] = 0;
    for (int f = 0; f < q.nf; ++f) {
      j.s[f] = s[q.f0 + f];
      j.m[f] = m[q.f0 + f];
      j.off[f] = off[q.f0 + f];
      int rn, rm, k;
      const Dims d = dims_of(s[q.f0 + f], m[q.f0 + f], p0, pc, b);
      product_dims(j, d, rn, rm, k);
      if (mode == kSchur) rm = rn;  // slots as the rows have them
      const int tn = q.rtn > 0 && mode == kTak ? q.rtn : tiles128(rn), tm = q.rtn > 0 && mode == kTakU ? q.rtn : tiles128(rm);
      const int nkt = k <= 0 ? 0 : (k + kK - 1) / kK;
      j.nkt = f == 0 || nkt == j.nkt ? nkt : 0;
      j.pref_n[f + 1] = j.pref_n[f] + (k > 0 ? tn : 0);  // K = 0 (Y[B,B] of a front without rows below): no operands
      j.pref_m[f + 1] = j.pref_m[f] + (k > 0 ? tm : 0);
      const int out = mode == kSchur ? tiles128(update_of(d, j.g0, j.k0, j.width).cols) : 0, rest = tn - out;
      j.pref_o[f + 1] = j.pref_o[f] + (mode == kSchur ? (gen ? tn * tn - rest * rest : out * (out + 1) / 2 + rest * out)
                                       : triangular(mode, gen) ? tn * (tn + 1) / 2 : tn * tm);
    }
    return j.pref_o[q.nf] * q.np;
  }
  int n_slots(const Job& j) const { return j.pref_n[j.nf] * j.np; }
  int m_slots(const Job& j) const { return j.pref_m[j.nf] * j.np; }

  // Bytes that the conversion of an operand reads and writes, in whole slots.
  double slot_bytes(const Job& j, Operand a) const {
    return double(m_side(a) ? m_slots(j) : n_slots(j)) * double(j.slot) * (1.0 + 8.0 / 30.0);
  }
  void conv(const Job& j, const Piece& q, Operand a) const { conv2(j, q, a, a, false); }
  void conv(const Job& j, const Piece& q, Operand a, Operand c) const { conv2(j, q, a, c, true); }
  void conv2(const Job& j, const Piece& q, Operand a, Operand c, bool both) const {
    const int oc = j.kt <= 2 ? 8 : 32, g = 32 / oc;
    auto blocks = [&](Operand op) { return ((m_side(op) ? m_slots(j) : n_slots(j)) * 16 + g - 1) / g; };
    const int na = blocks(a), n = na + (both ? blocks(c) : 0);
    if (n <= 0) return;
    if (oc == 8) launch_chained(k_rns_conv<T, 8>, n, 256, 0, st, F, Y, j, sc.planes, a, na, c);
    else launch_chained(k_rns_conv<T, 32>, n, 256, 0, st, F, Y, j, sc.planes, a, na, c);
  }

  // The product and its reconstruction, in pieces of the output scratch.
  void product(Job& j, const Piece& q, int tiles) const {
    const int cap = int(std::min<int64_t>(sc.out_bytes / (int64_t(kRnsOutTile) * (CPLX ? 2 : 1)), kItems * sc.sms / kRnsModuli));
    for (int o = 0; o < tiles; o += cap) {
      j.o0 = o;
      j.on = std::min(cap, tiles - o);
      launch_chained(k_rns_gemm<CPLX>, std::min(sc.sms, j.on * kRnsModuli), kThreads, gemm_smem(CPLX), st, j, sc.planes,
                     sc.out, sc.fail, sc.wait_ns, sc.hold);
      launch_chained(k_rns_recon<T>, dim3(j.on, (CPLX ? 2 : 1) * kRnsTile * kRnsTile / 4 / kReconThreads), kReconThreads, 0,
                     st, reinterpret_cast<double*>(F), reinterpret_cast<double*>(Y), j, sc.planes, sc.out);
    }
  }
};


// Scratch for the operands of a front's update by a group of g blocks (complex,
// also for real fronts): the most over the plan's fronts of more than a block.
int64_t group_bytes(const pexsi_plan* p, int g) {
  int64_t most = 0;
  const int blk = rns_block(p->b);
  for (const Level& lv : p->levels)
    for (size_t f = 0; f < lv.s.size() && lv.s[f] > blk; ++f)
      most = std::max(most, 2 * tiles128(lv.m[f]) * rns_slot_bytes(std::min(lv.s[f], g * blk), true));
  return most;
}

// Blocks of a group: as many as the scratch has room for the operands of, by the
// plan's largest fronts and not by a level's or a batch's, so that a front's sums
// are grouped alike whatever runs beside it (rns_scratch_range reserves the room
// for whole groups; only the least scratch has smaller ones). Each block alone, the rest of a front is read, reconstructed and written
// once per 256 columns and the products' K is 256; in groups the operands of a
// group are converted again. Groups of 1, 2 and 4 blocks: 55.4, 52.7 and 51.3 ms
// for the inertia counts of 256 atoms in a fluid, 60.8, 58.9 and 58.1 ms for the
// density matrix of 512, 53.0, 51.7 and 51.4 ms for a sheet of 14 x 14; fronts of
// a few hundred columns do not care.
int group_of(const pexsi_plan* p, int64_t cap) {
  int g = kRnsGroup;
  while (g > 1 && group_bytes(p, g) > cap) g /= 2;
  return g;
}

// Slots of the launch sequences of one front.
Slots sweep_slots(const Dims& d, int b) {
  if (d.bw <= b) return {0, 0, 32};
  return {2 * tiles128(d.bw) + 1, 0, b};
}
Slots refine_slots(const Dims& d, int b) { return {d.bw > b ? 3 * tiles128(d.bw) : 0, 0, d.bw}; }
Slots gen_sweep_slots(const Dims& d, int b) {
  if (d.bw <= b) return {0, 0, 32};
  return {2 * tiles128(d.bw) + 2, 0, b};
}
Slots gen_refine_slots(const Dims& d, int b) { return {d.bw > b ? 2 * tiles128(d.bw) : 0, 0, d.bw}; }
Slots schur_slots(const Dims& d) { return {d.mp > 0 ? 2 * tiles128(d.mp) + tiles128(d.bw) : 0, 0, d.bw}; }
Slots tak_slots(const Dims& d) {
  const int tm = tiles128(d.bw), tn = tiles128(d.mp);
  return {d.mp > 0 ? tm : 0, d.mp > 0 ? std::max(tn, tm) : 0, d.mp};
}

}  // namespace

void launch_rns_scales(const double* H, const double* S, int wide, const BatchShifts& sh, const int64_t* colptr,
                       const int64_t* diag, int64_t n, int64_t c0, int64_t e0, const int32_t* row, const int32_t* col,
                       int16_t* h, int16_t* g0, int16_t* g, int64_t stride, int* scaled, bool first, cudaStream_t st) {
  auto grid = [](int64_t k) { return int(std::min<int64_t>(k, 152 * 8)); };
  auto run = [&](auto w) {
    constexpr int W = decltype(w)::value;
    k_rns_diag_scale<W><<<dim3(grid((n + 255) / 256), sh.nb), 256, 0, st>>>(H, S, diag, n, c0, e0, sh, stride, h, g0, scaled, first);
    k_rns_scale<W><<<dim3(grid((n + 7) / 8), (sh.nb + 7) / 8), 256, 0, st>>>(H, S, colptr, row, col, n, e0, sh, stride, h, g0, g, scaled);
  };
  if (wide == 1) run(std::integral_constant<int, 1>{});
  else run(std::integral_constant<int, 2>{});
}

cudaError_t rns_configure() {
  cudaError_t e = cudaFuncSetAttribute(k_rns_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(true));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_rns_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(false));
  return e;
}

// Scratch bytes below which some front's operands do not fit (a front's Y[S,S]
// is taken in pieces of at least its panel operand's tiles), what whole groups of
// blocks need (group_of), and what lets every level run in one piece.
void rns_scratch_range(const pexsi_plan* p, int batch, int64_t& least, int64_t& whole, int64_t& want) {
  least = want = 0;
  for (const Level& lv : p->levels) {
    int64_t lw = 0, tw = 0, sw = 0;
    int ks = 32, kt = 32;
    for (size_t t = 0; t < lv.s.size(); ++t) {
      const Dims d = dims_of(lv.s[t], lv.m[t], 0, 0, p->b);
      const Slots a = sweep_slots(d, p->b), c = schur_slots(d), y = tak_slots(d), e = refine_slots(d, p->b);
      const int64_t one = std::max({(a.fixed + 1) * rns_slot_bytes(a.k, true), e.fixed * rns_slot_bytes(e.k, true), c.fixed * rns_slot_bytes(c.k, true),
                                    2 * y.fixed * rns_slot_bytes(y.k, true)});
      least = std::max(least, one);
      sw += a.fixed;
      lw += c.fixed;
      tw += y.fixed + y.n;
      ks = std::max({ks, c.k, std::min<int>(lv.s[t], kRnsGroup * rns_block(p->b))});
      kt = std::max(kt, y.k);
    }
    want = std::max({want, sw * batch * rns_slot_bytes(p->b, true), lw * batch * rns_slot_bytes(ks, true),
                     tw * batch * rns_slot_bytes(kt, true)});
  }
  least += rns_slot_bytes(32, true);
  whole = std::max(least, group_bytes(p, kRnsGroup));
  want = std::max(want, whole);
}

int64_t rns_out_bytes(const pexsi_plan* p, int batch, int most) {
  int64_t tiles = 1;
  for (const Level& lv : p->levels) {
    int64_t t = 0;
    for (size_t f = 0; f < lv.s.size(); ++f) {
      const int64_t n = tiles128(lv.m[f]);
      t += std::max<int64_t>(3, n * (n + 1) / 2);
    }
    tiles = std::max(tiles, t * batch);
  }
  return std::min<int64_t>(tiles, most) * kRnsOutTile * 2;
}

// Eliminates the block of columns [p0, p0 + 256) of the level's fronts (the
// first nact, those with s > p0): inverts the diagonal block, L[S,B] and the
// update of F[S,S].
template <typename T>
void rns_factor_block(const pexsi_plan* p, const Level& lv, const RnsScratch& sc, T* F, T* Y, int nact, int p0,
                      const BatchShifts& sh, DevStatus status, Profiler& pf, cudaStream_t st) {
  const int b = p->b, *s = lv.s.data(), *m = lv.m.data();
  const DevFronts fr = p->fronts();
  const int32_t* dfr = p->d_level_fronts + lv.front_off;
  Runner<T> r{sc, F, Y, s, m, lv.off.data(), fr.pool, b, st};
  constexpr bool CPLX = sizeof(T) == 16;
  r.group = group_of(p, sc.plane_bytes);
  const int bw = std::min(rns_block(b), s[0] - p0);  // the widest front's block
  r.keep(fr, dfr, nact, p0, sh.nb);
  if (bw > b) launch_chained(k_rns_save<T>, dim3((bw + 15) / 16, nact, sh.nb), 256, 0, st, F, Y, fr, dfr, p0, b, 0);
  for (int pc = 0; pc < bw; pc += b) {
    int n = 0;
    while (n < nact && s[n] > p0 + pc) ++n;
    cudaEvent_t a = pf.begin(st);
    launch_diag_inv<T>(F, fr, dfr, n, p0 + pc, b, sh, status, st);
    pf.end(a, P_DIAG, st, 0.0, 0.0);
    if (bw <= b) continue;
    a = pf.begin(st);
    auto slots = [&](int f) { return sweep_slots(dims_of(s[f], m[f], p0, pc, b), b); };
    int kernels = 0;
    for (const Piece& q : pieces_of(n, sh.nb, sc.plane_bytes, CPLX, slots)) {
      const int kt = (b + kK - 1) / kK;
      Job t, u;
      const int to = r.job(t, kSweepT, q, p0, pc, kt), uo = r.job(u, kSweepU, q, p0, pc, kt);
      if (to == 0) continue;
      t.n_base = u.m_base = 0;  // V, T, D
      u.n_base = int64_t(r.n_slots(t)) * t.slot;
      t.m_base = 2 * u.n_base;
      r.conv(t, q, kOpV, kOpD);
      r.product(t, q, to);
      r.conv(u, q, kOpT);
      r.product(u, q, uo);
      kernels += 6;
    }
    pf.end(a, P_PANEL, st, 0.0, 0.0, kernels);
  }
  // One Newton step X += X (I - B X) on the swept inverse: a panel block that is
  // nearly singular within a well conditioned B leaves large intermediate
  // inverses, whose rounding the sweeps keep; the residual product is accurate
  // to 2^-59 of the norms, so the step brings X to FP64 accuracy of B^-1.
  if (bw > b) {
    cudaEvent_t a = pf.begin(st);
    int kernels = 0;
    auto rslots = [&](int f) { return refine_slots(dims_of(s[f], m[f], p0, 0, b), b); };
    for (const Piece& q : pieces_of(nact, sh.nb, sc.plane_bytes, CPLX, rslots)) {
      const int kt = (std::min(rns_block(b), s[q.f0] - p0) + kK - 1) / kK;
      Job t, u;
      const int to = r.job(t, kResid, q, p0, 0, kt), uo = r.job(u, kRefine, q, p0, 0, kt);
      if (to == 0) continue;
      t.n_base = 0;  // B, X, R
      t.m_base = u.n_base = int64_t(r.n_slots(t)) * t.slot;
      u.m_base = 2 * t.m_base;
      Job c = t;
      c.n_base = u.m_base;
      r.conv(t, q, kOpR, kOpB);
      r.product(t, q, to);
      r.conv(c, q, kOpR);
      r.product(u, q, uo);
      kernels += 6;
    }
    pf.end(a, P_PANEL, st, 0.0, 0.0, kernels);
  }
  const bool joint = r.update_k(nact, p0) <= rns_block(b);  // the update's W is the panel product's operand
  auto slots = [&](int f) { return schur_slots(dims_of(s[f], m[f], p0, 0, b)); };
  for (const Piece& q : pieces_of(nact, sh.nb, sc.plane_bytes, CPLX, slots)) {
    const int kt = (std::min(rns_block(b), s[q.f0] - p0) + kK - 1) / kK;
    Job l, u;
    const int lo = r.job(l, kPanel, q, p0, 0, kt), uo = r.job(u, kSchur, q, p0, 0, kt);
    if (lo == 0) continue;
    l.n_base = 0;
    u.n_base = int64_t(r.n_slots(l)) * l.slot;
    l.m_base = 2 * u.n_base;  // W, L, B^-1
    u.m_base = 0;
    double fl = 0;
    if (pf.on)
      for (int f = q.f0; f < q.f0 + q.nf; ++f) {
        const Dims d = dims_of(s[f], m[f], p0, 0, b);
        fl += (CPLX ? 8.0 : 2.0) * q.np * d.mp * double(d.bw) * d.bw;
      }
    cudaEvent_t a = pf.begin(st);
    r.conv(l, q, kOpW, kOpB);
    pf.end(a, P_SLICE, st, 0.0, r.slot_bytes(l, kOpW) + r.slot_bytes(l, kOpB));
    a = pf.begin(st);
    r.product(l, q, lo);
    pf.end(a, P_PANEL, st, fl, 0.0, 2, fl * kRnsModuli);
    if (!joint) continue;
    a = pf.begin(st);
    r.conv(u, q, kOpL);
    pf.end(a, P_SLICE, st, 0.0, r.slot_bytes(u, kOpL));
    a = pf.begin(st);
    r.product(u, q, uo);
    const double sfl = pf.on ? r.update_flops(q, p0) : 0.0;
    pf.end(a, P_SCHUR, st, sfl, 0.0, 2, sfl * kRnsModuli);
  }
  if (!joint) r.apart(nact, p0, sh.nb, pf);
}

// Y[S,B], its mirror and Y[B,B] of the block at p0 of the level's first nact fronts.
void rns_selinv_block(const pexsi_plan* p, const Level& lv, const RnsScratch& sc, double2* Y, double2* F, int nact,
                      int p0, int nb, Profiler& pf, cudaStream_t st) {
  const int b = p->b, *s = lv.s.data(), *m = lv.m.data();
  Runner<double2> r{sc, F, Y, s, m, lv.off.data(), p->sym.front_elems, b, st};
  auto slots = [&](int f) { return tak_slots(dims_of(s[f], m[f], p0, 0, b)); };
  for (const Piece& q : pieces_of(nact, nb, sc.plane_bytes, true, slots)) {
    int k = 32;
    double fl = 0;
    for (int f = q.f0; f < q.f0 + q.nf; ++f) {
      const Dims d = dims_of(s[f], m[f], p0, 0, b);
      k = std::max(k, d.mp);
      fl += 8.0 * q.np * double(d.bw) * d.mp * (q.rtn > 0 ? double(q.rtn) * kRnsTile : d.mp);
    }
    const int kt = (k + kK - 1) / kK;
    Job t, g;
    const int to = r.job(t, kTak, q, p0, 0, kt), go = r.job(g, kDiag, q, p0, 0, kt);
    const bool more = q.rtn > 0, first = !more || q.rt0 == 0;
    // the front's last piece also takes Y[B,B]
    const bool last = !more || q.rt0 + q.rtn >= tiles128(dims_of(s[q.f0], m[q.f0], p0, 0, b).mp);
    t.m_base = g.m_base = 0;
    t.n_base = g.n_base = int64_t(r.m_slots(t)) * t.slot;
    if (to > 0) {
      cudaEvent_t a = pf.begin(st);
      if (first) r.conv(t, q, kOpLt, kOpY);
      else r.conv(t, q, kOpY);
      pf.end(a, P_SLICE, st, 0.0, r.slot_bytes(t, kOpY) + (first ? r.slot_bytes(t, kOpLt) : 0.0));
      a = pf.begin(st);
      r.product(t, q, to);
      pf.end(a, P_OFFDIAG, st, fl, 0.0, 2, fl * kRnsModuli);
    }
    if (last) {
      cudaEvent_t a = pf.begin(st);
      if (to > 0) r.conv(g, q, kOpYt);
      r.product(g, q, go);
      pf.end(a, P_DPART, st, 0.0, 0.0, 3);
    }
  }
}

// The same for LDU fronts: B, X and the panels are not symmetric.
void rns_factor_block_gen(const pexsi_plan* p, const Level& lv, const RnsScratch& sc, double2* F, double2* Y, int nact,
                          int p0, const BatchShifts& sh, DevStatus status, Profiler& pf, cudaStream_t st) {
  const int b = p->b, *s = lv.s.data(), *m = lv.m.data();
  const DevFronts fr = p->fronts();
  const int32_t* dfr = p->d_level_fronts + lv.front_off;
  Runner<double2> r{sc, F, Y, s, m, lv.off.data(), fr.pool, b, st, 1};
  r.group = group_of(p, sc.plane_bytes);
  const int bw = std::min(rns_block(b), s[0] - p0);
  const int kb = (b + kK - 1) / kK;
  r.keep(fr, dfr, nact, p0, sh.nb);
  if (bw > b) launch_chained(k_rns_save<double2>, dim3((bw + 15) / 16, nact, sh.nb), 256, 0, st, F, Y, fr, dfr, p0, b, 1);
  for (int pc = 0; pc < bw; pc += b) {
    int n = 0;
    while (n < nact && s[n] > p0 + pc) ++n;
    cudaEvent_t a = pf.begin(st);
    launch_diag_inv_gen(F, fr, dfr, n, p0 + pc, b, sh, status, st);
    pf.end(a, P_DIAG, st, 0.0, 0.0);
    if (bw <= b) continue;
    a = pf.begin(st);
    int kernels = 0;
    auto slots = [&](int f) { return gen_sweep_slots(dims_of(s[f], m[f], p0, pc, b), b); };
    for (const Piece& q : pieces_of(n, sh.nb, sc.plane_bytes, true, slots)) {
      Job t, x, u;
      const int to = r.job(t, kSweepT, q, p0, pc, kb), xo = r.job(x, kSweepDU, q, p0, pc, kb),
                uo = r.job(u, kSweepU, q, p0, pc, kb);
      if (to == 0) continue;
      const int64_t rows = int64_t(r.n_slots(t)) * t.slot, pan = int64_t(r.m_slots(t)) * t.slot;
      t.n_base = 0;                      // V, T
      u.n_base = 0;
      x.m_base = u.m_base = rows;        // U
      t.m_base = 2 * rows;               // columns of D^-1
      x.n_base = 2 * rows + pan;         // rows of D^-1
      r.conv(t, q, kOpV, kOpD);
      r.conv(x, q, kOpDr, kOpU);
      r.product(t, q, to);
      r.product(x, q, xo);
      r.conv(u, q, kOpT);
      r.product(u, q, uo);
      kernels += 9;
    }
    pf.end(a, P_PANEL, st, 0.0, 0.0, kernels);
  }
  if (bw > b) {
    cudaEvent_t a = pf.begin(st);
    int kernels = 0;
    auto slots = [&](int f) { return gen_refine_slots(dims_of(s[f], m[f], p0, 0, b), b); };
    for (const Piece& q : pieces_of(nact, sh.nb, sc.plane_bytes, true, slots)) {
      const int kt = (std::min(rns_block(b), s[q.f0] - p0) + kK - 1) / kK;
      Job t, u;
      const int to = r.job(t, kResid, q, p0, 0, kt), uo = r.job(u, kRefine, q, p0, 0, kt);
      if (to == 0) continue;
      t.n_base = u.n_base = 0;  // rows of B, then of X
      t.m_base = u.m_base = int64_t(r.n_slots(t)) * t.slot;  // columns of X, then of R
      r.conv(t, q, kOpBr, kOpB);
      r.product(t, q, to);
      r.conv(u, q, kOpXr, kOpRc);
      r.product(u, q, uo);
      kernels += 6;
    }
    pf.end(a, P_PANEL, st, 0.0, 0.0, kernels);
  }
  const bool joint = r.update_k(nact, p0) <= rns_block(b);
  auto slots = [&](int f) { return schur_slots(dims_of(s[f], m[f], p0, 0, b)); };
  for (const Piece& q : pieces_of(nact, sh.nb, sc.plane_bytes, true, slots)) {
    const int kt = (std::min(rns_block(b), s[q.f0] - p0) + kK - 1) / kK;
    Job l, u, x;
    const int lo = r.job(l, kPanel, q, p0, 0, kt), uo = r.job(u, kSchur, q, p0, 0, kt), xo = r.job(x, kPanelU, q, p0, 0, kt);
    if (lo == 0) continue;
    const int64_t rows = int64_t(r.n_slots(l)) * l.slot;
    l.n_base = u.n_base = 0;       // W, then L
    u.m_base = x.m_base = rows;    // A[B,S]
    l.m_base = x.n_base = 2 * rows;  // columns, then rows of B^-1
    double fl = 0;
    if (pf.on)
      for (int f = q.f0; f < q.f0 + q.nf; ++f) {
        const Dims d = dims_of(s[f], m[f], p0, 0, b);
        fl += 16.0 * q.np * d.mp * double(d.bw) * d.bw;
      }
    cudaEvent_t a = pf.begin(st);
    r.conv(l, q, kOpW, kOpB);
    r.product(l, q, lo);
    if (joint) r.conv(u, q, kOpL, kOpA);
    else r.conv(x, q, kOpA);
    r.conv(x, q, kOpXr);
    r.product(x, q, xo);
    pf.end(a, P_PANEL, st, fl, 0.0, 7, fl * kRnsModuli);
    if (!joint) continue;
    a = pf.begin(st);
    r.product(u, q, uo);
    const double sfl = pf.on ? r.update_flops(q, p0) : 0.0;
    pf.end(a, P_SCHUR, st, sfl, 0.0, 2, sfl * kRnsModuli);
  }
  if (!joint) r.apart(nact, p0, sh.nb, pf);
}

void rns_selinv_block_gen(const pexsi_plan* p, const Level& lv, const RnsScratch& sc, double2* Y, double2* F, int nact,
                          int p0, int nb, Profiler& pf, cudaStream_t st) {
  const int b = p->b, *s = lv.s.data(), *m = lv.m.data();
  Runner<double2> r{sc, F, Y, s, m, lv.off.data(), p->sym.front_elems, b, st, 1};
  auto slots = [&](int f) { return tak_slots(dims_of(s[f], m[f], p0, 0, b)); };
  for (const Piece& q : pieces_of(nact, nb, sc.plane_bytes, true, slots)) {
    int k = 32;
    double fl = 0;
    for (int f = q.f0; f < q.f0 + q.nf; ++f) {
      const Dims d = dims_of(s[f], m[f], p0, 0, b);
      k = std::max(k, d.mp);
      fl += 16.0 * q.np * double(d.bw) * d.mp * (q.rtn > 0 ? double(q.rtn) * kRnsTile : d.mp);
    }
    const int kt = (k + kK - 1) / kK;
    Job t, u, g;
    const int to = r.job(t, kTak, q, p0, 0, kt), uo = r.job(u, kTakU, q, p0, 0, kt), go = r.job(g, kDiag, q, p0, 0, kt);
    const bool last = q.rtn == 0 || q.rt0 + q.rtn >= tiles128(dims_of(s[q.f0], m[q.f0], p0, 0, b).mp);
    // the panel operand (columns of L, then rows of U), then the rows or columns of Y[S,S], then the columns of Y[S,B]
    t.m_base = u.n_base = g.n_base = 0;
    t.n_base = u.m_base = g.m_base = int64_t(r.m_slots(t)) * t.slot;
    if (to > 0) {
      cudaEvent_t a = pf.begin(st);
      r.conv(t, q, kOpLt, kOpYr);
      r.product(t, q, to);
      r.conv(u, q, kOpUr, kOpYc);
      r.product(u, q, uo);
      pf.end(a, P_OFFDIAG, st, fl, 0.0, 6, fl * kRnsModuli);
    }
    if (last) {
      cudaEvent_t a = pf.begin(st);
      if (to > 0) r.conv(g, q, kOpYtc);
      r.product(g, q, go);
      pf.end(a, P_DPART, st, 0.0, 0.0, 3);
    }
  }
}

template void rns_factor_block<double>(const pexsi_plan*, const Level&, const RnsScratch&, double*, double*, int, int,
                                       const BatchShifts&, DevStatus, Profiler&, cudaStream_t);
template void rns_factor_block<double2>(const pexsi_plan*, const Level&, const RnsScratch&, double2*, double2*, int, int,
                                        const BatchShifts&, DevStatus, Profiler&, cudaStream_t);

}  // namespace pexsi
