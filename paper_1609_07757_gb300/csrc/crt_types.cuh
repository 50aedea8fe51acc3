// crt_types.cuh -- records of the residue-number contraction (kernels in
// crt.cuh, host side in crt.cu): FP64-accurate products T = A B^T from one
// bf16 tensor-core product per modulus.
#pragma once
#include <cuda.h>

#include <cstdint>
#include <vector>

namespace iscsi {

constexpr int kCrtMaxMods = 16;
constexpr int CRT_BM = 128;         // rows of A per CTA (256 per CTA pair)
constexpr int CRT_BK = 64;          // K per stage: one 128-byte row of bf16
constexpr int CRT_MAXN = 256;       // columns per tile (both CTAs' accumulators hold all of them)
constexpr int CRT_CHUNK = 4;        // stages per accumulator: K = 256 products of at most 2^16 stay exact in FP32
constexpr int CRT_STAGES = 7;
constexpr int CRT_A_BYTES = CRT_BM * CRT_BK * 2;
constexpr int CRT_B_BYTES = CRT_MAXN / 2 * CRT_BK * 2;
constexpr int CRT_STAGE_BYTES = CRT_A_BYTES + CRT_B_BYTES;
constexpr int CRT_SMEM_BYTES = CRT_STAGES * CRT_STAGE_BYTES + 1024;
constexpr int CRT_EPI_WARPS = 8;    // two per TMEM lane quarter, half of the columns each
constexpr int CRT_THREADS = 64 + 32 * CRT_EPI_WARPS;

// Pairwise coprime moduli whose symmetric residues are at most 256 in
// magnitude (integers that bf16 holds exactly), largest first.
constexpr int kCrtModuli[kCrtMaxMods] = {513, 512, 511, 509, 505, 503, 499, 493, 491, 487, 481, 479, 473, 467, 463, 461};

// Constants of the first nm moduli, each FP32 value twice in a 64-bit word
// (packed operations on two elements): the limbs' weights mod m (symmetric: 2^15, 2^30 and
// 2^45, or 2^13, 2^26, 2^39 and 2^52 for five limbs), 1 / m and -m.
struct CrtMods {
  int nm;
  int m[kCrtMaxMods];
  unsigned long long c[4][kCrtMaxMods], inv[kCrtMaxMods], neg[kCrtMaxMods];
};

// Reconstruction S = F M, F = sum_i r_i (M/m_i)^-1 / m_i mod 1, as a 78-bit
// fraction: weight i is hi 2^-32 + lo 2^-78 (lo of 46 bits, as 32 + 14).
struct CrtWeights {
  uint32_t hi[kCrtMaxMods], lo1[kCrtMaxMods], lo0[kCrtMaxMods];
  // multiples of m_i that make a pass's summed residues non-negative: first pass, later ones
  int off[kCrtMaxMods], off_next[kCrtMaxMods];
  uint32_t start_hi;             // minus the offsets' share of the sums (their rounding cancels)
  unsigned long long start_lo;
  unsigned long long mman;       // M = mman 2^mexp, top bit of mman set (truncated)
  int mexp;
};

// One product R[M][N] = A[M][K] B[N][K]^T, a residue matrix per modulus.
// Operands: bf16 residues in blocks of `rows` x 64 K (rows: 128 for A, bt for
// B), block (modulus, row block, k block) at index (mod * nblk + rb) * nkb +
// kb, K contiguous inside a row.  The tensor maps see them as [blocks * rows][64].
// Output tile (row block rt of 128, column tile nt), modulus mod: 128 x ntile
// signed 16-bit residues (at most 257 in magnitude) at ((rt * tn + nt) * nm + mod) * 128 * ntile, in groups of 8
// columns: [column group][row][8].
struct CrtProblem {
  CUtensorMap a, b;
  int16_t* res;
  int nblk_a, nkb_a, nblk_b, nkb_b;
  int ntile, tn, nm, rt;  // columns per tile (a multiple of 16), column tiles, moduli, row blocks in use
};

// One tile of one modulus: k blocks [kb0, kb0 + nkb) of product prob, then
// [kb0b, kb0b + nkbb) of product probb into the same sums (the same-spin part
// M_alpha C + C M_beta^T; nkbb = 0: none).  The tile is prob's.
struct CrtItem {
  int prob, mt, nt, mod;
  int kb0, nkb, ntile, probb;
  int kb0b, nkbb, pad0, pad1;
};

}  // namespace iscsi
