// crt.cuh -- FP64-accurate contraction T = A B^T through residue numbers: the
// arithmetic (the kernel is k_crt_gemm, crt_gemm.cuh).
//
// Each row of A and of B is scaled by a power of two and rounded to integers
// of b bits; the integer product S = sum_k A_k B_k is then exact, |S| <= K
// 2^(bA + bB) < M / 2, and known from its residues modulo pairwise coprime
// m_1 .. m_n, M = prod m_i (Chinese remainder theorem; the emulation of
// accurate matrix products this way: Ozaki, Uchino, Imamura, "Ozaki Scheme II",
// arXiv:2504.08009).  With m_i <= 513 the symmetric residues are at most 256 in
// magnitude, integers that bf16 holds exactly, so a residue matrix costs ONE
// bf16 tensor-core product: 13 products for FP64 accuracy where the error-free
// slices of ozaki.cuh need 28.  A chunk of 256 K sums products of
// at most 2^16 to at most 2^24: exact in the FP32 accumulator whatever its
// rounding.  Each chunk is reduced modulo m_i and the residues added up.
#pragma once
#include "crt_types.cuh"
#include "ozaki_digits.cuh"
#include "ozaki_types.cuh"
#include "tc_ptx.cuh"

namespace iscsi {

// v 2^(bits - e) rounded to an integer, |v| < 2^e, bits <= 62 (in integer
// arithmetic; zeros, subnormals and what is not finite give 0)
__device__ __forceinline__ long long crt_fixed(double v, int e, int bits) {
  const long long b = __double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7FF);
  if ((unsigned)(E - 1) >= 0x7FEu) return 0;
  const long long m = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int sh = 1075 - E + e - bits;  // v = m 2^(E - 1075); >= 53 - bits when |v| < 2^e
  long long N = 0;
  if (sh <= 0) N = m << (-sh & 15);
  else if (sh < 55) N = (m + (1ll << (sh - 1))) >> sh;
  return b < 0 ? -N : N;
}

// Two integers in limbs as packed FP32: a limb in the low mantissa bits of 2^23, less a constant.
// LIMBS = 4, |N| <= 2^59: N = l0 + l1 2^15 + l2 2^30 + l3 2^45 with -2^14 <= l0, l1, l2 < 2^14
// (balanced: the fields of N + 2^14 (1 + 2^15 + 2^30), less 2^14) and |l3| <= 2^14.
// LIMBS = 5, |N| <= 2^62: l0 + l1 2^13 + .. + l4 2^52, 0 <= l0 .. l3 < 2^13, |l4| <= 2^10.
template <int LIMBS>
struct CrtLimbs2 {
  unsigned long long l[LIMBS];
};
template <int LIMBS>
__device__ __forceinline__ CrtLimbs2<LIMBS> crt_limbs2(long long a, long long b) {
  static_assert(LIMBS == 4 || LIMBS == 5, "limbs of 15 or of 13 bits");
  constexpr int W = LIMBS == 4 ? 15 : 13;
  constexpr uint32_t kMask = (1u << W) - 1, kBias = LIMBS == 4 ? 1u << 14 : 0u;
  if (LIMBS == 4) {
    constexpr long long kAll = (1ll << 14) + (1ll << 29) + (1ll << 44);
    a += kAll;
    b += kAll;
  }
  auto mant = [](long long x) { return ((uint32_t)x & kMask) | 0x4B000000u; };
  auto pair = [](uint32_t lo, uint32_t hi) { return ((unsigned long long)hi << 32) | lo; };
  const unsigned long long k0 = pair(0xCB000000u + kBias, 0xCB000000u + kBias);  // -(2^23 + bias), twice
  CrtLimbs2<LIMBS> r;
#pragma unroll
  for (int i = 0; i + 1 < LIMBS; ++i) r.l[i] = tc::add2(pair(mant(a >> (W * i)), mant(b >> (W * i))), k0);
  // the last one signed: added to 1.5 2^23
  r.l[LIMBS - 1] = tc::add2(pair(0x4B400000u + (uint32_t)(int)(a >> (W * (LIMBS - 1))),
                                 0x4B400000u + (uint32_t)(int)(b >> (W * (LIMBS - 1)))),
                            pair(0xCB400000u, 0xCB400000u));
  return r;
}

// Residues of eight consecutive K values for every modulus, one 16-byte store
// each.  t = l0 + l1 c1 + .. is congruent to N, an exact FP32 integer (|t| below 2^23.4
// with four limbs, 2^22.2 with five); its quotient by m is rounded by adding 1.5 2^23 with
// an error below 0.8 of the 1 / (2 m) that separates t / m from a tie (over the sixteen
// moduli), so |t - q m| <= 256 and the upper halves of the floats are the bf16 residues.
// Packed FP32, 3.5 instructions per residue with four limbs, 4 with five, which bound it (five limbs: full
// CI in 60 orbitals 188 us, 4 + 4 electrons in 16 787; four 161 and 667); integer arithmetic took ~13.
template <int LIMBS>
__device__ __forceinline__ void crt_store8(const CrtLimbs2<LIMBS> (&x)[4], const CrtMods& M, __nv_bfloat16* out,
                                           long long mod_stride) {
  const unsigned long long mg = tc::f32x2(12582912.0f, 12582912.0f), ng = tc::f32x2(-12582912.0f, -12582912.0f);
#pragma unroll 2
  for (int i = 0; i < M.nm; ++i) {
    const unsigned long long inv = M.inv[i], neg = M.neg[i];
    uint32_t pk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      unsigned long long t = x[j].l[0];
#pragma unroll
      for (int k = 1; k < LIMBS; ++k) t = tc::fma2(x[j].l[k], M.c[k - 1][i], t);
      const unsigned long long q = tc::add2(tc::fma2(t, inv, mg), ng);
      const unsigned long long r = tc::fma2(q, neg, t);
      pk[j] = __byte_perm((uint32_t)r, (uint32_t)(r >> 32), 0x7632);
    }
    *reinterpret_cast<uint4*>(out) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    out += mod_stride;
  }
}

// S 2^e from the fraction of S / M held as hi 2^-32 + lo 2^-78 (mod 1, signed),
// built in integer arithmetic and rounded once
__device__ __forceinline__ double crt_value(unsigned long long a_lo, uint32_t a_hi, unsigned long long mman, int mexp,
                                            int e) {
  // 96-bit fraction (f2, lo)
  unsigned long long lo = a_lo << 18;
  uint32_t f2 = a_hi + (uint32_t)(a_lo >> 46);
  const bool neg = (f2 >> 31) != 0;
  if (neg) {
    lo = 0ull - lo;
    f2 = ~f2 + (lo == 0 ? 1u : 0u);
  }
  if ((f2 | (uint32_t)(lo >> 32) | (uint32_t)lo) == 0) return 0.0;
  // top 64 bits, leading one at bit 63
  unsigned long long top;
  int lz;
  if (f2) {
    lz = __clz(f2);
    top = ((unsigned long long)f2 << 32) | (lo >> 32);
    if (lz) top = (top << lz) | ((unsigned long long)((uint32_t)lo) >> (32 - lz));
  } else {
    lz = __clzll((long long)lo);
    top = lo << lz;
    lz += 32;
  }
  const unsigned long long p = __umul64hi(top, mman);  // |S| = p 2^(mexp - lz) to 2^-62
  const long long q = (long long)(p >> 1);
  return oz_i64_scaled(neg ? -q : q, mexp - lz + 1 + e);
}

}  // namespace iscsi
