// crt.cuh -- FP64-accurate contraction T = A B^T through residue numbers.
//
// Each row of A and of B is scaled by a power of two and rounded to integers
// of b bits; the integer product S = sum_k A_k B_k is then exact, |S| <= K
// 2^(bA + bB) < M / 2, and known from its residues modulo pairwise coprime
// m_1 .. m_n, M = prod m_i (Chinese remainder theorem; the emulation of
// accurate matrix products this way: Ozaki, Uchino, Imamura, "Ozaki Scheme II",
// arXiv:2504.08009).  With m_i <= 513 the symmetric residues are at most 256 in
// magnitude, integers that bf16 holds exactly, so a residue matrix costs ONE
// bf16 tensor-core product: 12 or 13 products for FP64 accuracy where the
// error-free slices of ozaki.cuh need 28.  A chunk of 256 K sums products of
// at most 2^16 to at most 2^24: exact in the FP32 accumulator whatever its
// rounding.  Each chunk is reduced modulo m_i and the residues added up.
//
// k_crt_gemm: persistent CTA pairs (tcgen05 cta_group::2) on 256 x 256 tiles.
// A plain bf16 product needs (m + n) / (m n) operand bytes per flop; one SM's
// 128 x 256 tile would read 96 bytes a clock from L2 at the full MMA rate, a
// pair's 256 x 256 tile 64 per SM, because each CTA loads only its half of B.
#pragma once
#include "crt_types.cuh"
#include "ozaki_digits.cuh"
#include "ozaki_types.cuh"
#include "tc_ptx.cuh"

namespace iscsi {

// v 2^(bits - e) rounded to an integer, |v| < 2^e, bits <= 53 (in integer
// arithmetic; zeros and subnormals give 0)
__device__ __forceinline__ long long crt_fixed(double v, int e, int bits) {
  const long long b = __double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) return 0;
  const long long m = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int sh = 1075 - E + e - bits;  // v = m 2^(E - 1075); >= 0 when |v| < 2^e
  long long N = 0;
  if (sh <= 0) N = m;  // only sh = 0 occurs
  else if (sh < 55) N = (m + (1ll << (sh - 1))) >> sh;
  return b < 0 ? -N : N;
}

// Two integers |N| <= 2^52 as N = l0 + l1 2^13 + l2 2^26 + l3 2^39 (0 <= l0, l1,
// l2 < 2^13), the limbs as packed FP32: a limb in the low mantissa bits of 2^23
// (l3, signed: added to 1.5 2^23), less that constant.
struct CrtLimbs2 {
  unsigned long long l0, l1, l2, l3;
};
__device__ __forceinline__ CrtLimbs2 crt_limbs2(long long a, long long b) {
  auto mant = [](uint32_t x) { return (x & 0x1FFFu) | 0x4B000000u; };
  auto pair = [](uint32_t lo, uint32_t hi) { return ((unsigned long long)hi << 32) | lo; };
  const unsigned long long k0 = pair(0xCB000000u, 0xCB000000u);  // -2^23, twice
  CrtLimbs2 r;
  r.l0 = tc::add2(pair(mant((uint32_t)a), mant((uint32_t)b)), k0);
  r.l1 = tc::add2(pair(mant((uint32_t)a >> 13), mant((uint32_t)b >> 13)), k0);
  r.l2 = tc::add2(pair(mant((uint32_t)(a >> 26)), mant((uint32_t)(b >> 26))), k0);
  r.l3 = tc::add2(pair(0x4B400000u + (uint32_t)((int)(a >> 32) >> 7), 0x4B400000u + (uint32_t)((int)(b >> 32) >> 7)),
                  pair(0xCB400000u, 0xCB400000u));
  return r;
}

// Residues of eight consecutive K values for every modulus, one 16-byte store
// each.  t = l0 + l1 c1 + l2 c2 + l3 c3 is congruent to N, an exact FP32 integer
// (|t| < 2^23); its quotient by m is rounded by adding 1.5 2^23 with an error
// below 2^-11, under the 1 / (2 m) > 2^-10.1 that separates t / m from a tie, so
// |t - q m| <= 256 and the upper halves of the floats are the bf16 residues.
// Packed FP32: 3.5 instructions per residue, where integer arithmetic took ~13
// (4 + 4 electrons in 16 orbitals, operand kernel: 750 us).
__device__ __forceinline__ void crt_store8(const CrtLimbs2 (&x)[4], const CrtMods& M, __nv_bfloat16* out,
                                           long long mod_stride) {
  const unsigned long long mg = tc::f32x2(12582912.0f, 12582912.0f), ng = tc::f32x2(-12582912.0f, -12582912.0f);
#pragma unroll 2
  for (int i = 0; i < M.nm; ++i) {
    const unsigned long long c1 = M.c1[i], c2 = M.c2[i], c3 = M.c3[i], inv = M.inv[i], neg = M.neg[i];
    uint32_t pk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned long long t = tc::fma2(x[j].l3, c3, tc::fma2(x[j].l2, c2, tc::fma2(x[j].l1, c1, x[j].l0)));
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

constexpr uint32_t CRT_TMEM_COLS = 512;  // two accumulators of 256 columns

// Per CTA of a pair:
//   warp 0    (one lane) loads its half of every stage: 128 rows of A, ntile / 2
//             rows of B, 64 K each; both CTAs' bytes count on the even CTA's
//             full[stage];
//   warp 1    (even CTA only, one elected lane) issues the stage's four MMAs of 256 x
//             ntile x 16 for the pair, releases the stage in both CTAs and, every
//             CRT_CHUNK stages, hands the accumulator to both epilogues;
//   warps 2-9 add each chunk's exact integers (FP32 in tensor memory) into
//             residues' sums while the next chunk runs into the other accumulator,
//             and store the tile's residues.
// Every wait is bounded (oz_wait_bounded).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(CRT_THREADS, 1)
    k_crt_gemm(const CrtProblem* __restrict__ probs, const CrtItem* __restrict__ items,
               const int* __restrict__ pair_start, const __grid_constant__ CrtMods mods, int* __restrict__ err) {
  extern __shared__ unsigned char crt_smem_raw[];
  // the two CTAs' buffers must sit at the same offsets: align the address itself (equal in both)
  unsigned char* smem = (unsigned char*)(((uintptr_t)crt_smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t s0 = tc::smem_u32(smem);
  __shared__ uint64_t full_b[CRT_STAGES], empty_b[CRT_STAGES], accf_b[2], acce_b[2], drain_b;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;

  const uint32_t rank = tc::cluster_ctarank();
  const int pair = blockIdx.x >> 1;
  const int it0 = pair_start[pair], it1 = pair_start[pair + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < CRT_STAGES; ++s) {
      tc::mbar_init(tc::smem_u32(&full_b[s]), 1);
      tc::mbar_init(tc::smem_u32(&empty_b[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(tc::smem_u32(&accf_b[b]), 1);
      tc::mbar_init(tc::smem_u32(&acce_b[b]), 2 * CRT_EPI_WARPS);
    }
    tc::mbar_init(tc::smem_u32(&drain_b), 1);
    abort_s = 0;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    tc::tmem_alloc_pair(tc::smem_u32(&tmem_s), CRT_TMEM_COLS);
    tc::tmem_relinquish_pair();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::cluster_sync();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_s;

  auto wait = [&](uint64_t* bar, uint32_t parity, int site, int detail) -> bool {
    return oz_wait_bounded(bar, parity, site, detail, &abort_s, OZ_SPIN);
  };

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int it = it0; it < it1 && ok; ++it) {
        const CrtItem I = items[it];
        const int bt = I.ntile >> 1;
        const uint32_t bytes = 2u * (uint32_t)(CRT_A_BYTES + bt * CRT_BK * 2);
        for (int seg = 0; seg < 2 && ok; ++seg) {
          const int nkb = seg ? I.nkbb : I.nkb, kb0 = seg ? I.kb0b : I.kb0;
          if (nkb == 0) continue;
          const CrtProblem& P = probs[seg ? I.probb : I.prob];
          const long long ra = (long long)I.mod * P.nblk_a + 2 * I.mt + rank;
          const long long rb = (long long)I.mod * P.nblk_b + 2 * I.nt + rank;
          int ya = (int)((ra * P.nkb_a + kb0) * CRT_BM), yb = (int)((rb * P.nkb_b + kb0) * bt);
          for (int k = 0; k < nkb; ++k, ++g, ya += CRT_BM, yb += bt) {
            const int st = g % CRT_STAGES;
            if (g >= CRT_STAGES && !wait(&empty_b[st], ((g / CRT_STAGES) - 1) & 1, OZ_SITE_EMPTY, it - it0)) {
              ok = false;
              break;
            }
            const uint32_t fb = tc::smem_u32(&full_b[st]);
            if (rank == 0) tc::mbar_arrive_expect_tx(fb, bytes);
            const uint32_t fl = tc::mapa(fb, 0);
            const uint32_t sa = s0 + st * CRT_STAGE_BYTES;
            tc::tma_load_2d_pair(sa, &P.a, 0, ya, fl);
            tc::tma_load_2d_pair(sa + CRT_A_BYTES, &P.b, 0, yb, fl);
          }
        }
      }
      // copies still in flight (only after an abort) must land before the
      // pair's shared memory is released: the last phase of each stage
      if (rank == 0)
        for (int q = g - CRT_STAGES > 0 ? g - CRT_STAGES : 0; q < g; ++q)
          tc::mbar_wait_bounded(tc::smem_u32(&full_b[q % CRT_STAGES]), (q / CRT_STAGES) & 1, OZ_SPIN);
    }
  } else if (warp == 1) {
    // The whole warp runs the loop and one elected lane issues: in a branch of a single lane
    // the compiler moves every MMA operand through per-thread registers, ~50 cycles an MMA, and the
    // tensor core ran dry between them (a stage of four: 722 cycles against 512 of products).
    if (rank == 0) {
      int g = 0, st = 0, chunk = 0;
      uint32_t ph = 0;
      bool ok = true;
      const uint64_t dA0 = tc::smem_desc_sw128(s0), dB0 = tc::smem_desc_sw128(s0 + CRT_A_BYTES);
      for (int it = it0; it < it1 && ok; ++it) {
        const int nkb = __ldg(&items[it].nkb) + __ldg(&items[it].nkbb);
        const uint32_t idesc = tc::idesc_bf16_f32(2 * CRT_BM, __ldg(&items[it].ntile));
        for (int k = 0; k < nkb; ++k, ++g) {
          const int buf = chunk & 1;
          const bool first = k % CRT_CHUNK == 0, last = k % CRT_CHUNK == CRT_CHUNK - 1 || k == nkb - 1;
          if (first && chunk >= 2) {
            ok = wait(&acce_b[buf], ((chunk >> 1) - 1) & 1, OZ_SITE_FREE, chunk);
            if (!__all_sync(0xffffffffu, ok)) {
              ok = false;
              break;
            }
          }
          ok = wait(&full_b[st], ph, OZ_SITE_FULL, g);
          if (!__all_sync(0xffffffffu, ok)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          if (tc::elect_one()) {
            const uint64_t off = (uint64_t)(st * (CRT_STAGE_BYTES >> 4));
            const uint32_t d = tmem + (uint32_t)(buf * CRT_MAXN);
#pragma unroll
            for (int j = 0; j < CRT_BK / 16; ++j)
              tc::mma_bf16_pair(d, dA0 + off + (uint64_t)(2 * j), dB0 + off + (uint64_t)(2 * j), idesc,
                                first && j == 0 ? 0u : 1u);
            tc::mma_commit_pair(tc::smem_u32(&empty_b[st]));
            if (last) tc::mma_commit_pair(tc::smem_u32(&accf_b[buf]));
          }
          __syncwarp();
          if (last) ++chunk;
          if (++st == CRT_STAGES) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {
        // let MMAs already issued finish before TMEM is released (bounded)
        if (tc::elect_one()) tc::mma_commit_pair(tc::smem_u32(&drain_b));
        __syncwarp();
        tc::mbar_wait_bounded(tc::smem_u32(&drain_b), 0, OZ_SPIN);
      }
    }
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const int row = quarter * 32 + lane;
    int chunk = 0;
    bool ok = true;
    CrtItem nx = items[it0];
    for (int it = it0; it < it1 && ok; ++it) {
      const CrtItem I = nx;
      if (it + 1 < it1) nx = items[it + 1];
      const int bt = I.ntile >> 1, c0 = half * bt;
      const int m = mods.m[I.mod];
      const float inv = 1.0f / (float)m;
      const unsigned long long inv2 = tc::f32x2(inv, inv), fm2 = tc::f32x2(-(float)m, -(float)m),
                               mg2 = tc::f32x2(12582912.0f, 12582912.0f), ng2 = tc::f32x2(-12582912.0f, -12582912.0f);
      // sums of the chunks' residues, two columns per word: at most 257 per chunk, exact
      unsigned long long acc[CRT_MAXN / 4];
#pragma unroll
      for (int j = 0; j < CRT_MAXN / 4; ++j) acc[j] = 0ull;
      // residues of two exact integers |x| <= 2^24 (at most m / 2 + 1 in magnitude): the quotient is
      // rounded by adding 1.5 2^23, x - q m is exact.  Packed FP32: a conversion to integer would take
      // the 16-lane XU pipe 2048 cycles per 128 x 256 chunk, as long as its MMAs, and unpacked FP32
      // held a stage at 814 cycles (packed: 636).
      auto fold = [&](unsigned long long x) -> unsigned long long {
        const unsigned long long q = tc::add2(tc::fma2(x, inv2, mg2), ng2);
        return tc::fma2(q, fm2, x);
      };
      const int nch = (I.nkb + I.nkbb + CRT_CHUNK - 1) / CRT_CHUNK;
      for (int ch = 0; ch < nch; ++ch, ++chunk) {
        const int buf = chunk & 1;
        const bool w_ok = wait(&accf_b[buf], (chunk >> 1) & 1, OZ_SITE_CHUNK, chunk);
        if (!__all_sync(0xffffffffu, w_ok)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
#pragma unroll
        for (int g = 0; g < CRT_MAXN / 32; ++g) {
          if (g * 16 >= bt) continue;
          uint32_t v[16];
          tc::tmem_ld16(tmem + lane_base + (uint32_t)(buf * CRT_MAXN + c0 + g * 16), v);
          tc::tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j)
            acc[g * 8 + j] = tc::add2(acc[g * 8 + j], fold(((unsigned long long)v[2 * j + 1] << 32) | v[2 * j]));
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive_cluster_relaxed(tc::mapa(tc::smem_u32(&acce_b[buf]), 0));
      }
      if (!ok) break;
      const CrtProblem& P = probs[I.prob];
      const int rt = 2 * I.mt + (int)rank;
      if (rt < P.rt) {
        int16_t* out = P.res + (((long long)rt * P.tn + I.nt) * P.nm + I.mod) * ((long long)CRT_BM * I.ntile) +
                        ((long long)(c0 >> 3) * CRT_BM + row) * 8;
#pragma unroll
        for (int g = 0; g < CRT_MAXN / 16; ++g) {
          if (g * 8 >= bt) continue;
          uint32_t w[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // the low mantissa bits of 1.5 2^23 + r are r in two's complement
            const unsigned long long r = tc::add2(fold(acc[g * 4 + j]), mg2);
            w[j] = __byte_perm((uint32_t)r, (uint32_t)(r >> 32), 0x5410);
          }
          *reinterpret_cast<uint4*>(out + (long long)g * CRT_BM * 8) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
  }
  __syncthreads();
  if (abort_s && threadIdx.x == 0) {
    atomicCAS(err, 0, abort_s + (int)min(blockIdx.x, 4095u) * OZ_WAIT_CTA);
    // the peer may have issued copies this CTA's barriers do not cover: let them land
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::cluster_sync();  // both CTAs are done with each other's barriers and tensor memory
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc_pair(tmem, CRT_TMEM_COLS);
  }
}

}  // namespace iscsi
