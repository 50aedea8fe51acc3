// crt_gemm.cuh -- the tensor-core kernel of the residue-number contraction
// (arithmetic in crt.cuh).
//
// k_crt_gemm: persistent CTA pairs (tcgen05 cta_group::2) on 256 x 256 tiles.
// A plain bf16 product needs (m + n) / (m n) operand bytes per flop; one SM's
// 128 x 256 tile would read 96 bytes a clock from L2 at the full MMA rate, a
// pair's 256 x 256 tile 64 per SM, because each CTA loads only its half of B.
#pragma once
#include "crt.cuh"
#include "crt_types.cuh"
#include "ozaki_types.cuh"
#include "tc_ptx.cuh"

namespace iscsi {

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
      const uint32_t dA0 = (uint32_t)tc::smem_desc_sw128(s0), dB0 = dA0 + (CRT_A_BYTES >> 4);
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
            const uint32_t off = (uint32_t)(st * (CRT_STAGE_BYTES >> 4));
            const uint32_t d = tmem + (uint32_t)(buf * CRT_MAXN);
#pragma unroll
            for (int j = 0; j < CRT_BK / 16; ++j)
              tc::mma_bf16_pair_sw128(d, dA0 + off + 2 * j, dB0 + off + 2 * j, idesc, first && j == 0 ? 0u : 1u);
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
