// tc32w.cuh -- the FP32-form contraction T = A * B^T on the bf16 tensor
// cores, tiles of 128 rows and BN = 256 or 128 columns (arithmetic in tc32.cuh): three
// bf16 terms per element, the six term pairs of order t + u <= 2, FP32
// accumulation in tensor memory over K chunks of 512 and round-to-nearest
// FP32 sums across chunks in registers.
//
// Two accumulators share the 512 TMEM columns: order 0 (A_0 B_0) has BN
// columns, orders 1 and 2 (five pairs, each at most 2^-8 of order 0) sum into
// another BN.  With BN = 128 there are two such buffers and the MMAs of chunk
// c + 1 run while the epilogue drains chunk c; with BN = 256 one, and the MMAs wait for
// the drain.  The MMAs of an element come in the same order for both, with the same results
// bit for bit.
//
// What bounds it is the issue of the MMAs, not the operands: without any loads the
// 128-column kernel took 94 % of its time (full CI n = 60: 834 us, tensor pipe 37 % busy), a
// K step of five MMAs (A_0 (B_0, B_1) as one of N = 256) taking 725 cycles of issue and waits against 384
// of products.  So BN = 256: six MMAs of N = 256 for twice the products; a stage of two K
// steps (TMA rows of 64 bytes, one wait for twelve MMAs); the stages of a turn of the ring unrolled, so
// that a descriptor is a base plus a constant, of which only the low word is computed.  Full CI
// n = 60, both spin parts in one launch: 834 -> 500 us, one sigma 1004 -> 671 (a step's and a tile's
// time: t3_tiles).
//
// Warp 0 loads (TMA; A in a box of 128 rows x all terms, B in boxes of 128 rows of a term), warp 1 issues
// the MMAs (its loop whole, one elected lane issuing), the others drain (BN / 64 per TMEM
// lane quarter, 64 columns each).  Problems, segments and tensor maps are the
// shared records (ozaki_types.cuh).  Every wait is bounded; a
// wait that runs out sets abort, the CTA waits (bounded) for its copies in
// flight, frees TMEM and reports through err.
#pragma once
#include <cuda_bf16.h>

#include "ozaki_types.cuh"
#include "tc_ptx.cuh"
#include "tc32.cuh"

namespace iscsi {

template <int BN>
struct T3wShape {
  static constexpr int STAGES = BN == 256 ? 3 : 4;
  static constexpr int A_SLICE = T3_BM * T3_STAGE_K * 2;  // bytes: 8192
  static constexpr int B_SLICE = BN * T3_STAGE_K * 2;
  static constexpr int STAGE = T3_S * (A_SLICE + B_SLICE);
  static constexpr int SMEM = STAGES * STAGE + 1024;
  static constexpr int BUFS = BN == 256 ? 1 : 2;
  static constexpr int EPI_WARPS = BN / 16;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;
};
constexpr int T3W_EPI_COLS = 64;
constexpr int T3W_TMEM_COLS = 512;

template <int BN>
__global__ void __launch_bounds__(T3wShape<BN>::THREADS, 1)
    k_tc32w_gemm(const OzProblem* __restrict__ probs, int nprobs, const OzSeg* __restrict__ segs,
                 const OzMaps* __restrict__ maps, float* tbase, float* const* __restrict__ tbases,
                 int* __restrict__ err) {
  using W = T3wShape<BN>;
  constexpr int T3W_STAGES = W::STAGES;
  extern __shared__ unsigned char t3w_smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)t3w_smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t s_stage0 = tc::smem_u32(smem);
  __shared__ uint64_t full_b[T3W_STAGES], empty_b[T3W_STAGES], chunk_b[2], free_b[2], drain_b;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  __shared__ OzSeg seg_s[OZ_MAX_SEGS];
  __shared__ int segid_s[OZ_MAX_SEGS];
  __shared__ int step0_s[OZ_MAX_SEGS + 1];
  __shared__ int nseg_s;

  int tile = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (probs[mid].tile_begin <= tile) lo = mid;
    else hi = mid - 1;
  }
  const OzProblem P = probs[lo];
  float* const Tp = P.t_rel ? (tbases ? tbases[P.tb] : tbase) + P.t : reinterpret_cast<float*>(P.t);
  const int tl = tile - P.tile_begin;
  const int m0 = (tl / P.tiles_n) * T3_BM, n0 = (tl % P.tiles_n) * BN;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int SPC = T3_CHUNK_STEPS;

  if (threadIdx.x == 0) {
    for (int s = 0; s < T3W_STAGES; ++s) {
      tc::mbar_init(tc::smem_u32(&full_b[s]), 1);
      tc::mbar_init(tc::smem_u32(&empty_b[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(tc::smem_u32(&chunk_b[b]), 1);
      tc::mbar_init(tc::smem_u32(&free_b[b]), 32 * W::EPI_WARPS);
    }
    tc::mbar_init(tc::smem_u32(&drain_b), 1);
    abort_s = 0;
    int ns = 0, steps = 0;
    for (int g = 0; g < P.seg_count && ns < OZ_MAX_SEGS; ++g) {
      OzSeg sg = segs[P.seg_begin + g];
      if (n0 >= sg.nrows_b || sg.K <= 0) continue;
      seg_s[ns] = sg;
      segid_s[ns] = P.seg_begin + g;
      step0_s[ns] = steps;
      steps += sg.K / T3_BK;
      ++ns;
    }
    step0_s[ns] = steps;
    nseg_s = ns;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(tc::smem_u32(&tmem_s), T3W_TMEM_COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_s;
  const int nseg = nseg_s;
  const int total = step0_s[nseg];
  const int nchunks = (total + SPC - 1) / SPC;

  // a wait that runs out records where (oz_wait_code) and stops every role
  auto wait = [&](uint64_t* bar, uint32_t parity, int site, int detail) -> bool {
    return oz_wait_bounded(bar, parity, site, detail, &abort_s, OZ_SPIN);
  };

  if (warp == 0) {
    // ---------------- producer (TMA): all terms of A and of B per K step
    if (lane == 0) {
      int it = 0;  // stages issued
      bool ok = true;
      for (int seg = 0; seg < nseg && ok; ++seg) {
        const OzSeg& S = seg_s[seg];
        const CUtensorMap *ma = &maps[segid_s[seg]].a, *mb = &maps[segid_s[seg]].b;
        const int ay = S.a_row0 + m0, by = S.b_row0 + n0;
        for (int k0 = 0; k0 < S.K; k0 += T3_STAGE_K, ++it) {
          const int st = it % T3W_STAGES;
          if (it >= T3W_STAGES && !wait(&empty_b[st], ((it / T3W_STAGES) - 1) & 1, OZ_SITE_EMPTY, it)) {
            ok = false;
            break;
          }
          const uint32_t fb = tc::smem_u32(&full_b[st]);
          const uint32_t sa = s_stage0 + st * W::STAGE;
          tc::mbar_arrive_expect_tx(fb, W::STAGE);
          tc::tma_load_3d(sa, ma, S.a_k0 + k0, ay, 0, fb);
          for (int t = 0; t < T3_S; ++t)
            for (int h = 0; h < BN / 128; ++h)
              tc::tma_load_3d(sa + T3_S * W::A_SLICE + t * W::B_SLICE + h * (W::B_SLICE / (BN / 128)), mb, S.b_k0 + k0,
                              by + 128 * h, t, fb);
        }
      }
      for (int g = it - T3W_STAGES > 0 ? it - T3W_STAGES : 0; g < it; ++g)
        tc::mbar_wait_bounded(tc::smem_u32(&full_b[g % T3W_STAGES]), (g / T3W_STAGES) & 1, OZ_SPIN);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the whole warp runs the loop, one elected lane issues
    // (in a branch of a single lane the compiler moves the MMAs' operands through per-thread
    // registers, and the tensor core runs dry between them)
    constexpr uint32_t N1 = tc::idesc_bf16_f32(T3_BM, BN), N2 = tc::idesc_bf16_f32(T3_BM, 256);
    const uint32_t dA0 = (uint32_t)tc::smem_desc_sw64(s_stage0), dB0 = dA0 + ((T3_S * W::A_SLICE) >> 4);
    constexpr uint32_t kSt = W::STAGE >> 4, kA = W::A_SLICE >> 4, kB = W::B_SLICE >> 4;
    // one K step: A_0 B_0 into order 0's columns, then the others' five pairs
    auto mmas = [&](uint32_t A, uint32_t B, uint32_t D0, bool restart) {
      const uint32_t D1 = D0 + BN;
      if constexpr (BN == 128) {
        // A_0 (B_0, B_1): order 0 and the first of orders 1-2 lie side by side, as B's slices do
        tc::mma_bf16_sw64(D0, A, B, N2, restart ? 0u : 1u);
      } else {
        tc::mma_bf16_sw64(D0, A, B, N1, restart ? 0u : 1u);
        tc::mma_bf16_sw64(D1, A, B + kB, N1, restart ? 0u : 1u);
      }
      tc::mma_bf16_sw64(D1, A + kA, B, N1, 1u);           // A_1 B_0
      tc::mma_bf16_sw64(D1, A, B + 2 * kB, N1, 1u);       // A_0 B_2
      tc::mma_bf16_sw64(D1, A + kA, B + kB, N1, 1u);      // A_1 B_1
      tc::mma_bf16_sw64(D1, A + 2 * kA, B, N1, 1u);       // A_2 B_0
    };
    bool ok = true;
    uint32_t ph = 0;
    int seg = -1, left = 0;      // steps left of the segment
    int g = 0, ch = 0, kin = 0;  // step, its chunk and place in it
    while (g < total && ok) {
#pragma unroll
      for (int st = 0; st < T3W_STAGES; ++st) {
        if (g >= total) break;
        while (left == 0) {
          ++seg;
          left = step0_s[seg + 1] - step0_s[seg];
        }
        const bool two = left > 1;
        left -= two ? 2 : 1;
        bool w = wait(&full_b[st], ph, OZ_SITE_FULL, g);
        if (kin == 0 && ch >= W::BUFS)
          w = w && wait(&free_b[ch % W::BUFS], ((ch / W::BUFS) - 1) & 1, OZ_SITE_FREE, ch);
        if (!__all_sync(0xffffffffu, w)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t A = dA0 + kSt * st, B = dB0 + kSt * st;
        uint32_t D = tmem + (uint32_t)((ch % W::BUFS) * 2 * BN);
        if (two && kin == SPC - 1) {
          // the chunk ends inside the stage (an odd segment before)
          if (tc::elect_one()) {
            mmas(A, B, D, false);
            tc::mma_commit(tc::smem_u32(&chunk_b[ch % W::BUFS]));
          }
          __syncwarp();
          ++ch;
          w = ch < W::BUFS || wait(&free_b[ch % W::BUFS], ((ch / W::BUFS) - 1) & 1, OZ_SITE_FREE, ch);
          if (!__all_sync(0xffffffffu, w)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          D = tmem + (uint32_t)((ch % W::BUFS) * 2 * BN);
          if (tc::elect_one()) {
            mmas(A + 2, B + 2, D, true);  // 32 bytes into the 64-byte rows
            tc::mma_commit(tc::smem_u32(&empty_b[st]));
            if (g + 2 == total) tc::mma_commit(tc::smem_u32(&chunk_b[ch % W::BUFS]));
          }
          kin = 1;
          g += 2;
        } else {
          const int n = two ? 2 : 1;
          if (tc::elect_one()) {
            mmas(A, B, D, kin == 0);  // the first step of a chunk restarts the buffer
            if (two) mmas(A + 2, B + 2, D, false);
            tc::mma_commit(tc::smem_u32(&empty_b[st]));
            if (kin + n == SPC || g + n == total) tc::mma_commit(tc::smem_u32(&chunk_b[ch % W::BUFS]));
          }
          kin += n;
          g += n;
          if (kin == SPC) {
            kin = 0;
            ++ch;
          }
        }
        __syncwarp();
      }
      ph ^= 1u;
    }
    if (__any_sync(0xffffffffu, abort_s != 0)) {
      if (tc::elect_one()) tc::mma_commit(tc::smem_u32(&drain_b));
      __syncwarp();
      tc::mbar_wait_bounded(tc::smem_u32(&drain_b), 0, OZ_SPIN);
    }
  } else {
    // ---------------- epilogue: lane quarter = warp % 4, columns 64 ((warp - 2) / 4)
    const int quarter = warp & 3;
    const int cbase = ((warp - 2) >> 2) * T3W_EPI_COLS;
    const uint32_t lane_base = ((uint32_t)(quarter * 32) << 16) + (uint32_t)cbase;
    float sums[T3W_EPI_COLS];
#pragma unroll
    for (int j = 0; j < T3W_EPI_COLS; ++j) sums[j] = 0.0f;
    bool ok = true;
    for (int ch = 0; ch < nchunks && ok; ++ch) {
      const int b = ch % W::BUFS;
      ok = wait(&chunk_b[b], (ch / W::BUFS) & 1, OZ_SITE_CHUNK, ch);
      if (!__all_sync(0xffffffffu, ok)) {  // tcgen05.ld is warp-collective
        ok = false;
        break;
      }
      tc::fence_after_sync();
      const uint32_t D = tmem + lane_base + (uint32_t)(b * 2 * BN);
#pragma unroll
      for (int c0 = 0; c0 < T3W_EPI_COLS; c0 += 8) {
        uint32_t r0[8], r1[8];
        tc::tmem_ld8(D + c0, r0);
        tc::tmem_ld8(D + BN + c0, r1);
        tc::tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) sums[c0 + j] += __uint_as_float(r0[j]) + __uint_as_float(r1[j]);
      }
      tc::fence_before_sync();
      tc::mbar_arrive(tc::smem_u32(&free_b[b]));
    }
    if (ok) {
      // the operand stages are done with: turn the warp's 32 x 64 block there, so that a store covers a
      // row's 32 columns (a thread's own row: 32 lines per store, 11 us per 128-column tile)
      float* buf = reinterpret_cast<float*>(smem) + (warp - 2) * 32 * (T3W_EPI_COLS + 1);
#pragma unroll
      for (int j = 0; j < T3W_EPI_COLS; ++j) buf[lane * (T3W_EPI_COLS + 1) + j] = sums[j];
      __syncwarp();
      const int rows = min(32, P.M - m0 - quarter * 32);
      float* dst = Tp + (long long)(m0 + quarter * 32) * P.ldt + n0 + cbase + lane;
      const bool c0 = n0 + cbase + lane < P.N, c1 = n0 + cbase + lane + 32 < P.N;
      // an accumulating block's old values eight rows at a time (a load before each store waited for 64 round
      // trips one after the other: 28 tiles of 3 + 3 electrons in 18 orbitals 40 us, now 20)
      for (int r0 = 0; r0 < rows; r0 += 8) {
        float o0[8], o1[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const bool on = P.accumulate && r0 + j < rows;
          o0[j] = on && c0 ? dst[(long long)(r0 + j) * P.ldt] : 0.0f;
          o1[j] = on && c1 ? dst[(long long)(r0 + j) * P.ldt + 32] : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = r0 + j;
          if (r >= rows) break;
          const float x0 = buf[r * (T3W_EPI_COLS + 1) + lane], x1 = buf[r * (T3W_EPI_COLS + 1) + lane + 32];
          if (c0) dst[(long long)r * P.ldt] = P.accumulate ? o0[j] + x0 : x0;
          if (c1) dst[(long long)r * P.ldt + 32] = P.accumulate ? o1[j] + x1 : x1;
        }
      }
    }
  }
  __syncthreads();
  if (abort_s && threadIdx.x == 0) atomicCAS(err, 0, abort_s + (int)min(blockIdx.x, 4095u) * OZ_WAIT_CTA);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, T3W_TMEM_COLS);
  }
}

}  // namespace iscsi
