// density.cu -- one- and two-body density matrices (Sec. "Density matrices",
// Eqs. d1 and d2) on the GPU, spin-resolved:
//   d1[s][p][q]       = <bra| a+_ps a_qs |ket>
//   d2[b][p][q][r][t] = <bra| a+_ps a+_ru a_tu a_qs |ket>,  (s,u) = aa, ab, bb
//
// The paper builds them with the sigma step's class loops, a product of two CI
// coefficients in place of the integral.  Here each two-body block is one
// Gram-type contraction of "lifted" vectors, on the tensor cores with FP64
// accuracy:
//   ab: L[(q,t)][(X,Y)] = <X,Y| a_tu a_qs |ket> (X, Y: strings with one alpha
//       and one beta electron removed -- the sigma step's hole strings and its
//       lift tables), so d2_ab[p,q,r,t] = sum_XY L_bra[(p,r)] L_ket[(q,t)];
//   aa: L[{u<v}][(Z,B)] = <Z| a_v a_u |A> c[A,B] with A = Z u {u,v} (Z: strings
//       with two alpha electrons removed), so d2_aa[p,q,r,t] =
//       s(p,r) s(q,t) sum_ZB L_bra[{p,r}] L_ket[{q,t}], s(x,y) = +1 if x < y,
//       -1 if x > y; bb likewise with the roles of the spins exchanged.
// Rows of L are orbital pairs sorted by excitation level and columns are
// grouped by their level class c, so class c only reaches the rows with level
// <= k - c: the product is a sum of prefix blocks, cut into row/column regions
// (the block's "staircase"), one tensor-core problem per region pair.  With
// ket = bra the result is symmetric and only the upper regions (and, in a
// diagonal region, the tiles right of each 128-row block's start) are computed.
// The products go through residue numbers (crt.cuh): one integer scale per vector,
// |d2| <= |bra| |ket| by Cauchy-Schwarz (a row of L holds each coefficient at most
// once), 13 moduli.  Contexts whose residues do not fit take the exact bf16
// slices of ozaki.cuh instead.
// An expansion kernel writes the n^4 tensors from the pair-indexed results.
// d1 comes from d2's partial trace when d2 is computed for that spin (sum_r
// d2_ss[p,q,r,r] = (N_s - 1) d1_s[p,q]), else
// from a direct kernel over the one-hole strings.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "crt.cuh"
#include "crt_host.cuh"
#include "internal.cuh"
#include "ozaki_digits.cuh"

namespace iscsi {

constexpr int kDmMaxBnd = 2 * kMaxElec + 2;

// ---------------------------------------------------------------------------
// host plan

struct DmPart {            // one column level class of a block (kb0, nkb: its 64-wide K blocks in the residues)
  int kb0 = 0, nkb = 0;
  int col_start = 0;       // first column in the block's column list
  int ncol = 0;            // columns (K)
  int rows = 0;            // rows reached (pairs with level <= k - c)
  int ld = 0;              // ncol rounded up to 16
  int rows_pad = 0;        // rows rounded up to 128
  size_t sl_off = 0;       // element offset of its slices in a slice workspace
};

struct DmBlock {
  int kind = 0;            // 0: ab, 1: aa, 2: bb
  int R = 0;               // rows of the pair-indexed result (largest part rows)
  std::vector<DmPart> parts;
  std::vector<int> bnd;    // region boundaries: 0 = bnd[0] < ... < bnd[nreg] = R
  size_t q_off = 0;        // double offset of the R x R result in the result workspace
  size_t exp_off = 0;      // int offset of its row exponents (parts x R128) in an exponent workspace
  int R128 = 0;
  // residue operands: R256 rows of nkb K blocks per modulus, at res_off
  int R256 = 0, nkb = 0;
  size_t res_off = 0;
  int bits = 0;            // of a row's largest element: 2 bits + log2(columns) below the moduli's product
  int row0 = 0;            // its first row in the lists of all blocks' rows
};

constexpr int kDmMods = 13, kDmModsMax = 16;  // moduli: the fewest with kDmBits bits
constexpr int kDmBits = 50;                    // (the slices: 49)
constexpr int kDmNotFinite = -(1 << 20);  // scale of a row with an infinity or NaN: its elements of the result are NaN

struct DensityPlan {
  bool built = false;
  // residues (unless they do not fit: ket = bra / general): operands of bra and
  // ket, output residues, scales
  bool no_room[2] = {false, false};
  CrtHeld res_held;
  DevBuf res_bra, res_ket, res_out, scale;  // scale: per row of bra, of ket, then partial maxima
  int nmods = kDmMods, res_rows = 0;        // moduli; rows of all blocks
  CrtJob res_job[2];             // ket = bra / general
  bool res_ready[2] = {false, false};
  size_t res_out_off[3] = {0, 0, 0};
  bool slices = false;           // the slice workspaces below are allocated
  DmBlock blk[3];
  // same-spin tables per spin: pair row of {u<v}, two-hole lift, column list (Z, other string)
  DevBuf pp_row[2], lift2[2], cols[2];
  int nz[2] = {0, 0};
  DevBuf q;                      // FP64 results of all blocks
  DevBuf sl_bra, sl_ket;         // bf16 slices of the bra / ket operands
  DevBuf ex_bra, ex_ket;         // row exponents
  size_t sl_elems = 0, q_elems = 0, ex_elems = 0;
  OzJob job_sym, job_gen;        // ket = bra (upper regions only) / general
  bool sym_ready = false, gen_ready = false;
  double bf16_flops[2] = {0, 0}; // bf16 MMA flops of one launch of each job
  double fp64_flops[2] = {0, 0}; // 2 M N K of the computed regions
  cudaEvent_t ev[2] = {nullptr, nullptr};  // around the last contraction launch
  bool timed = false;
  ~DensityPlan() {
    for (cudaEvent_t e : ev)
      if (e) cudaEventDestroy(e);
  }
};

void density_release(Context& ctx) {
  delete ctx.dm;
  ctx.dm = nullptr;
}

bool density_drop(Context& ctx) {
  if (!ctx.dm || ctx.dm->res_held.bytes == 0) return false;
  DensityPlan& P = *ctx.dm;
  for (DevBuf* d : {&P.res_bra, &P.res_ket, &P.res_out}) d->release();
  P.res_held.add(0 - P.res_held.bytes);
  P.res_ready[0] = P.res_ready[1] = false;
  return true;
}

static inline int rup(int x, int m) { return (x + m - 1) / m * m; }

// sorted position of an ascending orbital list: colex rank through the context's rank table
static int host_colex(const int* o, int ne) {
  long long r = 0;
  for (int i = 0; i < ne; ++i) r += binom_ll(o[i], i + 1);
  return (int)r;
}

// same-spin tables of spin s: pairs {u<v} sorted by level, strings Z with two
// electrons removed, the two-hole lift <Z| a_v a_u |A>, and the column list
// (Z, string of the other spin) grouped by level class
static int build_samespin(Context& ctx, DensityPlan& P, int s, DmBlock& B) {
  const int n = ctx.n, ne = ctx.sp[s].ne, nocc = ctx.sp[s].nocc, o = 1 - s;
  const SpinSpace& SO = ctx.sp[o];
  std::vector<int> pos(ctx.sp[s].count);
  ISCSI_CUDA(cudaMemcpy(pos.data(), ctx.sp[s].pos.p, sizeof(int) * pos.size(), cudaMemcpyDeviceToHost));
  // pairs u < v by level lu + lv, then (u, v)
  std::vector<std::pair<int, int>> pairs;
  for (int lev = 0; lev <= 2; ++lev)
    for (int u = 0; u < n; ++u)
      for (int v = u + 1; v < n; ++v)
        if ((u >= nocc) + (v >= nocc) == lev) pairs.push_back({u, v});
  const int npp = (int)pairs.size();
  std::vector<int> pp_row(n * n, -1), pair_lev(npp);
  for (int i = 0; i < npp; ++i) {
    pp_row[pairs[i].first * n + pairs[i].second] = i;
    pair_lev[i] = (pairs[i].first >= nocc) + (pairs[i].second >= nocc);
  }
  // strings Z of ne - 2 electrons (lexicographic), with their levels
  std::vector<std::vector<int>> Z;
  {
    int k = ne - 2;
    std::vector<int> c(k);
    for (int i = 0; i < k; ++i) c[i] = i;
    while (true) {
      Z.push_back(c);
      int i = k - 1;
      while (i >= 0 && c[i] == n - k + i) --i;
      if (i < 0) break;
      ++c[i];
      for (int j = i + 1; j < k; ++j) c[j] = c[j - 1] + 1;
    }
  }
  const int nz = (int)Z.size();
  if ((long long)npp * nz >= (1ll << 31)) {
    set_error("iscsi_density: two-hole string table too large");
    return kErrArg;
  }
  std::vector<int> zlev(nz), lift2((size_t)npp * nz, -1);
  for (int z = 0; z < nz; ++z) {
    int l = 0;
    for (int x : Z[z]) l += (x >= nocc);
    zlev[z] = l;
    for (int i = 0; i < npp; ++i) {
      int u = pairs[i].first, v = pairs[i].second;
      if (std::find(Z[z].begin(), Z[z].end(), u) != Z[z].end() ||
          std::find(Z[z].begin(), Z[z].end(), v) != Z[z].end())
        continue;
      std::vector<int> A = Z[z];
      A.push_back(u);
      A.push_back(v);
      std::sort(A.begin(), A.end());
      // a_u acts first on |A>, then a_v on |A \ u>: signs from the occupied orbitals below each
      int below_u = 0, below_v = 0;
      for (int x : A) {
        if (x < u) ++below_u;
        if (x < v && x != u) ++below_v;
      }
      lift2[(size_t)i * nz + z] = (pos[host_colex(A.data(), ne)] << 1) | ((below_u + below_v) & 1);
    }
  }
  // columns (Z, O) by class c = level(Z) + level(O); O over the other spin's level-sorted strings
  int maxc = 0;
  for (int z = 0; z < nz; ++z) maxc = std::max(maxc, zlev[z] + SO.maxlevel);
  std::vector<int> cols;
  B.parts.clear();
  for (int c = 0; c <= maxc; ++c) {
    DmPart pt;
    pt.col_start = (int)(cols.size() / 2);
    for (int z = 0; z < nz; ++z) {
      int lo = c - zlev[z];
      if (lo < 0 || lo > SO.maxlevel) continue;
      for (int O = SO.level_start[lo]; O < SO.level_start[lo + 1]; ++O) {
        cols.push_back(z);
        cols.push_back(O);
      }
    }
    pt.ncol = (int)(cols.size() / 2) - pt.col_start;
    int rows = 0;
    for (int i = 0; i < npp; ++i)
      if (pair_lev[i] <= ctx.kmax - c) rows = i + 1;
    pt.rows = rows;
    if (pt.ncol > 0 && pt.rows > 0) B.parts.push_back(pt);
  }
  P.nz[s] = nz;
  ISCSI_TRY(P.pp_row[s].alloc(sizeof(int) * pp_row.size()));
  ISCSI_CUDA(cudaMemcpy(P.pp_row[s].p, pp_row.data(), sizeof(int) * pp_row.size(), cudaMemcpyHostToDevice));
  ISCSI_TRY(P.lift2[s].alloc(sizeof(int) * std::max<size_t>(1, lift2.size())));
  ISCSI_CUDA(cudaMemcpy(P.lift2[s].p, lift2.data(), sizeof(int) * lift2.size(), cudaMemcpyHostToDevice));
  ISCSI_TRY(P.cols[s].alloc(sizeof(int) * std::max<size_t>(2, cols.size())));
  if (!cols.empty())
    ISCSI_CUDA(cudaMemcpy(P.cols[s].p, cols.data(), sizeof(int) * cols.size(), cudaMemcpyHostToDevice));
  return kOk;
}

static void set_regions(DmBlock& B) {
  std::vector<int> b = {0};
  for (const DmPart& p : B.parts) b.push_back(p.rows);
  std::sort(b.begin(), b.end());
  b.erase(std::unique(b.begin(), b.end()), b.end());
  B.bnd = b;
  B.R = b.back();
  B.R128 = rup(std::max(B.R, 1), OZ_BM);
}

static int plan_build(Context& ctx) {
  if (!ctx.dm) ctx.dm = new DensityPlan();
  DensityPlan& P = *ctx.dm;
  if (P.built) return kOk;
  cudaStream_t st = stream();
  ISCSI_CUDA(cudaStreamSynchronize(st));
  for (int b = 0; b < 3; ++b) {
    P.blk[b] = DmBlock();
    P.blk[b].kind = b;
  }
  // ab: the sigma step's pairs, hole-pair classes and lift tables
  if (ctx.have_ab || (ctx.na > 0 && ctx.nb > 0)) {
    DmBlock& B = P.blk[0];
    for (int c = 0; c < (int)ctx.cls.size(); ++c) {
      const ColClass& cc = ctx.cls[c];
      if (cc.ncol == 0 || cc.mrows == 0) continue;
      DmPart pt;
      pt.col_start = ctx.hp_class_start[c];
      pt.ncol = cc.ncol;
      pt.rows = cc.mrows;
      B.parts.push_back(pt);
    }
  }
  if (ctx.na >= 2) ISCSI_TRY(build_samespin(ctx, P, 0, P.blk[1]));
  if (ctx.nb >= 2) ISCSI_TRY(build_samespin(ctx, P, 1, P.blk[2]));
  // consecutive classes that reach the same rows are one part (their columns
  // are adjacent in the column lists): one longer K instead of several segments
  for (int b = 0; b < 3; ++b) {
    std::vector<DmPart> merged;
    for (const DmPart& pt : P.blk[b].parts) {
      if (!merged.empty() && merged.back().rows == pt.rows &&
          merged.back().col_start + merged.back().ncol == pt.col_start)
        merged.back().ncol += pt.ncol;
      else
        merged.push_back(pt);
    }
    P.blk[b].parts = merged;
  }
  // workspace layout
  size_t sl = 0, q = 0, ex = 0;
  for (int b = 0; b < 3; ++b) {
    DmBlock& B = P.blk[b];
    if (B.parts.empty()) continue;
    if ((int)B.parts.size() > OZ_MAX_SEGS) {
      set_error("iscsi_density: too many column classes for one tensor-core problem");
      return kErrArg;
    }
    set_regions(B);
    for (DmPart& pt : B.parts) {
      pt.ld = rup(pt.ncol, OZ_BK);
      pt.rows_pad = rup(pt.rows, OZ_BM);
      pt.sl_off = sl;
      sl += (size_t)OZ_S * pt.rows_pad * pt.ld;
      sl = (sl + 127) / 128 * 128;  // 256-byte aligned slice arrays (TMA wants 16)
    }
    B.q_off = q;
    q += (size_t)B.R * B.R;
    q = (q + 31) / 32 * 32;
    B.exp_off = ex;
    ex += (size_t)B.parts.size() * B.R128;
    B.R256 = rup(std::max(B.R, 1), 2 * CRT_BM);
    B.nkb = 0;
    for (DmPart& pt : B.parts) {
      pt.kb0 = B.nkb;
      pt.nkb = rup(pt.ncol, CRT_BK) / CRT_BK;
      B.nkb += pt.nkb;
    }
  }
  P.res_rows = 0;
  for (P.nmods = kDmMods;; ++P.nmods) {
    int least = 64;
    for (DmBlock& B : P.blk) {
      long long cols = 1;
      for (const DmPart& pt : B.parts) cols += pt.ncol;
      // |sum| <= cols 2^(2 bits), below half the moduli's product
      B.bits = std::min(52, (int)std::floor((crt_log2_product(P.nmods) - 1.01 - std::log2((double)cols)) / 2.0));
      if (!B.parts.empty()) least = std::min(least, B.bits);
    }
    if (least >= kDmBits || P.nmods == kDmModsMax) break;
  }
  for (DmBlock& B : P.blk) {
    B.row0 = P.res_rows;
    if (!B.parts.empty()) P.res_rows += B.R;
  }
  for (cudaEvent_t& e : P.ev) ISCSI_CUDA(cudaEventCreate(&e));
  P.sl_elems = sl;
  P.q_elems = q;
  P.ex_elems = ex;
  if (q) ISCSI_TRY(P.q.alloc(sizeof(double) * q));
  P.built = true;
  return kOk;
}

// workspaces of the slices (contexts without residues)
static int slices_alloc(DensityPlan& P) {
  if (P.slices) return kOk;
  if (P.sl_elems) ISCSI_TRY(P.sl_bra.alloc(sizeof(__nv_bfloat16) * P.sl_elems));
  if (P.ex_elems) {
    ISCSI_TRY(P.ex_bra.alloc(sizeof(int) * P.ex_elems));
    ISCSI_CUDA(cudaMemset(P.ex_bra.p, 0, sizeof(int) * P.ex_elems));
  }
  P.slices = true;
  return kOk;
}

// ---------------------------------------------------------------------------
// device: operand values, exponents, slices

struct DmGather {
  int kind;                       // 0 ab, 1 aa, 2 bb
  int n, nholeA, nholeB, nz;
  const int* pair_of;             // ab rows -> q * n + t
  const int* hp_inv;              // ab columns -> X * nholeB + Y
  const int* liftA;
  const int* liftB;
  const int* lift2;               // aa / bb: [pair row][Z] -> (string << 1 | neg) or -1
  const int* cols;                // aa / bb: (Z, other string) per column
  const int8_t* alevel;
  const int* nballow;
  const long long* off;
  unsigned div_mul;               // 2^div_shift / nholeB rounded up
  int div_shift;
};

// xy / nholeB for 0 <= xy < 2^31 by one wide product (div_mul, div_shift of gather_of)
__device__ __forceinline__ int dm_div(const DmGather& g, int xy) {
  return (int)(((unsigned long long)(unsigned)xy * g.div_mul) >> g.div_shift);
}

// x, or -x when bit 0 of neg is set, on the integer units (a negation by the FP64 pipe takes 64 cycles a warp)
__device__ __forceinline__ double dm_signed(double x, int neg) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)(neg & 1) << 63));
}

__device__ __forceinline__ double dm_value(const DmGather& g, int col, int row, const double* __restrict__ c) {
  int A, B, neg;
  if (g.kind == 0) {
    int xy = g.hp_inv[col];
    int X = dm_div(g, xy), Y = xy - X * g.nholeB;
    int qt = g.pair_of[row];
    int q = qt / g.n, t = qt - q * g.n;
    int ea = g.liftA[q * g.nholeA + X], eb = g.liftB[t * g.nholeB + Y];
    if (ea < 0 || eb < 0) return 0.0;
    A = ea >> 1;
    B = eb >> 1;
    neg = (ea ^ eb) & 1;
  } else {
    int z = g.cols[2 * col], O = g.cols[2 * col + 1];
    int e = g.lift2[(long long)row * g.nz + z];
    if (e < 0) return 0.0;
    A = g.kind == 1 ? (e >> 1) : O;
    B = g.kind == 1 ? O : (e >> 1);
    neg = e & 1;
  }
  if (B >= g.nballow[g.alevel[A]]) return 0.0;
  return dm_signed(c[g.off[A] + B], neg);
}

// One block per row of L (rows_pad rows, ld columns): gathers the row once
// (held in registers, kDmRowRegs values per thread, or re-gathered beyond
// that), takes the row exponent e with max |L[row][:]| 2^-e < 1 (0 for an
// all-zero row, and for the padding rows) and writes the row's slices
// out[s][row][k], zero padded.
// With STAGED (the alpha-beta block with at most kDmStage hole strings per
// spin) the row's lift entries -- a+_q |X> and a+_t |Y> for every X and Y,
// with the target alpha string's offset and allowed beta count -- are staged
// in shared memory first, so an element costs the hole-pair table and c.
constexpr int kDmRowRegs = 16;
constexpr int kDmStage = 256;
constexpr int kDmMaxSplit = 8;  // blocks per row in k_dm_cut
struct DmStageRow {
  int a[kDmStage], b[kDmStage], lim[kDmStage];
  long long off[kDmStage];
};

template <bool STAGED>
__device__ __forceinline__ double dm_row_value(const DmGather& g, const DmStageRow& S, int col, int row,
                                               const double* __restrict__ c) {
  if (!STAGED) return dm_value(g, col, row, c);
  const int xy = g.hp_inv[col];
  const int X = dm_div(g, xy), Y = xy - X * g.nholeB;
  const int ea = S.a[X], eb = S.b[Y];
  if (ea < 0 || eb < 0) return 0.0;
  const int B = eb >> 1;
  if (B >= S.lim[X]) return 0.0;
  return dm_signed(c[S.off[X] + B], ea ^ eb);
}

template <bool STAGED>
__global__ void __launch_bounds__(256) k_dm_lift_slice(DmGather g, int col_start, int ncol, int rows, int ld,
                                                       int rows_pad, const double* __restrict__ c,
                                                       int* __restrict__ e, __nv_bfloat16* __restrict__ out) {
  const int r = blockIdx.x;
  const long long total = (long long)rows_pad * ld;
  __shared__ DmStageRow S;
  if (STAGED && r < rows) {
    const int qt = g.pair_of[r];
    const int q = qt / g.n, t = qt - (qt / g.n) * g.n;
    for (int X = threadIdx.x; X < g.nholeA; X += blockDim.x) {
      const int ea = g.liftA[q * g.nholeA + X];
      S.a[X] = ea;
      if (ea >= 0) {
        const int A = ea >> 1;
        S.off[X] = g.off[A];
        S.lim[X] = g.nballow[g.alevel[A]];
      }
    }
    for (int Y = threadIdx.x; Y < g.nholeB; Y += blockDim.x) S.b[Y] = g.liftB[t * g.nholeB + Y];
  }
  __syncthreads();
  double v[kDmRowRegs];
  int m = 0;
#pragma unroll
  for (int i = 0; i < kDmRowRegs; ++i) {
    const int k = threadIdx.x + i * blockDim.x;
    v[i] = (r < rows && k < ncol) ? dm_row_value<STAGED>(g, S, col_start + k, r, c) : 0.0;
    m = max(m, oz_exp_field(v[i]));
  }
  for (int k = threadIdx.x + kDmRowRegs * blockDim.x; k < ncol; k += blockDim.x)
    if (r < rows) m = max(m, oz_exp_field(dm_row_value<STAGED>(g, S, col_start + k, r, c)));
  m = __reduce_max_sync(0xffffffffu, m);
  __shared__ int sm[8];
  __shared__ int ex_s;
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    int x = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) x = max(x, sm[i]);
    ex_s = x > 0 ? x - 1022 : 0;
    if (r < rows) e[r] = ex_s;
  }
  __syncthreads();
  const int ex = ex_s;
  __nv_bfloat16* row = out + (long long)r * ld;
  int a[OZ_S];
#pragma unroll
  for (int i = 0; i < kDmRowRegs; ++i) {
    const int k = threadIdx.x + i * blockDim.x;
    if (k < ld) {
      oz_digits(v[i], ex, a);
      oz_store_digits(a, row + k, total);
    }
  }
  for (int k = threadIdx.x + kDmRowRegs * blockDim.x; k < ld; k += blockDim.x) {
    const double x = (r < rows && k < ncol) ? dm_row_value<STAGED>(g, S, col_start + k, r, c) : 0.0;
    oz_digits(x, ex, a);
    oz_store_digits(a, row + k, total);
  }
}

// Residues of all rows of L of all blocks, one thread block per row (and vector, blockIdx.z): 8
// consecutive columns per thread (row entries staged as in k_dm_lift_slice).  A row's unit
// is 2^-scale with scale = bits - e, max |L[row][:]| < 2^e: small rows keep their
// bits however large others are.  Rows a part does not reach and padding are zero from the
// buffer's first clearing on.  Rows of few columns take their maximum and their residues in one
// launch (MODE 0: a thread's first chunk stays in shared memory in between, later ones are gathered
// twice); longer ones are split over blockIdx.y, MODE 1 leaving partial maxima for MODE 2.
// 26 bytes written per element; latency of the gathers and the row staging bound it.  (One unit per
// vector, from its 2-norm, in a launch per vector, block and column class: one density of 2 + 2 electrons in 60 orbitals 975
// us, now 998, in 8 orbitals 70, now 49; 3 + 3 in 20, whose rows are split, 460, now 544.)
struct DmCutBlock {
  DmGather g;
  int row0, R, bits, nparts, nkb;
  int col_start[OZ_MAX_SEGS], ncol[OZ_MAX_SEGS], kb0[OZ_MAX_SEGS], rows[OZ_MAX_SEGS];
  long long base, mod_stride;
};
struct DmCut {
  DmCutBlock blk[3];
  const double* v[2];
  __nv_bfloat16* out[2];
  int* scale;   // [vector][row]
  int* pmax;    // [vector][row][gridDim.y]
  int rows;
};
template <bool STAGED, int MODE>
__global__ void __launch_bounds__(256, 4) k_dm_cut(const __grid_constant__ DmCut D,
                                                                const __grid_constant__ CrtMods M) {
  const int grow = blockIdx.x, vec = blockIdx.z;
  const int b = (D.blk[2].R > 0 && grow >= D.blk[2].row0) ? 2 : (D.blk[1].R > 0 && grow >= D.blk[1].row0) ? 1 : 0;
  const DmCutBlock& K = D.blk[b];
  const DmGather& g = K.g;
  const int r = grow - K.row0;
  const double* __restrict__ c = D.v[vec];
  const bool staged = STAGED && b == 0;
  __shared__ DmStageRow S;
  if (staged) {
    const int qt = g.pair_of[r];
    const int q = qt / g.n, t = qt - (qt / g.n) * g.n;
    for (int X = threadIdx.x; X < g.nholeA; X += blockDim.x) {
      const int ea = g.liftA[q * g.nholeA + X];
      S.a[X] = ea;
      if (ea >= 0) {
        const int A = ea >> 1;
        S.off[X] = g.off[A];
        S.lim[X] = g.nballow[g.alevel[A]];
      }
    }
    for (int Y = threadIdx.x; Y < g.nholeB; Y += blockDim.x) S.b[Y] = g.liftB[t * g.nholeB + Y];
    __syncthreads();
  }
  const int kc0 = blockIdx.y * 256 + threadIdx.x, step = 256 * gridDim.y, nch = 8 * K.nkb;
  __shared__ int sm[8];
  __shared__ double keep[MODE == 0 ? 8 : 1][256];  // a thread's first chunk
  int m = 0, sc = 0;
  if (MODE == 2)
    for (int i = 0; i < (int)gridDim.y; ++i) m = max(m, D.pmax[((long long)vec * D.rows + grow) * gridDim.y + i]);
  __nv_bfloat16* row = D.out[vec] + K.base + (long long)(r >> 7) * K.nkb * (CRT_BM * CRT_BK) + (r & 127) * CRT_BK;
#pragma unroll 1
  for (int pass = MODE == 2 ? 1 : 0; pass < (MODE == 1 ? 1 : 2); ++pass) {
    if (pass == 1) {
      sc = m == 0x7FF ? kDmNotFinite : m > 0 ? K.bits - (m - 1022) : 0;
      if (threadIdx.x == 0 && blockIdx.y == 0) D.scale[(long long)vec * D.rows + grow] = sc;
    }
#pragma unroll 1
    for (int kc = kc0; kc < nch; kc += step) {
      double v[8];
      int p = 0;
      while (p + 1 < K.nparts && (kc >> 3) >= K.kb0[p + 1]) ++p;
      if (r >= K.rows[p]) continue;  // the chunk's part does not reach the row
      if (MODE == 0 && pass == 1 && kc == kc0) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = keep[j][threadIdx.x];
      } else {
        const int k0 = kc * 8 - K.kb0[p] * CRT_BK, left = K.ncol[p] - k0, col = K.col_start[p] + k0;
        if (staged) {
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = j < left ? dm_row_value<true>(g, S, col + j, r, c) : 0.0;
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = j < left ? dm_value(g, col + j, r, c) : 0.0;
        }
      }
      if (pass == 0) {
#pragma unroll
        for (int j = 0; j < 8; ++j) m = max(m, oz_exp_field(v[j]));
        if (MODE == 0 && kc == kc0)
#pragma unroll
          for (int j = 0; j < 8; ++j) keep[j][threadIdx.x] = v[j];
      } else {
        CrtLimbs2<4> x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = crt_limbs2<4>(crt_fixed(v[2 * j], 0, sc), crt_fixed(v[2 * j + 1], 0, sc));
        crt_store8<4>(x, M, row + (long long)(kc >> 3) * (CRT_BM * CRT_BK) + (kc & 7) * 8, K.mod_stride);
      }
    }
    if (pass == 0) {
      m = __reduce_max_sync(0xffffffffu, m);
      if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
      __syncthreads();
      for (int w = 0; w < 8; ++w) m = max(m, sm[w]);
      if (MODE == 1 && threadIdx.x == 0) D.pmax[((long long)vec * D.rows + grow) * gridDim.y + blockIdx.y] = m;
    }
  }
}

// Q (R x R) from the residues of L_bra L_ket^T: a warp 32 rows x 8 columns, its rows' runs turned
// across lane octets; ket = bra: only the tiles on and above the diagonal exist, their mirror
// images are written with them (32 rows of a column at once).  All moduli's loads in flight, one
// launch for the three blocks (four in flight and a launch per block: 160 us at n = 60, now 96;
// the slices' kernel rebuilt in its epilogue and mirrored in 46).
struct DmRebuild {
  const int16_t* res[3];
  double* q[3];
  int R[3], tn[3], tile0[4];  // of the blocks ab, aa, bb; tile0: first tile of each in the grid
  int row0[3];                // first of each in the lists of rows' scales
};
template <int NM>
__global__ void __launch_bounds__(256) k_dm_rebuild(const __grid_constant__ DmRebuild D, int sym,
                                                    const int* __restrict__ scale_bra, const int* __restrict__ scale_ket,
                                                    const __grid_constant__ CrtWeights W) {
  const int blk = ((int)blockIdx.x >= D.tile0[1] ? 1 : 0) + ((int)blockIdx.x >= D.tile0[2] ? 1 : 0);
  const int tl = blockIdx.x - D.tile0[blk], R = D.R[blk], tn = D.tn[blk];
  double* __restrict__ q = D.q[blk];
  const int rt = tl / tn, nt = tl - rt * tn;
  if (sym && (rt >> 1) > nt) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int tile = CRT_BM * CRT_MAXN;
  const int16_t* base = D.res[blk] + ((long long)rt * tn + nt) * NM * tile;
  const int *sb = scale_bra + D.row0[blk], *sk = scale_ket + D.row0[blk];
  for (int w = warp; w < 32; w += 8) {
    const int cg = blockIdx.y * 8 + (w >> 2), quarter = w & 3;
    const int r0 = rt * CRT_BM + quarter * 32, col = nt * CRT_MAXN + cg * 8;
    if (r0 >= R || col >= R) continue;
    unsigned long long lo[8];
    uint32_t hi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      lo[j] = W.start_lo;
      hi[j] = W.start_hi;
    }
    const int16_t* src = base + (cg * CRT_BM + quarter * 32 + lane) * 8;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(src + (long long)i * tile));
      const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
      const uint32_t w0 = W.lo0[i], w1 = W.lo1[i], w2 = W.hi[i];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t t = (uint32_t)((int)(int16_t)(xw[j >> 1] >> (16 * (j & 1))) + W.off[i]);
        lo[j] += (unsigned long long)t * w0;
        lo[j] += (unsigned long long)(t * w1) << 32;
        hi[j] += t * w2;
      }
    }
    double v[8];
    const int er = sb[min(r0 + lane, R - 1)];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int ec = sk[min(col + j, R - 1)], e = -(er + ec);
      // crt_value gives 0 below the normal range: rounded there by a product
      if (min(er, ec) == kDmNotFinite) v[j] = __longlong_as_double(0x7FF8000000000000ll);
      else if (e < -900) v[j] = crt_value(lo[j], hi[j], W.mman, W.mexp, e + 600) * 0x1p-600;
      else v[j] = crt_value(lo[j], hi[j], W.mman, W.mexp, e);
    }
    if (sym && (rt >> 1) < nt && r0 + lane < R)
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (col + j < R) q[(long long)(col + j) * R + r0 + lane] = v[j];
    oz_lane_transpose<8>(v, lane);
    const int rr = r0 + (lane & ~7), cc = col + (lane & 7);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (cc < R && rr + k < R) q[(long long)(rr + k) * R + cc] = v[k];
  }
}

// ---------------------------------------------------------------------------
// device: expansion to the n^4 tensors, one-body matrices

struct DmResult {
  const double* q;   // R x R, row-major
  int R, nreg;
  int bnd[kDmMaxBnd];
};

// whether entry (x, y) of a ket = bra result is computed by the contraction:
// regions i < j, or the same region right of the 128-row block's first row
__device__ __forceinline__ bool dm_computed(const DmResult& Q, int x, int y) {
  int i = 0, j = 0;
  while (i + 1 < Q.nreg && x >= Q.bnd[i + 1]) ++i;
  while (j + 1 < Q.nreg && y >= Q.bnd[j + 1]) ++j;
  return i < j || (i == j && y >= Q.bnd[i] + ((x - Q.bnd[i]) / OZ_BM) * OZ_BM);
}

// ket = bra: every entry that was not computed is copied from its transpose,
// 32 x 32 tiles through shared memory (reads and writes coalesced).  Tiles
// wholly above the diagonal are all computed (x < y lies in the computed part).
__global__ void __launch_bounds__(256) k_dm_mirror(DmResult Q, double* __restrict__ q) {
  __shared__ double tile[32][33];
  const int x0 = blockIdx.y * 32, y0 = blockIdx.x * 32;  // destination rows x, columns y
  if (x0 + 31 < y0) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8) {  // source rows y0 + i, columns x0 + tx
    const int ys = y0 + i, xs = x0 + tx;
    tile[i][tx] = (ys < Q.R && xs < Q.R) ? q[(long long)ys * Q.R + xs] : 0.0;
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {  // destination row x0 + i, column y0 + tx
    const int x = x0 + i, y = y0 + tx;
    if (x < Q.R && y < Q.R && !dm_computed(Q, x, y)) q[(long long)x * Q.R + y] = tile[tx][i];
  }
}

struct DmExpand {
  int n, na, nb;
  DmResult blk[3];        // in d2's block order: aa, ab, bb
  const int* pair_index;  // ab: (p, r) -> row
  const int* pp_row[2];   // aa / bb: {u < v} -> row
};

// One block per (p, r) and d2 block b writes d2[b][p][q][r][t] for all (q, t): b = 1 (ab)
// Q[(p,r)][(q,t)], b = 0 (aa) or 2 (bb) s(p,r) s(q,t) Q[{p,r}][{q,t}].  A block reads one row
// of Q, which stays in L1 however the pairs {q,t} jump about in it (blocks over (p, q) read columns
// t < q of it one sector per element); a warp takes a q, lanes run over t, eight q
// in flight.  Bound by the 3 n^4 stores; n = 60: 157 us by (p, q), 101 now.
__global__ void __launch_bounds__(256) k_dm_expand(DmExpand E, double* __restrict__ d2) {
  const int n = E.n, p = blockIdx.x / n, r = blockIdx.x - (blockIdx.x / n) * n, b = blockIdx.y;
  const long long n2 = (long long)n * n;
  const bool ab = b == 1 && E.na > 0 && E.nb > 0;
  const bool ss = b != 1 && (b == 0 ? E.na : E.nb) >= 2;
  const DmResult& Q = E.blk[b];
  const int* __restrict__ rows = ab ? E.pair_index : ss ? E.pp_row[b == 0 ? 0 : 1] : nullptr;
  int x = -1;
  if (ab) x = rows[p * n + r];
  else if (ss && p != r) x = rows[min(p, r) * n + max(p, r)];
  const double* __restrict__ row = x >= 0 && x < Q.R ? Q.q + (long long)x * Q.R : nullptr;
  double* __restrict__ out = d2 + (((long long)b * n + p) * n2 + r) * n;  // + q n^2 + t
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sx = p < r ? 1 : 0;
  for (int q0 = warp; q0 < n; q0 += 64)
    for (int t = lane; t < n; t += 32) {
      int y[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int q = q0 + 8 * j;
        const bool on = row && q < n && (ab || q != t);
        y[j] = on ? __ldg(rows + (ab ? q * n + t : min(q, t) * n + max(q, t))) : -1;
      }
      long long v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = y[j] >= 0 && y[j] < Q.R ? __double_as_longlong(__ldg(row + y[j])) : 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int q = q0 + 8 * j;
        if (q >= n) continue;
        const int sg = ss ? sx ^ (q < t ? 1 : 0) : 0;
        const long long w = v[j] == 0 ? 0 : v[j] ^ ((long long)sg << 63);
        __stcs(out + q * n2 + t, __longlong_as_double(w));
      }
    }
}

// d1_s[p][q] = sum_r d2_ss[p,q,r,r] / (N_s - 1) of a spin with N_s >= 2, a warp per (p, q)
__global__ void __launch_bounds__(256) k_dm_trace(DmExpand E, double* __restrict__ d1) {
  const int spin = blockIdx.y;
  if ((spin == 0 ? E.na : E.nb) < 2) return;
  const int n = E.n, lane = threadIdx.x & 31;
  const int pq = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (pq >= n * n) return;
  const int p = pq / n, q = pq - p * n;
  const DmResult& Q = E.blk[2 * spin];
  const int* __restrict__ rows = E.pp_row[spin];
  double s = 0.0;
  for (int r = lane; r < n; r += 32) {
    if (r == p || r == q) continue;
    const int x = rows[min(p, r) * n + max(p, r)], y = rows[min(q, r) * n + max(q, r)];
    if (x < 0 || y < 0 || x >= Q.R || y >= Q.R) continue;
    const double v = Q.q[(long long)x * Q.R + y];
    s += (p < r) == (q < r) ? v : -v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) d1[(long long)spin * n * n + pq] = s / (double)((spin == 0 ? E.na : E.nb) - 1);
}

// d1_s[p][q] = sum_X s(p,X) s(q,X) sum_O bra[X u p, O] ket[X u q, O] over the
// one-hole strings X of spin s (the lift tables), one block per (p, q)
__global__ void __launch_bounds__(256) k_dm_gamma_direct(int n, int spin, int nhole, const int* __restrict__ lift,
                                                         int na_count, const int8_t* __restrict__ alevel,
                                                         const int* __restrict__ nballow,
                                                         const long long* __restrict__ off,
                                                         const double* __restrict__ bra,
                                                         const double* __restrict__ ket, double* __restrict__ d1) {
  const int p = blockIdx.x / n, q = blockIdx.x % n;
  double acc = 0.0;
  for (int X = 0; X < nhole; ++X) {
    int e1 = lift[p * nhole + X], e2 = lift[q * nhole + X];
    if (e1 < 0 || e2 < 0) continue;
    const double sg = ((e1 ^ e2) & 1) ? -1.0 : 1.0;
    const int s1 = e1 >> 1, s2 = e2 >> 1;
    double part = 0.0;
    if (spin == 0) {
      const int m = min(nballow[alevel[s1]], nballow[alevel[s2]]);
      const double* x = bra + off[s1];
      const double* y = ket + off[s2];
      for (int B = threadIdx.x; B < m; B += blockDim.x) part += x[B] * y[B];
    } else {
      for (int A = threadIdx.x; A < na_count; A += blockDim.x) {
        const int nbA = nballow[alevel[A]];
        if (s1 < nbA && s2 < nbA) part += bra[off[A] + s1] * ket[off[A] + s2];
      }
    }
    acc += sg * part;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ double sm[8];
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sm[i];
    d1[spin * n * n + blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------------------
// host: operands, work lists, launches

static DmGather gather_of(const Context& ctx, const DensityPlan& P, int b) {
  DmGather g;
  std::memset(&g, 0, sizeof(g));
  g.kind = b;
  g.n = ctx.n;
  g.nholeA = ctx.sp[0].nhole;
  g.nholeB = ctx.sp[1].nhole;
  g.pair_of = ctx.pair_of.as<int>();
  g.hp_inv = ctx.hp_inv.as<int>();
  g.liftA = ctx.sp[0].lift.as<int>();
  g.liftB = ctx.sp[1].lift.as<int>();
  if (b > 0) {
    g.lift2 = P.lift2[b - 1].as<int>();
    g.cols = P.cols[b - 1].as<int>();
    g.nz = P.nz[b - 1];
  }
  g.alevel = ctx.sp[0].level.as<int8_t>();
  g.nballow = ctx.nballow.as<int>();
  g.off = ctx.off.as<long long>();
  const int d = std::max(1, g.nholeB);
  int l = 0;
  while ((1ll << l) < d) ++l;
  g.div_shift = 31 + l;
  g.div_mul = (unsigned)(((1ull << (31 + l)) + d - 1) / d);
  return g;
}

// slices and row exponents of every part of every block for one vector
static int cut_operands(Context& ctx, const double* v, __nv_bfloat16* sl, int* ex, cudaStream_t st) {
  DensityPlan& P = *ctx.dm;
  for (int b = 0; b < 3; ++b) {
    const DmBlock& B = P.blk[b];
    if (B.parts.empty()) continue;
    DmGather g = gather_of(ctx, P, b);
    for (size_t i = 0; i < B.parts.size(); ++i) {
      const DmPart& pt = B.parts[i];
      int* e = ex + B.exp_off + i * B.R128;
      if (b == 0 && g.nholeA <= kDmStage && g.nholeB <= kDmStage)
        k_dm_lift_slice<true><<<pt.rows_pad, 256, 0, st>>>(g, pt.col_start, pt.ncol, pt.rows, pt.ld, pt.rows_pad, v,
                                                           e, sl + pt.sl_off);
      else
        k_dm_lift_slice<false><<<pt.rows_pad, 256, 0, st>>>(g, pt.col_start, pt.ncol, pt.rows, pt.ld, pt.rows_pad,
                                                            v, e, sl + pt.sl_off);
      ISCSI_COUNT_LAUNCH();
    }
  }
  ISCSI_CUDA(cudaGetLastError());
  return kOk;
}

// one problem (rows [r0, r1) x columns [c0, c1) of block B's result) with the
// parts that reach both ranges
static int add_problem(DensityPlan& P, OzJob& job, const DmBlock& B, int r0, int r1, int c0, int c1, bool sym,
                       int reg_rows_end, int reg_cols_end, double* flops) {
  OzProblem pr;
  std::memset(&pr, 0, sizeof(pr));
  pr.t = reinterpret_cast<long long>(P.q.as<double>() + B.q_off + (size_t)r0 * B.R + c0);
  pr.t_rel = 0;
  pr.ldt = B.R;
  pr.M = r1 - r0;
  pr.N = c1 - c0;
  pr.seg_begin = (int)job.segs.size();
  pr.accumulate = 0;
  const __nv_bfloat16* abase = P.sl_bra.as<__nv_bfloat16>();
  const __nv_bfloat16* bbase = sym ? abase : P.sl_ket.as<__nv_bfloat16>();
  const int* aex = P.ex_bra.as<int>();
  const int* bex = sym ? aex : P.ex_ket.as<int>();
  for (size_t i = 0; i < B.parts.size(); ++i) {
    const DmPart& pt = B.parts[i];
    if (pt.rows < reg_rows_end || pt.rows < reg_cols_end) continue;
    SliceArray a{abase + pt.sl_off, pt.ld, pt.rows_pad, (long long)pt.rows_pad * pt.ld};
    SliceArray b{bbase + pt.sl_off, pt.ld, pt.rows_pad, (long long)pt.rows_pad * pt.ld};
    ISCSI_TRY(oz_job_add_seg(job, a, r0, aex + B.exp_off + i * B.R128 + r0, b, c0, bex + B.exp_off + i * B.R128 + c0,
                             pt.ld, pr.N));
    flops[0] += 28.0 * 2.0 * pr.M * (double)pr.N * pt.ld;
    flops[1] += 2.0 * pr.M * (double)pr.N * pt.ncol;
  }
  pr.seg_count = (int)job.segs.size() - pr.seg_begin;
  if (pr.seg_count > 0) job.probs.push_back(pr);
  return kOk;
}

static int build_job(Context& ctx, bool sym) {
  DensityPlan& P = *ctx.dm;
  OzJob& job = sym ? P.job_sym : P.job_gen;
  job.probs.clear();
  job.segs.clear();
  job.maps.clear();
  job.sh.clear();
  double f[2] = {0.0, 0.0};
  for (int b = 0; b < 3; ++b) {
    const DmBlock& B = P.blk[b];
    if (B.parts.empty()) continue;
    const int nreg = (int)B.bnd.size() - 1;
    for (int i = 0; i < nreg; ++i)
      for (int j = sym ? i : 0; j < nreg; ++j) {
        const int r0 = B.bnd[i], r1 = B.bnd[i + 1], c0 = B.bnd[j], c1 = B.bnd[j + 1];
        if (sym && i == j) {
          // diagonal region: per 128-row block, the columns from the block's first row on
          for (int rb = r0; rb < r1; rb += OZ_BM)
            ISCSI_TRY(add_problem(P, job, B, rb, std::min(rb + OZ_BM, r1), rb, c1, true, r1, c1, f));
        } else {
          ISCSI_TRY(add_problem(P, job, B, r0, r1, c0, c1, sym, r1, c1, f));
        }
      }
  }
  P.bf16_flops[sym ? 0 : 1] = f[0];
  P.fp64_flops[sym ? 0 : 1] = f[1];
  ISCSI_TRY(oz_job_upload(job, stream()));
  (sym ? P.sym_ready : P.gen_ready) = true;
  return kOk;
}

// residue operands, products and schedule (sym: ket = bra); kErrNoMem: they do not fit
static int residues_build(Context& ctx, bool sym) {
  DensityPlan& P = *ctx.dm;
  const int idx = sym ? 0 : 1;
  if (P.res_ready[idx]) return kOk;
  cudaStream_t st = stream();
  size_t elems = 0, out = 0;
  const int nm = P.nmods;
  for (int b = 0; b < 3; ++b) {
    DmBlock& B = P.blk[b];
    if (B.parts.empty()) continue;
    B.res_off = elems;
    elems += (size_t)nm * B.R256 * B.nkb * CRT_BK;
    P.res_out_off[b] = out;
    out += (size_t)nm * B.R256 * B.R256;
    // sums of chunk residues stay exact below 2^24 / 257 chunks; tensor map rows are 32-bit
    if (B.nkb > CRT_CHUNK * 60000 || (long long)nm * B.R256 * B.nkb >= (1ll << 31)) return kErrNoMem;
  }
  DevBuf* ops[2] = {&P.res_bra, sym ? nullptr : &P.res_ket};
  for (DevBuf* d : ops)
    if (d && d->bytes < sizeof(__nv_bfloat16) * elems) {
      ISCSI_TRY(crt_alloc(*d, sizeof(__nv_bfloat16) * elems, P.res_held));
      ISCSI_CUDA(cudaMemsetAsync(d->p, 0, d->bytes, st));
    }
  if (P.res_out.bytes < sizeof(int16_t) * out) ISCSI_TRY(crt_alloc(P.res_out, sizeof(int16_t) * out, P.res_held));
  if (!P.scale.p) {
    ISCSI_TRY(P.scale.alloc(sizeof(int) * (size_t)std::max(1, P.res_rows) * 2 * (1 + kDmMaxSplit)));
  }
  CrtJob& job = P.res_job[idx];
  job.probs.clear();
  double f64 = 0.0;
  for (int b = 0; b < 3; ++b) {
    const DmBlock& B = P.blk[b];
    if (B.parts.empty()) continue;
    CrtHostProblem H;
    std::memset(&H.p, 0, sizeof(H.p));
    H.p.ntile = CRT_MAXN;
    H.p.tn = B.R256 / CRT_MAXN;
    H.p.nm = nm;
    H.p.rt = rup(B.R, CRT_BM) / CRT_BM;
    H.p.nblk_a = H.p.nblk_b = B.R256 / CRT_BM;
    H.p.nkb_a = H.p.nkb_b = B.nkb;
    H.p.res = P.res_out.as<int16_t>() + P.res_out_off[b];
    H.mt = B.R256 / (2 * CRT_BM);
    std::vector<DmPart> parts = B.parts;
    H.range = [parts, sym](int mt, int nt, int& k0, int& k1) {
      if (sym && mt > nt) return false;
      // the classes that reach both row ranges: a prefix
      k0 = k1 = 0;
      for (const DmPart& pt : parts)
        if (pt.rows > std::max(mt, nt) * 2 * CRT_BM) k1 = pt.kb0 + pt.nkb;
      return true;
    };
    const __nv_bfloat16* a = P.res_bra.as<__nv_bfloat16>() + B.res_off;
    ISCSI_TRY(crt_encode(H.p, a, sym ? a : P.res_ket.as<__nv_bfloat16>() + B.res_off, nm));
    job.probs.push_back(H);
    for (const DmPart& pt : B.parts) f64 += 2.0 * pt.ncol * pt.rows * (sym ? 0.5 * (pt.rows + 1.0) : (double)pt.rows);
  }
  ISCSI_TRY(job.upload(st));
  P.bf16_flops[idx] = job.flops;
  P.fp64_flops[idx] = f64;
  P.res_ready[idx] = true;
  return kOk;
}

// residues of bra and ket (null: bra only)
static int residues_cut(Context& ctx, const double* bra, const double* ket, cudaStream_t st) {
  DensityPlan& P = *ctx.dm;
  const CrtMods mods = crt_make_mods(P.nmods);
  DmCut D;
  std::memset(&D, 0, sizeof(D));
  int nkb = 0;
  for (int b = 0; b < 3; ++b) {
    const DmBlock& B = P.blk[b];
    DmCutBlock& K = D.blk[b];
    K.row0 = B.row0;
    if (B.parts.empty()) continue;
    K.g = gather_of(ctx, P, b);
    K.R = B.R;
    K.bits = B.bits;
    K.nkb = B.nkb;
    K.base = (long long)B.res_off;
    K.mod_stride = (long long)B.R256 * B.nkb * CRT_BK;
    for (const DmPart& pt : B.parts) {
      const int i = K.nparts++;
      K.col_start[i] = pt.col_start;
      K.ncol[i] = pt.ncol;
      K.kb0[i] = pt.kb0;
      K.rows[i] = pt.rows;
    }
    nkb = std::max(nkb, B.nkb);
  }
  if (P.res_rows == 0) return kOk;
  D.v[0] = bra;
  D.v[1] = ket;
  D.out[0] = P.res_bra.as<__nv_bfloat16>();
  D.out[1] = P.res_ket.as<__nv_bfloat16>();
  D.rows = P.res_rows;
  D.scale = P.scale.as<int>();
  D.pmax = D.scale + 2ll * P.res_rows;
  // at least two chunks of eight columns for each of a block's threads
  const dim3 grid(P.res_rows, std::max(1, std::min(kDmMaxSplit, nkb / 64)), ket ? 2 : 1);
  const bool staged = ctx.sp[0].nhole <= kDmStage && ctx.sp[1].nhole <= kDmStage && !P.blk[0].parts.empty();
  auto launch = [&](auto mode) {
    constexpr int MODE = decltype(mode)::value;
    if (staged)
      k_dm_cut<true, MODE><<<grid, 256, 0, st>>>(D, mods);
    else
      k_dm_cut<false, MODE><<<grid, 256, 0, st>>>(D, mods);
    ISCSI_COUNT_LAUNCH();
  };
  if (grid.y == 1) {
    launch(std::integral_constant<int, 0>());
  } else {
    launch(std::integral_constant<int, 1>());
    launch(std::integral_constant<int, 2>());
  }
  ISCSI_CUDA(cudaGetLastError());
  return kOk;
}

template <int NM>
static void launch_rebuild(const DmRebuild& D, int sym, const int* sb, const int* sk, cudaStream_t st) {
  static const CrtWeights weights = crt_make_weights(NM, 1);
  k_dm_rebuild<NM><<<dim3(D.tile0[3], CRT_MAXN / 64), 256, 0, st>>>(D, sym, sb, sk, weights);
  ISCSI_COUNT_LAUNCH();
}

int density_run(Context& ctx, const double* bra, const double* ket, double* d1, double* d2) {
  cudaStream_t st = stream();
  const bool sym = (ket == nullptr || ket == bra);
  if (!ket) ket = bra;
  const int n = ctx.n;
  DensityPlan* Pp = nullptr;
  DmExpand E;
  std::memset(&E, 0, sizeof(E));
  E.n = n;
  E.na = ctx.na;
  E.nb = ctx.nb;
  E.pair_index = ctx.pair_index.as<int>();
  if (d2) {
    ISCSI_TRY(plan_build(ctx));
    Pp = ctx.dm;
    DensityPlan& P = *Pp;
    bool res = !P.no_room[sym ? 0 : 1];
    if (res) {
      const int rc = residues_build(ctx, sym);
      if (rc == kErrNoMem) {
        cudaGetLastError();
        density_drop(ctx);
        P.no_room[1] = true;  // a ket of its own takes more
        P.no_room[0] = P.no_room[0] || sym;
        res = false;
      } else {
        ISCSI_TRY(rc);
      }
    }
    const bool ev = !ctx.capturing;
    if (res) {
      ISCSI_TRY(residues_cut(ctx, bra, sym ? nullptr : ket, st));
      const CrtJob& job = P.res_job[sym ? 0 : 1];
      if (job.grid > 0) {
        ISCSI_TRY(tc_err_buf(ctx));
        if (ev) ISCSI_CUDA(cudaEventRecord(P.ev[0], st));
        ISCSI_TRY(job.launch(ctx.oz_err.as<int>(), st));
        if (ev) ISCSI_CUDA(cudaEventRecord(P.ev[1], st));
        P.timed = ev;
      }
      DmRebuild D;
      D.tile0[0] = 0;
      for (int b = 0; b < 3; ++b) {
        const DmBlock& B = P.blk[b];
        const bool some = !B.parts.empty();
        D.res[b] = P.res_out.as<int16_t>() + P.res_out_off[b];
        D.q[b] = P.q.as<double>() + B.q_off;
        D.R[b] = some ? B.R : 0;
        D.row0[b] = B.row0;
        D.tn[b] = some ? B.R256 / CRT_MAXN : 1;
        D.tile0[b + 1] = D.tile0[b] + (some ? (rup(B.R, CRT_BM) / CRT_BM) * D.tn[b] : 0);
      }
      if (D.tile0[3] > 0) {
        const int *sb = P.scale.as<int>(), *sk = sb + (sym ? 0 : P.res_rows);
        switch (P.nmods) {
          case 13: launch_rebuild<13>(D, sym, sb, sk, st); break;
          case 14: launch_rebuild<14>(D, sym, sb, sk, st); break;
          case 15: launch_rebuild<15>(D, sym, sb, sk, st); break;
          default: launch_rebuild<16>(D, sym, sb, sk, st); break;
        }
      }
      ISCSI_CUDA(cudaGetLastError());
    } else {
      ISCSI_TRY(slices_alloc(P));
      if (!sym && !P.sl_ket.p && P.sl_elems) {
        ISCSI_TRY(P.sl_ket.alloc(sizeof(__nv_bfloat16) * P.sl_elems));
        ISCSI_TRY(P.ex_ket.alloc(sizeof(int) * P.ex_elems));
        ISCSI_CUDA(cudaMemsetAsync(P.ex_ket.p, 0, sizeof(int) * P.ex_elems, st));
      }
      if (sym ? !P.sym_ready : !P.gen_ready) ISCSI_TRY(build_job(ctx, sym));
      ISCSI_TRY(cut_operands(ctx, bra, P.sl_bra.as<__nv_bfloat16>(), P.ex_bra.as<int>(), st));
      if (!sym) ISCSI_TRY(cut_operands(ctx, ket, P.sl_ket.as<__nv_bfloat16>(), P.ex_ket.as<int>(), st));
      const OzJob& job = sym ? P.job_sym : P.job_gen;
      if (job.tiles > 0) {
        if (ev) ISCSI_CUDA(cudaEventRecord(P.ev[0], st));
        ISCSI_TRY(oz_job_launch(ctx, job, st));
        if (ev) ISCSI_CUDA(cudaEventRecord(P.ev[1], st));
        P.timed = ev;
      }
    }
    // expansion: slot 0 = aa, 1 = ab, 2 = bb (d2's block order)
    const int slot_of_plan[3] = {1, 0, 2};
    for (int b = 0; b < 3; ++b) {
      const DmBlock& B = P.blk[b];
      DmResult& R = E.blk[slot_of_plan[b]];
      R.q = P.q.as<double>() + B.q_off;
      R.R = B.parts.empty() ? 0 : B.R;
      R.nreg = B.parts.empty() ? 0 : (int)B.bnd.size() - 1;
      for (int i = 0; i < (int)B.bnd.size() && i < kDmMaxBnd; ++i) R.bnd[i] = B.bnd[i];
    }
    E.pp_row[0] = P.pp_row[0].as<int>();
    E.pp_row[1] = P.pp_row[1].as<int>();
    if (sym && !res)
      for (int b = 0; b < 3; ++b) {
        const DmResult& R = E.blk[b];
        if (R.R == 0) continue;
        dim3 grid((R.R + 31) / 32, (R.R + 31) / 32);
        k_dm_mirror<<<grid, 256, 0, st>>>(R, const_cast<double*>(R.q)); ISCSI_COUNT_LAUNCH();
      }
    k_dm_expand<<<dim3(n * n, 3), 256, 0, st>>>(E, d2); ISCSI_COUNT_LAUNCH();
    if (d1 && (ctx.na >= 2 || ctx.nb >= 2)) {
      k_dm_trace<<<dim3((n * n + 7) / 8, 2), 256, 0, st>>>(E, d1); ISCSI_COUNT_LAUNCH();
    }
    ISCSI_CUDA(cudaGetLastError());
  }
  if (d1) {
    for (int s = 0; s < 2; ++s) {
      const int ne = s == 0 ? ctx.na : ctx.nb;
      if (d2 && ne >= 2) {
        // k_dm_trace above
      } else if (ne == 0) {
        ISCSI_CUDA(cudaMemsetAsync(d1 + (size_t)s * n * n, 0, sizeof(double) * n * n, st));
      } else {
        k_dm_gamma_direct<<<n * n, 256, 0, st>>>(n, s, ctx.sp[s].nhole, ctx.sp[s].lift.as<int>(), ctx.sp[0].count,
                                                 ctx.sp[0].level.as<int8_t>(), ctx.nballow.as<int>(),
                                                 ctx.off.as<long long>(), bra, ket, d1); ISCSI_COUNT_LAUNCH();
      }
    }
    ISCSI_CUDA(cudaGetLastError());
  }
  return kOk;
}

double density_gemm_ms(Context& ctx) {
  if (!ctx.dm || !ctx.dm->timed) return 0.0;
  if (cudaEventSynchronize(ctx.dm->ev[1]) != cudaSuccess) return 0.0;
  float ms = 0.0f;
  if (cudaEventElapsedTime(&ms, ctx.dm->ev[0], ctx.dm->ev[1]) != cudaSuccess) return 0.0;
  return ms;
}

double density_flops(const Context& ctx, int sym, int which) {
  if (!ctx.dm) return 0.0;
  return which == 0 ? ctx.dm->bf16_flops[sym ? 0 : 1] : ctx.dm->fp64_flops[sym ? 0 : 1];
}

}  // namespace iscsi
