// crt.cu -- the FP64 sigma step's contractions through residue numbers
// (crt.cuh): operands, work list, schedule and reconstruction.
//
//   k_crt_cmax      largest exponent of each CI vector
//   k_crt_operands  residues of the lifted vector Ct^T (one row (X, Y, v) per
//                   column of T) and of C and C^T (the same-spin operands)
//   k_crt_gemm      every product's residues, one persistent launch
//   k_crt_fold      sigma: the residues of every T element of a determinant and
//                   of its same-spin part are added, then turned into FP64 once
//
// One scale per side: all units (G, M_alpha, M_beta) are integers of 2^-sh, a
// vector's coefficients integers of 2^(e - bc) with |c| < 2^e, so that products
// of different rows, columns and parts add up as residues and a determinant
// costs one reconstruction instead of one per T element (4 of them for 2 + 2
// electrons, 16 for 4 + 4).  |sigma| is bounded by the units' row 1-norms, taken
// at set-up, times 2^bc; the moduli are the fewest whose product holds that
// bound with the largest coefficient at kCrtCBits bits and the largest unit at kCrtUnitBits.
//
// kCrtCBits: every coefficient is rounded to 2^-58 of the vector's largest one, so a sigma
// element that only small coefficients reach is known to 2^-58 max |c| sum_J |H_IJ| and no
// better.  The slices have an exponent per column (49 bits).  Largest error of an element
// over its sum |G| |c| (2 + 2 electrons in 10 orbitals, coefficients falling by 10^-D with the
// excitation level; 50 bits, 12 moduli / 58 bits, 13 moduli / slices): D = 0 4e-15 / 4e-15 /
// 1.5e-14, 4 4e-13 / 3e-14 / 8e-13, 6 7e-12 / 1e-13 / 3e-12, 8 7e-10 / 5e-12 / 1e-11, 12 5e-8 /
// 1e-10 / 2e-11; falling along the determinants or at random the 58 bits stay below the
// slices to D = 12.
//
// Order: pairs (p, r) by level, then p, then r, and hole pairs by class, then X,
// then Y, so that a determinant row's T elements -- rows (p, *), columns (X, *) for
// the ne holes of its alpha string -- are a few dense blocks, read once and turned
// in shared memory.  In full CI (every class reaches every row) the levels are
// dropped: one block of n x nhole per hole.  Classes that reach the same rows
// are one product.  The same-spin products cover all levels at once: C is the
// [alpha strings][beta strings] matrix with zeros outside the space, rows and
// columns sorted by level, so a tile's K range is a range of strings.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <memory>
#include <queue>
#include <vector>

#include "internal.cuh"
#include "crt.cuh"
#include "crt_gemm.cuh"
#include "crt_host.cuh"
#include "ozaki_digits.cuh"
#include "tma_map.h"

namespace iscsi {

constexpr double kCrtUnitBits = 49.9;  // least bits of the largest unit (the error-free slices: 49)
constexpr int kCrtUnitBitsMax = 52;    // bits that are left over go to the unit up to here, then to the coefficients
constexpr int kCrtCBits = 58;          // least bits of the largest coefficient
constexpr int kCrtCBitsMax = 59, kCrtIntBits = 62;  // of coefficients (four limbs) and of units (five)

// ---------------------------------------------------------------------------
// constants

// modular inverse of a mod m (coprime)
static int mod_inverse(int a, int m) {
  long long t = 0, nt = 1, r = m, nr = a % m;
  while (nr) {
    const long long q = r / nr;
    std::swap(t -= q * nt, nt);
    std::swap(r -= q * nr, nr);
  }
  return (int)(t < 0 ? t + m : t);
}

CrtMods crt_make_mods(int nm, int limbs) {
  CrtMods c;
  std::memset(&c, 0, sizeof(c));
  c.nm = nm;
  for (int i = 0; i < kCrtMaxMods; ++i) {
    const int m = kCrtModuli[i];
    auto twice = [](float f) {
      uint32_t b;
      std::memcpy(&b, &f, sizeof(b));
      return ((unsigned long long)b << 32) | b;
    };
    auto sym = [&](long long x) {
      const int r = (int)(x % m);
      return twice((float)(2 * r > m ? r - m : r));
    };
    c.m[i] = m;
    for (int k = 1; k < limbs; ++k) c.c[k - 1][i] = sym(1ll << ((limbs == 4 ? 15 : 13) * k));
    c.inv[i] = twice(1.0f / (float)m);
    c.neg[i] = twice(-(float)m);
  }
  return c;
}

// reconstruction weights: M's top 64 bits and the fractions (M/m)^-1 / m to 78
// bits by long division; terms: residues of the first pass of k_crt_fold, of each later pass, later passes
CrtWeights crt_make_weights(int nm, int terms, int terms_next, int passes_next) {
  CrtWeights W;
  std::memset(&W, 0, sizeof(W));
  std::vector<uint32_t> M(1, 1);
  for (int i = 0; i < nm; ++i) {
    unsigned long long carry = 0;
    for (uint32_t& x : M) {
      const unsigned long long p = (unsigned long long)x * kCrtModuli[i] + carry;
      x = (uint32_t)p;
      carry = p >> 32;
    }
    if (carry) M.push_back((uint32_t)carry);
  }
  int bits = 32 * (int)(M.size() - 1);
  for (uint32_t x = M.back(); x; x >>= 1) ++bits;
  for (int b = 0; b < 64; ++b) {
    const int at = bits - 1 - b;
    W.mman = (W.mman << 1) | (at >= 0 ? (M[at / 32] >> (at % 32)) & 1u : 0u);
  }
  W.mexp = bits - 64;
  unsigned __int128 start = 0;
  for (int i = 0; i < nm; ++i) {
    const int m = kCrtModuli[i];
    long long rest = 1;
    for (int j = 0; j < nm; ++j)
      if (j != i) rest = rest * kCrtModuli[j] % m;
    unsigned __int128 w = 0;
    unsigned rem = (unsigned)mod_inverse((int)rest, m);
    for (int b = 0; b < 78; ++b) {
      rem <<= 1;
      w = (w << 1) | (rem >= (unsigned)m ? 1u : 0u);
      if (rem >= (unsigned)m) rem -= m;
    }
    if (2 * rem >= (unsigned)m) ++w;
    W.hi[i] = (uint32_t)(w >> 46);
    W.lo1[i] = (uint32_t)(w >> 32) & 0x3FFFu;
    W.lo0[i] = (uint32_t)w;
    W.off[i] = (terms * kCrtResMax + m - 1) / m * m;
    W.off_next[i] = (terms_next * kCrtResMax + m - 1) / m * m;
    start -= w * (unsigned)(W.off[i] + passes_next * W.off_next[i]);
  }
  W.start_lo = (unsigned long long)start & ((1ull << 46) - 1);
  W.start_hi = (uint32_t)(start >> 46);
  return W;
}

double crt_log2_product(int nm) {
  double s = 0.0;
  for (int i = 0; i < nm; ++i) s += std::log2((double)kCrtModuli[i]);
  return s;
}

static inline int up(int x, int m) { return (x + m - 1) / m * m; }

// columns per tile: as few tiles as 256 columns allow, equally wide
static int tile_cols(int N) {
  const int nt = (N + CRT_MAXN - 1) / CRT_MAXN;
  return std::max(16, up((N + nt - 1) / nt, 16));
}

// ---------------------------------------------------------------------------
// operand kernels

// largest row 1-norm and element of a matrix, X(r, k) = X[r * ld + k] or
// X[k * ld + r] when trans: out[0], out[1] (bit patterns of non-negative doubles
// order like integers)
__global__ void __launch_bounds__(256) k_crt_norms(const double* __restrict__ X, int cols, long long ld, int trans,
                                                   unsigned long long* __restrict__ out) {
  const int r = blockIdx.x;
  double s = 0.0, m = 0.0;
  for (int k = threadIdx.x; k < cols; k += blockDim.x) {
    const double x = fabs(trans ? X[(long long)k * ld + r] : X[(long long)r * ld + k]);
    s += x;
    m = x <= m ? m : x;  // keeps a NaN
  }
  __shared__ double ss[256], sm[256];
  ss[threadIdx.x] = s;
  sm[threadIdx.x] = m;
  __syncthreads();
  for (int o = 128; o; o >>= 1) {
    if ((int)threadIdx.x < o) {
      ss[threadIdx.x] += ss[threadIdx.x + o];
      const double x = sm[threadIdx.x + o];
      sm[threadIdx.x] = x <= sm[threadIdx.x] ? sm[threadIdx.x] : x;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    atomicMax(out, (unsigned long long)__double_as_longlong(ss[0]));
    atomicMax(out + 1, (unsigned long long)__double_as_longlong(sm[0]));
  }
}

// residues of a matrix in integers of 2^-sh, in blocks of bt rows: one thread
// per row and 8-wide K chunk, rows_pad rows and nkb k blocks (zeros beyond the
// matrix); row r and column k of the result are those of X at map[r], map[k]
// (or r, k)
__global__ void __launch_bounds__(256) k_crt_cut(const double* __restrict__ X, int rows, int cols, long long ld,
                                                 int trans, const int* __restrict__ map, int sh, int bt, int rows_pad,
                                                 int nkb, const __grid_constant__ CrtMods M,
                                                 __nv_bfloat16* __restrict__ out) {
  const long long t = blockIdx.x * 256ll + threadIdx.x;
  const int nch = 8 * nkb;
  if (t >= (long long)rows_pad * nch) return;
  // neighbouring threads read neighbouring elements: chunks of a row, or rows of a transposed matrix
  const int r = trans ? (int)(t % rows_pad) : (int)(t / nch);
  const int kc = trans ? (int)(t / rows_pad) : (int)(t % nch);
  CrtLimbs2<5> x[4];
  auto value = [&](int k) -> long long {
    if (r >= rows || k >= cols) return 0;
    const long long rr = map ? map[r] : r, kk = map ? map[k] : k;
    return crt_fixed(trans ? X[kk * ld + rr] : X[rr * ld + kk], 0, sh);
  };
#pragma unroll
  for (int j = 0; j < 4; ++j) x[j] = crt_limbs2<5>(value(kc * 8 + 2 * j), value(kc * 8 + 2 * j + 1));
  const int rb = r / bt;
  __nv_bfloat16* o = out + (((long long)rb * nkb + (kc >> 3)) * bt + (r - rb * bt)) * CRT_BK + (kc & 7) * 8;
  crt_store8(x, M, o, (long long)rows_pad * nkb * CRT_BK);
}

// Infinities and NaN of a vector: their number, and the determinants of the first kCrtBad of them
constexpr int kCrtBad = 64;
struct CrtBadList {
  int* count;        // this call's, cleared by k_crt_fold
  int* count_now;    // k_crt_operands' copy for k_crt_fold
  long long* det;    // [vector][kCrtBad]
};

// exponent field of the largest finite |c| of each vector, and its elements that are not finite;
// acc and the counts start at zero (k_crt_fold clears them again)
__global__ void __launch_bounds__(256) k_crt_cmax(const double* __restrict__ c, long long ndet, int* __restrict__ acc,
                                                  CrtBadList bad) {
  const double* v = c + (long long)blockIdx.y * ndet;
  const long long stride = (long long)gridDim.x * 256;
  int m = 0;
  long long i = blockIdx.x * 256ll + threadIdx.x;
  for (; i + 3 * stride < ndet; i += 4 * stride) {
    const double a = __ldg(v + i), b = __ldg(v + i + stride), d = __ldg(v + i + 2 * stride), e = __ldg(v + i + 3 * stride);
    m = max(m, max(max(oz_exp_field(a), oz_exp_field(b)), max(oz_exp_field(d), oz_exp_field(e))));
  }
  for (; i < ndet; i += stride) m = max(m, oz_exp_field(__ldg(v + i)));
  if (m == 0x7FF) {
    m = 0;
    for (i = blockIdx.x * 256ll + threadIdx.x; i < ndet; i += stride) {
      const int f = oz_exp_field(__ldg(v + i));
      if (f < 0x7FF) {
        m = max(m, f);
      } else {
        const int k = atomicAdd(bad.count + blockIdx.y, 1);
        if (k < kCrtBad) bad.det[(long long)blockIdx.y * kCrtBad + k] = i;
      }
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(acc + blockIdx.y, m);
}

// A group of column classes of the lifted vector (one product)
struct CrtLiftGroup {
  int hp_start, ncol, krows, nkb, bt, wpc;
  long long base, mod_stride;  // its block of the residue buffer (elements)
};
struct CrtOperands {
  int nvec, ngroups, n, nholeA, nholeB, cbits;
  CrtLiftGroup g[2 * kMaxElec];
  int blk_start[2 * kMaxElec + 1];  // first block of each group's columns; then the C tiles
  const int *pair, *hp_inv;  // K order -> (q << 16) | s; column order -> X * nholeB + Y (null: the same)
  const int *liftA, *liftB;
  const int8_t* alevel;
  const int* nballow;
  const long long* off;
  long long ndet;
  int *cmax, *cexp;          // exponent fields: largest of this call, and the copy for k_crt_fold
  CrtBadList bad;
  __nv_bfloat16* lift;
  // same spin
  int na, nb, ctx_x, ctx_y;  // strings; 64 x 64 tiles along beta and alpha (0: no same-spin part)
  __nv_bfloat16 *ca, *ct;    // C (rows alpha, blocks of 128) and C^T (rows beta, blocks of bt); either may be null
  long long ca_mod, ct_mod, ca_vec, ct_vec;
  int nkb_ca, nkb_ct, bt;
};

// lift entries of a column for n orbitals in dynamic shared memory: off[n], a[n], b[n], lim[n]
struct CrtLiftView {
  long long* off;
  int *a, *b, *lim;
};
__host__ __device__ constexpr int crt_lift_col_bytes(int n) { return (20 * n + 7) / 8 * 8; }

__device__ __forceinline__ double crt_lift_value(const CrtLiftView& L, int qs, const double* __restrict__ cv) {
  const int q = qs >> 16, s = qs & 0xFFFF;
  const int ea = L.a[q], eb = L.b[s];
  if (ea < 0 || eb < 0) return 0.0;
  const int Bp = eb >> 1;
  if (Bp >= L.lim[q]) return 0.0;
  // (the sign by the integer units: a negation on the FP64 pipe takes 64 cycles a warp)
  return __longlong_as_double(__double_as_longlong(cv[L.off[q] + Bp]) ^ ((long long)((ea ^ eb) & 1) << 63));
}

// Blocks of lift columns first (eight warps: one, two, four or eight per
// column by its length), then 64 x 64 tiles of C.  A lane gathers 8 consecutive K
// values and writes their residues as 16 bytes per modulus, eight lanes a full
// 128-byte line.  Elements outside the space, and padding, are zero from the
// buffers' first clearing on.
__global__ void __launch_bounds__(256) k_crt_operands(const __grid_constant__ CrtOperands O,
                                                      const __grid_constant__ CrtMods M,
                                                      const double* __restrict__ c) {
  extern __shared__ __align__(16) unsigned char crt_dyn[];
  const int nlift = O.blk_start[O.ngroups];
  if (blockIdx.x == 0)
    for (int v = threadIdx.x; v < O.nvec; v += 256) {
      O.cexp[v] = O.cmax[v];
      O.bad.count_now[v] = O.bad.count[v];
    }
  if ((int)blockIdx.x < nlift) {
    int gi = 0;
    while ((int)blockIdx.x >= O.blk_start[gi + 1]) ++gi;
    const CrtLiftGroup& G = O.g[gi];
    const int wpc = G.wpc, cpb = 8 / wpc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wc = warp / wpc, wk = warp % wpc;
    const int col = ((int)blockIdx.x - O.blk_start[gi]) * cpb + wc;
    const bool live = col < G.ncol * O.nvec;
    const int n = O.n;
    unsigned char* tab = crt_dyn + wc * crt_lift_col_bytes(n);
    CrtLiftView L;
    L.off = reinterpret_cast<long long*>(tab);
    L.a = reinterpret_cast<int*>(tab + 8 * n);
    L.b = L.a + n;
    L.lim = L.b + n;
    const int v = live ? col / G.ncol : 0;
    if (live) {
      const int hp = G.hp_start + col - v * G.ncol;
      const int xy = O.hp_inv ? O.hp_inv[hp] : hp;
      const int X = xy / O.nholeB, Y = xy - X * O.nholeB;
      for (int q = wk * 32 + lane; q < n; q += 32 * wpc) {
        const int ea = O.liftA[q * O.nholeA + X];
        L.a[q] = ea;
        L.b[q] = O.liftB[q * O.nholeB + Y];
        if (ea >= 0) {
          const int A = ea >> 1;
          L.off[q] = O.off[A];
          L.lim[q] = O.nballow[O.alevel[A]];
        }
      }
    }
    __syncthreads();
    if (!live) return;
    const double* cv = c + (long long)v * O.ndet;
    const int f = O.cmax[v], ex = f > 0 ? f - 1022 : 0;
    const int rb = col / G.bt;
    __nv_bfloat16* row = O.lift + G.base + ((long long)rb * G.nkb * G.bt + (col - rb * G.bt)) * CRT_BK;
    for (int kc = wk * 32 + lane; kc < 8 * G.nkb; kc += 32 * wpc) {
      // the pair table is padded to whole k blocks; pairs beyond the group's rows give zero
      const int4 k0 = __ldg(reinterpret_cast<const int4*>(O.pair) + 2 * kc);
      const int4 k1 = __ldg(reinterpret_cast<const int4*>(O.pair) + 2 * kc + 1);
      const int qs[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
      double val[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) val[j] = kc * 8 + j < G.krows ? crt_lift_value(L, qs[j], cv) : 0.0;
      CrtLimbs2<4> x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        x[j] = crt_limbs2<4>(crt_fixed(val[2 * j], ex, O.cbits), crt_fixed(val[2 * j + 1], ex, O.cbits));
      crt_store8(x, M, row + (long long)(kc >> 3) * G.bt * CRT_BK + (kc & 7) * 8, G.mod_stride);
    }
    return;
  }
  // a 64 x 64 tile of C, turned in shared memory
  double(*tile)[65] = reinterpret_cast<double(*)[65]>(crt_dyn);
  int t = (int)blockIdx.x - nlift;
  const int z = t / (O.ctx_x * O.ctx_y);
  t -= z * O.ctx_x * O.ctx_y;
  const int A0 = (t / O.ctx_x) * 64, B0 = (t % O.ctx_x) * 64;
  if (O.nballow[O.alevel[A0]] <= B0) return;  // outside the space (levels ascend, prefixes shrink)
  const double* cv = c + (long long)z * O.ndet;
  for (int i = threadIdx.x; i < 64 * 64; i += 256) {
    const int a = i >> 6, b = i & 63, A = A0 + a, B = B0 + b;
    double x = 0.0;
    if (A < O.na && B < O.nballow[O.alevel[A]]) x = cv[O.off[A] + B];
    tile[a][b] = x;
  }
  __syncthreads();
  const int f = O.cmax[z], ex = f > 0 ? f - 1022 : 0;
  for (int i = threadIdx.x; i < 1024; i += 256) {
    const bool tr = i >= 512;  // a chunk of C^T (a beta string, 8 alpha strings) or of C
    const int r = (i & 511) >> 3, kc = i & 7;
    const int R = (tr ? B0 : A0) + r;
    if ((tr ? O.ct : O.ca) == nullptr || R >= (tr ? O.nb : O.na)) continue;
    CrtLimbs2<4> x[4];
    auto value = [&](int j) { return crt_fixed(tr ? tile[kc * 8 + j][r] : tile[r][kc * 8 + j], ex, O.cbits); };
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = crt_limbs2<4>(value(2 * j), value(2 * j + 1));
    const int bt = tr ? O.bt : CRT_BM, rb = R / bt, kb = (tr ? A0 : B0) / CRT_BK;
    __nv_bfloat16* o = (tr ? O.ct + z * O.ct_vec : O.ca + z * O.ca_vec) +
                       (((long long)rb * (tr ? O.nkb_ct : O.nkb_ca) + kb) * bt + (R - rb * bt)) * CRT_BK + kc * 8;
    crt_store8(x, M, o, tr ? O.ct_mod : O.ca_mod);
  }
}

// ---------------------------------------------------------------------------
// fold and reconstruction

struct CrtFoldGroup {
  long long res;  // first residue of the group's product
  int ncol, ntile, tn;
};
struct CrtFold {
  int na, nb, n, nholeB, nvec, nm, na_strings;
  int parts;                 // 1: opposite spin, 2: same spin
  const int16_t* res;
  CrtFoldGroup g[2 * kMaxElec];
  const int *decA, *decB;
  // rows of (p, *): one run of all r, or two split at rsplit; columns of (X, *):
  // one run of all Y, or one per level of Y
  int rruns, rsplit, yruns, kmax;
  int ystart[kMaxElec + 2];
  const int* rowrun;         // [n][rruns] first row
  const int2* colrun;        // [nholeA][yruns] (group, first column in it)
  int xlev;                  // 0: no levels
  // same spin
  long long ss_res, ss_vec;
  int ss_ntile, ss_tn;
  const long long* off;
  const int8_t* alevel;
  const int* nballow;
  long long ndet;
  int *cmax, *cexp;
  CrtBadList bad;
  int ebias;                 // -(bits of the coefficients) - sh
  const int* ypos;           // per Y: run << 24 | position in a staged row (before the run's shift)
  int ypad[kMaxElec + 2];    // first position of each run in a staged row (multiples of 8)
  // a staged hole: rows r < rsplit of stride elements, the others of stride1 from base1 on (in a
  // truncated space these lack the runs of Y whose levels they cannot reach); odd numbers of
  // 16-byte units
  int stride, stride1, base1, hole_elems;
  int row0;                  // first alpha string of this launch
  int ni;                    // holes staged together
  int nbuf, stage_bytes;     // buffers (2 to 4: nbuf - 1 moduli are copied ahead) and their size
};
constexpr int kFoldPer = 4;  // determinants per thread
constexpr int kFoldThreads = 1024;

// first element of orbital r's row in a staged hole
__device__ __forceinline__ int fold_row(const CrtFold& F, int r) {
  return r < F.rsplit ? r * F.stride : F.base1 + (r - F.rsplit) * F.stride1;
}

// whether a determinant of the list lies within two excitations of (A, B): where H reaches it (the orbitals of a
// string are those of its dec entries)
__device__ __forceinline__ bool crt_reached(const CrtFold& F, const long long* det, int count, int A, int B) {
  if (count > kCrtBad) return true;
  for (int k = 0; k < count; ++k) {
    int a = 0, hi = F.na_strings;
    while (hi - a > 1) {
      const int mid = (a + hi) >> 1;
      if (F.off[mid] <= det[k]) a = mid;
      else hi = mid;
    }
    const int b = (int)(det[k] - F.off[a]);
    int moved = F.na + F.nb;
    for (int i = 0; i < F.na; ++i)
      for (int j = 0; j < F.na; ++j) moved -= ((F.decA[A * F.na + i] ^ F.decA[a * F.na + j]) & 0x1FE) == 0;
    for (int i = 0; i < F.nb; ++i)
      for (int j = 0; j < F.nb; ++j) moved -= ((F.decB[B * F.nb + i] ^ F.decB[b * F.nb + j]) & 0x1FE) == 0;
    if (moved <= 2) return true;
  }
  return false;
}

// One block per alpha string (and vector, and share of its beta strings): for
// each modulus the T blocks of the string's holes are copied into shared
// memory as they lie (16-byte units, one modulus ahead), every determinant adds
// its na nb entries with their signs and its same-spin residue, and the sum goes
// into its 78-bit fraction.  NB: beta electrons whose offsets stay in registers
// (0: any number, looked up each time).  Each T element is read once, in whole
// 16-byte units of consecutive rows.
// MR: several runs of Y (a truncated space).  The phase of a hole is (-1)^i for
// the i-th orbital of its string (the order of the dec tables), so signs need no
// look-up.
template <int NB, bool MR>
__global__ void __launch_bounds__(kFoldThreads) k_crt_fold(const __grid_constant__ CrtFold F,
                                                           const __grid_constant__ CrtWeights W,
                                                           double* __restrict__ sigma) {
  extern __shared__ __align__(16) unsigned char crt_dyn[];
  __shared__ int shift_s[kMaxElec * (kMaxElec + 1)];  // per hole and run of Y: columns before its first in a row
  __shared__ int units_s;
  const int A = F.row0 + blockIdx.x, v = blockIdx.z;
  const int lim = F.nballow[F.alevel[A]];
  const int B0 = blockIdx.y * (blockDim.x * kFoldPer) + threadIdx.x;
  if ((int)(blockIdx.y * (blockDim.x * kFoldPer)) >= lim) return;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) F.cmax[v] = F.bad.count[v] = 0;  // for the next call
  const bool ab = (F.parts & 1) != 0, ss = (F.parts & 2) != 0;
  int16_t* const stage = reinterpret_cast<int16_t*>(crt_dyn);
  uint2* const unit = reinterpret_cast<uint2*>(crt_dyn + (size_t)F.nbuf * F.stage_bytes);
  const int hs = F.hole_elems;  // elements of one staged hole

  unsigned long long lo[kFoldPer];
  uint32_t hi[kFoldPer];
  int offs[kFoldPer][NB ? NB : 1];  // position in a hole's block; MR: << 5 | run of Y
  int ssoff[kFoldPer];              // position of the same-spin residue in the row's tiles (modulus 0)
  const int ss_tile = CRT_BM * F.ss_ntile;
#pragma unroll
  for (int u = 0; u < kFoldPer; ++u) {
    lo[u] = W.start_lo;
    hi[u] = W.start_hi;
    const int B = min(B0 + u * (int)blockDim.x, lim - 1);
    if (NB && ab) {
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int db = F.decB[B * NB + j];
        const int yp = F.ypos[db >> 9];
        const int at = fold_row(F, (db >> 1) & 255) + (yp & 0xFFFFFF);
        offs[u][j] = MR ? (at << 5) | (yp >> 24) : at;
      }
    }
    ssoff[u] = 0;
    if (ss) {
      const int nt = B / F.ss_ntile, cc = B - nt * F.ss_ntile;
      ssoff[u] = nt * F.nm * ss_tile + (cc >> 3) * (CRT_BM * 8) + (cc & 7);
    }
  }
  const int16_t* const ssrow = F.res + F.ss_res + v * F.ss_vec + (long long)(A >> 7) * F.ss_tn * F.nm * ss_tile + (A & 127) * 8;

  for (int i0 = 0; i0 == 0 || (ab && i0 < F.na); i0 += F.ni) {
    const int i1 = ab ? min(F.na, i0 + F.ni) : 0;
    int nunits = 0;
    if (ab) {
      // the 16-byte units of holes [i0, i1): source in units from F.res (modulus 0),
      // destination unit | group << 24
      __syncthreads();  // the previous holes' units are copied and read
      if (threadIdx.x == 0) units_s = 0;
      __syncthreads();
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
      int cnt = 0;
      for (int i = i0; i < i1; ++i) {
        const int da = F.decA[A * F.na + i];
        const int X = da >> 9, p = (da >> 1) & 255;
        for (int yy = 0; yy < F.yruns; ++yy) {
          const int y0 = F.ystart[yy], nc = F.ystart[yy + 1] - y0;
          if (nc <= 0) continue;
          const int2 cr = F.colrun[X * F.yruns + yy];
          const CrtFoldGroup& G = F.g[cr.x];
          const int J0 = v * G.ncol + cr.y;
          if (threadIdx.x == 0) shift_s[(i - i0) * F.yruns + yy] = J0 & 7;
          const int ncg = ((J0 + nc - 1) >> 3) - (J0 >> 3) + 1;
          for (int rr = 0; rr < F.rruns; ++rr) {
            const int r0 = rr ? F.rsplit : 0, nr = (rr + 1 < F.rruns ? F.rsplit : F.n) - r0;
            if (nr <= 0) continue;
            if (F.xlev && F.alevel[A] + rr + yy > F.kmax) continue;  // outside the space
            const int R0 = F.rowrun[p * F.rruns + rr];
            for (int w = warp; w < ncg; w += nwarps) {
              const int col = (J0 & ~7) + w * 8;
              const int nt = col / G.ntile, cg = (col - nt * G.ntile) >> 3;
              const long long src = (G.res >> 3) + (long long)nt * F.nm * (16 * G.ntile) + cg * CRT_BM;
              const long long rts = (long long)G.tn * F.nm * (16 * G.ntile);
              for (int r = lane; r < nr; r += 32) {
                const int row = R0 + r;
                unit[cnt + w * nr + r] =
                    make_uint2((uint32_t)(src + (row >> 7) * rts + (row & 127)),
                               (uint32_t)(((i - i0) * hs + fold_row(F, r0 + r) + F.ypad[yy]) / 8 + w) | ((uint32_t)cr.x << 24));
              }
            }
            cnt += ncg * nr;
          }
        }
      }
      if (threadIdx.x == 0) units_s = cnt;
      __syncthreads();
      nunits = units_s;
    }
    auto copy = [&](int mod) {
      const uint32_t dst = tc::smem_u32(stage) + (mod % F.nbuf) * F.stage_bytes;
      for (int q = threadIdx.x; q < nunits && mod < F.nm; q += blockDim.x) {
        const uint2 x = unit[q];
        const uint4* src = reinterpret_cast<const uint4*>(F.res) + x.x + (size_t)mod * (16 * F.g[x.y >> 24].ntile);
        tc::cp_async16(dst + (x.y & 0xFFFFFFu) * 16, src);
      }
      tc::cp_async_commit();
    };
    if (ab)
      for (int m = 0; m + 1 < F.nbuf; ++m) copy(m);
#pragma unroll 1
    for (int mod = 0; mod < F.nm; ++mod) {
      int sum[kFoldPer];
#pragma unroll
      for (int u = 0; u < kFoldPer; ++u) sum[u] = ss && i0 == 0 ? ssrow[ssoff[u] + mod * ss_tile] : 0;
      if (ab) {
        // modulus mod has arrived for every thread, and all are done with the buffer that the
        // copy nbuf - 1 moduli ahead goes to
        if (F.nbuf >= 4) tc::cp_async_wait<2>();
        else if (F.nbuf == 3) tc::cp_async_wait<1>();
        else tc::cp_async_wait<0>();
        __syncthreads();
        copy(mod + F.nbuf - 1);
        const int16_t* st = stage + (size_t)(mod % F.nbuf) * (F.stage_bytes / 2);
        for (int i = i0; i < i1; ++i, st += hs) {
          const int sgn = 1 - 2 * (i & 1);
          const int* sh = shift_s + (i - i0) * F.yruns;
          const int16_t* sti = MR ? st : st + sh[0];
#pragma unroll
          for (int u = 0; u < kFoldPer; ++u) {
            int s = 0;
            if (NB) {
#pragma unroll
              for (int j = 0; j < NB; ++j) {
                const int o = offs[u][j];
                const int x = MR ? sti[(o >> 5) + sh[o & 31]] : sti[o];
                s = (j & 1) ? s - x : s + x;
              }
            } else {
              const int B = min(B0 + u * (int)blockDim.x, lim - 1);
              for (int j = 0; j < F.nb; ++j) {
                const int db = F.decB[B * F.nb + j];
                const int yp = F.ypos[db >> 9];
                const int x = st[fold_row(F, (db >> 1) & 255) + (yp & 0xFFFFFF) + sh[yp >> 24]];
                s += (j & 1) ? -x : x;
              }
            }
            sum[u] += s * sgn;
          }
        }
      }
      const uint32_t w0 = W.lo0[mod], w1 = W.lo1[mod], w2 = W.hi[mod];
      const int off = i0 == 0 ? W.off[mod] : W.off_next[mod];
#pragma unroll
      for (int u = 0; u < kFoldPer; ++u) {
        const uint32_t t = (uint32_t)(sum[u] + off);
        lo[u] += (unsigned long long)t * w0;
        lo[u] += (unsigned long long)(t * w1) << 32;
        hi[u] += t * w2;
      }
    }
#pragma unroll
    for (int u = 0; u < kFoldPer; ++u) {  // keep the low part within its 46 bits between passes
      hi[u] += (uint32_t)(lo[u] >> 46);
      lo[u] &= (1ull << 46) - 1;
    }
  }
  const int f = F.cexp[v];
  const int e = (f > 0 ? f - 1022 : 0) + F.ebias;
  double* out = sigma + v * F.ndet + F.off[A];
#pragma unroll
  for (int u = 0; u < kFoldPer; ++u) {
    const int B = B0 + u * (int)blockDim.x;
    if (B < lim) out[B] = crt_value(lo[u], hi[u], W.mman, W.mexp, e);
  }
  const int nbad = F.bad.count_now[v];
  if (nbad == 0) return;
#pragma unroll 1
  for (int B = B0; B < lim && B < B0 + kFoldPer * (int)blockDim.x; B += blockDim.x)
    if (crt_reached(F, F.bad.det + v * kCrtBad, nbad, A, B)) out[B] = __longlong_as_double(0x7FF8000000000000ll);
}

// ---------------------------------------------------------------------------
// work list and schedule
// items in the order that keeps the pairs on neighbouring tiles of one modulus
// (their operands shared in L2), dealt out in that order to the pair with the
// least work so far; the products with the largest tiles first
static void crt_schedule(const std::vector<CrtHostProblem>& probs, int npairs, std::vector<CrtItem>& items,
                         std::vector<int>& start, double& flops) {
  std::vector<int> order(probs.size());
  std::vector<double> big(probs.size(), 0.0);
  for (size_t i = 0; i < probs.size(); ++i) {
    order[i] = (int)i;
    big[i] = (double)probs[i].p.nkb_a * probs[i].p.ntile;
  }
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return big[x] > big[y]; });
  std::vector<std::vector<CrtItem>> of(npairs);
  using Q = std::pair<double, int>;
  std::priority_queue<Q, std::vector<Q>, std::greater<Q>> heap;
  for (int b = 0; b < npairs; ++b) heap.push({0.0, b});
  flops = 0.0;
  constexpr int kBand = 8;
  for (int pi : order) {
    const CrtHostProblem& H = probs[pi];
    if (!H.own) continue;
    for (int mod = 0; mod < H.p.nm; ++mod)
      for (int m0 = 0; m0 < H.mt; m0 += kBand)
        for (int nt = 0; nt < H.p.tn; ++nt)
          for (int mt = m0; mt < std::min(H.mt, m0 + kBand); ++mt) {
            int k0 = 0, k1 = 0;
            if (!H.range(mt, nt, k0, k1)) continue;
            CrtItem it{pi, mt, nt, mod, k0, std::max(0, k1 - k0), H.p.ntile, -1, 0, 0, 0, 0};
            if (H.second >= 0) {
              it.probb = pi + H.second;
              probs[it.probb].range(mt, nt, k0, k1);
              it.kb0b = k0;
              it.nkbb = std::max(0, k1 - k0);
            }
            const int nkb = it.nkb + it.nkbb;
            Q q = heap.top();
            heap.pop();
            of[q.second].push_back(it);
            // cycles: four MMAs of ntile / 2 cycles per k block (at least the loads' time), the epilogue's store
            q.first += nkb * std::max(4.0 * it.ntile / 2.0, 400.0) + 1500.0;
            heap.push(q);
            flops += 2.0 * 256.0 * it.ntile * 64.0 * nkb;
          }
  }
  items.clear();
  start.assign(1, 0);
  for (int b = 0; b < npairs; ++b) {
    if (of[b].empty()) continue;
    items.insert(items.end(), of[b].begin(), of[b].end());
    start.push_back((int)items.size());
  }
}

int CrtJob::upload(cudaStream_t st) {
  std::vector<CrtItem> items;
  std::vector<int> start;
  crt_schedule(probs, tc_sm_count() / 2, items, start, flops);
  grid = 2 * ((int)start.size() - 1);
  nitems = (int)items.size();
  std::vector<CrtProblem> pr;
  for (const CrtHostProblem& h : probs) pr.push_back(h.p);
  ISCSI_TRY(d_probs.grow(sizeof(CrtProblem) * std::max<size_t>(1, pr.size())));
  ISCSI_TRY(d_items.grow(sizeof(CrtItem) * std::max<size_t>(1, items.size())));
  ISCSI_TRY(d_start.grow(sizeof(int) * start.size()));
  if (!pr.empty())
    ISCSI_CUDA(cudaMemcpyAsync(d_probs.p, pr.data(), sizeof(CrtProblem) * pr.size(), cudaMemcpyHostToDevice, st));
  if (!items.empty())
    ISCSI_CUDA(
        cudaMemcpyAsync(d_items.p, items.data(), sizeof(CrtItem) * items.size(), cudaMemcpyHostToDevice, st));
  ISCSI_CUDA(cudaMemcpyAsync(d_start.p, start.data(), sizeof(int) * start.size(), cudaMemcpyHostToDevice, st));
  ISCSI_CUDA(cudaStreamSynchronize(st));  // the host vectors end here
  return kOk;
}

int CrtJob::launch(int* err, cudaStream_t st) const {
  if (grid == 0) return kOk;
  static bool attr = false;
  if (!attr) {
    ISCSI_CUDA(cudaFuncSetAttribute(k_crt_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, CRT_SMEM_BYTES));
    attr = true;
  }
  static const CrtMods all = crt_make_mods(kCrtMaxMods);  // the kernel reads the moduli themselves
  k_crt_gemm<<<grid, CRT_THREADS, CRT_SMEM_BYTES, st>>>(d_probs.as<CrtProblem>(), d_items.as<CrtItem>(),
                                                        d_start.as<int>(), all, err); ISCSI_COUNT_LAUNCH();
  ISCSI_CUDA(cudaGetLastError());
  return kOk;
}

// ---------------------------------------------------------------------------
// a context's state

struct CrtGroup {
  int hp_start = 0, ncol = 0, rows = 0;  // hole pairs, rows (= K) reached
};

// one launch of k_crt_fold: a range of alpha strings
struct CrtFoldLaunch {
  CrtFold f;
  CrtWeights w;
  int rows = 0, threads = 0, blocks = 0, smem = 0;
};

constexpr int kCrtMaxVecs = 65535;  // vectors are a grid dimension of k_crt_cmax and k_crt_fold

struct CrtState {
  bool off = false;  // its units are not finite: the context stays on the slices
  int max_vecs = kCrtMaxVecs;  // larger blocks did not fit: they take the slices
  CrtHeld held;      // residue buffers (crt_alloc)
  bool flat = false;  // every class reaches every row: no levels in the orders
  std::vector<CrtGroup> groups;
  std::vector<int> ystart;
  std::vector<int> ypad;
  DevBuf pair, map, rowrun, colrun, ypos;
  // scales: units are integers of 2^-sh
  CrtMods mods, unit_mods;              // of the vectors, and of G and the string matrices
  int sh = 0, cbits = 0;                // and a vector's coefficients of 2^(e - cbits)
  double bound = 0.0;                   // the bound of |sigma| / max |c| that sh was chosen for
  int g_cut[2] = {-1, 0}, m_cut[2] = {-1, 0};  // moduli and sh of the residues in g_res, ma_res / mb_res
  double rg = 0.0, gmax = 0.0;          // G's row 1-norm and largest element (-1: not taken)
  bool g_norm = false;
  DevBuf norms;
  DevBuf g_res, b_res;                  // G, lifted vector
  DevBuf ma_res, mb_res, ca_res, ct_res;  // string matrices, C, C^T
  DevBuf cfield;                        // of the vectors: lists of non-finite elements, exponent fields and counts (this call's, copies)
  DevBuf out;                           // residues of the products
  CrtOperands ops;
  CrtFold fold;
  CrtJob job;
  std::vector<CrtFoldLaunch> folds;
  int ops_smem = 0, ops_blocks = 0;
  int nvec = -1, parts = 0;  // what job was built for (parts: 1 opposite spin, 2 same spin)
};

void crt_release(Context& ctx) {
  if (ctx.crt) ++ctx.crt_version;
  delete ctx.crt;
  ctx.crt = nullptr;
}

void crt_invalidate(Context& ctx) {
  if (!ctx.crt) return;
  ctx.crt->nvec = -1;
  ++ctx.crt_version;
}

constexpr int kFoldMaxSmem = 220 * 1024;

static CrtState& crt_state(Context& ctx) {
  if (ctx.crt) return *ctx.crt;
  CrtState* S = new CrtState();
  ctx.crt = S;
  for (int c = 0; ctx.have_ab && c < (int)ctx.cls.size(); ++c) {
    const ColClass& cc = ctx.cls[c];
    if (cc.ncol == 0 || cc.mrows == 0) continue;
    if (S->groups.empty() || S->groups.back().rows != cc.mrows ||
        S->groups.back().hp_start + S->groups.back().ncol != ctx.hp_class_start[c]) {
      CrtGroup g;
      g.hp_start = ctx.hp_class_start[c];
      g.rows = cc.mrows;
      S->groups.push_back(g);
    }
    S->groups.back().ncol += cc.ncol;
  }
  S->flat = S->groups.size() == 1 && S->groups[0].rows == ctx.npairs &&
            (long long)S->groups[0].ncol == (long long)ctx.sp[0].nhole * ctx.sp[1].nhole;
  if (!S->groups.empty()) {
    // runs of the beta hole strings (their levels, sorted; one run without levels) and a row of a
    // staged block: every run on a 16-byte boundary with room for its shift of up to 7 columns, an
    // odd number of 16-byte units so that the units of consecutive rows spread over the banks
    const SpinSpace& HB = ctx.sp[1];
    S->ystart.assign(1, 0);
    if (S->flat) {
      S->ystart.push_back(HB.nhole);
    } else {
      for (int l = 0; l <= HB.hole_maxlevel; ++l) {
        int e = S->ystart.back();
        while (e < HB.nhole && HB.hole_level[e] == l) ++e;
        S->ystart.push_back(e);
      }
      if (S->ystart.back() != HB.nhole) S->off = true;
    }
    int at = 0;
    for (size_t y = 0; y + 1 < S->ystart.size(); ++y) {
      S->ypad.push_back(at);
      at += up(S->ystart[y + 1] - S->ystart[y] + 7, 8);
    }
    S->ypad.push_back(at);
  }
  return *S;
}

// shared memory of k_crt_fold for alpha strings of level lev and above: all holes
// of a string together and up to three moduli copied ahead while two blocks fit an
// SM, else fewer buffers, else one hole at a time
struct FoldShape {
  int ni = 0, nbuf = 0, stride = 0, stride1 = 0, base1 = 0, hole = 0, smem = 0;
};
static FoldShape fold_shape(const Context& ctx, const CrtState& S, int lev) {
  FoldShape f;
  auto row = [&](int runs) {  // a row of the first `runs` runs
    const int at = S.ypad[std::min<int>(runs, (int)S.ypad.size() - 1)];
    return (at / 8) % 2 ? at : at + 8;
  };
  const int all = (int)S.ypad.size() - 1;
  const int nob = S.flat ? ctx.n : ctx.sp[1].nocc;
  const int room = ctx.kmax - lev;  // levels left for r and Y
  f.stride = row(S.flat ? all : std::min(all, room + 1));
  f.stride1 = row(S.flat ? all : std::max(0, std::min(all, room)));
  f.base1 = nob * f.stride;
  f.hole = f.base1 + (ctx.n - nob) * f.stride1;
  const long long units = 8ll * (f.hole / 8 + 8);
  const int together = ctx.na * ctx.nb <= 25 ? ctx.na : 1;  // (at most 26 residues per pass: sums below 2^64)
  // two blocks per SM (113 KB) before all holes in one pass: 4 + 4 electrons in 16 orbitals 182 KB in one
  // pass 710 us, 91 KB in two passes 545 (12 moduli; 13: 559); but one hole per pass is slower (CISDT, 100
  // orbitals: 302 against 279)
  const struct { int ni, nbuf; long long limit; } tries[] = {
      {together, 4, 56 * 1024}, {together, 3, 75 * 1024}, {together, 2, 113 * 1024},
      {(together + 1) / 2, 2, together > 2 ? 113 * 1024 : 0}, {together, 2, kFoldMaxSmem}, {1, 2, kFoldMaxSmem}};
  for (const auto& t : tries) {
    const long long b = t.ni * (t.nbuf * 2ll * f.hole + units);
    if (b <= t.limit) {
      f.ni = t.ni;
      f.nbuf = t.nbuf;
      f.smem = (int)b;
      return f;
    }
  }
  return f;
}

// The opposite-spin contraction goes through residues when its columns fill
// the tiles: a residue product reads nm bf16 matrices of G where the slices
// read seven, so a column group narrower than kCrtMinCols that reaches many
// rows is bound by G's bytes and stays on the slices.  A hole's block of T has
// to fit k_crt_fold's shared memory.
constexpr int kCrtMinCols = 64;
constexpr int kCrtMinRows = 16;

bool crt_ab_active(Context& ctx, int nvec) {
  if (!ctx.have_ab) return false;
  CrtState& S = crt_state(ctx);
  if (S.off || nvec > S.max_vecs || S.groups.empty() || fold_shape(ctx, S, 0).ni == 0) return false;
  double heavy = 0.0, good = 0.0;
  for (const CrtGroup& g : S.groups) {
    const double w = (double)g.rows * g.rows;
    heavy += w;
    if ((long long)g.ncol * nvec >= kCrtMinCols || g.rows <= 1024) good += w;
    if ((long long)g.ncol * nvec > (1 << 30)) return false;
  }
  return good >= 0.9 * heavy && S.groups[0].rows >= kCrtMinRows;
}

// Strings of the space: alpha strings with an allowed beta string, and the longest allowed beta
// prefix (both are sorted by level).  A truncated space of many electrons reaches few of all strings (4 + 4
// electrons in 30 orbitals, doubles: 2055 of 27405), and the string matrices are cut for these alone.
static int alpha_strings(const Context& ctx) {
  int l = 0;
  while (l <= ctx.sp[0].maxlevel && ctx.nb_allowed_lvl[l] > 0) ++l;
  return ctx.sp[0].level_start[l];
}
static int beta_strings(const Context& ctx) {
  long long most = 0;
  for (int l = 0; l <= ctx.sp[0].maxlevel; ++l)
    if (ctx.sp[0].level_start[l + 1] > ctx.sp[0].level_start[l]) most = std::max(most, ctx.nb_allowed_lvl[l]);
  return (int)most;
}

void crt_strings(const Context& ctx, int& sa, int& sb) {
  sa = alpha_strings(ctx);
  sb = beta_strings(ctx);
}

bool crt_full(Context& ctx) { return crt_state(ctx).flat; }

// the same-spin products, all levels at once, when the strings fill a tile or so
bool crt_ss_active(Context& ctx, int nvec) {
  CrtState& S = crt_state(ctx);
  return !S.off && nvec <= S.max_vecs && alpha_strings(ctx) >= kCrtMinRows && beta_strings(ctx) >= kCrtMinRows;
}

int crt_encode(CrtProblem& P, const void* a, const void* b, int nm) {
  if (crt_encode_map(&P.a, a, (long long)nm * P.nblk_a * P.nkb_a * CRT_BM, CRT_BM) ||
      crt_encode_map(&P.b, b, (long long)nm * P.nblk_b * P.nkb_b * (P.ntile / 2), P.ntile / 2)) {
    set_error("residue contraction: TMA descriptor rejected");
    return kErrCuda;
  }
  return kOk;
}

static int cut_matrix(const double* X, int rows, int cols, long long ld, int trans, const int* map, int sh, int bt,
                      int rows_pad, int nkb, const CrtMods& M, __nv_bfloat16* out, cudaStream_t st) {
  const long long threads = (long long)rows_pad * nkb * 8;
  k_crt_cut<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(X, rows, cols, ld, trans, map, sh, bt, rows_pad, nkb, M,
                                                                out); ISCSI_COUNT_LAUNCH();
  ISCSI_CUDA(cudaGetLastError());
  return kOk;
}

// the stored beta matrix is M_beta^T (or the symmetric alpha matrix when shared)
static const double* beta_matrix(const Context& ctx, int& trans) {
  trans = ctx.beta_alias ? 0 : 1;
  return ctx.beta_alias ? ctx.M64[0].as<double>() : ctx.M64[1].as<double>();
}

// row 1-norms and largest elements (synchronises); what: 1 G, 2 the string matrices
static int take_norms(Context& ctx, int what, double& rm, double& mmax) {
  CrtState& S = *ctx.crt;
  cudaStream_t st = stream();
  if (!S.norms.p) ISCSI_TRY(S.norms.alloc(6 * sizeof(double)));
  ISCSI_CUDA(cudaMemsetAsync(S.norms.p, 0, 6 * sizeof(double), st));
  unsigned long long* d = S.norms.as<unsigned long long>();
  if (what & 1) {
    k_crt_norms<<<ctx.npairs, 256, 0, st>>>(ctx.G64.as<double>(), ctx.npairs, ctx.npairs, 0, d); ISCSI_COUNT_LAUNCH();
  }
  if ((what & 2) && ctx.na > 0 && ctx.M64[0].p) {
    const int NA = alpha_strings(ctx);
    k_crt_norms<<<NA, 256, 0, st>>>(ctx.M64[0].as<double>(), NA, ctx.sp[0].count, 0, d + 2); ISCSI_COUNT_LAUNCH();
  }
  if ((what & 2) && ctx.nb > 0) {
    int trans = 0;
    const double* Mb = beta_matrix(ctx, trans);
    const int NB = beta_strings(ctx);
    k_crt_norms<<<NB, 256, 0, st>>>(Mb, NB, ctx.sp[1].count, trans, d + 4); ISCSI_COUNT_LAUNCH();
  }
  ISCSI_CUDA(cudaGetLastError());
  double h[6];
  ISCSI_CUDA(cudaMemcpyAsync(h, S.norms.p, sizeof(h), cudaMemcpyDeviceToHost, st));
  ISCSI_CUDA(cudaStreamSynchronize(st));
  if (what & 1) {
    S.rg = h[0];
    S.gmax = h[1];
    S.g_norm = true;
  }
  rm = h[2] + h[4];
  mmax = std::max(h[3], h[5]);
  if (h[3] != h[3] || h[5] != h[5]) mmax = h[3] + h[5];
  return kOk;
}

// bound of |sigma_I| over max |c| from the norms (with the sums' own rounding)
static double sigma_bound(const Context& ctx, const CrtState& S, int parts, double rm) {
  return 1.000001 * (((parts & 1) ? (double)ctx.na * ctx.nb * S.rg : 0.0) + ((parts & 2) ? rm : 0.0));
}

// moduli, sh and the coefficients' bits for a bound of |sigma| / max|c|, the largest unit maxel and the
// unit whose bits count
static void choose_scale(double bound, double maxel, double ref, int& nm, int& sh, int& cbits) {
  if (bound <= 0.0) bound = 1.0;
  if (maxel <= 0.0) maxel = 1.0;
  if (ref <= 0.0) ref = maxel;
  const int cap = kCrtIntBits - 1 - (int)std::floor(std::log2(maxel));
  for (nm = 10; nm <= kCrtMaxMods; ++nm) {
    // 2^(sh + bc) bound < M / 2, a hundredth of a bit apart (the roundings of the integers)
    const double room = crt_log2_product(nm) - 1.01 - std::log2(bound);
    sh = std::min(cap, (int)std::floor(room - kCrtCBits));
    if (nm < kCrtMaxMods && sh < cap && room - kCrtCBits + std::log2(ref) < kCrtUnitBits) continue;
    sh = std::min(sh, (int)std::ceil(kCrtUnitBitsMax - std::log2(ref)));
    cbits = std::min(kCrtCBitsMax, (int)std::floor(room - sh));
    return;
  }
}

// string matrices' residues
static int crt_cut_m(Context& ctx) {
  CrtState& S = *ctx.crt;
  cudaStream_t st = stream();
  const int NA = alpha_strings(ctx), NB = beta_strings(ctx);
  const int ntile = tile_cols(NB), bt = ntile / 2, tn = (NB + ntile - 1) / ntile;
  const int ka = up(NA, CRT_BK) / CRT_BK, kb = up(NB, CRT_BK) / CRT_BK;
  if (ctx.na > 0 && ctx.M64[0].p) {
    const int rp = up(NA, 2 * CRT_BM);
    const size_t bytes = sizeof(__nv_bfloat16) * (size_t)S.mods.nm * rp * ka * CRT_BK;
    if (S.ma_res.bytes < bytes) ISCSI_TRY(crt_alloc(S.ma_res, bytes, S.held));
    ISCSI_TRY(cut_matrix(ctx.M64[0].as<double>(), NA, NA, ctx.sp[0].count, 0, nullptr, S.sh, CRT_BM, rp, ka, S.unit_mods,
                         S.ma_res.as<__nv_bfloat16>(), st));
  }
  if (ctx.nb > 0) {
    int trans = 0;
    const double* Mb = beta_matrix(ctx, trans);
    const int rp = tn * ntile;
    const size_t bytes = sizeof(__nv_bfloat16) * (size_t)S.mods.nm * rp * kb * CRT_BK;
    if (S.mb_res.bytes < bytes) ISCSI_TRY(crt_alloc(S.mb_res, bytes, S.held));
    ISCSI_TRY(cut_matrix(Mb, NB, NB, ctx.sp[1].count, trans, nullptr, S.sh, bt, rp, kb, S.unit_mods,
                         S.mb_res.as<__nv_bfloat16>(), st));
  }
  S.m_cut[0] = S.mods.nm;
  S.m_cut[1] = S.sh;
  return kOk;
}

// the string matrices changed in place (a per-step one-body term): cut them again,
// on the same scale while their bound still fits it, else everything anew
int crt_matrices_changed(Context& ctx) {
  if (!ctx.crt || ctx.crt->nvec < 0 || !(ctx.crt->parts & 2)) {
    if (ctx.crt) ctx.crt->m_cut[0] = -1;
    return kOk;
  }
  CrtState& S = *ctx.crt;
  double rm = 0.0, mmax = 0.0;
  ISCSI_TRY(take_norms(ctx, 2, rm, mmax));
  const double b = sigma_bound(ctx, S, S.parts, rm);
  if (!(b <= S.bound) || !(std::log2(std::max(mmax, 1e-300)) + S.sh < kCrtIntBits - 1.0)) {
    crt_invalidate(ctx);
    S.m_cut[0] = -1;
    return kOk;
  }
  return crt_cut_m(ctx);
}

// buffers, products and schedule for nvec vectors and the given parts
static int crt_build(Context& ctx, int nvec, int parts) {
  CrtState& S = *ctx.crt;
  cudaStream_t st = stream();
  const SpinSpace &SA = ctx.sp[0], &SB = ctx.sp[1];
  const int NA = alpha_strings(ctx), NB = beta_strings(ctx), n = ctx.n;
  // scale: 1.25 times the bound of today's string matrices, so that a small per-step one-body term keeps it
  {
    double rm = 0.0, mmax = 0.0;
    ISCSI_TRY(take_norms(ctx, ((parts & 1) && !S.g_norm ? 1 : 0) | (parts & 2), rm, mmax));
    const double b = sigma_bound(ctx, S, parts, 1.25 * rm);
    const double maxel = std::max((parts & 1) ? S.gmax : 0.0, (parts & 2) ? 1.25 * mmax : 0.0);
    if (!std::isfinite(b) || !std::isfinite(maxel) || b > 1e200 || (b > 0.0 && b < 1e-200)) {
      S.off = true;
      return kErrNoMem;  // the caller takes the slices
    }
    int nm = 0;
    choose_scale(b, maxel, (parts & 1) ? S.gmax : mmax, nm, S.sh, S.cbits);
    S.bound = b;
    S.mods = crt_make_mods(nm);
    S.unit_mods = crt_make_mods(nm, 5);
  }
  const int nm = S.mods.nm;
  S.job.probs.clear();
  CrtOperands& O = S.ops;
  CrtFold& F = S.fold;
  std::memset(&O, 0, sizeof(O));
  std::memset(&F, 0, sizeof(F));
  const size_t per_vec = 4 * sizeof(int) + kCrtBad * sizeof(long long);
  if (S.cfield.bytes < per_vec * nvec) ISCSI_TRY(S.cfield.grow(per_vec * nvec));
  ISCSI_CUDA(cudaMemsetAsync(S.cfield.p, 0, S.cfield.bytes, st));
  O.nvec = F.nvec = nvec;
  O.n = F.n = n;
  O.bad.det = S.cfield.as<long long>();
  O.cmax = F.cmax = reinterpret_cast<int*>(O.bad.det + (size_t)nvec * kCrtBad);
  O.cexp = F.cexp = O.cmax + nvec;
  O.bad.count = O.cmax + 2 * (size_t)nvec;
  O.bad.count_now = O.cmax + 3 * (size_t)nvec;
  F.bad = O.bad;
  O.nholeA = SA.nhole;
  O.nholeB = F.nholeB = SB.nhole;
  O.off = F.off = ctx.off.as<long long>();
  O.alevel = F.alevel = SA.level.as<int8_t>();
  O.nballow = F.nballow = ctx.nballow.as<int>();
  O.ndet = F.ndet = ctx.ndet;
  F.parts = parts;
  F.nm = nm;
  F.na = ctx.na;
  F.nb = ctx.nb;
  F.na_strings = SA.count;
  F.decA = SA.dec.as<int>();
  F.decB = SB.dec.as<int>();
  F.kmax = ctx.kmax;
  F.ni = F.nbuf = 1;
  F.ebias = -S.cbits - S.sh;
  O.cbits = S.cbits;
  size_t out_elems = 0;
  std::vector<size_t> out_off;
  auto add_out = [&](const CrtProblem& P) {
    out_off.push_back(out_elems);
    out_elems += (size_t)P.rt * P.tn * P.nm * CRT_BM * P.ntile;
  };
  S.ops_smem = 0;
  if (parts & 1) {
    const int np = ctx.npairs, gk = up(np, CRT_BK) / CRT_BK, rp = up(np, 2 * CRT_BM);
    if (!S.pair.p) {
      // orders (see the top of the file)
      std::vector<int> idx(np), pair, map;
      ISCSI_CUDA(cudaMemcpy(idx.data(), ctx.pair_index.p, sizeof(int) * np, cudaMemcpyDeviceToHost));
      const int rr = S.flat ? 1 : 2, noa = SA.nocc, nob = SB.nocc;
      std::vector<int> rowrun((size_t)n * rr, 0);
      for (int lvl = 0; lvl < (S.flat ? 1 : 3); ++lvl)
        for (int p = 0; p < n; ++p)
          for (int r = 0; r < n; ++r) {
            if (!S.flat && (p >= noa) + (r >= nob) != lvl) continue;
            if (r == 0 || (!S.flat && r == nob)) rowrun[(size_t)p * rr + (!S.flat && r >= nob ? 1 : 0)] = (int)pair.size();
            pair.push_back((p << 16) | r);
            map.push_back(idx[p * n + r]);
          }
      pair.resize((size_t)gk * CRT_BK, 0);
      const int yr = (int)S.ystart.size() - 1;
      std::vector<int2> colrun((size_t)SA.nhole * yr, make_int2(0, 0));
      if (S.flat) {
        for (int X = 0; X < SA.nhole; ++X) colrun[X] = make_int2(0, X * SB.nhole);
      } else {
        std::vector<int> at(ctx.cls.size(), 0), gr(ctx.cls.size(), -1);
        for (int c = 0; c < (int)ctx.cls.size(); ++c)
          for (int g = 0; g < (int)S.groups.size(); ++g)
            if (ctx.hp_class_start[c] >= S.groups[g].hp_start &&
                ctx.hp_class_start[c] < S.groups[g].hp_start + S.groups[g].ncol && ctx.cls[c].ncol > 0) {
              gr[c] = g;
              at[c] = ctx.hp_class_start[c] - S.groups[g].hp_start;
            }
        for (int X = 0; X < SA.nhole; ++X)
          for (int y = 0; y < yr; ++y) {
            const int c = SA.hole_level[X] + y;
            if (c < (int)gr.size() && gr[c] >= 0) {
              colrun[(size_t)X * yr + y] = make_int2(gr[c], at[c]);
              at[c] += S.ystart[y + 1] - S.ystart[y];
            }
          }
      }
      std::vector<int> ypos(SB.nhole);
      for (int y = 0; y < yr; ++y)
        for (int Y = S.ystart[y]; Y < S.ystart[y + 1]; ++Y) ypos[Y] = (y << 24) | (S.ypad[y] + Y - S.ystart[y]);
      ISCSI_TRY(S.ypos.alloc(sizeof(int) * SB.nhole));
      ISCSI_CUDA(cudaMemcpy(S.ypos.p, ypos.data(), sizeof(int) * SB.nhole, cudaMemcpyHostToDevice));
      ISCSI_TRY(S.map.alloc(sizeof(int) * np));
      ISCSI_TRY(S.rowrun.alloc(sizeof(int) * rowrun.size()));
      ISCSI_TRY(S.colrun.alloc(sizeof(int2) * colrun.size()));
      ISCSI_TRY(S.pair.alloc(sizeof(int) * pair.size()));
      ISCSI_CUDA(cudaMemcpy(S.map.p, map.data(), sizeof(int) * np, cudaMemcpyHostToDevice));
      ISCSI_CUDA(cudaMemcpy(S.rowrun.p, rowrun.data(), sizeof(int) * rowrun.size(), cudaMemcpyHostToDevice));
      ISCSI_CUDA(cudaMemcpy(S.colrun.p, colrun.data(), sizeof(int2) * colrun.size(), cudaMemcpyHostToDevice));
      ISCSI_CUDA(cudaMemcpy(S.pair.p, pair.data(), sizeof(int) * pair.size(), cudaMemcpyHostToDevice));
    }
    const size_t gbytes = sizeof(__nv_bfloat16) * (size_t)nm * rp * gk * CRT_BK;
    if (S.g_res.bytes < gbytes) {
      ISCSI_TRY(crt_alloc(S.g_res, gbytes, S.held));
      S.g_cut[0] = -1;
    }
    if (S.g_cut[0] != nm || S.g_cut[1] != S.sh) {
      ISCSI_TRY(cut_matrix(ctx.G64.as<double>(), np, np, np, 0, S.map.as<int>(), S.sh, CRT_BM, rp, gk, S.unit_mods,
                           S.g_res.as<__nv_bfloat16>(), st));
      S.g_cut[0] = nm;
      S.g_cut[1] = S.sh;
    }
    size_t elems = 0;
    int cpb = 1;
    for (const CrtGroup& g : S.groups) {
      CrtLiftGroup L;
      L.hp_start = g.hp_start;
      L.ncol = g.ncol;
      L.krows = g.rows;
      L.nkb = up(g.rows, CRT_BK) / CRT_BK;
      const int N = g.ncol * nvec, ntile = tile_cols(N), tn = (N + ntile - 1) / ntile;
      L.bt = ntile / 2;
      // 8-wide chunks of the column, at least a lane's worth per warp
      L.wpc = L.nkb >= 32 ? 8 : L.nkb >= 16 ? 4 : L.nkb >= 8 ? 2 : 1;
      cpb = std::max(cpb, 8 / L.wpc);
      L.base = (long long)elems;
      L.mod_stride = (long long)tn * ntile * L.nkb * CRT_BK;
      elems += (size_t)nm * L.mod_stride;
      const int gi = O.ngroups++;
      O.g[gi] = L;
      O.blk_start[gi + 1] = O.blk_start[gi] + (N + 8 / L.wpc - 1) / (8 / L.wpc);
    }
    S.ops_smem = crt_lift_col_bytes(n) * cpb;
    if (S.b_res.bytes < sizeof(__nv_bfloat16) * elems) ISCSI_TRY(crt_alloc(S.b_res, sizeof(__nv_bfloat16) * elems, S.held));
    // the padding rows of every group stay zero from here on
    ISCSI_CUDA(cudaMemsetAsync(S.b_res.p, 0, S.b_res.bytes, st));
    O.lift = S.b_res.as<__nv_bfloat16>();
    O.pair = S.pair.as<int>();
    O.hp_inv = S.flat ? nullptr : ctx.hp_inv.as<int>();
    O.liftA = SA.lift.as<int>();
    O.liftB = SB.lift.as<int>();
    for (int gi = 0; gi < O.ngroups; ++gi) {
      const CrtLiftGroup& L = O.g[gi];
      CrtHostProblem H;
      std::memset(&H.p, 0, sizeof(H.p));
      H.p.ntile = 2 * L.bt;
      H.p.tn = (L.ncol * nvec + H.p.ntile - 1) / H.p.ntile;
      H.p.nm = nm;
      H.p.rt = up(L.krows, CRT_BM) / CRT_BM;
      H.p.nblk_a = rp / CRT_BM;
      H.p.nkb_a = gk;
      H.p.nblk_b = 2 * H.p.tn;
      H.p.nkb_b = L.nkb;
      H.mt = (H.p.rt + 1) / 2;
      const int nkb = L.nkb;
      H.range = [nkb](int, int, int& k0, int& k1) {
        k0 = 0;
        k1 = nkb;
        return true;
      };
      ISCSI_TRY(crt_encode(H.p, S.g_res.p, S.b_res.as<__nv_bfloat16>() + L.base, nm));
      F.g[gi].res = (long long)out_elems;
      F.g[gi].ncol = L.ncol;
      F.g[gi].ntile = H.p.ntile;
      F.g[gi].tn = H.p.tn;
      add_out(H.p);
      S.job.probs.push_back(H);
    }
    F.rruns = S.flat ? 1 : 2;
    F.rsplit = S.flat ? n : SB.nocc;
    F.yruns = (int)S.ystart.size() - 1;
    for (int y = 0; y <= F.yruns; ++y) F.ystart[y] = S.ystart[y];
    F.rowrun = S.rowrun.as<int>();
    F.colrun = S.colrun.as<int2>();
    F.xlev = S.flat ? 0 : 1;
    F.ypos = S.ypos.as<int>();
    for (int y = 0; y < F.yruns; ++y) F.ypad[y] = S.ypad[y];
  }
  S.ops_blocks = O.blk_start[O.ngroups];
  if (parts & 2) {
    const int ntile = tile_cols(NB), tn = (NB + ntile - 1) / ntile;
    const int ka = up(NA, CRT_BK) / CRT_BK, kb = up(NB, CRT_BK) / CRT_BK, rp = up(NA, 2 * CRT_BM);
    const bool al = ctx.na > 0 && ctx.M64[0].p, be = ctx.nb > 0;
    if (S.m_cut[0] != nm || S.m_cut[1] != S.sh) ISCSI_TRY(crt_cut_m(ctx));
    O.ct_mod = (long long)tn * ntile * ka * CRT_BK;
    O.ca_mod = (long long)rp * kb * CRT_BK;
    O.ct_vec = O.ct_mod * nm;
    O.ca_vec = O.ca_mod * nm;
    O.nkb_ct = ka;
    O.nkb_ca = kb;
    O.bt = ntile / 2;
    O.na = NA;
    O.nb = NB;
    O.ctx_x = (NB + 63) / 64;
    O.ctx_y = (NA + 63) / 64;
    const size_t ctb = sizeof(__nv_bfloat16) * (size_t)O.ct_vec * nvec, cab = sizeof(__nv_bfloat16) * (size_t)O.ca_vec * nvec;
    if (al && S.ct_res.bytes < ctb) ISCSI_TRY(crt_alloc(S.ct_res, ctb, S.held));
    if (be && S.ca_res.bytes < cab) ISCSI_TRY(crt_alloc(S.ca_res, cab, S.held));
    // elements outside the space (and padding) stay zero from here on
    if (al) ISCSI_CUDA(cudaMemsetAsync(S.ct_res.p, 0, S.ct_res.bytes, st));
    if (be) ISCSI_CUDA(cudaMemsetAsync(S.ca_res.p, 0, S.ca_res.bytes, st));
    if (al) O.ct = S.ct_res.as<__nv_bfloat16>();
    if (be) O.ca = S.ca_res.as<__nv_bfloat16>();
    S.ops_blocks += O.ctx_x * O.ctx_y * nvec;
    S.ops_smem = std::max(S.ops_smem, 64 * 65 * (int)sizeof(double));
    const std::vector<int> ls = SA.level_start;
    const std::vector<long long> nba = ctx.nb_allowed_lvl;
    const int maxl = SA.maxlevel;
    auto level_of = [ls, maxl](int A) {
      int l = 0;
      while (l < maxl && ls[l + 1] <= A) ++l;
      return l;
    };
    F.ss_res = (long long)out_elems;
    F.ss_ntile = ntile;
    F.ss_tn = tn;
    for (int v = 0; v < nvec; ++v) {
      bool first = true;
      for (int part = 0; part < 2; ++part) {
        if (part == 0 ? !al : !be) continue;
        CrtHostProblem H;
        std::memset(&H.p, 0, sizeof(H.p));
        H.p.ntile = ntile;
        H.p.tn = tn;
        H.p.nm = nm;
        H.p.rt = up(NA, CRT_BM) / CRT_BM;
        H.p.nblk_a = rp / CRT_BM;
        H.p.nkb_a = part == 0 ? ka : kb;
        H.p.nblk_b = 2 * tn;
        H.p.nkb_b = H.p.nkb_a;
        H.mt = rp / (2 * CRT_BM);
        if (part == 0) {
          // alpha strings with an allowed prefix beyond the tile's first column, within two
          // levels of the tile's rows
          H.range = [=](int mt, int nt, int& k0, int& k1) {
            const int lo = level_of(mt * 256), hi = level_of(std::min(mt * 256 + 255, NA - 1));
            if (nba[lo] <= (long long)nt * ntile) return false;
            int l1 = 0;  // levels with columns in this tile
            while (l1 <= maxl && nba[l1] > (long long)nt * ntile) ++l1;
            l1 = std::min(l1, hi + 3);
            const int l0 = std::max(0, lo - 2);
            k0 = ls[l0] / CRT_BK;
            k1 = (ls[std::min(l1, maxl + 1)] + CRT_BK - 1) / CRT_BK;
            return true;
          };
          ISCSI_TRY(crt_encode(H.p, S.ma_res.p, S.ct_res.as<__nv_bfloat16>() + O.ct_vec * v, nm));
          if (be) H.second = 1;
        } else {
          // the allowed beta prefix of the tile's first (lowest) level
          H.range = [=](int mt, int nt, int& k0, int& k1) {
            const int lo = level_of(mt * 256);
            if (nba[lo] <= (long long)nt * ntile) return false;
            k0 = 0;
            k1 = (int)((nba[lo] + CRT_BK - 1) / CRT_BK);
            return true;
          };
          ISCSI_TRY(crt_encode(H.p, S.ca_res.as<__nv_bfloat16>() + O.ca_vec * v, S.mb_res.p, nm));
        }
        if (first) {
          if (v == 1) F.ss_vec = (long long)out_elems - F.ss_res;
          add_out(H.p);
        } else {
          H.own = false;
          out_off.push_back(0);
        }
        first = false;
        S.job.probs.push_back(H);
      }
    }
  }
  if (out_elems >> 35) return kErrNoMem;  // k_crt_fold addresses 16-byte units of it with 32 bits
  if (S.out.bytes < sizeof(int16_t) * out_elems) ISCSI_TRY(crt_alloc(S.out, sizeof(int16_t) * out_elems, S.held));
  for (size_t i = 0; i < S.job.probs.size(); ++i) S.job.probs[i].p.res = S.out.as<int16_t>() + out_off[i];
  F.res = S.out.as<int16_t>();
  // the fold's launches: levels of alpha strings with their own staged shape (fewer than 64 strings
  // join the next level); a block covers its row in one pass, or a quarter of a few much longer rows
  S.folds.clear();
  for (int l = 0; l <= SA.maxlevel;) {
    const int l0 = l;
    while (l < SA.maxlevel && (S.flat || SA.level_start[l + 1] - SA.level_start[l0] < 64)) ++l;
    ++l;
    const int r0 = SA.level_start[l0], r1 = SA.level_start[l];
    if (r1 <= r0 || ctx.nb_allowed_lvl[l0] <= 0) continue;
    CrtFoldLaunch L;
    L.f = F;
    L.f.row0 = r0;
    L.rows = r1 - r0;
    L.smem = 0;
    int ni = ctx.na, passes = 1;
    if (parts & 1) {
      const FoldShape fs = fold_shape(ctx, S, S.flat ? 0 : l0);
      L.f.ni = ni = fs.ni;
      L.f.nbuf = fs.nbuf;
      L.f.stride = fs.stride;
      L.f.stride1 = fs.stride1;
      L.f.base1 = fs.base1;
      L.f.hole_elems = fs.hole;
      L.f.stage_bytes = fs.ni * fs.hole * 2;
      L.smem = fs.smem;
      passes = (ctx.na + ni - 1) / ni;
    }
    L.w = crt_make_weights(nm, ((parts & 1) ? ni * ctx.nb : 0) + 1, ni * ctx.nb, passes - 1);
    int lim = (int)ctx.nb_allowed_lvl[l0], most = (int)ctx.nb_allowed_lvl[l - 1];
    L.threads = std::min(kFoldThreads, std::max(64, up((std::max(most, (lim + 3) / 4) + kFoldPer - 1) / kFoldPer, 32)));
    L.blocks = (lim + L.threads * kFoldPer - 1) / (L.threads * kFoldPer);
    L.threads = std::min(L.threads, up(((lim + L.blocks - 1) / L.blocks + kFoldPer - 1) / kFoldPer, 32));
    S.folds.push_back(L);
  }
  ISCSI_TRY(S.job.upload(st));
  S.nvec = nvec;
  S.parts = parts;
  ++ctx.crt_version;
  return kOk;
}

static size_t g_crt_held = 0;

void CrtHeld::add(size_t n) {
  bytes += n;
  g_crt_held += n;
}

int crt_alloc(DevBuf& d, size_t bytes, CrtHeld& held) {
  held.add(0 - std::min(held.bytes, d.bytes));
  d.release();
  size_t free_b = 0, total = 0;
  ISCSI_CUDA(cudaMemGetInfo(&free_b, &total));
  if (g_crt_held + bytes > (free_b + g_crt_held) / 2) {
    set_error("residues: less than half of the free memory would be left");
    return kErrNoMem;
  }
  ISCSI_TRY(d.alloc(bytes));
  held.add(bytes);
  return kOk;
}

bool crt_drop(Context& ctx) {
  if (!ctx.crt || ctx.crt->held.bytes == 0) return false;
  const int most = ctx.crt->max_vecs;
  crt_release(ctx);
  crt_state(ctx).max_vecs = most;
  return true;
}

// Operands of this call's vectors (building buffers and work list when they
// changed).  parts: 1 opposite spin, 2 same spin.  kErrNoMem leaves blocks of this
// many vectors and more without residues (the caller takes the slices instead).
int crt_operands(Context& ctx, const double* c, int nvec, int parts) {
  CrtState& S = crt_state(ctx);
  cudaStream_t st = stream();
  if (!ctx.oz_err.p) {
    ISCSI_TRY(ctx.oz_err.alloc(sizeof(int)));
    ISCSI_CUDA(cudaMemsetAsync(ctx.oz_err.p, 0, sizeof(int), st));
  }
  if (S.nvec != nvec || S.parts != parts) {
    S.nvec = -1;
    const int rc = crt_build(ctx, nvec, parts);
    if (rc == kErrNoMem) {
      // blocks of fewer vectors may still fit
      const bool off = S.off;
      cudaStreamSynchronize(st);
      crt_release(ctx);
      crt_state(ctx).off = off;
      crt_state(ctx).max_vecs = nvec - 1;
      cudaGetLastError();
    }
    ISCSI_TRY(rc);
  }
  const int vb = (int)std::min<long long>(2 * tc_sm_count(), (ctx.ndet + 1023) / 1024);
  k_crt_cmax<<<dim3(vb, nvec), 256, 0, st>>>(c, ctx.ndet, S.ops.cmax, S.ops.bad); ISCSI_COUNT_LAUNCH();
  k_crt_operands<<<S.ops_blocks, 256, S.ops_smem, st>>>(S.ops, S.mods, c); ISCSI_COUNT_LAUNCH();
  ISCSI_CUDA(cudaGetLastError());
  return kOk;
}

int crt_gemm(Context& ctx) { return ctx.crt->job.launch(ctx.oz_err.as<int>(), stream()); }

template <int NB, bool MR>
static int launch_fold(const CrtState& S, double* sigma, cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    ISCSI_CUDA(cudaFuncSetAttribute(k_crt_fold<NB, MR>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldMaxSmem));
    attr = true;
  }
  for (const CrtFoldLaunch& L : S.folds) {
    k_crt_fold<NB, MR><<<dim3(L.rows, L.blocks, S.nvec), L.threads, L.smem, st>>>(L.f, L.w, sigma); ISCSI_COUNT_LAUNCH();
  }
  ISCSI_CUDA(cudaGetLastError());
  return kOk;
}

// sigma (overwritten): the parts that went through residues
int crt_fold(Context& ctx, double* sigma) {
  const CrtState& S = *ctx.crt;
  cudaStream_t st = stream();
  const bool mr = (S.parts & 1) && S.ystart.size() > 2;
  switch (ctx.nb) {
    case 1: return mr ? launch_fold<1, true>(S, sigma, st) : launch_fold<1, false>(S, sigma, st);
    case 2: return mr ? launch_fold<2, true>(S, sigma, st) : launch_fold<2, false>(S, sigma, st);
    case 3: return mr ? launch_fold<3, true>(S, sigma, st) : launch_fold<3, false>(S, sigma, st);
    case 4: return mr ? launch_fold<4, true>(S, sigma, st) : launch_fold<4, false>(S, sigma, st);
    default: return launch_fold<0, true>(S, sigma, st);
  }
}

// several contexts' products on one schedule; rebuilt when one of them was
struct CrtBatch {
  CrtJob job;
  std::vector<std::pair<Context*, long long>> src;
};

int crt_batch_launch(CrtBatch*& b, const std::vector<Context*>& ctxs, int* err, cudaStream_t st) {
  if (ctxs.empty()) return kOk;
  if (!b) b = new CrtBatch();
  std::vector<std::pair<Context*, long long>> src;
  for (Context* c : ctxs) src.push_back({c, c->crt_version});
  if (src != b->src) {
    b->job.probs.clear();
    for (Context* c : ctxs) b->job.probs.insert(b->job.probs.end(), c->crt->job.probs.begin(), c->crt->job.probs.end());
    ISCSI_TRY(b->job.upload(st));
    b->src = src;
  }
  return b->job.launch(err, st);
}

void crt_batch_release(CrtBatch*& b) {
  delete b;
  b = nullptr;
}

void crt_stats(const Context& ctx, double& flops, int& items, int& grid, int& moduli) {
  const bool on = ctx.crt && ctx.crt->nvec > 0;
  flops = on ? ctx.crt->job.flops : 0.0;
  items = on ? ctx.crt->job.nitems : 0;
  grid = on ? ctx.crt->job.grid : 0;
  moduli = on ? ctx.crt->mods.nm : 0;
}

}  // namespace iscsi
