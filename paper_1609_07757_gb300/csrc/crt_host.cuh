// crt_host.cuh -- host side of the residue-number contraction shared by its
// users (crt.cu, density.cu): products, work list, constants.
#pragma once
#include <functional>
#include <vector>

#include "crt_types.cuh"
#include "internal.cuh"

namespace iscsi {

constexpr int kCrtResMax = 257;   // |residue| as k_crt_gemm stores it

// host description of a product: which tiles it has and their k blocks
struct CrtHostProblem {
  CrtProblem p;
  int mt;                          // pairs of row blocks
  std::function<bool(int, int, int&, int&)> range;  // tile (mt, nt) -> its k blocks; false: no tile
  int second = -1;                 // product added into the same tiles (relative index), its k blocks by its own range
  bool own = true;                 // false: only as another's second product
};

// a list of products on the device with its schedule (one context's, or several merged)
struct CrtJob {
  std::vector<CrtHostProblem> probs;
  DevBuf d_probs, d_items, d_start;
  int grid = 0, nitems = 0;
  double flops = 0.0;
  int upload(cudaStream_t st);
  int launch(int* err, cudaStream_t st) const;
};

// constants of the first nm moduli for integers in four or five limbs; weights of the reconstruction from sums of `terms`
// stored residues (later passes: terms_next each); log2 of the moduli's product
CrtMods crt_make_mods(int nm, int limbs = 4);
CrtWeights crt_make_weights(int nm, int terms, int terms_next = 0, int passes_next = 0);
double crt_log2_product(int nm);
// Bytes of residue buffers of one user, counted for the process as well.
struct CrtHeld {
  size_t bytes = 0;
  CrtHeld() = default;
  CrtHeld(const CrtHeld&) = delete;
  CrtHeld& operator=(const CrtHeld&) = delete;
  ~CrtHeld() { add(0 - bytes); }
  void add(size_t n);  // (modulo 2^64: also takes back)
};
// A residue buffer: the residues take a few times the memory of the slices, and are taken only while
// all of the process's stay below half of what the device would have free without them, so that a
// program's own vectors and other contexts find the room they found with the slices.  kErrNoMem otherwise.
int crt_alloc(DevBuf& d, size_t bytes, CrtHeld& held);
// tensor maps of a product's operands
int crt_encode(CrtProblem& P, const void* a, const void* b, int nm);

}  // namespace iscsi
