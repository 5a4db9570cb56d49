// reconstruct.cuh -- summing boxes of any levels down to leaves, in two parts: the leaves' tree, which depends on
// the keys alone, and the coefficients, for one function or for two held on the same boxes.
#pragma once

#include <vector>

#include "mra_internal.cuh"

namespace mra {

// One function on the input boxes: box b has the coefficients at row[b] (none where row[b] < 0), row b when
// row is null; the leaves' coefficients go to out.
struct SumDown {
  const double *coeffs = nullptr;
  const int64_t *row = nullptr;
  double *out = nullptr;
};

class Reconstruct {
 public:
  explicit Reconstruct(cudaStream_t stream) : s(stream) {}
  ~Reconstruct();
  // The result's tree from n >= 1 sorted, unique keys (checked); leaves() is known afterwards.
  int plan(int k, int64_t n, const uint64_t *keys);
  int64_t leaves() const { return nout; }
  // The leaves' keys in order (leaves() of them).
  int place(uint64_t *out_keys);
  // The coefficients of one or two functions, one launch per level for both.
  int run(int nf, const SumDown *f);

 private:
  cudaStream_t s;
  std::vector<void *> held;
  int k = 0, nmin = 0, nmax = 0;
  int64_t n_in = 0, ni = 0, nout = 0, info[24] = {};
  const uint64_t *keys = nullptr, *ik = nullptr;
  int *top = nullptr;
  double *Ub = nullptr;
  int64_t *dst = nullptr, *own = nullptr, *iown = nullptr;
  unsigned char *start = nullptr;
  void *dalloc(size_t bytes);
  void drop(void *p);
};

}  // namespace mra
