// functions.cu -- products and inner products of functions held on different leaf trees.
//
// Two trees of disjoint leaves are first brought onto their common refinement: each tree's
// leaves plus empty boxes at the other tree's leaf keys are summed down (reconstruct.cuh), which
// gives both functions on the same leaves.  The product then uses the third representation of
// Sec. 2.1: the values at the k Gauss-Legendre points of every box.  With V[q][i] = phi_i(x_q)
// and weights w_q on (0,1), a leaf of width h holds f = h^{-3/2} (V x V x V) s at its points,
// and coefficients come back as s = h^{3/2} (V^T W)^{x3} f, so the product's coefficients are
//     s_ab = h^{-3/2} (V^T W)^{x3} [ (V^{x3} s_a) * (V^{x3} s_b) ],
// the product interpolated at the points.  The inner product is the coefficient dot product
// over the common leaves (the basis is orthonormal).
#include <algorithm>
#include <cmath>
#include <vector>

#include <cub/cub.cuh>

#include "mra_internal.cuh"
#include "reconstruct.cuh"

namespace mra {
namespace {

// c <- alpha c over n * k3 coefficients (grid-stride).
__global__ void scale_kernel(int64_t n, double alpha, double *c) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    c[i] *= alpha;
}

// First position in the sorted keys[0 .. n) that is not below x.
__device__ __forceinline__ int64_t lower_bound(const uint64_t *keys, int64_t n, uint64_t x) {
  int64_t a = 0, b = n;
  while (a < b) {
    const int64_t m = (a + b) / 2;
    if (keys[m] < x) a = m + 1;
    else b = m;
  }
  return a;
}

// flags: 1 the first tree's keys are not strictly increasing, 2 the second's, 4 the keys differ.
__global__ void compare_keys_kernel(int64_t na, const uint64_t *a, int64_t nb, const uint64_t *b, int *flags) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int f = na != nb ? 4 : 0;
  if (i > 0 && i < na && a[i] <= a[i - 1]) f |= 1;
  if (i > 0 && i < nb && b[i] <= b[i - 1]) f |= 2;
  if (i < na && i < nb && a[i] != b[i]) f |= 4;
  f = __reduce_or_sync(0xffffffffu, f);
  if (f && (threadIdx.x & 31) == 0) atomicOr(flags, f);
}

// fresh[j] = 1 for a box of b that a does not have; fresh[nb] = 0 (so that its scan ends with the count).
__global__ void fresh_kernel(int64_t na, const uint64_t *a, int64_t nb, const uint64_t *b, int64_t *fresh) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j > nb) return;
  const int64_t p = j < nb ? lower_bound(a, na, b[j]) : 0;
  fresh[j] = j < nb && !(p < na && a[p] == b[j]);
}

// The boxes of either tree in order, with the row each tree has them at (-1: not there).  before[j]: boxes of
// b[0 .. j) that a does not have.
__global__ void union_kernel(int64_t na, const uint64_t *a, int64_t nb, const uint64_t *b, const int64_t *before,
                             uint64_t *u, int64_t *ra, int64_t *rb) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < na) {
    const int64_t p = lower_bound(b, nb, a[i]), at = i + before[p];
    u[at] = a[i];
    ra[at] = i;
    rb[at] = p < nb && b[p] == a[i] ? p : -1;
  } else if (i < na + nb) {
    const int64_t j = i - na;
    if (before[j + 1] == before[j]) return;
    const int64_t at = before[j] + lower_bound(a, na, b[j]);
    u[at] = b[j];
    ra[at] = -1;
    rb[at] = j;
  }
}

// One CTA per leaf: s_ab = h^{-3/2} (V^T W)^{x3} [(V^{x3} s_a) (V^{x3} s_b)].  VW[q][i] holds
// V[q][i] and VW[k*k + i*k + q] holds w_q V[q][i].  Shared memory: 4 k^3 doubles.
__global__ void product_kernel(int k, double L, int64_t n, const uint64_t *keys, const double *a, const double *b,
                               const double *VW, double *out) {
  extern __shared__ double sh[];
  const int64_t leaf = blockIdx.x;
  if (leaf >= n) return;
  const int k2 = k * k, k3 = k2 * k;
  double *x = sh, *y = x + k3, *t = y + k3, *u = t + k3;
  const double *V = VW, *VtW = VW + k2;
  const double h = 2.0 * L / (double)(1LL << key_level(keys[leaf]));
  // values of a (into x) and of b (into y): three mode products each
  for (int pass = 0; pass < 2; ++pass) {
    const double *src = pass == 0 ? a : b;
    double *dst = pass == 0 ? x : y;
    for (int e = threadIdx.x; e < k3; e += blockDim.x) t[e] = src[leaf * k3 + e];
    __syncthreads();
    for (int e = threadIdx.x; e < k3; e += blockDim.x) {  // u[q][j][l] = sum_i V[q][i] t[i][j][l]
      const int q = e / k2, r = e % k2;
      double v = 0.0;
      for (int i = 0; i < k; ++i) v += V[q * k + i] * t[i * k2 + r];
      u[e] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < k3; e += blockDim.x) {  // t[q][p][l] = sum_j V[p][j] u[q][j][l]
      const int q = e / k2, p = (e / k) % k, l = e % k;
      double v = 0.0;
      for (int j = 0; j < k; ++j) v += V[p * k + j] * u[(q * k + j) * k + l];
      t[e] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < k3; e += blockDim.x) {  // dst[q][p][r] = sum_l V[r][l] t[q][p][l]
      const int qp = e / k, r = e % k;
      double v = 0.0;
      for (int l = 0; l < k; ++l) v += V[r * k + l] * t[qp * k + l];
      dst[e] = v;
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < k3; e += blockDim.x) t[e] = x[e] * y[e];
  __syncthreads();
  for (int e = threadIdx.x; e < k3; e += blockDim.x) {  // back: u[i][p][r] = sum_q VtW[i][q] t[q][p][r]
    const int i = e / k2, r = e % k2;
    double v = 0.0;
    for (int q = 0; q < k; ++q) v += VtW[i * k + q] * t[q * k2 + r];
    u[e] = v;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < k3; e += blockDim.x) {
    const int i = e / k2, j = (e / k) % k, r = e % k;
    double v = 0.0;
    for (int p = 0; p < k; ++p) v += VtW[j * k + p] * u[(i * k + p) * k + r];
    x[e] = v;
  }
  __syncthreads();
  const double scale = 1.0 / (h * sqrt(h));
  for (int e = threadIdx.x; e < k3; e += blockDim.x) {
    const int ij = e / k, l = e % k;
    double v = 0.0;
    for (int r = 0; r < k; ++r) v += VtW[l * k + r] * x[ij * k + r];
    out[leaf * k3 + e] = scale * v;
  }
}

__global__ void dot_rows_kernel(int64_t n, int k3, const double *a, const double *b, double *d) {
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  double s = 0.0;
  for (int e = lane; e < k3; e += 32) s += a[i * k3 + e] * b[i * k3 + e];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) d[i] = s;
}

// Device buffers released on scope exit (stream-ordered).
struct Pool {
  cudaStream_t s;
  std::vector<void *> held;
  explicit Pool(cudaStream_t st) : s(st) {}
  ~Pool() {
    for (void *p : held) cudaFreeAsync(p, s);
    cudaStreamSynchronize(s);
  }
  void *get(size_t bytes) {
    void *p = nullptr;
    if (pool_malloc(&p, bytes ? bytes : 1, s) != cudaSuccess) return nullptr;
    held.push_back(p);
    return p;
  }
};

int check_leaf_view(const mra_tree_view *v, const char *what) {
  if (!v) return fail(MRA_ERR_ARG, "%s: NULL tree", what);
  if (v->n < 0 || (v->n > 0 && (!v->keys || !v->coeffs))) return fail(MRA_ERR_ARG, "%s: bad tree view", what);
  if (v->k < 1 || v->k > MRA_MAX_K) return fail(MRA_ERR_ARG, "%s: k=%d outside 1..%d", what, v->k, MRA_MAX_K);
  return MRA_OK;
}

// Both trees on their common leaves: keys (shared), and each tree's coefficients there.  The common leaves depend
// on the union of the keys alone, so one plan serves both trees and each level is one launch for both.
// What binds it is latency (two sorts, a kernel per level, four host reads).  In an iteration of the bound-state
// solver (7,680 leaves, k = 6) the product takes 0.88 ms and the three inner products 1.37; with the union made on
// the host and each tree summed down by itself they took 1.25 and 2.0.
int align(const mra_tree_view &a, const mra_tree_view &b, Pool &pool, cudaStream_t s, int64_t *n_out,
          uint64_t **keys_out, double **ca, double **cb) {
  const int k3 = a.k * a.k * a.k;
  int *d_flags = (int *)pool.get(3 * sizeof(int));
  if (!d_flags) return fail(MRA_ERR_CUDA, "mra_multiply/inner: out of device memory");
  MRA_CUDA_TRY(cudaMemsetAsync(d_flags, 0, 3 * sizeof(int), s));
  const auto grid = [](int64_t n) { return counted((unsigned)((n + 255) / 256)); };
  compare_keys_kernel<<<grid(std::max(a.n, b.n)), 256, 0, s>>>(a.n, a.keys, b.n, b.keys, d_flags);
  MRA_CUDA_TRY(cudaGetLastError());
  int flags = 0;
  MRA_CUDA_TRY(cudaMemcpyAsync(&flags, d_flags, sizeof(int), cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (flags & 1) return fail(MRA_ERR_ARG, "mra_multiply/inner: first tree's keys not sorted and unique");
  if (flags & 2) return fail(MRA_ERR_ARG, "mra_multiply/inner: second tree's keys not sorted and unique");
  if (!(flags & 4)) {  // already on the same leaves
    *n_out = a.n;
    *keys_out = a.keys;
    *ca = a.coeffs;
    *cb = b.coeffs;
    return MRA_OK;
  }
  const int64_t nab = a.n + b.n;
  size_t tb = 0;
  MRA_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, (int64_t *)nullptr, (int64_t *)nullptr, b.n + 1, s));
  int64_t *fresh = (int64_t *)pool.get((b.n + 1) * 8), *before = (int64_t *)pool.get((b.n + 1) * 8);
  uint64_t *u = (uint64_t *)pool.get(nab * 8);
  int64_t *ra = (int64_t *)pool.get(nab * 8), *rb = (int64_t *)pool.get(nab * 8);
  void *tmp = pool.get(tb);
  if (!fresh || !before || !u || !ra || !rb || !tmp) return fail(MRA_ERR_CUDA, "mra_multiply/inner: out of device memory");
  fresh_kernel<<<grid(b.n + 1), 256, 0, s>>>(a.n, a.keys, b.n, b.keys, fresh);
  MRA_CUDA_TRY(cudaGetLastError());
  MRA_CUDA_TRY(cub::DeviceScan::ExclusiveSum(tmp, tb, fresh, before, b.n + 1, s));
  union_kernel<<<grid(nab), 256, 0, s>>>(a.n, a.keys, b.n, b.keys, before, u, ra, rb);
  MRA_CUDA_TRY(cudaGetLastError());
  int64_t more = 0;
  MRA_CUDA_TRY(cudaMemcpyAsync(&more, before + b.n, 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t nu = a.n + more;
  if (nu >= (1LL << 31)) return fail(MRA_ERR_ARG, "mra_multiply/inner: more than 2^31 boxes");
  Reconstruct rec(s);
  int rc = rec.plan(a.k, nu, u);
  if (rc) return rc;
  const int64_t n = rec.leaves();
  uint64_t *keys = (uint64_t *)pool.get(n * 8);
  if (!keys) return fail(MRA_ERR_CUDA, "mra_multiply/inner: out of device memory");
  if ((rc = rec.place(keys)) != MRA_OK) return rc;
  // a tree whose own leaves are the common leaves (the other's are all at or above them) is used as it is
  int own[2] = {4, 4};
  for (int t = 0; t < 2; ++t) {
    const mra_tree_view &v = t == 0 ? a : b;
    if (v.n != n) continue;
    compare_keys_kernel<<<grid(n), 256, 0, s>>>(n, v.keys, n, keys, d_flags + 1 + t);
    MRA_CUDA_TRY(cudaGetLastError());
    MRA_CUDA_TRY(cudaMemcpyAsync(&own[t], d_flags + 1 + t, sizeof(int), cudaMemcpyDeviceToHost, s));
  }
  if (a.n == n || b.n == n) MRA_CUDA_TRY(cudaStreamSynchronize(s));
  SumDown f[2];
  int nf = 0;
  for (int t = 0; t < 2; ++t) {
    const mra_tree_view &v = t == 0 ? a : b;
    double **c = t == 0 ? ca : cb;
    if (own[t] == 0) {
      *c = v.coeffs;
      continue;
    }
    *c = (double *)pool.get(n * k3 * 8);
    if (!*c) return fail(MRA_ERR_CUDA, "mra_multiply/inner: out of device memory");
    f[nf++] = SumDown{v.coeffs, t == 0 ? ra : rb, *c};
  }
  if (nf > 0 && (rc = rec.run(nf, f)) != MRA_OK) return rc;
  *n_out = n;
  *keys_out = keys;
  return MRA_OK;
}

}  // namespace
}  // namespace mra

using namespace mra;

extern "C" int mra_multiply(const mra_tree_view *a, const mra_tree_view *b, mra_tree_view *out, void *stream) {
  int rc = check_leaf_view(a, "mra_multiply(a)");
  if (rc) return rc;
  rc = check_leaf_view(b, "mra_multiply(b)");
  if (rc) return rc;
  if (!out || out->k != a->k || out->cap < 0 || (out->cap > 0 && (!out->keys || !out->coeffs)))
    return fail(MRA_ERR_ARG, "mra_multiply: bad output view");
  if (b->k != a->k || b->L != a->L) return fail(MRA_ERR_ARG, "mra_multiply: trees of different k or L");
  out->L = a->L;
  if (a->n == 0 || b->n == 0) {
    out->n = 0;
    return MRA_OK;
  }
  cudaStream_t s = (cudaStream_t)stream;
  Pool pool(s);
  int64_t n = 0;
  uint64_t *keys = nullptr;
  double *ca = nullptr, *cb = nullptr;
  rc = align(*a, *b, pool, s, &n, &keys, &ca, &cb);
  if (rc) return rc;
  if (n > out->cap) {
    out->n = n;
    return fail(MRA_ERR_CAPACITY, "mra_multiply: %lld leaves, capacity %lld", (long long)n, (long long)out->cap);
  }
  const int k = a->k, k3 = k * k * k;
  // V[q][i] = phi_i(x_q) and w_q V[q][i] (stored transposed) at the k Gauss-Legendre points on (0,1)
  std::vector<double> gx(k), gw(k), VW(2 * k * k);
  gauss_legendre(k, gx.data(), gw.data());
  for (int q = 0; q < k; ++q) {
    const double xq = 0.5 * (gx[q] + 1.0), wq = 0.5 * gw[q], t = 2.0 * xq - 1.0;
    double p0 = 1.0, p1 = t;
    for (int i = 0; i < k; ++i) {
      double P = i == 0 ? 1.0 : (i == 1 ? t : 0.0);
      if (i >= 2) {
        P = ((2.0 * i - 1.0) * t * p1 - (i - 1.0) * p0) / i;
        p0 = p1;
        p1 = P;
      }
      const double phi = sqrt(2.0 * i + 1.0) * P;
      VW[q * k + i] = phi;
      VW[k * k + i * k + q] = wq * phi;
    }
  }
  double *dVW = (double *)pool.get(VW.size() * 8);
  if (!dVW) return fail(MRA_ERR_CUDA, "mra_multiply: out of device memory");
  MRA_CUDA_TRY(cudaMemcpyAsync(dVW, VW.data(), VW.size() * 8, cudaMemcpyHostToDevice, s));
  MRA_CUDA_TRY(cudaFuncSetAttribute(product_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(4 * k3 * sizeof(double))));
  product_kernel<<<counted((unsigned)n), 128, 4 * k3 * sizeof(double), s>>>(k, a->L, n, keys, ca, cb, dVW, out->coeffs);
  MRA_CUDA_TRY(cudaGetLastError());
  MRA_CUDA_TRY(cudaMemcpyAsync(out->keys, keys, (size_t)n * 8, cudaMemcpyDeviceToDevice, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  out->n = n;
  return MRA_OK;
}

extern "C" int mra_inner(const mra_tree_view *a, const mra_tree_view *b, double *result, void *stream) {
  int rc = check_leaf_view(a, "mra_inner(a)");
  if (rc) return rc;
  rc = check_leaf_view(b, "mra_inner(b)");
  if (rc) return rc;
  if (!result) return fail(MRA_ERR_ARG, "mra_inner: NULL result");
  if (b->k != a->k || b->L != a->L) return fail(MRA_ERR_ARG, "mra_inner: trees of different k or L");
  *result = 0.0;
  if (a->n == 0 || b->n == 0) return MRA_OK;
  cudaStream_t s = (cudaStream_t)stream;
  Pool pool(s);
  int64_t n = 0;
  uint64_t *keys = nullptr;
  double *ca = nullptr, *cb = nullptr;
  rc = align(*a, *b, pool, s, &n, &keys, &ca, &cb);
  if (rc) return rc;
  const int k3 = a->k * a->k * a->k;
  double *d = (double *)pool.get(n * 8), *sum = (double *)pool.get(8);
  if (!d || !sum) return fail(MRA_ERR_CUDA, "mra_inner: out of device memory");
  dot_rows_kernel<<<counted((unsigned)((n + 7) / 8)), 256, 0, s>>>(n, k3, ca, cb, d);
  MRA_CUDA_TRY(cudaGetLastError());
  size_t tb = 0;
  MRA_CUDA_TRY(cub::DeviceReduce::Sum(nullptr, tb, d, sum, (int)n, s));
  void *tmp = pool.get(tb);
  if (!tmp) return fail(MRA_ERR_CUDA, "mra_inner: out of device memory");
  MRA_CUDA_TRY(cub::DeviceReduce::Sum(tmp, tb, d, sum, (int)n, s));
  MRA_CUDA_TRY(cudaMemcpyAsync(result, sum, 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  return MRA_OK;
}

extern "C" int mra_scale(mra_tree_view *t, double alpha, void *stream) {
  if (!t) return fail(MRA_ERR_ARG, "mra_scale: NULL tree view");
  if (t->n < 0 || t->n > t->cap) return fail(MRA_ERR_ARG, "mra_scale: bad n/cap");
  if (t->k < 1 || t->k > MRA_MAX_NS_K) return fail(MRA_ERR_ARG, "mra_scale: k=%d invalid", t->k);
  if (!std::isfinite(alpha)) return fail(MRA_ERR_ARG, "mra_scale: alpha is not finite");
  if (t->n == 0) return MRA_OK;
  if (!t->coeffs) return fail(MRA_ERR_ARG, "mra_scale: NULL coefficients");
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t n = t->n * (int64_t)t->k * t->k * t->k;
  const unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16);
  scale_kernel<<<counted(grid), 256, 0, s>>>(n, alpha, t->coeffs);
  MRA_CUDA_TRY(cudaGetLastError());
  return MRA_OK;
}
