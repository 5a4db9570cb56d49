// twoscale.cuh -- the two-scale transforms of one box by one CTA (Sec. 2.2), FP64.
//
// U[i][j] is U^{(0)} (k x k).  phi_j has degree j, so U[i][j] = 0 for i > j, and reflection gives
// U^{(1)}[i][j] = (-1)^{i+j} U[i][j].  Down (parent to children), one dimension: with
// e_i = sum_{j >= i, j - i even} U[i][j] d_j and o_i = sum_{j > i, j - i odd} U[i][j] d_j the children get e_i + o_i
// and e_i - o_i.  Up (children to parent): s_j = sum_{i <= j, j - i even} U[i][j] (S0_i + S1_i) +
// sum_{i < j, j - i odd} U[i][j] (S0_i - S1_i).  A quarter of the products of the full (2k) x k matrix; the
// FP64 pipe binds these transforms (a 3-D transform of a box took 14 k^4 FMAs, now about 3.5 k^4).  Sum-down and
// truncation of 16,166 boxes at k = 10, with the trees made from the keys beforehand: 7.06 -> 2.33 ms.
#pragma once

namespace mra {
namespace twoscale {

// Row i of U times a vector of stride st, even and odd parts.
__device__ __forceinline__ void even_odd(int k, int i, const double *U, const double *v, int st, double &e, double &o) {
  e = o = 0.0;
  const double *u = U + i * k;
  int j = i;
  for (; j + 1 < k; j += 2) {
    e = fma(u[j], v[j * st], e);
    o = fma(u[j + 1], v[(j + 1) * st], o);
  }
  if (j < k) e = fma(u[j], v[j * st], e);
}

// Children of the k^3 tensor d: emit(I, J, L, value) for every element of the (2k)^3 tensor (I = c k + i ...).
// U, d, a (2 k^3 doubles), b (4 k^3 doubles) in shared memory, a and b distinct from d; d is complete (the
// caller has synchronised); emit runs without a barrier after it.
template <class Emit>
__device__ __forceinline__ void down(int k, const double *U, const double *d, double *a, double *b, Emit emit) {
  const int kk = 2 * k, k2 = k * k;
  for (int q = threadIdx.x; q < k * k2; q += blockDim.x) {  // a[I][j][l]
    const int i = q / k2, r = q - i * k2;
    double e, o;
    even_odd(k, i, U, d + r, k2, e, o);
    a[i * k2 + r] = e + o;
    a[(k + i) * k2 + r] = e - o;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < k * kk * k; q += blockDim.x) {  // b[I][J][l]
    const int i = q / (kk * k), r = q - i * kk * k, I = r / k, l = r - I * k;
    double e, o;
    even_odd(k, i, U, a + I * k2 + l, k, e, o);
    b[(I * kk + i) * k + l] = e + o;
    b[(I * kk + k + i) * k + l] = e - o;
  }
  __syncthreads();
  // the last dimension: rows i and k-1-i by one thread, k+1 products for every lane of a warp
  const int h = (k + 1) / 2;
  for (int q = threadIdx.x; q < kk * kk * h; q += blockDim.x) {
    const int IJ = q / h, i = q - IJ * h, i2 = k - 1 - i, I = IJ / kk, J = IJ - I * kk;
    const double *v = b + IJ * k;
    const int n1 = k - i, n = i2 != i ? k + 1 : n1;
    double e = 0.0, o = 0.0, e1 = 0.0, o1 = 0.0;
    int at = i * k + i, j = i;
    for (int t = 0; t < n; ++t) {
      if (t == n1) {
        e1 = e;
        o1 = o;
        e = o = 0.0;
        at = i2 * k + i2;
        j = i2;
      }
      const double f = fma(U[at], v[j], e);  // the two parities take turns
      e = o;
      o = f;
      ++at;
      ++j;
    }
    if (n == n1) {
      e1 = e;
      o1 = o;
    }
    if (n1 & 1) {
      const double s = e1;
      e1 = o1;
      o1 = s;
    }
    emit(I, J, i, e1 + o1);
    emit(I, J, k + i, e1 - o1);
    if (n != n1) {
      if ((n - n1) & 1) {
        const double s = e;
        e = o;
        o = s;
      }
      emit(I, J, i2, e + o);
      emit(I, J, k + i2, e - o);
    }
  }
}

// x0 + x1 and x0 - x1 in place, for the pairs of the two halves (stride half) of n pairs spaced by `step` blocks.
__device__ __forceinline__ void sums_and_differences(double *S, int outer, int half) {
  for (int q = threadIdx.x; q < outer * half; q += blockDim.x) {
    double *x = S + (q / half) * 2 * half + q % half;
    const double x0 = x[0], x1 = x[half];
    x[0] = x0 + x1;
    x[half] = x0 - x1;
  }
}

// Column j of U over sums p (stride st) and differences m = p + off.
__device__ __forceinline__ double column(int k, int j, const double *U, const double *p, int st, int off) {
  double v = 0.0, w = 0.0;
  int i = j;
  for (; i >= 1; i -= 2) {
    v = fma(U[i * k + j], p[i * st], v);
    w = fma(U[(i - 1) * k + j], p[(i - 1) * st + off], w);
  }
  if (i == 0) v = fma(U[j], p[0], v);
  return v + w;
}

// The first dimension of the filter from S (shared memory, (2k)^3, overwritten) into a[j][J][L] (4 k^3).
__device__ __forceinline__ void up_first(int k, const double *U, double *S, double *a) {
  const int k4 = 4 * k * k;
  sums_and_differences(S, 1, k * k4);
  __syncthreads();
  for (int q = threadIdx.x; q < k * k4; q += blockDim.x) {
    const int j = q / k4, r = q - j * k4;
    a[q] = column(k, j, U, S + r, k4, k * k4);
  }
  __syncthreads();
}

// The other two dimensions: a[j][J][L] (overwritten) through b (2 k^3) to s (k^3); complete on return.
__device__ __forceinline__ void up_rest(int k, const double *U, double *a, double *b, double *s) {
  const int kk = 2 * k, k2 = k * k;
  sums_and_differences(a, k, k * kk);
  __syncthreads();
  for (int q = threadIdx.x; q < k * k * kk; q += blockDim.x) {  // b[x][j][L]
    const int j = q / (k * kk), r = q - j * k * kk, x = r / kk, L = r - x * kk;
    b[(x * k + j) * kk + L] = column(k, j, U, a + x * kk * kk + L, kk, k * kk);
  }
  __syncthreads();
  sums_and_differences(b, k2, k);
  __syncthreads();
  for (int q = threadIdx.x; q < k2 * k; q += blockDim.x) {  // s[x][y][j]
    const int xy = q / k, j = q - xy * k;
    s[q] = column(k, j, U, b + xy * kk, 1, k);
  }
  __syncthreads();
}

}  // namespace twoscale
}  // namespace mra
