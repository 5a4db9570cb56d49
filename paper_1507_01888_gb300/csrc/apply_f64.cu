// apply_f64.cu -- FP64 apply of the records with |l|_inf <= 1, source-stationary, in parity components.
//
// The FP64 pipe is what bounds this apply (about two FMAs per SM and clock), so the kernel is built
// around doing fewer of them.  Two facts about the terms c_m R_{m,lx} x R_{m,ly} x R_{m,lz} s_b
// (Sec. 2.3) of one source b:
//   * the first mode product depends on (m, lx) only and the first two on (m, lx, ly), so they
//     are shared by the terms that differ in the later displacements: 3 + 9 + 27 products for a
//     full neighbourhood instead of 3 x 27;
//   * reflecting the source and the displacement gives R_{-l}[i][j] = (-1)^{i+j} R_l[i][j].  So
//     R_0 has entries with i + j even only, and R_{+1} = E + O, R_{-1} = E - O with E the entries
//     with i + j even and O the others.  The three products R_0 x, E x, O x cost k^2/2 FMAs each
//     (1.5 k^2 in all) and give what three full products (3 k^2) give; E and O parts are carried
//     through all three stages and added and subtracted once, after the sum over m.
// A full neighbourhood takes 19.5 k^4 FMAs per source and term instead of 81 k^4.  Measured on the
// whole apply against the per-destination gather with full products (apply_f64_kernel, now for wider
// displacements only): bound-state Helmholtz M = 60, k = 10, 17,200 boxes, 5.92 M kept terms 314 ->
// 78.6 ms (0.567 T FMA/s, 90% of two per SM and clock); order 20, 1,408 leaves in non-standard form, all levels in
// one apply, 931 -> 71.6 ms; 64 boxes, k = 6, M = 20 1.51 -> 0.29 ms (0.39 before the apply's small kernels were joined).
//
// Work decomposition.  The output index ix of the first product is carried unchanged through the
// other two, so the work of a source splits without redundancy into slices (cx, ix), cx = 0, E, O:
// per m, a slice is one k x k matrix t1 = (row ix of the cx block) s, three k x k matrices
// t2[cy], and nine accumulators [cy][cz] of k x k elements, kept in registers over all m.  A CTA
// takes 2 nx slices of one source: nx values of ix with E and O (the records lx = +-1), or 2 nx
// values with cx = 0 (the records lx = 0).  Each thread owns PT/2 elements of both halves, i.e.
// PT x 9 accumulators.  The sums of each record are written once, as FP64 partials indexed by the
// record, and dest_sum_f64_kernel adds the partials of every destination in the order of the sorted
// records.  The partial buffer is bounded: larger applies run in ranges of records (an addition
// chain per destination in the same order, so the result does not depend on the ranges).  Where not even
// the smallest buffer is to be had, the apply is the gather's (apply.cu), which needs none.
#include <algorithm>

#include "apply_internal.cuh"

namespace mra {

namespace {

constexpr int PT = 4;               // elements per thread (9 accumulators each)
constexpr int F64_MAX_THREADS = 416;
constexpr size_t F64_MAX_SMEM = 200 * 1024;  // dynamic shared memory of a CTA
constexpr size_t F64_PARTIAL_BYTES = (size_t)4 << 30;      // most scratch of one range of records
constexpr size_t F64_PARTIAL_BYTES_MIN = (size_t)64 << 20;  // smallest: a range fills the chip a few times over

__host__ __device__ constexpr int par_half(int k) { return (k + 1) / 2; }
// doubles of one (level, m) entry of the parity table: [3 components][half of the j][k], even
__host__ __device__ constexpr int par_entry(int k) { return (3 * par_half(k) * k + 1) & ~1; }

// Sign of child c's coefficient i in the combination of parity a of the doubled basis: reflection
// maps child 0's phi_i to (-1)^i child 1's phi_i, so (phi_{0,i} +- (-1)^i phi_{1,i}) / sqrt 2 are even and odd.
__device__ __forceinline__ double pair_sign(int c, int i, int a) { return c && ((i + a) & 1) ? -1.0 : 1.0; }

// Parity table of every level (blockIdx.y): entry m holds W[comp][jj][i], comp 0: R_0, 1: E, 2: O (of l = 1), the
// entry [i][j] of the block with j = 2 jj + (i & 1) for comp 0 and 1 and 2 jj + 1 - (i & 1) for O
// (zero beyond k).  Non-standard operators (pairs = 1) are first turned into the basis of even and
// odd child combinations, index 2 i + parity.
__global__ void parity_table_kernel(int k, int M, int min_level, const int *Dlev, const int64_t *level_off,
                                    const double *R, double *W, int pairs) {
  const int m = blockIdx.x, lev = min_level + blockIdx.y, D = Dlev[lev], h = par_half(k), nl = 2 * D + 1, hk = k / 2;
  const double *Rm = R + (level_off[lev] + (int64_t)m * nl) * k * k;
  double *Wm = W + ((int64_t)blockIdx.y * M + m) * par_entry(k);
  for (int e = threadIdx.x; e < par_entry(k); e += blockDim.x) {
    const int comp = e / (h * k), jj = (e / k) % h, i = e % k;
    const int j = 2 * jj + (comp == 2 ? 1 - (i & 1) : (i & 1));
    double v = 0.0;
    if (comp < 3 && j < k && (comp == 0 || D >= 1)) {
      const double *B = Rm + (D + (comp ? 1 : 0)) * k * k;
      if (!pairs) {
        v = B[i * k + j];
      } else {
        for (int c = 0; c < 2; ++c)
          for (int d = 0; d < 2; ++d)
            v += pair_sign(c, i >> 1, i & 1) * pair_sign(d, j >> 1, j & 1) * B[(c * hk + (i >> 1)) * k + d * hk + (j >> 1)];
        v *= 0.5;
      }
    }
    Wm[e] = v;
  }
}

struct F64Args {
  int k, nx, n0, n1;              // slices: nx per half; CTAs per source with lx = 0 and with lx = +-1
  int pairs;                      // 1: doubled (non-standard) basis
  int M, min_level;
  const double *W, *c;            // parity table [level - min_level][m][par_entry], coefficients
  const double *R;                // the blocks themselves (terms whose mirror image is not kept)
  const int *Dlev;
  const int64_t *level_off;
  const uint64_t *in_keys;
  const double *in_coeffs;
  const int64_t *rec_cnt, *rec_off;
  const int *rec_l;
  const uint64_t *rec_mask;
  double *partial;                // [p1 - p0][k^3]
  int64_t p0, p1;                 // records of this launch
  int64_t n_src, n_rec;
  const int *skip;                // see FixedSizes
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One term c_m R_lx x R_ly x R_lz s at one element, straight from the blocks (k^3 FMAs): for the
// rare term that the screen keeps for a displacement and drops for its mirror image, because the
// two computed block norms differ in the last bit and the threshold lies between the two bounds.
__device__ __noinline__ double lone_term(const F64Args &a, const double *s, int n, int m, int lx, int ly, int lz, int ix, int iy,
                            int iz) {
  const int k = a.k, Dop = a.Dlev[n], nl = 2 * Dop + 1, hk = k / 2;
  const double *B = a.R + (a.level_off[n] + (int64_t)m * nl + Dop) * k * k;
  // entry [i][j] of the block of displacement l, in the basis of s
  auto at = [&](int l, int i, int j) {
    const double *Bl = B + (int64_t)l * k * k;
    if (!a.pairs) return Bl[i * k + j];
    double v = 0.0;
    for (int c = 0; c < 2; ++c)
      for (int d = 0; d < 2; ++d)
        v += pair_sign(c, i >> 1, i & 1) * pair_sign(d, j >> 1, j & 1) * Bl[(c * hk + (i >> 1)) * k + d * hk + (j >> 1)];
    return 0.5 * v;
  };
  double v = 0.0;
  for (int x = 0; x < k; ++x) {
    double vy = 0.0;
    for (int y = 0; y < k; ++y) {
      double vz = 0.0;
      for (int z = 0; z < k; ++z) vz += at(lz, iz, z) * s[(x * k + y) * k + z];
      vy += at(ly, iy, y) * vz;
    }
    v += at(lx, ix, x) * vy;
  }
  return a.c[m] * v;
}

__global__ void __launch_bounds__(F64_MAX_THREADS, 1) apply_f64_sym_kernel(const __grid_constant__ F64Args a) {
  extern __shared__ __align__(16) double sh[];
  __shared__ unsigned long long all[4][2], any[4][2];  // kept-term masks by (|ly|, |lz|): AND and OR over the signs
  __shared__ int rec[2][9];                            // record of (sign of lx, ly, lz), -1 = none in range
  __shared__ int lone;                                 // some mask differs from its mirror images'
  if (a.skip && *a.skip) return;
  const int k = a.k, k2 = k * k, k3 = k2 * k, h = par_half(k), nx = a.nx, we = par_entry(k);
  const int64_t b = blockIdx.x;
  const int ch = blockIdx.y;
  const int ax = ch < a.n1 ? 1 : 0;                    // |lx| of this CTA's records (the longer work first)
  const int ix0 = ax ? ch * nx : (ch - a.n1) * 2 * nx;
  const int64_t r0 = a.rec_off[b];
  const int rc = (int)a.rec_cnt[b];                    // at most 27
  if (rc == 0 || r0 >= a.p1 || r0 + rc <= a.p0) return;
  const int tid = threadIdx.x, nt = blockDim.x;
  double *W0 = sh, *W1 = W0 + we, *s = W1 + we, *t1 = s + k3 + (k3 & 1), *t2 = t1 + 2 * nx * k2;
  if (tid < 8) {
    all[tid >> 1][tid & 1] = ~0ull;
    any[tid >> 1][tid & 1] = 0ull;
  }
  if (tid < 18) rec[tid / 9][tid % 9] = -1;
  if (tid == 0) lone = 0;
  __syncthreads();
  if (tid < rc) {
    const int64_t p = MRA_IDX(r0 + tid, a.n_rec);
    const int lp = a.rec_l[p];
    const int lx = (lp & 255) - 128, ly = ((lp >> 8) & 255) - 128, lz = ((lp >> 16) & 255) - 128;
    if (abs(lx) == ax) {
      const int q = (abs(ly) << 1) | abs(lz);
      for (int w = 0; w < 2; ++w) {
        atomicAnd(&all[q][w], (unsigned long long)a.rec_mask[2 * p + w]);
        atomicOr(&any[q][w], (unsigned long long)a.rec_mask[2 * p + w]);
      }
      if (p >= a.p0 && p < a.p1) rec[lx < 0 ? 1 : 0][(ly + 1) * 3 + lz + 1] = (int)(p - a.p0);
    }
  }
  __syncthreads();
  uint64_t um[2] = {0ull, 0ull}, om[2] = {0ull, 0ull};
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const uint64_t both = all[q][w] & any[q][w];
      um[w] |= both;
      om[w] |= any[q][w];
      if (tid == 0 && both != any[q][w]) lone = 1;
    }
  if (!(om[0] | om[1])) return;  // no record with this |lx|
  const int n = key_level(a.in_keys[b]);
  const double *Wl = a.W + (int64_t)(n - a.min_level) * a.M * we;
  // the source's coefficients, in the doubled basis turned into even and odd child combinations
  const double *sb = a.in_coeffs + (int64_t)MRA_IDX(b, a.n_src) * k3;
  if (!a.pairs) {
    for (int e = tid; e < k3; e += nt) s[e] = sb[e];
  } else {
    const int hk = k / 2;
    for (int e = tid; e < k3; e += nt) {
      const int x = e / k2, y = (e / k) % k, z = e % k;
      double v = 0.0;
      for (int c = 0; c < 8; ++c) {
        const int cx = c >> 2, cy = (c >> 1) & 1, cz = c & 1;
        v += pair_sign(cx, x >> 1, x & 1) * pair_sign(cy, y >> 1, y & 1) * pair_sign(cz, z >> 1, z & 1) *
             sb[((cx * hk + (x >> 1)) * k + cy * hk + (y >> 1)) * k + cz * hk + (z >> 1)];
      }
      s[e] = v;  // 8^{1/2} times the orthonormal combination; dest_sum_f64_kernel divides by 8, exactly
    }
  }
  // this thread's elements: (ix within the half, iy, iz) of both halves
  int ex[PT / 2], ey[PT / 2], ez[PT / 2], jb[PT / 2];
#pragma unroll
  for (int q = 0; q < PT / 2; ++q) {
    const int e = tid + q * nt;
    const bool in = e < nx * k2;
    ex[q] = in ? e / k2 : -1;
    ey[q] = (e / k) % k;
    ez[q] = e % k;
    jb[q] = e % k2;
  }
  // half hf of element q: its ix (or -1), and where its slice starts in t1
  auto ix_of = [&](int hf, int q) {
    const int ix = ix0 + (ax ? 0 : hf * nx) + ex[q];
    return ex[q] >= 0 && ix < k ? ix : -1;
  };
  double acc[PT][3][3];
#pragma unroll
  for (int q = 0; q < PT; ++q)
#pragma unroll
    for (int y = 0; y < 3; ++y)
#pragma unroll
      for (int z = 0; z < 3; ++z) acc[q][y][z] = 0.0;
  auto next_term = [&](uint64_t *u) {
    int m = -1;
    if (u[0]) {
      m = __ffsll((long long)u[0]) - 1;
      u[0] &= u[0] - 1;
    } else if (u[1]) {
      m = 64 + __ffsll((long long)u[1]) - 1;
      u[1] &= u[1] - 1;
    }
    return m;
  };
  auto fetch = [&](int m, double *dst) {
    const double *src = Wl + (int64_t)m * we;
    for (int e = 2 * tid; e < we; e += 2 * nt) cp_async16(dst + e, src + e);
  };
  int m = next_term(um);
  if (m >= 0) fetch(m, W0);
  const int pk = k - 1;  // rows beyond the last (odd k) are read from it, with weight zero
  while (m >= 0) {
    cp_async_wait();
    __syncthreads();  // the term's blocks (and, the first time, the source) are there; t2 and the other block buffer are free
    const int mn = next_term(um);
    if (mn >= 0) fetch(mn, W1);
    // ---- stage 1: slice (cx, ix), contraction jx
    const double cm = a.c[m];
#pragma unroll
    for (int q = 0; q < PT; ++q) {
      const int hf = q / (PT / 2), qq = q % (PT / 2), ix = ix_of(hf, qq);
      if (ix < 0) continue;
      const int comp = ax ? 1 + hf : 0, par = comp == 2 ? 1 - (ix & 1) : (ix & 1);
      const double *w = W0 + comp * h * k + ix, *x = s + jb[qq];
      double v = 0.0;
      for (int jj = 0; jj < h; ++jj) v = fma(w[jj * k], x[min(2 * jj + par, pk) * k2], v);
      t1[(hf * nx + ex[qq]) * k2 + jb[qq]] = cm * v;
    }
    // which products this term needs
    bool need[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) need[q] = ((all[q][m >> 6] & any[q][m >> 6]) >> (m & 63)) & 1ull;
    const bool y0 = need[0] || need[1], y1 = need[2] || need[3];
    __syncthreads();
    // ---- stage 2: components cy, contraction jy
#pragma unroll
    for (int q = 0; q < PT; ++q) {
      const int hf = q / (PT / 2), qq = q % (PT / 2);
      if (ix_of(hf, qq) < 0) continue;
      const int iy = ey[qq], py = iy & 1, sl = hf * nx + ex[qq];
      const double *w = W0 + iy, *x = t1 + sl * k2 + ez[qq];
      double v0 = 0.0, v1 = 0.0, v2 = 0.0;
      if (y0 && y1) {
        for (int jj = 0; jj < h; ++jj) {
          const double u = x[min(2 * jj + py, pk) * k], o = x[min(2 * jj + 1 - py, pk) * k];
          v0 = fma(w[jj * k], u, v0);
          v1 = fma(w[(h + jj) * k], u, v1);
          v2 = fma(w[(2 * h + jj) * k], o, v2);
        }
      } else if (y0) {
        for (int jj = 0; jj < h; ++jj) v0 = fma(w[jj * k], x[min(2 * jj + py, pk) * k], v0);
      } else {
        for (int jj = 0; jj < h; ++jj) {
          v1 = fma(w[(h + jj) * k], x[min(2 * jj + py, pk) * k], v1);
          v2 = fma(w[(2 * h + jj) * k], x[min(2 * jj + 1 - py, pk) * k], v2);
        }
      }
      double *o = t2 + sl * k2 + jb[qq];
      if (y0) o[0] = v0;
      if (y1) {
        o[2 * nx * k2] = v1;
        o[4 * nx * k2] = v2;
      }
    }
    __syncthreads();
    // ---- stage 3: components cz, contraction jz, into the accumulators
#pragma unroll
    for (int q = 0; q < PT; ++q) {
      const int hf = q / (PT / 2), qq = q % (PT / 2);
      if (ix_of(hf, qq) < 0) continue;
      const int iz = ez[qq], pz = iz & 1, sl = hf * nx + ex[qq];
      const double *w = W0 + iz;
#pragma unroll
      for (int cy = 0; cy < 3; ++cy) {
        if (!(cy == 0 ? y0 : y1)) continue;
        const bool z0 = need[cy == 0 ? 0 : 2], z1 = need[cy == 0 ? 1 : 3];
        const double *x = t2 + (cy * 2 * nx + sl) * k2 + ey[qq] * k;
        double v0 = acc[q][cy][0], v1 = acc[q][cy][1], v2 = acc[q][cy][2];
        if (z0 && z1) {
          for (int jj = 0; jj < h; ++jj) {
            const double u = x[min(2 * jj + pz, pk)], o = x[min(2 * jj + 1 - pz, pk)];
            v0 = fma(w[jj * k], u, v0);
            v1 = fma(w[(h + jj) * k], u, v1);
            v2 = fma(w[(2 * h + jj) * k], o, v2);
          }
        } else if (z0) {
          for (int jj = 0; jj < h; ++jj) v0 = fma(w[jj * k], x[min(2 * jj + pz, pk)], v0);
        } else if (z1) {
          for (int jj = 0; jj < h; ++jj) {
            v1 = fma(w[(h + jj) * k], x[min(2 * jj + pz, pk)], v1);
            v2 = fma(w[(2 * h + jj) * k], x[min(2 * jj + 1 - pz, pk)], v2);
          }
        }
        acc[q][cy][0] = v0;
        acc[q][cy][1] = v1;
        acc[q][cy][2] = v2;
      }
    }
    m = mn;
    double *t = W0;
    W0 = W1;
    W1 = t;
  }
  __syncthreads();  // lone; and the source, when no term ran
  // ---- E +- O in y and z, then in x; the records' sums
#pragma unroll
  for (int q = 0; q < PT / 2; ++q) {
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      double(&c)[3][3] = acc[hf * (PT / 2) + q];
#pragma unroll
      for (int y = 0; y < 3; ++y) {  // z: 1, 2 -> +, -
        const double e = c[y][1], o = c[y][2];
        c[y][1] = e + o;
        c[y][2] = e - o;
      }
#pragma unroll
      for (int z = 0; z < 3; ++z) {
        const double e = c[1][z], o = c[2][z];
        c[1][z] = e + o;
        c[2][z] = e - o;
      }
    }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {  // lx = 0: the half's own ix; else lx = +1 and -1 of the same ix
      const int ix = ix_of(hf, q);
      if (ix < 0) continue;
      const int elem = (ix * k + ey[q]) * k + ez[q];
#pragma unroll
      for (int y = 0; y < 3; ++y)
#pragma unroll
        for (int z = 0; z < 3; ++z) {
          // component index 0, 1, 2 stands for displacement 0, +1, -1
          const int ly = y == 0 ? 0 : (y == 1 ? 1 : -1), lz = z == 0 ? 0 : (z == 1 ? 1 : -1);
          const int p = rec[ax ? hf : 0][(ly + 1) * 3 + lz + 1];
          if (p < 0) continue;
          const double u = acc[q][y][z], v = acc[PT / 2 + q][y][z];
          double r = ax ? (hf ? u - v : u + v) : (hf ? v : u);
          if (lone) {
            const int qm = (abs(ly) << 1) | abs(lz), lx = ax ? (hf ? -1 : 1) : 0;
            for (int w = 0; w < 2; ++w) {
              uint64_t bits = a.rec_mask[2 * (a.p0 + p) + w] & ~all[qm][w];
              while (bits) {
                r += lone_term(a, s, n, 64 * w + __ffsll((long long)bits) - 1, lx, ly, lz, ix, ey[q], ez[q]);
                bits &= bits - 1;
              }
            }
          }
          a.partial[(int64_t)p * k3 + elem] = r;
        }
    }
  }
}

// Sum the partials of every destination over the records [p0, p1) in sorted order (ascending record
// index within a destination, so one contiguous run), one CTA per destination: HBM-bound, k^3
// doubles read per record.  first: start from zero, else from the earlier ranges' sums in the
// output; last: doubled-basis sums are turned back into child coefficients.
__global__ void dest_sum_f64_kernel(int k, const int64_t *seg, const int *perm, const double *partial, int64_t p0,
                                    int64_t p1, int first, int last, int pairs, const uint64_t *dest_key,
                                    uint64_t *out_keys, double *out_coeffs, int64_t n_rec, const int *skip) {
  extern __shared__ __align__(16) double sum[];  // k^3, doubled basis only
  if (skip && *skip) return;
  const int64_t d = blockIdx.x;
  const int k2 = k * k, k3 = k2 * k;
  int64_t r0 = seg[d], r1 = seg[d + 1];
  if (p0 > 0 || p1 < n_rec) {
    auto lower = [&](int64_t p) {
      int64_t lo = seg[d], hi = seg[d + 1];
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (perm[MRA_IDX(mid, n_rec)] < p) lo = mid + 1; else hi = mid;
      }
      return lo;
    };
    r0 = lower(p0);
    r1 = lower(p1);
  }
  if (first && threadIdx.x == 0) out_keys[d] = dest_key[d];
  if (r0 == r1 && !first && !(last && pairs)) return;
  double *o = out_coeffs + d * k3;
  for (int e = threadIdx.x; e < k3; e += blockDim.x) {
    double v = first ? 0.0 : o[e];
    auto rec = [&](int64_t r) {
      return __ldcs(partial + ((int64_t)MRA_IDX((int64_t)perm[MRA_IDX(r, n_rec)], n_rec) - p0) * k3 + e);
    };
    int64_t r = r0;
    for (; r + 4 <= r1; r += 4) {
      const double a0 = rec(r), a1 = rec(r + 1), a2 = rec(r + 2), a3 = rec(r + 3);
      v += a0;
      v += a1;
      v += a2;
      v += a3;
    }
    for (; r < r1; ++r) v += rec(r);
    if (pairs && last)
      sum[e] = v;
    else
      o[e] = v;
  }
  if (!(pairs && last)) return;
  __syncthreads();
  const int hk = k / 2;
  for (int e = threadIdx.x; e < k3; e += blockDim.x) {
    const int x = e / k2, y = (e / k) % k, z = e % k;
    const int cx = x / hk, cy = y / hk, cz = z / hk, i = x % hk, j = y % hk, l = z % hk;
    double v = 0.0;
    for (int q = 0; q < 8; ++q) {
      const int pa = q >> 2, pb = (q >> 1) & 1, pc = q & 1;
      v += pair_sign(cx, i, pa) * pair_sign(cy, j, pb) * pair_sign(cz, l, pc) *
           sum[((2 * i + pa) * k + 2 * j + pb) * k + 2 * l + pc];
    }
    o[e] = 0.125 * v;
  }
}

size_t f64_smem(int k, int nx) {
  const int k2 = k * k, k3 = k2 * k;
  return (size_t)(2 * par_entry(k) + k3 + (k3 & 1) + 8 * nx * k2) * sizeof(double);
}

// Slices per half and threads of a CTA.  The time of the most loaded SM is modelled as its warps'
// FP64 instructions, idle lanes and slices included (an SM's FP64 pipe takes a warp instruction in
// 16 cycles), times 8 / (resident warps) where fewer than eight warps are there to hide their own
// latency; the least wins.  Large trees get the split with the fewest idle lanes (k = 10: 5 slices,
// 256 threads, two elements of each half per thread), small ones more CTAs of fewer elements per thread.
// 64 boxes, k = 6, M = 20, whole call when it was chosen: 1 slice and two elements in one warp 501 us, 6 slices and
// one element in seven warps 394 us (now 293).
void f64_shape(int k, int64_t n_src, int sms, int *nx_out, int *threads_out) {
  double best = -1.0;
  for (int nx = 1; nx <= k; ++nx)
    for (int ept = PT / 2; ept >= 1; --ept) {
      const int threads = ((nx * k * k + ept - 1) / ept + 31) / 32 * 32, warps = threads / 32;
      const size_t smem = f64_smem(k, nx) + 1024;
      if (threads > F64_MAX_THREADS || smem > F64_MAX_SMEM) continue;
      const int64_t ctas = n_src * ((k + 2 * nx - 1) / (2 * nx) + (k + nx - 1) / nx);
      const int64_t per_sm = (ctas + sms - 1) / sms;
      const int64_t resident = std::min<int64_t>(per_sm, std::min<int64_t>(512 / threads, (228 * 1024) / smem));
      const double cost = (double)per_sm * warps * 2 * ept *
                          std::max(1.0, 8.0 / (double)(std::max<int64_t>(resident, 1) * warps)) *
                          (1.0 + 0.25 / (warps * ept));  // staging the source once per CTA
      if (best < 0.0 || cost < best) {
        best = cost;
        *nx_out = nx;
        *threads_out = threads;
      }
    }
}

}  // namespace

int f64_parity_build(Operator &op, cudaStream_t s) {
  const size_t we = (size_t)par_entry(op.k), levels = op.D.size();
  if (!op.d_W) MRA_CUDA_TRY(cudaMalloc((void **)&op.d_W, levels * op.M * we * sizeof(double)));
  parity_table_kernel<<<counted(dim3((unsigned)op.M, (unsigned)levels)), 128, 0, s>>>(
      op.k, op.M, op.min_level, op.d_D, op.d_level_off, op.d_R, op.d_W, op.non_standard ? 1 : 0);
  MRA_CUDA_TRY(cudaGetLastError());
  return MRA_OK;
}

// Bytes of the partial buffer of P records: all of them, or as many as the bound holds.
size_t f64_partial_bytes(int k, int64_t P) {
  const size_t row = (size_t)k * k * k * sizeof(double);
  return std::min((size_t)P * row, std::max(F64_PARTIAL_BYTES, row));
}

size_t f64_partial_least(int k, int64_t P) {
  const size_t row = (size_t)k * k * k * sizeof(double);
  return std::min(f64_partial_bytes(k, P), std::max(F64_PARTIAL_BYTES_MIN, row));
}

int apply_f64_run(const Operator &op, const mra_tree_view &in, mra_tree_view &out, const ApplyWork &wk, cudaStream_t s,
                  bool *ran) {
  *ran = false;
  const int k = op.k, k3 = k * k * k;
  const int64_t P = wk.P, nd = wk.n_dest;
  const size_t row = (size_t)k3 * sizeof(double);
  int dev = 0, sms = 0;
  MRA_CUDA_TRY(cudaGetDevice(&dev));
  MRA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  size_t bytes = wk.fx ? wk.fx->partial_bytes : f64_partial_bytes(k, P);
  const size_t least = f64_partial_least(k, P);
  double *partial = wk.fx ? (double *)wk.fx->partial : nullptr;
  if (!wk.fx) {
    // when memory is short, smaller ranges of records
    while (pool_malloc((void **)&partial, bytes, s) != cudaSuccess) {
      cudaGetLastError();
      if (bytes <= least) return MRA_OK;
      bytes = std::max(bytes / 2, least);
    }
  }
  if (!partial) return MRA_OK;
  *ran = true;
  const int64_t range = (int64_t)(bytes / row);
  if (range < 1) return fail(MRA_ERR_ARG, "mra_apply: partial-sum buffer smaller than one record");
  F64Args a{};
  a.k = k;
  int threads = 32;
  a.nx = 1;
  f64_shape(k, in.n, sms, &a.nx, &threads);
  a.n0 = (k + 2 * a.nx - 1) / (2 * a.nx);
  a.n1 = (k + a.nx - 1) / a.nx;
  a.pairs = op.non_standard ? 1 : 0;
  a.M = op.M;
  a.min_level = op.min_level;
  a.W = op.d_W;
  a.c = op.d_c;
  a.R = op.d_R;
  a.Dlev = op.d_D;
  a.level_off = op.d_level_off;
  a.in_keys = in.keys;
  a.in_coeffs = in.coeffs;
  a.rec_cnt = wk.rec_cnt;
  a.rec_off = wk.rec_off;
  a.rec_l = wk.rec_l;
  a.rec_mask = wk.rec_mask;
  a.partial = partial;
  a.n_src = in.n;
  a.n_rec = P;
  a.skip = wk.skip();
  const size_t smem = f64_smem(k, a.nx), dsm = a.pairs ? row : 0;
  // the same limit whatever the order, so that callers on several threads do not lower it for one another
  cudaError_t e = cudaFuncSetAttribute(apply_f64_sym_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F64_MAX_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(dest_sum_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             MRA_MAX_NS_K * MRA_MAX_NS_K * MRA_MAX_NS_K * (int)sizeof(double));
  if (e == cudaSuccess && wk.ev0) e = cudaEventRecord(wk.ev0, s);
  for (int64_t p0 = 0; p0 < P && e == cudaSuccess; p0 += range) {
    a.p0 = p0;
    a.p1 = std::min(P, p0 + range);
    apply_f64_sym_kernel<<<counted(dim3((unsigned)in.n, (unsigned)(a.n0 + a.n1))), threads, smem, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    dest_sum_f64_kernel<<<counted((unsigned)nd), k3 >= 512 ? 256 : 128, dsm, s>>>(
        k, wk.seg, wk.perm, partial, a.p0, a.p1, p0 == 0, a.p1 == P, a.pairs, wk.dest_key, out.keys, out.coeffs, P, wk.skip());
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && wk.ev1) e = cudaEventRecord(wk.ev1, s);
  if (!wk.fx) cudaFreeAsync(partial, s);
  if (e != cudaSuccess) return fail(MRA_ERR_CUDA, "mra_apply: FP64 apply: %s", cudaGetErrorString(e));
  return MRA_OK;
}

int debug_line_f64(cudaStream_t s) { return debug_take_line(s); }

}  // namespace mra
