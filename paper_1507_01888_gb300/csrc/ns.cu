// ns.cu -- the operator in non-standard form and its apply on uniform trees (Sec. 2.2).
//
// With P^{n+1} = P^n + Q^n the level-N operator T^N = P^N T P^N splits into
//     T^N = T^{n0} + sum_{n=n0}^{N-1} (A^n + B^n + C^n),
// A^n = Q^n T Q^n, B^n = Q^n T P^n, C^n = P^n T Q^n.  On level n's 2k basis -- a box's
// children's k^3 coefficients side by side, S[(cx,i)][(cy,j)][(cz,l)] -- the level-(n+1)
// operator has the blocks
//     R2k^n_{m,l}[(ci,i)][(cj,j)] = R^{n+1}_{m, 2l+ci-cj}[i][j]
// and A^n + B^n + C^n = T2k^n - Ubar T^n Ubar^T with Ubar[(c,i)][j] = U^(c)[i][j].  Its
// blocks decay with the displacement (A as r^(-2k-1), B and C as r^(-k-1)), so a small
// displacement range per level reaches the operator's long range through the coarse levels.
//
// The apply (uniform level N, every box present):
//   compress   s^n = (Ubar^T)^{x3} S^n, S^n = children of level n, for n = N-1 .. n0;
//   coarsest   r^{n0} = T^{n0} s^{n0} with every displacement of level n0;
//   per level  Y^n = T2k^n S^n and Z^n = T^n s^n (the library's apply on level n's boxes,
//              |l|_inf <= max_disp, FP64 or split BF16), then
//              r^{n+1}(children of b) = (Ubar)^{x3} (r^n_b - Z^n_b) + Y^n_b;
// r^N is the result.  With every displacement it equals the plain level-N apply.
#include <algorithm>
#include <vector>

#include <cub/cub.cuh>

#include "apply_internal.cuh"
#include "reconstruct.cuh"
#include "twoscale.cuh"

namespace mra {

namespace {

// ---------------------------------------------------------------- 2k blocks
// Blocks of every level n (blockIdx.y) of the non-standard operator from the level-(n+1) blocks of op.
__global__ void ns_blocks_kernel(int k, int M, int min_level, const int *Dns, const int64_t *ns_off, const int *Dop,
                                 const int64_t *op_off, const double *Rop, double *Rns) {
  const int n = min_level + blockIdx.y, D = Dns[n], Dc = Dop[n + 1];
  const int64_t ns_base = ns_off[n], op_base = op_off[n + 1];
  const int nl = 2 * D + 1, nlc = 2 * Dc + 1, kk = 2 * k;
  const int q = blockIdx.x;  // m * nl + (l + D)
  if (q >= M * nl) return;
  const int m = q / nl, l = q % nl - D;
  double *B = Rns + (ns_base + q) * (int64_t)kk * kk;
  for (int e = threadIdx.x; e < kk * kk; e += blockDim.x) {
    const int I = e / kk, J = e % kk, ci = I / k, i = I % k, cj = J / k, j = J % k;
    const int lc = 2 * l + ci - cj;
    B[e] = Rop[(op_base + (int64_t)m * nlc + lc + Dc) * k * k + i * k + j];
  }
}

// Frobenius norm of every block (for the norm screen).
__global__ void block_norms_kernel(int64_t nblocks, int kk2, const double *R, double *N) {
  const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= nblocks) return;
  double s = 0.0;
  for (int e = lane; e < kk2; e += 32) {
    const double v = R[b * kk2 + e];
    s += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) N[b] = sqrt(s);
}

// ---------------------------------------------------------------- uniform levels
// Keys of every box of level n in key order (x slowest): box i at (i / nb^2, i / nb % nb, i % nb).
__global__ void level_keys_kernel(int n, int64_t nbox, uint64_t *keys) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nbox) return;
  const int64_t nb = 1LL << n;
  keys[i] = make_key(n, i / (nb * nb), (i / nb) % nb, i % nb);
}

__global__ void check_uniform_kernel(int n, int64_t nbox, const uint64_t *keys, int *err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nbox) return;
  const int64_t nb = 1LL << n;
  if (keys[i] != make_key(n, i / (nb * nb), (i / nb) % nb, i % nb)) atomicExch(err, 1);
}

// Rows of an apply's output (keys of level n, any subset) into a zeroed dense level array.
__global__ void scatter_dense_kernel(int64_t n_rows, const uint64_t *keys, const double *rows, int rowlen,
                                     double *dense) {
  const int64_t r = blockIdx.x;
  if (r >= n_rows) return;
  const uint64_t key = keys[r];
  const int64_t nb = 1LL << key_level(key);
  const int64_t d = (key_x(key) * nb + key_y(key)) * nb + key_z(key);
  for (int e = threadIdx.x; e < rowlen; e += blockDim.x) dense[d * rowlen + e] = rows[r * rowlen + e];
}

// The same for rows of several whole levels, n0 first, back to back.
__global__ void scatter_levels_kernel(int64_t n_rows, const uint64_t *keys, const double *rows, int rowlen, int n0,
                                      double *dense) {
  const int64_t r = blockIdx.x;
  if (r >= n_rows) return;
  const uint64_t key = keys[r];
  const int n = key_level(key);
  const int64_t nb = 1LL << n;
  int64_t d = (key_x(key) * nb + key_y(key)) * nb + key_z(key);
  for (int m = n0; m < n; ++m) d += 1LL << (3 * m);
  for (int e = threadIdx.x; e < rowlen; e += blockDim.x) dense[d * rowlen + e] = rows[r * rowlen + e];
}

// ---------------------------------------------------------------- two-scale transforms
// Threads of the kernels that transform one box per CTA.  A level often has fewer boxes than the chip has
// room for, so a launch lasts as long as one box does: 512 threads instead of 256.
constexpr int BOX_THREADS = 512;
// Shared memory of the transforms: U (k^2) and the buffers up (S 8 k^3, a 4 k^3) and down (7 k^3) need.
size_t up_smem(int k) { return (size_t)(k * k + 12 * k * k * k) * 8; }
size_t down_smem(int k) { return (size_t)(k * k + 7 * k * k * k) * 8; }
// The kernels' dynamic shared memory limit: one value for every order, so that callers on several threads do not
// lower it for one another (at order 16 a box takes 226 KB, beside up to 1 KB of static shared memory).
constexpr int BOX_SMEM = 226 * 1024;

// S (shared, complete, overwritten) filtered to the parent's coefficients, written to s_out.
__device__ __forceinline__ void filter_box(int k, const double *U, double *S, double *a, double *s_out) {
  const int k3 = k * k * k;
  twoscale::up_first(k, U, S, a);
  double *b = S, *sv = S + 2 * k3;
  twoscale::up_rest(k, U, a, b, sv);
  for (int e = threadIdx.x; e < k3; e += blockDim.x) s_out[e] = sv[e];
}

// One CTA per box of level n: S = the children (dense level n+1) as a (2k)^3 tensor, written
// out, and s = (Ubar^T)^{x3} S.
__global__ void compress_kernel(int k, int n, const double *fine, const double *Ub, double *S_out,
                                double *s_out) {
  extern __shared__ double sh[];
  const int kk = 2 * k, k3 = k * k * k, kk3 = kk * kk * kk;
  double *U = sh, *S = U + k * k, *a = S + kk3;
  const int64_t box = blockIdx.x, nb = 1LL << n, nf = 2 * nb;
  const int64_t x = box / (nb * nb), y = (box / nb) % nb, z = box % nb;
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) U[e] = Ub[e];
  for (int e = threadIdx.x; e < kk3; e += blockDim.x) {
    const int I = e / (kk * kk), J = (e / kk) % kk, Lq = e % kk;
    const int64_t child = ((2 * x + I / k) * nf + 2 * y + J / k) * nf + 2 * z + Lq / k;
    const double v = fine[child * k3 + ((I % k) * k + J % k) * k + Lq % k];
    S[e] = v;
    S_out[box * kk3 + e] = v;
  }
  __syncthreads();
  filter_box(k, U, S, a, s_out + box * k3);
}

// One CTA per box of level n: r^{n+1}(children) = (Ubar)^{x3} (r_b - Z_b) + Y_b, into the
// dense level n+1 array.
__global__ void sum_down_kernel(int k, int n, const double *r, const double *Z, const double *Y,
                                const double *Ub, double *fine) {
  extern __shared__ double sh[];
  const int kk = 2 * k, k3 = k * k * k, kk3 = kk * kk * kk;
  double *U = sh, *d = U + k * k, *a = d + k3, *b = a + 2 * k3;
  const int64_t box = blockIdx.x, nb = 1LL << n, nf = 2 * nb;
  const int64_t x = box / (nb * nb), y = (box / nb) % nb, z = box % nb;
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) U[e] = Ub[e];
  for (int e = threadIdx.x; e < k3; e += blockDim.x) d[e] = r[box * k3 + e] - Z[box * k3 + e];
  __syncthreads();
  twoscale::down(k, U, d, a, b, [&](int I, int J, int Lq, double v) {
    const int64_t child = ((2 * x + I / k) * nf + 2 * y + J / k) * nf + 2 * z + Lq / k;
    fine[child * k3 + ((I % k) * k + J % k) * k + Lq % k] = Y[box * kk3 + (I * kk + J) * kk + Lq] + v;
  });
}

// ---------------------------------------------------------------- adaptive trees
__device__ __forceinline__ int64_t find_sorted(const uint64_t *keys, int64_t n, uint64_t key) {
  int64_t lo = 0, hi = n - 1;
  while (lo <= hi) {
    const int64_t mid = (lo + hi) >> 1;
    const uint64_t v = keys[mid];
    if (v == key) return mid;
    if (v < key) lo = mid + 1; else hi = mid - 1;
  }
  return -1;
}

// Leaf checks: keys strictly increasing, every leaf deeper than n0; deepest level -> *maxlev.
__global__ void leaf_check_kernel(int64_t n, const uint64_t *keys, int n0, int *err, int *maxlev) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int lv = key_level(keys[i]);
  if (lv <= n0 || (i > 0 && keys[i] <= keys[i - 1])) atomicExch(err, 1);
  atomicMax(maxlev, lv);
}

// Ancestor on level n of every leaf deeper than n (others: the largest key, dropped later).
// Entry (j, i): the level-(n0+j) ancestor of leaf i when the leaf is deeper, else the largest key.
__global__ void ancestor_kernel(int64_t n_leaf, const uint64_t *keys, int n0, int nlev, uint64_t *anc) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_leaf * nlev) return;
  const int64_t i = e % n_leaf;
  const int n = n0 + (int)(e / n_leaf);
  const uint64_t k = keys[i];
  const int lv = key_level(k);
  anc[e] = lv > n ? make_key(n, key_x(k) >> (lv - n), key_y(k) >> (lv - n), key_z(k) >> (lv - n)) : ~0ull;
}

// One CTA per interior node of level n: its children (leaves or interior nodes of level n+1)
// as the (2k)^3 tensor S, and s = (Ubar^T)^{x3} S.  A missing child sets *err.
__global__ void compress_tree_kernel(int k, int n, const uint64_t *ikeys, int64_t n_int, const uint64_t *lkeys,
                                     const double *lcoeffs, int64_t n_leaf, const uint64_t *ckeys,
                                     const double *ccoeffs, int64_t n_child_int, const double *Ub, double *S_out,
                                     double *s_out, int *err) {
  extern __shared__ double sh[];
  __shared__ const double *src[8];
  const int kk = 2 * k, k3 = k * k * k, kk3 = kk * kk * kk;
  double *U = sh, *S = U + k * k, *a = S + kk3;
  const int64_t box = blockIdx.x;
  if (box >= n_int) return;
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) U[e] = Ub[e];
  const uint64_t key = ikeys[box];
  if (threadIdx.x < 8) {
    const int cx = threadIdx.x >> 2, cy = (threadIdx.x >> 1) & 1, cz = threadIdx.x & 1;
    const uint64_t ck = make_key(n + 1, 2 * key_x(key) + cx, 2 * key_y(key) + cy, 2 * key_z(key) + cz);
    const int64_t li = find_sorted(lkeys, n_leaf, ck);
    const double *p = nullptr;
    if (li >= 0) {
      p = lcoeffs + li * k3;
    } else {
      const int64_t ci = find_sorted(ckeys, n_child_int, ck);
      if (ci >= 0) p = ccoeffs + ci * k3;
    }
    if (!p) atomicExch(err, 2);
    src[threadIdx.x] = p;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kk3; e += blockDim.x) {
    const int I = e / (kk * kk), J = (e / kk) % kk, Lq = e % kk;
    const double *p = src[((I / k) << 2) | ((J / k) << 1) | (Lq / k)];
    const double v = p ? p[((I % k) * k + J % k) * k + Lq % k] : 0.0;
    S[e] = v;
    S_out[box * kk3 + e] = v;
  }
  __syncthreads();
  filter_box(k, U, S, a, s_out + box * k3);
}

// The halo of the level's sources: every in-cell box within |l|_inf <= D of one (others: the
// largest key, dropped later).
__global__ void halo_kernel(int64_t ni, const uint64_t *ikeys, int D, uint64_t *out) {
  const int w = 2 * D + 1, w3 = w * w * w;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ni * w3) return;
  const uint64_t k = ikeys[e / w3];
  const int l = (int)(e % w3), lx = l / (w * w) - D, ly = (l / w) % w - D, lz = l % w - D;
  const int n = key_level(k);
  const int64_t nb = 1LL << n, x = key_x(k) + lx, y = key_y(k) + ly, z = key_z(k) + lz;
  out[e] = (x < 0 || x >= nb || y < 0 || y >= nb || z < 0 || z >= nb) ? ~0ull : make_key(n, x, y, z);
}

// Children of the halo boxes (all levels; entry 8 j + c): a child that lies in the next level's halo is
// refined there (its rank in the whole halo list goes to dst), the others are leaves of the result
// (their keys to leaf_key, the largest key elsewhere).  *found counts the refined children.
__global__ void halo_children_kernel(int64_t nh, const uint64_t *hkeys, const int64_t *off, int nmax, int64_t *dst,
                                     uint64_t *leaf_key, int *id, unsigned long long *found) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool in = false;
  if (e < 8 * nh) {
    const uint64_t k = hkeys[e >> 3];
    const int n = key_level(k), c = (int)(e & 7);
    const uint64_t ck = make_key(n + 1, 2 * key_x(k) + (c >> 2), 2 * key_y(k) + ((c >> 1) & 1), 2 * key_z(k) + (c & 1));
    int64_t p = -1;
    if (n + 1 < nmax) p = find_sorted(hkeys + off[n + 1], off[n + 2] - off[n + 1], ck);
    in = p >= 0;
    dst[e] = in ? off[n + 1] + p : -1;
    leaf_key[e] = in ? ~0ull : ck;
    id[e] = (int)e;
  }
  const unsigned b = __ballot_sync(0xffffffffu, in);
  if ((threadIdx.x & 31) == 0 && b) atomicAdd(found, (unsigned long long)__popc(b));
}

// Leaf i in key order: its place in the output, kept at its child entry as -2 - i, and its key.
__global__ void leaf_places_kernel(int64_t n_leaf, const uint64_t *sorted, const int *id, int64_t *dst, uint64_t *okeys) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_leaf) return;
  dst[id[i]] = -2 - i;
  okeys[i] = sorted[i];
}

// The output rows of the two applies at every halo box (-1: a screened apply wrote none).
__global__ void halo_rows_kernel(int64_t nh, const uint64_t *hkeys, const uint64_t *ykeys, int64_t ny,
                                 const uint64_t *zkeys, int64_t nz, int64_t *yi, int64_t *zi) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nh) return;
  yi[j] = find_sorted(ykeys, ny, hkeys[j]);
  zi[j] = find_sorted(zkeys, nz, hkeys[j]);
}

// Every target row of an apply must lie in the sources' halo.
__global__ void targets_in_kernel(int64_t nt, const uint64_t *tkeys, const uint64_t *rkeys, int64_t nr, int *err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nt) return;
  if (find_sorted(rkeys, nr, tkeys[i]) < 0) atomicExch(err, 3);
}

// One CTA per halo box of one level (j0 + blockIdx.x): its children get (Ubar)^{x3} (r - Z) + Y (absent rows
// as zero), written to the next level's r where the child is refined there, else to the result.
__global__ void sum_down_tree_kernel(int k, int64_t j0, double *r, const int64_t *yi, const double *Y,
                                     const int64_t *zi, const double *Z, const int64_t *dst, const double *Ub,
                                     double *out) {
  extern __shared__ double sh[];
  __shared__ double *to[8];
  const int64_t p = j0 + blockIdx.x;
  const int kk = 2 * k, k3 = k * k * k, kk3 = kk * kk * kk;
  double *U = sh, *d = U + k * k, *a = d + k3, *b = a + 2 * k3;
  const int64_t y = yi[p], z = zi[p];
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) U[e] = Ub[e];
  for (int e = threadIdx.x; e < k3; e += blockDim.x) d[e] = r[p * k3 + e] - (z >= 0 ? Z[z * k3 + e] : 0.0);
  if (threadIdx.x < 8) {
    const int64_t t = dst[8 * p + threadIdx.x];
    to[threadIdx.x] = t >= 0 ? r + t * k3 : out + (-2 - t) * k3;
  }
  __syncthreads();
  twoscale::down(k, U, d, a, b, [&](int I, int J, int Lq, double v) {
    const int child = ((I / k) << 2) | ((J / k) << 1) | (Lq / k);
    to[child][((I % k) * k + J % k) * k + Lq % k] = (y >= 0 ? Y[y * kk3 + (I * kk + J) * kk + Lq] : 0.0) + v;
  });
}

// ---------------------------------------------------------------- reconstruct
// Level of the shallowest input box above box b or b itself (the input is sorted and unique).
__global__ void top_level_kernel(int64_t n, const uint64_t *keys, int *top) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const uint64_t k = keys[b];
  const int lv = key_level(k);
  int t = lv;
  for (int m = 0; m < lv; ++m)
    if (find_sorted(keys, n, make_key(m, key_x(k) >> (lv - m), key_y(k) >> (lv - m), key_z(k) >> (lv - m))) >= 0) {
      t = m;
      break;
    }
  top[b] = t;
}

// Interior boxes of levels n0 .. n0+nlev-1 at once: entry (j, b) is the level-(n0+j) ancestor of
// input box b when b is deeper and has an input box at or above that level on its path, else
// the largest key (dropped after the sort: its level field is beyond every level).
__global__ void interior_all_kernel(int64_t n_in, const uint64_t *keys, const int *top, int n0, int nlev,
                                    uint64_t *out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_in * nlev) return;
  const int64_t b = e % n_in;
  const int n = n0 + (int)(e / n_in);
  const uint64_t k = keys[b];
  const int lv = key_level(k);
  out[e] = (lv > n && top[b] <= n) ? make_key(n, key_x(k) >> (lv - n), key_y(k) >> (lv - n), key_z(k) >> (lv - n))
                                   : ~0ull;
}
// off[l] = first position of level l (0 <= l <= 20) in the sorted keys[0 .. *n)
__global__ void level_offsets_kernel(const uint64_t *keys, const int64_t *n, int64_t *off) {
  const int l = threadIdx.x;
  if (l > 20) return;
  const uint64_t x = (uint64_t)l << 57;
  int64_t a = 0, b = *n;
  while (a < b) {
    const int64_t m = (a + b) / 2;
    if (keys[m] < x) a = m + 1;
    else b = m;
  }
  off[l] = a;
}

// Keys strictly increasing and no level above 19 (*bad otherwise); off[l] = first position of level l, l <= 20.
__global__ void leaf_offsets_kernel(int64_t n, const uint64_t *keys, int64_t *off, int64_t *bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n) return;
  const int lv = i < n ? min(key_level(keys[i]), 21) : 21;
  const int pv = i > 0 ? min(key_level(keys[i - 1]), 21) : -1;
  if (i < n && (lv > MRA_MAX_LEVEL || (i > 0 && keys[i] <= keys[i - 1])))
    atomicMax((unsigned long long *)bad, lv > MRA_MAX_LEVEL ? 2ull : 1ull);
  for (int l = pv + 1; l <= min(lv, 20); ++l) off[l] = i;
}

// Input boxes that are tops (no input box above them): all of them and those that are interior too.
__global__ void count_tops_kernel(int64_t n, const uint64_t *keys, const int *top, const uint64_t *ikeys,
                                  const int64_t *ni, unsigned long long *count) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool t = false, in = false;
  if (b < n) {
    t = top[b] == key_level(keys[b]);
    if (t) in = find_sorted(ikeys, *ni, keys[b]) >= 0;
  }
  const unsigned bt = __ballot_sync(0xffffffffu, t), bi = __ballot_sync(0xffffffffu, in);
  if ((threadIdx.x & 31) == 0) {
    if (bt) atomicAdd(count, (unsigned long long)__popc(bt));
    if (bi) atomicAdd(count + 1, (unsigned long long)__popc(bi));
  }
}

// The nodes of the result by entry: 8 j + c, child c of interior box j, then 8 ni + b, input box b.  A child
// that is interior is passed on (dst = its rank), the other children and the tops that are not interior are
// leaves (their keys in leaf_key, the largest key elsewhere).  own: the input box at the child, or -1;
// start[j], iown[j]: interior box j is a top, the input box at it.
__global__ void recon_nodes_kernel(int64_t ni, const uint64_t *ikeys, int64_t n_in, const uint64_t *keys, const int *top,
                                   int64_t *dst, int64_t *own, int64_t *iown, unsigned char *start, uint64_t *leaf_key,
                                   int *id) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * ni + n_in) return;
  id[e] = (int)e;
  if (e >= 8 * ni) {
    const int64_t b = e - 8 * ni;
    const bool leaf = top[b] == key_level(keys[b]) && find_sorted(ikeys, ni, keys[b]) < 0;
    leaf_key[e] = leaf ? keys[b] : ~0ull;
    dst[e] = -1;
    return;
  }
  const int64_t j = e >> 3;
  const uint64_t k = ikeys[j];
  const int n = key_level(k), c = (int)(e & 7);
  const uint64_t ck = make_key(n + 1, 2 * key_x(k) + (c >> 2), 2 * key_y(k) + ((c >> 1) & 1), 2 * key_z(k) + (c & 1));
  const int64_t p = find_sorted(ikeys, ni, ck);
  dst[e] = p >= 0 ? p : -1;
  own[e] = p >= 0 ? -1 : find_sorted(keys, n_in, ck);
  leaf_key[e] = p >= 0 ? ~0ull : ck;
  if (c == 0) {
    const int64_t b = find_sorted(keys, n_in, k);
    iown[j] = b;
    start[j] = b >= 0 && top[b] == n;
  }
}

// One or two functions on the same boxes (blockIdx.y): their input, the sums on the interior boxes, the leaves.
struct SumDownSets {
  SumDown f[2];
  double *r[2];
};
__device__ __forceinline__ const double *box_coeffs(const SumDown &f, int64_t b, int k3) {
  if (b >= 0 && f.row) b = f.row[b];
  return b >= 0 ? f.coeffs + b * k3 : nullptr;
}

// The tops that are leaves, copied to their places.
__global__ void copy_tops_kernel(int64_t n_in, int64_t base, int k3, const int64_t *dst,
                                 const __grid_constant__ SumDownSets sets) {
  const int64_t b = blockIdx.x, t = dst[base + b];
  if (t == -1) return;
  const SumDown f = blockIdx.y ? sets.f[1] : sets.f[0];
  const double *c = box_coeffs(f, b, k3);
  double *o = f.out + (-2 - t) * k3;
  for (int e = threadIdx.x; e < k3; e += blockDim.x) o[e] = c ? c[e] : 0.0;
}

// One CTA per interior box of one level (j0 + blockIdx.x): what it was passed plus its own input coefficients,
// to its eight children by the two-scale relation; a leaf child adds its own input coefficients.
__global__ void pass_down_kernel(int k, int64_t j0, const int64_t *iown, const unsigned char *start, const int64_t *dst,
                                 const int64_t *own, const double *Ub, const __grid_constant__ SumDownSets sets) {
  extern __shared__ double sh[];
  __shared__ double *to[8];
  __shared__ const double *add[8];
  const int64_t p = j0 + blockIdx.x;
  const int k3 = k * k * k;
  const SumDown f = blockIdx.y ? sets.f[1] : sets.f[0];
  double *r = blockIdx.y ? sets.r[1] : sets.r[0];
  double *U = sh, *d = U + k * k, *a = d + k3, *b = a + 2 * k3;
  const double *in = box_coeffs(f, iown[p], k3);
  const bool first = start[p];
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) U[e] = Ub[e];
  for (int e = threadIdx.x; e < k3; e += blockDim.x) {
    double v = first ? 0.0 : r[p * k3 + e];
    if (in) v = first ? in[e] : v + in[e];
    d[e] = v;
  }
  if (threadIdx.x < 8) {
    const int64_t t = dst[8 * p + threadIdx.x];
    to[threadIdx.x] = t >= 0 ? r + t * k3 : f.out + (-2 - t) * k3;
    add[threadIdx.x] = box_coeffs(f, own[8 * p + threadIdx.x], k3);
  }
  __syncthreads();
  twoscale::down(k, U, d, a, b, [&](int I, int J, int Lq, double v) {
    const int child = ((I / k) << 2) | ((J / k) << 1) | (Lq / k), e = ((I % k) * k + J % k) * k + Lq % k;
    const double *w = add[child];
    to[child][e] = w ? v + w[e] : v;
  });
}

// ---------------------------------------------------------------- truncate
// Boxes that could hold a merged parent: a box all of whose eight children are leaves or merged parents
// holds the leaf at its low corner.  So leaf i proposes its ancestors as long as it is their low corner,
// each box at most once; *count and the per-level counts of what is written to cand.
__global__ void corner_parents_kernel(int64_t n, const uint64_t *keys, uint64_t *cand, unsigned long long *count,
                                      unsigned long long *level_count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t k = keys[i];
  const int lv = key_level(k);
  int64_t x = key_x(k), y = key_y(k), z = key_z(k);
  for (int m = lv - 1; m >= 0 && !((x | y | z) & 1); --m) {
    x >>= 1;
    y >>= 1;
    z >>= 1;
    cand[atomicAdd(count, 1ull)] = make_key(m, x, y, z);
    atomicAdd(level_count + m, 1ull);
  }
}

// Child c of candidate j (entry 8 j + c): the leaf there, or -2 - (candidate there), or -1.
__global__ void merge_children_kernel(int64_t nc, const uint64_t *cand, int64_t n_in, const uint64_t *keys, int64_t *child) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * nc) return;
  const uint64_t k = cand[e >> 3];
  const int n = key_level(k), c = (int)(e & 7);
  const uint64_t ck = make_key(n + 1, 2 * key_x(k) + (c >> 2), 2 * key_y(k) + ((c >> 1) & 1), 2 * key_z(k) + (c & 1));
  int64_t p = find_sorted(keys, n_in, ck);
  if (p < 0) {
    p = find_sorted(cand, nc, ck);
    p = p >= 0 ? -2 - p : -1;
  }
  child[e] = p;
}

// One CTA per candidate of one level (j0 + blockIdx.x): if its eight children are leaves or merged, S from the
// eight, s = (Ubar^T)^{x3} S and the detail d = S - Ubar^{x3} s; if ||d||_F <= thresh the eight are gone
// (gone: leaves, then candidates), the candidate holds s (pv) and ||d||^2 is kept.  Shared memory: U,
// S (8 k^3) and 4 k^3 with s_smem, else 7 k^3 and S read from the children's rows (k > 12, where S does not fit).
__global__ void truncate_level_kernel(int k, int64_t j0, int64_t n_in, const int64_t *child, const double *coeffs,
                                      double thresh, const double *Ub, int *gone, int *merged, double *d2, double *pv,
                                      int s_smem) {
  extern __shared__ double sh[];
  __shared__ const double *src[8];
  __shared__ int all;
  __shared__ double red[BOX_THREADS / 32];
  const int64_t j = j0 + blockIdx.x;
  const int kk = 2 * k, k3 = k * k * k, kk3 = kk * kk * kk;
  if (threadIdx.x == 0) all = 1;
  __syncthreads();
  if (threadIdx.x < 8) {
    const int64_t c = child[8 * j + threadIdx.x];
    const bool there = c >= 0 || (c <= -2 && merged[-2 - c]);
    src[threadIdx.x] = c >= 0 ? coeffs + c * k3 : (there ? pv + (-2 - c) * k3 : nullptr);
    if (!there) all = 0;
  }
  __syncthreads();
  if (!all) return;
  // S[(I, J, L)] = child (I/k, J/k, L/k)'s coefficient (I%k, J%k, L%k)
  auto s_at = [&](int I, int J, int Lq) {
    return src[((I / k) << 2) | ((J / k) << 1) | (Lq / k)][((I % k) * k + J % k) * k + Lq % k];
  };
  double *U = sh, *S = U + k * k, *a, *b, *sv, *c;  // b also serves the way down (2 k^3), as does a (4 k^3)
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) U[e] = Ub[e];
  if (s_smem) {
    a = S + kk3;
    b = S;
    sv = S + 2 * k3;
    c = S + 3 * k3;
    for (int q = threadIdx.x; q < kk3; q += blockDim.x) S[q] = s_at(q / (kk * kk), (q / kk) % kk, q % kk);
    __syncthreads();
    twoscale::up_first(k, U, S, a);
  } else {
    a = S;
    b = a + 4 * k3;
    sv = b + 2 * k3;
    c = b;
    __syncthreads();
    for (int q = threadIdx.x; q < k * kk * kk; q += blockDim.x) {
      const int jx = q / (kk * kk), J = (q / kk) % kk, Lq = q % kk;
      double t = 0.0;
      for (int i = jx; i >= 0; --i) {
        const double x0 = s_at(i, J, Lq), x1 = s_at(k + i, J, Lq);
        t = fma(U[i * k + jx], ((jx - i) & 1) ? x0 - x1 : x0 + x1, t);
      }
      a[q] = t;
    }
    __syncthreads();
  }
  twoscale::up_rest(k, U, a, b, sv);
  double part = 0.0;
  twoscale::down(k, U, sv, c, a, [&](int I, int J, int Lq, double v) {
    const double dd = s_at(I, J, Lq) - v;
    part = fma(dd, dd, part);
  });
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  __shared__ int merge;
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    merge = sqrt(tot) <= thresh;
    if (merge) {
      merged[j] = 1;
      d2[j] = tot;
    }
  }
  __syncthreads();
  if (!merge) return;
  if (threadIdx.x < 8) {
    const int64_t q = child[8 * j + threadIdx.x];
    gone[q >= 0 ? q : n_in + (-2 - q)] = 1;
  }
  for (int q = threadIdx.x; q < k3; q += blockDim.x) pv[j * k3 + q] = sv[q];
}

// Survivors, entries as gone's (leaves, then candidates), one more entry of zero.
__global__ void keep_flags_kernel(int64_t n_in, int64_t nc, const int *gone, const int *merged, int *keep) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n_in + nc) return;
  keep[i] = i < n_in + nc && !gone[i] && (i < n_in || merged[i - n_in]) ? 1 : 0;
}

// One CTA per entry: a survivor to its place among all survivors in key order, its rank among its own kind
// plus the survivors of the other kind with smaller keys (pos: exclusive sum of keep).
__global__ void emit_kept_kernel(int64_t n_in, int64_t nc, int k3, const uint64_t *keys, const double *coeffs,
                                 const uint64_t *cand, const double *pv, const int *keep, const int *pos, int64_t cap,
                                 uint64_t *okeys, double *ocoeffs) {
  const int64_t i = blockIdx.x;
  if (!keep[i] || pos[n_in + nc] > cap) return;
  const bool leaf = i < n_in;
  const uint64_t key = leaf ? keys[i] : cand[i - n_in];
  const uint64_t *other = leaf ? cand : keys;
  int64_t lo = 0, hi = leaf ? nc : n_in;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (other[mid] < key) lo = mid + 1; else hi = mid;
  }
  const int64_t o = leaf ? (int64_t)pos[i] + pos[n_in + lo] - pos[n_in] : (int64_t)pos[i] - pos[n_in] + pos[lo];
  const double *v = leaf ? coeffs + i * k3 : pv + (i - n_in) * k3;
  if (threadIdx.x == 0) okeys[o] = key;
  for (int e = threadIdx.x; e < k3; e += blockDim.x) ocoeffs[o * k3 + e] = v[e];
}

// Sum of v in a fixed order, one CTA.
__global__ void sum_kernel(int64_t n, const double *v, double *out) {
  __shared__ double red[32];
  double t = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) t += v[i];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double w = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) w += red[q];
    *out = w;
  }
}

inline size_t al(size_t v) { return (v + 255) & ~(size_t)255; }
inline int64_t boxes(int n) { return 1LL << (3 * n); }

// Levels whose applies run as one: from level `first` on to the returned level (exclusive), as long as the bound on
// their records together stays below this.  Coarse levels leave most SMs idle and each apply pays its launches and
// synchronisations; a level with more records than this fills the chip by itself, and beside the others it
// would only add to the scratch (some 150 bytes a record, and the output rows).  Whole levels at k = 6, M = 8, bound
// of 2^16, 2^19, 2^22 records and none: |l| <= 3, 4,096 leaves 27.6, 21.4, 21.4, 21.4 ms; |l| <= 1, 32,768 leaves 14.6,
// 14.0, 14.0, 14.0; 262,144 leaves 79.4, 78.9, 78.1, 78.1; FP64 with |l| <= 3, 32,768 leaves 1044, 1036, 996, 996.
constexpr int64_t NS_GROUP_RECORDS = 1 << 22;
template <class Boxes>
int group_end(const Operator &op, const mra_apply_opts &o, int first, int last, Boxes boxes_in) {
  int m = first + 1;
  while (m < last && apply_max_records(op, o, boxes_in(first, m + 1)) < NS_GROUP_RECORDS) ++m;
  return m;
}

// Options of the per-level applies and of the coarsest level's complete apply.
mra_apply_opts level_opts(const mra_apply_opts &o) { return o; }
mra_apply_opts coarse_opts(const mra_apply_opts &o, int n0) {
  mra_apply_opts c = o;
  c.stencil = MRA_STENCIL_SHELLS;
  c.max_disp = (int)((1LL << n0) - 1);
  return c;
}

// Workspace of mra_apply_ns: dense s^n, S^n (n0 <= n < N, back to back), r ping-pong, Y, Z (of the
// largest group of levels), Ubar, an error word, the levels' keys, the applies' outputs (keys +
// coefficients of Y and of Z / the coarse r), and the largest apply's workspace.
struct NsLayout {
  std::vector<int64_t> first;  // first box of level n among all levels' (n0 <= n <= N)
  std::vector<int> group;      // the levels [n0, group[0]), [group[0], group[1]), ... up to N
  size_t s, S, rA, rB, Yd, Zd, Ub, err, keys, yk, yc, zk, zc, apply, total;
  size_t apply_bytes;
};

NsLayout ns_layout(const Operator &op, const Operator &ns, int N, int n0, const mra_apply_opts &o) {
  NsLayout L{};
  const int k = op.k, kk = 2 * k;
  const size_t k3 = (size_t)k * k * k, kk3 = (size_t)kk * kk * kk;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t at = off;
    off = al(off + (bytes ? bytes : 1));
    return at;
  };
  L.first.assign(N + 1, 0);
  for (int n = n0; n < N; ++n) L.first[n + 1] = L.first[n] + boxes(n);
  const int64_t nt = L.first[N];
  int64_t ng = 0;  // boxes of the largest group
  const mra_apply_opts lo = level_opts(o);
  for (int a = n0; a < N;) {
    const int b = group_end(op, lo, a, N, [&](int x, int y) { return L.first[y] - L.first[x]; });
    L.group.push_back(b);
    ng = std::max(ng, L.first[b] - L.first[a]);
    a = b;
  }
  L.s = take(nt * k3 * 8);
  L.S = take(nt * kk3 * 8);
  L.rA = take(boxes(N - 1) * k3 * 8);
  L.rB = take(boxes(N - 1) * k3 * 8);
  L.Yd = take(ng * kk3 * 8);
  L.Zd = take(ng * k3 * 8);
  L.Ub = take((size_t)kk * k * 8);
  L.err = take(8);
  L.keys = take(nt * 8);
  L.yk = take(ng * 8);
  L.yc = take(ng * kk3 * 8);
  L.zk = take(ng * 8);
  L.zc = take(ng * k3 * 8);
  size_t ab = apply_workspace_bytes(op, coarse_opts(o, n0), boxes(n0));
  ab = std::max(ab, apply_workspace_bytes(op, lo, ng));
  ab = std::max(ab, apply_workspace_bytes(ns, lo, ng));
  L.apply_bytes = ab;
  L.apply = take(ab);
  L.total = off;
  return L;
}

int ns_check(const Operator *op, const Operator *ns, const mra_tree_view *in, int n0, const mra_apply_opts *o,
             int *N_out) {
  if (!op || !ns) return fail(MRA_ERR_ARG, "mra_apply_ns: NULL operator");
  if (!in || !o) return fail(MRA_ERR_ARG, "mra_apply_ns: NULL argument");
  if (ns->k != 2 * op->k || ns->M != op->M || ns->L != op->L)
    return fail(MRA_ERR_ARG, "mra_apply_ns: the second operator is not the non-standard form of the first");
  if (in->k != op->k || in->L != op->L) return fail(MRA_ERR_ARG, "mra_apply_ns: tree k or L differs from the operator");
  if (in->n <= 0 || !in->keys || !in->coeffs) return fail(MRA_ERR_ARG, "mra_apply_ns: empty input tree");
  int N = -1;
  for (int n = 1; n <= 10; ++n)
    if (in->n == boxes(n)) N = n;
  if (N < 0) return fail(MRA_ERR_ARG, "mra_apply_ns: %lld boxes is not a whole level 1..10", (long long)in->n);
  if (n0 < 0 || n0 >= N) return fail(MRA_ERR_ARG, "mra_apply_ns: coarsest level %d outside 0..%d", n0, N - 1);
  if (n0 < op->min_level || N - 1 > op->max_level || n0 < ns->min_level || N - 1 > ns->max_level)
    return fail(MRA_ERR_ARG, "mra_apply_ns: levels %d..%d outside the operators' tables", n0, N - 1);
  if (o->precision != MRA_PREC_FP64 && o->precision != MRA_PREC_SPLIT_BF16)
    return fail(MRA_ERR_ARG, "mra_apply_ns: unknown precision %d", o->precision);
  if (o->precision == MRA_PREC_SPLIT_BF16 && (o->pieces < 2 || o->pieces > 3))
    return fail(MRA_ERR_ARG, "mra_apply_ns: pieces must be 2 or 3");
  if (o->dest_hi != 0) return fail(MRA_ERR_ARG, "mra_apply_ns: no destination range in the non-standard form");
  if (o->precision == MRA_PREC_SPLIT_BF16 && ns->k > MRA_MAX_K)
    return fail(MRA_ERR_UNSUPPORTED, "mra_apply_ns: order 2k=%d is applied in FP64 only (split precision to %d)",
                ns->k, MRA_MAX_K);
  if (o->screen != MRA_SCREEN_NONE && o->screen != MRA_SCREEN_NORM)
    return fail(MRA_ERR_ARG, "mra_apply_ns: screen must be MRA_SCREEN_NONE or MRA_SCREEN_NORM");
  if (o->screen == MRA_SCREEN_NORM && !(o->tau >= 0.0)) return fail(MRA_ERR_ARG, "mra_apply_ns: tau must be >= 0");
  if (o->stencil != MRA_STENCIL_SHELLS && o->stencil != MRA_STENCIL_NEAREST)
    return fail(MRA_ERR_ARG, "mra_apply_ns: unknown stencil %d", o->stencil);
  const int D = o->stencil == MRA_STENCIL_NEAREST ? 1 : o->max_disp;
  if (D < 0 || D > ns->max_disp || D > op->max_disp)
    return fail(MRA_ERR_ARG, "mra_apply_ns: max_disp %d outside the operators' range", D);
  if ((1LL << n0) - 1 > op->max_disp)
    return fail(MRA_ERR_ARG, "mra_apply_ns: the complete level-%d apply needs an operator with max_disp >= %lld", n0,
                (long long)((1LL << n0) - 1));
  *N_out = N;
  return MRA_OK;
}

}  // namespace

}  // namespace mra

using namespace mra;

extern "C" int mra_operator_ns_create(const mra_operator *h, int max_disp, mra_operator **out, void *stream) {
  const Operator *op = reinterpret_cast<const Operator *>(h);
  if (!op || !out) return fail(MRA_ERR_ARG, "mra_operator_ns_create: NULL argument");
  *out = nullptr;
  if (2 * op->k > MRA_MAX_NS_K)
    return fail(MRA_ERR_ARG, "mra_operator_ns_create: 2k=%d above %d", 2 * op->k, MRA_MAX_NS_K);
  if (op->max_level <= op->min_level)
    return fail(MRA_ERR_ARG, "mra_operator_ns_create: the operator needs at least two levels");
  if (max_disp < 0) return fail(MRA_ERR_ARG, "mra_operator_ns_create: max_disp < 0");
  cudaStream_t s = (cudaStream_t)stream;
  Operator *ns = new Operator();
  auto bail = [&](int code) {
    free_operator(ns);
    return code;
  };
  ns->kernel = op->kernel;
  ns->non_standard = true;
  ns->mu = op->mu;
  ns->M = op->M;
  ns->k = 2 * op->k;
  ns->L = op->L;
  ns->min_level = op->min_level;
  ns->max_level = op->max_level - 1;
  ns->max_disp = max_disp;
  ns->h_fit = op->h_fit;
  ns->s_lo = op->s_lo;
  ns->fit_err = op->fit_err;
  ns->r_lo = op->r_lo;
  ns->r_hi = op->r_hi;
  ns->c = op->c;
  ns->t = op->t;
  std::vector<int> Dabs(20, 0);
  std::vector<int64_t> off_abs(20, -1);
  int64_t nb = 0;
  for (int n = ns->min_level; n <= ns->max_level; ++n) {
    const int D = (int)std::min<int64_t>(max_disp, (1LL << n) - 1);
    if (2 * D + 1 > op->D[n + 1 - op->min_level])
      return bail(fail(MRA_ERR_ARG, "mra_operator_ns_create: level %d needs the operator's max_disp >= %d", n + 1,
                       2 * D + 1));
    Dabs[n] = D;
    off_abs[n] = nb;
    ns->D.push_back(D);
    ns->level_off.push_back(nb);
    nb += (int64_t)ns->M * (2 * D + 1);
  }
  ns->n_blocks = nb;
  const size_t kk2 = (size_t)ns->k * ns->k;
  if (cudaMalloc((void **)&ns->d_c, ns->M * 8) != cudaSuccess || cudaMalloc((void **)&ns->d_t, ns->M * 8) != cudaSuccess ||
      cudaMalloc((void **)&ns->d_R, nb * kk2 * 8) != cudaSuccess || cudaMalloc((void **)&ns->d_N, nb * 8) != cudaSuccess ||
      cudaMalloc((void **)&ns->d_D, 20 * sizeof(int)) != cudaSuccess ||
      cudaMalloc((void **)&ns->d_level_off, 20 * sizeof(int64_t)) != cudaSuccess)
    return bail(fail(MRA_ERR_CUDA, "mra_operator_ns_create: cudaMalloc failed"));
  cudaError_t e = cudaMemcpyAsync(ns->d_c, ns->c.data(), ns->M * 8, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ns->d_t, ns->t.data(), ns->M * 8, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ns->d_D, Dabs.data(), 20 * sizeof(int), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ns->d_level_off, off_abs.data(), 20 * sizeof(int64_t), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    const int most = 2 * *std::max_element(ns->D.begin(), ns->D.end()) + 1;
    ns_blocks_kernel<<<counted(dim3((unsigned)(ns->M * most), (unsigned)ns->D.size())), 256, 0, s>>>(
        op->k, ns->M, ns->min_level, ns->d_D, ns->d_level_off, op->d_D, op->d_level_off, op->d_R, ns->d_R);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    block_norms_kernel<<<counted((unsigned)((nb + 7) / 8)), 256, 0, s>>>(nb, (int)kk2, ns->d_R, ns->d_N);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return bail(fail(MRA_ERR_CUDA, "mra_operator_ns_create: %s", cudaGetErrorString(e)));
  {  // parity components of the blocks, for the FP64 path
    int rc = f64_parity_build(*ns, s);
    if (rc != MRA_OK) return bail(rc);
  }
  if (ns->k <= MRA_MAX_K) {  // BF16 pieces of the 2k blocks for the tensor-core path
    int rc = split_blocks_build(*ns, s);
    if (rc != MRA_OK) return bail(rc);
  }
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return bail(fail(MRA_ERR_CUDA, "mra_operator_ns_create: %s", cudaGetErrorString(e)));
  *out = reinterpret_cast<mra_operator *>(ns);
  return MRA_OK;
}

extern "C" int mra_apply_ns_workspace_size(const mra_operator *h, const mra_operator *hns, const mra_tree_view *in,
                                           int n0, const mra_apply_opts *o, size_t *bytes) {
  const Operator *op = reinterpret_cast<const Operator *>(h);
  const Operator *ns = reinterpret_cast<const Operator *>(hns);
  if (!bytes) return fail(MRA_ERR_ARG, "mra_apply_ns_workspace_size: NULL bytes");
  int N = 0;
  int rc = ns_check(op, ns, in, n0, o, &N);
  if (rc) return rc;
  *bytes = ns_layout(*op, *ns, N, n0, *o).total;
  return MRA_OK;
}

extern "C" int mra_apply_ns(const mra_operator *h, const mra_operator *hns, const mra_tree_view *in, int n0,
                            const mra_apply_opts *o, mra_tree_view *out, void *workspace, size_t workspace_bytes,
                            mra_apply_stats *stats, void *stream) {
  const Operator *op = reinterpret_cast<const Operator *>(h);
  const Operator *ns = reinterpret_cast<const Operator *>(hns);
  int N = 0;
  int rc = ns_check(op, ns, in, n0, o, &N);
  if (rc) return rc;
  if (!out || !out->keys || !out->coeffs || out->k != op->k)
    return fail(MRA_ERR_ARG, "mra_apply_ns: output view missing or of another k");
  if (out->cap < in->n) {
    out->n = in->n;
    return fail(MRA_ERR_CAPACITY, "mra_apply_ns: output capacity %lld < %lld", (long long)out->cap,
                (long long)in->n);
  }
  const NsLayout Lw = ns_layout(*op, *ns, N, n0, *o);
  if (!workspace || workspace_bytes < Lw.total)
    return fail(MRA_ERR_CAPACITY, "mra_apply_ns: workspace of %zu bytes < %zu needed", workspace_bytes, Lw.total);
  cudaStream_t s = (cudaStream_t)stream;
  char *w = (char *)workspace;
  const int k = op->k, kk = 2 * k;
  const int k3 = k * k * k, kk3 = kk * kk * kk;
  double *Ub = (double *)(w + Lw.Ub);
  int *d_err = (int *)(w + Lw.err);
  uint64_t *keys = (uint64_t *)(w + Lw.keys);
  // Ubar[(c,i)][j] = U^(c)[i][j]
  std::vector<double> U(2 * k * k), Ubh(2 * k * k);
  two_scale(k, U.data());
  for (int c = 0; c < 2; ++c)
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < k; ++j) Ubh[(c * k + i) * k + j] = U[c * k * k + i * k + j];
  MRA_CUDA_TRY(cudaMemcpyAsync(Ub, Ubh.data(), Ubh.size() * 8, cudaMemcpyHostToDevice, s));
  MRA_CUDA_TRY(cudaMemsetAsync(d_err, 0, sizeof(int), s));
  check_uniform_kernel<<<counted((unsigned)((in->n + 255) / 256)), 256, 0, s>>>(N, in->n, in->keys, d_err);
  MRA_CUDA_TRY(cudaGetLastError());
  int herr = 0;
  MRA_CUDA_TRY(cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (herr) return fail(MRA_ERR_ARG, "mra_apply_ns: the input is not every box of level %d in key order", N);

  // ---- compress: S^n and s^n for n = N-1 .. n0
  const size_t sh_c = up_smem(k), sh_d = down_smem(k);
  MRA_CUDA_TRY(cudaFuncSetAttribute(compress_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BOX_SMEM));
  MRA_CUDA_TRY(cudaFuncSetAttribute(sum_down_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BOX_SMEM));
  double *s_all = (double *)(w + Lw.s), *S_all = (double *)(w + Lw.S);
  for (int n = N - 1; n >= n0; --n) {
    const double *fine = n == N - 1 ? in->coeffs : s_all + Lw.first[n + 1] * k3;
    compress_kernel<<<counted((unsigned)boxes(n)), BOX_THREADS, sh_c, s>>>(k, n, fine, Ub, S_all + Lw.first[n] * kk3,
                                                                   s_all + Lw.first[n] * k3);
    MRA_CUDA_TRY(cudaGetLastError());
    level_keys_kernel<<<counted((unsigned)((boxes(n) + 255) / 256)), 256, 0, s>>>(n, boxes(n), keys + Lw.first[n]);
    MRA_CUDA_TRY(cudaGetLastError());
  }

  mra_apply_stats acc{};
  auto add_stats = [&](const mra_apply_stats &st) {
    acc.pairs += st.pairs;
    acc.terms_kept += st.terms_kept;
    acc.terms_screened += st.terms_screened;
    acc.terms_issued += st.terms_issued;
    acc.sources_truncated += st.sources_truncated;
    acc.skipped_bound += st.skipped_bound;
    acc.kernel_ms += st.kernel_ms;
    acc.main_kernel_ms += st.main_kernel_ms;
    acc.mma_passes += st.mma_passes;
    acc.kernel = st.kernel;
    acc.algo_flops += st.algo_flops;
    for (int q = 0; q <= MRA_MAX_LEVEL; ++q) {
      acc.level_sources[q] += st.level_sources[q];
      acc.level_terms_kept[q] += st.level_terms_kept[q];
    }
  };
  void *aws = w + Lw.apply;
  // one apply on every box of the levels [a, b); *dense: its rows in the boxes' order, which is its own output
  // when every box has a row (both are in key order), else scattered into the zeroed array
  auto levels_apply = [&](const Operator &opx, int a, int b, double *coeffs, const mra_apply_opts &oo,
                          uint64_t *okeys, double *ocoeffs, double *zeroed, double **dense) -> int {
    const int64_t nbx = Lw.first[b] - Lw.first[a];
    const int rowlen = opx.k * opx.k * opx.k;
    mra_tree_view vin{nbx, nbx, keys + Lw.first[a], coeffs, opx.k, opx.L};
    mra_tree_view vout{0, nbx, okeys, ocoeffs, opx.k, opx.L};
    mra_apply_stats st{};
    int rc2 = apply_run(opx, vin, oo, vout, aws, Lw.apply_bytes, &st, s);
    if (rc2 != MRA_OK) return rc2;
    add_stats(st);
    *dense = ocoeffs;
    if (vout.n == nbx) return MRA_OK;
    *dense = zeroed;
    MRA_CUDA_TRY(cudaMemsetAsync(zeroed, 0, (size_t)nbx * rowlen * 8, s));
    if (vout.n > 0) {
      scatter_levels_kernel<<<counted((unsigned)vout.n), 128, 0, s>>>(vout.n, okeys, ocoeffs, rowlen, a, zeroed);
      MRA_CUDA_TRY(cudaGetLastError());
    }
    return MRA_OK;
  };
  uint64_t *yk = (uint64_t *)(w + Lw.yk), *zk = (uint64_t *)(w + Lw.zk);
  double *yc = (double *)(w + Lw.yc), *zc = (double *)(w + Lw.zc);
  double *rcur = (double *)(w + Lw.rA), *rnext = (double *)(w + Lw.rB);

  // ---- coarsest level: T^{n0} with every displacement
  double *r0 = nullptr, *Y = nullptr, *Z = nullptr;
  rc = levels_apply(*op, n0, n0 + 1, s_all, coarse_opts(*o, n0), zk, zc, (double *)(w + Lw.Zd), &r0);
  if (rc != MRA_OK) return rc;
  MRA_CUDA_TRY(cudaMemcpyAsync(rcur, r0, (size_t)boxes(n0) * k3 * 8, cudaMemcpyDeviceToDevice, s));
  // ---- levels n0 .. N-1: their applies do not depend on one another, so the levels of a group in one apply each
  int a = n0;
  for (const int b : Lw.group) {
    rc = levels_apply(*ns, a, b, S_all + Lw.first[a] * kk3, level_opts(*o), yk, yc, (double *)(w + Lw.Yd), &Y);
    if (rc != MRA_OK) return rc;
    rc = levels_apply(*op, a, b, s_all + Lw.first[a] * k3, level_opts(*o), zk, zc, (double *)(w + Lw.Zd), &Z);
    if (rc != MRA_OK) return rc;
    for (int n = a; n < b; ++n) {
      double *fine = n == N - 1 ? out->coeffs : rnext;
      const int64_t at = Lw.first[n] - Lw.first[a];
      sum_down_kernel<<<counted((unsigned)boxes(n)), BOX_THREADS, sh_d, s>>>(k, n, rcur, Z + at * k3, Y + at * kk3, Ub, fine);
      MRA_CUDA_TRY(cudaGetLastError());
      std::swap(rcur, rnext);
    }
    a = b;
  }
  MRA_CUDA_TRY(cudaMemcpyAsync(out->keys, in->keys, (size_t)in->n * 8, cudaMemcpyDeviceToDevice, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  out->n = in->n;
  out->L = op->L;
  if (stats) {
    acc.n_in = in->n;
    acc.n_out = in->n;
    *stats = acc;
  }
  return MRA_OK;
}

// ---------------------------------------------------------------- adaptive trees
// The non-standard form apply on an adaptive tree (leaves of a complete octree, every leaf
// deeper than n0).  Sources of level n are the interior nodes I_n (S = children, s = filter);
// the result tree starts with every box of level n0 (r = T^{n0} s^{n0}, every displacement)
// and at each level refines the nodes in the halo of the level's sources -- every box an
// unscreened apply reaches, |l|_inf <= D (children get Ubar^{x3} (r_p - Z_p) + Y_p, absent
// rows of screened applies as zero); the other nodes, and every node of the deepest leaf
// level, are the result's leaves.  The halo keeps every later level's targets inside the
// result: a target's parent lies in the previous level's halo.
// The tree depends on the keys alone and the levels' applies on one another's results not at all, so
// the structure is made first (two sorts over all levels) and then the applies run: the
// coarsest level's, and T2k and T over the sources of a group of levels (see group_end).  Level by level, each
// with two applies of few boxes, the launches, their synchronisations and the idle SMs took longer than
// the kernels' work.
extern "C" int mra_apply_ns_tree(const mra_operator *h, const mra_operator *hns, const mra_tree_view *in, int n0,
                                 const mra_apply_opts *o, mra_tree_view *out, mra_apply_stats *stats, void *stream) {
  const Operator *op = reinterpret_cast<const Operator *>(h);
  const Operator *ns = reinterpret_cast<const Operator *>(hns);
  if (!op || !ns || !in || !o || !out) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: NULL argument");
  if (ns->k != 2 * op->k || ns->M != op->M || ns->L != op->L)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: the second operator is not the non-standard form of the first");
  if (in->k != op->k || in->L != op->L) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: tree k or L differs");
  if (in->n <= 0 || !in->keys || !in->coeffs) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: empty input tree");
  if (in->n >= (1LL << 31)) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: more than 2^31 leaves");
  if (out->k != op->k || out->cap < 0 || (out->cap > 0 && (!out->keys || !out->coeffs)))
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: bad output view");
  if (o->dest_hi != 0) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: no destination range in the non-standard form");
  if (o->precision != MRA_PREC_FP64 && o->precision != MRA_PREC_SPLIT_BF16)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: unknown precision %d", o->precision);
  if (o->precision == MRA_PREC_SPLIT_BF16 && (o->pieces < 2 || o->pieces > 3))
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: pieces must be 2 or 3");
  if (o->screen != MRA_SCREEN_NONE && o->screen != MRA_SCREEN_NORM)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: screen must be MRA_SCREEN_NONE or MRA_SCREEN_NORM");
  if (o->stencil != MRA_STENCIL_SHELLS && o->stencil != MRA_STENCIL_NEAREST)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: unknown stencil %d", o->stencil);
  const int D = o->stencil == MRA_STENCIL_NEAREST ? 1 : o->max_disp;
  if (D < 0 || D > ns->max_disp || D > op->max_disp)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: max_disp %d outside the operators' range", D);
  if (n0 < 0 || (1LL << n0) - 1 > op->max_disp)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: the complete level-%d apply needs max_disp >= %lld", n0,
                (long long)((1LL << n0) - 1));
  cudaStream_t s = (cudaStream_t)stream;
  const int k = op->k, kk = 2 * k, k3 = k * k * k;
  const int64_t n_leaf = in->n;
  std::vector<void *> held;  // stream-ordered allocations, released on every return
  struct Release {
    std::vector<void *> &v;
    cudaStream_t s;
    ~Release() {
      for (void *p : v) cudaFreeAsync(p, s);
      cudaStreamSynchronize(s);
    }
  } release{held, s};
  auto dalloc = [&](size_t bytes) -> void * {
    void *p = nullptr;
    if (pool_malloc(&p, bytes ? bytes : 1, s) != cudaSuccess) return nullptr;
    held.push_back(p);
    return p;
  };
  auto drop = [&](void *p) {  // release one allocation early
    auto it = std::find(held.begin(), held.end(), p);
    if (it != held.end()) {
      cudaFreeAsync(p, s);
      held.erase(it);
    }
  };
#define NS_ALLOC(var, type, count)                                                              \
  type *var = (type *)dalloc((size_t)(count) * sizeof(type));                                   \
  if (!var) return fail(MRA_ERR_CUDA, "mra_apply_ns_tree: out of device memory (%s)", #var);

  // ---- leaves: order, depth
  NS_ALLOC(d_int, int, 4);
  MRA_CUDA_TRY(cudaMemsetAsync(d_int, 0, 4 * sizeof(int), s));
  leaf_check_kernel<<<counted((unsigned)((n_leaf + 255) / 256)), 256, 0, s>>>(n_leaf, in->keys, n0, d_int, d_int + 1);
  MRA_CUDA_TRY(cudaGetLastError());
  int hint[2] = {0, 0};
  MRA_CUDA_TRY(cudaMemcpyAsync(hint, d_int, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (hint[0]) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: leaves must be sorted, unique and deeper than level %d", n0);
  const int Nmax = hint[1];
  if (n0 < op->min_level || Nmax - 1 > op->max_level || n0 < ns->min_level || Nmax - 1 > ns->max_level)
    return fail(MRA_ERR_ARG, "mra_apply_ns_tree: levels %d..%d outside the operators' tables", n0, Nmax - 1);
  NS_ALLOC(Ub, double, kk * k);
  std::vector<double> U(2 * k * k), Ubh(2 * k * k);
  two_scale(k, U.data());
  for (int c = 0; c < 2; ++c)
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < k; ++j) Ubh[(c * k + i) * k + j] = U[c * k * k + i * k + j];
  MRA_CUDA_TRY(cudaMemcpyAsync(Ub, Ubh.data(), Ubh.size() * 8, cudaMemcpyHostToDevice, s));

  // ---- interior nodes of every level: the leaves' ancestors, sorted and unique, all levels in
  // one sort (keys order by level first, so each level is one range)
  std::vector<uint64_t *> Ik(Nmax + 1, nullptr);
  std::vector<int64_t> In(Nmax + 1, 0), off_int(21, 0);
  {
    const int nlev = std::max(Nmax - n0, 1);
    if (n_leaf * nlev >= (int64_t)INT32_MAX) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: too many leaves x levels");
    const int64_t na = n_leaf * nlev;
    NS_ALLOC(anc, uint64_t, na);
    NS_ALLOC(anc_s, uint64_t, na);
    NS_ALLOC(d_nsel, int64_t, 1);
    NS_ALLOC(d_off, int64_t, 21);
    size_t t1 = 0, t2 = 0;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(nullptr, t1, anc, anc_s, (int)na, 0, 64, s));
    MRA_CUDA_TRY(cub::DeviceSelect::Unique(nullptr, t2, anc_s, anc, d_nsel, (int)na, s));
    size_t tb = std::max(t1, t2);
    NS_ALLOC(tmp, unsigned char, tb);
    ancestor_kernel<<<counted((unsigned)((na + 255) / 256)), 256, 0, s>>>(n_leaf, in->keys, n0, nlev, anc);
    MRA_CUDA_TRY(cudaGetLastError());
    size_t tt = tb;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(tmp, tt, anc, anc_s, (int)na, 0, 64, s));
    tt = tb;
    MRA_CUDA_TRY(cub::DeviceSelect::Unique(tmp, tt, anc_s, anc, d_nsel, (int)na, s));
    level_offsets_kernel<<<counted(1), 32, 0, s>>>(anc, d_nsel, d_off);
    MRA_CUDA_TRY(cudaGetLastError());
    std::vector<int64_t> &off = off_int;
    MRA_CUDA_TRY(cudaMemcpyAsync(off.data(), d_off, 21 * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MRA_CUDA_TRY(cudaStreamSynchronize(s));
    for (int n = n0; n < Nmax; ++n) {
      Ik[n] = anc + off[n];
      In[n] = off[n + 1] - off[n];
    }
    drop(anc_s);
    drop(tmp);
  }
  if (In[n0] != boxes(n0)) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: level %d is not complete", n0);

  const int64_t n_int = off_int[Nmax] - off_int[n0];

  // ---- the halo of every level's sources, sorted and unique, all levels in one sort: the boxes that are
  // refined.  It fixes the whole result tree: the children of the halo boxes are the next level's halo
  // boxes and the result's leaves, so every size and place is known before any apply runs.
  const int64_t w3 = (int64_t)(2 * D + 1) * (2 * D + 1) * (2 * D + 1);
  const int64_t nh_all = n_int * w3;
  std::vector<int64_t> hoff(21, 0);
  NS_ALLOC(d_hoff, int64_t, 21);
  uint64_t *hk = nullptr;
  {
    NS_ALLOC(hal, uint64_t, nh_all);
    NS_ALLOC(hal_s, uint64_t, nh_all);
    NS_ALLOC(d_nh, int64_t, 1);
    size_t t1 = 0, t2 = 0;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(nullptr, t1, hal, hal_s, nh_all, 0, 64, s));
    MRA_CUDA_TRY(cub::DeviceSelect::Unique(nullptr, t2, hal_s, hal, d_nh, nh_all, s));
    const size_t tb = std::max(t1, t2);
    NS_ALLOC(tmph, unsigned char, tb);
    halo_kernel<<<counted((unsigned)((nh_all + 255) / 256)), 256, 0, s>>>(n_int, Ik[n0], D, hal);
    MRA_CUDA_TRY(cudaGetLastError());
    size_t tt = tb;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(tmph, tt, hal, hal_s, nh_all, 0, 64, s));
    tt = tb;
    MRA_CUDA_TRY(cub::DeviceSelect::Unique(tmph, tt, hal_s, hal, d_nh, nh_all, s));
    level_offsets_kernel<<<counted(1), 32, 0, s>>>(hal, d_nh, d_hoff);
    MRA_CUDA_TRY(cudaGetLastError());
    MRA_CUDA_TRY(cudaMemcpyAsync(hoff.data(), d_hoff, 21 * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MRA_CUDA_TRY(cudaStreamSynchronize(s));
    drop(hal_s);
    drop(tmph);
    hk = hal;
  }
  const int64_t nh = hoff[Nmax];  // halo boxes, levels n0 .. Nmax-1
  if (hoff[n0 + 1] - hoff[n0] != boxes(n0))
    return fail(MRA_ERR_NUMERIC, "mra_apply_ns_tree: the halo of level %d is not the whole level", n0);
  if (8 * nh >= (int64_t)INT32_MAX) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: too many result boxes");
  const int64_t nout = 8 * nh - (nh - boxes(n0));
  mra_apply_stats acc{};
  acc.n_in = n_leaf;
  acc.n_out = nout;
  if (nout > out->cap) {
    out->L = op->L;
    out->n = nout;
    if (stats) *stats = acc;
    return fail(MRA_ERR_CAPACITY, "mra_apply_ns_tree: %lld result leaves, capacity %lld", (long long)nout,
                (long long)out->cap);
  }
  NS_ALLOC(dst, int64_t, 8 * nh);
  const uint64_t *leaf_sorted = nullptr;
  const int *leaf_id = nullptr;
  {
    NS_ALLOC(lk, uint64_t, 8 * nh);
    NS_ALLOC(lks, uint64_t, 8 * nh);
    NS_ALLOC(id, int, 8 * nh);
    NS_ALLOC(ids, int, 8 * nh);
    size_t tb = 0;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, lk, lks, id, ids, (int)(8 * nh), 0, 64, s));
    NS_ALLOC(tmp, unsigned char, tb);
    NS_ALLOC(found, unsigned long long, 1);
    MRA_CUDA_TRY(cudaMemsetAsync(found, 0, 8, s));
    halo_children_kernel<<<counted((unsigned)((8 * nh + 255) / 256)), 256, 0, s>>>(nh, hk, d_hoff, Nmax, dst, lk, id, found);
    MRA_CUDA_TRY(cudaGetLastError());
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortPairs(tmp, tb, lk, lks, id, ids, (int)(8 * nh), 0, 64, s));
    unsigned long long hfound = 0;
    MRA_CUDA_TRY(cudaMemcpyAsync(&hfound, found, 8, cudaMemcpyDeviceToHost, s));
    MRA_CUDA_TRY(cudaStreamSynchronize(s));
    if ((int64_t)hfound != nh - boxes(n0))  // every halo box is a child of one of the level above
      return fail(MRA_ERR_NUMERIC, "mra_apply_ns_tree: a halo box lies outside the result tree");
    for (void *p : {(void *)lk, (void *)id, (void *)tmp, (void *)found}) drop(p);
    leaf_sorted = lks;
    leaf_id = ids;
  }

  // ---- compress, from the deepest interior level up; all levels' S and s back to back in key order
  const size_t sh_c = up_smem(k), sh_d = down_smem(k);
  const int kk3 = kk * kk * kk;
  MRA_CUDA_TRY(cudaFuncSetAttribute(compress_tree_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BOX_SMEM));
  MRA_CUDA_TRY(cudaFuncSetAttribute(sum_down_tree_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BOX_SMEM));
  NS_ALLOC(S_all, double, n_int * kk3);
  NS_ALLOC(s_all, double, n_int * k3);
  auto first = [&](int n) { return off_int[n] - off_int[n0]; };
  for (int n = Nmax - 1; n >= n0; --n) {
    const bool deeper = n + 1 < Nmax;
    compress_tree_kernel<<<counted((unsigned)In[n]), BOX_THREADS, sh_c, s>>>(
        k, n, Ik[n], In[n], in->keys, in->coeffs, n_leaf, deeper ? Ik[n + 1] : nullptr,
        deeper ? s_all + first(n + 1) * k3 : nullptr, deeper ? In[n + 1] : 0, Ub, S_all + first(n) * kk3,
        s_all + first(n) * k3, d_int);
    MRA_CUDA_TRY(cudaGetLastError());
  }
  MRA_CUDA_TRY(cudaMemcpyAsync(hint, d_int, sizeof(int), cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (hint[0]) return fail(MRA_ERR_ARG, "mra_apply_ns_tree: the leaves are not a complete octree");
  // the input has been read: the result may be written (also where it shares the input's buffers)
  leaf_places_kernel<<<counted((unsigned)((nout + 255) / 256)), 256, 0, s>>>(nout, leaf_sorted, leaf_id, dst, out->keys);
  MRA_CUDA_TRY(cudaGetLastError());

  // one library apply of opx on the interior boxes [b0, b1) (their coefficients at coeffs): its rows appended
  // at okeys/ocoeffs + *nout_rows
  auto run_apply = [&](const Operator &opx, int64_t b0, int64_t b1, double *coeffs, const mra_apply_opts &oo, int64_t rows_cap,
                       uint64_t *okeys, double *ocoeffs, int64_t *nout_rows) -> int {
    const int64_t rl = (int64_t)opx.k * opx.k * opx.k;
    const size_t wb = apply_workspace_bytes(opx, oo, b1 - b0);
    void *ws = dalloc(wb);
    if (!ws) return fail(MRA_ERR_CUDA, "mra_apply_ns_tree: out of device memory");
    mra_tree_view vin{b1 - b0, b1 - b0, Ik[n0] + b0, coeffs + b0 * rl, opx.k, opx.L};
    mra_tree_view vout{0, rows_cap - *nout_rows, okeys + *nout_rows, ocoeffs + *nout_rows * rl, opx.k, opx.L};
    mra_apply_stats st{};
    const int rc2 = apply_run(opx, vin, oo, vout, ws, wb, &st, s);
    drop(ws);
    if (rc2 != MRA_OK) return rc2;
    acc.pairs += st.pairs;
    acc.terms_kept += st.terms_kept;
    acc.terms_screened += st.terms_screened;
    acc.terms_issued += st.terms_issued;
    acc.skipped_bound += st.skipped_bound;
    acc.kernel_ms += st.kernel_ms;
    acc.main_kernel_ms += st.main_kernel_ms;
    acc.mma_passes += st.mma_passes;
    acc.kernel = st.kernel;
    acc.algo_flops += st.algo_flops;
    for (int q = 0; q <= MRA_MAX_LEVEL; ++q) {
      acc.level_sources[q] += st.level_sources[q];
      acc.level_terms_kept[q] += st.level_terms_kept[q];
    }
    *nout_rows += vout.n;
    return MRA_OK;
  };
  // the applies of the levels are independent: the levels of a group in one apply
  auto run_levels = [&](const Operator &opx, double *coeffs, uint64_t *okeys, double *ocoeffs, int64_t *rows) -> int {
    for (int n = n0; n < Nmax;) {
      const int m = group_end(opx, level_opts(*o), n, Nmax, [&](int x, int y) { return first(y) - first(x); });
      const int rc2 = run_apply(opx, first(n), first(m), coeffs, level_opts(*o), nh, okeys, ocoeffs, rows);
      if (rc2 != MRA_OK) return rc2;
      n = m;
    }
    return MRA_OK;
  };

  // ---- coarsest level: every box, T^{n0} with every displacement
  NS_ALLOC(r, double, nh * k3);
  {
    NS_ALLOC(ok, uint64_t, boxes(n0));
    NS_ALLOC(oc, double, boxes(n0) * k3);
    int64_t no = 0;
    const int rc = run_apply(*op, 0, boxes(n0), s_all, coarse_opts(*o, n0), boxes(n0), ok, oc, &no);
    if (rc != MRA_OK) return rc;
    MRA_CUDA_TRY(cudaMemsetAsync(r, 0, (size_t)boxes(n0) * k3 * 8, s));
    if (no > 0) {
      scatter_dense_kernel<<<counted((unsigned)no), 128, 0, s>>>(no, ok, oc, k3, r);  // level n0 is complete: dense order
      MRA_CUDA_TRY(cudaGetLastError());
    }
    drop(ok);
    drop(oc);
  }
  // ---- T2k^n S^n and T^n s^n of every level
  NS_ALLOC(yk, uint64_t, nh);
  NS_ALLOC(yc, double, nh * kk3);
  NS_ALLOC(zk, uint64_t, nh);
  NS_ALLOC(zc, double, nh * k3);
  int64_t ny = 0, nz = 0;
  int rc = run_levels(*ns, S_all, yk, yc, &ny);
  if (rc != MRA_OK) return rc;
  rc = run_levels(*op, s_all, zk, zc, &nz);
  if (rc != MRA_OK) return rc;
  MRA_CUDA_TRY(cudaMemsetAsync(d_int, 0, sizeof(int), s));
  if (ny > 0) targets_in_kernel<<<counted((unsigned)((ny + 255) / 256)), 256, 0, s>>>(ny, yk, hk, nh, d_int);
  if (nz > 0) targets_in_kernel<<<counted((unsigned)((nz + 255) / 256)), 256, 0, s>>>(nz, zk, hk, nh, d_int);
  MRA_CUDA_TRY(cudaGetLastError());
  // ---- down the levels
  NS_ALLOC(yi, int64_t, nh);
  NS_ALLOC(zi, int64_t, nh);
  halo_rows_kernel<<<counted((unsigned)((nh + 255) / 256)), 256, 0, s>>>(nh, hk, yk, ny, zk, nz, yi, zi);
  MRA_CUDA_TRY(cudaGetLastError());
  for (int n = n0; n < Nmax; ++n) {
    const int64_t j0 = hoff[n], nj = hoff[n + 1] - hoff[n];
    if (nj == 0) continue;
    sum_down_tree_kernel<<<counted((unsigned)nj), BOX_THREADS, sh_d, s>>>(k, j0, r, yi, yc, zi, zc, dst, Ub, out->coeffs);
    MRA_CUDA_TRY(cudaGetLastError());
  }
  MRA_CUDA_TRY(cudaMemcpyAsync(hint, d_int, sizeof(int), cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (hint[0]) return fail(MRA_ERR_NUMERIC, "mra_apply_ns_tree: an apply reached a box outside the result tree");
  out->L = op->L;
  out->n = nout;
  if (stats) *stats = acc;
  return MRA_OK;
#undef NS_ALLOC
}


// ---------------------------------------------------------------- reconstruct (host)
namespace mra {

Reconstruct::~Reconstruct() {
  for (void *p : held) cudaFreeAsync(p, s);
}

void *Reconstruct::dalloc(size_t bytes) {
  void *p = nullptr;
  if (pool_malloc(&p, bytes ? bytes : 1, s) != cudaSuccess) return nullptr;
  held.push_back(p);
  return p;
}

void Reconstruct::drop(void *p) {
  auto it = std::find(held.begin(), held.end(), p);
  if (it != held.end()) {
    cudaFreeAsync(p, s);
    held.erase(it);
  }
}

#define RC_GET(var, type, count)                        \
  var = (type *)dalloc((size_t)(count) * sizeof(type)); \
  if (!var) return fail(MRA_ERR_CUDA, "mra_reconstruct: out of device memory (%s)", #var);
#define RC_ALLOC(var, type, count) \
  type *var = nullptr;             \
  RC_GET(var, type, count)

int Reconstruct::plan(int k_, int64_t n, const uint64_t *keys_) {
  k = k_;
  n_in = n;
  keys = keys_;
  const int kk = 2 * k;
  // order and the level ranges of the sorted input
  RC_ALLOC(d_off, int64_t, 22);
  MRA_CUDA_TRY(cudaMemsetAsync(d_off, 0, 22 * 8, s));
  leaf_offsets_kernel<<<counted((unsigned)((n_in + 256) / 256)), 256, 0, s>>>(n_in, keys, d_off, d_off + 21);
  MRA_CUDA_TRY(cudaGetLastError());
  RC_GET(top, int, n_in);
  top_level_kernel<<<counted((unsigned)((n_in + 255) / 256)), 256, 0, s>>>(n_in, keys, top);
  MRA_CUDA_TRY(cudaGetLastError());
  RC_GET(Ub, double, kk * k);
  std::vector<double> U(2 * k * k);
  two_scale(k, U.data());  // [c][i][j]: the rows (c, i) of Ubar in order
  MRA_CUDA_TRY(cudaMemcpyAsync(Ub, U.data(), U.size() * 8, cudaMemcpyHostToDevice, s));
  int64_t off[22];
  MRA_CUDA_TRY(cudaMemcpyAsync(off, d_off, 22 * 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (off[21] == 2) return fail(MRA_ERR_ARG, "mra_reconstruct: level above %d", MRA_MAX_LEVEL);
  if (off[21]) return fail(MRA_ERR_ARG, "mra_reconstruct: keys must be sorted and unique");
  nmin = 0, nmax = MRA_MAX_LEVEL;
  while (off[nmin + 1] == 0) ++nmin;
  while (off[nmax] == n_in) --nmax;
  // The result's tree depends on the keys alone: the interior boxes of all levels (one sort), their children and
  // the tops that stay leaves (one sort for the leaves' order).  Then each level is one kernel that
  // passes its interior boxes' sums down into the next level's or to the leaves' places.
  const int nlev = std::max(nmax - nmin, 1);
  if (n_in * nlev >= (int64_t)INT32_MAX) return fail(MRA_ERR_ARG, "mra_reconstruct: too many boxes x levels");
  const int64_t na = n_in * nlev;
  RC_ALLOC(anc, uint64_t, na);
  RC_ALLOC(iall, uint64_t, na);
  RC_ALLOC(d_info, int64_t, 24);  // offsets of the interior levels, then tops, interior tops, interior boxes
  MRA_CUDA_TRY(cudaMemsetAsync(d_info, 0, 24 * 8, s));
  int64_t *d_ni = d_info + 23;
  interior_all_kernel<<<counted((unsigned)((na + 255) / 256)), 256, 0, s>>>(n_in, keys, top, nmin, nlev, anc);
  MRA_CUDA_TRY(cudaGetLastError());
  {
    size_t tb = 0, t2 = 0;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(nullptr, tb, anc, iall, (int)na, 0, 64, s));
    MRA_CUDA_TRY(cub::DeviceSelect::Unique(nullptr, t2, iall, anc, d_ni, (int)na, s));
    tb = std::max(tb, t2);
    RC_ALLOC(tmp, unsigned char, tb);
    size_t tt = tb;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(tmp, tt, anc, iall, (int)na, 0, 64, s));
    tt = tb;
    MRA_CUDA_TRY(cub::DeviceSelect::Unique(tmp, tt, iall, anc, d_ni, (int)na, s));
    drop(tmp);
  }
  ik = anc;  // the unique interior keys, in key order (so level by level)
  level_offsets_kernel<<<counted(1), 32, 0, s>>>(ik, d_ni, d_info);
  MRA_CUDA_TRY(cudaGetLastError());
  count_tops_kernel<<<counted((unsigned)((n_in + 255) / 256)), 256, 0, s>>>(n_in, keys, top, ik, d_info + 20,
                                                                            (unsigned long long *)(d_info + 21));
  MRA_CUDA_TRY(cudaGetLastError());
  MRA_CUDA_TRY(cudaMemcpyAsync(info, d_info, 24 * 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  drop(iall);
  const int64_t ntop = info[21], itop = info[22];
  ni = info[20];
  nout = 8 * ni - (ni - itop) + (ntop - itop);
  return MRA_OK;
}

int Reconstruct::place(uint64_t *out_keys) {
  const int64_t nn = 8 * ni + n_in;
  if (nn >= (int64_t)INT32_MAX) return fail(MRA_ERR_ARG, "mra_reconstruct: too many boxes in the result");
  RC_GET(dst, int64_t, nn);
  RC_GET(own, int64_t, 8 * ni);
  RC_GET(iown, int64_t, ni);
  RC_GET(start, unsigned char, ni);
  RC_ALLOC(lk, uint64_t, nn);
  RC_ALLOC(lks, uint64_t, nn);
  RC_ALLOC(id, int, nn);
  RC_ALLOC(ids, int, nn);
  size_t tb = 0;
  MRA_CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, lk, lks, id, ids, (int)nn, 0, 64, s));
  RC_ALLOC(tmp, unsigned char, tb);
  recon_nodes_kernel<<<counted((unsigned)((nn + 255) / 256)), 256, 0, s>>>(ni, ik, n_in, keys, top, dst, own, iown, start, lk,
                                                                           id);
  MRA_CUDA_TRY(cudaGetLastError());
  MRA_CUDA_TRY(cub::DeviceRadixSort::SortPairs(tmp, tb, lk, lks, id, ids, (int)nn, 0, 64, s));
  leaf_places_kernel<<<counted((unsigned)((nout + 255) / 256)), 256, 0, s>>>(nout, lks, ids, dst, out_keys);
  MRA_CUDA_TRY(cudaGetLastError());
  return MRA_OK;
}

int Reconstruct::run(int nf, const SumDown *f) {
  const int k3 = k * k * k;
  SumDownSets sets{};
  for (int i = 0; i < nf; ++i) {
    sets.f[i] = f[i];
    RC_GET(sets.r[i], double, ni * k3);
  }
  copy_tops_kernel<<<counted(dim3((unsigned)n_in, (unsigned)nf)), 128, 0, s>>>(n_in, 8 * ni, k3, dst, sets);
  MRA_CUDA_TRY(cudaGetLastError());
  const size_t sh_d = down_smem(k);
  MRA_CUDA_TRY(cudaFuncSetAttribute(pass_down_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BOX_SMEM));
  for (int n = nmin; n < nmax; ++n) {
    const int64_t nj = info[n + 1] - info[n];
    if (nj == 0) continue;
    pass_down_kernel<<<counted(dim3((unsigned)nj, (unsigned)nf)), BOX_THREADS, sh_d, s>>>(k, info[n], iown, start, dst, own, Ub,
                                                                                     sets);
    MRA_CUDA_TRY(cudaGetLastError());
  }
  return MRA_OK;
}
#undef RC_ALLOC
#undef RC_GET

}  // namespace mra

extern "C" int mra_reconstruct(const mra_tree_view *in, mra_tree_view *out, void *stream) {
  if (!in || !out) return fail(MRA_ERR_ARG, "mra_reconstruct: NULL argument");
  if (in->n < 0 || (in->n > 0 && (!in->keys || !in->coeffs))) return fail(MRA_ERR_ARG, "mra_reconstruct: bad input");
  if (in->k < 1 || in->k > MRA_MAX_K) return fail(MRA_ERR_ARG, "mra_reconstruct: k=%d outside 1..%d", in->k, MRA_MAX_K);
  if (in->n >= (1LL << 31)) return fail(MRA_ERR_ARG, "mra_reconstruct: more than 2^31 boxes");
  if (out->k != in->k || out->cap < 0 || (out->cap > 0 && (!out->keys || !out->coeffs)))
    return fail(MRA_ERR_ARG, "mra_reconstruct: bad output view");
  out->L = in->L;
  if (in->n == 0) {
    out->n = 0;
    return MRA_OK;
  }
  cudaStream_t s = (cudaStream_t)stream;
  Reconstruct rec(s);
  int rc = rec.plan(in->k, in->n, in->keys);
  if (rc) return rc;
  if (rec.leaves() > out->cap) {
    out->n = rec.leaves();
    return fail(MRA_ERR_CAPACITY, "mra_reconstruct: %lld leaves, capacity %lld", (long long)out->n, (long long)out->cap);
  }
  if ((rc = rec.place(out->keys)) != MRA_OK) return rc;
  const SumDown f{in->coeffs, nullptr, out->coeffs};
  if ((rc = rec.run(1, &f)) != MRA_OK) return rc;
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  out->n = rec.leaves();
  return MRA_OK;
}


// ---------------------------------------------------------------- truncate (host)
extern "C" int mra_truncate(const mra_tree_view *in, double thresh, mra_tree_view *out, double *err2, void *stream) {
  if (!in || !out) return fail(MRA_ERR_ARG, "mra_truncate: NULL argument");
  if (in->n < 0 || (in->n > 0 && (!in->keys || !in->coeffs))) return fail(MRA_ERR_ARG, "mra_truncate: bad input");
  if (in->k < 1 || in->k > MRA_MAX_K) return fail(MRA_ERR_ARG, "mra_truncate: k=%d outside 1..%d", in->k, MRA_MAX_K);
  if (in->n >= (1LL << 31)) return fail(MRA_ERR_ARG, "mra_truncate: more than 2^31 leaves");
  if (!(thresh >= 0.0)) return fail(MRA_ERR_ARG, "mra_truncate: thresh must be >= 0");
  if (out->k != in->k || out->cap < 0 || (out->cap > 0 && (!out->keys || !out->coeffs)))
    return fail(MRA_ERR_ARG, "mra_truncate: bad output view");
  out->L = in->L;
  if (err2) *err2 = 0.0;
  if (in->n == 0) {
    out->n = 0;
    return MRA_OK;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int k = in->k, kk = 2 * k, k3 = k * k * k;
  const int64_t n_in = in->n;
  std::vector<void *> held;
  struct Release {
    std::vector<void *> &v;
    cudaStream_t s;
    ~Release() {
      for (void *p : v) cudaFreeAsync(p, s);
      cudaStreamSynchronize(s);
    }
  } release{held, s};
  auto dalloc = [&](size_t bytes) -> void * {
    void *p = nullptr;
    if (pool_malloc(&p, bytes ? bytes : 1, s) != cudaSuccess) return nullptr;
    held.push_back(p);
    return p;
  };
#define TR_ALLOC(var, type, count)                                                              \
  type *var = (type *)dalloc((size_t)(count) * sizeof(type));                                   \
  if (!var) return fail(MRA_ERR_CUDA, "mra_truncate: out of device memory (%s)", #var);

  TR_ALLOC(Ub, double, kk * k);
  std::vector<double> U(2 * k * k);
  two_scale(k, U.data());  // [c][i][j]: the rows (c, i) of Ubar in order
  MRA_CUDA_TRY(cudaMemcpyAsync(Ub, U.data(), U.size() * 8, cudaMemcpyHostToDevice, s));
  // The boxes where a merge is possible are known from the keys (their low corner is a leaf's); sorted once,
  // they are worked through from the deepest level up, one kernel per level.
  TR_ALLOC(d_info, int64_t, 44);  // leaf level offsets [0..20], bad [21], candidates [22], per level [23..42]
  MRA_CUDA_TRY(cudaMemsetAsync(d_info, 0, 44 * 8, s));
  leaf_offsets_kernel<<<counted((unsigned)((n_in + 256) / 256)), 256, 0, s>>>(n_in, in->keys, d_info, d_info + 21);
  MRA_CUDA_TRY(cudaGetLastError());
  int64_t info[44];
  MRA_CUDA_TRY(cudaMemcpyAsync(info, d_info, 22 * 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  if (info[21] == 2) return fail(MRA_ERR_ARG, "mra_truncate: level above 19");
  if (info[21]) return fail(MRA_ERR_ARG, "mra_truncate: keys must be sorted and unique");
  // a level-l leaf proposes at most l boxes
  int64_t nc_max = 0;
  for (int l = 0; l < 20; ++l) nc_max += l * (info[l + 1] - info[l]);
  TR_ALLOC(cand0, uint64_t, nc_max);
  corner_parents_kernel<<<counted((unsigned)((n_in + 255) / 256)), 256, 0, s>>>(
      n_in, in->keys, cand0, (unsigned long long *)(d_info + 22), (unsigned long long *)(d_info + 23));
  MRA_CUDA_TRY(cudaGetLastError());
  MRA_CUDA_TRY(cudaMemcpyAsync(info, d_info, 44 * 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t nc = info[22];
  if (n_in + nc >= (int64_t)INT32_MAX) return fail(MRA_ERR_ARG, "mra_truncate: too many boxes");
  TR_ALLOC(cand, uint64_t, nc);
  TR_ALLOC(child, int64_t, 8 * nc);
  TR_ALLOC(flags, int, n_in + 2 * nc);  // gone (leaves, candidates), merged
  TR_ALLOC(d2, double, nc + 1);
  TR_ALLOC(pv, double, nc * k3);
  int *gone = flags, *merged = flags + n_in + nc;
  MRA_CUDA_TRY(cudaMemsetAsync(flags, 0, (size_t)(n_in + 2 * nc) * sizeof(int), s));
  MRA_CUDA_TRY(cudaMemsetAsync(d2, 0, (size_t)(nc + 1) * 8, s));
  if (nc > 0) {
    size_t tb = 0;
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(nullptr, tb, cand0, cand, (int)nc, 0, 62, s));
    TR_ALLOC(tmp, unsigned char, tb);
    MRA_CUDA_TRY(cub::DeviceRadixSort::SortKeys(tmp, tb, cand0, cand, (int)nc, 0, 62, s));
    merge_children_kernel<<<counted((unsigned)((8 * nc + 255) / 256)), 256, 0, s>>>(nc, cand, n_in, in->keys, child);
    MRA_CUDA_TRY(cudaGetLastError());
    // S stays in shared memory up to k = 12 (96 k^3 bytes); above, only the filter's pieces (56 k^3)
    const int s_smem = k <= 12 ? 1 : 0;
    const size_t sh = s_smem ? up_smem(k) : down_smem(k);
    MRA_CUDA_TRY(cudaFuncSetAttribute(truncate_level_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BOX_SMEM));
    int64_t end = nc;
    for (int n = 19; n >= 0; --n) {
      const int64_t here = info[23 + n];
      if (here == 0) continue;
      truncate_level_kernel<<<counted((unsigned)here), BOX_THREADS, sh, s>>>(k, end - here, n_in, child, in->coeffs, thresh, Ub,
                                                                     gone, merged, d2, pv, s_smem);
      MRA_CUDA_TRY(cudaGetLastError());
      end -= here;
    }
  }
  // survivors in key order
  const int64_t ne = n_in + nc;
  TR_ALLOC(keep, int, ne + 1);
  TR_ALLOC(pos, int, ne + 1);
  keep_flags_kernel<<<counted((unsigned)((ne + 256) / 256)), 256, 0, s>>>(n_in, nc, gone, merged, keep);
  MRA_CUDA_TRY(cudaGetLastError());
  size_t tsc = 0;
  MRA_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tsc, keep, pos, (int)(ne + 1), s));
  TR_ALLOC(tmp2, unsigned char, tsc);
  MRA_CUDA_TRY(cub::DeviceScan::ExclusiveSum(tmp2, tsc, keep, pos, (int)(ne + 1), s));
  sum_kernel<<<counted(1), 1024, 0, s>>>(nc, d2, d2 + nc);
  MRA_CUDA_TRY(cudaGetLastError());
  // where the result shares the input's buffers, it is put together elsewhere first
  auto overlap = [](const void *a, size_t na, const void *b, size_t nb) {
    return (const char *)a < (const char *)b + nb && (const char *)b < (const char *)a + na;
  };
  const size_t row = (size_t)k3 * sizeof(double), cap = (size_t)std::min<int64_t>(out->cap, ne);
  const bool shared = overlap(in->keys, n_in * 8, out->keys, cap * 8) || overlap(in->coeffs, n_in * row, out->coeffs, cap * row);
  uint64_t *okeys = out->keys;
  double *ocoeffs = out->coeffs;
  if (shared) {
    TR_ALLOC(tk, uint64_t, cap);
    TR_ALLOC(tv, double, cap * k3);
    okeys = tk;
    ocoeffs = tv;
  }
  emit_kept_kernel<<<counted((unsigned)ne), 128, 0, s>>>(n_in, nc, k3, in->keys, in->coeffs, cand, pv, keep, pos, out->cap,
                                                         okeys, ocoeffs);
  MRA_CUDA_TRY(cudaGetLastError());
  int nout = 0;
  double e2 = 0.0;
  MRA_CUDA_TRY(cudaMemcpyAsync(&nout, pos + ne, sizeof(int), cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaMemcpyAsync(&e2, d2 + nc, 8, cudaMemcpyDeviceToHost, s));
  MRA_CUDA_TRY(cudaStreamSynchronize(s));
  out->n = nout;
  if (nout > out->cap)
    return fail(MRA_ERR_CAPACITY, "mra_truncate: %d leaves, capacity %lld", nout, (long long)out->cap);
  if (shared) {
    MRA_CUDA_TRY(cudaMemcpyAsync(out->keys, okeys, (size_t)nout * 8, cudaMemcpyDeviceToDevice, s));
    MRA_CUDA_TRY(cudaMemcpyAsync(out->coeffs, ocoeffs, (size_t)nout * row, cudaMemcpyDeviceToDevice, s));
    MRA_CUDA_TRY(cudaStreamSynchronize(s));
  }
  if (err2) *err2 = e2;
  return MRA_OK;
#undef TR_ALLOC
}
