// setup.cu -- set-up kernels: Gaussian-fit search, 1-D operator blocks, projection.
//
// Everything here is FP64 and runs once per operator or per input function, outside the
// applies; the fit also runs in every refit, so in every step of the bound-state solver.  Compiled with --fmad=false so that
// the fit search evaluates its error exactly as written.
#include <cooperative_groups.h>
#include <math.h>

#include "mra_internal.cuh"

namespace mra {

namespace cg = cooperative_groups;

namespace {

constexpr int GLQ = 20;  // points per panel of the composite Gauss-Legendre rules
__constant__ double c_glx[GLQ], c_glw[GLQ];

__device__ __forceinline__ void legendre_phi(int k, double x01, double *out) {
  // phi_i(x) = sqrt(2i+1) P_i(2x-1), i < k (Sec. 2.1, eq. scalingfunc); zero outside [0,1]
  if (x01 < 0.0 || x01 > 1.0) {
    for (int i = 0; i < k; ++i) out[i] = 0.0;
    return;
  }
  double x = 2.0 * x01 - 1.0, p0 = 1.0, p1 = x;
  out[0] = 1.0;
  if (k > 1) out[1] = sqrt(3.0) * x;
  for (int m = 1; m + 1 < k; ++m) {
    double p2 = ((2.0 * m + 1.0) * x * p1 - (double)m * p0) / (m + 1.0);
    p0 = p1;
    p1 = p2;
    out[m + 1] = sqrt(2.0 * m + 3.0) * p2;
  }
}

// --------------------------------------------------------------------------- fit search
// A candidate (h, s_lo) of the grid h = (5+i)/100, s_lo = (j-100)/4 has the error
// max_p |sum_m c_m exp(-t_m r_p^2) - K(r_p)| / K(r_p) over the log-spaced points p = 0 .. 2999; over a
// subset of the points it is a lower bound of that (a maximum over some of the same values).
constexpr int FIT_NS = 113, FIT_NP = 3000;  // s_lo values per h (116 h values), points
constexpr int FIT_SUB = 16;                 // points of the lower bounds

// r_p and K(r_p) of every point.
__global__ void fit_points_kernel(double mu, double r_lo, double r_hi, double *rk) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= FIT_NP) return;
  const double r = r_lo * pow(r_hi / r_lo, (double)p / (double)(FIT_NP - 1));
  rk[p] = r;
  rk[FIT_NP + p] = exp(-mu * r) / r;
}

__device__ __forceinline__ void fit_term(double mu, int cand, int m, double &c, double &t) {
  const int i = cand / FIT_NS, j = cand % FIT_NS;
  const double h = (5.0 + i) / 100.0, s_lo = (j - 100.0) / 4.0;
  const double two_over_sqrtpi = 2.0 / sqrt(3.14159265358979323846264338327950288);
  const double s = s_lo + m * h;
  c = two_over_sqrtpi * h * exp(s - mu * mu * exp(-2.0 * s) / 4.0);
  t = exp(2.0 * s);
}

__device__ __forceinline__ double fit_error(int M, const double *c, const double *t, double r, double K) {
  double sum = 0.0;
  for (int m = 0; m < M; ++m) sum += c[m] * exp(-t[m] * r * r);
  return fabs(sum - K) / K;
}

// Lower bounds of every candidate over the FIT_SUB points pts: half a warp per candidate, a lane per point
// (one CTA per candidate used 16 of its 256 threads: 1.5 of the 2.45 ms of a fit went there).
__global__ void fit_lower_kernel(double mu, int M, int n_cand, const int *pts, const double *rk, double *err) {
  extern __shared__ double sh[];  // [candidates of the CTA][2][M]
  const int half = threadIdx.x / FIT_SUB, lane = threadIdx.x % FIT_SUB;
  const int cand = blockIdx.x * (blockDim.x / FIT_SUB) + half;
  double *c = sh + half * 2 * M, *t = c + M;
  if (cand < n_cand)
    for (int m = lane; m < M; m += FIT_SUB) fit_term(mu, cand, m, c[m], t[m]);
  __syncwarp();
  double worst = 0.0;
  if (cand < n_cand) {
    const int p = pts[lane];
    const double e = fit_error(M, c, t, rk[p], rk[FIT_NP + p]);
    worst = e > worst ? e : worst;
  }
  for (int o = FIT_SUB / 2; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  if (cand < n_cand && lane == 0) err[cand] = worst;
}

// Full errors of the listed candidates: CTA (candidate, 256 points), the maximum by atomics on the bits (the errors
// are not negative, so their bits order as they do; err is zero before).  A candidate on one CTA kept 16 SMs busy.
__global__ void fit_full_kernel(double mu, int M, const int *cands, const double *rk, double *err) {
  extern __shared__ double sh[];
  double *c = sh, *t = sh + M;
  for (int m = threadIdx.x; m < M; m += blockDim.x) fit_term(mu, cands[blockIdx.x], m, c[m], t[m]);
  __syncthreads();
  const int p = blockIdx.y * blockDim.x + threadIdx.x;
  double worst = 0.0;
  if (p < FIT_NP) {
    const double e = fit_error(M, c, t, rk[p], rk[FIT_NP + p]);
    worst = e > worst ? e : worst;
  }
  for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  if ((threadIdx.x & 31) == 0) atomicMax((unsigned long long *)err + blockIdx.x, (unsigned long long)__double_as_longlong(worst));
}

// --------------------------------------------------------------------------- blocks
// R^n_{m,l}[i][j] = h int_{-1}^{1} exp(-T (z+l)^2) C_ij(z) dz,
//   C_ij(z) = int_{max(0,z)}^{min(1,1+z)} phi_i(u) phi_j(u-z) du  (exact: (k+1)-point GL),
// the cross-correlation form of h int int phi_i(u) exp(-T(u-v+l)^2) phi_j(v) du dv with z = u - v.
// The outer integral runs over w = z + l on the two halves z in [-1,0], [0,1]
// (C has a kink at z = 0), restricted to |w| <= sqrt(wmin^2 + 46/T) (the rest is
// below e^-46 of the maximum on that half), with uniform panels no wider than
// min(1/8, 1/(2 sqrt T), 1/(T wmin)) and 20-point Gauss-Legendre per panel.
struct HalfRange {
  double lo, hi;
  int npan;
};

// `wide`: panels of at most 1, 1/sqrt(T) and 2/(T wmin) instead of 1/8, 1/2 and 1 of these.  Enough for the Gaussian
// times a polynomial of degree below 16: on such a panel a polynomial of degree 24 is within 1e-23 of the
// Gaussian's own scale there, and 20 points integrate the product of the two exactly.
__device__ HalfRange half_range(double T, double wa, double wb, bool wide = false) {
  HalfRange r;
  double wmin = wa > 0.0 ? wa : (wb < 0.0 ? -wb : 0.0);
  r.lo = wa;
  r.hi = wb;
  wide = wide && T > 0.0;
  double width = wide ? 1.0 : 0.125;
  const double grow = wide ? 2.0 : 1.0;
  if (T > 0.0) {
    double W = sqrt(wmin * wmin + 46.0 / T);
    if (-W > r.lo) r.lo = -W;
    if (W < r.hi) r.hi = W;
    width = fmin(width, grow * 0.5 / sqrt(T));
    if (wmin > 0.0) width = fmin(width, grow / (T * wmin));
  }
  if (r.hi <= r.lo) {
    r.npan = 0;
    return r;
  }
  double np = ceil((r.hi - r.lo) / width);
  r.npan = (int)fmin(np, 1024.0);
  return r;
}

constexpr int ZB = 8;  // z nodes per shared-memory round

__global__ void blocks_kernel(int k, double L, int min_level, int nlev, const int *Dlev,
                              const int64_t *level_off, const double *t, int M, const double *glxk,
                              const double *glwk, double *R, double *N) {
  extern __shared__ double sm[];
  // phi tables for ZB z-nodes: A[zb][q][i] = phi_i(u_q), B[zb][q][j] = phi_j(u_q - z)
  int kq = k + 1;
  double *A = sm;
  double *B = A + ZB * kq * k;
  double *wq = B + ZB * kq * k;  // [ZB][kq] quadrature weight (incl. Gaussian and Jacobians)
  __shared__ double red[32];
  int64_t blk = blockIdx.x;
  int lev = min_level;
  for (int q = 0; q < nlev; ++q)
    if (blk >= level_off[min_level + q]) lev = min_level + q;
  int D = Dlev[lev];
  int nl = 2 * D + 1;
  int64_t local = blk - level_off[lev];
  int m = (int)(local / nl);
  int l = (int)(local % nl) - D;
  double h = 2.0 * L / (double)(1LL << lev);
  double T = t[m] * h * h;
  HalfRange hr[2] = {half_range(T, -1.0 + l, 0.0 + l), half_range(T, 0.0 + l, 1.0 + l)};
  int n0 = hr[0].npan * GLQ, ntot = n0 + hr[1].npan * GLQ;
  int tid = threadIdx.x;
  int ii = tid / k, jj = tid % k;
  double acc = 0.0;
  for (int base = 0; base < ntot; base += ZB) {
    // build tables for nodes base..base+ZB-1
    for (int e = tid; e < ZB * kq; e += blockDim.x) {
      int zb = e / kq, q = e % kq;
      int node = base + zb;
      double wgt = 0.0, z = 0.0;
      if (node < ntot) {
        int half = node < n0 ? 0 : 1;
        int idx = half ? node - n0 : node;
        int p = idx / GLQ, g = idx % GLQ;
        const HalfRange &r = hr[half];
        double pw = (r.hi - r.lo) / r.npan;
        double w = r.lo + pw * (p + 0.5 + 0.5 * c_glx[g]);
        z = w - (double)l;
        double ua = z > 0.0 ? z : 0.0, ub = z < 0.0 ? 1.0 + z : 1.0;
        double u = ua + (ub - ua) * 0.5 * (glxk[q] + 1.0);
        wgt = 0.5 * pw * c_glw[g] * exp(-T * w * w) * 0.5 * (ub - ua) * glwk[q];
        legendre_phi(k, u, A + (zb * kq + q) * k);
        legendre_phi(k, u - z, B + (zb * kq + q) * k);
      } else {
        for (int i = 0; i < k; ++i) {
          A[(zb * kq + q) * k + i] = 0.0;
          B[(zb * kq + q) * k + i] = 0.0;
        }
      }
      wq[zb * kq + q] = wgt;
    }
    __syncthreads();
    if (tid < k * k) {
      for (int e = 0; e < ZB * kq; ++e) acc += wq[e] * A[e * k + ii] * B[e * k + jj];
    }
    __syncthreads();
  }
  double v = (tid < k * k) ? h * acc : 0.0;
  if (tid < k * k) R[blk * k * k + tid] = v;
  double s2 = v * v;
  for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  if ((tid & 31) == 0) red[tid >> 5] = s2;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += red[q];
    N[blk] = sqrt(s);
  }
}

// --------------------------------------------------------------------------- projection
// s_b[ix][iy][iz] = sum_g coef_g X_g[ix] Y_g[iy] Z_g[iz] with the 1-D factors
// X_g[i] = h^{1/2} int_0^1 exp(-a_g h^2 (u - uc)^2) phi_i(u) du, uc = (c_g + L)/h - b_x  (eq. projection).
// A factor depends on (level, dimension, coordinate) and the Gaussian only, and the boxes of a
// refined neighbourhood share their coordinates, so the integrals are done once per distinct
// coordinate (an "entry") and not once per box.  8 Gaussians, k = 10, 17,200 leaves: the integrals
// 179 -> 0.50 ms, the refinement test 8.0 -> 0.49 ms with the children's assembly, the call 190 -> 2.2 ms
// (FP64-bound exponentials, recurrences and products; the rest is the host's decision after every level).

// A factor entry: level, dimension and coordinate.
__host__ __device__ inline uint64_t make_entry(int level, int dim, int64_t x) {
  return ((uint64_t)level << 40) | ((uint64_t)dim << 32) | (uint64_t)x;
}

// Legendre polynomials of leading coefficient one, Q_{m+1} = x Q_m - b_m Q_{m-1}, and sqrt(2i+1) P_i / Q_i.
__constant__ double c_leg_b[MRA_MAX_K], c_leg_s[MRA_MAX_K];

constexpr int FACTOR_THREADS = 128, FACTOR_SUB = 8;  // threads per sum over the nodes, one sum per i
static_assert(FACTOR_SUB * MRA_MAX_K <= FACTOR_THREADS, "a group of threads for every i");

// Where the factors of a set of entries go: F[(e * ng + g) * stride + i], i < k; nz[e * ng + g] = 0 when all
// k are zero, which needs no quadrature where the Gaussian underflows on the whole box.
struct FactorSet {
  int stride;
  double *F;
  unsigned char *nz;
};

// One CTA per (entry, Gaussian), the first n_first entries into one set and the rest into the other (parents and
// children in one launch); threads stride over the nodes of the panel rule over the offset w = u - uc
// (the sums over the threads go through shared memory, an eighth of a shuffle reduction's additions; with it
// and a recurrence of leading coefficient one 0.64 -> 0.50 ms).
// A level has few tasks of up to 280 nodes, each with an exponential and a serial recurrence: with one warp per task
// and panels of half the width latency bound (63 us a launch, two launches a level; 8 Gaussians, k = 10: 1.52 ms of
// a projection), now the FP64 pipe does at the larger levels (42 us a level, 0.50 ms).
__global__ void __launch_bounds__(FACTOR_THREADS) factor_kernel(int64_t n_entries, int64_t n_first, int ng, const double *g,
                                                                int k, double L, const uint64_t *entries,
                                                                const __grid_constant__ FactorSet first,
                                                                const __grid_constant__ FactorSet rest) {
  __shared__ double glx[GLQ], glw[GLQ], sum[MRA_MAX_K][FACTOR_THREADS + FACTOR_SUB];
  if (threadIdx.x < GLQ) {
    glx[threadIdx.x] = c_glx[threadIdx.x];
    glw[threadIdx.x] = c_glw[threadIdx.x];
  }
  __syncthreads();
  for (int64_t task = blockIdx.x; task < n_entries * ng; task += gridDim.x) {
    const int64_t en = task / ng;
    const int gi = (int)(task - en * ng);
    const uint64_t ent = entries[en];
    const int n = (int)(ent >> 40), d = (int)(ent >> 32) & 255;
    const double bx = (double)(ent & 0xFFFFFFFFull);
    const double h = 2.0 * L / (double)(1LL << n);
    const double T = g[ng + gi] * h * h;
    const double x = (g[(2 + d) * ng + gi] + L) / h;  // uc = x - b
    const double wa = bx - x;                         // w at u = 0
    const double wb = (bx + 1.0) - x;                 // w at u = 1
    double acc[MRA_MAX_K];
#pragma unroll
    for (int i = 0; i < MRA_MAX_K; ++i) acc[i] = 0.0;
    const double wmin = wa > 0.0 ? wa : (wb < 0.0 ? -wb : 0.0);
    if (T * wmin * wmin < 760.0) {  // exp(-745.2) is the smallest positive double
      const HalfRange r = half_range(T, wa, wb, true);
      const int nn = r.npan * GLQ;
      const double pw = r.npan > 0 ? (r.hi - r.lo) / r.npan : 0.0;
      for (int node = threadIdx.x; node < nn; node += FACTOR_THREADS) {
        const int p = node / GLQ, q = node % GLQ;
        const double w = r.lo + pw * (p + 0.5 + 0.5 * glx[q]);
        const double wt = 0.5 * pw * glw[q] * exp(-T * w * w);
        const double t = 2.0 * (w - wa) - 1.0;  // u = w + uc, formed from the box end
        double p0 = 1.0, p1 = t;
        acc[0] += wt;
#pragma unroll
        for (int i = 1; i < MRA_MAX_K; ++i) {
          if (i < k) {
            acc[i] = fma(wt, p1, acc[i]);
            const double p2 = fma(t, p1, -c_leg_b[i] * p0);
            p0 = p1;
            p1 = p2;
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < MRA_MAX_K; ++i)
      if (i < k) sum[i][threadIdx.x] = acc[i];
    __syncthreads();
    const int i = threadIdx.x / FACTOR_SUB, sub = threadIdx.x % FACTOR_SUB;
    double v = 0.0;
    if (i < k)
      for (int q = sub; q < FACTOR_THREADS; q += FACTOR_SUB) v += sum[i][q];
    for (int o = FACTOR_SUB / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const FactorSet to = en < n_first ? first : rest;
    const int64_t row = (en < n_first ? en : en - n_first) * ng + gi;
    if (i < k) {
      v *= c_leg_s[i] * sqrt(h);
      if (sub == 0) to.F[row * to.stride + i] = v;
    }
    const int some = __syncthreads_or(v != 0.0);  // NaN counts as nonzero
    if (threadIdx.x == 0) to.nz[row] = some ? 1 : 0;
  }
}

// The parents' factors on their children, X' = U^{(c)} X (two-scale relation of Sec. 2.2 in one dimension),
// beside the children's own: child entry 2 e + c, F_child[((2 e + c) * ng + g) * 2k + k + i].
__global__ void lift_kernel(int64_t n, int ng, int k, const double *Fp, const unsigned char *nzp, const double *U,
                            double *Fc, unsigned char *nzc) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // (child entry, g, i)
  if (q >= n * 2 * ng * k) return;
  const int i = (int)(q % k);
  const int64_t cg = q / k, ce = cg / ng, pg = (ce >> 1) * ng + cg % ng;
  const double *Uc = U + (ce & 1) * k * k + i * k, *X = Fp + pg * k;
  double v = 0.0;
  for (int j = 0; j < k; ++j) v = fma(Uc[j], X[j], v);
  Fc[cg * 2 * k + k + i] = v;
  if (i == 0 && nzp[pg]) nzc[cg] |= 2;  // bit 0: the child's own factor is nonzero, bit 1: the parent's
}

constexpr int ASM_THREADS = 256, ASM_G = 16;  // Gaussians staged at a time

// A thread has the elements (ix, iy, sub + q S), q < EPT, of a box: S threads per (ix, iy), so that X Y is formed
// once for all of a thread's iz.
struct Elements {
  int ix, iy, sub, S;
  bool active;
  __device__ Elements(int k) {
    const int k2 = k * k;
    S = max(1, min(k, ASM_THREADS / k2));
    const int pair = min((int)threadIdx.x / S, k2 - 1);
    active = (int)threadIdx.x < k2 * S;
    ix = pair / k;
    iy = pair % k;
    sub = (int)threadIdx.x % S;
  }
  // the element's place in the box's coefficients, or -1
  __device__ int at(int k, int q) const {
    const int iz = sub + q * S;
    return active && iz < k ? (ix * k + iy) * k + iz : -1;
  }
};

// Sum over the Gaussians at this thread's elements of one box with the
// factor entries e[0..2], added to own[q], and with TEST the parent's projection there, to par[q].  Gaussians
// whose product is exactly zero are left out; the others are added in order.
template <int EPT, bool TEST>
__device__ void sum_gaussians(int ng, int k, const Elements &el, const double *coef, const double *F, const unsigned char *nz,
                              const int64_t *e, double *stage, int *list, int *count, double *own, double *par) {
  const int st = TEST ? 2 * k : k;
  for (int g0 = 0; g0 < ng;) {
    __syncthreads();  // the list and the staged factors of the previous round have been used
    if (threadIdx.x < 32) {  // the next ASM_G Gaussians that matter, in order
      int have = 0, next = g0;
      while (next < ng && have < ASM_G) {
        const int gi = next + (int)threadIdx.x;
        int f = 0;
        if (gi < ng) {
          f = nz[e[0] * ng + gi] & nz[e[1] * ng + gi] & nz[e[2] * ng + gi];
          if (!isfinite(coef[gi])) f = 1;  // its product with zero is not zero
        }
        const unsigned b = __ballot_sync(0xffffffffu, f != 0);
        const int at = have + __popc(b & ((1u << threadIdx.x) - 1u));
        if (f && at < ASM_G) list[at] = gi;
        const int n = __popc(b);
        if (have + n > ASM_G) {  // resume after the last one taken
          int left = ASM_G - have;
          unsigned bb = b;
          int last = 0;
          while (left-- > 0) {
            last = __ffs(bb) - 1;
            bb &= bb - 1;
          }
          next += last + 1;
          have = ASM_G;
        } else {
          have += n;
          next += 32;
        }
      }
      if (threadIdx.x == 0) {
        count[0] = have;
        count[1] = min(next, ng);
      }
    }
    __syncthreads();
    const int have = count[0];
    g0 = count[1];
    for (int q = threadIdx.x; q < have * 3 * st; q += ASM_THREADS) {
      const int l = q / (3 * st), r = q - l * 3 * st, d = r / st, i = r - d * st;
      const double v = F[(e[d] * ng + list[l]) * st + i];
      stage[q] = d == 0 ? coef[list[l]] * v : v;
    }
    __syncthreads();
    for (int l = 0; l < have; ++l) {
      const double *X = stage + l * 3 * st, *Y = X + st, *Z = Y + st;
      const double xy = X[el.ix] * Y[el.iy], pxy = TEST ? X[k + el.ix] * Y[k + el.iy] : 0.0;
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int iz = el.sub + q * el.S;
        if (iz < k) {
          own[q] = fma(xy, Z[iz], own[q]);
          if (TEST) par[q] = fma(pxy, Z[k + iz], par[q]);
        }
      }
    }
  }
}

// A cluster of eight CTAs per parent: each has one child's coefficients, together ||s_children - U s_parent||_F
// (the refinement test of Sec. 2.1), the parent's projection on a child being the sum of the lifted factors'
// products: no k^4 transform.  pidx: the parent's entry in each dimension.  One CTA for the eight children in
// turn, X Y formed for every element, took 61 us a level (k = 10, 8 Gaussians, up to 376 parents), now 41.
template <int EPT>
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(ASM_THREADS)
    children_kernel(int ng, int k, const double *coef, const double *F, const unsigned char *nz, const int *pidx, double *out,
                    double *dnorm) {
  extern __shared__ double stage[];  // [ASM_G][3][2k]
  __shared__ int list[ASM_G], count[2];
  __shared__ double red[ASM_THREADS / 32], total;
  const cg::cluster_group cluster = cg::this_cluster();
  const int c = (int)cluster.block_rank();
  const int64_t p = blockIdx.x >> 3;
  const int k3 = k * k * k;
  const Elements el(k);
  const int64_t e[3] = {2 * (int64_t)pidx[3 * p] + (c >> 2), 2 * (int64_t)pidx[3 * p + 1] + ((c >> 1) & 1),
                        2 * (int64_t)pidx[3 * p + 2] + (c & 1)};
  double own[EPT] = {}, par[EPT] = {}, part = 0.0;
  sum_gaussians<EPT, true>(ng, k, el, coef, F, nz, e, stage, list, count, own, par);
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    const int m = el.at(k, q);
    if (m >= 0) {
      out[(8 * p + c) * k3 + m] = own[q];
      const double d = own[q] - par[q];
      part = fma(d, d, part);
    }
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int q = 0; q < ASM_THREADS / 32; ++q) v += red[q];
    total = v;
  }
  cluster.sync();
  if (c == 0 && threadIdx.x == 0) {
    double v = 0.0;
    for (int q = 0; q < 8; ++q) v += *cluster.map_shared_rank(&total, q);
    dnorm[p] = sqrt(v);
  }
  cluster.sync();  // the totals have been read
}

// One CTA per box of a whole level (entry of dimension d and coordinate x: d 2^n + x).
template <int EPT>
__global__ void __launch_bounds__(ASM_THREADS) boxes_kernel(int ng, int k, const double *coef, const double *F,
                                                            const unsigned char *nz, const uint64_t *keys, double *out,
                                                            int add) {
  extern __shared__ double stage[];  // [ASM_G][3][k]
  __shared__ int list[ASM_G], count[2];
  const int64_t b = blockIdx.x;
  const uint64_t key = keys[b];
  const int64_t nb = 1LL << key_level(key);
  const int64_t e[3] = {key_x(key), nb + key_y(key), 2 * nb + key_z(key)};
  const Elements el(k);
  double own[EPT] = {}, par[EPT];
  if (add) {
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int m = el.at(k, q);
      if (m >= 0) own[q] = out[b * k * k * k + m];
    }
  }
  sum_gaussians<EPT, false>(ng, k, el, coef, F, nz, e, stage, list, count, own, par);
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    const int m = el.at(k, q);
    if (m >= 0) out[b * k * k * k + m] = own[q];
  }
}

// The rules' nodes and the recurrence's coefficients, written on stream s before the kernels that read them
// (always the same values).
cudaError_t upload_tables(cudaStream_t s) {
  struct Tables {
    double x[GLQ], w[GLQ], b[MRA_MAX_K], r[MRA_MAX_K];
    Tables() {
      gauss_legendre(GLQ, x, w);
      double lead = 1.0;  // of P_m
      for (int m = 0; m < MRA_MAX_K; ++m) {
        b[m] = (double)(m * m) / (4.0 * m * m - 1.0);
        r[m] = sqrt(2.0 * m + 1.0) * lead;
        lead *= (2.0 * m + 1.0) / (m + 1.0);
      }
    }
  };
  static const Tables t;
  cudaError_t e = cudaMemcpyToSymbolAsync(c_glx, t.x, sizeof(t.x), 0, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_glw, t.w, sizeof(t.w), 0, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_leg_b, t.b, sizeof(t.b), 0, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_leg_s, t.r, sizeof(t.r), 0, cudaMemcpyHostToDevice, s);
  return e;
}

}  // namespace

size_t fit_points_bytes() { return 2 * FIT_NP * sizeof(double); }

cudaError_t launch_fit_lower(double mu, int M, double r_lo, double r_hi, const int *d_pts, double *d_rk, int n_cand,
                             double *d_err, cudaStream_t s) {
  fit_points_kernel<<<counted((FIT_NP + 255) / 256), 256, 0, s>>>(mu, r_lo, r_hi, d_rk);
  const int per = 128 / FIT_SUB;
  fit_lower_kernel<<<counted((unsigned)((n_cand + per - 1) / per)), 128, per * 2 * M * sizeof(double), s>>>(mu, M, n_cand, d_pts,
                                                                                                          d_rk, d_err);
  return cudaGetLastError();
}

cudaError_t launch_fit_full(double mu, int M, const int *d_cands, int n_cands, const double *d_rk, double *d_err,
                            cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(d_err, 0, n_cands * sizeof(double), s);
  if (e != cudaSuccess) return e;
  fit_full_kernel<<<counted(dim3((unsigned)n_cands, (FIT_NP + 255) / 256)), 256, 2 * M * sizeof(double), s>>>(mu, M, d_cands,
                                                                                                             d_rk, d_err);
  return cudaGetLastError();
}

cudaError_t launch_blocks(const Operator &op, const double *d_glxk, const double *d_glwk,
                          cudaStream_t s) {
  cudaError_t e = upload_tables(s);
  if (e != cudaSuccess) return e;
  int kq = op.k + 1;
  size_t smem = (size_t)(2 * ZB * kq * op.k + ZB * kq) * sizeof(double);
  int threads = 256;
  int nlev = op.max_level - op.min_level + 1;
  blocks_kernel<<<counted((unsigned)op.n_blocks), threads, smem, s>>>(op.k, op.L, op.min_level, nlev, op.d_D,
                                                             op.d_level_off, op.d_t, op.M, d_glxk,
                                                             d_glwk, op.d_R, op.d_N);
  return cudaGetLastError();
}

// Factors of the entries (device array) for every Gaussian, the first n_first into one set, the others into the rest.
static cudaError_t launch_factors(int64_t n_entries, int64_t n_first, int ng, const double *d_g, int k, double L,
                                  const uint64_t *d_entries, FactorSet first, FactorSet rest, cudaStream_t s) {
  const int64_t tasks = n_entries * ng;
  if (tasks <= 0) return cudaSuccess;
  factor_kernel<<<counted((unsigned)std::min<int64_t>(tasks, 1 << 20)), FACTOR_THREADS, 0, s>>>(n_entries, n_first, ng, d_g, k, L,
                                                                                               d_entries, first, rest);
  return cudaGetLastError();
}

cudaError_t launch_project_level(int ng, const double *d_g, int k, double L, int64_t n_entries, const uint64_t *d_entries,
                                 double *F, unsigned char *nz, int64_t nbox, const uint64_t *d_keys, double *d_out,
                                 bool add, cudaStream_t s) {
  if (nbox <= 0) return cudaSuccess;
  cudaError_t e = upload_tables(s);
  const FactorSet f{k, F, nz};
  if (e == cudaSuccess) e = launch_factors(n_entries, n_entries, ng, d_g, k, L, d_entries, f, f, s);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)ASM_G * 3 * k * sizeof(double);
  if (k <= 10)
    boxes_kernel<5><<<counted((unsigned)nbox), ASM_THREADS, smem, s>>>(ng, k, d_g, F, nz, d_keys, d_out, add);
  else
    boxes_kernel<16><<<counted((unsigned)nbox), ASM_THREADS, smem, s>>>(ng, k, d_g, F, nz, d_keys, d_out, add);
  return cudaGetLastError();
}

cudaError_t launch_project_children(int ng, const double *d_g, int k, double L, int64_t n_entries,
                                    const uint64_t *d_entries, const double *d_U, double *Fp, double *Fc,
                                    unsigned char *nzp, unsigned char *nzc, int64_t np, const int *d_pidx, double *d_out,
                                    double *d_dnorm, cudaStream_t s) {
  if (np <= 0) return cudaSuccess;
  // the parents' entries, then their children's (2 e + c)
  cudaError_t e = launch_factors(3 * n_entries, n_entries, ng, d_g, k, L, d_entries, FactorSet{k, Fp, nzp},
                                 FactorSet{2 * k, Fc, nzc}, s);
  if (e != cudaSuccess) return e;
  if (ng > 0) {
    const int64_t nl = n_entries * 2 * ng * k;
    lift_kernel<<<counted((unsigned)((nl + 255) / 256)), 256, 0, s>>>(n_entries, ng, k, Fp, nzp, d_U, Fc, nzc);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const size_t smem = (size_t)ASM_G * 6 * k * sizeof(double);
  if (k <= 10)
    children_kernel<5><<<counted((unsigned)(8 * np)), ASM_THREADS, smem, s>>>(ng, k, d_g, Fc, nzc, d_pidx, d_out, d_dnorm);
  else
    children_kernel<16><<<counted((unsigned)(8 * np)), ASM_THREADS, smem, s>>>(ng, k, d_g, Fc, nzc, d_pidx, d_out, d_dnorm);
  return cudaGetLastError();
}

cudaError_t project_tables(cudaStream_t s) { return upload_tables(s); }
uint64_t factor_entry(int level, int dim, int64_t x) { return make_entry(level, dim, x); }

}  // namespace mra
