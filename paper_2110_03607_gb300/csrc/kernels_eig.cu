// FP64 eigen-solver for the symmetric environment matrices A^(j), A'^(j) (Sec. 4.2.5,
// Eqs. SVD_N / SVD_P), and the choice / truncation / sign gauge of the isometries
// (Secs. 2, 4.2.6-4.2.8).
//
// A = Q T Q^T by Householder reflections (Golub & Van Loan, Sec. 8.3.1), one thread-block
// cluster per matrix; T = Z diag(lambda) Z^T by Cuppen's divide and conquer with the
// eigenvectors of Gu & Eisenstat (SIAM J. Matrix Anal. Appl. 16, 172, 1995); V = Q Z.  Every
// stage is backward stable: eigenvalues to a few eps ||A||, V orthogonal to a few eps n.  A's rows
// fall off by many orders, and their rounding with them: what one-sided Jacobi sweeps would resolve
// beyond eps ||A|| for the kept vectors is put right at the end from W = A V (eig_gram_kernel).
//
// Why not Jacobi: one-sided Jacobi spends about 11 n^3 FP64 multiply-adds per sweep and n - 1
// grid-wide barriers, and needed 4 to 16 sweeps after its FP32 start (the part of the spectrum
// below the FP32 resolution starts from nothing); GB300 issues 2 FP64 FMA per clock and SM, so
// the count of operations is what matters: n^3 (reduction) + up to 4/3 n^3 (merges, less what
// deflates) + n^3 (back-transformation) + 2 n^3 (W = A V and its Gram
// matrix).  Measured, before and after: 4 matrices of 32 rows 1.4 and 0.58 ms, 8 of 128 9.1 and 1.4,
// 4 of 288 (2D, chi = 24, zero field) 85 and 3.9.
//
// Which vectors are taken from a degenerate eigenspace matters: the run goes on from them, and on
// an isotropic lattice many pairs are degenerate, each vector with a symmetry of its own.  So the
// symmetries are taken out first, as Jacobi rotations from the unit vectors would leave them:
//  * where A commutes with the exchange of hat and check up to a sign per index (a lattice that is
//    symmetric under the reflection of the current axis; the signs are the parities that the
//    leg's indices have under it), it is turned to the even and odd combinations;
//  * the indices are ordered by the connected components of the pattern of elements above
//    rounding, elements between components count as zero, and a reflector never mixes two
//    components.  Exact zeros between parities stay exact.
//
// A batch of up to kJacobiMax rows (the caller gives the matrices up to there and those above as
// two batches) goes through one-sided Jacobi sweeps (jacobi_onesided_kernel): they cost no
// more there (n = 16: 0.2 ms), and they move nearly degenerate pairs, which the first steps of a
// split run have at the 1e-8 of its rounding, less than the reduction's few eps.
#include <cooperative_groups.h>

#include <algorithm>

#include "eig_class.h"
#include "hotrg_internal.cuh"
#include "../../include/hotrg.h"

namespace cg = cooperative_groups;

namespace hotrg {

namespace {
constexpr double kEps = 2.220446049250313e-16;
constexpr int kRb = 16;          // reflectors per block of the back-transformation
constexpr int kLeaf = 9;         // largest tridiagonal leaf solved by implicit QR in one warp
constexpr int kJacobiMax = kEigSmall;   // largest order left to the Jacobi sweeps
constexpr int kPolish = 96;      // columns of a group of close eigenvalues
constexpr int kEigMaxN = 1024;   // chi_j^2 <= 32^2
constexpr int kTriThreads = 256;
constexpr int kVecThreads = 128;   // of them, those with the work of order n: a warp per quarter of the SM

// per-matrix control words
struct EigCtl {
  double unscale;    // power of two: max |A| / unscale in [0.5, 1)
  int bad;           // a non-finite element: eigenvalues and vectors are set to NaN
  int mixed;         // a row is coupled to another label: the components need more rounds; in the correction:
                     // whether the pass has angles (1), one above 2^-24 (2) or 2^-12 (3) among them
  int settled;       // a pass of the correction found no angle above 2^-24: it left none above 2^-48
  int iters;         // most QR iterations an eigenvalue of a leaf took
  unsigned long long amax;   // bits of max |A|
  double top;        // max |A| / unscale
};
// per-merge control words
struct MergeCtl {
  int k;             // eigenvalues left in the secular equation
  int nrot;          // plane rotations of the deflation
  int ntop, nbot;    // columns with entries in the first / second half's rows
};

// views of the workspace of a batch of matrices, and their orders
constexpr int kEigMaxMat = 16;
struct EigWs {
  int n, nmat;            // leading dimension of the batch, matrices
  int na[kEigMaxMat];     // order of each matrix (<= n)
  int keep[kEigMaxMat];   // leading eigenvectors that may be kept
  double* vh;        // [nmat][n][n] Householder vectors (row k: v_k), then S of the merges
  double* q0;        // [nmat][n][n] eigenvectors of the nodes (column-major)
  double* q1;
  double* s;         // [nmat][n][n] d_i - lambda_j, then the merge's eigenvectors
  double* d;         // [nmat][n] diagonal of T
  double* e;         // [nmat][n] off-diagonal
  double* tau;       // [nmat][n]
  double* tf;        // [nmat][blocks][kRb][kRb] T factors of the blocked reflectors
  double* ev0;       // [nmat][n] eigenvalues of the nodes, ascending within a node
  double* ev1;
  double* dk;        // [nmat][n] poles of the secular equation
  double* zk;        // [nmat][n] its weights z_i
  double* zh;        // [nmat][n] the weights recomputed from the roots
  double* val;       // [nmat][n] new eigenvalues: roots, then deflated
  double* rc;        // [nmat][n] rotation cosines
  double* rs;        // [nmat][n] sines
  double* w2;        // [nmat][n][n] turned columns of the correction
  double* w3;        // [nmat][n][n]
  double* ap;        // [nmat][n][n] A, scaled, in the basis of the exchange's combinations
  const int* swp;    // [nmat][n] partner of every index under the exchange
  int* perm;         // [nmat][n] component order
  int* comp;         // [nmat][n] component label
  int* sgn;          // [nmat][n] sign of every index under the exchange
  int* okc;          // [nmat][n] by label: the exchange holds in the component
  int* sym;          // [nmat][n] by index: it does in this one's
  int* cls;          // [nmat][n] by eigenvector: (label + 1) even, -(label + 1) odd, 0 without the exchange
  int* lost;         // [nmat][n] by eigenvector: 1 where a turn ended its class
  int* icl;          // [nmat][n] the same as cls by index of the turned basis
  int* idx;          // [nmat][n] columns of the secular equation
  int* defl;         // [nmat][n] deflated columns
  int* rp;           // [nmat][n] rotation columns
  int* rq;
  int* top;          // [nmat][n] entries with support in the first half
  int* bot;
  EigCtl* ctl;       // [nmat]
  MergeCtl* mc;      // [nmat][nodes]
};

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// sums of four values over the warp: halves are exchanged while there is more than one value per
// lane (6 additions instead of 20: an FP64 warp instruction takes 16 issue slots)
__device__ __forceinline__ void warp_sum4(double& a, double& b, double& c, double& e) {
  const int lane = threadIdx.x & 31;
  const bool h4 = (lane & 16) != 0, h3 = (lane & 8) != 0;
  double x0 = h4 ? c : a, y0 = h4 ? a : c;
  double x1 = h4 ? e : b, y1 = h4 ? b : e;
  x0 += __shfl_xor_sync(0xffffffffu, y0, 16);
  x1 += __shfl_xor_sync(0xffffffffu, y1, 16);
  double x = h3 ? x1 : x0;
  const double y = h3 ? x0 : x1;
  x += __shfl_xor_sync(0xffffffffu, y, 8);
  x += __shfl_xor_sync(0xffffffffu, x, 4);
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  a = __shfl_sync(0xffffffffu, x, 0);
  b = __shfl_sync(0xffffffffu, x, 8);
  c = __shfl_sync(0xffffffffu, x, 16);
  e = __shfl_sync(0xffffffffu, x, 24);
}

__device__ __forceinline__ int rr_slot(int i, int r, int mp) {
  // circle method: player 0 fixed, the others rotate by r (0 <= i - 1 + r < 2 (mp - 1), so
  // one conditional subtraction replaces the modulo)
  if (i == 0) return 0;
  int x = i - 1 + r;
  if (x >= mp - 1) x -= mp - 1;
  return 1 + x;
}

// 1 / sqrt(a) for normal a > 0: an FP32 estimate for the mantissa m in [1, 4), a = m 4^k, and two
// Newton steps y <- y (3 - m y^2) / 2, then the exponent (a rotation's chain of dependent FP64
// operations is what a leaf costs; sqrt and a division would be twice as long)
__device__ __forceinline__ double rsqrt_newton(double a) {
  const int hi = __double2hiint(a), ex = ((hi >> 20) - 1023) & ~1;
  const double m = __hiloint2double(hi - (ex << 20), __double2loint(a));
  double y = (double)rsqrtf((float)m);
  y = y * fma(-0.5 * m * y, y, 1.5);
  y = y * fma(-0.5 * m * y, y, 1.5);
  return __hiloint2double(__double2hiint(y) - ((ex >> 1) << 20), __double2loint(y));
}
}  // namespace

// ---------------------------------------------------------------------------
// Scale, symmetry, order
// ---------------------------------------------------------------------------
// What counts as rounding in an environment's element (i, j): 128 eps sqrt(max |A| max(A_ii, A_jj)),
// and eps max |A| / 32 at the least.  The sums over a tensor whose elements carry an absolute error
// of order eps leave up to that much in rows of norm sqrt(A_ii) (measured on 2D runs at chi = 24:
// 1 to 60 eps in the first form, 1e-3 eps max |A| in rows below 1e-20 max |A|).
struct Noise {
  double rel2, abs;   // (128 eps)^2 max |A|, eps max |A| / 32
  __device__ explicit Noise(double amax, double times = 1.0)
      : rel2(times * times * (128.0 * kEps) * (128.0 * kEps) * amax), abs(times * 0.03125 * kEps * amax) {}
  __device__ bool coupled(double a, double di, double dj) const {
    return fabs(a) > abs && a * a > rel2 * fmax(fabs(di), fabs(dj));
  }
};

// max |A| and non-finite elements: a warp per row
__global__ void __launch_bounds__(256) eig_check_kernel(const double* __restrict__ A, EigWs ws) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const double* Am = A + (long long)mat * ld * ld;
  double amax = 0.0;
  int bad = 0;
  for (int j = lane; j < n; j += 32) {
    const double a = fabs(Am[(long long)i * ld + j]);
    if (!(a <= 1.7976931348623157e308)) bad = 1;
    amax = fmax(amax, a);
  }
  for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    EigCtl* c = ws.ctl + mat;
    if (bad) c->bad = 1;
    else atomicMax(&c->amax, (unsigned long long)__double_as_longlong(amax));
  }
}

// ap = 2^-e A (max |ap| in [0.5, 1)), and a first label: the row's first coupled column, which a
// dense block shares.  A warp per row.
__global__ void __launch_bounds__(256) eig_scale_kernel(const double* __restrict__ A, EigWs ws) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const EigCtl c = ws.ctl[mat];
  if (c.bad) return;
  int ex = 0;
  const double amax = __longlong_as_double((long long)c.amax);
  if (amax > 0.0) frexp(amax, &ex);
  ex = ex < -1000 ? -1000 : ex > 1000 ? 1000 : ex;   // both factors stay finite
  const double scale = ldexp(1.0, -ex);
  if (i == 0 && lane == 0) {
    ws.ctl[mat].unscale = ldexp(1.0, ex);
    ws.ctl[mat].top = amax * scale;
  }
  const double* Am = A + (long long)mat * ld * ld;
  double* out = ws.q0 + (long long)mat * ld * ld + (long long)i * ld;
  for (int j = lane; j < n; j += 32) out[j] = Am[(long long)i * ld + j] * scale;
}

// first labels of M: a warp per row
__global__ void __launch_bounds__(256) eig_label_kernel(const double* __restrict__ M, EigWs ws) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const EigCtl c = ws.ctl[mat];
  if (i == 0 && lane == 0) ws.ctl[mat].mixed = 0;
  const double* Mm = M + (long long)mat * ld * ld;
  int first = c.bad ? 0 : i;
  if (!c.bad) {
    const Noise nz(c.top);
    const double di = Mm[(long long)i * ld + i];
    for (int j0 = 0; j0 < i; j0 += 32) {
      const int j = j0 + lane;
      const unsigned m = __ballot_sync(
          0xffffffffu, j < i && nz.coupled(Mm[(long long)i * ld + j], di, Mm[(long long)j * ld + j]));
      if (m) {
        first = j0 + __ffs(m) - 1;
        break;
      }
    }
  }
  if (lane == 0) ws.comp[mat * ld + i] = first;
}

// whether a row is coupled to another label
__global__ void __launch_bounds__(256) eig_mixed_kernel(const double* __restrict__ M, EigWs ws) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const EigCtl c = ws.ctl[mat];
  if (c.bad) return;
  const double* Mm = M + (long long)mat * ld * ld;
  const Noise nz(c.top);
  const double di = Mm[(long long)i * ld + i];
  const int* lab = ws.comp + mat * ld;
  const int l = lab[i];
  int mixed = 0;
#pragma unroll 4
  for (int j = lane; j < n; j += 32)
    if (lab[j] != l && nz.coupled(Mm[(long long)i * ld + j], di, Mm[(long long)j * ld + j])) mixed = 1;
  if (__any_sync(0xffffffffu, mixed) && lane == 0) ws.ctl[mat].mixed = 1;
}

// One CTA per matrix: components by minimum-label hooking with pointer jumping where the first
// labels did not settle them.  SIGNS: then the signs s_i of the exchange P, A_ij = s_i s_j A_PiPj:
// an index takes its sign from its largest coupling to one that has it.  Else the order of the
// rows, stable within a component.
template <bool SIGNS>
__global__ void __launch_bounds__(1024) eig_order_kernel(const double* __restrict__ M, EigWs ws) {
  __shared__ int lab[kEigMaxN], nxt[kEigMaxN], nsg[kEigMaxN];
  __shared__ double diag[kEigMaxN];
  __shared__ int s_changed;
  const int mat = blockIdx.x, n = ws.na[mat], ld = ws.n;
  const EigCtl c = ws.ctl[mat];
  const double* Mm = M + (long long)mat * ld * ld;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const Noise nz(c.top), far(c.top, 1048576.0);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    lab[i] = ws.comp[mat * ld + i];
    diag[i] = c.bad ? 0.0 : Mm[(long long)i * ld + i];
  }
  __syncthreads();
  for (int round = 0; round < n && c.mixed; ++round) {
    if (threadIdx.x == 0) s_changed = 0;
    __syncthreads();
    for (int i = warp; i < n; i += nw) {
      int l = lab[i];
#pragma unroll 4
      for (int j = lane; j < n; j += 32)
        if (nz.coupled(Mm[(long long)i * ld + j], diag[i], diag[j])) l = min(l, lab[j]);
      l = __reduce_min_sync(0xffffffffu, l);
      if (lane == 0) nxt[i] = l;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      int l = nxt[i];
      for (int hop = 0; hop < 16; ++hop) {   // the label's own label stays within the component
        const int l2 = nxt[l];
        if (l2 >= l) break;
        l = l2;
      }
      if (l != lab[i]) s_changed = 1;
      lab[i] = l;
    }
    __syncthreads();
    const int ch = s_changed;
    __syncthreads();
    if (!ch) break;
  }
  if (SIGNS) {
    const int* sw = ws.swp + mat * ld;
    int* sg = nxt;   // 0: none yet
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      sg[i] = lab[i] == i ? 1 : 0;
      nsg[i] = 0;
    }
    __syncthreads();
    // first over couplings far above rounding, then over any
    int strict = 1;
    for (int round = 0; round < 2 * n && !c.bad; ++round) {
      if (threadIdx.x == 0) s_changed = 0;
      __syncthreads();
      for (int i = warp; i < n; i += nw) {
        if (sg[i]) continue;
        double best = 0.0;
        int bj = -1;
        for (int j = lane; j < n; j += 32) {
          if (lab[j] != lab[i] || sg[j] == 0) continue;
          const double x = Mm[(long long)i * ld + j];
          if (fabs(x) > best && (strict ? far : nz).coupled(x, diag[i], diag[j])) {
            best = fabs(x);
            bj = j;
          }
        }
        for (int o = 16; o > 0; o >>= 1) {
          const double b2 = __shfl_xor_sync(0xffffffffu, best, o);
          const int j2 = __shfl_xor_sync(0xffffffffu, bj, o);
          if (b2 > best || (b2 == best && j2 > bj)) {
            best = b2;
            bj = j2;
          }
        }
        if (bj >= 0 && lane == 0) {
          const double x = Mm[(long long)i * ld + bj], y = Mm[(long long)sw[i] * ld + sw[bj]];
          nsg[i] = (x < 0.0) == (y < 0.0) ? sg[bj] : -sg[bj];
          s_changed = 1;
        }
      }
      __syncthreads();
      const int ch = s_changed;
      for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (!sg[i]) sg[i] = nsg[i];
      __syncthreads();
      if (!ch) {
        if (!strict) break;
        strict = 0;
      }
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      ws.sgn[mat * ld + i] = sg[i];
      ws.comp[mat * ld + i] = lab[i];
      ws.okc[mat * ld + i] = 1;
    }
  } else {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int l = lab[i];
      int pos = 0;
      for (int j = 0; j < n; ++j) pos += (lab[j] < l) || (lab[j] == l && j < i);
      ws.perm[mat * ld + (c.bad ? i : pos)] = i;
      ws.comp[mat * ld + i] = l;
    }
  }
}

// components in which the exchange holds to eight times the rounding (an asymmetry that the run
// itself built up): a warp per row
__global__ void __launch_bounds__(256) eig_verify_kernel(const double* __restrict__ M, EigWs ws) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const EigCtl c = ws.ctl[mat];
  if (c.bad) return;
  const double* Mm = M + (long long)mat * ld * ld;
  const int *sw = ws.swp + mat * ld, *lab = ws.comp + mat * ld, *sg = ws.sgn + mat * ld;
  const int pi = sw[i], l = lab[i];
  const Noise nz(c.top, 8.0);
  const double di = Mm[(long long)i * ld + i];
  int odd = sg[i] == 0 || sg[i] != sg[pi] || lab[pi] != l;
#pragma unroll 4
  for (int j = lane; j < n; j += 32) {
    if (lab[j] != l) continue;
    const double x = Mm[(long long)i * ld + j], y = Mm[(long long)pi * ld + sw[j]];
    if (nz.coupled(sg[i] == sg[j] ? x - y : x + y, di, Mm[(long long)j * ld + j])) odd = 1;
  }
  if (__any_sync(0xffffffffu, odd) && lane == 0) ws.okc[mat * ld + l] = 0;
}

// ap: in the components where the exchange holds, the combinations (e_i + s e_Pi) / sqrt 2 at the
// smaller and (e_i - s e_Pi) / sqrt 2 at the larger index of a pair, zeros between even and odd;
// zeros between components
__global__ void __launch_bounds__(256) eig_basis_kernel(const double* __restrict__ M, EigWs ws) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  if (ws.ctl[mat].bad) return;
  const double* Mm = M + (long long)mat * ld * ld;
  double* out = ws.ap + (long long)mat * ld * ld + (long long)i * ld;
  const int *sw = ws.swp + mat * ld, *lab = ws.comp + mat * ld, *sg = ws.sgn + mat * ld;
  const int l = lab[i];
  const bool sym = ws.okc[mat * ld + l] != 0;
  if (lane == 0) ws.sym[mat * ld + i] = sym;
  const int pi = sym ? sw[i] : i, i0 = min(i, pi), i1 = max(i, pi), si = sg[i];
  const bool fi = pi == i;
  const int ci = fi ? si : (i == i0 ? 1 : -1);   // class: +1 even, -1 odd
  if (lane == 0) ws.icl[mat * ld + i] = sym ? ci * (l + 1) : 0;
  for (int j = lane; j < n; j += 32) {
    double x = 0.0;
    if (lab[j] == l) {
      if (!sym) {
        x = Mm[(long long)i * ld + j];
      } else {
        const int pj = sw[j], j0 = min(j, pj), j1 = max(j, pj), sj = sg[j];
        const bool fj = pj == j;
        const int cj = fj ? sj : (j == j0 ? 1 : -1);
        if (ci == cj) {
          // averaged over the exchange: (i0, j0) with (i1, j1), (i0, j1) with (i1, j0)
          const double ss = si == sj ? 1.0 : -1.0;
          const double a = 0.5 * (Mm[(long long)i0 * ld + j0] + ss * Mm[(long long)i1 * ld + j1]);
          const double b = 0.5 * (Mm[(long long)i0 * ld + j1] + ss * Mm[(long long)i1 * ld + j0]);
          if (fi && fj) x = a;
          else if (fi) x = 0.70710678118654752440 * (a + (cj * sj > 0 ? b : -b));
          else if (fj) x = 0.70710678118654752440 * (a + (ci * si > 0 ? ss * b : -ss * b));
          else x = a + (cj * sj > 0 ? b : -b);
        }
      }
    }
    out[j] = x;
  }
}

// ---------------------------------------------------------------------------
// Householder reduction: a cluster of C CTAs per matrix, row i of the (full, symmetric)
// matrix on CTA i mod C, in shared memory while n^2 / C doubles fit, else in `rowbuf`.  Step k:
//   u = row k beyond its diagonal, u_{k+1} -= beta, H = I - tau u u^T (the reflector is the row
//   itself but for one element), then one fused pass over the rows below k: the rank-2 update of
//   step k - 1 and the product with u, 3 FP64 FMA per element, two rows per warp.
// Everything of order n (w, the next row, beta and tau) is computed by every CTA for itself, so a
// step needs one cluster barrier: the entries of A u are pushed to all CTAs, row k + 1 is pulled
// from its owner.  Bound by the chain of FP64 warp instructions of a step: each holds a quarter of
// the SM for about 64 clocks (measured: a warp alone issues one per 64, whether they depend on one
// another or not), so the order-n work is spread over four warps and every sum over lanes counts.
// ---------------------------------------------------------------------------
template <int EPT>   // elements of a row per thread
__global__ void __launch_bounds__(kTriThreads, 1) eig_tridiag_kernel(EigWs ws, int in_smem, double* rowbuf) {
  extern __shared__ __align__(16) double tsm[];
  __shared__ double s_part[2][kVecThreads / 32], s_tau, s_ht;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int mat = blockIdx.x / C, n = ws.na[mat], ld = ws.n, nrow = (n + C - 1) / C;
  const long long nn = (long long)ld * ld;
  double* q = tsm;              // [2][n] A u, pushed by every CTA
  double* vb = q + 2 * n;       // [2][n] u of this step and of the one before
  double* w = vb + 2 * n;       // [n]
  double* rows = in_smem ? w + n : rowbuf + (long long)mat * (ld + 16) * ld + (long long)rank * nrow * n;
  const double* Am = ws.ap + (long long)mat * nn;
  const int* pm = ws.perm + mat * ld;
  const int* cm = ws.comp + mat * ld;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = kTriThreads / 32;
  double* gd = ws.d + mat * ld;
  double* ge = ws.e + mat * ld;
  double* gt = ws.tau + mat * ld;
  double* gv = ws.vh + (long long)mat * nn;
  for (int lr = warp; lr < nrow; lr += NW) {
    const int i = lr * C + rank;
    if (i >= n) break;
    const double* src = Am + (long long)pm[i] * ld;
    const int ci = cm[pm[i]];
    for (int j = lane; j < n; j += 32) rows[(long long)lr * n + j] = cm[pm[j]] == ci ? src[pm[j]] : 0.0;
  }
  // sum of one value per thread over the first four warps, in each of their threads
  auto vec_sum = [&](double x, double* part) {
    x = warp_sum(x);
    if (lane == 0) part[warp] = x;
    asm volatile("bar.sync 1, %0;" ::"n"(kVecThreads) : "memory");
    x = part[lane & 3];
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    return x;
  };
  double beta = 0.0, tau = 0.0;
  // warp 0: beta of the row in v with x2 = sum of its squares beyond k + 1; u_{k+1} = alpha - beta.
  // Sums below 1e-60 (entries below 1e-30 of the largest element) count as zero: H = I, u = 0.
  auto reflector = [&](int k, double* v, double x2) {
    const double alpha = v[k + 1];
    const bool zero = !(x2 > 1e-60);
    beta = alpha;
    if (!zero) {
      x2 = fma(alpha, alpha, x2);
      beta = -copysign(x2 * rsqrt_newton(x2), alpha);
    }
    __syncwarp();
    if (lane == 0) v[k + 1] = zero ? 0.0 : alpha - beta;
    if (zero)
      for (int j = k + 2 + lane; j < n; j += 32) v[j] = 0.0;
  };
  {
    const double* src = Am + (long long)pm[0] * ld;
    if (tid < kVecThreads) {
      double x2 = 0.0;
      for (int j = tid; j < n; j += kVecThreads) {
        const double x = cm[pm[j]] == cm[pm[0]] ? src[pm[j]] : 0.0;
        vb[j] = x;
        w[j] = 0.0;
        vb[n + j] = 0.0;
        if (j >= 2) x2 = fma(x, x, x2);
      }
      x2 = vec_sum(x2, s_part[0]);
      if (warp == 0 && n > 2) reflector(0, vb, x2);
    }
  }
  __syncthreads();
  cluster.sync();   // every CTA of the cluster runs before any remote access
  for (int k = 0; k + 2 < n; ++k) {
    double* v = vb + (k & 1) * n;
    double* vo = vb + ((k + 1) & 1) * n;
    double* qk = q + (k & 1) * n;
    // ---- tau and the record of the reflector, behind the other warps' rows
    if (warp == 0) {
      const double u1 = v[k + 1];
      tau = u1 == 0.0 ? 0.0 : -1.0 / (beta * u1);
      if (lane == 0) {
        s_tau = tau;
        s_ht = 0.5 * tau * tau;
        if (rank == 0) {
          gd[k] = v[k];
          ge[k] = beta;
          gt[k] = tau;
        }
      }
    }
    if (rank == 0)
      for (int j = k + 1 + tid; j < n; j += kTriThreads) gv[(long long)k * ld + j] = v[j];
    // ---- rows i > k: the update of step k - 1, then q_i = A_i . u
    {
      int l0 = (k + 1 - rank + C - 1) / C;   // first local row with i > k
      if (l0 < 0) l0 = 0;
      const int lend = (n - rank + C - 1) / C;   // rows of this CTA
      for (int lr = l0 + 2 * (NW - 1 - warp); lr < lend; lr += 2 * NW) {   // warp 0 last: it has tau to form
        const bool two = lr + 1 < lend;
        const int i0 = lr * C + rank, i1 = two ? i0 + C : i0;
        double* row0 = rows + (long long)lr * n;
        double* row1 = two ? row0 + n : row0;
        const double v0 = vo[i0], w0 = w[i0], v1 = vo[i1], w1 = w[i1];
        double s0 = 0.0, s1 = 0.0;
        // loads of two chunks ahead of the arithmetic (the stores to the rows keep the compiler from
        // moving loads up)
        for (int j = ((k + 1) & ~31) + lane; j < n; j += 64) {
          const int j2 = j + 32;
          const bool a_in = j > k, b_in = j2 < n;
          double a0 = 0.0, a1 = 0.0, b0 = 0.0, b1 = 0.0;
          double wa = 0.0, oa = 0.0, va = 0.0, wb = 0.0, ob = 0.0, vv = 0.0;
          if (a_in) {
            a0 = row0[j];
            a1 = row1[j];
            wa = w[j];
            oa = vo[j];
            va = v[j];
          }
          if (b_in) {
            b0 = row0[j2];
            b1 = row1[j2];
            wb = w[j2];
            ob = vo[j2];
            vv = v[j2];
          }
          a0 = fma(-w0, oa, fma(-v0, wa, a0));
          s0 = fma(a0, va, s0);
          if (two) {
            a1 = fma(-w1, oa, fma(-v1, wa, a1));
            s1 = fma(a1, va, s1);
          }
          if (a_in) {
            row0[j] = a0;
            if (two) row1[j] = a1;
          }
          if (j - lane + 32 < n) {   // the second chunk holds columns
            b0 = fma(-w0, ob, fma(-v0, wb, b0));
            s0 = fma(b0, vv, s0);
            if (two) {
              b1 = fma(-w1, ob, fma(-v1, wb, b1));
              s1 = fma(b1, vv, s1);
            }
            if (b_in) {
              row0[j2] = b0;
              if (two) row1[j2] = b1;
            }
          }
        }
        // both sums at once: lanes 0 .. 15 keep the first, 16 .. 31 the second
        double x = lane < 16 ? s0 : s1;
        x += __shfl_xor_sync(0xffffffffu, lane < 16 ? s1 : s0, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        // lane l < 16 pushes q_i0 to CTA l, lane 16 + l q_i1
        if ((lane & 15) < C && (two || lane < 16)) *cluster.map_shared_rank(qk + (lane < 16 ? i0 : i1), lane & 15) = x;
      }
    }
    cluster.sync();
    // ---- w, row k + 1 after this step's update (into the other buffer), its reflector
    if (tid < kVecThreads) {
      const int own = (k + 1) % C, olr = (k + 1) / C;
      const double* orow = in_smem ? cluster.map_shared_rank(rows + (long long)olr * n, own)
                                   : rowbuf + (long long)mat * (ld + 16) * ld + ((long long)own * nrow + olr) * n;
      const double v1 = v[k + 1], q1 = qk[k + 1];
      tau = s_tau;
      double rr[EPT], qq[EPT], vv[EPT], p = 0.0;
#pragma unroll
      for (int u = 0; u < EPT; ++u) {
        const int j = tid + kVecThreads * u;
        const bool in = j > k && j < n;
        rr[u] = in ? (in_smem ? orow[j] : __ldcg(orow + j)) : 0.0;
        qq[u] = in ? qk[j] : 0.0;
        vv[u] = in ? v[j] : 0.0;
        p = fma(qq[u], vv[u], p);
      }
      p = vec_sum(p, s_part[0]);
      const double hc = s_ht * p;
      const double w1 = fma(tau, q1, -hc * v1);
      double x2 = 0.0;
#pragma unroll
      for (int u = 0; u < EPT; ++u) {
        const int j = tid + kVecThreads * u;
        const double wj = fma(tau, qq[u], -hc * vv[u]);
        const double x = fma(-v1, wj, fma(-w1, vv[u], rr[u]));
        if (j > k && j < n) {
          w[j] = wj;
          vo[j] = x;
        }
        if (j > k + 2) x2 = fma(x, x, x2);   // beyond n: zeros
      }
      x2 = vec_sum(x2, s_part[1]);
      if (warp == 0 && k + 3 < n) reflector(k + 1, vo, x2);
    }
    __syncthreads();
  }
  // ---- the last two rows
  if (n >= 2) {
    // row n - 2 as the last step left it (n = 2: row 0 as loaded)
    const double* r = n > 2 ? vb + ((n - 2) & 1) * n : vb;
    const double* vl = vb + ((n - 3) & 1) * n;
    if (rank == 0 && tid == 0) {
      gd[n - 2] = r[n - 2];
      ge[n - 2] = r[n - 1];
    }
    if (rank == (n - 1) % C && tid == 0) {
      const double a = rows[(long long)((n - 1) / C) * n + n - 1];
      gd[n - 1] = n > 2 ? fma(-2.0 * vl[n - 1], w[n - 1], a) : a;
    }
  } else if (rank == 0 && tid == 0) {
    gd[0] = vb[0];
  }
  cluster.sync();   // remote rows may still be being read
}

// ---------------------------------------------------------------------------
// Leaves: one warp per tridiagonal leaf (at most kLeaf rows), implicit QR with Wilkinson
// shifts (Golub & Van Loan, Alg. 8.3.2-8.3.3).  Lane l holds row l of the vectors.  A split
// point between rows b - 1 and b takes |e_{b-1}| from both diagonals (Cuppen).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(32) eig_leaf_kernel(EigWs ws, int leaves, double* ev, double* Q, DevState* st) {
  __shared__ double d[32], e[32], z[32 * 33];
  const int lane = threadIdx.x & 31;
  const int gl = blockIdx.x;
  const int mat = gl / leaves, leaf = gl % leaves, n = ws.na[mat], ld = ws.n;
  if (ws.ctl[mat].bad) return;
  const int lo = (int)((long long)leaf * n / leaves), hi = (int)((long long)(leaf + 1) * n / leaves), m = hi - lo;
  const double* gd = ws.d + mat * ld;
  const double* ge = ws.e + mat * ld;
  if (lane < m) {
    double x = gd[lo + lane];
    if (lane == 0 && lo > 0) x -= fabs(ge[lo - 1]);
    if (lane == m - 1 && hi < n) x -= fabs(ge[hi - 1]);
    d[lane] = x;
    e[lane] = lane + 1 < m ? ge[lo + lane] : 0.0;
    for (int j = 0; j < m; ++j) z[lane * 33 + j] = j == lane ? 1.0 : 0.0;
  }
  __syncwarp();
  double big = lane < m ? fabs(d[lane]) + fabs(e[lane]) : 0.0;
  for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
  // the matrix is scaled to max |A| in [0.5, 1): couplings below eps / 1024 change no eigenvalue's
  // leading digits (and a leaf of pure rounding noise would never converge relative to itself)
  const double floor_ = fmax(big * 0.015625, 0.0009765625) * kEps;
  int most = 0;
  // every lane runs the same scalar recurrence on the shared d, e; lane 0 stores them
  for (int m1 = m - 1; m1 > 0;) {
    int it = 0;
    while (true) {
      // smallest l with no negligible coupling in l .. m1
      int l = m1;
      while (l > 0) {
        if (fabs(e[l - 1]) <= kEps * (fabs(d[l - 1]) + fabs(d[l])) + floor_) break;
        --l;
      }
      if (l == m1) break;
      if (++it > 80) {
        if (lane == 0 && st->status == 0) st->status = HOTRG_ENOTCONV;
        break;
      }
      const double b1 = e[m1 - 1], dm = d[m1];
      const double hd = 0.5 * (d[m1 - 1] - dm);
      const double mu = dm - b1 * b1 / (hd + copysign(sqrt(fma(hd, hd, b1 * b1)), hd));
      double x = d[l] - mu, zz = e[l];
      double dk = d[l], ek = e[l];
      for (int k = l; k < m1; ++k) {
        const double r2 = fma(x, x, zz * zz);
        double c = 1.0, s = 0.0, rr = 0.0;
        if (r2 > 1e-290) {
          const double ir = rsqrt_newton(r2);
          c = x * ir;
          s = zz * ir;
          rr = r2 * ir;
        }
        const double dn = d[k + 1], en = k + 1 < m1 ? e[k + 1] : 0.0;
        const double cs = c * s, c2 = c * c, s2 = s * s;
        const double nd = fma(c2, dk, fma(2.0 * cs, ek, s2 * dn));
        const double nd1 = fma(s2, dk, fma(-2.0 * cs, ek, c2 * dn));
        const double ne = fma(c2 - s2, ek, cs * (dn - dk));
        __syncwarp();
        if (lane == 0) {
          if (k > l) e[k - 1] = rr;
          d[k] = nd;
          if (k + 1 == m1) {
            d[m1] = nd1;
            e[k] = ne;
          }
        }
        if (lane < m) {
          const double z0 = z[lane * 33 + k], z1 = z[lane * 33 + k + 1];
          z[lane * 33 + k] = fma(c, z0, s * z1);
          z[lane * 33 + k + 1] = fma(c, z1, -s * z0);
        }
        x = ne;
        zz = s * en;
        dk = nd1;
        ek = c * en;
      }
      __syncwarp();
    }
    most = most > it ? most : it;
    --m1;
  }
  __syncwarp();
  // ascending
  if (lane < m) {
    const double x = d[lane];
    int pos = 0;
    for (int j = 0; j < m; ++j) pos += d[j] < x || (d[j] == x && j < lane);
    ev[mat * ld + lo + pos] = x;
    e[lane] = (double)pos;
  }
  __syncwarp();
  double* Qm = Q + (long long)mat * ld * ld;
  for (int j = 0; j < m; ++j)
    if (lane < m) Qm[(long long)(lo + (int)e[j]) * ld + lo + lane] = z[lane * 33 + j];
  if (lane == 0) atomicMax(&ws.ctl[mat].iters, most);
}

// ---------------------------------------------------------------------------
// Merge of two nodes, T = diag(T1, T2) + rho u u^T = Q (D + rho z z^T) Q^T, in five kernels:
// prep (order, deflation), roots, weights, vectors, product.  grid.y: (matrix, node).
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool merge_view(const EigWs& ws, int nodes, int g, int& mat, int& lo, int& mid, int& hi) {
  mat = g / nodes;
  const int node = g % nodes, n = ws.na[mat];
  lo = (int)((long long)node * n / nodes);
  hi = (int)((long long)(node + 1) * n / nodes);
  mid = (int)((long long)(2 * node + 1) * n / (2 * nodes));
  return ws.ctl[mat].bad == 0;
}

// The order of the poles and the deflation (LAPACK Users' Guide's criteria: a weight, or the
// coupling that a rotation of two close poles would leave, below 8 eps).
__global__ void __launch_bounds__(256) eig_prep_kernel(EigWs ws, int nodes, const double* __restrict__ ev,
                                                       const double* __restrict__ Q) {
  __shared__ double sd[kEigMaxN], sz[kEigMaxN];
  __shared__ short scol[kEigMaxN];
  __shared__ unsigned char styp[kEigMaxN];
  __shared__ short surv[kEigMaxN], acc[kEigMaxN], ltop[kEigMaxN], lbot[kEigMaxN];
  __shared__ unsigned char flag[kEigMaxN];
  __shared__ double redm[16], s_tol;
  __shared__ int s_ns, s_nd, s_k, s_nt, s_nb;
  int mat, lo, mid, hi;
  if (!merge_view(ws, nodes, blockIdx.x, mat, lo, mid, hi)) return;
  const int n = ws.n, m = hi - lo, n1 = mid - lo, n2 = hi - mid;
  const double* evm = ev + mat * n;
  const double* Qm = Q + (long long)mat * n * n;
  // an empty half (orders far below the batch's): no coupling, every column is kept
  const double off = n1 > 0 && n2 > 0 ? ws.e[mat * n + mid - 1] : 0.0;
  const double rho = 2.0 * fabs(off), sg = off < 0.0 ? -1.0 : 1.0;
  const double rt = 0.70710678118654752440;
  double md = 0.0, mz = 0.0;
  for (int t = threadIdx.x; t < m; t += blockDim.x) {
    const int col = lo + t;
    const double x = evm[col];
    int pos;
    if (t < n1) {   // own index + entries of the second half below x
      int a = 0, b = n2;
      while (a < b) {
        const int c = (a + b) >> 1;
        if (evm[mid + c] < x) a = c + 1;
        else b = c;
      }
      pos = t + a;
    } else {        // own index + entries of the first half not above x
      int a = 0, b = n1;
      while (a < b) {
        const int c = (a + b) >> 1;
        if (evm[lo + c] <= x) a = c + 1;
        else b = c;
      }
      pos = t - n1 + a;
    }
    const double z = t < n1 ? (n2 > 0 ? rt * Qm[(long long)col * n + mid - 1] : 0.0)
                            : (n1 > 0 ? sg * rt * Qm[(long long)col * n + mid] : 0.0);
    sd[pos] = x;
    sz[pos] = z;
    scol[pos] = (short)col;
    styp[pos] = t < n1 ? 1 : 2;
    md = fmax(md, fabs(x));
    mz = fmax(mz, fabs(z));
  }
  for (int o = 16; o > 0; o >>= 1) {
    md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
    mz = fmax(mz, __shfl_xor_sync(0xffffffffu, mz, o));
  }
  if ((threadIdx.x & 31) == 0) redm[threadIdx.x >> 5] = fmax(md, mz);
  __syncthreads();
  if (threadIdx.x == 0) {
    double tol = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tol = fmax(tol, redm[q]);
    tol *= 8.0 * kEps;
    s_tol = tol;
  }
  __syncthreads();
  const double tol = s_tol;
  const int base = mat * n + lo;
  // poles with a negligible weight deflate (val is filled from its end: val[m - 1 - i] belongs
  // to defl[i]); the others are packed, warp 0 counting
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int ns = 0, nd = 0;
    for (int t0 = 0; t0 < m; t0 += 32) {
      const int t = t0 + lane;
      const bool in = t < m, keep = in && rho * fabs(sz[t]) > tol;
      const unsigned mk = __ballot_sync(0xffffffffu, keep), md_ = __ballot_sync(0xffffffffu, in && !keep);
      const unsigned below = (1u << lane) - 1u;
      if (keep) surv[ns + __popc(mk & below)] = (short)t;
      if (in && !keep) {
        const int i = nd + __popc(md_ & below);
        ws.val[base + m - 1 - i] = sd[t];
        ws.defl[base + i] = scol[t];
      }
      ns += __popc(mk);
      nd += __popc(md_);
    }
    if (lane == 0) {
      s_ns = ns;
      s_nd = nd;
    }
  }
  __syncthreads();
  const int ns = s_ns;
  // close neighbours: the coupling that a rotation would leave is negligible
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    bool close = false;
    if (i > 0) {
      const int a = surv[i - 1], b = surv[i];
      close = fabs((sd[b] - sd[a]) * sz[a] * sz[b]) <= tol * fma(sz[a], sz[a], sz[b] * sz[b]);
    }
    flag[i] = close ? 1 : 0;
  }
  __syncthreads();
  // one thread walks the packed poles: without close pairs it only copies; after a rotation the
  // surviving pole has moved, and its next neighbour is tested again
  if (threadIdx.x == 0) {
    int K = 0, nd = s_nd, nr = 0, nt = 0, nb = 0;
    bool moved = false;
    for (int i = 1; i <= ns; ++i) {
      const int a = surv[i - 1];
      bool close = false;
      if (i < ns) {
        const int b = surv[i];
        close = flag[i] != 0;
        if (moved) close = fabs((sd[b] - sd[a]) * sz[a] * sz[b]) <= tol * fma(sz[a], sz[a], sz[b] * sz[b]);
        if (close) {
          const double pd = sd[a], pz = sz[a], xd = sd[b], xz = sz[b];
          const double tz = sqrt(fma(pz, pz, xz * xz)), c = xz / tz, s = -pz / tz;
          ws.rp[base + nr] = scol[a];
          ws.rq[base + nr] = scol[b];
          ws.rc[base + nr] = c;
          ws.rs[base + nr] = s;
          ++nr;
          ws.val[base + m - 1 - nd] = fma(pd * c, c, xd * s * s);
          ws.defl[base + nd++] = scol[a];
          sd[b] = fma(pd * s, s, xd * c * c);
          sz[b] = tz;
          styp[b] |= styp[a];
        }
      }
      moved = close;
      if (!close) {
        acc[K] = (short)a;
        if (styp[a] & 1) ltop[nt++] = (short)K;
        if (styp[a] & 2) lbot[nb++] = (short)K;
        ++K;
      }
    }
    MergeCtl c;
    c.k = K;
    c.nrot = nr;
    c.ntop = nt;
    c.nbot = nb;
    ws.mc[blockIdx.x] = c;
    s_k = K;
    s_nt = nt;
    s_nb = nb;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < s_k; i += blockDim.x) {
    const int a = acc[i];
    ws.dk[base + i] = sd[a];
    ws.zk[base + i] = sz[a];
    ws.idx[base + i] = scol[a];
    if (i < s_nt) ws.top[base + i] = ltop[i];
    if (i < s_nb) ws.bot[base + i] = lbot[i];
  }
}

// Roots of 1 + rho sum_i z_i^2 / (d_i - x): one warp per root, x = d_org + mu with the nearer
// pole as origin, so that the differences d_i - x are accurate.  Each step matches the value and
// the slope of the poles on either side (Bunch, Nielsen & Sorensen; Li's form of the quadratic),
// inside a bracket.  Row j of `s` receives d_i - x_j.
// Two warps per CTA: the FP64 unit belongs to the SM, so the roots are spread over the chip.
__global__ void __launch_bounds__(64) eig_roots_kernel(EigWs ws, int nodes) {
  int mat, lo, mid, hi;
  if (!merge_view(ws, nodes, blockIdx.y, mat, lo, mid, hi)) return;
  const int K = ws.mc[blockIdx.y].k;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= K) return;
  const int n = ws.n, base = mat * n + lo;
  const double rho = 2.0 * fabs(ws.e[mat * n + mid - 1]);
  const double* d = ws.dk + base;
  const double* z = ws.zk + base;
  const bool last = j == K - 1;
  const double dj = d[j], gap = last ? 0.0 : d[j + 1] - dj;
  double zz2 = 0.0;
  if (last)
    for (int i = lane; i < K; i += 32) zz2 = fma(z[i], z[i], zz2);
  zz2 = warp_sum(zz2);
  // f and the sums over the poles up to j and after it, at d_org + mu
  double psi, dpsi, phi, dphi;
  auto eval = [&](double dorg, double mu) {
    double a = 0.0, b = 0.0, c = 0.0, e = 0.0;
    for (int i = lane; i < K; i += 32) {
      const double inv = 1.0 / ((d[i] - dorg) - mu);
      const double t = rho * z[i] * z[i] * inv;
      if (i <= j) {
        a += t;
        b = fma(t, inv, b);
      } else {
        c += t;
        e = fma(t, inv, e);
      }
    }
    warp_sum4(a, b, c, e);
    psi = a;
    dpsi = b;
    phi = c;
    dphi = e;
    return 1.0 + psi + phi;
  };
  double dorg = dj, mu, blo, bhi, f;
  double p1 = 0.0, p2 = 0.0;   // poles j and j + 1 relative to the origin
  if (last) {
    blo = 0.0;
    bhi = rho * zz2 * (1.0 + 8.0 * kEps);   // above the root, which with one pole is rho z^2 itself
    mu = 0.5 * bhi;
    f = eval(dorg, mu);
  } else {
    mu = 0.5 * gap;
    f = eval(dj, mu);
    p2 = gap;
    if (f >= 0.0) {
      blo = 0.0;
      bhi = mu;
    } else {
      dorg = d[j + 1];
      p1 = -gap;
      p2 = 0.0;
      mu = -0.5 * gap;
      blo = mu;
      bhi = 0.0;
    }
  }
  for (int it = 0; it < 100; ++it) {
    if (fabs(f) <= 4.0 * kEps * (1.0 + fabs(psi) + fabs(phi))) break;
    if (f < 0.0) blo = mu;
    else bhi = mu;
    if (bhi - blo <= 2.0 * kEps * fmax(fabs(blo), fabs(bhi))) break;
    double eta;
    const double D1 = p1 - mu, D2 = p2 - mu;
    if (last) {
      // (1 + p) + q / (D1 - eta) = 0 with q = psi' D1^2, p = psi - psi' D1
      const double c = f - dpsi * D1;
      eta = c > 0.0 ? D1 + dpsi * D1 * D1 / c : bhi;
    } else {
      // c eta^2 - a eta + b = 0, scaled by a power of two and solved in FP32: the correction needs
      // only a few digits, the sums above carry the accuracy
      const double c = f - dpsi * D1 - dphi * D2;
      const double a = (D1 + D2) * f - D1 * D2 * (dpsi + dphi);
      const double b = D1 * D2 * f;
      const int ea = 0x7fe00000 - (__double2hiint(fmax(fabs(a), fabs(b))) & 0x7ff00000);
      const double sc = __hiloint2double(ea, 0);   // 2^-exponent
      const float af = (float)(a * sc), bf = (float)(b * sc), cf = (float)(c * sc);
      const float disc = sqrtf(fmaxf(0.0f, fmaf(af, af, -4.0f * bf * cf)));
      eta = (double)(af <= 0.0f ? (af - disc) / (2.0f * cf) : 2.0f * bf / (af + disc));
    }
    double nx = mu + eta;
    if (!(nx > blo && nx < bhi)) {
      // bisection, on the logarithm where the bracket spans more than a factor of four
      const double al = fmin(fabs(blo), fabs(bhi)), ah = fmax(fabs(blo), fabs(bhi));
      const double sgn = bhi > 0.0 ? 1.0 : -1.0;
      if (al == 0.0) nx = sgn * ah * 0.0625;
      else if (ah > 4.0 * al) nx = sgn * sqrt(al) * sqrt(ah);
      else nx = 0.5 * (blo + bhi);
      if (!(nx > blo && nx < bhi)) break;
    }
    if (nx == mu) break;
    mu = nx;
    f = eval(dorg, mu);
  }
  double* row = ws.s + (long long)mat * n * n + (long long)(lo + j) * n + lo;
  for (int i = lane; i < K; i += 32) row[i] = (d[i] - dorg) - mu;
  if (lane == 0) ws.val[base + j] = dorg + mu;
}

// Weights of which the computed roots are the exact ones (Gu & Eisenstat, Eq. 3.3, by Loewner's
// formula): z^_i^2 = (x_i - d_i) prod_{j != i} (x_j - d_i) / (d_j - d_i), up to a common factor.
// Threads along i (coalesced columns of s), eight slices of j.
__global__ void __launch_bounds__(256) eig_weights_kernel(EigWs ws, int nodes) {
  __shared__ double part[8][33];
  int mat, lo, mid, hi;
  if (!merge_view(ws, nodes, blockIdx.y, mat, lo, mid, hi)) return;
  const int K = ws.mc[blockIdx.y].k;
  if ((int)blockIdx.x * 32 >= K) return;
  const int n = ws.n, base = mat * n + lo;
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), y = threadIdx.x >> 5;
  const double* d = ws.dk + base;
  const double* s = ws.s + (long long)mat * n * n + (long long)lo * n + lo;
  double p = 1.0;
  if (i < K) {
    const double di = d[i];
    for (int j = y; j < K; j += 8) {
      const double x = s[(long long)j * n + i];
      p *= j == i ? -x : x / (di - d[j]);
    }
  }
  part[y][threadIdx.x & 31] = p;
  __syncthreads();
  if (y == 0 && i < K) {
    for (int q = 1; q < 8; ++q) p *= part[q][threadIdx.x & 31];
    ws.zh[base + i] = copysign(sqrt(fabs(p)), ws.zk[base + i]);
  }
}

// Vectors of the secular equation, s_ji = z^_i / (d_i - x_j), normalised (warps j < k), and the
// place of every new eigenvalue in the ascending order (all warps): the deflated ones keep
// their columns.
__global__ void __launch_bounds__(256) eig_vectors_kernel(EigWs ws, int nodes, double* __restrict__ ev, int* pos) {
  int mat, lo, mid, hi;
  if (!merge_view(ws, nodes, blockIdx.y, mat, lo, mid, hi)) return;
  const int K = ws.mc[blockIdx.y].k, n = ws.n, m = hi - lo, base = mat * n + lo;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= m) return;
  if (j < K) {
    double* row = ws.s + (long long)mat * n * n + (long long)(lo + j) * n + lo;
    const double* zh = ws.zh + base;
    double a = 0.0;
    for (int i = lane; i < K; i += 32) {
      const double x = zh[i] / row[i];
      row[i] = x;
      a = fma(x, x, a);
    }
    a = 1.0 / sqrt(warp_sum(a));
    for (int i = lane; i < K; i += 32) row[i] *= a;
  }
  // val: roots in 0 .. K-1, the value of deflated column i at m - 1 - i
  const double* val = ws.val + base;
  const double x = j < K ? val[j] : val[m - 1 - (j - K)];
  int c = 0;
  for (int i = lane; i < m; i += 32) {
    const double y = i < K ? val[i] : val[m - 1 - (i - K)];
    c += y < x || (y == x && i < j);
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) {
    pos[base + j] = lo + c;
    ev[base + c] = x;
  }
}

// The deflation's rotations on the columns of Q, a thread per row.  A rotation's second column
// is always untouched before it, so its loads run ahead; the first is the one just written or
// an untouched one.
__global__ void __launch_bounds__(64) eig_rotate_kernel(EigWs ws, int nodes, double* Q) {
  int mat, lo, mid, hi;
  if (!merge_view(ws, nodes, blockIdx.y, mat, lo, mid, hi)) return;
  const int nr = ws.mc[blockIdx.y].nrot;
  const int row = lo + blockIdx.x * 64 + threadIdx.x;
  if (nr == 0 || row >= hi) return;
  const int n = ws.n, base = mat * n + lo;
  double* Qm = Q + (long long)mat * n * n + row;
  const int* rp = ws.rp + base;
  const int* rq = ws.rq + base;
  int prev = -1;
  double carry = 0.0;
  for (int t0 = 0; t0 < nr; t0 += 8) {
    double y[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) y[u] = t0 + u < nr ? Qm[(long long)rq[t0 + u] * n] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int t = t0 + u;
      if (t >= nr) break;
      const int p = rp[t];
      if (p != prev) {
        if (prev >= 0) Qm[(long long)prev * n] = carry;
        carry = Qm[(long long)p * n];
      }
      const double c = ws.rc[base + t], s = ws.rs[base + t];
      Qm[(long long)p * n] = fma(c, carry, s * y[u]);
      carry = fma(c, y[u], -s * carry);
      prev = rq[t];
    }
  }
  Qm[(long long)prev * n] = carry;
}

// New vectors: column pos[j] = sum_i s_ji Q[:, idx_i] for the roots (rows of the first half sum
// over `top` only, those of the second over `bot`), a copy for the deflated.  32 x 32 tiles
// (FP64 issue bounds it, and small tiles spread n^3 over the chip), 2 x 2 per thread.
__global__ void __launch_bounds__(256) eig_product_kernel(EigWs ws, int nodes, const double* __restrict__ Q,
                                                          double* __restrict__ Qn, const int* __restrict__ pos) {
  constexpr int BK = 16;
  __shared__ double As[BK][33], Bs[BK][33];
  int mat, lo, mid, hi;
  if (!merge_view(ws, nodes, blockIdx.z, mat, lo, mid, hi)) return;
  const MergeCtl mc = ws.mc[blockIdx.z];
  const int n = ws.n, m = hi - lo, K = mc.k, base = mat * n + lo;
  // row tiles: first half, then second
  const int t1 = (mid - lo + 31) / 32;
  const bool second = (int)blockIdx.x >= t1;
  const int r0 = second ? mid + ((int)blockIdx.x - t1) * 32 : lo + (int)blockIdx.x * 32;
  const int rend = second ? hi : mid;
  if (r0 >= rend) return;
  const int j0 = blockIdx.y * 32;
  if (j0 >= m) return;
  const int kk = second ? mc.nbot : mc.ntop;
  const int* list = (second ? ws.bot : ws.top) + base;
  const int* idx = ws.idx + base;
  const double* S = ws.s + (long long)mat * n * n + (long long)lo * n + lo;
  const double* Qm = Q + (long long)mat * n * n;
  double* Qo = Qn + (long long)mat * n * n;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;   // tx: rows, ty: columns j
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  if (j0 < K) {
    for (int k0 = 0; k0 < kk; k0 += BK) {
      {
        // As[k][r]: rows contiguous in Q; Bs[k][j]: gathered from row j of S
        const int r = tid & 31, kq = tid >> 5;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = k0 + kq + 8 * u;
          As[kq + 8 * u][r] = (k < kk && r0 + r < rend) ? Qm[(long long)idx[list[k]] * n + r0 + r] : 0.0;
        }
        const int k = k0 + (tid & 15), jq = tid >> 4;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int j = j0 + jq + 16 * u;
          Bs[tid & 15][jq + 16 * u] = (k < kk && j < K) ? S[(long long)j * n + list[k]] : 0.0;
        }
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < BK; ++k) {
        const double a0 = As[k][tx], a1 = As[k][tx + 16], b0 = Bs[k][ty], b1 = Bs[k][ty + 16];
        acc[0][0] = fma(a0, b0, acc[0][0]);
        acc[0][1] = fma(a0, b1, acc[0][1]);
        acc[1][0] = fma(a1, b0, acc[1][0]);
        acc[1][1] = fma(a1, b1, acc[1][1]);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int j = j0 + ty + 16 * v;
    if (j >= m) continue;
    double* out = Qo + (long long)pos[base + j] * n;
    const double* src = j < K ? nullptr : Qm + (long long)ws.defl[base + j - K] * n;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = r0 + tx + 16 * u;
      if (r < rend) out[r] = j < K ? acc[u][v] : src[r];
    }
  }
}

// V = H_0 H_1 .. H_{n-3} Z in blocks of kRb reflectors, H_b .. H_{b+r-1} = I - U^T T U (rows of U
// the reflectors, T upper triangular: Schreiber & Van Loan's compact form).
constexpr int kStrip = 8;    // eigenvectors per CTA

// T of every block: T_ii = tau_i, T[0:i, i] = -tau_i T[0:i, 0:i] (U u_i)[0:i]
__global__ void __launch_bounds__(256) eig_tfactor_kernel(EigWs ws, double* tf) {
  __shared__ double g[kRb][kRb + 1], t[kRb][kRb + 1];
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n, b0 = blockIdx.x * kRb;
  const int r = min(kRb, n - 2 - b0);
  if (r <= 0) return;
  const double* vh = ws.vh + (long long)mat * ld * ld;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // pairs (p, q > p) of the block: u_q begins at q + 1
  for (int e = warp; e < kRb * kRb; e += 8) {
    const int p = e / kRb, q = e % kRb;
    if (p >= q || q >= r) continue;
    const double *up = vh + (long long)(b0 + p) * ld, *uq = vh + (long long)(b0 + q) * ld;
    double a = 0.0;
    for (int i = b0 + q + 1 + lane; i < n; i += 32) a = fma(up[i], uq[i], a);
    a = warp_sum(a);
    if (lane == 0) g[p][q] = a;
  }
  __syncthreads();
  if (warp == 0) {
    const double* tau = ws.tau + mat * ld + b0;
    for (int q = 0; q < kRb; ++q) {
      double x = 0.0;
      if (q < r) {
        if (lane < q) {
          for (int c = lane; c < q; ++c) x = fma(t[lane][c], g[c][q], x);
          x *= -tau[q];
        } else if (lane == q) {
          x = tau[q];
        }
      }
      if (lane < kRb) t[lane][q] = x;
      __syncwarp();
    }
  }
  __syncthreads();
  double* out = tf + ((long long)mat * gridDim.x + blockIdx.x) * kRb * kRb;
  out[threadIdx.x] = t[threadIdx.x / kRb][threadIdx.x % kRb];
}

// A CTA holds kStrip eigenvectors in shared memory and applies the blocks from the last to the
// first: W = U Z (a thread per output and half of the sum, no shuffles), W <- T W, Z -= U^T W.  The FP64
// unit bounds it: n^3 multiply-adds per matrix over the chip (4 x 288: 0.16 ms at the full rate).
// Rows return to A's order; NaN for a matrix with non-finite elements.
__global__ void __launch_bounds__(256) eig_back_kernel(EigWs ws, const double* __restrict__ Z,
                                                       const double* __restrict__ ev, const double* __restrict__ tf,
                                                       int nblk, double* __restrict__ V, double* __restrict__ lam) {
  extern __shared__ double bsm[];
  const int ld = ws.n, mat = blockIdx.y, n = ws.na[mat], j0 = blockIdx.x * kStrip;
  if (j0 >= n) return;
  const int zp = n | 1, tid = threadIdx.x;   // odd pitch: the eight columns land on different banks
  double* z = bsm;                       // [kStrip][zp]
  double* u = z + kStrip * zp;           // [kRb][zp]
  double* wp = u + kRb * zp;             // [2][kRb][kStrip]
  double* w = wp + 2 * kRb * kStrip;     // [kRb][kStrip]
  const long long nn = (long long)ld * ld;
  const bool bad = ws.ctl[mat].bad != 0;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  const double* vh = ws.vh + mat * nn;
  const int cols = min(kStrip, n - j0);
  for (int e = tid; e < kStrip * n; e += 256) {
    const int c = e / n, i = e - c * n;
    z[c * zp + i] = c < cols ? (bad ? nan : Z[mat * nn + (long long)(j0 + c) * ld + i]) : 0.0;
  }
  const int nb = (n - 2 + kRb - 1) / kRb;
  for (int b = (n > 2 && !bad) ? nb - 1 : -1; b >= 0; --b) {
    const int b0 = b * kRb, r = min(kRb, n - 2 - b0), i0 = b0 + 1;   // rows i0 .. n - 1 are touched
    __syncthreads();
    for (int q = tid >> 5; q < kRb; q += 8)
      for (int i = i0 + (tid & 31); i < n; i += 32)
        u[q * zp + i] = (q < r && i > b0 + q) ? vh[(long long)(b0 + q) * ld + i] : 0.0;
    __syncthreads();
    {
      // output (q, c), half h of the rows
      const int h = tid >> 7, q = (tid >> 3) & 15, c = tid & 7;
      const int mid = i0 + (n - i0) / 2;
      const int lo = h ? mid : i0, hi = h ? n : mid;
      double a0 = 0.0, a1 = 0.0;
      int i = lo;
      for (; i + 1 < hi; i += 2) {
        a0 = fma(u[q * zp + i], z[c * zp + i], a0);
        a1 = fma(u[q * zp + i + 1], z[c * zp + i + 1], a1);
      }
      if (i < hi) a0 = fma(u[q * zp + i], z[c * zp + i], a0);
      wp[tid] = a0 + a1;
    }
    __syncthreads();
    if (tid < kRb * kStrip) {
      const int q = tid >> 3, c = tid & 7;
      const double* t = tf + ((long long)mat * nblk + b) * kRb * kRb + q * kRb;
      double a = 0.0;
      for (int p = q; p < r; ++p) a = fma(t[p], wp[p * kStrip + c] + wp[kRb * kStrip + p * kStrip + c], a);
      w[tid] = -a;
    }
    __syncthreads();
    // thread: rows i, i + 32, .. of column c (warp c)
    {
      const int c = tid >> 5;
      double wr[kRb];
#pragma unroll
      for (int q = 0; q < kRb; ++q) wr[q] = w[q * kStrip + c];
      for (int i = i0 + (tid & 31); i < n; i += 32) {
        double a = z[c * zp + i];
#pragma unroll
        for (int q = 0; q < kRb; ++q) a = fma(u[q * zp + i], wr[q], a);
        z[c * zp + i] = a;
      }
    }
  }
  __syncthreads();
  // back to A's order and basis
  const int* pm = ws.perm + mat * ld;
  for (int e = tid; e < cols * n; e += 256) {
    const int c = e / n, i = e - c * n;
    u[c * zp + pm[i]] = z[c * zp + i];
  }
  __syncthreads();
  const int* sw = ws.swp + mat * ld;
  const int *lab = ws.sym + mat * ld, *sg = ws.sgn + mat * ld;   // 1: combinations at this index
  for (int e = tid; e < cols * n; e += 256) {
    const int c = e / n, i = e - c * n;
    double x = u[c * zp + i];
    if (!bad && lab[i] && sw[i] != i) {
      // x, y: the even and the odd combination's entries (in either order)
      const double y = u[c * zp + sw[i]];
      x = 0.70710678118654752440 * (i < sw[i] ? x + y : (sg[i] > 0 ? y - x : x - y));
    }
    V[mat * nn + (long long)(j0 + c) * ld + i] = x;
  }
  // class: that of the component that holds the vector
  if (tid < cols) {
    int k = 0;
    for (int i = 1; i < n; ++i)
      if (fabs(z[tid * zp + i]) > fabs(z[tid * zp + k])) k = i;
    ws.cls[mat * ld + j0 + tid] = bad ? 0 : ws.icl[mat * ld + pm[k]];
  }
  if (tid < cols) lam[mat * ld + j0 + tid] = bad ? nan : ev[mat * ld + j0 + tid] * ws.ctl[mat].unscale;
}

// ---------------------------------------------------------------------------
// One-sided (Hestenes) Jacobi for the smallest orders: W = A V is orthogonalised column pair by
// column pair by plane rotations applied to W and V; at convergence A v_i = lambda_i v_i with
// |lambda_i| = ||w_i||.  Round-robin ordering (n/2 disjoint pairs per round, n - 1 rounds per
// sweep), a warp per pair over the whole grid (the FP64 units of many SMs), a grid barrier
// between rounds.  A pair whose inner product is exactly 0 is never rotated, which keeps an
// exact block pattern of A exact.
//
// Stopping rule: a sweep counts only the rotations of pairs in which a column's squared norm
// exceeds (4 n eps)^2 times the largest squared column norm at the start: the near-null columns
// (rounding noise of order n eps lambda_1) are rotated too, but do not keep the sweeps going.
// ---------------------------------------------------------------------------
struct JacobiOrders {
  int n[kEigMaxMat];
};
__global__ void __launch_bounds__(256) jacobi_onesided_kernel(const double* __restrict__ A, double* W, double* V,
                                                              double* lam, int n, JacobiOrders na, int nmat, int max_sweeps,
                                                              int* counters, unsigned long long* colmax,
                                                              int* sweeps_out, DevState* st) {
  cg::grid_group grid = cg::this_grid();
  const int nn = n * n;
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
  const int gthreads = gridDim.x * blockDim.x;
  for (int e = gtid; e < nmat * nn; e += gthreads) {
    const int r = e % nn;
    __stcg(W + e, A[e]);                // A symmetric: row i = column i
    __stcg(V + e, r / n == r % n ? 1.0 : 0.0);
  }
  if (gtid < 3 * nmat) counters[gtid] = 0;
  if (gtid < nmat) colmax[gtid] = 0ull;
  grid.sync();

  const int npairs = (n + 1) / 2, rounds = 2 * npairs - 1;
  const int lane = threadIdx.x & 31;
  // consecutive tasks go to different blocks (SMs), spreading the FP64 work
  const int gw = (int)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int nw = gthreads >> 5;
  const int ntasks = nmat * npairs;
  // largest squared column norm of every matrix (non-negative doubles order like their
  // bit patterns, so an integer maximum is exact and independent of the order)
  for (int task = gw; task < nmat * n; task += nw) {
    const double x = lane < n ? __ldcg(W + task * n + lane) : 0.0;
    const double a = warp_sum(x * x);
    if (lane == 0 && a > 0.0) atomicMax(colmax + task / n, (unsigned long long)__double_as_longlong(a));
  }
  grid.sync();
  // the computed inner product carries rounding of order n eps sqrt(a b): a tolerance below that
  // level would keep rotating rounding noise forever.  A pair is rotated only if |g| > tol
  // max(a, b), not tol sqrt(a b): the rotation it would apply to V is g / (a - b), below tol either
  // way, but a column at rounding level carries noise of order eps times the large column it was
  // last rotated against, and the relative test would rotate that pair forever.  Columns with a
  // squared norm below 1e-280 are left alone: tol max(a, b) underflows to 0 there.
  int sweep = 1;
  unsigned settled = 0u;   // matrices that have had their last sweep
  bool converged = false;
  for (; sweep <= max_sweeps; ++sweep) {
    int *cur = counters + (sweep % 3) * nmat, *prev = counters + ((sweep + 2) % 3) * nmat;
    if (blockIdx.x == 0 && (int)threadIdx.x < nmat) counters[((sweep + 1) % 3) * nmat + threadIdx.x] = 0;
    for (int r = 0; r < rounds; ++r) {
      for (int task = gw; task < ntasks; task += nw) {
        // a matrix takes the turns of its own order, and none after its last sweep, whatever its batch
        const int mat = task / npairs, k = task % npairs, nm = na.n[mat], mp = nm + (nm & 1);
        if (k >= mp / 2 || r >= mp - 1 || (sweep > 1 && __ldcg(prev + mat) == 0)) continue;
        int p = rr_slot(k, r, mp), q = rr_slot(mp - 1 - k, r, mp);
        if (p >= nm || q >= nm) continue;
        if (p > q) { const int t = p; p = q; q = t; }
        const bool in = lane < n;
        const int ip = mat * nn + p * n + lane, iq = mat * nn + q * n + lane;
        // the V columns are loaded with the W columns (one L2 round trip), used if the pair rotates
        const double x = in ? __ldcg(W + ip) : 0.0, y = in ? __ldcg(W + iq) : 0.0;
        const double vx = in ? __ldcg(V + ip) : 0.0, vy = in ? __ldcg(V + iq) : 0.0;
        const double a = warp_sum(x * x), b = warp_sum(y * y), g = warp_sum(x * y);
        const double big = fmax(a, b);
        const double tol = 4.0 * (double)nm * kEps;
        if (!((g != 0.0) && big > 1e-280 && (fabs(g) > tol * big))) continue;
        const bool counts = big > tol * tol * __longlong_as_double((long long)__ldcg(colmax + mat));
        const double zeta = (b - a) / (2.0 * g);
        const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        const double c = 1.0 / sqrt(1.0 + t * t);
        const double s = c * t;
        if (in) {
          __stcg(W + ip, c * x - s * y);
          __stcg(W + iq, s * x + c * y);
          __stcg(V + ip, c * vx - s * vy);
          __stcg(V + iq, s * vx + c * vy);
        }
        if (lane == 0 && counts) atomicAdd(cur + mat, 1);
      }
      grid.sync();
    }
    int total = 0;
    for (int m = 0; m < nmat; ++m) {
      const int rotated = __ldcg(cur + m);
      if (gtid == 0 && !(settled >> m & 1u)) {
        sweeps_out[m] = sweep;
        if (rotated == 0) settled |= 1u << m;
      }
      total += rotated;
    }
    if (total == 0) {
      converged = true;
      break;
    }
  }
  for (int task = gw; task < nmat * n; task += nw) {
    const double x = lane < n ? __ldcg(W + task * n + lane) : 0.0;
    const double a = warp_sum(x * x);
    if (lane == 0) lam[task] = sqrt(a);
  }
  if (gtid == 0 && !converged && st->status == 0) st->status = HOTRG_ENOTCONV;
}

// ---------------------------------------------------------------------------
// The graded part.  Backward error of a few eps ||A|| turns vectors with eigenvalues lambda, mu by eps
// lambda_1 / |lambda - mu|, far more than A's elements leave open where lambda and mu are small.  So
// W = A V is formed and its columns are made orthogonal to 4 n eps (one-sided Jacobi's test): groups
// of close eigenvalues by plane rotations, the others, whose angles are small, all at once by 1 + M + M^2 / 2 +
// M^3 / 8 (M skew, its elements the angles: orthogonal to M^6 / 64), as far as the angles need it.  A kept
// vector's angles against those far below it reach 8 eps lambda_1 / lambda, 2^-9 for the least lambda that the
// selection tells from its neighbours, 1e-12 lambda_1; a pass leaves their products, so there are three.
// ---------------------------------------------------------------------------
// Vectors of opposite classes are left as they are (turn_forbidden); what else ends a class is noted in
// `lost` by the polish alone, whose turns are ordered by barriers, and applied by the last pass.

// EIG_AV: out[0] = X Y[0] / unscale.  With the angles as X, for V (0) and W (1): EIG_FIRST: out = Y + X Y where the
// matrix has any; EIG_SECOND: out = Z + X (Z - Y) / 2 with Z = Y + X Y where one is above 2^-24; EIG_THIRD: the same
// with 1 / 4, Z of second and Y of first order, where one is above 2^-12.  32 x 32 tiles, 2 x 2 per thread.
enum EigProduct { EIG_AV, EIG_FIRST, EIG_SECOND, EIG_THIRD };
struct EigPair {
  double* p[2];
};
template <EigProduct KIND>
__global__ void __launch_bounds__(256) eig_nn_kernel(const double* __restrict__ X, EigPair Yp, EigPair Zp, EigWs ws,
                                                     EigPair outp) {
  constexpr int BK = 16;
  __shared__ double As[BK][33], Bs[BK][33];
  const int mat = KIND == EIG_AV ? blockIdx.z : blockIdx.z >> 1, which = KIND == EIG_AV ? 0 : blockIdx.z & 1;
  const int n = ws.na[mat], ld = ws.n, c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  if (c0 >= n || r0 >= n) return;
  const EigCtl ctl = ws.ctl[mat];
  if (ctl.bad || (KIND != EIG_AV && ctl.mixed < (int)KIND)) return;
  const double* __restrict__ Y = Yp.p[which];
  const double* __restrict__ Z = KIND >= EIG_SECOND ? Zp.p[which] : nullptr;
  double* __restrict__ out = outp.p[which];
  const long long o = (long long)mat * ld * ld;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int k0 = 0; k0 < n; k0 += BK) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = r0 + (tid >> 4) + 16 * u, k = k0 + (tid & 15);
      As[tid & 15][(tid >> 4) + 16 * u] = (r < n && k < n) ? X[o + (long long)r * ld + k] : 0.0;
      const int kb = k0 + (tid >> 5) + 8 * u, c = c0 + (tid & 31);
      const long long eb = o + (long long)kb * ld + c;
      Bs[(tid >> 5) + 8 * u][tid & 31] = (kb < n && c < n) ? (KIND >= EIG_SECOND ? Z[eb] - Y[eb] : Y[eb]) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const double a0 = As[k][ty], a1 = As[k][ty + 16], b0 = Bs[k][tx], b1 = Bs[k][tx + 16];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
  const double sc = KIND == EIG_AV ? 1.0 / ctl.unscale : 1.0;   // a power of two
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = r0 + ty + 16 * u, c = c0 + tx + 16 * v;
      if (r < n && c < n) {
        const long long e = o + (long long)r * ld + c;
        out[e] = KIND == EIG_AV ? acc[u][v] * sc : KIND == EIG_FIRST ? Y[e] + acc[u][v]
                                                                          : fma(KIND == EIG_SECOND ? 0.5 : 0.25, acc[u][v], Z[e]);
      }
    }
}

// squared norms of W's columns (into dk); LAST: the eigenvalues, and no class where the polish ended it
template <bool LAST>
__global__ void __launch_bounds__(256) eig_norm_kernel(const double* __restrict__ W, EigWs ws, double* lam, int pass) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const EigCtl ctl = ws.ctl[mat];
  if (c == 0 && lane == 0 && !LAST) {
    if (pass > 0 && ctl.mixed < 2) ws.ctl[mat].settled = 1;
    ws.ctl[mat].mixed = 0;
  }
  if (c >= n || ctl.bad) return;
  const double* w = W + (long long)mat * ld * ld + (long long)c * ld;
  double a = 0.0;
  for (int i = lane; i < n; i += 32) a = fma(w[i], w[i], a);
  a = warp_sum(a);
  if (lane == 0) {
    if (LAST) {
      lam[mat * ld + c] = sqrt(a) * ctl.unscale;
      if (ws.lost[mat * ld + c]) ws.cls[mat * ld + c] = 0;
    } else {
      ws.dk[mat * ld + c] = a;
    }
  }
}

// Angles: the Gram matrix of W's columns (upper 32 x 32 tiles), and for every pair that is not
// orthogonal to 4 n eps of its norms the tangent t of its plane rotation, w_p -= t w_q, w_q += t w_p, in M.  (Of
// the larger norm, as in the sweeps, would leave what two small columns have of a large one, and the product of
// the two would pass for an angle between them: 3e-11 of a vector at 6e-12 lambda_1.)
// Angles above 2^-9 are left: between kept vectors, or across the cut, the groups have taken them.  So are the
// vectors below 1e-12 lambda_1, which are rounding: their angles would come back to the others.
__global__ void __launch_bounds__(256) eig_gram_kernel(const double* __restrict__ W, EigWs ws, double* __restrict__ M) {
  constexpr int BK = 16;
  __shared__ double As[BK][33], Bs[BK][33];
  const int mat = blockIdx.z, n = ws.na[mat], ld = ws.n, q0 = blockIdx.x * 32, p0 = blockIdx.y * 32;
  if (q0 >= n || p0 > q0 || ws.ctl[mat].bad || ws.ctl[mat].settled) return;
  const long long o = (long long)mat * ld * ld;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int k0 = 0; k0 < n; k0 += BK) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = (tid >> 4) + 16 * u, k = k0 + (tid & 15);
      As[tid & 15][r] = (p0 + r < n && k < n) ? W[o + (long long)(p0 + r) * ld + k] : 0.0;
      Bs[tid & 15][r] = (q0 + r < n && k < n) ? W[o + (long long)(q0 + r) * ld + k] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const double a0 = As[k][ty], a1 = As[k][ty + 16], b0 = Bs[k][tx], b1 = Bs[k][tx + 16];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
  const double* nrm = ws.dk + mat * ld;
  const double tol = 4.0 * n * kEps;
  const int first = n - ws.keep[mat];   // pairs of two vectors behind the kept ones stay
  const double line = 1e-24 * nrm[n - 1];
  const int *cls = ws.cls + mat * ld, *lost = ws.lost + mat * ld;
  int any = 0;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int p = p0 + ty + 16 * u, q = q0 + tx + 16 * v;
      if (p >= n || q >= n || p > q) continue;
      double t = 0.0;
      if (p < q) {
        const double a = nrm[p], b = nrm[q], g = acc[u][v], big = fmax(a, b);
        if (q >= first && big > line && fabs(g) > tol * sqrt(a) * sqrt(b) &&
            !turn_forbidden(cls[p], lost[p] != 0, cls[q], lost[q] != 0)) {
          const double zeta = (b - a) / (2.0 * g);
          t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
          if (fabs(t) > 0.001953125) t = 0.0;
          if (t != 0.0) any = max(any, fabs(t) > 0.000244140625 ? 3 : fabs(t) > 5.9604644775390625e-8 ? 2 : 1);
        }
      }
      M[o + (long long)p * ld + q] = -t;
      M[o + (long long)q * ld + p] = t;
    }
  if (any) atomicMax(&ws.ctl[mat].mixed, any);
}

// V and W take the turned columns, of the highest order that was formed
__global__ void __launch_bounds__(256) eig_take_kernel(EigWs ws, EigPair first, EigPair second, EigPair third, EigPair to,
                                                       int most) {
  const int mat = blockIdx.y, n = ws.na[mat], ld = ws.n;
  const EigCtl ctl = ws.ctl[mat];
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n || ctl.bad || !ctl.mixed) return;
  const long long o = (long long)mat * ld * ld + (long long)c * ld;
  const int order = min(ctl.mixed, most);
  const double* v = order > 2 ? third.p[0] : order > 1 ? second.p[0] : first.p[0];
  const double* w = order > 2 ? third.p[1] : order > 1 ? second.p[1] : first.p[1];
  for (int i = lane; i < n; i += 32) {
    to.p[0][o + i] = v[o + i];
    to.p[1][o + i] = w[o + i];
  }
}

// Groups of neighbouring eigenvalues, 2e-8 lambda_1 apart at most, above 4 n eps lambda_1 and not wholly
// behind the kept ones: their columns of W are orthogonalised by one-sided Jacobi sweeps.  One CTA per
// matrix; without a group it reads the eigenvalues and ends.  At most kPolish columns of a group are
// taken, those with the largest eigenvalues.
__global__ void __launch_bounds__(256) eig_polish_kernel(EigWs ws, double* V, double* W, const double* __restrict__ lam) {
  __shared__ double l[kEigMaxN];
  __shared__ int s_rot;
  const int mat = blockIdx.x, n = ws.na[mat], ld = ws.n;
  if (ws.ctl[mat].bad || n < 2) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const long long nn = (long long)ld * ld;
  for (int i = threadIdx.x; i < n; i += blockDim.x) l[i] = lam[mat * ld + i];   // ascending
  __syncthreads();
  const double top = fmax(fabs(l[0]), fabs(l[n - 1])), thr = 2e-8 * top, floor_ = 4.0 * n * kEps * top;
  const double tol = 4.0 * n * kEps;
  double* Vm = V + mat * nn;
  double* Wm = W + mat * nn;
  const int first = n - ws.keep[mat];
  for (int hi = n; hi > 1 && hi > first && l[hi - 1] > floor_;) {
    int lo = hi - 1;
    // behind the kept ones only as far as the last of them reaches
    while (lo > 0 && l[max(lo, first)] - l[lo - 1] <= thr && l[lo - 1] > floor_ && hi - lo < kPolish) --lo;
    const int m = hi - lo;
    if (m < 2) {
      --hi;
      continue;
    }
    const int mp = m + (m & 1);
    const int* cls = ws.cls + mat * ld + lo;
    volatile int* lost = ws.lost + mat * ld + lo;
    for (int sweep = 0; sweep < 30; ++sweep) {
      __syncthreads();
      if (threadIdx.x == 0) s_rot = 0;
      __syncthreads();
      for (int r = 0; r < mp - 1; ++r) {
        for (int k = warp; k < mp / 2; k += nw) {
          const int p = rr_slot(k, r, mp), q = rr_slot(mp - 1 - k, r, mp);
          if (p >= m || q >= m) continue;
          // the pairs of a round are disjoint, and a barrier ends the round
          const int cp = cls[p], cq = cls[q];
          const bool lp = lost[p] != 0, lq = lost[q] != 0;
          if (turn_forbidden(cp, lp, cq, lq)) continue;
          double *wp = Wm + (long long)(lo + p) * ld, *wq = Wm + (long long)(lo + q) * ld;
          double a = 0.0, b = 0.0, g = 0.0;
          for (int i = lane; i < n; i += 32) {
            a = fma(wp[i], wp[i], a);
            b = fma(wq[i], wq[i], b);
            g = fma(wp[i], wq[i], g);
          }
          a = warp_sum(a);
          b = warp_sum(b);
          g = warp_sum(g);
          const double big = fmax(a, b);
          if (!(g != 0.0 && big > 1e-280 && fabs(g) > tol * big)) continue;
          const double zeta = (b - a) / (2.0 * g);
          const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
          const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
          double *vp = Vm + (long long)(lo + p) * ld, *vq = Vm + (long long)(lo + q) * ld;
          for (int i = lane; i < n; i += 32) {
            const double x = wp[i], y = wq[i], vx = vp[i], vy = vq[i];
            wp[i] = c * x - s * y;
            wq[i] = s * x + c * y;
            vp[i] = c * vx - s * vy;
            vq[i] = s * vx + c * vy;
          }
          if (lane == 0) {
            s_rot = 1;
            if (turn_ends_class(cp, lp, cq, lq, t)) lost[p] = lost[q] = 1;
          }
          __syncwarp();
        }
        __syncthreads();
      }
      const int rot = s_rot;
      if (!rot) break;
    }
    hi = lo;
  }
}

__global__ void eig_iters_kernel(EigWs ws, int* out) {
  if ((int)threadIdx.x < ws.nmat) out[threadIdx.x] = ws.ctl[threadIdx.x].iters + 1;
}

namespace {
struct EigLayout {
  size_t bytes = 0;
  size_t take(size_t b) {
    const size_t o = bytes;
    bytes += (b + 255) & ~size_t(255);
    return o;
  }
};

int eig_leaves(int n) {
  int l = 1;
  while ((n + l - 1) / l > kLeaf) l *= 2;
  return l;
}

// lays the workspace out from `base` (null: sizes only)
size_t eig_layout(char* base, int n, int nmat, EigWs* w, int** pos) {
  EigLayout L;
  const size_t nn = (size_t)n * n * nmat, nv = (size_t)n * nmat;
  auto dbl = [&](size_t c) { return (double*)(base + L.take(sizeof(double) * c)); };
  auto i32 = [&](size_t c) { return (int*)(base + L.take(sizeof(int) * c)); };
  w->n = n;
  w->nmat = nmat;
  w->vh = dbl(nn);
  w->q0 = dbl(nn);
  w->q1 = dbl(nn);
  w->ap = dbl(nn);
  w->w2 = dbl(nn);
  w->w3 = dbl(nn);
  w->s = dbl((size_t)(n + 16) * n * nmat);   // also the rows of a reduction that exceeds shared memory
  w->tf = dbl((size_t)((n + kRb - 1) / kRb) * kRb * kRb * nmat);
  for (double** p : {&w->d, &w->e, &w->tau, &w->ev0, &w->ev1, &w->dk, &w->zk, &w->zh, &w->val, &w->rc, &w->rs})
    *p = dbl(nv);
  for (int** p : {&w->perm, &w->comp, &w->sgn, &w->okc, &w->sym, &w->lost, &w->icl, &w->idx, &w->defl, &w->rp, &w->rq, &w->top, &w->bot, pos}) *p = i32(nv);
  w->ctl = (EigCtl*)(base + L.take(sizeof(EigCtl) * nmat));
  w->mc = (MergeCtl*)(base + L.take(sizeof(MergeCtl) * nmat * eig_leaves(n)));
  return L.bytes;
}

// CTAs per matrix of the reduction, and whether its rows fit in shared memory
int tri_cluster(int n) { return n <= 32 ? 1 : n <= 48 ? 2 : n <= 96 ? 4 : n <= 192 ? 8 : 16; }
size_t tri_smem(int n, int c, bool rows) {
  const size_t nrow = (n + c - 1) / c;
  return sizeof(double) * (5 * (size_t)n + (rows ? nrow * n : 0));
}

template <int EPT>
int launch_tridiag_t(const EigWs& w, cudaStream_t s) {
  const int n = w.n;
  if (cudaFuncSetAttribute(eig_tridiag_kernel<EPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) !=
          cudaSuccess ||
      cudaFuncSetAttribute(eig_tridiag_kernel<EPT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return -1;
  for (int c = tri_cluster(n);; c = 8) {
    const bool fits = tri_smem(n, c, true) <= 220 * 1024;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c * w.nmat);
    cfg.blockDim = dim3(kTriThreads);
    cfg.dynamicSmemBytes = tri_smem(n, c, fits);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (c > 8) {   // sixteen CTAs are not portable: eight if the device cannot place them
      int active = 0;
      if (cudaOccupancyMaxActiveClusters(&active, eig_tridiag_kernel<EPT>, &cfg) != cudaSuccess || active < 1) {
        cudaGetLastError();
        continue;
      }
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, eig_tridiag_kernel<EPT>, w, fits ? 1 : 0, w.s);
    ++g_launches;
    return e == cudaSuccess ? 0 : -1;
  }
}

int launch_tridiag(const EigWs& w, cudaStream_t s) {
  if (w.n <= kVecThreads) return launch_tridiag_t<1>(w, s);
  if (w.n <= 2 * kVecThreads) return launch_tridiag_t<2>(w, s);
  if (w.n <= 3 * kVecThreads) return launch_tridiag_t<3>(w, s);
  if (w.n <= 5 * kVecThreads) return launch_tridiag_t<5>(w, s);
  return launch_tridiag_t<8>(w, s);
}
}  // namespace

size_t eig_workspace_bytes(int n, int nmat) {
  EigWs w;
  int* pos;
  return eig_layout(nullptr, n, nmat, &w, &pos);
}

// V (rows: eigenvectors) and lam of nmat symmetric matrices of orders na[] <= n, with leading
// dimension n; A is overwritten; keep[]: the leading eigenvectors that may be kept; swp [nmat][n]: the partner of every index under the exchange of hat and check;
// iters: one word per matrix
int launch_eig(double* A, int n, int nmat, const int* na, const int* keep, const int* swp, void* work, double* V,
               double* lam, int* cls, int* iters, DevState* st, cudaStream_t s) {
  if (n < 1 || n > kEigMaxN || nmat < 1 || nmat > kEigMaxMat) return -1;
  EigWs w;
  for (int m = 0; m < kEigMaxMat; ++m) {
    w.na[m] = m < nmat ? na[m] : 0;
    w.keep[m] = m < nmat ? std::min(keep[m], na[m]) : 0;
    if (m < nmat && (na[m] < 1 || na[m] > n)) return -1;
  }
  int* pos;
  eig_layout((char*)work, n, nmat, &w, &pos);
  w.cls = cls;
  if (cudaMemsetAsync(cls, 0, sizeof(int) * n * nmat, s) != cudaSuccess) return -1;
  if (n <= kJacobiMax) {
    // rows beyond a matrix's order are zero: their columns are never rotated
    int npairs = (n + 1) / 2, max_sweeps = 60;
    double* W = w.vh;
    int* counters = (int*)w.ctl;
    unsigned long long* colmax = (unsigned long long*)w.mc;
    const int blocks = std::max(1, std::min(nmat * npairs, sm_count()));
    JacobiOrders orders;
    for (int m = 0; m < kEigMaxMat; ++m) orders.n[m] = w.na[m];
    void* args[] = {&A, &W, &V, &lam, &n, &orders, &nmat, &max_sweeps, &counters, &colmax, &iters, &st};
    const cudaError_t e =
        cudaLaunchCooperativeKernel((void*)jacobi_onesided_kernel, dim3(blocks), dim3(256), args, 0, s);
    ++g_launches;
    return e == cudaSuccess ? 0 : -1;
  }
  w.swp = swp;
  if (cudaMemsetAsync(w.ctl, 0, sizeof(EigCtl) * nmat, s) != cudaSuccess ||
      cudaMemsetAsync(w.lost, 0, sizeof(int) * n * nmat, s) != cudaSuccess)
    return -1;
  const dim3 rows((n + 7) / 8, nmat);
  double* m = w.q0;   // A scaled: the vectors' buffer is not needed yet
  eig_check_kernel<<<rows, 256, 0, s>>>(A, w);
  eig_scale_kernel<<<rows, 256, 0, s>>>(A, w);
  eig_label_kernel<<<rows, 256, 0, s>>>(m, w);
  eig_mixed_kernel<<<rows, 256, 0, s>>>(m, w);
  eig_order_kernel<true><<<nmat, 1024, 0, s>>>(m, w);
  eig_verify_kernel<<<rows, 256, 0, s>>>(m, w);
  eig_basis_kernel<<<rows, 256, 0, s>>>(m, w);
  eig_label_kernel<<<rows, 256, 0, s>>>(w.ap, w);
  eig_mixed_kernel<<<rows, 256, 0, s>>>(w.ap, w);
  eig_order_kernel<false><<<nmat, 1024, 0, s>>>(w.ap, w);
  g_launches += 10;
  const size_t qbytes = (size_t)((char*)w.ap - (char*)w.q0);
  if (cudaMemsetAsync(w.q0, 0, qbytes, s) != cudaSuccess) return -1;   // blocks between nodes read as zero
  if (launch_tridiag(w, s) != 0) return -1;
  const int leaves = eig_leaves(n);
  eig_leaf_kernel<<<nmat * leaves, 32, 0, s>>>(w, leaves, w.ev0, w.q0, st);
  ++g_launches;
  double *q = w.q0, *qn = w.q1, *ev = w.ev0, *evn = w.ev1;
  for (int nodes = leaves / 2; nodes >= 1; nodes /= 2) {
    const int m = n / nodes + 1, g = nmat * nodes;
    const int mm = m < n ? m : n;
    eig_prep_kernel<<<g, 256, 0, s>>>(w, nodes, ev, q);
    eig_roots_kernel<<<dim3((mm + 1) / 2, g), 64, 0, s>>>(w, nodes);
    eig_weights_kernel<<<dim3((mm + 31) / 32, g), 256, 0, s>>>(w, nodes);
    eig_vectors_kernel<<<dim3((mm + 7) / 8, g), 256, 0, s>>>(w, nodes, evn, pos);
    eig_rotate_kernel<<<dim3((mm + 63) / 64, g), 64, 0, s>>>(w, nodes, q);
    const int half = mm / 2 + 1;
    eig_product_kernel<<<dim3(2 * ((half + 31) / 32), (mm + 31) / 32, g), 256, 0, s>>>(w, nodes, q, qn, pos);
    g_launches += 6;
    double* t = q;
    q = qn;
    qn = t;
    t = ev;
    ev = evn;
    evn = t;
  }
  const int nblk = n > 2 ? (n - 2 + kRb - 1) / kRb : 0;
  const size_t smem = sizeof(double) * ((size_t)(kStrip + kRb) * (n + 1) + 3 * kRb * kStrip);
  if (cudaFuncSetAttribute(eig_back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess)
    return -1;
  if (nblk > 0) {
    eig_tfactor_kernel<<<dim3(nblk, nmat), 256, 0, s>>>(w, w.tf);
    ++g_launches;
  }
  eig_back_kernel<<<dim3((n + kStrip - 1) / kStrip, nmat), 256, smem, s>>>(w, q, ev, w.tf, nblk, V, lam);
  ++g_launches;
  // W = A V, the close groups, then the small angles
  const int tn = (n + 31) / 32;
  const dim3 tiles(tn, tn, nmat), both(tn, tn, 2 * nmat);
  double *W = w.q0, *M = w.s;   // free by now, as the buffers of the turned columns are
  const EigPair cur = {{V, W}}, one = {{w.q1, w.ap}}, two = {{w.vh, w.w2}}, three = {{A, w.w3}}, none = {{nullptr, nullptr}};
  eig_nn_kernel<EIG_AV><<<tiles, 256, 0, s>>>(V, EigPair{{A, nullptr}}, none, w, EigPair{{W, nullptr}});
  eig_polish_kernel<<<nmat, 256, 0, s>>>(w, V, W, lam);
  for (int pass = 0; pass < 3; ++pass) {
    eig_norm_kernel<false><<<rows, 256, 0, s>>>(W, w, lam, pass);
    eig_gram_kernel<<<tiles, 256, 0, s>>>(W, w, M);
    eig_nn_kernel<EIG_FIRST><<<both, 256, 0, s>>>(M, cur, none, w, one);
    // the second pass has angles up to 2^-18, the third up to 2^-36
    if (pass < 2) eig_nn_kernel<EIG_SECOND><<<both, 256, 0, s>>>(M, cur, one, w, two);
    if (pass < 1) eig_nn_kernel<EIG_THIRD><<<both, 256, 0, s>>>(M, one, two, w, three);
    eig_take_kernel<<<rows, 256, 0, s>>>(w, one, two, three, cur, 3 - pass);
  }
  eig_norm_kernel<true><<<rows, 256, 0, s>>>(W, w, lam, 0);
  g_launches += 18;
  eig_iters_kernel<<<1, 32, 0, s>>>(w, iters);
  ++g_launches;
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// Choice, truncation and sign gauge for one transverse leg.
// Matrices 0 (A^(j)) and 1 (A'^(j)) of V and lam are used.
// Orders the eigenpairs by lambda = |eigenvalue| descending; values within 1e-12 lambda_1 of
// their predecessor form a tie group ordered by pivot index (the lowest row whose magnitude is
// within 1e-6 of the column maximum).  epsilon = sum of the eigenvalues after the first nnew;
// U^(j) is taken if epsilon < epsilon' - 1e-10 max(lambda_1, lambda'_1), else U'^(j); each kept
// column is flipped so that its pivot entry is positive.
// Three launches: pivots (a warp per eigenvector), order and choice (one CTA, every rank by
// counting: a tie group of the near-null space has hundreds of members), U (a thread per entry).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) select_pivot_kernel(const double* __restrict__ V, int n, int* piv, int* sgn) {
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;   // column of either side
  if (c >= 2 * n) return;
  const double* v = V + (long long)c * n;   // the two matrices are contiguous
  double vmax = 0.0;
  for (int k = lane; k < n; k += 32) vmax = fmax(vmax, fabs(v[k]));
  for (int o = 16; o > 0; o >>= 1) vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
  int first = n;
  for (int k0 = 0; k0 < n && first == n; k0 += 32) {
    const int k = k0 + lane;
    const bool hit = k < n && fabs(v[k]) >= (1.0 - 1e-6) * vmax;
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    if (m) first = k0 + __ffs(m) - 1;
  }
  if (first >= n) first = 0;   // no entry found (a NaN column): stay in range; the trace reports it
  if (lane == 0) {
    piv[c] = first;
    sgn[c] = v[first] < 0.0 ? -1 : 1;
  }
}

__global__ void __launch_bounds__(1024) select_kernel(const double* __restrict__ lam_in, const int* __restrict__ piv,
                                                      int n, int nnew, double* lam_sorted, int* order_out,
                                                      LegResult* res, const int* sweeps, const int* __restrict__ cls,
                                                      int* rank_out, int* cls_out) {
  extern __shared__ double sm[];
  double* lam = sm;                  // [2][n] by eigenvector, -1 for a NaN
  double* srt = lam + 2 * n;         // [2][n] descending
  int* order = (int*)(srt + 2 * n);  // [2][n]
  int* grp = order + 2 * n;          // [2][n] first place of the tie group
  int* fin = grp + 2 * n;            // [2][n]
  __shared__ double s_eps[2], s_part[2][32];
  __shared__ int s_choice;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < 2 * n; e += blockDim.x) {
    const double x = fabs(lam_in[e]);
    lam[e] = isnan(x) ? -1.0 : x;   // a NaN ranks below every number, so that the ranks stay a permutation
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 2 * n; e += blockDim.x) {
    const int side = e >= n ? 1 : 0, i = e - side * n;
    const double* l = lam + side * n;
    const double li = l[i];
    int rank = 0;
    for (int k = 0; k < n; ++k) rank += (l[k] > li) || (l[k] == li && k < i);
    order[side * n + rank] = i;
    srt[side * n + rank] = li;
  }
  __syncthreads();
  // tie groups: a place starts one if it lies more than tol below its predecessor; the group of
  // a place is the last start at or before it (warp 0 and 1 walk a side, 32 places at a time)
  if (warp < 2) {
    const double* l = srt + warp * n;
    const double tol = 1e-12 * l[0];
    int cur = 0;
    for (int r0 = 0; r0 < n; r0 += 32) {
      const int r = r0 + lane;
      const bool brk = r < n && r > 0 && l[r - 1] - l[r] > tol;
      const unsigned m = __ballot_sync(0xffffffffu, brk);
      const unsigned below = m & (0xffffffffu >> (31 - lane));
      if (r < n) grp[warp * n + r] = below ? r0 + 31 - __clz(below) : cur;
      if (m) cur = r0 + 31 - __clz(m);
    }
  }
  __syncthreads();
  // place within the group: by pivot, then by the order before (stable)
  for (int e = threadIdx.x; e < 2 * n; e += blockDim.x) {
    const int side = e >= n ? 1 : 0, r = e - side * n;
    const int *ord = order + side * n, *g = grp + side * n, *pv = piv + side * n;
    const int g0 = g[r], mine = pv[ord[r]];
    int place = g0;
    for (int k = g0; k < n && g[k] == g0; ++k) {
      const int o = pv[ord[k]];
      place += o < mine || (o == mine && k < r);
    }
    fin[side * n + place] = ord[r];
  }
  __syncthreads();
  for (int side = 0; side < 2; ++side) {
    double a = 0.0;
    for (int r = nnew + threadIdx.x; r < n; r += blockDim.x) {
      const double x = lam_in[side * n + fin[side * n + r]];
      a += fabs(x);
    }
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) s_part[side][warp] = a;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double a = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += s_part[threadIdx.x][w];
    s_eps[threadIdx.x] = a;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double l1a = fabs(lam_in[fin[0]]), l1b = fabs(lam_in[n + fin[n]]);
    const double tol = 1e-10 * fmax(l1a, l1b);
    const int prime = !(s_eps[0] < s_eps[1] - tol) ? 1 : 0;
    s_choice = prime;
    const double* lc = lam_in + prime * n;
    const int* oc = fin + prime * n;
    res->eps[0] = s_eps[0];
    res->eps[1] = s_eps[1];
    res->lam1[0] = l1a;
    res->lam1[1] = l1b;
    res->chose_prime = prime;
    res->sweeps[0] = sweeps ? sweeps[0] : 0;
    res->sweeps[1] = sweeps ? sweeps[1] : 0;
    const double top = fabs(lc[oc[0]]);
    res->gap = (nnew < n && top > 0.0) ? (fabs(lc[oc[nnew - 1]]) - fabs(lc[oc[nnew]])) / top : 1e300;
  }
  __syncthreads();
  const int side = s_choice;
  for (int e = threadIdx.x; e < 2 * n; e += blockDim.x) lam_sorted[e] = fabs(lam_in[(e >= n ? n : 0) + fin[e]]);
  for (int r = threadIdx.x; r < nnew; r += blockDim.x) order_out[r] = side * n + fin[side * n + r];
  if (rank_out)   // rank of every eigenvector of the chosen side in the sorted order, and its class by rank
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
      rank_out[fin[side * n + r]] = r;
      cls_out[r] = cls[side * n + fin[side * n + r]];
    }
}

// U = the kept eigenvectors in order, sign-fixed (order: row of the two stacked matrices)
__global__ void __launch_bounds__(256) select_u_kernel(const double* __restrict__ V, const int* __restrict__ order,
                                                       const int* __restrict__ sgn, int n, int nnew, double* U64,
                                                       float* U32) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * nnew) return;
  const int row = e / nnew, col = e - row * nnew;
  const int src = order[col];
  const double v = V[(long long)src * n + row] * (double)sgn[src];
  U64[e] = v;
  U32[e] = (float)v;
}

// scratch: 5 n words
void launch_select(const double* lam, const double* V, int n, int nnew, double* lam_sorted, double* U64, float* U32,
                   LegResult* res, const int* sweeps, int* scratch, cudaStream_t s, const int* cls, int* rank_out,
                   int* cls_out) {
  const size_t smem = (size_t)4 * n * sizeof(double) + (size_t)6 * n * sizeof(int);
  if (smem > 47 * 1024) raise_smem_limit(select_kernel, 56 * kEigMaxN);
  int *piv = scratch, *sgn = scratch + 2 * n, *order = scratch + 4 * n;
  select_pivot_kernel<<<(2 * n + 7) / 8, 256, 0, s>>>(V, n, piv, sgn);
  select_kernel<<<1, 1024, smem, s>>>(lam, piv, n, nnew, lam_sorted, order, res, sweeps, cls, rank_out, cls_out);
  select_u_kernel<<<(n * nnew + 255) / 256, 256, 0, s>>>(V, order, sgn, n, nnew, U64, U32);
  g_launches += 3;
}

}  // namespace hotrg
