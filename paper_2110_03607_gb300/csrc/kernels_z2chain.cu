// The two large stages of the tensor-times-isometry chains in the Z2 block form (d >= 3): the last
// prime stage, which writes the blocks of the bottleneck's B operand, and the first non-prime stage,
// which reads the blocks of its product C.
//
// U~ is nonzero only where par(hat) ^ par(check) = par(new), and an output is wanted (prime), or is not
// identically zero (non-prime), for the new indices of one parity only.  So with the check and new
// indices sorted by parity, an output vector needs half the terms of half the columns, a quarter of the
// multiply-adds and half of the loads of the dense stage.  The terms that remain are summed in the order
// of the dense stage, and those left out are exact zeros: the results are the same bit for bit.
//
// The prime stage is bound by instruction issue (splitting into pieces and storing them is half of it)
// and close to the rate at which HBM takes its output; the non-prime stage by its shared-memory reads of
// U~ (one 16-byte read for 4 multiply-adds) and the reads of C.
#include "hotrg_internal.cuh"

namespace hotrg {

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// two FP32 multiply-adds (adds) in one instruction, each rounded as fmaf (as +)
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// acc[0 .. NH) += x * row[0 .. NH)
template <int NH>
__device__ __forceinline__ void fma_row2(float x, const float* row, u64 (&acc)[NH / 2]) {
  const u64 xx = pack2(x, x);
#pragma unroll
  for (int n = 0; n < NH; n += 4) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(row + n);
    acc[n / 2] = fma2(xx, u.x, acc[n / 2]);
    acc[n / 2 + 1] = fma2(xx, u.y, acc[n / 2 + 1]);
  }
}

struct Lists {
  int b[2][32];   // check indices of each parity, ascending
  int n[2][32];   // new indices of each parity
};

// U~ rows in shared memory: of hat a, the check indices sorted by parity (ascending within one), each
// with the columns n of parity par(a) ^ par(b), padded with zeros to NH.  Four words between the hats
// put the rows of neighbouring hats on other banks.
template <int NH>
__device__ __forceinline__ int hat_pitch(int chi) {
  return chi * NH + 4;
}
template <int NH>
__device__ void load_u(const Z2Chain& p, float* us, Lists* l) {
  if (threadIdx.x < 64) {   // the lists, by rank among the indices of the same parity
    const int i = threadIdx.x & 31;
    const bool of_n = threadIdx.x >= 32;
    const unsigned mask = of_n ? p.mask_n : p.mask_b;
    if (i < (of_n ? p.nn : p.chi)) {
      const int par = (mask >> i) & 1;
      const int rank = __popc((par ? mask : ~mask) & ((1u << i) - 1u));
      if (of_n) l->n[par][rank] = i;
      else l->b[par][rank] = i;
    }
  }
  __syncthreads();
  const int nb0 = p.chi - __popc(p.mask_b);
  const int nn1 = __popc(p.mask_n), nn0 = p.nn - nn1;
  for (int e = threadIdx.x; e < p.chi * p.chi * NH; e += blockDim.x) {
    const int i = e % NH, r = (e / NH) % p.chi, a = e / (NH * p.chi);
    const int pb = r >= nb0 ? 1 : 0;
    const int b = l->b[pb][pb ? r - nb0 : r];
    const int pn = (int)((p.mask_b >> a) & 1) ^ pb;
    us[a * hat_pitch<NH>(p.chi) + r * NH + i] =
        i < (pn ? nn1 : nn0) ? p.U[(long long)(a + b * p.chi) * p.ldu + l->n[pn][i]] : 0.0f;
  }
  __syncthreads();
}

template <int PF>
__device__ __forceinline__ void store_pair(char* o, long long pbytes, int npieces, float v0, float v1) {
  if (PF == PIECE_TF32) {
    for (int q = 0; q < npieces; ++q) {
      const float w0 = round_tf32(v0), w1 = round_tf32(v1);
      *reinterpret_cast<float2*>(o) = make_float2(w0, w1);
      v0 -= w0;
      v1 -= w1;
      o += pbytes;
    }
  } else {
    for (int q = 0; q < npieces; ++q) {
      const __nv_bfloat162 w = __floats2bfloat162_rn(v0, v1);
      *reinterpret_cast<__nv_bfloat162*>(o) = w;
      v0 -= __low2float(w);
      v1 -= __high2float(w);
      o += pbytes;
    }
  }
}

}  // namespace

// Last prime stage.  Input (FP32, contiguous): [g1][rho][nc][b][h] with g1 = (c', the new indices so
// far), nc = all check indices, b = the check index summed here, h = the hat indices so far; output row
// (g1, n, nc), column k = (rho, h, a) at its position in the list of k's parity.
// A warp takes 64 positions of one block's K list, two neighbours a lane (so that pieces are stored in
// pairs), and goes through GPER row groups (g1, nc) with them: the positions are decoded once.
template <int PF, int NH>
__global__ void __launch_bounds__(256, NH <= 8 ? 3 : (NH <= 16 ? 2 : 1)) z2_prime_kernel(Z2Chain p, const float* __restrict__ in, int H, int chi_c, int P,
                                                       int groups, int gper, const int* __restrict__ kcat, int rb0,
                                                       int R, Z2Blocks zo) {
  extern __shared__ __align__(16) unsigned char smem_u[];
  __shared__ Lists l;
  float* us = reinterpret_cast<float*>(smem_u);
  load_u<NH>(p, us, &l);
  const int lane = threadIdx.x & 31;
  // class sizes (selects, not arrays: an indexed array would live in local memory)
  const int nb1 = __popc(p.mask_b), nb0 = p.chi - nb1, nc1 = __popc(p.mask_n), nc0 = p.nn - nc1;
  const int chunks0 = (rb0 + 63) / 64, chunks = chunks0 + (R - rb0 + 63) / 64;
  const int pn0 = (int)(p.mask_n & 1u);
  const long long tasks = (long long)chunks * ((groups + gper - 1) / gper);
  const int hp = hat_pitch<NH>(p.chi);
  constexpr int UB = NH <= 8 ? 8 : 4;
  for (long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); t < tasks; t += (long long)gridDim.x * 8) {
    const int chunk = (int)(t % chunks);
    const int g_lo = (int)(t / chunks) * gper, g_hi = min(groups, g_lo + gper);
    const int kb = chunk >= chunks0 ? 1 : 0;
    const int kpos = (kb ? chunk - chunks0 : chunk) * 64 + 2 * lane;
    const int cnt = kb ? R - rb0 : rb0;
    const bool ok0 = kpos < cnt, ok1 = kpos + 1 < cnt;
    // the two k of this lane: input offset and hat index
    int a0 = 0, a1 = 0;
    long long o0 = 0, o1 = 0;
    if (ok0) {
      const int k = kcat[(kb ? rb0 : 0) + kpos], rh = k / p.chi, rho = rh / H;
      a0 = k - rh * p.chi;
      o0 = (long long)rho * P * p.chi * H + (rh - rho * H);
      a1 = a0;
      o1 = o0;
    }
    if (ok1) {
      const int k = kcat[(kb ? rb0 : 0) + kpos + 1], rh = k / p.chi, rho = rh / H;
      a1 = k - rh * p.chi;
      o1 = (long long)rho * P * p.chi * H + (rh - rho * H);
    }
    const int pa0 = (int)(p.mask_b >> a0) & 1, pa1 = (int)(p.mask_b >> a1) & 1;
    const bool shared_a = __all_sync(0xffffffffu, a0 == a1);
    char* ob = (char*)(kb ? zo.blk[1] : zo.blk[0]) + (long long)kpos * (PF == PIECE_TF32 ? 4 : 2);
    const long long ldb = (kb ? zo.ld[1] : zo.ld[0]) * (PF == PIECE_TF32 ? 4 : 2);
    const long long psb = (kb ? zo.pstride[1] : zo.pstride[0]) * (PF == PIECE_TF32 ? 4 : 2);
    // a row group's parity and the positions of its rows (lane i: the i-th of either parity of the new
    // index) are read one group ahead
    const long long lr0 = lane < nc0 ? (long long)l.n[0][lane] * P : 0, lr1 = lane < nc1 ? (long long)l.n[1][lane] * P : 0;
    int g1 = g_lo / P, nc = g_lo - g1 * P;
    long long row0 = (long long)g1 * p.nn * P + nc;
    int blk_n = zo.cblk[row0], pos_n0 = zo.cpos[row0 + lr0], pos_n1 = zo.cpos[row0 + lr1];
    for (int g = g_lo; g < g_hi; ++g) {
      // the parity of new index that block kb takes from this row group
      const int sig = blk_n ^ pn0 ^ zo.q ^ kb;
      const int ncols = sig ? nc1 : nc0;
      const int pos = sig ? pos_n1 : pos_n0;
      const float* x = in + ((long long)g1 * chi_c * P + nc) * p.chi * H;
      if (++nc == P) {
        nc = 0;
        ++g1;
      }
      if (g + 1 < g_hi) {
        row0 = (long long)g1 * p.nn * P + nc;
        blk_n = zo.cblk[row0];
        pos_n0 = zo.cpos[row0 + lr0];
        pos_n1 = zo.cpos[row0 + lr1];
      }
      if (ncols == 0) continue;
      u64 acc0[NH / 2], acc1[NH / 2];
#pragma unroll
      for (int n = 0; n < NH / 2; ++n) acc0[n] = acc1[n] = 0ULL;
      if (shared_a) {
        const int pb = sig ^ pa0, m = pb ? nb1 : nb0;
        const float* row = us + a0 * hp + (pb ? nb0 : 0) * NH;
        const int* bl = l.b[pb];
        for (int i = 0; i < m; i += UB) {
          float x0[UB], x1[UB];
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const bool in_list = i + u < m;
            const long long ofs = in_list ? (long long)bl[i + u] * H : 0;
            x0[u] = in_list ? x[o0 + ofs] : 0.0f;
            x1[u] = in_list ? x[o1 + ofs] : 0.0f;
          }
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            if (i + u >= m) break;
            const float* ur = row + (i + u) * NH;
            const u64 xx0 = pack2(x0[u], x0[u]), xx1 = pack2(x1[u], x1[u]);
#pragma unroll
            for (int n = 0; n < NH; n += 4) {
              const ulonglong2 uu = *reinterpret_cast<const ulonglong2*>(ur + n);
              acc0[n / 2] = fma2(xx0, uu.x, acc0[n / 2]);
              acc0[n / 2 + 1] = fma2(xx0, uu.y, acc0[n / 2 + 1]);
              acc1[n / 2] = fma2(xx1, uu.x, acc1[n / 2]);
              acc1[n / 2 + 1] = fma2(xx1, uu.y, acc1[n / 2 + 1]);
            }
          }
        }
      } else {
        const int pb0 = sig ^ pa0, pb1 = sig ^ pa1;
        const float* r0 = us + a0 * hp + (pb0 ? nb0 : 0) * NH;
        const float* r1 = us + a1 * hp + (pb1 ? nb0 : 0) * NH;
        for (int i = 0; i < (pb0 ? nb1 : nb0); ++i) fma_row2<NH>(x[o0 + (long long)l.b[pb0][i] * H], r0 + i * NH, acc0);
        for (int i = 0; i < (pb1 ? nb1 : nb0); ++i) fma_row2<NH>(x[o1 + (long long)l.b[pb1][i] * H], r1 + i * NH, acc1);
      }
#pragma unroll
      for (int n = 0; n < NH; n += 2) {
        float v0, w0, v1, w1;
        unpack2(acc0[n / 2], v0, w0);
        unpack2(acc1[n / 2], v1, w1);
        if (n >= ncols) break;
        const int z = __shfl_sync(0xffffffffu, pos, n);
        // past the end of the list stands the K padding, which reads as zero
        if (ok0) store_pair<PF>(ob + z * ldb, psb, zo.npieces, v0, ok1 ? v1 : 0.0f);
        if (n + 1 >= ncols) break;
        const int z1 = __shfl_sync(0xffffffffu, pos, n + 1);
        if (ok0) store_pair<PF>(ob + z1 * ldb, psb, zo.npieces, w0, ok1 ? w1 : 0.0f);
      }
    }
  }
}

// First non-prime stage.  C rows (rr, a), columns (cc, b); output [rr][cc][n], FP32, zero where the
// parities forbid it.  A warp takes 32 neighbouring cc of one rr.  In a block's row the check indices of
// one cc stand next to each other (VEC: class sizes and so their starts are multiples of VEC), so a
// lane's terms for one hat index are one or two vector loads and a warp reads a contiguous stretch.
template <int NH, int VEC>
__global__ void __launch_bounds__(256, NH <= 8 ? 4 : (NH <= 12 ? 3 : 2)) z2_nonprime_kernel(Z2Chain p, Z2In zi, long long rrs, long long ccs,
                                                          float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_u[];
  __shared__ Lists l;
  float* us = reinterpret_cast<float*>(smem_u);
  const int hp = hat_pitch<NH>(p.chi);
  load_u<NH>(p, us, &l);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* tile = us + p.chi * hp + warp * 32 * (p.nn + 1);
  // class sizes (selects, not arrays: an indexed array would live in local memory)
  const int nb1 = __popc(p.mask_b), nb0 = p.chi - nb1, nc1 = __popc(p.mask_n), nc0 = p.nn - nc1;
  const int pb0 = (int)(p.mask_b & 1u);
  constexpr int MB = NH <= 16 ? NH : 8;
  const long long chunks = (ccs + 31) / 32, tasks = rrs * chunks;
  for (long long t = (long long)blockIdx.x * 8 + warp; t < tasks; t += (long long)gridDim.x * 8) {
    const long long rr = t / chunks, cc0 = (t - rr * chunks) * 32;
    const int live = (int)min(32LL, ccs - cc0);
    const long long cc = cc0 + min(lane, live - 1);
    // rows: lane a holds the position and block of (rr, a)
    unsigned zr = 0u;
    if (lane < p.chi) zr = (unsigned)zi.rpos[rr * p.chi + lane] | ((unsigned)zi.rblk[rr * p.chi + lane] << 31);
    // columns: the block of (cc, b) is blk0 ^ par(b); the first of each parity
    const int cpar = zi.cblk[cc * p.chi] ^ pb0 ^ zi.q;
    const int s0 = nb0 ? zi.cpos[cc * p.chi + l.b[0][0]] : 0, s1 = nb1 ? zi.cpos[cc * p.chi + l.b[1][0]] : 0;
    u64 acc[NH / 2];
#pragma unroll
    for (int n = 0; n < NH / 2; ++n) acc[n] = 0ULL;
    int sig = 0;   // the parity of the new indices with a nonzero result: that of (rr, cc)
    // the terms of one hat index: their count, their rows of U~ and (up to MB of them) their values; the
    // next hat index is read while one is summed
    auto fetch = [&](int a, int& m, const float*& ur, const float*& x, float (&v)[MB]) {
      const unsigned z = __shfl_sync(0xffffffffu, zr, a);
      const int rb = (int)(z >> 31), pb = rb ^ cpar;
      if (a == 0) sig = pb ^ (int)(p.mask_b & 1u);
      const float* cr = rb ? zi.c[1] : zi.c[0];
      m = cr ? (pb ? nb1 : nb0) : 0;
      ur = us + a * hp + (pb ? nb0 : 0) * NH;
      x = cr + (long long)(z & 0x7fffffffu) * zi.ld + (pb ? s1 : s0);
      if (VEC == 4) {
#pragma unroll
        for (int i = 0; i + 3 < MB; i += 4)
          if (i < m) *reinterpret_cast<float4*>(v + i) = *reinterpret_cast<const float4*>(x + i);
      } else if (VEC == 2) {
#pragma unroll
        for (int i = 0; i + 1 < MB; i += 2)
          if (i < m) *reinterpret_cast<float2*>(v + i) = *reinterpret_cast<const float2*>(x + i);
      } else {
#pragma unroll
        for (int i = 0; i < MB; ++i)
          if (i < m) v[i] = x[i];
      }
    };
    int m;
    const float *ur, *x;
    alignas(16) float v[MB];
    fetch(0, m, ur, x, v);
    for (int a = 0; a < p.chi; ++a) {
      int m1 = 0;
      const float *ur1 = ur, *x1 = x;
      alignas(16) float v1[MB];
      if (a + 1 < p.chi) fetch(a + 1, m1, ur1, x1, v1);
      u64 part[NH / 2];
#pragma unroll
      for (int n = 0; n < NH / 2; ++n) part[n] = 0ULL;
#pragma unroll
      for (int i = 0; i < MB; ++i)
        if (i < m) fma_row2<NH>(v[i], ur + i * NH, part);
      for (int i = MB; i < m; ++i) fma_row2<NH>(x[i], ur + i * NH, part);
#pragma unroll
      for (int n = 0; n < NH / 2; ++n) acc[n] = add2(acc[n], part[n]);
      m = m1;
      ur = ur1;
      x = x1;
#pragma unroll
      for (int i = 0; i < MB; ++i) v[i] = v1[i];
    }
    // through shared memory, so that the warp's outputs leave in one contiguous stretch
    const int ncols = sig ? nc1 : nc0;
    float* mine = tile + lane * (p.nn + 1);
#pragma unroll
    for (int n = 0; n < NH; n += 2) {
      float v, w;
      unpack2(acc[n / 2], v, w);
      if (n < ncols) mine[l.n[sig][n]] = v;
      if (n + 1 < ncols) mine[l.n[sig][n + 1]] = w;
    }
    for (int n = 0; n < p.nn - ncols; ++n) mine[l.n[sig ^ 1][n]] = 0.0f;
    __syncwarp();
    float* o = out + (rr * ccs + cc0) * p.nn;
    int i = lane / p.nn, n = lane - i * p.nn;
    for (int e = lane; e < live * p.nn; e += 32) {
      o[e] = tile[i * (p.nn + 1) + n];
      n += 32;
      while (n >= p.nn) {
        n -= p.nn;
        ++i;
      }
    }
    __syncwarp();
  }
}

namespace {

int half_width(const Z2Chain& p) {   // columns of the larger parity class
  const int n1 = __builtin_popcount(p.mask_n);
  return n1 > p.nn - n1 ? n1 : p.nn - n1;
}

// the kernel's shared-memory limit, raised where U~ needs more than the default; false: it does not fit
template <typename K>
bool room(K kernel, size_t smem) {
  if (smem > 226 * 1024) return false;
  return smem <= 40 * 1024 ||
         cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
}

template <int PF, int NH>
bool prime_nh(const Z2Chain& p, const float* in, int H, int chi_c, int P, int groups, const int* kcat, int rb0, int R,
              const Z2Blocks& zo, int ctas_per_sm, cudaStream_t s) {
  const size_t smem = sizeof(float) * p.chi * (p.chi * NH + 4);
  auto kernel = z2_prime_kernel<PF, NH>;
  if (!room(kernel, smem)) return false;
  const long long chunks = (rb0 + 63) / 64 + (R - rb0 + 63) / 64;
  const long long warps = 8LL * ctas_per_sm * sm_count();
  int gper = 8;   // row groups a warp takes per decoding, fewer where there are not enough warps
  while (gper > 1 && chunks * ((groups + gper - 1) / gper) < 2 * warps) gper >>= 1;
  const long long tasks = chunks * ((groups + gper - 1) / gper);
  long long blocks = (tasks + 7) / 8;
  if (blocks > warps / 8) blocks = warps / 8;
  kernel<<<(unsigned)blocks, 256, smem, s>>>(p, in, H, chi_c, P, groups, gper, kcat, rb0, R, zo);
  ++g_launches;
  return true;
}

template <int PF>
bool prime_pf(const Z2Chain& p, const float* in, int H, int chi_c, int P, int groups, const int* kcat, int rb0, int R,
              const Z2Blocks& zo, int cps, cudaStream_t s) {
  const int w = half_width(p);
  if (w <= 4) return prime_nh<PF, 4>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 8) return prime_nh<PF, 8>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 12) return prime_nh<PF, 12>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 16) return prime_nh<PF, 16>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  return prime_nh<PF, 32>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
}

template <int NH, int VEC>
bool nonprime_one(const Z2Chain& p, const Z2In& zi, long long rrs, long long ccs, float* out, int cps, cudaStream_t s) {
  const size_t smem = sizeof(float) * (p.chi * (p.chi * NH + 4) + 8 * 32 * (p.nn + 1));
  auto kernel = z2_nonprime_kernel<NH, VEC>;
  if (!room(kernel, smem)) return false;
  long long blocks = (rrs * ((ccs + 31) / 32) + 7) / 8;
  if (blocks > (long long)cps * sm_count()) blocks = (long long)cps * sm_count();
  kernel<<<(unsigned)blocks, 256, smem, s>>>(p, zi, rrs, ccs, out);
  ++g_launches;
  return true;
}

template <int NH>
bool nonprime_nh(const Z2Chain& p, const Z2In& zi, long long rrs, long long ccs, float* out, int cps, cudaStream_t s) {
  const int b1 = __builtin_popcount(p.mask_b), b0 = p.chi - b1;
  if ((b0 | b1) % 4 == 0 && zi.ld % 4 == 0) return nonprime_one<NH, 4>(p, zi, rrs, ccs, out, cps, s);
  if ((b0 | b1) % 2 == 0 && zi.ld % 2 == 0) return nonprime_one<NH, 2>(p, zi, rrs, ccs, out, cps, s);
  return nonprime_one<NH, 1>(p, zi, rrs, ccs, out, cps, s);
}

}  // namespace

bool launch_z2_prime(const Z2Chain& p, const float* in, int H, int chi_c, int P, long long groups, const int* kcat,
                     int rb0, int R, const Z2Blocks& zo, int pfmt, int ctas_per_sm, cudaStream_t s) {
  if (groups < 1 || groups >= (1LL << 31)) return false;
  return pfmt == PIECE_TF32
             ? prime_pf<PIECE_TF32>(p, in, H, chi_c, P, (int)groups, kcat, rb0, R, zo, ctas_per_sm, s)
             : prime_pf<PIECE_BF16>(p, in, H, chi_c, P, (int)groups, kcat, rb0, R, zo, ctas_per_sm, s);
}

bool launch_z2_nonprime(const Z2Chain& p, const Z2In& zi, long long rrs, long long ccs, float* out, int ctas_per_sm,
                        cudaStream_t s) {
  const int w = half_width(p);
  if (w <= 4) return nonprime_nh<4>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 8) return nonprime_nh<8>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 12) return nonprime_nh<12>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 16) return nonprime_nh<16>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  return nonprime_nh<32>(p, zi, rrs, ccs, out, ctas_per_sm, s);
}

}  // namespace hotrg
