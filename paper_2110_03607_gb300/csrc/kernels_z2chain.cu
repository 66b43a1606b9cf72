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
// The dense form runs through the same kernels as one block with one parity.
//
// 3D chi = 16, one c'-slice (0.8 GB of B written, 0.54 GB of C read): prime 0.85 -> 0.30 ms, bound by
// instruction issue (67 % of the slots: forming, packing and storing the pieces is half of it), 2.7 TB/s
// written; non-prime 0.57 -> 0.22 ms, bound by the L1 pipe (reads of U~, then of C), 2.4 TB/s read.  Per step
// at chi = 20: 108 -> 47 and 119 -> 32 ms.
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

template <int PF, int NP>
__device__ __forceinline__ void store_pair(char* o, long long pbytes, float v0, float v1) {
  if (PF == PIECE_TF32) {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const float w0 = round_tf32(v0), w1 = round_tf32(v1);
      *reinterpret_cast<float2*>(o) = make_float2(w0, w1);
      v0 -= w0;
      v1 -= w1;
      o += pbytes;
    }
  } else {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
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
template <int PF, int NP, int NH>
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
  constexpr int UB = 4;
  __shared__ int bo[64];   // offset of the i-th check index of a parity
  if (threadIdx.x < 64) bo[threadIdx.x] = (threadIdx.x & 31) < (threadIdx.x < 32 ? nb0 : nb1) ? l.b[threadIdx.x >> 5][threadIdx.x & 31] * H : 0;
  __syncthreads();
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
        const int* bl = bo + pb * 32;
        const float *xa = x + o0, *xb = x + o1;
        for (int i = 0; i < m; i += UB) {
          float x0[UB], x1[UB];
#pragma unroll
          for (int u = 0; u < UB; ++u)
            if (i + u < m) {
              const int ofs = bl[i + u];
              x0[u] = xa[ofs];
              x1[u] = xb[ofs];
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
        if (ok0) store_pair<PF, NP>(ob + z * ldb, psb, v0, ok1 ? v1 : 0.0f);
        if (n + 1 >= ncols) break;
        const int z1 = __shfl_sync(0xffffffffu, pos, n + 1);
        if (ok0) store_pair<PF, NP>(ob + z1 * ldb, psb, w0, ok1 ? w1 : 0.0f);
      }
    }
  }
}

// First non-prime stage.  C rows (rr, a), columns (cc, b); output [rr][cc][n], FP32, zero where the
// parities forbid it.  A warp takes 128 neighbouring cc of one rr and goes through those of either parity
// by themselves, two a lane: the rows of U~ are then the same for all its lanes and serve two outputs a
// read (with both parities together and one output a lane these reads took 92 % of the L1 pipe).  In a
// block's row the check indices of one cc stand next to each other (VEC: class sizes, and so their
// starts, are multiples of VEC), so that a lane's terms for one hat index are one or two vector loads of
// whole sectors.
constexpr int kCcs = 128;
template <int NH, int VEC>
__global__ void __launch_bounds__(256, NH <= 8 ? 3 : (NH <= 16 ? 2 : 1)) z2_nonprime_kernel(Z2Chain p, Z2In zi, long long rrs, long long ccs,
                                                          float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_u[];
  __shared__ Lists l;
  __shared__ unsigned char s_list[8][kCcs];
  float* us = reinterpret_cast<float*>(smem_u);
  const int hp = hat_pitch<NH>(p.chi);
  load_u<NH>(p, us, &l);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* tile = us + p.chi * hp + warp * 64 * (p.nn + 1);
  unsigned char* list = s_list[warp];   // even ones from the front, odd ones from the back
  const int nb1 = __popc(p.mask_b), nb0 = p.chi - nb1, nc1 = __popc(p.mask_n), nc0 = p.nn - nc1;
  const int pb0 = (int)(p.mask_b & 1u);
  constexpr int MB = NH <= 16 ? NH : 8;
  const long long chunks = (ccs + kCcs - 1) / kCcs, tasks = rrs * chunks;
  for (long long t = (long long)blockIdx.x * 8 + warp; t < tasks; t += (long long)gridDim.x * 8) {
    const long long rr = t / chunks, c0 = (t - rr * chunks) * kCcs;
    const int live = (int)min((long long)kCcs, ccs - c0);
    // rows: lane a holds the position and block of (rr, a)
    unsigned zr = 0u;
    if (lane < p.chi) zr = (unsigned)zi.rpos[rr * p.chi + lane] | ((unsigned)zi.rblk[rr * p.chi + lane] << 31);
    // the block of column (cc, b) is cpar ^ par(b)
    int count[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < kCcs / 32; ++q) {
      const int i = q * 32 + lane;
      const bool ok = i < live;
      const int cpar = ok ? zi.cblk[(c0 + i) * p.chi] ^ pb0 ^ zi.q : 0;
      const unsigned odd = __ballot_sync(0xffffffffu, ok && cpar), even = __ballot_sync(0xffffffffu, ok && !cpar);
      const unsigned below = (1u << lane) - 1u;
      if (ok) list[cpar ? kCcs - 1 - count[1] - __popc(odd & below) : count[0] + __popc(even & below)] = (unsigned char)i;
      count[0] += __popc(even);
      count[1] += __popc(odd);
    }
    __syncwarp();
#pragma unroll 1
    for (int cpar = 0; cpar < 2; ++cpar) {
      const int cnt = cpar ? count[1] : count[0];
#pragma unroll 1
      for (int base = 0; base < cnt; base += 64) {
        const int e0 = min(base + lane, cnt - 1), e1 = min(base + lane + 32, cnt - 1);
        const long long k0 = (c0 + list[cpar ? kCcs - 1 - e0 : e0]) * p.chi, k1 = (c0 + list[cpar ? kCcs - 1 - e1 : e1]) * p.chi;
        // the first column of either class of check indices
        const int s00 = nb0 ? zi.cpos[k0 + l.b[0][0]] : 0, s01 = nb1 ? zi.cpos[k0 + l.b[1][0]] : 0;
        const int s10 = nb0 ? zi.cpos[k1 + l.b[0][0]] : 0, s11 = nb1 ? zi.cpos[k1 + l.b[1][0]] : 0;
        u64 acc0[NH / 2], acc1[NH / 2];
#pragma unroll
        for (int n = 0; n < NH / 2; ++n) acc0[n] = acc1[n] = 0ULL;
        int sig = 0;   // the parity of the new indices with a nonzero result: that of (rr, cc)
#pragma unroll 1
        for (int a = 0; a < p.chi; ++a) {
          const unsigned z = __shfl_sync(0xffffffffu, zr, a);
          const int rb = (int)(z >> 31), pb = rb ^ cpar, m = pb ? nb1 : nb0;
          if (a == 0) sig = pb ^ pb0;
          const float* cr = rb ? zi.c[1] : zi.c[0];
          if (!cr) continue;
          cr += (long long)(z & 0x7fffffffu) * zi.ld;
          const float *x0 = cr + (pb ? s01 : s00), *x1 = cr + (pb ? s11 : s10);
          const float* ur = us + a * hp + (pb ? nb0 : 0) * NH;
          u64 part0[NH / 2], part1[NH / 2];
#pragma unroll
          for (int n = 0; n < NH / 2; ++n) part0[n] = part1[n] = 0ULL;
          for (int i0 = 0; i0 < m; i0 += MB) {
            alignas(16) float v0[MB], v1[MB];
#pragma unroll
            for (int i = 0; i < MB; i += VEC)
              if (i0 + i < m) {
                if constexpr (VEC == 4) {
                  *reinterpret_cast<float4*>(v0 + i) = *reinterpret_cast<const float4*>(x0 + i0 + i);
                  *reinterpret_cast<float4*>(v1 + i) = *reinterpret_cast<const float4*>(x1 + i0 + i);
                } else if constexpr (VEC == 2) {
                  *reinterpret_cast<float2*>(v0 + i) = *reinterpret_cast<const float2*>(x0 + i0 + i);
                  *reinterpret_cast<float2*>(v1 + i) = *reinterpret_cast<const float2*>(x1 + i0 + i);
                } else {
                  v0[i] = x0[i0 + i];
                  v1[i] = x1[i0 + i];
                }
              }
#pragma unroll
            for (int i = 0; i < MB; ++i) {
              if (i0 + i >= m) break;
              const float* row = ur + (i0 + i) * NH;
              const u64 xx0 = pack2(v0[i], v0[i]), xx1 = pack2(v1[i], v1[i]);
#pragma unroll
              for (int n = 0; n < NH; n += 4) {
                const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(row + n);
                part0[n / 2] = fma2(xx0, u.x, part0[n / 2]);
                part0[n / 2 + 1] = fma2(xx0, u.y, part0[n / 2 + 1]);
                part1[n / 2] = fma2(xx1, u.x, part1[n / 2]);
                part1[n / 2 + 1] = fma2(xx1, u.y, part1[n / 2 + 1]);
              }
            }
          }
#pragma unroll
          for (int n = 0; n < NH / 2; ++n) {
            acc0[n] = add2(acc0[n], part0[n]);
            acc1[n] = add2(acc1[n], part1[n]);
          }
        }
        // through shared memory, so that the outputs of a cc leave together
        const int ncols = sig ? nc1 : nc0;
        float *mine0 = tile + lane * (p.nn + 1), *mine1 = mine0 + 32 * (p.nn + 1);
#pragma unroll
        for (int n = 0; n < NH; n += 2) {
          float v, w, v1, w1;
          unpack2(acc0[n / 2], v, w);
          unpack2(acc1[n / 2], v1, w1);
          if (n < ncols) {
            mine0[l.n[sig][n]] = v;
            mine1[l.n[sig][n]] = v1;
          }
          if (n + 1 < ncols) {
            mine0[l.n[sig][n + 1]] = w;
            mine1[l.n[sig][n + 1]] = w1;
          }
        }
        for (int n = 0; n < p.nn - ncols; ++n) mine0[l.n[sig ^ 1][n]] = mine1[l.n[sig ^ 1][n]] = 0.0f;
        __syncwarp();
        const int rows = min(64, cnt - base);
        int i = lane / p.nn, n = lane - i * p.nn;
        for (int e = lane; e < rows * p.nn; e += 32) {
          const int k = base + i;
          out[(rr * ccs + c0 + list[cpar ? kCcs - 1 - k : k]) * p.nn + n] = tile[i * (p.nn + 1) + n];
          n += 32;
          while (n >= p.nn) {
            n -= p.nn;
            ++i;
          }
        }
        __syncwarp();
      }
    }
    __syncwarp();
  }
}

namespace {

constexpr int kChainDynSmem = 224 * 1024;   // the kernels' lists take 2 KB of an SM's 227

int half_width(const Z2Chain& p) {   // columns of the larger parity class
  const int n1 = __builtin_popcount(p.mask_n);
  return n1 > p.nn - n1 ? n1 : p.nn - n1;
}

// the kernel's shared-memory limit, raised where U~ needs more than the default; false: it does not fit
template <typename K>
bool room(K kernel, size_t smem) {
  return smem <= kChainDynSmem && (smem <= 40 * 1024 || raise_smem_limit(kernel, kChainDynSmem));
}

template <int PF, int NP, int NH>
bool prime_nh(const Z2Chain& p, const float* in, int H, int chi_c, int P, int groups, const int* kcat, int rb0, int R,
              const Z2Blocks& zo, int ctas_per_sm, cudaStream_t s) {
  const size_t smem = sizeof(float) * p.chi * (p.chi * NH + 4);
  auto kernel = z2_prime_kernel<PF, NP, NH>;
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

template <int PF, int NP>
bool prime_pf(const Z2Chain& p, const float* in, int H, int chi_c, int P, int groups, const int* kcat, int rb0, int R,
              const Z2Blocks& zo, int cps, cudaStream_t s) {
  const int w = half_width(p);
  if (w <= 4) return prime_nh<PF, NP, 4>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 8) return prime_nh<PF, NP, 8>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 12) return prime_nh<PF, NP, 12>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 16) return prime_nh<PF, NP, 16>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 20) return prime_nh<PF, NP, 20>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  if (w <= 24) return prime_nh<PF, NP, 24>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
  return prime_nh<PF, NP, 32>(p, in, H, chi_c, P, groups, kcat, rb0, R, zo, cps, s);
}

template <int NH, int VEC>
bool nonprime_one(const Z2Chain& p, const Z2In& zi, long long rrs, long long ccs, float* out, int cps, cudaStream_t s) {
  const size_t smem = sizeof(float) * (p.chi * (p.chi * NH + 4) + 8 * 64 * (p.nn + 1));
  auto kernel = z2_nonprime_kernel<NH, VEC>;
  if (!room(kernel, smem)) return false;
  long long blocks = (rrs * ((ccs + kCcs - 1) / kCcs) + 7) / 8;
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
  if (groups < 1 || groups >= (1LL << 31) || zo.npieces < (pfmt == PIECE_TF32 ? 1 : 2) ||
      zo.npieces > (pfmt == PIECE_TF32 ? 2 : 3))
    return false;
  const int n = zo.npieces;
  if (pfmt == PIECE_TF32)
    return n == 1 ? prime_pf<PIECE_TF32, 1>(p, in, H, chi_c, P, (int)groups, kcat, rb0, R, zo, ctas_per_sm, s)
                  : prime_pf<PIECE_TF32, 2>(p, in, H, chi_c, P, (int)groups, kcat, rb0, R, zo, ctas_per_sm, s);
  return n == 2 ? prime_pf<PIECE_BF16, 2>(p, in, H, chi_c, P, (int)groups, kcat, rb0, R, zo, ctas_per_sm, s)
                : prime_pf<PIECE_BF16, 3>(p, in, H, chi_c, P, (int)groups, kcat, rb0, R, zo, ctas_per_sm, s);
}

bool launch_z2_nonprime(const Z2Chain& p, const Z2In& zi, long long rrs, long long ccs, float* out, int ctas_per_sm,
                        cudaStream_t s) {
  const int w = half_width(p);
  if (w <= 4) return nonprime_nh<4>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 8) return nonprime_nh<8>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 12) return nonprime_nh<12>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 16) return nonprime_nh<16>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 20) return nonprime_nh<20>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  if (w <= 24) return nonprime_nh<24>(p, zi, rrs, ccs, out, ctas_per_sm, s);
  return nonprime_nh<32>(p, zi, rrs, ccs, out, ctas_per_sm, s);
}

}  // namespace hotrg
