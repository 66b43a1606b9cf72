// FP64 products on the tensor cores: C = A . B^T from exact products of digits.
//
// The FP64 pipe of this chip does 2 multiply-adds per clock and SM (1.25 TFLOP/s); its BF16 tensor
// cores do 4096 times as many.  Following Ozaki, Ogita, Oishi and Rump (Numerical Algorithms 59, 2012),
// every row of an operand is written as integers of a common unit 2^(e - 62), 2^e > max |x|, rounded to
// nearest, and each integer as eight signed digits in base 256 (seven in [-128, 127], the leading one in
// [-65, 65]):
//   x = sum_a v_a 2^(e - 6 - 8 a).
// A digit is exact in BF16, a product of two is at most 2^14, and the tensor core adds into an FP32
// accumulator without error while every partial sum stays within 2^24.  The products v_a w_b with
// a + b = g share one accumulator (they share the weight 2^-8g): at most 8 products times 128
// along K, 2^14 2^3 2^7 = 2^24.  So each chunk of 128 along K gives nine exact integers P_0 .. P_8 per
// output; they are added, P_8 rounded to P_7's unit, into two 64-bit integers (hi: g = 0 .. 3, lo: g = 4 .. 8),
// and one rounding to FP64 ends the sum.
//
// What this leaves out, with alpha = |a| / 2^ea and beta = |b| / 2^eb in [0, 1) and results in units of
// 2^(ea + eb): of an element the bits below 2^-62, at most 2^-63 and of either sign, which is 2^-63.8
// sqrt(|alpha|^2 + |beta|^2) in the mean (2-norms of the rows) and 2^-63 sum (alpha + beta) at the most; of the
// digits' products those with a + b > 8, six of either sign at 2^-84 each: 2^-70 sqrt(K) in the mean, K 2^-67.4 at
// the most.  (a + b = 8 is needed for rows with the same digits, the diagonal of a Gram or equal rows of two
// operands: v_4^2 is positive, and 32,768 of them were 2e-15 of the sum of a row with one large element.)
// An FP64 sum has errors of a few 2^-54 of s = sum alpha beta in the mean and K 2^-53 s at the most.  So the
// digits are as good, entry by entry, where s >= 2^-9 (|alpha| + |beta|) (an error of 2^-54.8 s); where the
// large elements of one row meet the small ones of the other, or a row holds an infinity or a NaN, they are not.
// Therefore s is computed too, as one more product of BF16 (a ninth plane, alpha rounded down, and a tenth
// accumulator, summed over all of K in FP32), and f64_fix_kernel forms the entries that fail the test on the
// FP64 pipe.  Rows of coarse-grained tensors pass in general: no entry of the Grams and products of 3D steps
// (bonds 9 x 11 x 10 and 12 to 16, zero field or 0.01 and 0.02) fails at 2^-9, 0.1 % of the worst product at 2^-8.
// Near a trivial fixed point, where a few elements rule a tensor, or in a field of 1e-4, whose odd elements are
// that small, a tenth to two thirds do: there the digits lost up to all of an entry's own figures.
//
// Layout: tile 128 x 48 of C per CTA, its ten accumulators fill 480 of the 512 columns of TMEM.  A ring of
// two stages holds K slabs of 32 (64-byte rows), all nine planes of both operands (99 KB a stage).  44 products of
// 48 columns; with eight accumulators of 64 columns (36 products, entries unguarded) the FP64 products of a 3D step,
// bonds 9 x 11 x 10, took 12.8 ms with their slicing, so 22.4.
// The MMA warp goes through a slab by accumulator g, and waits for the epilogue once per g and chunk,
// so the drain of one accumulator runs under the MMAs of the next.
#include <stdio.h>

#include <algorithm>
#include <atomic>

#include "tcgen05.cuh"

namespace hotrg {

namespace {
constexpr int TM = 128, TN = 48, TK = 32, DIG = 8, STAGES = 2;
constexpr int PLANES = DIG + 1;                 // the digits and alpha
constexpr int ACCS = 9;                         // of the digits' products; the tenth sums alpha beta
constexpr int CHUNK = 4;                        // slabs per exact sum: 128 along K
constexpr int A_PLANE = TM * TK * 2, B_PLANE = TN * TK * 2;
constexpr int STAGE_BYTES = PLANES * (A_PLANE + B_PLANE);
constexpr int SMEM_BYTES = 1024 + STAGES * STAGE_BYTES + 512;
constexpr int EPI_WARPS = 8, W_PROD = 8, W_MMA = 9, NTHREADS = 320;
constexpr int NON_FINITE = 0x7fffffff;          // a row with an infinity or a NaN
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of one CTA");
static_assert((ACCS + 1) * TN <= 512 && TN % 16 == 0, "columns of TMEM");
constexpr float kTrust = 0.001953125f;          // 2^-9: the least s / (|alpha| + |beta|) of an entry taken from the digits

struct SliceDesc {
  const double* x;
  long long ld;
  int rows;
  __nv_bfloat16* v;        // plane a of element (r, k) at (a rows + r) kpad + k
  unsigned long long* q;   // per row: sum of alpha^2 in units of 2^-30
  int* e;                  // per row: biased exponent of the largest |x|, at least 1
};

// largest |x| of a row, as the high word of its bits (0 below 2^-1042: the row's unit is then that
// of the smallest normal numbers)
__device__ __forceinline__ int high_abs(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int row_exponent(int hi) {
  const int e = hi >> 20;
  return e == 0x7ff ? NON_FINITE : (e < 1 ? 1 : e);
}

// digits of x in a row whose largest exponent is E, packed: byte 7 - a holds v_a + 128
__device__ __forceinline__ unsigned long long digits(double x, int E) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  int be = (int)(bits >> 52) & 0x7ff;
  unsigned long long m = bits & 0xfffffffffffffULL;
  if (be) m |= 0x10000000000000ULL;
  else be = 1;
  const int sh = be - E + 9;                    // x = m 2^(be - 1075), unit 2^(E - 1084); sh <= 9
  unsigned long long f = sh >= 0 ? m << (sh & 15) : (sh > -64 ? (m + (1ULL << (-sh - 1))) >> -sh : 0ULL);
  if ((long long)bits < 0) f = 0ULL - f;
  return (f + 0x0080808080808080ULL) ^ 0x8000000000000000ULL;
}
// alpha = |x| 2^(1022 - E), as the bits of a BF16 number, rounded down; what is not zero is at least 2^-60, so
// that a sum of products is zero only if every product is
__device__ __forceinline__ unsigned alpha_bits(double x, int E) {
  const unsigned hi = (unsigned)high_abs(x);
  const int be = (int)(hi >> 20), ex = be - E - 1;
  if (be == 0) return (hi | (unsigned)__double2loint(x)) != 0u ? 67u << 7 : 0u;
  return ex < -60 ? 67u << 7 : (unsigned)(ex + 127) << 7 | ((hi >> 13) & 0x7fu);
}

// eight consecutive elements -> one 16-byte store per plane; the sum of alpha^2 is returned
__device__ __forceinline__ float store_planes(const double (&x)[8], int E, __nv_bfloat16* dst, long long dstride) {
  unsigned lo[8], hi[8], al[4];
  float sq = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned long long d = E == NON_FINITE ? 0x8080808080808080ULL : digits(x[i], E);
    lo[i] = (unsigned)d;
    hi[i] = (unsigned)(d >> 32);
    const unsigned a = E == NON_FINITE ? 0u : alpha_bits(x[i], E);
    al[i >> 1] = i & 1 ? al[i >> 1] | a << 16 : a;
    const float f = __uint_as_float(a << 16);
    sq = fmaf(f, f, sq);
  }
#pragma unroll
  for (int a = 0; a < DIG; ++a) {
    unsigned w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      unsigned f[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        // 2^23 + (v + 128) as an FP32 word, less 2^23 + 128: v, exact, its low 16 bits zero
        const unsigned word = a < 4 ? hi[2 * i + q] : lo[2 * i + q];
        const unsigned u = __byte_perm(word, 0x4b000000u, 0x7540 + (3 - (a & 3)));
        f[q] = __float_as_uint(__uint_as_float(u) - 8388736.0f);
      }
      w[i] = __byte_perm(f[0], f[1], 0x7632);
    }
    *reinterpret_cast<uint4*>(dst + a * dstride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  *reinterpret_cast<uint4*>(dst + DIG * dstride) = make_uint4(al[0], al[1], al[2], al[3]);
  return sq;
}
// a sum of alpha^2 in units of 2^-30, rounded up: integers add up to the same in any order
__device__ __forceinline__ unsigned long long norm_units(float sq) {
  return (unsigned long long)ceilf(sq * 1073741824.0f);
}

__device__ __forceinline__ void load8(const double* x, int n, double (&v)[8]) {
  if (n >= 8 && (((uintptr_t)x) & 15) == 0) {
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const double2 t = *reinterpret_cast<const double2*>(x + i);
      v[i] = t.x;
      v[i + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = i < n ? x[i] : 0.0;
  }
}

// Short rows (K <= 2048): 2^tprl threads per row of either operand, eight elements each; exponent and
// planes in one pass.
__global__ void __launch_bounds__(256) slice_short_kernel(SliceDesc A, SliceDesc B, int K, int kpad, int tprl) {
  const int tpr = 1 << tprl;
  const long long r0 = (long long)blockIdx.x * (256 >> tprl) + (threadIdx.x >> tprl);
  const int t = threadIdx.x & (tpr - 1), k = t * 8;
  const bool second = r0 >= A.rows;
  const SliceDesc& d = second ? B : A;
  const long long r = second ? r0 - A.rows : r0;
  const bool live = r < d.rows;
  double x[8];
  load8(d.x + (live ? r * d.ld + (k < K ? k : 0) : 0), live ? K - k : 0, x);
  int hi = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) hi = max(hi, high_abs(x[i]));
  __shared__ int wmax[8];
  __shared__ unsigned long long wsum[8];
  const int w = threadIdx.x >> 5, wpr = tpr >> 5;
  for (int o = min(tpr, 32) >> 1; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  if (tpr > 32) {
    if ((threadIdx.x & 31) == 0) wmax[w] = hi;
    __syncthreads();
    for (int q = 0; q < wpr; ++q) hi = max(hi, wmax[(w & ~(wpr - 1)) + q]);
  }
  const int E = row_exponent(hi);
  float sq = 0.0f;
  if (live && k < kpad) sq = store_planes(x, E, d.v + r * kpad + k, (long long)d.rows * kpad);
  unsigned long long n = norm_units(sq);
  for (int o = min(tpr, 32) >> 1; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if (tpr > 32) {
    if ((threadIdx.x & 31) == 0) wsum[w] = n;
    __syncthreads();
    n = 0;
    for (int q = 0; q < wpr; ++q) n += wsum[(w & ~(wpr - 1)) + q];
  }
  if (live && t == 0) {
    d.e[r] = E;
    d.q[r] = n;
  }
}

// Long rows: the exponents first (blocks of a row meet in an atomic maximum; e and q zeroed before) ...
__global__ void __launch_bounds__(256) slice_max_kernel(SliceDesc A, SliceDesc B, long long K) {
  const bool second = (int)blockIdx.x >= A.rows;
  const SliceDesc& d = second ? B : A;
  const int r = second ? (int)blockIdx.x - A.rows : (int)blockIdx.x;
  const double* x = d.x + r * d.ld;
  int hi = 0;
  for (long long k = ((long long)blockIdx.y * 256 + threadIdx.x) * 8; k < K; k += (long long)gridDim.y * 2048) {
    double v[8];
    load8(x + k, (int)min(8LL, K - k), v);
#pragma unroll
    for (int i = 0; i < 8; ++i) hi = max(hi, high_abs(v[i]));
  }
  for (int o = 16; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  if ((threadIdx.x & 31) == 0) atomicMax(d.e + r, row_exponent(hi));
}
// ... then the planes
__global__ void __launch_bounds__(256) slice_long_kernel(SliceDesc A, SliceDesc B, long long K, int kpad) {
  const bool second = (int)blockIdx.x >= A.rows;
  const SliceDesc& d = second ? B : A;
  const int r = second ? (int)blockIdx.x - A.rows : (int)blockIdx.x;
  const double* x = d.x + r * d.ld;
  const int E = d.e[r];
  __nv_bfloat16* v0 = d.v + (long long)r * kpad;
  unsigned long long n = 0;
  for (long long k = ((long long)blockIdx.y * 256 + threadIdx.x) * 8; k < kpad; k += (long long)gridDim.y * 2048) {
    double v[8];
    load8(x + (k < K ? k : 0), (int)max(0LL, min(8LL, K - k)), v);
    n += norm_units(store_planes(v, E, v0 + k, (long long)d.rows * kpad));
  }
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(d.q + r, n);
}

// (hi 2^32 + lo) 2^e, rounded once to nearest-even (twice where the result is subnormal); in integer
// arithmetic, because the FP64 pipe would take longer than the drain
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 32);
  unsigned l = (unsigned)lo;
  const bool neg = h < 0;
  if (neg) {
    h = ~h + (l == 0u ? 1 : 0);
    l = 0u - l;
  }
  if (h == 0 && l == 0u) return 0.0;
  const int n = h ? __clzll(h) : 32 + __clz(l) + 32;
  unsigned long long m;
  unsigned rest = 0u;
  if (n == 0) {
    m = (unsigned long long)h;
    rest = l;
  } else if (n < 32) {
    m = ((unsigned long long)h << n) | (l >> (32 - n));
    rest = l << n;
  } else if (n < 64) {
    m = ((unsigned long long)h << n) | ((unsigned long long)l << (n - 32));
  } else {
    m = (unsigned long long)l << (n - 32);
  }
  // value = m 2^(e + 32 - n), the top bit of m set
  unsigned long long q = m >> 11;
  const unsigned rem = (unsigned)m & 0x7ffu;
  if (rem > 0x400u || (rem == 0x400u && (rest != 0u || (q & 1ULL)))) ++q;
  const int be = e + 32 - n + 63 + 1023;   // biased exponent of the leading bit
  if (be >= 1 && be < 2046) {
    const unsigned long long bits = ((unsigned long long)(be - 1) << 52) + q;   // a carry moves the exponent
    return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ULL : 0ULL)));
  }
  const double r = scalbn((double)q, e + 32 - n + 11);
  return neg ? -r : r;
}

struct TcItems {
  int M, N, mt, nt, upper;       // tiles of C; upper: only those that reach the diagonal or above it
  int ntiles;
  int slabs, per;                // K slabs, and slabs of one split (a multiple of CHUNK)
  int nsplit;
};
}  // namespace

// item -> tile and K slabs; tiles run fastest, so the CTAs at work share their K range in L2
__device__ __forceinline__ void item_of(const TcItems& it, long long i, int* m0, int* n0, int* z, int* s0, int* cnt) {
  int t = (int)(i % it.ntiles);
  *z = (int)(i / it.ntiles);
  int ti, tj;
  if (it.upper) {
    // row tile ti: the column tiles from the one that holds column ti TM on
    ti = 0;
    while (t >= it.nt - ti * TM / TN) {
      t -= it.nt - ti * TM / TN;
      ++ti;
    }
    tj = ti * TM / TN + t;
  } else {
    ti = t % it.mt;
    tj = t / it.mt;
  }
  *m0 = ti * TM;
  *n0 = tj * TN;
  *s0 = *z * it.per;
  *cnt = min(it.per, it.slabs - *s0);
}

__global__ void __launch_bounds__(NTHREADS, 1)
    f64_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const int* __restrict__ ea, const int* __restrict__ eb, double* __restrict__ C, long long ldc,
                  long long split_stride, float* __restrict__ S, TcItems its, int* g_err) {
  extern __shared__ uint8_t smem_raw[];
  volatile int* gerr = g_err;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;      // [ACCS] MMA -> epilogue
  uint64_t* tempty = tfull + ACCS;       // [ACCS] epilogue -> MMA
  uint64_t* sfull = tempty + ACCS;       // the sum of alpha beta, once an item
  uint64_t* sempty = sfull + 1;
  uint64_t* drain = sempty + 1;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* cta_abort = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int g = 0; g < ACCS; ++g) {
      mbar_init(tfull + g, 1);
      mbar_init(tempty + g, EPI_WARPS);
    }
    mbar_init(sfull, 1);
    mbar_init(sempty, EPI_WARPS);
    mbar_init(drain, 1);
    *cta_abort = *gerr ? 1 : 0;   // an earlier launch or CTA gave up: do nothing
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmB) : "memory");
  }
  if (warp == W_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const long long nitems = *cta_abort ? 0 : (long long)its.ntiles * its.nsplit;

  if (warp == W_PROD) {
    if (lane == 0) {
      // ---------------- TMA producer: both operands' planes of one K slab per stage
      long long g = 0;
      bool ok = true;
      for (long long i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
        int m0, n0, z, s0, cnt;
        item_of(its, i, &m0, &n0, &z, &s0, &cnt);
        for (int kb = 0; kb < cnt; ++kb, ++g) {
          const int s = (int)(g % STAGES);
          if (!mbar_wait(empty + s, (uint32_t)((g / STAGES) & 1) ^ 1u, cta_abort, gerr)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + s * STAGE_BYTES;
          mbar_expect_tx(full + s, (uint32_t)STAGE_BYTES);
          tma_load_3d(&tmA, st, full + s, (s0 + kb) * TK, m0, 0);
          tma_load_3d(&tmB, st + PLANES * A_PLANE, full + s, (s0 + kb) * TK, n0, 0);
        }
      }
      // no arrival may be in flight when the CTA exits: the last slabs are consumed, or, after an
      // abort, have at least landed
      for (long long q = g > STAGES ? g - STAGES : 0; q < g; ++q) {
        const int s = (int)(q % STAGES);
        const uint32_t ph = (uint32_t)(q / STAGES) & 1u;
        const unsigned long long t0 = gtimer();
        if (ok && !mbar_wait(empty + s, ph, cta_abort, gerr)) ok = false;
        if (!ok)
          while (!mbar_try_wait(full + s, ph))
            if (gtimer() - t0 > WAIT_NS) break;
      }
    }
    __syncwarp();
  } else if (warp == W_MMA) {
    if (lane == 0) {
      // ---------------- MMA issuer: accumulator g of a slab takes the products with a + b = g
      constexpr uint32_t idesc = idesc_bf16_f32(TM, TN);
      bool ok = true;
      long long g = 0, ch = 0, item = 0;   // slabs, chunks and items of this CTA so far
      for (long long i = blockIdx.x; i < nitems && ok; i += gridDim.x, ++item) {
        int m0, n0, z, s0, cnt;
        item_of(its, i, &m0, &n0, &z, &s0, &cnt);
        for (int kb = 0; kb < cnt && ok; ++kb, ++g) {
          const int s = (int)(g % STAGES);
          const bool first = kb % CHUNK == 0, last = kb % CHUNK == CHUNK - 1 || kb == cnt - 1;
          if (!mbar_wait(full + s, (uint32_t)(g / STAGES) & 1u, cta_abort, gerr)) {
            ok = false;
            break;
          }
          const uint32_t st = su32(smem + s * STAGE_BYTES);
          const uint64_t a0 = sdesc_sw<TK * 2>(st), b0 = sdesc_sw<TK * 2>(st + PLANES * A_PLANE);
          for (int acc = 0; acc < ACCS; ++acc) {
            if (first && ch > 0 && !mbar_wait(tempty + acc, (uint32_t)(ch - 1) & 1u, cta_abort, gerr)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t dst = tmem + (uint32_t)(acc * TN);
            const int a_lo = acc < DIG ? 0 : acc - DIG + 1;
            for (int a = a_lo; a < DIG && a <= acc; ++a) {
              const uint64_t da = a0 + (uint64_t)(a * (A_PLANE >> 4)), db = b0 + (uint64_t)((acc - a) * (B_PLANE >> 4));
#pragma unroll
              for (int kk = 0; kk < TK / 16; ++kk)   // 16 BF16 = 32 bytes inside the swizzled row
                umma_bf16(dst, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                          first && a == a_lo && kk == 0 ? 0u : 1u);
            }
            if (last) umma_commit(tfull + acc);
          }
          if (!ok) break;
          // alpha beta, over all slabs of the item
          if (kb == 0 && item > 0 && !mbar_wait(sempty, (uint32_t)(item - 1) & 1u, cta_abort, gerr)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < TK / 16; ++kk)
            umma_bf16(tmem + (uint32_t)(ACCS * TN), a0 + (uint64_t)(DIG * (A_PLANE >> 4) + 2 * kk),
                      b0 + (uint64_t)(DIG * (B_PLANE >> 4) + 2 * kk), idesc, kb == 0 && kk == 0 ? 0u : 1u);
          if (kb == cnt - 1) umma_commit(sfull);
          umma_commit(empty + s);
          if (last) ++ch;
        }
      }
      if (*cta_abort || *gerr) {
        // TMEM is never released under a running MMA (bounded wait)
        umma_commit(drain);
        const unsigned long long t0 = gtimer();
        while (!mbar_try_wait(drain, 0))
          if (gtimer() - t0 > WAIT_NS) break;
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue warps: 32 rows (the warp's TMEM lanes) x TN / 2 columns each
    constexpr int EC = TN / 2;
    const int quarter = warp & 3, part = warp >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(part * EC);
    auto load_acc = [&](int acc, uint32_t (&v)[EC]) {
      uint32_t v0[16], v1[8];
      tmem_ld_async(lane_base + (uint32_t)(acc * TN), v0);
      tmem_ld_async(lane_base + (uint32_t)(acc * TN + 16), v1);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < EC; ++j) v[j] = j < 16 ? v0[j & 15] : v1[j & 7];
    };
    auto release = [&](uint64_t* bar) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(bar)) : "memory");
    };
    bool ok = true;
    long long ch = 0, item = 0;
    for (long long i = blockIdx.x; i < nitems && ok; i += gridDim.x, ++item) {
      int m0, n0, z, s0, cnt;
      item_of(its, i, &m0, &n0, &z, &s0, &cnt);
      long long hi[EC], lo[EC];
#pragma unroll
      for (int j = 0; j < EC; ++j) hi[j] = lo[j] = 0;
      const int nch = (cnt + CHUNK - 1) / CHUNK;
      for (int q = 0; q < nch && ok; ++q, ++ch) {
#pragma unroll
        for (int acc = 0; acc < ACCS; ++acc) {
          // one verdict per warp: tcgen05.ld is a warp-wide instruction
          if (ok) ok = __all_sync(0xffffffffu, mbar_wait(tfull + acc, (uint32_t)ch & 1u, cta_abort, gerr)) != 0;
          if (!ok) continue;
          tc_fence_after();
          uint32_t v[EC];
          load_acc(acc, v);
          release(tempty + acc);
#pragma unroll
          for (int j = 0; j < EC; ++j) {
            const int p = __float2int_rn(__uint_as_float(v[j]));
            if (acc < 4) hi[j] += (long long)p * (1 << (24 - 8 * (acc & 3)));
            else if (acc < 8) lo[j] += (long long)p * (1 << (24 - 8 * (acc & 3)));
            else lo[j] += (p + 128) >> 8;
          }
        }
      }
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(sfull, (uint32_t)item & 1u, cta_abort, gerr)) != 0;
      if (!ok) break;
      tc_fence_after();
      uint32_t sv[EC];
      load_acc(ACCS, sv);
      release(sempty);
      if (*cta_abort) break;
      const int row = m0 + quarter * 32 + lane, col0 = n0 + part * EC;
      if (row < its.M) {
        const int er = ea[row];
        double* dst = C + (long long)z * split_stride + (long long)row * ldc + col0;
        float* sdst = S + ((long long)z * its.M + row) * its.N + col0;
        // x = sum_a v_a 2^(E - 1022 - 6 - 8 a) of each operand; hi counts in units of 2^-24
        const int e0 = er - 2 * 1028 - 24 - 32;
#pragma unroll
        for (int j = 0; j < EC; ++j)
          if (col0 + j < its.N) {
            const int ec = eb[col0 + j];
            // rows that are not finite are left to f64_fix_kernel
            dst[j] = er == NON_FINITE || ec == NON_FINITE ? 0.0 : fixed_to_double(hi[j], lo[j], e0 + ec);
            sdst[j] = __uint_as_float(sv[j]);
          }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == W_MMA) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// S[0] = the sum over the splits: 32 entries a block, each by eight threads (a thread per entry waits for one load
// after another: 12.5 us for 128 x 128 in 64 splits, 4.3 so)
__global__ void __launch_bounds__(256) f64_sum_kernel(float* S, long long plane, int nsplit) {
  __shared__ float part[8][33];
  const int lane = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (long long i0 = (long long)blockIdx.x * 32; i0 < plane; i0 += (long long)gridDim.x * 32) {
    const long long i = i0 + lane;
    float s = 0.0f;
    if (i < plane) {
#pragma unroll 4
      for (int z = y; z < nsplit; z += 8) s += S[z * plane + i];
    }
    part[y][lane] = s;
    __syncthreads();
    if (y == 0 && i < plane) {
#pragma unroll
      for (int q = 1; q < 8; ++q) s += part[q][lane];
      S[i] = s;
    }
    __syncthreads();
  }
}

// The entries that the digits do not give as well as an FP64 sum, from the operands themselves: a warp
// sums up to four entries of a row at a time, in 32 chains and a tree, each by itself, so that an entry's bits
// do not depend on which others failed.  A tile of 16 x 64 and one split per CTA.  Where nothing failed this
// reads S: 41 us for 990 x 16,270, behind 2.3 ms of products, 5 us for 128 x 128 in 64 splits.  Where all did the
// FP64 pipe bounds it as it does gemm_nt_f64_kernel: 600 x 1800 x 1800 4.4 ms in all, 3.1 at the pipe's full rate.
// (Tiles of 64 x 64 left SMs without one: 7.2 ms; their code unrolled over the rows, 10 us for the 128 x 128.)
constexpr int FIX_M = 16, FIX_N = 64;
__global__ void __launch_bounds__(256)
    f64_fix_kernel(const double* __restrict__ A, long long lda, const double* __restrict__ B, long long ldb,
                   double* __restrict__ C, long long ldc, long long split_stride, int M, int N, long long K,
                   long long per, const float* __restrict__ S, const unsigned long long* __restrict__ qa,
                   const int* __restrict__ ea, const unsigned long long* __restrict__ qb, const int* __restrict__ eb,
                   int upper) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // this warp's 32 columns of 4 rows
  const int r0 = blockIdx.y * FIX_M + (warp >> 1) * 4, c0 = blockIdx.x * FIX_N + (warp & 1) * 32, c = c0 + lane;
  if (r0 >= M || c0 >= N || (upper && c0 + 31 < r0)) return;
  // 2^-9 |alpha|; infinite for a row that is not finite
  auto line_of = [](const unsigned long long* q, const int* e, int r) {
    return e[r] == NON_FINITE ? __int_as_float(0x7f800000)
                              : kTrust * 3.0517578125e-5f * sqrtf((float)q[r]);   // 2^-15 sqrt(q)
  };
  float s[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) s[u] = r0 + u < M && c < N ? S[(long long)(r0 + u) * N + c] : 0.0f;
  const float line_c = c < N ? line_of(qb, eb, c) : 0.0f;
  unsigned mine = 0u;   // lane u: the entries of row u to form
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = r0 + u;
    const float line = line_c + (r < M ? line_of(qa, ea, r) : 0.0f);
    // a sum of exact zeros needs nothing; an infinite line is never reached
    const bool good = s[u] >= line || (s[u] == 0.0f && line < __int_as_float(0x7f800000));
    const unsigned todo = __ballot_sync(0xffffffffu, r < M && c < N && !(upper && c < r) && !good);
    if (lane == u) mine = todo;
  }
  unsigned rows = __ballot_sync(0xffffffffu, mine != 0u);
  const long long k_lo = (long long)blockIdx.z * per, k_hi = k_lo + per < K ? k_lo + per : K;
  double* Cz = C + (long long)blockIdx.z * split_stride;
#pragma unroll 1
  for (; rows != 0u; rows &= rows - 1u) {
    const int u = __ffs(rows) - 1;
    unsigned todo = __shfl_sync(0xffffffffu, mine, u);
    const double* a = A + (long long)(r0 + u) * lda;
#pragma unroll 1
    while (todo != 0u) {
      int col[4], cnt = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        col[q] = c0;
        if (todo != 0u) {
          col[q] += __ffs(todo) - 1;
          todo &= todo - 1u;
          cnt = q + 1;
        }
      }
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
      for (long long k = k_lo + lane; k < k_hi; k += 32) {
        const double x = a[k];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < cnt) acc[q] = fma(x, B[(long long)col[q] * ldb + k], acc[q]);
      }
      // the four sums over the lanes: halves are exchanged while there is more than one value a lane, the
      // same tree for each; lanes 8 q end with sum q
      const bool h4 = (lane & 16) != 0, h3 = (lane & 8) != 0;
      double x0 = h4 ? acc[2] : acc[0], x1 = h4 ? acc[3] : acc[1];
      x0 += __shfl_xor_sync(0xffffffffu, h4 ? acc[0] : acc[2], 16);
      x1 += __shfl_xor_sync(0xffffffffu, h4 ? acc[1] : acc[3], 16);
      double x = h3 ? x1 : x0;
      x += __shfl_xor_sync(0xffffffffu, h3 ? x0 : x1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      const int q = lane >> 3;
      if ((lane & 7) == 0 && q < cnt) {
        const int to = q == 0 ? col[0] : q == 1 ? col[1] : q == 2 ? col[2] : col[3];
        Cz[(long long)(r0 + u) * ldc + to] = x;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {
constexpr size_t kWsCap = (size_t)512 << 20;    // workspace of a pass; larger products go in several passes
constexpr size_t kSumCap = (size_t)64 << 20;    // of it, for the sums of alpha beta of all splits
constexpr int kMostChunks = 8192;               // of one 64-bit sum

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
int padded(long long K) { return (int)((K + TK - 1) / TK * TK); }
size_t plane_bytes(long long rows, long long K) { return align256((size_t)2 * PLANES * padded(K) * rows); }
size_t row_bytes(long long rows) { return align256((size_t)12 * rows); }
size_t operand_bytes(long long rows, long long K) { return plane_bytes(rows, K) + row_bytes(rows); }

// bytes that a row of B takes: its planes, its norm and exponent, a column of sums
double column_bytes(long long M, long long K) { return 2.0 * PLANES * padded(K) + 12.0 + 4.0 * M; }
size_t pass_bytes(long long m, long long n, long long K) {
  return operand_bytes(m, K) + operand_bytes(n, K) + align256((size_t)4 * m * n);
}
// whether a product without partials is done in a workspace of `cap` bytes: room for 32 rows of A and 16 of B.  It
// depends on K alone, so that the rows and columns of a product may come in any groups.
bool fits(long long K, size_t cap) {
  return pass_bytes(32, 16, K) <= cap && (padded(K) / TK + CHUNK - 1) / CHUNK <= kMostChunks;
}

// How a product goes through a workspace of `cap` bytes: whole, in passes along K (each leaves partials of its own;
// where partials are allowed), or along N, and along M where A and 256 rows of B are more than that.
struct Plan {
  long long kp;      // terms of a pass
  int pieces;        // passes along K
  int mp, np;        // rows and columns of a pass
  int nsplit;        // most splits of a pass
  bool shared;       // B's planes are A's
  size_t bytes;
};
bool make_plan(long long M, long long N, long long K, bool same, int max_split, size_t cap, Plan* p) {
  p->kp = K;
  p->pieces = 1;
  p->mp = (int)M;
  p->np = (int)N;
  p->nsplit = 1;
  p->shared = same;
  if (max_split > 1) {
    const size_t plane = (size_t)4 * M * N;
    p->nsplit = (int)std::max<size_t>(1, std::min<size_t>((size_t)max_split, kSumCap / plane));
    const size_t sums = align256(plane * p->nsplit);
    p->bytes = operand_bytes(M, K) + (same ? 0 : operand_bytes(N, K)) + sums;
    if (p->bytes > cap) {
      const double rows = (double)(M + (same ? 0 : N));
      const double left = (double)cap - (double)sums - 12.0 * rows - 4096.0;
      p->kp = (long long)(left / (2.0 * PLANES * rows)) / 128 * 128;
      if (p->kp < 1024) return false;
      p->pieces = (int)((K + p->kp - 1) / p->kp);
      if (p->pieces > max_split) return false;
      p->nsplit = std::min(p->nsplit, max_split / p->pieces);
      p->bytes = operand_bytes(M, p->kp) + (same ? 0 : operand_bytes(N, p->kp)) + sums;
      if (p->bytes > cap) return false;
    }
    return (padded(p->kp) / TK + CHUNK - 1) / CHUNK <= (long long)kMostChunks * p->nsplit;
  }
  p->bytes = same ? operand_bytes(M, K) + align256((size_t)4 * M * N) : pass_bytes(M, N, K);
  if (p->bytes <= cap) return true;
  p->shared = false;
  auto columns = [&](int mp) {   // of a pass of mp rows
    return (long long)(((double)cap - (double)operand_bytes(mp, K) - 4096.0) / column_bytes(mp, K));
  };
  if (columns(p->mp) < std::min(N, 256LL)) {
    // half of the workspace each: whole tiles of rows if it holds one, else quarters of a tile
    const long long rows = (long long)(0.5 * (double)cap / (2.0 * PLANES * padded(K) + 12.0));
    p->mp = (int)std::min(M, std::max(32LL, rows >= TM ? rows / TM * TM : rows / 32 * 32));
  }
  const long long n = columns(p->mp);
  p->np = (int)std::min(N, n >= 64 ? n / 64 * 64 : n / 16 * 16);
  if (p->np < 1) return false;
  p->bytes = pass_bytes(p->mp, p->np, K);
  return p->bytes <= cap;
}

bool smem_attr_set() {
  static std::atomic<int> done[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (dev >= 0 && dev < kMaxDevices && done[dev].load(std::memory_order_acquire)) return true;
  if (!raise_smem_limit(f64_tc_kernel, SMEM_BYTES)) return false;
  if (dev >= 0 && dev < kMaxDevices) done[dev].store(1, std::memory_order_release);
  return true;
}

int launch_slices(const SliceDesc& a, const SliceDesc& b, long long K, cudaStream_t s) {
  const int kpad = padded(K);
  const int rows = a.rows + b.rows;
  if (rows == 0) return 0;
  if (K <= 2048) {
    int tprl = 2;
    while ((8 << tprl) < kpad) ++tprl;
    const int rpb = 256 >> tprl;
    slice_short_kernel<<<(rows + rpb - 1) / rpb, 256, 0, s>>>(a, b, (int)K, kpad, tprl);
    ++g_launches;
    return 0;
  }
  // q and e of an operand are one array
  if ((a.rows && cudaMemsetAsync(a.q, 0, 12 * (size_t)a.rows, s) != cudaSuccess) ||
      (b.rows && cudaMemsetAsync(b.q, 0, 12 * (size_t)b.rows, s) != cudaSuccess))
    return -1;
  const long long most = (K + 2047) / 2048, fill = (8LL * sm_count() + rows - 1) / rows;
  const dim3 grid((unsigned)rows, (unsigned)std::max(1LL, std::min({most, fill, 65535LL})));
  slice_max_kernel<<<grid, 256, 0, s>>>(a, b, K);
  slice_long_kernel<<<grid, 256, 0, s>>>(a, b, K, kpad);
  g_launches += 2;
  return 0;
}
}  // namespace

size_t f64_tc_bytes(long long M, long long N, long long K, bool same, int max_split, size_t cap) {
  if (M < 1 || N < 1 || K < 1 || M >= (1LL << 31) || N >= (1LL << 31) || K >= (1LL << 31) - TK) return 0;
  cap = std::min(cap, kWsCap);
  if (max_split <= 1 && !fits(K, cap)) return 0;
  Plan p;
  return make_plan(M, N, K, same, max_split, cap, &p) ? p.bytes : 0;
}

double f64_tc_column_bytes(long long M, long long K) { return column_bytes(M, K); }

// Partial products written (at most max_split); 0: not done (the caller takes the FP64 pipe),
// negative: an error
int launch_gemm_nt_f64_tc(const double* A, long long lda, const double* B, long long ldb, double* C, long long ldc,
                          long long split_stride, int M, int N, long long K, int max_split, int upper_only, void* ws,
                          size_t ws_bytes, int* err_flag, cudaStream_t s, size_t cap) {
  const bool same = A == B && lda == ldb && M == N;
  Plan pl;
  if (!ws || !tc_gemm_ready() || !smem_attr_set() ||
      !make_plan(M, N, K, same, max_split, std::min(cap, kWsCap), &pl) || pl.bytes > ws_bytes)
    return 0;
  if (upper_only && (pl.np < N || pl.mp < M)) return 0;
  int used = 0;
  for (int p = 0; p < pl.pieces; ++p) {
    const long long k0 = p * pl.kp, Kp = std::min(pl.kp, K - k0);
    const int kpad = padded(Kp);
    char* w = (char*)ws;
    auto operand = [&](const double* x, long long ld, int rows) {
      SliceDesc d;
      d.x = x + k0;
      d.ld = ld;
      d.rows = rows;
      d.v = (__nv_bfloat16*)w;
      w += plane_bytes(rows, Kp);
      d.q = (unsigned long long*)w;
      d.e = (int*)(d.q + rows);
      w += row_bytes(rows);
      return d;
    };
    const SliceDesc a0 = operand(A, lda, pl.mp), b0 = pl.shared ? a0 : operand(B, ldb, pl.np);
    float* sums = (float*)w;
    for (int m0 = 0; m0 < M; m0 += pl.mp)
      for (int n0 = 0; n0 < N; n0 += pl.np) {
        const int mc = std::min(pl.mp, M - m0), nc = std::min(pl.np, N - n0);
        SliceDesc a = a0, b = b0;
        a.x += (long long)m0 * lda;
        a.rows = mc;
        a.e = (int*)(a.q + mc);
        if (pl.shared) {
          b = a;
        } else {
          b.x += (long long)n0 * ldb;
          b.rows = nc;
          b.e = (int*)(b.q + nc);
        }
        SliceDesc sa = a, sb = b;
        if (n0 > 0) sa.rows = 0;   // the planes of A are there
        if (pl.shared || (m0 > 0 && pl.np >= N)) sb.rows = 0;
        if (launch_slices(sa, sb, Kp, s) != 0) return -1;
        CUtensorMap ma, mb;
        if (make_piece_map(&ma, a.v, mc, kpad, PLANES, TM, TK, false, PLANES) ||
            make_piece_map(&mb, b.v, nc, kpad, PLANES, TN, TK, false, PLANES))
          return -1;
        TcItems it;
        it.M = mc;
        it.N = nc;
        it.mt = (mc + TM - 1) / TM;
        it.nt = (nc + TN - 1) / TN;
        it.upper = upper_only;
        it.ntiles = it.mt * it.nt;
        if (upper_only) {
          it.ntiles = 0;
          for (int t = 0; t < it.mt; ++t) it.ntiles += it.nt - t * TM / TN;
        }
        it.slabs = kpad / TK;
        const int chunks = (it.slabs + CHUNK - 1) / CHUNK;
        // splits: the rounds of the items over the SMs times an item's chunks, the epilogue as two more
        const long long sms = sm_count();
        long long best = -1;
        int ns_best = 1;
        for (int ns = 1; ns <= std::max(1, std::min(pl.nsplit, chunks)); ++ns) {
          const int cps = (chunks + ns - 1) / ns;
          if (cps > kMostChunks) continue;
          const int real = (chunks + cps - 1) / cps;
          const long long cost = ((long long)it.ntiles * real + sms - 1) / sms * (cps + 2);
          if (best < 0 || cost < best) {
            best = cost;
            ns_best = real;
          }
        }
        const int cps = (chunks + ns_best - 1) / ns_best;
        it.nsplit = (chunks + cps - 1) / cps;
        it.per = cps * CHUNK;
        const long long items = (long long)it.ntiles * it.nsplit;
        double* Cp = C + (long long)m0 * ldc + n0 + (long long)used * split_stride;
        f64_tc_kernel<<<(unsigned)std::min(items, sms), NTHREADS, SMEM_BYTES, s>>>(ma, mb, a.e, b.e, Cp, ldc,
                                                                                   split_stride, sums, it, err_flag);
        ++g_launches;
        if (it.nsplit > 1) {
          const long long plane = (long long)mc * nc;
          f64_sum_kernel<<<(unsigned)std::min((plane + 31) / 32, 64 * sms), 256, 0, s>>>(sums, plane, it.nsplit);
          ++g_launches;
        }
        const dim3 grid((nc + FIX_N - 1) / FIX_N, (mc + FIX_M - 1) / FIX_M, it.nsplit);
        f64_fix_kernel<<<grid, 256, 0, s>>>(a.x, lda, b.x, ldb, Cp, ldc, split_stride, mc, nc, Kp,
                                            (long long)it.per * TK, sums, a.q, a.e, b.q, b.e, upper_only);
        ++g_launches;
        if (m0 + mc >= M && n0 + nc >= N) used += it.nsplit;
      }
  }
  if (cudaPeekAtLastError() != cudaSuccess) {
    fprintf(stderr, "hotrg: FP64 product on the tensor cores: launch error (M %d, N %d, K %lld)\n", M, N, K);
    return -1;
  }
  return used;
}

}  // namespace hotrg
