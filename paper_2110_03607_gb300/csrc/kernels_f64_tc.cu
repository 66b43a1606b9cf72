// FP64 products on the tensor cores: C = A . B^T from exact products of digits.
//
// The FP64 pipe of this chip does 2 multiply-adds per clock and SM (1.25 TFLOP/s); its BF16 tensor
// cores do 4096 times as many.  Following Ozaki, Ogita, Oishi and Rump (Numerical Algorithms 59, 2012),
// every row of an operand is written as integers of a common unit 2^(e - 62), 2^e > max |x|, and each
// integer as eight signed digits in base 256 (seven in [-128, 127], the leading one in [-65, 65]):
//   x = sum_a v_a 2^(e - 6 - 8 a).
// A digit is exact in BF16, a product of two is at most 2^14, and the tensor core adds into an FP32
// accumulator without error while every partial sum stays within 2^24.  The products v_a w_b with
// a + b = g <= 7 share one accumulator (they share the weight 2^-8g): at most 8 products times 128
// along K, 2^14 2^3 2^7 = 2^24.  So each chunk of 128 along K gives eight exact integers P_g per
// output; they are added, still exactly, into two 64-bit integers (hi: g = 0 .. 3, lo: g = 4 .. 7),
// and one rounding to FP64 ends the sum.  Left out are the bits of an element below 2^-62 of its
// row's largest and the products with a + b > 7, at most 2^-61 of the two rows' largest and of either
// sign: less than the roundings of an FP64 sum.  Only where the two rows have the same digits, on the
// diagonal of a Gram, do the squares among them add up (v_4^2 of every term: 2e-15 of the sum at
// K = 32,768).  A symmetric product therefore takes a ninth accumulator, a + b = 8, in tiles of 48
// columns; it enters lo rounded to its unit once a chunk.
//
// Layout: tile 128 x 64 of C per CTA, its eight accumulators fill the 512 columns of TMEM.  A ring of
// two stages holds K slabs of 32 (64-byte rows), all eight digits of both operands (96 KB a stage).
// The MMA warp goes through a slab by accumulator g, and waits for the epilogue once per g and chunk,
// so the drain of one accumulator runs under the MMAs of the next.
#include <stdio.h>

#include <algorithm>
#include <atomic>

#include "tcgen05.cuh"

namespace hotrg {

namespace {
constexpr int TM = 128, TK = 32, DIG = 8, STAGES = 2;
constexpr int CHUNK = 4;                        // slabs per exact sum: 128 along K
constexpr int A_DIG = TM * TK * 2;
// the tile width for a number of accumulators: 64 for 8, 48 for 9
__host__ __device__ constexpr int tile_n(int accs) { return 512 / accs / 16 * 16; }
__host__ __device__ constexpr int stage_bytes(int accs) { return DIG * (A_DIG + tile_n(accs) * TK * 2); }
__host__ __device__ constexpr int smem_bytes(int accs) { return 1024 + STAGES * stage_bytes(accs) + 512; }
constexpr int EPI_WARPS = 8, W_PROD = 8, W_MMA = 9, NTHREADS = 320;
constexpr int NON_FINITE = 0x7fffffff;          // a row with an infinity or a NaN
static_assert(smem_bytes(8) <= 227 * 1024, "shared memory of one CTA");
static_assert(tile_n(8) == 64 && tile_n(9) == 48, "tile widths");

struct SliceDesc {
  const double* x;
  long long ld;
  int rows;
  __nv_bfloat16* v;    // digit a of element (r, k) at (a rows + r) kpad + k
  int* e;              // per row: biased exponent of the largest |x|, at least 1
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
  unsigned long long f = sh >= 0 ? m << (sh & 15) : (sh > -64 ? m >> -sh : 0ULL);
  if ((long long)bits < 0) f = 0ULL - f;
  return (f + 0x0080808080808080ULL) ^ 0x8000000000000000ULL;
}

// eight consecutive elements -> one 16-byte store per digit
__device__ __forceinline__ void store_digits(const double (&x)[8], int E, __nv_bfloat16* dst, long long dstride) {
  unsigned lo[8], hi[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned long long d = E == NON_FINITE ? 0x8080808080808080ULL : digits(x[i], E);
    lo[i] = (unsigned)d;
    hi[i] = (unsigned)(d >> 32);
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
// digits in one pass.
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
  for (int o = min(tpr, 32) >> 1; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  if (tpr > 32) {
    const int w = threadIdx.x >> 5, wpr = tpr >> 5;
    if ((threadIdx.x & 31) == 0) wmax[w] = hi;
    __syncthreads();
    for (int q = 0; q < wpr; ++q) hi = max(hi, wmax[(w & ~(wpr - 1)) + q]);
  }
  const int E = row_exponent(hi);
  if (!live) return;
  if (t == 0) d.e[r] = E;
  if (k < kpad) store_digits(x, E, d.v + r * kpad + k, (long long)d.rows * kpad);
}

// Long rows: the exponents first (blocks of a row meet in an atomic maximum; e zeroed before) ...
__global__ void __launch_bounds__(256) slice_max_kernel(SliceDesc A, SliceDesc B, long long K) {
  const bool second = (int)blockIdx.y >= A.rows;
  const SliceDesc& d = second ? B : A;
  const int r = second ? (int)blockIdx.y - A.rows : (int)blockIdx.y;
  const double* x = d.x + r * d.ld;
  int hi = 0;
  for (long long k = ((long long)blockIdx.x * 256 + threadIdx.x) * 8; k < K; k += (long long)gridDim.x * 2048) {
    double v[8];
    load8(x + k, (int)min(8LL, K - k), v);
#pragma unroll
    for (int i = 0; i < 8; ++i) hi = max(hi, high_abs(v[i]));
  }
  for (int o = 16; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  if ((threadIdx.x & 31) == 0) atomicMax(d.e + r, row_exponent(hi));
}
// ... then the digits
__global__ void __launch_bounds__(256) slice_long_kernel(SliceDesc A, SliceDesc B, long long K, int kpad) {
  const bool second = (int)blockIdx.y >= A.rows;
  const SliceDesc& d = second ? B : A;
  const int r = second ? (int)blockIdx.y - A.rows : (int)blockIdx.y;
  const double* x = d.x + r * d.ld;
  const int E = d.e[r];
  __nv_bfloat16* v0 = d.v + (long long)r * kpad;
  for (long long k = ((long long)blockIdx.x * 256 + threadIdx.x) * 8; k < kpad; k += (long long)gridDim.x * 2048) {
    double v[8];
    load8(x + (k < K ? k : 0), (int)max(0LL, min(8LL, K - k)), v);
    store_digits(v, E, v0 + k, (long long)d.rows * kpad);
  }
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
template <int TN>
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

template <int ACCS>
__global__ void __launch_bounds__(NTHREADS, 1)
    f64_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const int* __restrict__ ea, const int* __restrict__ eb, double* __restrict__ C, long long ldc,
                  long long split_stride, TcItems its, int* g_err) {
  constexpr int TN = tile_n(ACCS), B_DIG = TN * TK * 2, STAGE_BYTES = stage_bytes(ACCS);
  extern __shared__ uint8_t smem_raw[];
  volatile int* gerr = g_err;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;      // [ACCS] MMA -> epilogue
  uint64_t* tempty = tfull + ACCS;       // [ACCS] epilogue -> MMA
  uint64_t* drain = tempty + ACCS;
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
      // ---------------- TMA producer: both operands' digits of one K slab per stage
      long long g = 0;
      bool ok = true;
      for (long long i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
        int m0, n0, z, s0, cnt;
        item_of<TN>(its, i, &m0, &n0, &z, &s0, &cnt);
        for (int kb = 0; kb < cnt; ++kb, ++g) {
          const int s = (int)(g % STAGES);
          if (!mbar_wait(empty + s, (uint32_t)((g / STAGES) & 1) ^ 1u, cta_abort, gerr)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + s * STAGE_BYTES;
          mbar_expect_tx(full + s, (uint32_t)STAGE_BYTES);
          tma_load_3d(&tmA, st, full + s, (s0 + kb) * TK, m0, 0);
          tma_load_3d(&tmB, st + DIG * A_DIG, full + s, (s0 + kb) * TK, n0, 0);
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
      long long g = 0, ch = 0;   // slabs and chunks of this CTA so far
      for (long long i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
        int m0, n0, z, s0, cnt;
        item_of<TN>(its, i, &m0, &n0, &z, &s0, &cnt);
        for (int kb = 0; kb < cnt && ok; ++kb, ++g) {
          const int s = (int)(g % STAGES);
          const bool first = kb % CHUNK == 0, last = kb % CHUNK == CHUNK - 1 || kb == cnt - 1;
          if (!mbar_wait(full + s, (uint32_t)(g / STAGES) & 1u, cta_abort, gerr)) {
            ok = false;
            break;
          }
          const uint32_t st = su32(smem + s * STAGE_BYTES);
          const uint64_t a0 = sdesc_sw<TK * 2>(st), b0 = sdesc_sw<TK * 2>(st + DIG * A_DIG);
          for (int acc = 0; acc < ACCS; ++acc) {
            if (first && ch > 0 && !mbar_wait(tempty + acc, (uint32_t)(ch - 1) & 1u, cta_abort, gerr)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t dst = tmem + (uint32_t)(acc * TN);
            const int a_lo = acc < DIG ? 0 : acc - DIG + 1;
            for (int a = a_lo; a < DIG && a <= acc; ++a) {
              const uint64_t da = a0 + (uint64_t)(a * (A_DIG >> 4)), db = b0 + (uint64_t)((acc - a) * (B_DIG >> 4));
#pragma unroll
              for (int kk = 0; kk < TK / 16; ++kk)   // 16 BF16 = 32 bytes inside the swizzled row
                umma_bf16(dst, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                          first && a == a_lo && kk == 0 ? 0u : 1u);
            }
            if (last) umma_commit(tfull + acc);
          }
          if (!ok) break;
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
    bool ok = true;
    long long ch = 0;
    for (long long i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
      int m0, n0, z, s0, cnt;
      item_of<TN>(its, i, &m0, &n0, &z, &s0, &cnt);
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
          if constexpr (EC == 32) {
            tmem_ld_async(lane_base + (uint32_t)(acc * TN), v);
            tmem_wait_ld();
          } else {
            uint32_t v0[16], v1[8];
            tmem_ld_async(lane_base + (uint32_t)(acc * TN), v0);
            tmem_ld_async(lane_base + (uint32_t)(acc * TN + 16), v1);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < EC; ++j) v[j] = j < 16 ? v0[j & 15] : v1[j & 7];
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(tempty + acc)) : "memory");
#pragma unroll
          for (int j = 0; j < EC; ++j) {
            const int p = __float2int_rn(__uint_as_float(v[j]));
            if (acc < 4) hi[j] += (long long)p * (1 << (24 - 8 * (acc & 3)));
            else if (acc < 8) lo[j] += (long long)p * (1 << (24 - 8 * (acc & 3)));
            else lo[j] += (p + 128) >> 8;
          }
        }
      }
      if (!ok || *cta_abort) break;
      const int row = m0 + quarter * 32 + lane, col0 = n0 + part * EC;
      if (row < its.M) {
        const int er = ea[row];
        double* dst = C + (long long)z * split_stride + (long long)row * ldc + col0;
        // x = sum_a v_a 2^(E - 1022 - 6 - 8 a) of each operand; hi counts in units of 2^-24
        const int e0 = er - 2 * 1028 - 24 - 32;
#pragma unroll
        for (int j = 0; j < EC; ++j)
          if (col0 + j < its.N) {
            const int ec = eb[col0 + j];
            dst[j] = er == NON_FINITE || ec == NON_FINITE ? __longlong_as_double(0x7ff8000000000000LL)
                                                          : fixed_to_double(hi[j], lo[j], e0 + ec);
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

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {
constexpr long long kWsCap = 512LL << 20;   // digits of a pass; larger products go in several passes

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
int padded(long long K) { return (int)((K + TK - 1) / TK * TK); }
size_t ws_of(long long rows_a, long long rows_b, long long K) {
  return align256((size_t)16 * padded(K) * rows_a) + align256((size_t)16 * padded(K) * rows_b) +
         align256(4 * (size_t)rows_a) + align256(4 * (size_t)rows_b);
}

bool smem_attr_set() {
  static std::atomic<int> done[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (dev >= 0 && dev < kMaxDevices && done[dev].load(std::memory_order_acquire)) return true;
  if (cudaFuncSetAttribute(f64_tc_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(8)) !=
          cudaSuccess ||
      cudaFuncSetAttribute(f64_tc_kernel<9>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(9)) != cudaSuccess)
    return false;
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
  if (rows > 65535) return -1;
  if ((a.rows && cudaMemsetAsync(a.e, 0, 4 * (size_t)a.rows, s) != cudaSuccess) ||
      (b.rows && cudaMemsetAsync(b.e, 0, 4 * (size_t)b.rows, s) != cudaSuccess))
    return -1;
  const long long most = (K + 2047) / 2048, fill = (8LL * sm_count() + rows - 1) / rows;
  const dim3 grid((unsigned)std::max(1LL, std::min(most, fill)), (unsigned)rows);
  slice_max_kernel<<<grid, 256, 0, s>>>(a, b, K);
  slice_long_kernel<<<grid, 256, 0, s>>>(a, b, K, kpad);
  g_launches += 2;
  return 0;
}
}  // namespace

// Where the digits pay: the FP64 pipe does 0.6e12 multiply-adds a second, so 2^24 of them take 28 us
// there, about as long as the launches and the first tiles of this path.  A Gram over less than 1024
// terms (2D runs: K = chi_c chi_j) stays on the pipe too: at a degenerate cut the kept vector follows the
// rounding of the Gram (ordered 2D phase, chi = 24, step 11: a pair 2.8e-15 lambda_1 apart), and such runs
// go on as they did; it would save 0.1 ms of a Gram of 576 rows.
size_t f64_tc_bytes(long long M, long long N, long long K, bool same, int upper) {
  if (M < 32 || N < 16 || K < 32 || M >= (1LL << 31) || N >= (1LL << 31) || K >= (1LL << 31) - TK) return 0;
  if (same && K < 1024) return 0;
  if ((double)M * (double)N * (double)K * (upper ? 0.5 : 1.0) < 16777216.0) return 0;
  return std::min(ws_of(M, same ? 0 : N, K), (size_t)kWsCap);
}

double f64_tc_column_bytes(long long M, long long K) {
  (void)M;
  return 16.0 * padded(K) + 4.0;
}

// Partial products written (at most max_split); 0: not done (the caller takes the FP64 pipe),
// negative: an error
int launch_gemm_nt_f64_tc(const double* A, long long lda, const double* B, long long ldb, double* C, long long ldc,
                          long long split_stride, int M, int N, long long K, int max_split, int upper_only, void* ws,
                          size_t ws_bytes, int* err_flag, cudaStream_t s) {
  const bool same = A == B && lda == ldb && M == N;
  if (!ws || !tc_gemm_ready() || !smem_attr_set()) return 0;
  // passes along K (more partials) or along N, so that the digits fit the workspace
  long long kp = K;
  int np = N;
  if (ws_of(M, same ? 0 : N, K) > ws_bytes) {
    if (max_split > 1) {
      const double per = 16.0 * (M + (same ? 0 : N));
      kp = (long long)(((double)ws_bytes - 4096.0 - 8.0 * (M + (double)N)) / per) / 128 * 128;
      if (kp < 1024 || (K + kp - 1) / kp > max_split) return 0;
    } else {
      if (same) return 0;
      const double left = (double)ws_bytes - 4096.0 - (16.0 * padded(K) + 4.0) * M;
      const double rows = left / (16.0 * padded(K) + 4.0);
      if (rows < 256.0) return 0;
      np = (int)std::min((double)N, rows) / 64 * 64;
    }
  }
  if (K > 2048 && (long long)M + np > 65535) {
    if (M > 32768) return 0;
    np = std::min(np, 32704);
  }
  const int pieces = (int)((K + kp - 1) / kp);
  const int accs = same ? 9 : 8, TN = tile_n(accs);
  if (np < N && (same || pieces > 1)) return 0;
  int used = 0;
  for (int p = 0; p < pieces; ++p) {
    const long long k0 = p * kp, Kp = std::min(kp, K - k0);
    const int kpad = padded(Kp);
    char* w = (char*)ws;
    SliceDesc a, b;
    a.x = A + k0;
    a.ld = lda;
    a.rows = M;
    a.v = (__nv_bfloat16*)w;
    w += align256((size_t)16 * kpad * M);
    b = a;
    if (!same) {
      b.v = (__nv_bfloat16*)w;
      w += align256((size_t)16 * kpad * np);
    }
    a.e = (int*)w;
    b.e = same ? a.e : (int*)(w + align256(4 * (size_t)M));
    for (int n0 = 0; n0 < N; n0 += np) {
      const int nc = std::min(np, N - n0);
      SliceDesc sa = a, sb = b;
      if (!same) {
        sb.x = B + (long long)n0 * ldb + k0;
        sb.ld = ldb;
      }
      sb.rows = same ? 0 : nc;
      if (n0 > 0) sa.rows = 0;   // the digits of A are there
      if (launch_slices(sa, sb, Kp, s) != 0) return -1;
      CUtensorMap ma, mb;
      if (make_piece_map(&ma, a.v, M, kpad, DIG, TM, TK, false, DIG) ||
          make_piece_map(&mb, b.v, same ? M : nc, kpad, DIG, TN, TK, false, DIG))
        return -1;
      TcItems it;
      it.M = M;
      it.N = nc;
      it.mt = (M + TM - 1) / TM;
      it.nt = (nc + TN - 1) / TN;
      it.upper = upper_only;
      it.ntiles = it.mt * it.nt;
      if (upper_only) {
        it.ntiles = 0;
        for (int t = 0; t < it.mt; ++t) it.ntiles += it.nt - t * TM / TN;
      }
      it.slabs = kpad / TK;
      const int chunks = (it.slabs + CHUNK - 1) / CHUNK;
      if (chunks > 8192 * (long long)std::max(1, max_split / pieces)) return -1;   // 64-bit sums: 2^14 chunks
      // splits: the rounds of the items over the SMs times an item's chunks, the epilogue as two more
      const long long sms = sm_count();
      long long best = -1;
      int ns_best = 1;
      for (int ns = 1; ns <= std::max(1, std::min(max_split / pieces, chunks)); ++ns) {
        const int cps = (chunks + ns - 1) / ns;
        if (cps > 8192) continue;
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
      (same ? f64_tc_kernel<9> : f64_tc_kernel<8>)<<<(unsigned)std::min(items, sms), NTHREADS, smem_bytes(accs), s>>>(
          ma, mb, a.e, b.e, C + n0 + (long long)used * split_stride, ldc, split_stride, it, err_flag);
      ++g_launches;
      if (n0 + nc >= N) used += it.nsplit;
    }
  }
  if (cudaPeekAtLastError() != cudaSuccess) {
    fprintf(stderr, "hotrg: FP64 product on the tensor cores: launch error (M %d, N %d, K %lld)\n", M, N, K);
    return -1;
  }
  return used;
}

}  // namespace hotrg
