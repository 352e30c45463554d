// The plain FP64 sweep (Sec. II-B) with its contraction Z i on the tensor
// cores, as sums of integers: each operand is held as 55-bit fixed point with
// one power-of-two scale per row, cut into seven balanced 8-bit digits stored
// in FP16 (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numerical
// Algorithms 59, 2012).  A product of two digits is an integer of at most
// 2^14 (2^16), so 1024 (256) of them sum exactly in the FP32 accumulator; the epilogue
// adds those sums in 32-bit integers.  The complex product uses three real
// ones (Re, Im and Re + Im, the sums formed as integers, so the scheme's
// cancellations are exact), and the products of digits p and q are kept for
// p + q <= 6.  What the fixed point and the products left out cost is about
// 2^-55 of a row's largest entry times the operand's largest, times the square
// root of n.  Every kept bit is an integer, so a result does not depend on the
// tile, the batch or the order of the sums.
//
// An FP64 sum's rounding goes with the sum of its terms' magnitudes instead,
// so where a row's large entries meet small ones of the operand the fixed
// point would be the less exact.  A 22nd product tells those rows: of the
// leading digits of |Re| + |Im| (8 bits, rounded down), the sum of magnitudes
// in units of the two scales.  Rows where it is below SPLIT_WEAK are formed in
// FP64 by the step kernel, from the matrix and the operand themselves, over
// the unknowns of the row's own part of the network; a row of the plain sweep
// only if the digits' error could show beside the rounding of its voltage.
//
// Why: this GPU does 1.25 TFLOP/s in FP64 and about 1.9 PFLOP/s in FP16; the
// 28 digit products of 6 n^2 operations each are 168 n^2 operations at 1500
// times the rate.
//
// Measured per sweep against the FP64 contraction (k_currents_f64 +
// k_gemm3m_f64 + the stop test): 1000 scenarios of 3069 unknowns 66 -> 1.29 ms
// (contraction 1.03), 4096 of 381 3.5 -> 0.23 ms (0.091).
//
// One sweep is two kernels: k_split_gemm (the 22 partial products of every
// active scenario) and k_split_step (recombination, update, stop test, active
// list and the operand of the next sweep, one block per scenario).
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>

#include "adj_loads.cuh"
#include "loads.cuh"
#include "split.cuh"
#include "tc_ptx.cuh"

namespace zbus {
namespace {

using namespace tc;

constexpr int GEMM_THREADS = 320;      // TMA, MMA and eight epilogue warps
// Least sum of leading digits (unit 2^-14 of the product of the scales) of a
// row that keeps its digit products: 1.5.  Root mean square error of a row over
// that of the FP64 contraction, by this sum (99 and 255 unknowns; loads and
// upstream gradients of one size, one bus of 100 or 10^4 times the others, sizes
// over twelve decades): below 0.25 4 to 10^4, 0.5 to 0.75 1.0 to 2.4, 1 to 1.25
// 1.0 to 1.5, 1.25 to 1.5 1.0 to 1.25, 1.5 to 2 0.8 to 1.15, above 2 at most 0.95
// (0.1 at 32, where most rows of a large feeder are).  With loads of one size the
// rows below are those of the small parts, a few buses behind a line of their own
// at the slack; the gradient of 4096 scenarios of 128 buses takes 5.52 ms without
// them, 5.67 so and 5.93 with the line at 2.
constexpr int SPLIT_WEAK = 3 << 13;
constexpr int EPI_WARPS = 8;
constexpr int TMEM_COLS = 512;         // two accumulators of up to 256 columns
constexpr int ACC_STRIDE = 256;
constexpr unsigned long long SPLIT_DRAIN_NS = 2000000000ull;

#ifdef ZBUS_CHECKED
// checked build: zbus_checked_set_wait lowers the limit of the pipeline's waits
__device__ unsigned long long g_split_wait_ns = WAIT_NS;
__device__ __forceinline__ unsigned long long split_wait_ns() { return g_split_wait_ns; }
#else
__device__ __forceinline__ unsigned long long split_wait_ns() { return WAIT_NS; }
#endif

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(su32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(su32(bar))
      : "memory");
}

__device__ __forceinline__ void st_i8(int32_t* p, const int* v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// ---------------------------------------------------------------------------
// Work of the contraction: one item is the 128 x BN block (mt, nt) of one
// partial product (c, d): component c (Re, Im, Re + Im; 3, the magnitudes, has
// one digit) and digit weight d, the sum over p <= d of X_p Z_{d-p}^T.  Items
// are listed from the longest (d = 6) to the shortest and dealt to the blocks
// back and forth, so every block gets about the same number of k-blocks.
// ---------------------------------------------------------------------------
struct SplitItem {
  int c, d, mt, nt;
};

__device__ __forceinline__ SplitItem split_item(int g, int mtiles, int ntn) {
  const int per = mtiles * ntn;
  const int cls = g / per, t = g % per;
  SplitItem it;
  it.d = cls < 3 * SPLIT_S ? SPLIT_S - 1 - cls / 3 : 0;
  it.c = cls < 3 * SPLIT_S ? cls % 3 : 3;
  it.mt = t / ntn;
  it.nt = t % ntn;
  return it;
}

// k-blocks whose digit products sum exactly (to at most 2^24) in the FP32
// accumulator: digits are at most 128, the first digit of Re + Im and the
// magnitudes 256.
__device__ __forceinline__ int split_chunk(const SplitItem& it) {
  return (it.c < 2 ? 1024 : it.d > 0 ? 512 : 256) / BK;
}

__device__ __forceinline__ int split_deal(int round) {
  const int G = gridDim.x;
  return round * G + ((round & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
}

// ---------------------------------------------------------------------------
// Partial products.  Warp roles: 0 = TMA producer, 1 = TMEM owner and MMA
// issuer, 2..9 = epilogue (warp w reads TMEM lanes 32 (w % 4) .. + 31 of one
// half of the columns).  The accumulator is drained before its sum can pass
// 2^24 (split_chunk) into 32-bit integer registers, the next chunk's MMAs running meanwhile in
// the other accumulator.  Bound by the tensor pipe at large batches: 16384
// scenarios of 3069 unknowns in 14.1 ms, 1.87 PFLOP/s of digit products (0.98
// of the measured cuBLAS rate); a few scenarios read the 415 MB of slices of
// Z once per sweep (0.15 ms).  Every wait is bounded as in k_contract_group, and
// a block that gives up records its code and leaves nothing in flight.
// ---------------------------------------------------------------------------
template <int BN, int STAGES>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
k_split_gemm(SolveCtx* __restrict__ ctx, const __grid_constant__ CUtensorMap tmX,
             const __grid_constant__ CUtensorMap tmZ, int n, int num_kb, int64_t rows) {
  constexpr int A_BYTES = BM * BK * 2;
  constexpr int B_BYTES = BN * BK * 2;
  constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  constexpr int HN = BN / 2;   // columns of one epilogue warp
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_holder = (uint32_t*)(drain + 1);

  const int count = ctx->count;
  const int mtiles = (count + BM - 1) / BM;
  const int ntn = (n + BN - 1) / BN;
  const int total = SPLIT_PLANES * mtiles * ntn;
  if ((int)blockIdx.x >= total) return;   // whole block, before any barrier
  const int rounds = (total + gridDim.x - 1) / gridDim.x;
  const unsigned long long wait_ns = split_wait_ns();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int u = 0; u < 2; ++u) {
      mbar_init(&tfull[u], 1);
      mbar_init(&tempty[u], EPI_WARPS);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_holder)),
                 "r"((uint32_t)TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == 0) {
    if (lane == 0) {
      uint32_t kc = 0;   // stage fills issued
      bool ok = true;
      for (int r = 0; r < rounds && ok; ++r) {
        const int g = split_deal(r);
        if (g >= total) continue;
        const SplitItem it = split_item(g, mtiles, ntn);
        // digit q of Z ascending in every item, so items of other weights
        // running at the same time read the same slices of Z
        for (int q = 0; q <= it.d && ok; ++q)
          for (int kb = 0; kb < num_kb; ++kb) {
            const int s = kc % STAGES;
            const uint32_t round = kc / STAGES;
            if (!mbar_wait(&empty[s], (round & 1) ^ 1, wait_ns)) {
              atomicCAS(&ctx->err, 0, 111);
              ok = false;
              break;
            }
            uint8_t* st = smem + s * STAGE_BYTES;
            mbar_expect_tx(&full[s], STAGE_BYTES);
            tma_load_3d(st, &tmX, &full[s], kb * BK, it.mt * BM, it.c * SPLIT_S + it.d - q);
            tma_load_3d(st + A_BYTES, &tmZ, &full[s], kb * BK, it.nt * BN,
                        it.c * SPLIT_S + q);
            ++kc;
          }
      }
      // drain: the last fill of every stage has landed
      const uint32_t first = kc > (uint32_t)STAGES ? kc - STAGES : 0u;
      for (uint32_t j = first; j < kc; ++j)
        if (!mbar_wait(&full[j % STAGES], (j / STAGES) & 1, SPLIT_DRAIN_NS)) {
          atomicCAS(&ctx->err, 0, 115);
          break;
        }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // kind::f16 instruction descriptor: D f32, A and B f16, both K-major
      const uint32_t idesc =
          (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      uint32_t kc = 0, ch = 0;   // stages and accumulator chunks used
      bool ok = true, issued = false;
      for (int r = 0; r < rounds && ok; ++r) {
        const int g = split_deal(r);
        if (g >= total) continue;
        const SplitItem it = split_item(g, mtiles, ntn);
        const int blocks = (it.d + 1) * num_kb, chunk = split_chunk(it);
        for (int b0 = 0; b0 < blocks && ok; b0 += chunk, ++ch) {
          const int buf = ch & 1;
          if (!mbar_wait(&tempty[buf], ((ch >> 1) & 1) ^ 1, wait_ns)) {
            atomicCAS(&ctx->err, 0, 114);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(buf * ACC_STRIDE);
          const int b1 = min(blocks, b0 + chunk);
          for (int b = b0; b < b1; ++b, ++kc) {
            const int s = kc % STAGES;
            if (!mbar_wait(&full[s], (kc / STAGES) & 1, wait_ns)) {
              atomicCAS(&ctx->err, 0, 112);
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t a0 = su32(smem + s * STAGE_BYTES);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              umma_f16(d, sw128_desc(a0 + kk * 32), sw128_desc(a0 + A_BYTES + kk * 32), idesc,
                       (b != b0 || kk != 0) ? 1u : 0u);
            issued = true;
            umma_commit(&empty[s]);
          }
          if (ok) umma_commit(&tfull[buf]);
        }
      }
      // drain: every MMA this thread issued has completed before the tensor
      // memory is freed
      if (issued) {
        umma_commit(drain);
        if (!mbar_wait(drain, 0, SPLIT_DRAIN_NS)) atomicCAS(&ctx->err, 0, 116);
      }
    }
  } else {
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int ld = (n + 7) & ~7;
    int32_t* const D = ctx->D;
    uint32_t ch = 0;
    bool ok = true;
    for (int r = 0; r < rounds && ok; ++r) {
      const int g = split_deal(r);
      if (g >= total) continue;
      const SplitItem it = split_item(g, mtiles, ntn);
      const int blocks = (it.d + 1) * num_kb, chunk = split_chunk(it);
      int acc[HN];
#pragma unroll
      for (int t = 0; t < HN; ++t) acc[t] = 0;
      for (int b0 = 0; b0 < blocks; b0 += chunk, ++ch) {
        const int buf = ch & 1;
        // the warp goes on, or gives up, as one: its loads need every lane
        ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], (ch >> 1) & 1, wait_ns));
        tc_fence_after();
        if (!ok) {
          if (lane == 0) atomicCAS(&ctx->err, 0, 113);
          break;
        }
        const uint32_t ta =
            tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * ACC_STRIDE + half * HN);
#pragma unroll
        for (int c = 0; c < HN / 32; ++c) {
          float v[32];
          tmem_ld32(ta + (uint32_t)(c * 32), v);
          if (c == HN / 32 - 1) {
            // the accumulator is in registers now: hand it back
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
          }
#pragma unroll
          for (int t = 0; t < 32; ++t) acc[c * 32 + t] += __float2int_ru(v[t]);
        }
      }
      const int64_t row = (int64_t)it.mt * BM + q * 32 + lane;
      if (ok && row < count) {
        const int col0 = it.nt * BN + half * HN;
        int32_t* dst = D + ((int64_t)(it.c * SPLIT_S + it.d) * rows + row) * ld + col0;
#pragma unroll
        for (int t = 0; t < HN; t += 8)
          if (col0 + t < ld) st_i8(dst + t, acc + t);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------
// Fixed point and digits.
// ---------------------------------------------------------------------------

// Exponent e of a row whose largest magnitude has the bit pattern `top`:
// every entry is below 2^e.  Clamped so that the scales stay finite (entries
// below 2^-900 2^-55 become zero).
__device__ __forceinline__ int row_exponent(unsigned long long top) {
  return max(-900, (int)(top >> 52) - 1022);
}

// round(x 2^(55 - e)) with integer instructions (the conversion instruction
// runs on the FP64 units); |x| < 2^e.
__device__ __forceinline__ long long fixed_point(double x, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((u >> 52) & 0x7FF);
  unsigned long long m = u & 0xFFFFFFFFFFFFFull;
  m = ex ? m | (1ull << 52) : m;
  // x = m 2^(max(ex, 1) - 1075)
  const int sh = max(ex, 1) - 1075 + SPLIT_BITS - e;   // at most 2
  if (sh >= 0) {
    m <<= sh;
  } else if (sh < -55) {
    m = 0ull;
  } else {
    m = (m + (1ull << (-sh - 1))) >> -sh;
  }
  return (u >> 63) ? -(long long)m : (long long)m;
}

// Slices of one row of n complex values, by all threads of the block: digit p
// of component c of value(j) goes to plane c * 7 + p of out, `plane` halves
// apart, the leading digits of |Re| + |Im| to plane 21; a thread takes four
// columns of one component at a time.  A magnitude below one digit is 2^-12, so
// that a sum of products is zero (rounded up, k_split_gemm) only where each is.
template <typename Load>
__device__ __forceinline__ void write_slices(Load value, int n, int K_pad, int e, __half* out,
                                             int64_t plane) {
  const __half2 bias = __floats2half2_rn(1280.f, 1280.f);
  const int groups = K_pad / 4;
  for (int u = threadIdx.x; u < 3 * groups; u += blockDim.x) {
    const int c = u / groups, g = u - c * groups;
    long long y[4];
    uint32_t mag[2] = {0x65006500u, 0x65006500u};   // 1280 + the magnitude's digit
    uint32_t tiny[2] = {0u, 0u};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = g * 4 + i;
      const double2 v = j < n ? value(j) : make_double2(0.0, 0.0);
      y[i] = fixed_point(c == 1 ? v.y : v.x, e);
      if (c == 2) {
        const long long im = fixed_point(v.y, e);
        const uint32_t d = (uint32_t)((llabs(y[i]) + llabs(im)) >> (SPLIT_BITS - 7));
        mag[i >> 1] += d << (16 * (i & 1));
        if (d == 0 && has_load(v)) tiny[i >> 1] |= 0x0C00u << (16 * (i & 1));   // 2^-12
        y[i] += im;
      }
    }
    __half* dst = out + (int64_t)c * SPLIT_S * plane + g * 4;
    if (c == 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const __half2 hv = __hsub2(*reinterpret_cast<const __half2*>(&mag[i]), bias);
        mag[i] = *reinterpret_cast<const uint32_t*>(&hv) | tiny[i];   // of a half that is 0
      }
      *reinterpret_cast<uint2*>(dst + SPLIT_S * plane) = make_uint2(mag[0], mag[1]);
    }
#pragma unroll
    for (int p = SPLIT_S - 1; p >= 0; --p) {
      uint32_t w[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint32_t pair = 0x64006400u;   // the halves 1024 + (digit + 256), minus 1280 below
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          long long& v = y[2 * i + h];
          int d;
          if (p > 0) {
            d = (int)(((uint32_t)v + 128u) & 255u) - 128;
            v = (v - d) >> 8;
          } else {
            d = (int)v;   // at most 256 in magnitude
          }
          pair += (uint32_t)(d + 256) << (16 * h);
        }
        const __half2 hv = __hsub2(*reinterpret_cast<const __half2*>(&pair), bias);
        w[i] = *reinterpret_cast<const uint32_t*>(&hv);
      }
      *reinterpret_cast<uint2*>(dst + p * plane) = make_uint2(w[0], w[1]);
    }
  }
}

__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}

// Maximum over the block (valid in every thread); red: one word per warp.
__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long x,
                                                            unsigned long long* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = max_u64(x, __shfl_xor_sync(0xffffffffu, x, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  x = red[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) x = max_u64(x, red[w]);
  return x;
}

// Matrix rows (one block each): slices and scale 2^(e - 31) of row i.
__global__ void __launch_bounds__(256)
k_split_pack(const double* __restrict__ Zr, const double* __restrict__ Zi, int n, int n_pad,
             int K_pad, __half* __restrict__ out, double* __restrict__ zs) {
  __shared__ unsigned long long red[8];
  const int i = blockIdx.x;
  const double* zr = Zr + (int64_t)i * n_pad;
  const double* zi = Zi + (int64_t)i * n_pad;
  unsigned long long top = 0ull;
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    top = max_u64(top, max_u64(abs_bits(zr[j]), abs_bits(zi[j])));
  top = block_max_u64(top, red);
  const int e = row_exponent(top);
  write_slices([&](int j) { return make_double2(zr[j], zi[j]); }, n, K_pad, e,
               out + (int64_t)i * K_pad, (int64_t)n * K_pad);
  if (threadIdx.x == 0) zs[i] = ldexp(1.0, e - 31);
}

// ---------------------------------------------------------------------------
// Update, stop test and next operand, one block per active scenario.
//   v_i <- w_i + 2^(ez_i + ex_b - 62) sum_d D_d 2^(8 (6 - d))
// with the three components combined as integers (T1 - T2, T3 - T1 - T2) in
// two 64-bit words of four and three digit weights, exact until one rounding.
// The block then holds the scenario's new voltages, so it decides the stop
// and, if the scenario goes on, takes a slot of the next sweep and writes the
// slices of i(v) (or of conj(lambda)) there.  The slot order may differ
// between runs; no result depends on it.
//
// Bound by the FP64 pipe (about 34 operations an unknown at two a clock and
// SM: 91 us for 4096 scenarios of 381 unknowns; 75 % busy) and by the
// latencies between the block's barriers: 136 us there, 203 before the
// voltages had a thread per unknown and the slices one per four columns, 156
// before the tests for absent loads left the FP64 pipe.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double exact_double(long long x) {   // |x| < 2^51
  return __longlong_as_double(x + 0x4338000000000000ll) - 6755399441055744.0;
}

// hi 2^24 + lo, rounded once: hi's low 24 bits join lo, so both conversions
// are exact for every size the path takes.
__device__ __forceinline__ double recombine(long long hi, long long lo) {
  return fma(exact_double(hi >> 24), 0x1p48, exact_double(((hi & 0xFFFFFFll) << 24) + lo));
}

template <bool ADJ>
__device__ __forceinline__ void operand_of_bus(const SolveCtx& c, int b, int n, int j0, int m,
                                               double inv_s, const double2 (&v)[3],
                                               double2 (&x)[3]) {
  const int64_t e = (int64_t)b * n + j0;
  double2 sw[3], sd[3];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    sw[p] = (c.S_wye && p < m) ? c.S_wye[e + p] : make_double2(0.0, 0.0);
    sd[p] = (c.S_del && p < m) ? c.S_del[e + p] : make_double2(0.0, 0.0);
  }
  if (!ADJ) {
    bus_injection_one(v, sw, sd, m, x);
  } else {
    double2 vf[3], g[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      vf[p] = p < m ? c.Vf[e + p] : make_double2(1.0, 0.0);
      g[p] = p < m ? c.G[e + p] : make_double2(0.0, 0.0);
    }
    adjoint_rhs(vf, v, g, inv_s, sw, sd, m, x);
  }
#pragma unroll
  for (int p = 0; p < 3; ++p)
    if (p >= m) x[p] = make_double2(0.0, 0.0);
}

// The matrix in FP64 and its parts (SplitOps).
struct SplitRows {
  const double* Zr;
  const double* Zi;
  const int2* part;
  const int32_t* part_col;
  int n_pad;
  __device__ int size(int j) const {   // unknowns of j's part
    const int2 r = __ldg(part + j);
    return r.y - r.x;
  }
};

// The block's weak rows (list, cnt of them) in FP64, over the unknowns of their
// parts, into out[row]; x: the operand.  Four rows a warp, eight lanes a row:
// most are of parts of a few buses.  Columns without current cost no
// arithmetic.
__device__ __noinline__ void weak_rows(const uint16_t* list, int cnt, int n, const SplitRows& m,
                                       const double2* x, double2* out) {
  const int lane = threadIdx.x & 31;
  for (int r0 = (threadIdx.x >> 5) * 4; r0 < cnt; r0 += blockDim.x >> 3) {
    const int r = r0 + (lane >> 3);
    const int row = r < cnt ? list[r] : -1;
    double2 a = make_double2(0.0, 0.0);
    if (row >= 0) {
      const int2 cols = __ldg(m.part + row);
      const double* zr = m.Zr + (int64_t)row * m.n_pad;
      const double* zi = m.Zi + (int64_t)row * m.n_pad;
#pragma unroll 4
      for (int t = cols.x + (lane & 7); t < cols.y; t += 8) {
        const int k = __ldg(m.part_col + t);
        if (!ZB_IN(k, n, 0x602u)) continue;
        const double2 xk = x[k];
        if (has_load(xk)) a = cfma(make_double2(__ldg(zr + k), __ldg(zi + k)), xk, a);
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    }
    if (row >= 0 && (lane & 7) == 0) out[row] = a;
  }
}

// Whether the digits' error in a row of scale s with m terms, some 2^-55.6 sqrt(m)
// of 2^62 s, is within 2^-57 of the larger part of its new voltage, whose own rounding is
// some 2^-54.8 of it: by the exponents.
__device__ __forceinline__ bool beside_voltage(double s, double vx, double vy, int m) {
  const int es = __double2hiint(s) >> 20;
  const int ev = max(__double2hiint(vx) & 0x7FFFFFFF, __double2hiint(vy) & 0x7FFFFFFF) >> 20;
  return es <= ev - 64 - (33 - __clz(m)) / 2;
}

// Blocks of 256 threads an SM holds: at 2 the FP64 pipe waits (176 us a sweep
// of 4096 scenarios of 381 unknowns against 156, with comparisons on it), at 4
// the spills cost a few
// scenarios (92 us a sweep of 16 of 3069 unknowns against 76).
constexpr int STEP_MIN = 3;

template <bool ADJ, bool FIRST>
__global__ void __launch_bounds__(256, STEP_MIN)
k_split_step(SolveCtx* __restrict__ ctx, const double* __restrict__ zs, SplitRows m64,
             const double2* __restrict__ w, int n, int K_pad, int64_t rows,
             cudaGraphConditionalHandle h, int use_handle) {
  extern __shared__ double2 op[];   // [n] operand of the next sweep
  uint16_t* const weak = reinterpret_cast<uint16_t*>(op + n);   // [n] rows for FP64
  __shared__ unsigned long long red[8];
  __shared__ double sred[8];
  __shared__ int s_keep, s_slot, s_weak;
  const SolveCtx& c = *ctx;
  const int tid = threadIdx.x;
  if (tid == 0) s_weak = 0;
  __syncthreads();
  const int ld = (n + 7) & ~7;
  const int nb = (n + 2) / 3;
  const int par = c.iter & 1;
  const int32_t* const list = par ? c.list2 : c.list;
  int32_t* const list_out = FIRST ? nullptr : (par ? c.list : c.list2);
  const double* const xs = c.xs + (int64_t)par * rows;
  double* const xs_out = c.xs + (int64_t)(FIRST ? par : par ^ 1) * rows;
  const int it = c.iter + 1;
  const bool summag = c.rule == ZBUS_CONV_SUMMAG;
  const int count = c.count;
  for (int slot = blockIdx.x; slot < count; slot += gridDim.x) {
    const int b = list[slot];
    const bool in = ZB_IN(b, c.B, 0x601u);
    int out_slot = slot;
    double2* const V = c.V + (int64_t)(in ? b : 0) * n;
    double2* const xop = c.xop + (int64_t)(in ? b : 0) * n;
    unsigned long long top = 0ull;       // largest |Re|, |Im| of the operand
    unsigned long long st2 = 0ull;       // largest squared step, bit pattern
    unsigned long long sth = 0ull;       // largest step whose square leaves the range
    double dsum = 0.0;
    const double xb = FIRST ? 0.0 : xs[slot];
    const double inv_s = ADJ ? 1.0 / c.gscale[in ? b : 0] : 0.0;
    // the new voltage, step and magnitudes of unknown j: w_j + s (re, im)
    const auto update = [&](int j, double re, double im, double s, double2 vo, double2 wj) {
      const double2 v = make_double2(fma(re, s, wj.x), fma(im, s, wj.y));
      V[j] = v;
      op[j] = v;
      const double dx = v.x - vo.x, dy = v.y - vo.y;
      const unsigned long long qb = abs_bits(fma(dx, dx, dy * dy));
      if ((unsigned)(qb >> 52) - 128u < 1792u) {   // far inside the range of squares
        st2 = max_u64(st2, qb);
      } else if ((abs_bits(dx) | abs_bits(dy)) != 0ull) {
        const unsigned long long hb = abs_bits(hypot(dx, dy));
        sth = max_u64(sth, hb > 0x7FF0000000000000ull ? 0x7FF0000000000000ull : hb);
      }
      if (summag) dsum += hypot(v.x, v.y) - hypot(vo.x, vo.y);
    };
    unsigned long long mine = 0ull;      // this thread's weak rows, a bit an iteration
    // voltages, a thread per unknown
    if (in)
      for (int j = tid, i = 0; j < n; j += blockDim.x, ++i) {
        if (FIRST) {
          op[j] = V[j];
          continue;
        }
        const int32_t* D = c.D + (int64_t)slot * ld + j;
        const int64_t plane = rows * ld;
        int32_t t[3][SPLIT_S];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
          for (int d = 0; d < SPLIT_S; ++d) t[q][d] = D[(q * SPLIT_S + d) * plane];
        const int mag = D[3 * SPLIT_S * plane];
        const double2 vo = V[j];
        const double2 wj = ADJ ? make_double2(0.0, 0.0) : w[j];
        const double s = zs[j] * xb;
        long long hi[3], lo[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          hi[q] = ((long long)t[q][0] << 24) + ((long long)t[q][1] << 16) +
                  ((long long)t[q][2] << 8) + t[q][3];
          lo[q] = ((long long)t[q][4] << 16) + ((long long)t[q][5] << 8) + t[q][6];
        }
        const double re = recombine(hi[0] - hi[1], lo[0] - lo[1]);
        const double im = recombine(hi[2] - hi[0] - hi[1], lo[2] - lo[0] - lo[1]);
        // a sum of zero is exact; a scale that is not a number goes to every row
        if (mag > 0 && mag < SPLIT_WEAK && xb > 0.0 &&
            (ADJ || !beside_voltage(s, fma(re, s, wj.x), fma(im, s, wj.y), m64.size(j)))) {
          mine |= 1ull << i;
          weak[atomicAdd(&s_weak, 1)] = (uint16_t)j;
        } else {
          update(j, re, im, s, vo, wj);
        }
      }
    if (!FIRST) {
      __syncthreads();
      const int cnt = s_weak;
      if (cnt > 0) {
        weak_rows(weak, cnt, n, m64, xop, op);
        __syncthreads();
        for (int j = tid; mine; j += blockDim.x, mine >>= 1)
          if (mine & 1ull) {
            const double2 d = op[j];
            update(j, d.x, d.y, 1.0, V[j], ADJ ? make_double2(0.0, 0.0) : w[j]);
          }
        if (tid == 0) s_weak = 0;
      }
      st2 = block_max_u64(st2, red);
      sth = block_max_u64(sth, red);
      if (summag) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
        if ((tid & 31) == 0) sred[tid >> 5] = dsum;
        __syncthreads();
      }
      if (tid == 0) {
        double delta = fmax(sqrt(__longlong_as_double((long long)st2)),
                            __longlong_as_double((long long)sth));
        if (summag) {
          double u = 0.0;
          for (int q = 0; q < (int)(blockDim.x >> 5); ++q) u += sred[q];
          delta = fabs(u);
        }
        int keep = 0;
        if (in) {
          c.iters[b] = it;
          if (!isfinite(delta) || c.err != 0) {
            c.conv[b] = 0;
          } else if (delta <= c.tol) {
            c.conv[b] = 1;
          } else if (it < c.max_iter) {
            keep = 1;
          }
        }
        s_keep = keep;
        if (keep) {
          const int o = atomicAdd(&ctx->next, 1);
          list_out[o] = b;
          s_slot = o;
        }
      }
      __syncthreads();
      if (!s_keep) {
        __syncthreads();
        continue;
      }
      out_slot = s_slot;
    } else {
      __syncthreads();
    }
    // operand in their place, a thread per bus
    if (in)
      for (int k = tid; k < nb; k += blockDim.x) {
        const int j0 = 3 * k, m = min(3, n - j0);
        double2 v[3], x[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) v[p] = p < m ? op[j0 + p] : make_double2(1.0, 0.0);
        operand_of_bus<ADJ>(c, b, n, j0, m, inv_s, v, x);
#pragma unroll
        for (int p = 0; p < 3; ++p)
          if (p < m) {
            op[j0 + p] = x[p];
            top = max_u64(top, max_u64(abs_bits(x[p].x), abs_bits(x[p].y)));
          }
      }
    top = block_max_u64(top, red);
    // a value that is not finite: the scale carries it to every output
    const bool bad = top >= 0x7FF0000000000000ull;
    const int e = bad ? 0 : row_exponent(top);
    __half* out = reinterpret_cast<__half*>(c.X) + (int64_t)out_slot * K_pad;
    const int64_t plane = rows * K_pad;
    if (in)
      for (int j = tid; j < n; j += blockDim.x) xop[j] = op[j];
    if (bad) {
      write_slices([&](int) { return make_double2(0.0, 0.0); }, n, K_pad, 0, out, plane);
    } else {
      write_slices([&](int j) { return op[j]; }, n, K_pad, e, out, plane);
    }
    if (tid == 0)
      xs_out[out_slot] = bad    ? __longlong_as_double(0x7FF8000000000000ll)
                         : top ? ldexp(1.0, e - 31)
                               : 0.0;
    __syncthreads();
  }
  if (FIRST) return;
  // the last block closes the sweep
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(&ctx->done, 1) == (int)gridDim.x - 1) {
      __threadfence();
      const int left = atomicAdd(&ctx->next, 0);
      if (c.hist && it - 1 < c.hist_n) c.hist[it - 1] = count;
      ctx->count = left;
      ctx->iter = it;
      ctx->next = 0;
      ctx->done = 0;
      if (use_handle) cudaGraphSetConditional(h, left > 0 ? 1u : 0u);
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

// Planes [22][rows][K_pad] of FP16 as a 3D tensor, boxes of 64 x box_rows;
// rows past the end read as zero.
zbus_status make_map(CUtensorMap* map, const void* base, int K_pad, int64_t rows, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return fail(ZBUS_ERR_UNSUPPORTED, "cuTensorMapEncodeTiled is not available");
  cuuint64_t dims[3] = {(cuuint64_t)K_pad, (cuuint64_t)rows, (cuuint64_t)SPLIT_PLANES};
  cuuint64_t strides[2] = {(cuuint64_t)K_pad * 2, (cuuint64_t)K_pad * 2 * (cuuint64_t)rows};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides,
                  box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return fail(ZBUS_ERR_CUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
  return ZBUS_OK;
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

int num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      sms = 0;
  }
  return sms ? sms : 148;
}

constexpr int STAGES_256 = 4, STAGES_192 = 5;
template <int BN, int STAGES>
constexpr size_t gemm_smem() {
  return (size_t)STAGES * (BM + BN) * BK * 2 + 1024 + (2 * STAGES + 5) * 8 + 16;
}

template <int BN, int STAGES>
zbus_status launch_gemm(SolveCtx* ctx, const SplitScratch& s, const SplitOps& ops, int n,
                        int64_t batch, cudaStream_t st) {
  constexpr size_t smem = gemm_smem<BN, STAGES>();
  ZB_CUDA(cudaFuncSetAttribute(k_split_gemm<BN, STAGES>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int64_t items = (int64_t)SPLIT_PLANES * ((batch + BM - 1) / BM) * ((n + BN - 1) / BN);
  const int grid = (int)std::min<int64_t>(items, num_sms());
  k_split_gemm<BN, STAGES><<<grid, GEMM_THREADS, smem, st>>>(ctx, s.map, ops.map, n,
                                                             split_kpad(n) / BK, s.rows);
  return ZBUS_OK;
}

// Operand and list of a block: 16 and 2 bytes an unknown.
size_t step_smem(int n) { return (size_t)n * (sizeof(double2) + sizeof(uint16_t)); }

int step_threads(int n) { return n <= 3 * 160 ? 128 : 256; }

int step_grid(int64_t batch) {
  return (int)std::min<int64_t>(batch, (int64_t)num_sms() * 16);
}

}  // namespace

size_t split_scratch_bytes(int n, int64_t rows) {
  return a256((size_t)SPLIT_PLANES * rows * split_kpad(n) * 2) +
         a256((size_t)SPLIT_PLANES * rows * split_ld(n) * 4) +
         a256((size_t)rows * n * sizeof(double2)) + a256((size_t)rows * 2 * 8) +
         a256((size_t)rows * 4);
}

zbus_status split_scratch_bind(SplitScratch* s, void* base, int n, int64_t rows) {
  char* p = (char*)base;
  s->rows = rows;
  s->X = p;
  p += a256((size_t)SPLIT_PLANES * rows * split_kpad(n) * 2);
  s->D = (int32_t*)p;
  p += a256((size_t)SPLIT_PLANES * rows * split_ld(n) * 4);
  s->xop = (double2*)p;
  p += a256((size_t)rows * n * sizeof(double2));
  s->xs = (double*)p;
  p += a256((size_t)rows * 2 * 8);
  s->list2 = (int32_t*)p;
  return make_map(&s->map, s->X, split_kpad(n), rows, BM);
}

zbus_status split_parts(zbus_network net, const std::vector<int32_t>& ptr,
                        const std::vector<int32_t>& col, cudaStream_t st) {
  const int n = net->n;
  std::vector<int32_t> root(n);
  for (int i = 0; i < n; ++i) root[i] = i;
  auto find = [&](int i) {
    while (root[i] != i) i = root[i] = root[root[i]];
    return i;
  };
  for (int i = 0; i < n; ++i)
    for (int t = ptr[i]; t < ptr[i + 1]; ++t) {
      const int a = find(i), b = find(col[t]);
      root[std::max(a, b)] = std::min(a, b);
    }
  std::vector<int32_t> order(n);
  for (int i = 0; i < n; ++i) {
    root[i] = find(i);
    order[i] = i;
  }
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return root[a] < root[b]; });
  std::vector<int2> range(n);
  for (int i = 0, e = 0; i < n; i = e) {
    for (e = i; e < n && root[order[e]] == root[order[i]]; ++e) {
    }
    for (int t = i; t < e; ++t) range[order[t]] = make_int2(i, e);
  }
  ZB_CUDA(cudaMalloc((void**)&net->part, (size_t)n * sizeof(int2)));
  ZB_CUDA(cudaMalloc((void**)&net->part_col, (size_t)n * sizeof(int32_t)));
  ZB_CUDA(cudaMemcpyAsync(net->part, range.data(), (size_t)n * sizeof(int2),
                          cudaMemcpyHostToDevice, st));
  ZB_CUDA(cudaMemcpyAsync(net->part_col, order.data(), (size_t)n * sizeof(int32_t),
                          cudaMemcpyHostToDevice, st));
  ZB_CUDA(cudaStreamSynchronize(st));
  return ZBUS_OK;
}

namespace {

// One value for every size, so that calls of several host threads cannot lower
// each other's.
template <bool ADJ, bool FIRST>
cudaError_t allow_step_smem() {
  return cudaFuncSetAttribute(k_split_step<ADJ, FIRST>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)step_smem(SPLIT_MAX_NPAD));
}

}  // namespace

zbus_status split_pack(SplitOps* ops, const double* Zr, const double* Zi, int n, int n_pad,
                       const int2* part, const int32_t* part_col, cudaStream_t st) {
  if (ops->Z) return ZBUS_OK;
  ops->Zr = Zr;
  ops->Zi = Zi;
  ops->n_pad = n_pad;
  ops->part = part;
  ops->part_col = part_col;
  ZB_CUDA((allow_step_smem<false, true>()));
  ZB_CUDA((allow_step_smem<false, false>()));
  ZB_CUDA((allow_step_smem<true, true>()));
  ZB_CUDA((allow_step_smem<true, false>()));
  const int K = split_kpad(n);
  // N-tile: 192 or 256 outputs, whichever leaves less of the last tile idle
  ops->BN = round_up(n, 192) < round_up(n, 256) ? 192 : 256;
  zbus_status s = ZBUS_OK;
  cudaError_t ce;
  if ((ce = cudaMalloc(&ops->Z, (size_t)SPLIT_PLANES * n * K * 2)) != cudaSuccess ||
      (ce = cudaMalloc((void**)&ops->zs, (size_t)n * sizeof(double))) != cudaSuccess) {
    s = cuda_fail(ce, "cudaMalloc(slices of Z)", __FILE__, __LINE__);
  } else {
    k_split_pack<<<n, 256, 0, st>>>(Zr, Zi, n, n_pad, K, (__half*)ops->Z, ops->zs);
    if ((ce = cudaGetLastError()) != cudaSuccess ||
        (ce = cudaStreamSynchronize(st)) != cudaSuccess)
      s = cuda_fail(ce, "slices of Z", __FILE__, __LINE__);
    else
      s = make_map(&ops->map, ops->Z, K, n, ops->BN);
  }
  if (s != ZBUS_OK) split_release(ops);
  return s;
}

void split_release(SplitOps* ops) {
  cudaFree(ops->Z);
  cudaFree(ops->zs);
  ops->Z = nullptr;
  ops->zs = nullptr;
}

void split_fill_ctx(SolveCtx* h, const SplitScratch& s) {
  h->X = s.X;
  h->D = s.D;
  h->xs = s.xs;
  h->xop = s.xop;
  h->list2 = s.list2;
  h->next = 0;
  h->done = 0;
}

zbus_status launch_split_gemm(SolveCtx* ctx, const SplitScratch& s, const SplitOps& ops, int n,
                              int64_t batch, cudaStream_t st) {
  return ops.BN == 192 ? launch_gemm<192, STAGES_192>(ctx, s, ops, n, batch, st)
                       : launch_gemm<256, STAGES_256>(ctx, s, ops, n, batch, st);
}

namespace {

template <bool ADJ, bool FIRST>
void launch_step(SolveCtx* ctx, const SplitOps& ops, const double2* w, int n, int64_t batch,
                 int64_t rows, cudaGraphConditionalHandle h, bool use_handle, cudaStream_t st) {
  const SplitRows m64 = {ops.Zr, ops.Zi, ops.part, ops.part_col, ops.n_pad};
  k_split_step<ADJ, FIRST><<<step_grid(batch), step_threads(n), step_smem(n), st>>>(
      ctx, ops.zs, m64, w, n, split_kpad(n), rows, h, use_handle ? 1 : 0);
}

}  // namespace

void launch_split_first(SolveCtx* ctx, int n, int64_t batch, int64_t rows, bool adjoint,
                        cudaStream_t st) {
  if (adjoint)
    launch_step<true, true>(ctx, SplitOps(), nullptr, n, batch, rows, 0, false, st);
  else
    launch_step<false, true>(ctx, SplitOps(), nullptr, n, batch, rows, 0, false, st);
}

void launch_split_step(SolveCtx* ctx, const SplitOps& ops, const double2* w, int n, int64_t batch,
                       int64_t rows, bool adjoint, cudaGraphConditionalHandle h, bool use_handle,
                       cudaStream_t st) {
  if (adjoint)
    launch_step<true, false>(ctx, ops, nullptr, n, batch, rows, h, use_handle, st);
  else
    launch_step<false, false>(ctx, ops, w, n, batch, rows, h, use_handle, st);
}

ZB_CHECK_WORD_ACCESSOR(check_word_split)

cudaError_t split_set_wait(uint64_t wait_ns) {
#ifdef ZBUS_CHECKED
  return cudaMemcpyToSymbol(g_split_wait_ns, &wait_ns, sizeof(wait_ns));
#else
  (void)wait_ns;
  return cudaErrorNotSupported;
#endif
}

}  // namespace zbus
