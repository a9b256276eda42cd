// Tensor-times-matrix products on the tensor cores, and the contractions that turn
// them into concurrent MTTKRPs.
//
//   Y_a(r, c) = sum_i T_(a)(i, r) Ubar^(a)(i, c)           (ttm_kernel)
//   Mbar_n(i_n, c) = sum over the other indices of r of Y_a(r, c) times the
//                    remaining factors' entries             (contract_kernel)
//
// for a mode a != n (Eq. MTTKRP with its Khatri-Rao sum taken one mode at a
// time).  Y_a does not depend on the other factors, so every mode n != a that is
// updated before Ubar^(a) changes shares it: a sweep of N modes needs two of the
// products of 2 C prod(I) operations instead of N.
//
// The FP64 form's product, exact up to FP64 rounding on the BF16 tensor pipe: GB300 runs
// 1.1 TFLOP/s in FP64 and 1889 TFLOP/s in BF16, so 36 BF16 products per FP64 one still
// leave a factor of 48.  Every operand value x of a contraction vector whose magnitudes
// stay below 2^E is rounded to 58 fractional bits of 2^E and
// written in balanced digits, x = 2^(E-7) sum_k d_k 2^(-7k), |d_0| <= 128,
// |d_k| <= 64 (k = 1 .. 7; d_7 in steps of 1/4): BF16 holds each digit exactly.
// The products d_s e_t with s + t = l < 8 are summed per level l in one FP32
// accumulator in TMEM.  A level's terms are integers and its sum stays below
// (l + 3) 2^12 K <= 2^24 for chains of K <= kTtmChainMax, so levels 0 to 6 are
// exact whatever the order of the additions; level 7 may truncate in its own
// last bits (2^-63 of the product of the vectors' maxima).  The drain adds the levels as
// 64-bit integers and rounds once to FP64.
//
// Bound.  Let 2^E and 2^F bound the two vectors' magnitudes and S be the sum of the
// magnitudes of an entry's K terms.  Dropped are the operands' rounding (at most 2^-58 per
// term) and the products beyond level 7 (seven of at most 2^-58 per term): at most
// K 2^-55 2^(E+F), typically sqrt(7 K) 2^-60 2^(E+F).  That is measured by the vectors'
// maxima, not by the entry's own terms, so it is accepted only where S >= 2^-6 2^(E+F):
// the error is then at most 16 K 2^-53 S and typically 1.3 sqrt(K) 2^-53 S or less, and an
// MTTKRP's sum over many entries averages it (measured below).  The drain finds S from below
// by the entry's own value, or else by the products of the magnitudes' leading 16 bits
// (stored with the digits); an entry that neither certifies is computed as a plain FP64 dot
// product (plain_entries).  Of dense data of one scale none is, of noisy fluorescence-like
// data 0 to 3 entries in 100 (300x100x50, 1500 columns: 0.45 ms a sweep from the start,
// 0.57 ms at convergence; with 8-bit magnitudes and twice the threshold 1.2 ms).  Data whose
// vectors hardly overlap take more: 1.3 ms with 1% of the tensor non-zero, 7 ms for separated
// bumps without noise, against 16 ms of the CUDA-core kernel; 40x33x61: 0.2 against 0.35 ms.
//
// Along the contraction the two operands are equilibrated by powers of two
// (exact): T_(a)(i, :) 2^(-F_i) against Ubar^(a)(i, :) 2^(F_i), F_i the mean exponent of
// slice i's non-zero entries: slices of different scale (an outlying sample) then cost no
// digits, and a single large entry sets no slice's scale: it is the maximum of its own
// column of T_(a) alone, and only that column's entries need the dot products where a
// submodel leaves it out.
//
// Measured (GB300), against the CUDA-core MTTKRP of every mode: an FP64 sweep of
// 300x100x50 with 1500 columns 16.0 -> 0.45 ms, of 400x400x400 with 400 columns
// 192 -> 3.4 ms; loss and gradient of 100x60x60x40 with 800 columns 166 -> 4.3 ms.
// Largest error of an MTTKRP entry against quadruple precision, in units of 2^-53 of the sum
// of its own terms' magnitudes (41x61x35 to 300x100x50 and 4-way, uniform, normal and bumps,
// 0 to 40 sweeps): 0.1 to 5 where the CUDA-core kernel, with longer chains, has 0.2 to 33; of
// the largest entry 1.3e-16 to 7.1e-16 against 1.5e-16 to 1.9e-15.
//
// A column of Ubar^(a) with a non-finite entry is taken out of the digits and
// computed by plain FP64 dot products in the drain, so Inf and NaN propagate as
// in the CUDA-core kernel; a tensor with a non-finite entry never gets here.
#include <limits.h>
#include <math.h>

#include <type_traits>

#include "jk_common.cuh"
#include "jk_ptx.cuh"

namespace jk {
namespace {

using namespace ptx;

constexpr int kTileM = kTtmTileC;
constexpr int kRow = 32;                      // bytes of one operand row per stage: 16 BF16
constexpr uint32_t kABytes = kTileM * kRow;   // one digit of U for 16 rows k
// A stage holds the eight digits of 16 rows k: 32 KB of U's images and up to 16 KB of
// T's.  TMEM holds the eight level accumulators of BN columns, twice for BN = 32 (the
// drain then runs under the next tile).
constexpr int P = 8;
constexpr int ttm_sets(int BN) { return 2 * P * BN <= 512 ? 2 : 1; }
constexpr uint32_t kAStage = P * kABytes, kBStage = 16384, kStage = kAStage + kBStage;
constexpr int kStages = 4;
constexpr int kEpiWarps = 16;
constexpr int kTmaWarp = kEpiWarps, kMmaWarp = kEpiWarps + 1;
constexpr int kThreads = 32 * (kEpiWarps + 2);
constexpr uint32_t kTmemCols = 512;           // all of TMEM
constexpr uint32_t kListBytes = kEpiWarps * 32 * 16 * 2;   // the draining warps' lists (plain_entries)
constexpr size_t kSmem = 1024 + (size_t)kStages * kStage + kListBytes + (2 * kStages + 5) * 8 + 16;

// ---- digits ---------------------------------------------------------------------
// One operand matrix X (K x M, row stride ld; K the contraction) into stage images:
// per TILE columns m and 16 rows k, P digit tiles of TILE x 32 bytes, K-major in
// the 32-byte swizzle (16-byte chunk XOR bit 2 of the row): one bulk copy per
// operand and stage.  A block takes 8 columns, thread (m, g) the 8-row chunks g
// and g + 32, loaded once into registers (K <= kTtmChainMax: at most 56 chunks):
// first each column's exponent (expo[m].x: scaled magnitudes < 2^expo), then the
// digits.  sgn = +1 / -1 scales row k by 2^(+-kexp[k]).  Integer arithmetic
// throughout: an FP64 rint per digit would take 18 us of the FP64 pipe for
// 300 x 1500 entries.  counter: a sweep's first slicing also advances the sweep
// counter (null otherwise).  mag: every scaled magnitude in units of 2^(expo - 16),
// rounded down (32 nk bytes per column: for 16 rows, the high bytes, then the low ones);
// expo[m].y: how many have a high byte of at least kFlat.
constexpr int kSliceCols = 8;   // columns per block
constexpr uint32_t kFlat = 16;  // 2^-4 of a column's power of two, in a high byte's units of 2^-8

// Half of every digit's field below d_0: 256 of the last one's nine bits, 64 of the
// others' seven.
constexpr long long half_fields() {
  long long h = 256;
  for (int s = 1; s < P - 1; ++s) h += 64ll << (9 + 7 * (s - 1));
  return h;
}

// Columns whose products T Ubar^(a) (or those times another factor) may leave FP64's range
// where the Khatri-Rao product does not: a tensor or a factor of extreme scale (beyond about
// 1e60, 1e120).  Y holds such a column times 2^-column_power, so that it has T's own scale,
// and the contractions carry the power to the end.  ec: the column's exponent.
__device__ __forceinline__ int column_power(int ec, int2 range) {
  const bool ordinary = abs(range.x) <= 200 && abs(ec) <= 400 && ec + range.y <= 1014;
  return ordinary ? 0 : ec - range.x;
}

template <int TILE>
__global__ void __launch_bounds__(256) slice_f64_kernel(const double* __restrict__ X, int K, int64_t M, int64_t ld,
                                                        const int* __restrict__ kexp, int sgn, int nk, int64_t Mpad,
                                                        unsigned char* __restrict__ img, int2* __restrict__ expo,
                                                        unsigned char* __restrict__ mag,
                                                        const int2* __restrict__ range, int* __restrict__ power,
                                                        int* __restrict__ counter) {
  if (counter != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *counter += 1;
  constexpr int kCols = kSliceCols, kGroups = 256 / kCols;
  constexpr int kTop = 9 + 7 * (P - 2);   // position of d_0; the last digit's field has two bits more
  static_assert(2 * kGroups * 8 >= kTtmChainMax, "two chunks per thread hold a column");
  __shared__ int red[kGroups][kCols + 1];
  __shared__ int flat[kCols];
  const int ml = threadIdx.x % kCols, g = threadIdx.x / kCols;
  for (int64_t m0 = (int64_t)blockIdx.x * kCols; m0 < Mpad; m0 += (int64_t)gridDim.x * kCols) {
    const int64_t m = m0 + ml;
    const bool mv = m < M;
    double x[2][8];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int k = 8 * (g + j * kGroups) + e;
        x[j][e] = mv && k < K ? __ldg(X + (int64_t)k * ld + m) : 0.0;
      }
    int top = INT_MIN;   // largest biased exponent after scaling
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int k = 8 * (g + j * kGroups) + e;
        const unsigned long long u = (unsigned long long)__double_as_longlong(x[j][e]) & 0x7fffffffffffffffull;
        const int ef = (int)(u >> 52);
        if (ef == 2047)
          top = INT_MAX;
        else if (u != 0)
          top = max(top, (ef > 1 ? ef : 1) + sgn * __ldg(kexp + k));
      }
    __syncthreads();   // red of the previous columns is consumed
    red[g][ml] = top;
    if (g == 0) flat[ml] = 0;
    __syncthreads();
    for (int i = 0; i < kGroups; ++i) top = max(top, red[i][ml]);
    const bool col_bad = top == INT_MAX;
    const int E = (col_bad || top == INT_MIN) ? 0 : top - 1022;
    int nflat = 0;
    const int64_t tile = m / TILE;
    const int row = (int)(m - tile * TILE);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int ch = g + j * kGroups;
      if (ch >= 2 * nk) break;
      unsigned long long high = 0, low = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x[j][e]);
        const int ef = (int)((b >> 52) & 2047);
        if (ef > 0 && !col_bad) {   // a normal entry: 1.m 2^(ef - 1023), scaled below 2^E
          const int sh = E - 1 - (ef + sgn * __ldg(kexp + 8 * ch + e) - 1023);
          const uint32_t q = sh < 16 ? (0x8000u | (uint32_t)((b >> 37) & 0x7fff)) >> sh : 0u;
          high |= (unsigned long long)(q >> 8) << (8 * e);
          low |= (unsigned long long)(q & 255u) << (8 * e);
          nflat += (q >> 8) >= kFlat ? 1 : 0;
        }
      }
      unsigned long long* mg = reinterpret_cast<unsigned long long*>(mag + (m * nk + (ch >> 1)) * 32 + (ch & 1) * 8);
      mg[0] = high;
      mg[2] = low;
      uint32_t w[P][4];
#pragma unroll
      for (int pr = 0; pr < 4; ++pr) {
        uint32_t lo[P], hi[P];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int k = 8 * ch + 2 * pr + e;
          long long v = 0;
          const unsigned long long b = (unsigned long long)__double_as_longlong(x[j][2 * pr + e]);
          if ((b << 1) != 0 && !col_bad) {   // entries beyond K were loaded as zeros
            const int ef = (int)((b >> 52) & 2047);
            unsigned long long mant = b & 0xfffffffffffffull;
            if (ef > 0) mant |= 1ull << 52;
            // |x| 2^(kTop + 7 - E) rounded: shift <= kTop - 46 as |x| < 2^E
            const int sh = (ef > 0 ? ef : 1) + sgn * __ldg(kexp + k) - E - (1075 - kTop - 7);
            if (sh >= 0)
              mant <<= sh;
            else
              mant = sh < -54 ? 0ull : (mant + (1ull << (-sh - 1))) >> (-sh);
            v = (b >> 63) ? -(long long)mant : (long long)mant;
          }
          // balanced digits: add half of every field, read the fields unsigned
          constexpr long long kHalf = half_fields();
          v += kHalf;
          uint32_t d[P];
          d[0] = __float_as_uint(__int_as_float(0x4B400000 + (int)(v >> kTop)) - 12582912.f);
#pragma unroll
          for (int s = 1; s < P - 1; ++s)
            d[s] = __float_as_uint(__int_as_float(0x4B400000 - 64 + (int)((v >> (kTop - 7 * s)) & 127)) - 12582912.f);
          d[P - 1] = __float_as_uint((__int_as_float(0x4B400000 - 256 + (int)(v & 511)) - 12582912.f) * 0.25f);
#pragma unroll
          for (int s = 0; s < P; ++s) (e == 0 ? lo[s] : hi[s]) = d[s];
        }
#pragma unroll
        for (int s = 0; s < P; ++s) w[s][pr] = __byte_perm(lo[s], hi[s], 0x7632);   // high halves: BF16
      }
      unsigned char* dst = img + (tile * nk + (ch >> 1)) * (int64_t)(P * TILE * kRow) + (row >> 3) * (8 * kRow) +
                           (row & 7) * kRow + (((ch & 1) ^ ((row >> 2) & 1)) << 4);
#pragma unroll
      for (int s = 0; s < P; ++s)
        *reinterpret_cast<uint4*>(dst + s * (TILE * kRow)) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
    if (nflat > 0) atomicAdd(&flat[ml], nflat);
    __syncthreads();
    if (g == 0) {
      expo[m] = make_int2(col_bad ? kTtmBadExp : (top == INT_MIN ? kTtmZeroExp : E), flat[ml]);
      if (power != nullptr) power[m] = range == nullptr || col_bad || top == INT_MIN ? 0 : column_power(E, *range);
    }
  }
}

// kexp[i] = F_i, the mean exponent of slice i's non-zero entries (0 for a zero slice): no
// single entry, and no slice of another mode, sets it.  *bad = 1 if an entry is Inf or NaN.
__global__ void slice_exponent_kernel(const double* __restrict__ Tn, int64_t J, int* __restrict__ kexp,
                                      int* __restrict__ bad) {
  __shared__ long long sums[8], counts[8];
  const int64_t i = blockIdx.x;
  long long sum = 0, count = 0;
  bool finite = true;
  for (int64_t j = threadIdx.x; j < J; j += blockDim.x) {
    const unsigned long long u =
        (unsigned long long)__double_as_longlong(__ldg(Tn + i * J + j)) & 0x7fffffffffffffffull;
    const int ef = (int)(u >> 52);
    finite = finite && ef != 2047;
    if (u != 0) {
      sum += (ef > 1 ? ef : 1) - 1022;
      ++count;
    }
  }
  if (!finite) *bad = 1;
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    count += __shfl_xor_sync(0xffffffffu, count, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sums[threadIdx.x >> 5] = sum;
    counts[threadIdx.x >> 5] = count;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)blockDim.x / 32; ++w) {
      sum += sums[w];
      count += counts[w];
    }
    kexp[i] = count == 0 ? 0 : (int)(sum / count);
  }
}

// range: g, about T's own exponent, at most what keeps every sum of T(., r) and a column of
// size 1 finite, and the largest exponent of rexp.
__global__ void range_kernel(const int* __restrict__ kexp, int K, const int2* __restrict__ rexp, int64_t J,
                             int2* __restrict__ range) {
  __shared__ int red[32];
  int top = kTtmZeroExp;
#pragma unroll 8
  for (int64_t r = threadIdx.x; r < J; r += blockDim.x) top = max(top, __ldg(rexp + r).x);
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = top;
  __syncthreads();
  if (threadIdx.x == 0) {
    int sum = 0;
    for (int i = 0; i < K; ++i) sum += __ldg(kexp + i);
    for (int w = 0; w < (int)blockDim.x / 32; ++w) top = max(top, red[w]);
    *range = make_int2(min(sum / K, 1014 - top), top);   // K < 2^9 terms below 2^1014
  }
}

// ---- the product ------------------------------------------------------------------
__device__ __forceinline__ uint64_t smem_desc32(uint32_t saddr) {   // K-major, 32-byte swizzle
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)((8 * kRow) >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}

// m0 2^21 + m1 2^14 + m2 2^7 + m3 of four level sums (integers; the last one may
// carry a fraction, rounded here).  |m| <= 2^22: after adding 1.5 2^23 the low
// mantissa bits are the integer, and two levels fit 32 bits.  Chains of at most
// kTtmFastChain rows cannot exceed that; in longer ones (check) strongly correlated
// digits may reach 2^24 and are converted (a quarter of the rate).
constexpr int kTtmFastChain = 102;   // (l + 3) 2^12 K <= 2^22 for l <= 7

__device__ __forceinline__ long long sum_levels(uint32_t m0, uint32_t m1, uint32_t m2, uint32_t m3, bool check) {
  constexpr float kRound = 12582912.f;   // 1.5 * 2^23: bits 0x4B400000
  constexpr uint32_t kBias = 0x4B400000u * 129u;
  const uint32_t b0 = __float_as_uint(__uint_as_float(m0) + kRound), b1 = __float_as_uint(__uint_as_float(m1) + kRound);
  const uint32_t b2 = __float_as_uint(__uint_as_float(m2) + kRound), b3 = __float_as_uint(__uint_as_float(m3) + kRound);
  if (check) {
    const uint32_t chk = (b0 ^ 0x4B000000u) | (b1 ^ 0x4B000000u) | (b2 ^ 0x4B000000u) | (b3 ^ 0x4B000000u);
    if ((chk & 0xFF800000u) != 0)
      return ((long long)__float2int_rn(__uint_as_float(m0)) << 21) +
             ((long long)__float2int_rn(__uint_as_float(m1)) << 14) +
             ((long long)__float2int_rn(__uint_as_float(m2)) << 7) + (long long)__float2int_rn(__uint_as_float(m3));
  }
  const int t0 = (int)(b0 * 128u + b1 - kBias), t1 = (int)(b2 * 128u + b3 - kBias);
  return (long long)t0 * 16384 + t1;
}

// The eight levels (BN TMEM columns apart) of this warp's 32 lanes x NC columns at base:
// per column hi + lo 2^-28 in units of level 3.
template <int BN, int NC>
__device__ __forceinline__ void read_levels(uint32_t base, bool check, long long (&hi)[NC], uint32_t (&lo)[NC]) {
#pragma unroll
  for (int h = 0; h < NC / 4; ++h) {
    uint32_t v[4][4];
    __syncwarp();
#pragma unroll
    for (int l = 0; l < 4; ++l) tmem_ld4(base + (uint32_t)(l * BN + 4 * h), v[l]);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 4; ++k) hi[4 * h + k] = sum_levels(v[0][k], v[1][k], v[2][k], v[3][k], check);
    __syncwarp();
#pragma unroll
    for (int l = 0; l < 4; ++l) tmem_ld4(base + (uint32_t)((l + 4) * BN + 4 * h), v[l]);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long low = sum_levels(v[0][k], v[1][k], v[2][k], v[3][k], check);
      hi[4 * h + k] += low >> 28;
      lo[4 * h + k] = (uint32_t)low & 0xFFFFFFFu;
    }
  }
}

// (hi + lo 2^-28) 2^(ex - 35) rounded to FP64, |hi| < 2^47, lo < 2^28, in
// integers: one FP64 add per output would take 4096 cycles of GB300's FP64 pipe
// (two lanes per clock and SM) per tile.
__device__ __forceinline__ double round_levels(long long hi, uint32_t lo, int ex) {
  // magnitude by the ones' complement (off by one unit of level 7)
  const uint32_t s = (uint32_t)(hi >> 63);
  const uint32_t h1 = (uint32_t)((unsigned long long)hi >> 32) ^ s, h0 = (uint32_t)hi ^ s;
  const uint32_t l1 = (lo ^ s) << 4;   // 28 bits, left aligned
  const bool small = h1 == 0;
  const uint32_t w2 = small ? h0 : h1, w1 = small ? l1 : h0, w0 = small ? 0u : l1;
  const int n = __clz((int)w2);
  const uint32_t m1 = __funnelshift_l(w1, w2, n), m0 = __funnelshift_l(w0, w1, n);
  const int be = 1023 + 28 + ex - n - (small ? 32 : 0);
  if (w2 == 0 || be < 1 || be > 2045)
    // rare: zeros, sums below 2^-35 of the vectors' maxima, results outside the
    // normal range (both addends exact: one rounding, and scalbn's)
    return scalbn(fma((double)lo, 1.0 / 268435456.0, (double)hi), ex - 35);
  const unsigned long long q =
      ((((unsigned long long)m1 << 32) | m0) >> 11) + ((m0 >> 10) & 1u) + ((unsigned long long)(uint32_t)(be - 1) << 52);
  return __longlong_as_double((long long)(q | ((unsigned long long)(s & 0x80000000u) << 32)));
}

// What certifies an entry of the product (the bound is derived at the top of this file): the
// sum of its terms' magnitudes is at least 2^-6 of the product of the vectors' maxima,
//  - because so many of both vectors' entries are at least 2^-4 of their maxima that at
//    least kFlatTerms rows hold two of them (4 x 2^-8; decided for a warp's 32 columns and
//    rows at once: dense data of one scale, at no cost per entry),
//  - by the entry's own value, or
//  - by the magnitudes' leading 16 bits.
constexpr int kFlatTerms = 4;
constexpr long long kCertain = 1ll << 29;      // 2^-6 in units of level 3 (2^-35)
constexpr uint32_t kCertainMags = 1u << 18;    // 2^-6 in units of 2^-24

// Of the entries of this warp's tile rows that their own value does not certify (bits of open:
// rows r0 .. r0 + 7 of column c0 + lane), those that the magnitudes do not certify either.
__device__ __noinline__ uint32_t uncertified(const TtmArgs& a, int64_t r0, int c0, uint32_t open, int lane) {
  // the magnitudes of sixteen rows k of the contraction at a time, against all pending rows
  // together (their loads are in flight together): the products of the high bytes, which are
  // mostly enough, then those of high and low ones
  const uint4* mr = reinterpret_cast<const uint4*>(a.rmag) + r0 * a.nk * 2;
  const uint4* mc = reinterpret_cast<const uint4*>(a.cmag) + (int64_t)(c0 + lane) * a.nk * 2;   // padded, as the rows
  uint32_t sum[8] = {};
  auto dot = [](const uint4& x, const uint4& y, uint32_t s) {
    return __dp4a(x.x, y.x, __dp4a(x.y, y.y, __dp4a(x.z, y.z, __dp4a(x.w, y.w, s))));
  };
  for (int w = 0; w < a.nk && __any_sync(0xffffffffu, open != 0); ++w) {
    const uint4 y = __ldg(mc + 2 * w);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      sum[k] += dot(__ldg(mr + ((int64_t)k * a.nk + w) * 2), y, 0u) << 8;
      if (sum[k] >= kCertainMags) open &= ~(1u << k);
    }
  }
  for (int w = 0; w < a.nk && __any_sync(0xffffffffu, open != 0); ++w) {
    const uint4 yh = __ldg(mc + 2 * w), yl = __ldg(mc + 2 * w + 1);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint4* xp = mr + ((int64_t)k * a.nk + w) * 2;
      sum[k] = dot(__ldg(xp), yl, dot(__ldg(xp + 1), yh, sum[k]));
      if (sum[k] >= kCertainMags) open &= ~(1u << k);
    }
  }
  return open;
}

// Plain FP64 dot products for the entries in pending (bits as above): those that nothing
// certifies, and every entry of a column with a non-finite one.  They are gathered in list and
// taken 32 at a time, a lane each, or fewer by several lanes each: bound by the FP64 pipe
// (K / 2 clocks of an SM per entry), as submodels that share a factor fail together, rows of
// whole tiles at a time.
__device__ __noinline__ void plain_entries(const TtmArgs& a, int64_t r0, int c0, uint32_t pending,
                                           unsigned short* list, int lane) {
  int at = __popc(pending);
  for (int o = 1; o < 32; o <<= 1) {
    const int below = __shfl_up_sync(0xffffffffu, at, o);
    if (lane >= o) at += below;
  }
  const int total = __shfl_sync(0xffffffffu, at, 31);
  at -= __popc(pending);
  for (; pending != 0; pending &= pending - 1)
    list[at++] = (unsigned short)(((__ffs((int)pending) - 1) << 5) | lane);
  __syncwarp();   // the list, and the digits' sums before the stores below
  for (int base = 0; base < total; base += 32) {
    const int cnt = total - base < 32 ? total - base : 32;
    const int lg = cnt > 16 ? 0 : __clz(cnt > 1 ? cnt - 1 : 0) - 27;   // 32 >> lg entries at a time
    const int e = lane >> lg, part = lane & ((1 << lg) - 1);
    const int code = list[base + (e < cnt ? e : 0)];
    const int64_t r = r0 + (code >> 5);
    const int c = c0 + (code & 31);
    const double *t = a.Tn + r, *u = a.U + c;
    const int ec = __ldg(a.cexp + c).x;
    const int power = __ldg(a.power + c);
    double acc = 0.0;
    if (power != 0) {
      for (int i = part; i < a.K; i += 1 << lg) {
        const int f = __ldg(a.kexp + i);
        acc = fma(scalbn(__ldg(t + (int64_t)i * a.J), ec - power - f), scalbn(__ldg(u + (int64_t)i * a.C), f - ec), acc);
      }
    } else {
#pragma unroll 8
      for (int i = part; i < a.K; i += 1 << lg)
        acc = fma(__ldg(t + (int64_t)i * a.J), __ldg(u + (int64_t)i * a.C), acc);
    }
    __syncwarp();
    for (int o = 1; o < (1 << lg); o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (e < cnt && part == 0) a.Y[r * a.C + c] = acc;
  }
  __syncwarp();   // the list is free again
}

// Persistent: one CTA per SM (all of TMEM, 4 x 48 KB stages) walks the 128 x
// BN tiles of Y, C tiles fastest so that the CTAs in flight share T's images in L2.
//   warp 16  TMA: one lane refills the ring in order, across tile boundaries
//   warp 17  one lane issues the stage's 12 MMAs (B digits stacked along N, up to
//            256 wide: digit s of U against digits t0..t1 of T lands in levels
//            s + t0 .. s + t1, 64 columns each)
//   warps 0-15  drain: 32 columns c x a quarter of the rows r each, levels to Y
// Bound: shared-memory bandwidth.  Per 16 rows of the contraction and 128 x 64 tile the
// MMAs take 1152 cycles of the tensor pipe but read 120 KB of operands while TMA writes
// 48 KB: 168 KB at 128 bytes a clock are 1344 cycles, and about 1380 were measured
// (400x400x400, 400 columns: 1310 us).
// BN = 64 leaves room for one accumulator set, so the next tile's first MMA waits until
// every level is read (about 5000 cycles): the drain takes the levels into 64-bit integers
// first and rounds and stores them under the next tile's MMAs.  BN = 32 has two sets and
// hides the drain, but its MMAs (the narrow ones at their least time) take about 1130
// cycles per 16 rows of half a tile: 300x100x50 contracted over 100 rows took 157 us
// against 147 with BN = 64, 100x60x60x40 over 100 rows 828 against 767; over up to 64
// rows the halves are even, and fill the SMs more evenly.
template <int BN>
__global__ void __launch_bounds__(kThreads, 1) ttm_kernel(const __grid_constant__ TtmArgs a) {
  constexpr int NB = ttm_sets(BN);          // accumulator sets
  constexpr int NC = BN / 4;                // rows r of a draining warp
  constexpr int G = 256 / BN;               // digits of T stacked per MMA
  constexpr uint32_t kBBytes = BN * kRow;   // one digit of T for 16 rows k
  static_assert(P * kBBytes <= kBStage && NB * P * BN <= (int)kTmemCols && BN % 16 == 0, "tile");
  constexpr uint32_t kSetCols = kTmemCols / NB;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned short* lists = reinterpret_cast<unsigned short*>(ring + (size_t)kStages * kStage);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)kStages * kStage + kListBytes);
  uint64_t* empty = full + kStages;
  uint64_t* accum = empty + kStages;      // [2] a tile's MMAs into set b are complete
  uint64_t* tmem_empty = accum + 2;       // [2] the drain has read set b
  uint64_t* drain = accum + 4;            // abort path: the MMAs so far are complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accum[b], 1);
      mbar_init(&tmem_empty[b], kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kMmaWarp) tmem_alloc(tmem_slot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int64_t ntiles = (int64_t)a.tiles_c * a.tiles_r;
  const int nk = a.nk;

  if (warp == kTmaWarp) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true, issued = false;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int64_t tr = t / a.tiles_c;
        const unsigned char* srca = a.At + (t - tr * a.tiles_c) * nk * (int64_t)(P * kABytes);
        const unsigned char* srcb = a.Bt + tr * nk * (int64_t)(P * kBBytes);
        for (int ks = 0; ks < nk; ++ks) {
          ok = wait_bounded(&empty[s], ph ^ 1u, abort_flag, a.err, 1);
          if (!ok) break;
          unsigned char* dst = ring + (size_t)s * kStage;
          mbar_arrive_expect_tx(&full[s], kAStage + P * kBBytes);
          bulk_load(dst, srca + (int64_t)ks * kAStage, kAStage, &full[s]);
          bulk_load(dst + kAStage, srcb + (int64_t)ks * (P * kBBytes), P * kBBytes, &full[s]);
          issued = true;
          if (++s == kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (*abort_flag && issued) {   // let the copies in flight land before the CTA exits
        const uint64_t t0 = global_ns();
        while (global_ns() - t0 < 200000ull) {
        }
      }
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      const uint64_t desc0 = smem_desc32(smem_u32(ring));
      uint32_t idesc[G + 1];
#pragma unroll
      for (int c = 0; c <= G; ++c)   // FP32 accumulator, BF16 operands, both K-major, N >> 3, M >> 4
        idesc[c] = (1u << 4) | (1u << 7) | (1u << 10) | (((uint32_t)(c * BN) >> 3) << 17) |
                   ((uint32_t)(kTileM >> 4) << 24);
      int s = 0;
      uint32_t ph = 0, use = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++use) {
        const uint32_t b = use % NB;
        if (use >= NB) {
          ok = wait_bounded(&tmem_empty[b], (use / NB - 1) & 1u, abort_flag, a.err, 7);
          if (!ok) break;
          tc_fence_after();
        }
        const uint32_t td = tmem + b * kSetCols;
        for (int ks = 0; ks < nk; ++ks) {
          ok = wait_bounded(&full[s], ph, abort_flag, a.err, 2);
          if (!ok) break;
          tc_fence_after();
          const uint64_t ad = desc0 + (uint64_t)(((uint32_t)s * kStage) >> 4);
          const uint64_t bd = ad + (uint64_t)(kAStage >> 4);
#pragma unroll
          for (int p = 0; p < P; ++p) {
#pragma unroll
            for (int t0 = 0; t0 < P - p; t0 += G) {
              const int cnt = P - p - t0 < G ? P - p - t0 : G;
              tc_mma<kKindBF16>(td + (uint32_t)((p + t0) * BN), ad + (uint64_t)(p * (kABytes >> 4)),
                                bd + (uint64_t)(t0 * (kBBytes >> 4)), idesc[cnt], (ks == 0 && p == 0) ? 0u : 1u);
            }
          }
          tc_commit(&empty[s]);
          if (++s == kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (ok) tc_commit(&accum[b]);
      }
      if (!ok) {
        tc_commit(drain);
        wait_drain(drain, 0);
      }
    }
  } else {
    const int quarter = warp & 3, grp = warp >> 2;
    uint32_t use = 0;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++use) {
      const int64_t tr = t / a.tiles_c;
      const int c = (int)(t - tr * a.tiles_c) * kTileM + quarter * 32 + lane;
      const int64_t r0 = tr * BN + NC * grp;
      const int2 ce = __ldg(a.cexp + c);   // padded to whole tiles, as rexp
      const int ec = ce.x;
      const int power = __ldg(a.power + c);
      // this warp's row exponents, in flight while the tile's MMAs run
      const int2 re = __ldg(a.rexp + r0 + (lane < NC ? lane : 0));
      const uint32_t b = use % NB;
      const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + b * kSetCols + (uint32_t)(NC * grp);
      bool have = wait_sleepy(&accum[b], (use / NB) & 1u, abort_flag, a.err, 5);
      have = __all_sync(0xffffffffu, have);
      if (!have) break;
      tc_fence_after();
      // read the levels into integers, so that the next tile's MMAs start early ...
      long long hi[NC];
      uint32_t lo[NC];
      read_levels<BN, NC>(base, a.K > kTtmFastChain, hi, lo);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tmem_empty[b]);
      // ... and round and store them meanwhile
      const bool forced = ec == kTtmBadExp;
      const int ex = ec - power;
      double* y = a.Y + r0 * a.C + c;
      uint32_t pending = 0;   // rows whose sum is below kCertain of the vectors' maxima
#pragma unroll
      for (int k = 0; k < NC; ++k, y += a.C) {
        const int er = __shfl_sync(0xffffffffu, re.x, k);
        if (r0 + k >= a.J || c >= a.C) continue;
        const bool sure = (unsigned long long)(hi[k] + kCertain) >= 2ull * kCertain;
        if (forced || (!sure && er != kTtmZeroExp && ec != kTtmZeroExp)) pending |= 1u << k;
        if (!forced) *y = round_levels(hi[k], lo[k], ex + er);
      }
      const int rflat = __reduce_min_sync(0xffffffffu, re.y);
      if (ce.y + rflat >= a.K + kFlatTerms) pending = 0;
      if (__any_sync(0xffffffffu, pending != 0)) {
        // a column with a non-finite entry (its magnitudes are zero) needs all of its sums
        uint32_t left = 0;
#pragma unroll
        for (int h = 0; h < NC; h += 8) left |= uncertified(a, r0 + h, c - lane, (pending >> h) & 255u, lane) << h;
        if (__any_sync(0xffffffffu, left != 0)) plain_entries(a, r0, c - lane, left, lists + warp * (32 * 16), lane);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// ---- contraction with one more factor ------------------------------------------------
// v 2^e in exact factors (but for an underflow), without scalbn's registers.
__device__ __forceinline__ double times_power(double v, int e) {
#pragma unroll 1
  while (e != 0) {
    const int k = e > 1000 ? 1000 : (e < -1000 ? -1000 : e);
    v *= __hiloint2double((k + 1023) << 20, 0);
    e -= k;
  }
  return v;
}

// out[s][h][l][c] = sum over split s of m of X[h][m][l][c] U[m][c].  A thread takes RB
// outputs (h, l) of V adjacent columns: one load of U serves RB of X, and a load of two
// columns is 16 bytes.  A column that X holds times a power of two (see column_power) is
// contracted with its factor's column scaled to at most 1; the powers go into the result, or,
// if that is contracted again, to out_power.  Bound: X read once, or the FP64 pipe's two
// multiply-adds per clock and SM (400x400x400, 400 columns: 130 us, 512 MB at 3.9 TB/s and
// 490 G multiply-adds/s).
template <int RB, int V>
__global__ void __launch_bounds__(256) contract_kernel(const double* __restrict__ X, int64_t H, int Mm, int64_t L,
                                                       int C, const double* __restrict__ U, int mchunk,
                                                       const int* __restrict__ power, int* __restrict__ out_power,
                                                       double* __restrict__ out) {
  constexpr int UN = RB * V >= 8 ? 2 : (RB * V >= 4 ? 4 : 8);   // terms loaded together
  const int64_t HL = H * L, groups = (HL + RB - 1) / RB;
  const int CV = C / V;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= groups * CV) return;
  const int64_t g = idx / CV;
  const int c = (int)(idx - g * CV) * V;
  const int mb = blockIdx.y * mchunk, me = mb + mchunk < Mm ? mb + mchunk : Mm;
  const double* x[RB];
  double acc[RB][V];
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    const int64_t o = g * RB + q < HL ? g * RB + q : HL - 1;
    const int64_t hh = o / L;
    x[q] = X + ((hh * Mm + mb) * L + (o - hh * L)) * C + c;
#pragma unroll
    for (int w = 0; w < V; ++w) acc[q][w] = 0.0;
  }
  const int64_t step = L * C;
  const double* u = U + (int64_t)mb * C + c;
  auto load = [](const double* p, double (&v)[V]) {
    if constexpr (V == 2) {
      const double2 t = __ldg(reinterpret_cast<const double2*>(p));
      v[0] = t.x;
      v[1] = t.y;
    } else {
      v[0] = __ldg(p);
    }
  };
  bool shifted = false;
#pragma unroll
  for (int w = 0; w < V; ++w) shifted = shifted || __ldg(power + c + w) != 0;
  auto terms = [&](auto nt) {   // N <= UN terms, all loaded first
    constexpr int N = decltype(nt)::value;
    double uv[N][V], xv[N][RB][V];
#pragma unroll
    for (int e = 0; e < N; ++e) {
      load(u + (int64_t)e * C, uv[e]);
#pragma unroll
      for (int q = 0; q < RB; ++q) load(x[q] + e * step, xv[e][q]);
    }
#pragma unroll
    for (int e = 0; e < N; ++e)
#pragma unroll
      for (int q = 0; q < RB; ++q)
#pragma unroll
        for (int w = 0; w < V; ++w) acc[q][w] = fma(xv[e][q][w], uv[e][w], acc[q][w]);
    u += (int64_t)N * C;
#pragma unroll
    for (int q = 0; q < RB; ++q) x[q] += N * step;
  };
  if (shifted) {
#pragma unroll
    for (int w = 0; w < V; ++w) {
      int pw = __ldg(power + c + w);
      double most = 0.0;
#pragma unroll 1
      for (int k = 0; k < Mm; ++k) most = fmax(most, fabs(__ldg(U + (int64_t)k * C + c + w)));
      const int ue = pw != 0 && most > 0.0 && isfinite(most) ? (__double2hiint(most) >> 20) - 1022 : 0;
#pragma unroll 1
      for (int k = mb; k < me; ++k) {
        const double uv = times_power(__ldg(U + (int64_t)k * C + c + w), -ue);
#pragma unroll
        for (int q = 0; q < RB; ++q) acc[q][w] = fma(__ldg(x[q] + (k - mb) * step + w), uv, acc[q][w]);
      }
      pw += ue;   // true: acc 2^pw
      if (out_power != nullptr)
        out_power[c + w] = pw;   // the same from every thread of the column
      else
#pragma unroll
        for (int q = 0; q < RB; ++q) acc[q][w] = times_power(acc[q][w], pw);
    }
  } else {
    int m = mb;
    for (; m + UN <= me; m += UN) terms(std::integral_constant<int, UN>{});
    for (; m < me; ++m) terms(std::integral_constant<int, 1>{});
    if (out_power != nullptr)
#pragma unroll
      for (int w = 0; w < V; ++w) out_power[c + w] = 0;
  }
#pragma unroll
  for (int q = 0; q < RB; ++q)
    if (g * RB + q < HL) {
      double* o = out + ((int64_t)blockIdx.y * HL + g * RB + q) * C + c;
#pragma unroll
      for (int w = 0; w < V; ++w) o[w] = acc[q][w];
    }
}

template <int TILE>
cudaError_t launch_slice(const double* X, int K, int64_t M, int64_t ld, const int* kexp, int sgn, unsigned char* img,
                         int2* expo, unsigned char* mag, const int2* range, int* power, int* counter, cudaStream_t s) {
  const int64_t Mpad = (M + TILE - 1) / TILE * TILE;
  const int64_t blocks = Mpad / kSliceCols;
  slice_f64_kernel<TILE><<<(unsigned)(blocks < 65535 ? blocks : 65535), 256, 0, s>>>(
      X, K, M, ld, kexp, sgn, ttm_ksteps(K), Mpad, img, expo, mag, range, power, counter);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_slice_exponents(const double* Tn, int64_t I, int64_t J, int* kexp, int* bad, cudaStream_t s) {
  slice_exponent_kernel<<<(unsigned)I, 256, 0, s>>>(Tn, J, kexp, bad);
  return cudaGetLastError();
}

cudaError_t launch_range(const int* kexp, int K, const int2* rexp, int64_t J, int2* range, cudaStream_t s) {
  range_kernel<<<1, 1024, 0, s>>>(kexp, K, rexp, J, range);
  return cudaGetLastError();
}

cudaError_t launch_slice_tensor(const double* Tn, int I, int64_t J, const int* kexp, unsigned char* Bt, int2* rexp,
                                unsigned char* rmag, cudaStream_t s) {
  return ttm_tile_r(I) == 32 ? launch_slice<32>(Tn, I, J, J, kexp, -1, Bt, rexp, rmag, nullptr, nullptr, nullptr, s)
                             : launch_slice<64>(Tn, I, J, J, kexp, -1, Bt, rexp, rmag, nullptr, nullptr, nullptr, s);
}

cudaError_t launch_slice_factor(const double* U, int I, int C, const int* kexp, unsigned char* At, int2* cexp,
                                unsigned char* cmag, const int2* range, int* power, int* counter, cudaStream_t s) {
  return launch_slice<kTileM>(U, I, C, C, kexp, +1, At, cexp, cmag, range, power, counter, s);
}

cudaError_t prepare_ttm(int K) {
  return cudaFuncSetAttribute(ttm_tile_r(K) == 32 ? ttm_kernel<32> : ttm_kernel<64>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
}

cudaError_t launch_ttm(const TtmArgs& a, int num_sms, cudaStream_t s) {
  const int64_t tiles = (int64_t)a.tiles_c * a.tiles_r;
  const unsigned grid = (unsigned)(tiles < num_sms ? tiles : num_sms);
  if (ttm_tile_r(a.K) == 32)
    ttm_kernel<32><<<grid, kThreads, kSmem, s>>>(a);
  else
    ttm_kernel<64><<<grid, kThreads, kSmem, s>>>(a);
  return cudaGetLastError();
}

// Shape of a contraction: two columns per 16-byte load where C is even, four rows of
// outputs per thread where enough threads remain, and m split to fill the SMs, at least
// eight terms each.  A large X wants about 1280 threads per SM in flight (400x400x400,
// 400 columns: 128 us, with 512 per SM 165 us); a small one 512, as every split lengthens
// the sums of the update that follows.
namespace {
constexpr int64_t kContractSms = 152, kLargeX = 64ll << 20;

int contract_vec(int C) { return C % 2 == 0 ? 2 : 1; }

int contract_rb(int64_t HL, int Mm, int C, int V) {
  return HL >= 4 && (HL + 3) / 4 * (C / V) * ((Mm + 7) / 8) >= kContractSms * 512 ? 4 : 1;
}
}  // namespace

int contract_splits(int64_t HL, int Mm, int C) {
  const int V = contract_vec(C), RB = contract_rb(HL, Mm, C, V);
  const int64_t threads = (HL + RB - 1) / RB * (C / V);
  const int64_t want = kContractSms * (HL * Mm * C * 8 > kLargeX ? 1280 : 512);
  int64_t S = (want + threads - 1) / threads;
  if (S > (Mm + 7) / 8) S = (Mm + 7) / 8;
  if (S > 65535) S = 65535;   // grid.y
  if (S < 1) S = 1;
  const int chunk = (int)((Mm + S - 1) / S);
  return (Mm + chunk - 1) / chunk;
}

cudaError_t launch_contract(const double* X, int64_t H, int Mm, int64_t L, int C, const double* U, int S,
                            const int* power, int* out_power, double* out, cudaStream_t s) {
  const int64_t HL = H * L;
  const int chunk = (Mm + S - 1) / S;
  const int V = contract_vec(C), RB = contract_rb(HL, Mm, C, V);
  const dim3 grid((unsigned)(((HL + RB - 1) / RB * (C / V) + 255) / 256), (unsigned)S);
  if (RB == 4 && V == 2)
    contract_kernel<4, 2><<<grid, 256, 0, s>>>(X, H, Mm, L, C, U, chunk, power, out_power, out);
  else if (RB == 4)
    contract_kernel<4, 1><<<grid, 256, 0, s>>>(X, H, Mm, L, C, U, chunk, power, out_power, out);
  else if (V == 2)
    contract_kernel<1, 2><<<grid, 256, 0, s>>>(X, H, Mm, L, C, U, chunk, power, out_power, out);
  else
    contract_kernel<1, 1><<<grid, 256, 0, s>>>(X, H, Mm, L, C, U, chunk, power, out_power, out);
  return cudaGetLastError();
}

}  // namespace jk
