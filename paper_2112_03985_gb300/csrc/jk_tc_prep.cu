// Create-time operand preparation for the tensor-core MTTKRP: the padded,
// precision-split unfoldings, the transposed FP32 factor copies, and the
// per-row grids (row exponents, column maxima) of the exact-chain form.
#include <cuda_bf16.h>

#include <type_traits>

#include "jk_tc.cuh"

namespace jk {
namespace tc {
namespace {

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// One CTA per row: max |T| -> smallest F with max < 2^F.
__global__ void row_exponent_kernel(const double* __restrict__ Tn, int64_t J, int* __restrict__ rowexp) {
  __shared__ double red[256];
  const int64_t i = blockIdx.x;
  double m = 0.0;
  for (int64_t j = threadIdx.x; j < J; j += blockDim.x) m = fmax(m, fabs(Tn[i * J + j]));
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    int e = 0;
    if (red[0] > 0.0) frexp(red[0], &e);   // max = f 2^e, f in [0.5, 1) -> max < 2^e
    rowexp[i] = e;
  }
}

// Byte offset of element (r, col) of one part tile (BN rows x ROW bytes,
// K-major) in the ROW-byte swizzle of the MMA's shared-memory operands: rows
// in groups of 8 (8 * ROW bytes apart), the 16-byte chunk index XORed with
// the row (ROW = 128) or with row / 2 (ROW = 64).
__device__ __forceinline__ int64_t swizzled_offset(int r, int cb, int row_bytes) {
  const int sw = row_bytes == 128 ? (r & 7) : ((r >> 1) & 3);
  return (int64_t)(r >> 3) * (8 * row_bytes) + (int64_t)(r & 7) * row_bytes + (((cb >> 4) ^ sw) << 4) + (cb & 15);
}

// Tt holds, for N tile t and k-step s, the parts of rows t*BN .. t*BN+BN-1 and
// padded columns s*BK .. s*BK+BK-1 (see jk_tc.cuh).  Logical element (i, jp):
// jp = ia + Ia_pad * o with ia the index of the fastest mode a and o running
// mixed-radix over the remaining modes in increasing order; j is the Eq.
// kolda_mapping column of those indices; zero where i >= I, jp >= Jp or
// ia >= Ia.  Splits are taken from the FP64 value.  IT: 32-bit indices where the padded
// unfolding has fewer than 2^31 entries (six divisions per entry).
template <int PREC, typename IT>
__global__ void tile_unfold_kernel(const double* __restrict__ Tn, IT I, IT J, IT Ia, IT Ia_pad, IT Jp, UnfoldMap mp,
                                   const int* __restrict__ rowexp, int BN, int tiles_n, IT nkt,
                                   unsigned char* __restrict__ Tt) {
  constexpr int EB = (PREC == JKCALS_TF32 || PREC == JKCALS_3XTF32) ? 4 : 2;
  constexpr int ROW = PREC == JKCALS_EXACT_BF16 ? 64 : 128;
  constexpr int BK = ROW / EB;
  constexpr int NS = PREC == JKCALS_EXACT_BF16 ? 4 : (PREC == JKCALS_SPLIT_BF16 ? 3 : (PREC == JKCALS_3XTF32 ? 2 : 1));
  const IT cols = nkt * BK;
  const int64_t total = (int64_t)tiles_n * BN * cols;
  const int64_t part_bytes = (int64_t)BN * ROW;
  for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e0 < total;
       e0 += (int64_t)gridDim.x * blockDim.x) {
    const IT e = (IT)e0;
    const IT i = e / cols;
    const IT jp = e - i * cols;
    double x = 0.0;
    if (i < I && jp < Jp) {
      const IT o = jp / Ia_pad;
      const IT ia = jp - o * Ia_pad;
      if (ia < Ia) {
        IT j = ia * (IT)mp.sa, rem = o;
        for (int t = 0; t < mp.nq; ++t) {
          const IT qd = (IT)mp.qd[t], qq = rem / qd;
          j += (rem - qq * qd) * (IT)mp.qs[t];
          rem = qq;
        }
        x = Tn[(int64_t)i * J + j];
      }
    }
    float v[NS];
    if constexpr (PREC == JKCALS_TF32 || PREC == JKCALS_3XTF32) {
      const float h = tf32_rna((float)x);
      v[0] = h;
      if constexpr (NS > 1) v[1] = tf32_rna((float)(x - (double)h));
    } else if constexpr (PREC == JKCALS_EXACT_BF16) {
      // x = 2^(F-7) (s0 + s1 2^-7 + s2 2^-14 + s3 2^-21), |s_k| <= 128, stored as s_k 2^(-7k)
      const long long xb = __double_as_longlong(x);
      const int ef = (int)((xb >> 52) & 2047);
      const int sc = i < I ? kSliceBits - rowexp[i] : 0;
      if ((xb & 0x1fffffff) == 0 && (ef != 0 || (xb << 1) == 0) && ef != 2047) {
        // x has at most FP32's 24 significant bits (a tensor given in FP32): y is an
        // FP32 number, and every step below is exact there as in FP64 (whose rint and
        // ldexp sequences and 64-bit divisions took 75-80 us per mode of 300x100x50; a
        // job on it, create included, went from 5.66 to 5.49 ms).  y below FP32's normal
        // range has no digits.
        const int ey = ef - 896 + sc;   // biased FP32 exponent of y, at most 127 + 6
        float y = 0.f;
        if (ef != 0 && ey > 0)
          y = __int_as_float((int)((xb >> 32) & 0x80000000ll) | (ey << 23) | (int)((xb >> 29) & 0x7fffff));
        constexpr float kRound = 12582912.f;   // 1.5 * 2^23: rounds to the nearest even integer
        float unit = 1.f;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float d = __fsub_rn(__fadd_rn(y, kRound), kRound);
          v[s] = d * unit;
          y = __fsub_rn(y, d) * 128.f;
          unit *= 0.0078125f;
        }
      } else {
        double y = i < I ? ldexp(x, sc) : 0.0;
        const double s0 = rint(y);
        y = (y - s0) * 128.0;
        const double s1 = rint(y);
        y = (y - s1) * 128.0;
        const double s2 = rint(y);
        y = (y - s2) * 128.0;
        const double s3 = rint(y);
        v[0] = (float)s0;
        v[1] = (float)(s1 / 128.0);
        v[2] = (float)(s2 / 16384.0);
        v[3] = (float)(s3 / 2097152.0);
      }
    } else {
      const float h = __bfloat162float(__double2bfloat16(x));
      v[0] = h;
      if constexpr (NS > 1) {
        const double r1 = x - (double)h;
        const float m = __bfloat162float(__double2bfloat16(r1));
        v[1] = m;
        v[2] = __bfloat162float(__double2bfloat16(r1 - (double)m));
      }
    }
    const IT tn = i / (IT)BN, ks = jp / BK;
    const int r = (int)(i - tn * (IT)BN), col = (int)(jp - ks * BK);
    const int64_t tile = ((int64_t)tn * nkt + ks) * NS * part_bytes;
    const int64_t off = swizzled_offset(r, col * EB, ROW);
#pragma unroll
    for (int p = 0; p < NS; ++p) {
      unsigned char* dst = Tt + tile + p * part_bytes + off;
      if constexpr (EB == 4)
        *reinterpret_cast<float*>(dst) = v[p];
      else
        *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(v[p]);   // exact: v[p] is a BF16 value
    }
  }
}

__global__ void factor_to_ut_kernel(const double* __restrict__ U, int64_t I, int C, float* __restrict__ UT,
                                    float* __restrict__ UT_lo, int64_t I_pad) {
  const int64_t total = I * (int64_t)C;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = e / I;
    const int64_t i = e - c * I;
    const double u = U[i * C + c];
    const float hi = (float)u;
    UT[c * I_pad + i] = hi;
    if (UT_lo != nullptr) UT_lo[c * I_pad + i] = (float)(u - (double)hi);
  }
}

// One warp per column.
__global__ void colmax_kernel(const float* __restrict__ UT, int64_t I, int64_t I_pad, int C,
                              float* __restrict__ cmax) {
  const int c = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  float m = 0.f;
  for (int64_t i = lane; i < I; i += 32) m = fmaxf(m, fabsf(UT[(int64_t)c * I_pad + i]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) cmax[c] = m;
}

inline unsigned grid_for(int64_t total) {
  int64_t b = (total + 255) / 256;
  if (b > 65535 * 8) b = 65535 * 8;
  return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t launch_row_exponent(const double* Tn64, int64_t I, int64_t J, int* rowexp, cudaStream_t s) {
  row_exponent_kernel<<<(unsigned)I, 256, 0, s>>>(Tn64, J, rowexp);
  return cudaGetLastError();
}

cudaError_t launch_tile_unfold(int precision, const double* Tn64, int64_t I, int64_t J, int64_t Ia, int64_t Ia_pad,
                               int64_t Jp, const UnfoldMap& mp, const int* rowexp, int BN, int tiles_n, int64_t nkt,
                               void* Tt, cudaStream_t s) {
  const int64_t total = (int64_t)tiles_n * BN * nkt * form_bk(precision);
  const unsigned g = grid_for(total);
  unsigned char* out = static_cast<unsigned char*>(Tt);
  auto go = [&](auto prec) {
    constexpr int PREC = decltype(prec)::value;
    if (total < 2147483647LL && I * J < 2147483647LL)
      tile_unfold_kernel<PREC, uint32_t><<<g, 256, 0, s>>>(Tn64, (uint32_t)I, (uint32_t)J, (uint32_t)Ia,
                                                           (uint32_t)Ia_pad, (uint32_t)Jp, mp, rowexp, BN, tiles_n,
                                                           (uint32_t)nkt, out);
    else
      tile_unfold_kernel<PREC, int64_t><<<g, 256, 0, s>>>(Tn64, I, J, Ia, Ia_pad, Jp, mp, rowexp, BN, tiles_n, nkt, out);
    return cudaGetLastError();
  };
  switch (precision) {
    case JKCALS_TF32: return go(std::integral_constant<int, JKCALS_TF32>{});
    case JKCALS_3XTF32: return go(std::integral_constant<int, JKCALS_3XTF32>{});
    case JKCALS_BF16: return go(std::integral_constant<int, JKCALS_BF16>{});
    case JKCALS_SPLIT_BF16: return go(std::integral_constant<int, JKCALS_SPLIT_BF16>{});
    case JKCALS_EXACT_BF16: return go(std::integral_constant<int, JKCALS_EXACT_BF16>{});
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_factor_to_ut(const double* U, int64_t I, int C, float* UT, float* UT_lo, int64_t I_pad,
                                cudaStream_t s) {
  factor_to_ut_kernel<<<grid_for(I * (int64_t)C), 256, 0, s>>>(U, I, C, UT, UT_lo, I_pad);
  return cudaGetLastError();
}

cudaError_t launch_colmax(const float* UT, int64_t I, int64_t I_pad, int C, float* cmax, cudaStream_t s) {
  colmax_kernel<<<(unsigned)((C + 7) / 8), 256, 0, s>>>(UT, I, I_pad, C, cmax);
  return cudaGetLastError();
}

}  // namespace tc
}  // namespace jk
