// te_quant.cu - rounding of binary64 matrix values to the storage types of
// the mixed-precision forms (Section III-A): binary32, bfloat16, and FP8 E4M3
// with one binary32 scale per row.
//
// Round to nearest, ties to even, from the binary64 value directly (no
// intermediate binary32 rounding); a zero result is +0.  For |x| in
// [2^e, 2^(e+1)) and p significant bits the quantum is 2^(e+1-p), never below
// the format's smallest subnormal; |x| / quantum is exact and rint() rounds
// it to the nearest integer, ties to even.  FP8: scale_r = binary32 of
// max_j |a_rj| / 448 (1 for an all-zero row), code = round(a / scale_r)
// saturated at 448 (the largest finite E4M3 value).
#include "te_common.cuh"
#include "te_internal.h"

namespace te {

// GB300 runs binary64 at a small fraction of its other rates (a warp's
// instruction holds its scheduler's unit for 64 cycles, a division takes about
// 570), so the codes are found with integers and binary32 where those decide
// them for certain, and by the definition above (round_sig) elsewhere: outside
// binary32's normal range, and within the estimate's error of a tie.
//   - binary32 and bfloat16: round to nearest even on the binary64 pattern;
//   - E4M3: |a| / scale estimated in binary32 (relative error below 2^-21)
//     is rounded unless it lies within 2^-19 of the middle of two codes; the
//     scale is the rounded head of max|a| / 448 in double-float (error below
//     2^-44) unless the tail is within 2^-16 of half a unit of the head.
// 23 M entries, 1 M rows: E4M3 4,970 us with a binary64 division per entry and
// 420 us now, bfloat16 1,344 and 139 us.
TE_DEV double round_sig(double ax, int p, int qmin) {
  int qe = ilogb(ax) + 1 - p;
  if (qe < qmin) qe = qmin;
  const double q = scalbn(1.0, qe);
  return rint(ax / q) * q;
}

__device__ __noinline__ uint16_t bf16_code_exact(double x) {
  const double ax = fabs(x);
  if (!(ax > 0.0)) return 0;
  const double r = round_sig(ax, 8, -133);
  if (r == 0.0) return 0;
  const uint32_t bits = __float_as_uint((float)r);  // exact: 8 significant bits
  return (uint16_t)((bits >> 16) | (x < 0.0 ? 0x8000u : 0u));
}

TE_DEV uint8_t e4m3_code_exact(double x) {
  const double ax = fabs(x);
  if (!(ax > 0.0)) return 0;
  double r = round_sig(ax, 4, -9);
  if (r > 448.0) r = 448.0;
  if (r == 0.0) return 0;
  uint32_t code;
  if (r < 0x1p-6) {
    code = (uint32_t)(r * 512.0);  // subnormal: m * 2^-9, m in 1..7
  } else {
    const int e = ilogb(r);
    code = ((uint32_t)(e + 7) << 3) | ((uint32_t)scalbn(r, 3 - e) - 8u);
  }
  return (uint8_t)(code | (x < 0.0 ? 0x80u : 0u));
}

__device__ __noinline__ uint8_t e4m3_quotient_exact(double v, float s) {
  return e4m3_code_exact(v / (double)s);
}
__device__ __noinline__ float e4m3_scale_exact(double mx) {
  return __double2float_rn(mx / 448.0);
}

TE_DEV uint16_t bf16_code(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - 897u > 1150u - 897u) return bf16_code_exact(x);
  const unsigned c = ((e - 896u) << 7) | ((hi >> 13) & 0x7fu), rem = hi & 0x1fffu;
  const unsigned up = (rem > 0x1000u || (rem == 0x1000u && (lo != 0u || (c & 1u)))) ? 1u : 0u;
  return (uint16_t)((c + up) | ((hi >> 31) << 15));  // (a carry out of the largest is infinity)
}

// scale of a row with largest magnitude mx
TE_DEV float e4m3_scale(double mx) {
  if (!(mx > 0.0)) return 1.0f;
  const unsigned e = ((unsigned)__double2hiint(mx) >> 20) & 0x7ffu;
  if (e - 930u > 1140u - 930u) return e4m3_scale_exact(mx);
  const float ih = 0x1.24924ap-9f;                                // 1 / 448 =
  const float il = (float)(1.0 / 448.0 - 0x1.24924ap-9);          //   ih + il
  const float mh = f_head(mx), ml = f_tail(mx);
  float p, q;
  two_prod(mh, ih, p, q);
  q = __fadd_rn(q, __fmaf_rn(mh, il, __fmul_rn(ml, ih)));
  float zh, zl;
  fast_two_sum(p, q, zh, zl);
  // half a unit in the last place of zh
  const float half = __uint_as_float((__float_as_uint(zh) & 0x7f800000u) - (24u << 23));
  // (a power of two has a finer spacing below it)
  if (!(fabsf(zl) < 0.5f * half * (2.0f - 0x1p-15f)) || (__float_as_uint(zh) & 0x7fffffu) == 0u)
    return e4m3_scale_exact(mx);
  return zh;
}

// code of v in a row of scale s; is = 1 / s to binary32
TE_DEV uint8_t e4m3_code(double v, float s, float is) {
  const unsigned hi = (unsigned)__double2hiint(v);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if ((hi & 0x7fffffffu) == 0u && __double2loint(v) == 0) return 0;
  const float q = __fmul_rn(f_head(fabs(v)), is);
  const unsigned es = (__float_as_uint(s) >> 23) & 0xffu;
  bool fine = e - 930u <= 1110u - 930u && es - 30u <= 220u - 30u;
  unsigned c;
  if (q < 0x1p-6f) {  // a multiple of 2^-9
    const float t = q * 512.0f, r = rintf(t);
    c = (unsigned)r;
    fine = fine && fabsf(fabsf(t - r) - 0.5f) > t * 0x1p-19f + 0x1p-40f;
  } else {
    const unsigned b = __float_as_uint(q), rem = b & 0xfffffu;
    fine = fine && rem - (0x80000u - 32u) > 64u;
    c = min((b + 0x80000u) >> 20, (unsigned)((127 + 8) << 3 | 6)) - (120u << 3);
  }
  if (!fine) return e4m3_quotient_exact(v, s);
  return c == 0u ? 0 : (uint8_t)(c | ((hi >> 31) << 7));
}

__global__ void round_f32_kernel(const double* v, int64_t nnz, float* out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
       k += (int64_t)gridDim.x * blockDim.x)
    out[k] = f32_from_f64(v[k]);
}

__global__ void round_bf16_kernel(const double* v, int64_t nnz, uint16_t* out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
       k += (int64_t)gridDim.x * blockDim.x)
    out[k] = bf16_code(v[k]);
}

// one warp per row: the row's largest magnitude gives its scale
__global__ void quant_e4m3_kernel(const int64_t* rp, const double* v, int64_t n, uint8_t* out,
                                  float* scale) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < n;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t a = rp[r], b = rp[r + 1];
    long long mb = 0;  // magnitudes compare as integers; a NaN does not count, as in fmax
    for (int64_t k = a + lane; k < b; k += 32) {
      const long long m = __double_as_longlong(v[k]) & INT64_MAX;
      if (m > mb && m <= 0x7ff0000000000000ll) mb = m;
    }
    for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    const float s = e4m3_scale(__longlong_as_double(mb));
    const float is = __frcp_rn(s);
    if (lane == 0) scale[r] = s;
    for (int64_t k = a + lane; k < b; k += 32) out[k] = e4m3_code(v[k], s, is);
  }
}

cudaError_t launch_quantize(int to, const int64_t* rp, const double* val, int64_t n, int64_t nnz,
                            void* out, float* row_scale, cudaStream_t s) {
  const int threads = 256;
  if (to == TE_FP8_E4M3) {
    int64_t blocks = (n * 32 + threads - 1) / threads;
    if (blocks > 65536) blocks = 65536;
    if (blocks < 1) blocks = 1;
    quant_e4m3_kernel<<<(int)blocks, threads, 0, s>>>(rp, val, n, static_cast<uint8_t*>(out),
                                                       row_scale);
    return cudaGetLastError();
  }
  if (nnz <= 0) return cudaSuccess;
  int64_t blocks = (nnz + threads - 1) / threads;
  if (blocks > 65536) blocks = 65536;
  if (to == TE_BF16)
    round_bf16_kernel<<<(int)blocks, threads, 0, s>>>(val, nnz, static_cast<uint16_t*>(out));
  else if (to == TE_F32)
    round_f32_kernel<<<(int)blocks, threads, 0, s>>>(val, nnz, static_cast<float*>(out));
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace te
