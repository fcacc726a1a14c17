// te_refine.cu - binary64 Rayleigh-quotient refinement of the selected Ritz
// pairs, and the Gram matrix of a set of vectors (orthogonality metric).
//
// Refinement (for the mixed-precision forms): the Ritz vector u of a Ritz
// value theta is an approximate eigenvector of M; its Rayleigh quotient
// u'Mu / u'u against the binary64 matrix is a better eigenvalue estimate
// (the error is quadratic in the vector's error), and ||Mu - theta' u|| /
// ||u|| is the reconstruction error the paper reports (Section IV-D).  With
// y = M u and r = y - theta u (small, so no cancellation),
//   theta' = theta + u'r / u'u,   ||y - theta' u||^2 = r'r - (u'r)^2 / u'u.
//
// The products of up to eight vectors are taken together: the vectors lie by
// rows, so an entry (row, column) of the SpMV layout gathers one contiguous
// piece of the vectors' row for all of them, the matrix is read once per
// eight vectors, and the row of y goes straight from registers into the sums
// u'r, u'u, r'r (y is never stored).  A product per vector re-read the matrix
// and gathered 8 bytes per 32-byte sector every time.  Bound: binary64
// multiply-adds (a warp's instruction holds its scheduler's unit for 64
// cycles): R-MAT 2^22, 128 M entries, 16 vectors 6.0 ms against 9.7 ms, of
// which 4.1 are the multiply-adds.
// Per-block partial sums are added by the last block in a fixed order, so the
// result does not depend on scheduling.
#include <algorithm>

#include "te_common.cuh"
#include "te_internal.h"

namespace te {

constexpr int RQ_THREADS = 256;
constexpr int RQ_WARPS = RQ_THREADS / 32;

int refine_grid(int num_sms) { return num_sms * 2; }

// A lane holds NV vectors (1 or 2) of a row and LG lanes hold a row's LG * NV.
// `U`: vectors by rows, K of them with stride Kr; this launch takes vectors
// k0 ... k0 + LG * NV - 1 (those below K).
struct RefineArgs {
  LzState* st;
  const SellSlice* slices;
  const int32_t* vout;
  const int32_t* cols;
  const double* vals;
  const LongRow* lrows;
  const double* U;
  const unsigned char* filled;  // rows with entries
  double* vpart;                // cut rows' pieces: LG * NV sums each
  double* part;                 // [block][vector][3]: u'r, u'u, r'r
  int64_t n;
  int nslices, nlrows, K, Kr, k0, blocks;  // blocks: of the product kernel
};

template <int NV>
struct RefineVec {
  double v[NV];
};
template <int NV>
TE_DEV RefineVec<NV> refine_load(const RefineArgs& a, int64_t row, int k) {
  RefineVec<NV> x;
  const double* p = a.U + row * a.Kr + k;
  if constexpr (NV == 2) {  // (k is even and Kr too: 16-byte aligned)
    const double2 d = k < a.K ? __ldg(reinterpret_cast<const double2*>(p)) : make_double2(0., 0.);
    x.v[0] = d.x;
    x.v[1] = d.y;
  } else {
    x.v[0] = k < a.K ? __ldg(p) : 0.0;
  }
  return x;
}

// a lane's sums of u'r, u'u, r'r over its rows
template <int NV>
struct RefineSums {
  double ur[NV], uu[NV], rr[NV];
  TE_DEV void init() {
#pragma unroll
    for (int q = 0; q < NV; ++q) ur[q] = uu[q] = rr[q] = 0.0;
  }
  TE_DEV void row(const RefineVec<NV>& u, const RefineVec<NV>& y, const double* th) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const double res = fma(-th[q], u.v[q], y.v[q]);
      ur[q] = fma(u.v[q], res, ur[q]);
      uu[q] = fma(u.v[q], u.v[q], uu[q]);
      rr[q] = fma(res, res, rr[q]);
    }
  }
};

// the block's sums into part[block] (warps in order)
template <int LG, int NV>
TE_DEV void refine_block_sums(RefineSums<NV>& s, double* part, double (*red)[LG * NV * 3]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
#pragma unroll
    for (int o = 16; o >= LG; o >>= 1) {
      s.ur[q] += __shfl_xor_sync(0xffffffffu, s.ur[q], o);
      s.uu[q] += __shfl_xor_sync(0xffffffffu, s.uu[q], o);
      s.rr[q] += __shfl_xor_sync(0xffffffffu, s.rr[q], o);
    }
    if (lane < LG) {
      double* d = red[wid] + (lane * NV + q) * 3;
      d[0] = s.ur[q];
      d[1] = s.uu[q];
      d[2] = s.rr[q];
    }
  }
  __syncthreads();
  if (threadIdx.x < LG * NV * 3) {
    double t = 0.0;
    for (int w = 0; w < RQ_WARPS; ++w) t += red[w][threadIdx.x];
    part[(size_t)blockIdx.x * LG * NV * 3 + threadIdx.x] = t;
  }
}

constexpr int RQ_UNROLL = 8;  // entries in flight per lane

// Warps walk the slices of the SpMV layout; 32 / LG pieces of a slice at a
// time, LG rounds.  The two chains per sum and their order are the SpMV's.
template <int LG, int NV>
__global__ void __launch_bounds__(RQ_THREADS) refine_product_kernel(RefineArgs a) {
  __shared__ double red[RQ_WARPS][LG * NV * 3];
  constexpr int PW = 32 / LG;
  const int lane = threadIdx.x & 31, sub = lane % LG, pi = lane / LG;
  const int k = a.k0 + sub * NV;
  double th[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) th[q] = k + q < a.K ? a.st->theta_sel[k + q] : 0.0;
  RefineSums<NV> sums;
  sums.init();
  const uint64_t pol = policy_evict_first();
  for (int64_t sl = blockIdx.x * (int64_t)RQ_WARPS + (threadIdx.x >> 5); sl < a.nslices;
       sl += (int64_t)gridDim.x * RQ_WARPS) {
    const SellSlice S = a.slices[sl];
    for (int rnd = 0; rnd < LG; ++rnd) {
      const int piece = rnd * PW + pi;
      const int32_t out = a.vout[sl * SELL_C + piece];
      const int32_t* cp = a.cols + S.base + piece;
      const double* vp = a.vals + S.base + piece;
      double acc[2][NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) acc[0][q] = acc[1][q] = 0.0;
      for (int e = 0; e < S.len; e += RQ_UNROLL) {
        int32_t c[RQ_UNROLL];
        double v[RQ_UNROLL];
#pragma unroll
        for (int u = 0; u < RQ_UNROLL; ++u) {
          const bool ok = e + u < S.len;
          c[u] = ok ? ld_stream_i32(cp + (int64_t)(e + u) * SELL_C, pol) : 0;
          v[u] = ok ? ld_stream_f64(vp + (int64_t)(e + u) * SELL_C, pol) : 0.0;
        }
        RefineVec<NV> x[RQ_UNROLL];
#pragma unroll
        for (int u = 0; u < RQ_UNROLL; ++u)
          if (e + u < S.len) x[u] = refine_load<NV>(a, c[u], k);
#pragma unroll
        for (int u = 0; u < RQ_UNROLL; ++u)
          if (e + u < S.len)  // (uniform: no binary64 instruction for the tail)
#pragma unroll
            for (int q = 0; q < NV; ++q) acc[u & 1][q] = fma(v[u], x[u].v[q], acc[u & 1][q]);
      }
      RefineVec<NV> y;
#pragma unroll
      for (int q = 0; q < NV; ++q) y.v[q] = acc[0][q] + acc[1][q];
      if (out >= 0) {
        sums.row(refine_load<NV>(a, out, k), y, th);
      } else if (out != SELL_SKIP) {
        double* d = a.vpart + ((int64_t)(-1 - (int64_t)out) * LG + sub) * NV;
#pragma unroll
        for (int q = 0; q < NV; ++q) d[q] = y.v[q];
      }
    }
  }
  refine_block_sums<LG, NV>(sums, a.part, red);
}

// Cut rows (a warp per row: the lanes' strided pieces, then a shuffle tree)
// and rows without entries (y = 0); the last block adds every block's sums
// and writes theta', the residual and the eigenvalue outputs.
template <int LG, int NV>
__global__ void __launch_bounds__(RQ_THREADS) refine_finish_kernel(RefineArgs a) {
  __shared__ double red[RQ_WARPS][LG * NV * 3];
  __shared__ double tot[LG * NV * 3];
  __shared__ int last;
  constexpr int PW = 32 / LG;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, sub = lane % LG, pi = lane / LG;
  const int k = a.k0 + sub * NV;
  LzState* st = a.st;
  double th[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) th[q] = k + q < a.K ? st->theta_sel[k + q] : 0.0;
  RefineSums<NV> sums;
  sums.init();
  const int64_t w0 = blockIdx.x * (int64_t)RQ_WARPS + wid, nw = (int64_t)gridDim.x * RQ_WARPS;
  for (int64_t r = w0; r < a.nlrows; r += nw) {
    const LongRow lr = a.lrows[r];
    RefineVec<NV> y;
#pragma unroll
    for (int q = 0; q < NV; ++q) y.v[q] = 0.0;
    for (int c = pi; c < lr.count; c += PW) {
      const double* d = a.vpart + ((int64_t)(lr.first + c) * LG + sub) * NV;
#pragma unroll
      for (int q = 0; q < NV; ++q) y.v[q] += d[q];
    }
#pragma unroll
    for (int q = 0; q < NV; ++q)
#pragma unroll
      for (int o = 16; o >= LG; o >>= 1) y.v[q] += __shfl_xor_sync(0xffffffffu, y.v[q], o);
    if (pi == 0) sums.row(refine_load<NV>(a, lr.row, k), y, th);
  }
  for (int64_t r = w0 * PW + pi; r < a.n; r += nw * PW) {
    if (a.filled[r]) continue;
    RefineVec<NV> y;
#pragma unroll
    for (int q = 0; q < NV; ++q) y.v[q] = 0.0;
    sums.row(refine_load<NV>(a, r, k), y, th);
  }
  refine_block_sums<LG, NV>(sums, a.part + (size_t)a.blocks * LG * NV * 3, red);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int nb = a.blocks + (int)gridDim.x;
  for (int q = wid; q < LG * NV * 3; q += RQ_WARPS) {
    double t = 0.0;
    for (int blk = lane; blk < nb; blk += 32) t += __ldcg(a.part + (size_t)blk * LG * NV * 3 + q);
    t = warp_sum(t);
    if (lane == 0) tot[q] = t;
  }
  __syncthreads();
  const int kk = a.k0 + threadIdx.x;
  if (threadIdx.x < LG * NV && kk < a.K) {
    const double ur = tot[3 * threadIdx.x], uu = tot[3 * threadIdx.x + 1],
                 rr = tot[3 * threadIdx.x + 2];
    double thn = st->theta_sel[kk], res = 0.0;
    if (uu > 0.0) {
      thn += ur / uu;
      const double q = rr - ur * ur / uu;
      res = sqrt(q > 0.0 ? q : 0.0) / sqrt(uu);
    }
    st->theta_sel[kk] = thn;
    st->resid_est[kk] = res;
    if (st->eigvals_out) st->eigvals_out[kk] = thn;
  }
  if (threadIdx.x == 0) st->ticket = 0;
}

// filled[r] = 1 for the rows that a lane or a cut row writes
__global__ void refine_mark_kernel(const int32_t* vout, int64_t lanes, const LongRow* lrows,
                                   int nlrows, unsigned char* filled) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < lanes + nlrows;
       i += stride) {
    if (i < lanes) {
      const int32_t r = vout[i];
      if (r >= 0) filled[r] = 1;
    } else {
      filled[lrows[i - lanes].row] = 1;
    }
  }
}

template <int LG, int NV>
static cudaError_t refine_chunk(RefineArgs& a, int fin_blocks, cudaStream_t s) {
  refine_product_kernel<LG, NV><<<a.blocks, RQ_THREADS, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  refine_finish_kernel<LG, NV><<<fin_blocks, RQ_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_refine(LzState* st, const DevSell& S, int64_t n, int K, const double* U,
                          int64_t pieces, void* scratch, size_t scratch_bytes,
                          unsigned char* filled, int num_sms, int* kernels, cudaStream_t s) {
  RefineArgs a;
  a.st = st;
  a.slices = S.slices;
  a.vout = S.vout;
  a.cols = S.cols;
  a.vals = static_cast<const double*>(S.vals);
  a.lrows = S.lrows;
  a.U = U;
  a.filled = filled;
  a.n = n;
  a.nslices = S.nslices;
  a.nlrows = S.nlrows;
  a.K = K;
  a.Kr = (K + 1) & ~1;
  *kernels = 1;
  cudaError_t e = cudaMemsetAsync(filled, 0, (size_t)n, s);
  if (e != cudaSuccess) return e;
  const int64_t lanes = (int64_t)S.nslices * SELL_C;
  const int64_t marks = std::max<int64_t>((lanes + S.nlrows + 255) / 256, 1);
  refine_mark_kernel<<<(unsigned)std::min<int64_t>(marks, 8 * num_sms), 256, 0, s>>>(
      S.vout, lanes, S.lrows, S.nlrows, filled);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // as many vectors at a time as leave no lane idle and as the scratch (the
  // basis, free by now) holds the cut rows' sums of; at least one, whose sums
  // the plan's own array holds
  for (int k0 = 0; k0 < K;) {
    const int left = K - k0;
    int nv = left > 4 ? 8 : left > 2 ? 4 : left;
    // the blocks' sums come first
    auto need = [&](int v, int blocks) {
      return (size_t)blocks * v * 3 * sizeof(double) + (size_t)pieces * v * sizeof(double);
    };
    int pb = (int)std::min<int64_t>(std::max<int64_t>((S.nslices + RQ_WARPS - 1) / RQ_WARPS, 1),
                                    (int64_t)num_sms * 4);
    int fb = (int)std::min<int64_t>(
        std::max<int64_t>((n + 32 * RQ_WARPS - 1) / (32 * RQ_WARPS), 1), (int64_t)num_sms * 2);
    while (nv > 1 && need(nv, pb + fb) > scratch_bytes) nv /= 2;
    const size_t room = scratch_bytes / ((size_t)nv * 3 * sizeof(double));
    if ((size_t)(pb + fb) > room) {  // (a basis of a few tiles)
      pb = (int)std::max<size_t>(std::min<size_t>((size_t)pb, room / 2), 1);
      fb = (int)std::max<size_t>(std::min<size_t>((size_t)fb, room / 2), 1);
    }
    a.k0 = k0;
    a.blocks = pb;
    a.part = static_cast<double*>(scratch);
    a.vpart = nv > 1 ? a.part + (size_t)(pb + fb) * nv * 3 : static_cast<double*>(S.vpart);
    e = nv == 8   ? refine_chunk<4, 2>(a, fb, s)
        : nv == 4 ? refine_chunk<2, 2>(a, fb, s)
        : nv == 2 ? refine_chunk<1, 2>(a, fb, s)
                  : refine_chunk<1, 1>(a, fb, s);
    if (e != cudaSuccess) return e;
    *kernels += 2;
    k0 += nv;
  }
  return cudaSuccess;
}

// Thread per caller row: its K values are one contiguous row of src (read
// with 16-byte loads, up to eight in flight per thread), written to the K
// columns (coalesced across threads).
__global__ void copy_out_rows_kernel(const LzState* st, const double* __restrict__ src, int64_t n,
                                     int K, const int32_t* __restrict__ iperm) {
  double* __restrict__ dst = st->eigvecs_user;
  if (dst == nullptr) return;
  const int Kr = (K + 1) & ~1;
  constexpr int CH = 8;  // 16-byte loads of one row in flight per thread
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const double2* row =
        reinterpret_cast<const double2*>(src + (size_t)(iperm ? (int64_t)iperm[v] : v) * Kr);
    for (int k0 = 0; k0 < K; k0 += 2 * CH) {
      double2 t[CH];
#pragma unroll
      for (int q = 0; q < CH; ++q)
        if (k0 + 2 * q < K) t[q] = row[(k0 >> 1) + q];
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        const int k = k0 + 2 * q;
        if (k < K) dst[(size_t)k * n + v] = t[q].x;
        if (k + 1 < K) dst[(size_t)(k + 1) * n + v] = t[q].y;
      }
    }
  }
}

cudaError_t launch_copy_out_rows(LzState* st, const double* src, int64_t n, int K,
                                 const int32_t* iperm, int grid, cudaStream_t s) {
  copy_out_rows_kernel<<<grid, 256, 0, s>>>(st, src, n, K, iperm);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Gram matrix: G[a][b] = sum_r U[r, a] U[r, b] for a <= b (pair index p in
// row-major upper-triangle order).  Each block stages GR rows of U in shared
// memory and every thread accumulates up to GP pairs; per-block partials are
// summed over blocks in order by gram_reduce.
// ---------------------------------------------------------------------------
constexpr int GR = 32;  // rows staged per block iteration
constexpr int GT = 256;
constexpr int GP = (MAX_M * (MAX_M + 1) / 2 + GT - 1) / GT;  // pairs per thread

__global__ void __launch_bounds__(GT) gram_kernel(const double* U, int64_t n, int K,
                                                  double* partials) {
  __shared__ double tile[MAX_M][GR + 1];  // +1: pairs of a warp hit different banks
  const int np = K * (K + 1) / 2;
  int pa[GP], pb[GP];
  double acc[GP];
#pragma unroll
  for (int q = 0; q < GP; ++q) {
    acc[q] = 0.0;
    pa[q] = -1;
    pb[q] = 0;
    const int p = threadIdx.x + q * GT;
    if (p < np) {
      // invert p = a*K - a*(a-1)/2 + (b - a)
      int a = 0, base = 0;
      while (base + (K - a) <= p) {
        base += K - a;
        ++a;
      }
      pa[q] = a;
      pb[q] = a + (p - base);
    }
  }
  for (int64_t r0 = (int64_t)blockIdx.x * GR; r0 < n; r0 += (int64_t)gridDim.x * GR) {
    __syncthreads();
    for (int e = threadIdx.x; e < K * GR; e += GT) {
      const int a = e / GR, rr = e % GR;
      const int64_t r = r0 + rr;
      tile[a][rr] = r < n ? U[(size_t)a * (size_t)n + r] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < GP; ++q) {
      if (pa[q] < 0) continue;
      double t = acc[q];
      for (int rr = 0; rr < GR; ++rr) t = fma(tile[pa[q]][rr], tile[pb[q]][rr], t);
      acc[q] = t;
    }
  }
#pragma unroll
  for (int q = 0; q < GP; ++q) {
    const int p = threadIdx.x + q * GT;
    if (p < np) partials[(size_t)blockIdx.x * np + p] = acc[q];
  }
}

__global__ void gram_reduce(const double* partials, int blocks, int K, double* G) {
  const int np = K * (K + 1) / 2;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  double t = 0.0;
  for (int b = 0; b < blocks; ++b) t += partials[(size_t)b * np + p];
  int a = 0, base = 0;
  while (base + (K - a) <= p) {
    base += K - a;
    ++a;
  }
  const int bcol = a + (p - base);
  G[a * K + bcol] = t;
  G[bcol * K + a] = t;
}

cudaError_t launch_gram(const double* U, int64_t n, int K, double* partials, int grid,
                        double* G, cudaStream_t s) {
  gram_kernel<<<grid, GT, 0, s>>>(U, n, K, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int np = K * (K + 1) / 2;
  gram_reduce<<<(np + 127) / 128, 128, 0, s>>>(partials, grid, K, G);
  return cudaGetLastError();
}

}  // namespace te
