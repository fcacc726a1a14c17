// te_noalloc.cu - y = M x without any device allocation.
//
// Some callers cannot call cudaMalloc: a framework whose caching allocator has
// already reserved the device memory, a serving loop that must not take the
// allocator's locks or latency between requests, or a host application that
// hands this library a fixed memory budget and forbids driver allocations.
// te_spmv needs work memory (its row partition and long-row partial sums);
// te_spmv_noalloc is a variant of the same SpMV that keeps its work memory in
// one file-scope __device__ array instead, so it allocates nothing.
//
// Work decomposition: the non-zeros are cut into fixed chunks of CHUNK
// entries, one CTA each.  Every thread loads CHUNK / 256 entries with
// coalesced loads, all gathers of x in flight at once, and leaves the (value,
// x) pairs in shared memory; a mark at each row's first entry names the row.
// Then every thread sums its own CHUNK / 256 consecutive entries, closing a
// sum at each mark: rows that lie inside one thread are done, the others are
// joined by a segmented scan over the CTA (a shuffle scan per warp, then the
// eight warps in order).  So the work per entry does not depend on the row
// lengths.  The chunk's first and last row leave their partial sums in the
// scratch array, and a second kernel adds those partials in a fixed order
// (deterministic) and writes the empty rows.  The scratch holds one 32-byte
// record per chunk, so a matrix may have at most NOALLOC_MAX_CHUNKS chunks.
// A chunk's CTA walks every row its entries touch, empty ones included, and
// the second kernel visits every row: the cost grows with n as well as nnz.
//
// Bound: the gathers of x (one 32-byte sector each on a matrix without
// locality), about 0.95 per SM and clock; the matrix's own bytes take less
// than half of that time with binary32 values.
// GB300, R-MAT 2^22, 128 M entries, binary32 values, a whole call: 1797 us
// with a warp per row (10 of 32 lanes busy on short rows), 1200 us with marks
// but four-byte accesses (the walk's 32 shared-memory reads each wait behind
// other warps' gathers in the load queue), 790 us as it stands (ncu: L1 path
// 57 % busy, barriers the largest stall).
#include <cuda_runtime.h>

#include <condition_variable>
#include <mutex>
#include <string>

#include "te_common.cuh"
#include "te_internal.h"

namespace te {

constexpr int NOALLOC_THREADS = 256;
constexpr int NOALLOC_MAX_CHUNKS = 131072;  // 4 MiB of carry records
constexpr int NOALLOC_MAX_DEVICES = 64;

struct Carry {
  int32_t head, tail;  // first and last row touched by the chunk
  int32_t pad0, pad1;
  double sum_head;     // partial sum of the head row over the chunk (f64 or dw bits)
  double sum_tail;     // partial sum of the tail row over the chunk (if tail != head)
};
static_assert(sizeof(Carry) == 32, "carry record layout");

// Shared by every call on a device; keeps the last call's contents.
static __device__ __align__(256) unsigned char g_noalloc_scratch[256 + NOALLOC_MAX_CHUNKS * sizeof(Carry)];

template <int P>
struct NaTr;
template <>
struct NaTr<PREC_DDD> {
  using val_t = double;
  using x_t = double;
  static constexpr int CHUNK = 2048;
};
template <>
struct NaTr<PREC_FDF> {
  using val_t = float;
  using x_t = float;
  static constexpr int CHUNK = 4096;
};

// The last row r in [0, n) with rp[r] <= k (rp[0] = 0 <= k), by a whole warp:
// every step probes 31 inner points of the interval at once, so a search over
// 2^22 rows takes five dependent loads instead of 22 (the chunk's other warps
// load entries meanwhile).  Any row_ptr ends it in bounds: the interval
// shrinks at every step whatever the probes hold.
TE_DEV int32_t warp_row_of(const int64_t* rp, int64_t n, int64_t k, int lane) {
  int64_t lo = 0, hi = n;  // the answer lies in [lo, hi)
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t p = lo + step * lane;  // lane 0 probes lo itself
    const bool le = lane == 0 || (p < hi && __ldg(rp + p) <= k);
    const unsigned m = __ballot_sync(0xffffffffu, le);
    const int last = 31 - __clz((int)m);
    lo += step * last;
    if (lo + step < hi) hi = lo + step;
  }
  return (int32_t)lo;
}

// accumulator: double (DDD) or double-float (FDF); stored in 8 bytes
template <int P>
struct NaAcc;
template <>
struct NaAcc<PREC_DDD> {
  double v = 0.0;
  TE_DEV void add_prod(double a, double b) { v = fma(a, b, v); }
  TE_DEV void warp_reduce() { v = warp_sum(v); }
  TE_DEV void merge(const NaAcc& o) { v += o.v; }
  TE_DEV NaAcc up(int d) const {
    NaAcc o;
    o.v = __shfl_up_sync(0xffffffffu, v, d);
    return o;
  }
  TE_DEV double bits() const { return v; }
  TE_DEV void add_bits(double b) { v += b; }
  TE_DEV double value() const { return v; }
};
template <>
struct NaAcc<PREC_FDF> {
  dacc a = {0.f, 0.f};
  TE_DEV void add_prod(float x, float y) {
    float p, e;
    two_prod(x, y, p, e);
    dacc_add_pair(a, p, e);
  }
  TE_DEV void warp_reduce() { a = warp_sum(a); }
  TE_DEV void merge(const NaAcc& o) { a = dacc_merge(a, o.a); }
  TE_DEV NaAcc up(int d) const {
    NaAcc o;
    o.a.s = __shfl_up_sync(0xffffffffu, a.s, d);
    o.a.c = __shfl_up_sync(0xffffffffu, a.c, d);
    return o;
  }
  TE_DEV double bits() const {
    dw v = dacc_value(a);
    return __longlong_as_double(((long long)__float_as_int(v.lo) << 32) |
                                (unsigned int)__float_as_int(v.hi));
  }
  TE_DEV void add_bits(double b) {
    long long u = __double_as_longlong(b);
    dacc_add_pair(a, __int_as_float((int)(u & 0xffffffffu)), __int_as_float((int)(u >> 32)));
  }
  // (the integer conversion: most warps close a row at half of their steps, and
  // the binary64 pipe would take 16 cycles per instruction for a few lanes)
  TE_DEV double value() const { return dw_to_double_bits(dacc_value(a)); }
};

// A running sum and the row it belongs to: row = -1 when no row has started
// since the sum began (the sum continues the one before it).
template <int P>
struct NaSeg {
  NaAcc<P> acc;
  int32_t row = -1;
  // this segment placed after `p`
  TE_DEV void after(const NaSeg& p) {
    if (row >= 0) return;
    NaAcc<P> t = p.acc;
    t.merge(acc);
    acc = t;
    row = p.row;
  }
};

// A chunk in shared memory: runs of IPT entries, one per thread, each padded
// so that the threads' 16-byte reads of their own runs (and the writes, four
// entries at a time) touch different banks.  FDF: 57 KB, three CTAs per SM.
template <int P>
struct NaSmem {
  using val_t = typename NaTr<P>::val_t;
  using x_t = typename NaTr<P>::x_t;
  static constexpr int CH = NaTr<P>::CHUNK;
  static constexpr int IPT = CH / NOALLOC_THREADS;
  static constexpr int PPAD = 16 / (int)(2 * sizeof(val_t));
  static constexpr int PRUN = IPT + PPAD;  // a run of pairs: its bytes = 16 mod 128
  static constexpr int MRUN = IPT + 4;     // a run of marks
  struct __align__(2 * sizeof(val_t)) Pair {
    val_t v;
    x_t x;
  };
  struct __align__(16) Pair16 {
    Pair p[16 / sizeof(Pair)];
  };
  static constexpr int PPV = (int)(sizeof(Pair16) / sizeof(Pair));  // pairs per 16 bytes
  __align__(16) Pair pair[NOALLOC_THREADS * PRUN];
  __align__(16) int32_t mark[NOALLOC_THREADS * MRUN];  // the row whose first entry this is, else -1
  NaSeg<P> wtot[NOALLOC_THREADS / 32];
  int32_t hs, ts;
  TE_DEV static int pslot(int e) { return e / IPT * PRUN + e % IPT; }
  TE_DEV static int mslot(int e) { return e / IPT * MRUN + e % IPT; }
};

// Many chunks: the first and last row of every chunk, a warp per chunk,
// before the chunk kernel (16 us for 15,500 chunks).  Inside it the search's
// five dependent loads wait each time behind the gathers of the SM's other
// warps, in the same queue.
__global__ void __launch_bounds__(256) noalloc_search_kernel(const int64_t* rp, int64_t n,
                                                             int64_t nnz, int ch, int64_t nchunks,
                                                             unsigned char* scratch) {
  Carry* carry = reinterpret_cast<Carry*>(scratch + 256);
  const int lane = threadIdx.x & 31;
  const int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (c >= nchunks) return;
  const int64_t k1 = (c + 1) * ch < nnz ? (c + 1) * ch : nnz;
  const int32_t h = warp_row_of(rp, n, c * ch, lane);
  const int32_t t = warp_row_of(rp, n, k1 - 1, lane);
  if (lane == 0) *reinterpret_cast<int2*>(&carry[c]) = make_int2(h, t);
}

// VEC: col_idx and values are 16-byte aligned, so four entries per load
template <int P, bool VEC>
__global__ void __launch_bounds__(NOALLOC_THREADS, 3) noalloc_chunk_kernel(
    const int64_t* rp, const int32_t* ci, const void* val, const void* x, double* y, int64_t n,
    int64_t nnz, int searched, unsigned char* scratch, volatile int* status) {
  using val_t = typename NaTr<P>::val_t;
  using x_t = typename NaTr<P>::x_t;
  using Sm = NaSmem<P>;
  constexpr int CH = Sm::CH, IPT = Sm::IPT, G = IPT / 4;
  extern __shared__ __align__(16) unsigned char na_sm[];
  Sm& sm = *reinterpret_cast<Sm*>(na_sm);
  Carry* carry = reinterpret_cast<Carry*>(scratch + 256);

  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t c = blockIdx.x;
  const int64_t k0 = c * CH;
  const int64_t k1 = k0 + CH < nnz ? k0 + CH : nnz;
  const int nz = (int)(k1 - k0);
  const uint64_t keep = policy_evict_last();
  const int32_t* cp = ci + k0;
  const val_t* va = static_cast<const val_t*>(val) + k0;
  const x_t* xv = static_cast<const x_t*>(x);
  int2 ht = make_int2(0, 0);
  if (searched) ht = *reinterpret_cast<const int2*>(&carry[c]);
  // group g of this thread: entries (g * 256 + tid) * 4 ... + 3
  int32_t col[IPT];
  val_t v[IPT];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int e = (g * NOALLOC_THREADS + tid) * 4;
    if (VEC && e + 4 <= nz) {
      const int4 c4 = __ldcs(reinterpret_cast<const int4*>(cp + e));
      col[4 * g] = c4.x;
      col[4 * g + 1] = c4.y;
      col[4 * g + 2] = c4.z;
      col[4 * g + 3] = c4.w;
      if constexpr (P == PREC_FDF) {
        const float4 v4 = __ldcs(reinterpret_cast<const float4*>(va + e));
        v[4 * g] = v4.x;
        v[4 * g + 1] = v4.y;
        v[4 * g + 2] = v4.z;
        v[4 * g + 3] = v4.w;
      } else {
        const double2 a2 = __ldcs(reinterpret_cast<const double2*>(va + e));
        const double2 b2 = __ldcs(reinterpret_cast<const double2*>(va + e + 2));
        v[4 * g] = a2.x;
        v[4 * g + 1] = a2.y;
        v[4 * g + 2] = b2.x;
        v[4 * g + 3] = b2.y;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = e + u < nz;
        col[4 * g + u] = in ? cp[e + u] : 0;
        v[4 * g + u] = in ? va[e + u] : (val_t)0;
      }
    }
  }
  for (int e = tid; e < NOALLOC_THREADS * Sm::MRUN / 4; e += NOALLOC_THREADS)
    reinterpret_cast<int4*>(sm.mark)[e] = make_int4(-1, -1, -1, -1);
  if (!searched) {
    if (wid == 0) {
      const int32_t r = warp_row_of(rp, n, k0, lane);
      if (lane == 0) sm.hs = r;
    } else if (wid == 1) {
      const int32_t r = warp_row_of(rp, n, k1 - 1, lane);
      if (lane == 0) sm.ts = r;
    }
    __syncthreads();
    ht = make_int2(sm.hs, sm.ts);
  }
  const int32_t h = ht.x, t = ht.y;  // in [0, n), whatever row_ptr holds
  // the first rows' pointers, on their way before the gathers
  int64_t r = (int64_t)h + 1 + tid;
  int64_t rb = 0, re = 0;
  if (r <= t) {
    rb = __ldg(rp + r);
    re = __ldg(rp + r + 1);
  }
  bool bad = false;
  x_t xg[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) {  // (entries past nz gather x[0])
    const bool ok = col[i] >= 0 && (int64_t)col[i] < n;
    bad |= !ok;
    const int32_t g = ok ? col[i] : 0;
    if constexpr (P == PREC_FDF) xg[i] = ld_keep_f32(xv + g, keep);
    else xg[i] = ld_keep_f64(xv + g, keep);
  }
  if (bad) status[0] = 1;
  if (searched) __syncthreads();  // the marks are cleared
  // marks of the rows after the first; an empty row has no entry to mark
  while (r <= t) {
    if (rb < re && rb >= k0 && rb < k1) sm.mark[Sm::mslot((int)(rb - k0))] = (int32_t)r;
    r += NOALLOC_THREADS;
    if (r <= t) {
      rb = __ldg(rp + r);
      re = __ldg(rp + r + 1);
    }
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int at = Sm::pslot((g * NOALLOC_THREADS + tid) * 4);
#pragma unroll
    for (int u = 0; u < 4; u += Sm::PPV) {
      typename Sm::Pair16 w;
#pragma unroll
      for (int q = 0; q < Sm::PPV; ++q) {
        w.p[q].v = v[4 * g + u + q];
        w.p[q].x = xg[4 * g + u + q];
      }
      *reinterpret_cast<typename Sm::Pair16*>(&sm.pair[at + u]) = w;
    }
  }
  __syncthreads();

  // this thread's entries; `head`: what precedes its first mark
  NaSeg<P> mine;
  NaAcc<P> head;
  const int cnt = nz - tid * IPT;
  int4 mk[G];
#pragma unroll
  for (int g = 0; g < G; ++g) mk[g] = reinterpret_cast<const int4*>(sm.mark + tid * Sm::MRUN)[g];
  auto walk = [&](int g, NaSeg<P>& seg, NaAcc<P>& before) {  // four entries
    typename Sm::Pair16 w[4 / Sm::PPV];
#pragma unroll
    for (int u = 0; u < 4 / Sm::PPV; ++u)
      w[u] = *reinterpret_cast<const typename Sm::Pair16*>(
          &sm.pair[tid * Sm::PRUN + 4 * g + u * Sm::PPV]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (4 * g + u < cnt) {
        const int32_t row = u == 0 ? mk[g].x : u == 1 ? mk[g].y : u == 2 ? mk[g].z : mk[g].w;
        if (row >= 0) {
          if (seg.row >= 0) y[seg.row] = seg.acc.value();
          else before = seg.acc;
          seg.acc = NaAcc<P>();
          seg.row = row;
        }
        const typename Sm::Pair p = w[u / Sm::PPV].p[u % Sm::PPV];
        seg.acc.add_prod(p.v, p.x);
      }
    }
  };
  if constexpr (P == PREC_FDF) {
#pragma unroll
    for (int g = 0; g < G; ++g) walk(g, mine, head);
  } else {
    // two chains of four, joined: a chain of eight rounds more often than the sum
    // of a row by a tree (rows of 20 entries: error 1.69e-16 against 1.58e-16)
    static_assert(P == PREC_FDF || G == 2, "");
    NaSeg<P> part;
    NaAcc<P> between;
    walk(0, mine, head);
    walk(1, part, between);
    NaAcc<P> t = mine.acc;
    t.merge(part.row < 0 ? part.acc : between);
    if (part.row < 0) {
      mine.acc = t;
    } else {
      if (mine.row >= 0) y[mine.row] = t.value();
      else head = t;
      mine = part;
    }
  }
  // inclusive segmented scan over the warp, then what lies before this thread
  NaSeg<P> inc = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    // (short rows: no sum reaches further; the vote is cheaper than a merge:
    // uniform rows of 24 entries, 36.8 M of them, binary64 403 -> 366 us)
    if (!__any_sync(0xffffffffu, lane >= d && inc.row < 0)) break;
    NaSeg<P> p;
    p.acc = inc.acc.up(d);
    p.row = __shfl_up_sync(0xffffffffu, inc.row, d);
    if (lane >= d) inc.after(p);
  }
  if (lane == 31) sm.wtot[wid] = inc;
  NaSeg<P> ex;
  ex.acc = inc.acc.up(1);
  ex.row = __shfl_up_sync(0xffffffffu, inc.row, 1);
  if (lane == 0) ex = NaSeg<P>();
  __syncthreads();
  NaSeg<P> pre;  // the chunk starts inside (or at the start of) row h
  pre.row = h;
  for (int w = 0; w < wid; ++w) {
    NaSeg<P> q = sm.wtot[w];
    q.after(pre);
    pre = q;
  }
  ex.after(pre);
  if (mine.row >= 0) {  // the row open before this thread ends here
    NaAcc<P> s = ex.acc;
    s.merge(head);
    if (ex.row == h) carry[c].sum_head = s.bits();
    else y[ex.row] = s.value();
  }
  if (tid == NOALLOC_THREADS - 1) {  // the chunk's last row stays open
    mine.after(ex);
    if (mine.row == h) carry[c].sum_head = mine.acc.bits();
    else carry[c].sum_tail = mine.acc.bits();
    carry[c].head = h;
    carry[c].tail = t;
  }
}

// Adds the chunks' partial sums, writes the empty rows, and checks the row
// pointers (row_ptr[0] = 0, non-decreasing, row_ptr[n] = nnz): a malformed
// row_ptr sets the second status word.  The chunk kernel keeps every access
// in bounds whatever row_ptr holds; its results are discarded then.
// A warp per chunk completes the rows that start in it (a row is completed
// by the chunk in which it starts): its lanes add the chunks that the row
// covers, strided, and a shuffle tree joins the lanes - a row over a
// thousand chunks is a hub row's ordinary case, and one thread walking them
// would end long after everything else.  The first chunk_blocks blocks do
// this (a chain of dependent loads each), the others check the rows,
// NA_FIX_ROWS per thread, at the same time.
constexpr int NA_FIX_ROWS = 4;
template <int P>
__global__ void __launch_bounds__(256) noalloc_fixup_kernel(const int64_t* rp, double* y,
                                                            int64_t n, int64_t nnz,
                                                            int64_t nchunks, int chunk_blocks,
                                                            unsigned char* scratch,
                                                            volatile int* status) {
  constexpr int CH = NaTr<P>::CHUNK;
  const Carry* carry = reinterpret_cast<const Carry*>(scratch + 256);
  const int lane = threadIdx.x & 31;
  if ((int)blockIdx.x < chunk_blocks) {  // uniform per block
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= nchunks) return;
    const Carry rec = carry[i];
    const int64_t hb = __ldg(rp + rec.head), he = __ldg(rp + rec.head + 1);
    const int64_t te = __ldg(rp + rec.tail + 1);
#pragma unroll
    for (int side = 0; side < 2; ++side) {  // the chunk's first row, then its last
      if (side ? rec.tail == rec.head : hb != i * CH) continue;  // uniform
      const int32_t row = side ? rec.tail : rec.head;
      // the last chunk with entries of this row (clamped: row_ptr may be malformed)
      int64_t last = ((side ? te : he) - 1) / CH;
      if (last >= nchunks) last = nchunks - 1;
      NaAcc<P> s;
      if (lane == 0) s.add_bits(side ? rec.sum_tail : rec.sum_head);
      if (side || rec.tail == rec.head)
        for (int64_t c2 = i + 1 + lane; c2 <= last; c2 += 32) s.add_bits(carry[c2].sum_head);
      s.warp_reduce();
      if (lane == 0) y[row] = s.value();
    }
    return;
  }
  const int64_t b0 = (int64_t)(blockIdx.x - chunk_blocks) * (256 * NA_FIX_ROWS);
  if (b0 == 0 && threadIdx.x == 0 && (__ldg(rp) != 0 || __ldg(rp + n) != nnz)) status[1] = 1;
  int64_t b[NA_FIX_ROWS], e[NA_FIX_ROWS];
#pragma unroll
  for (int u = 0; u < NA_FIX_ROWS; ++u) {
    const int64_t i = b0 + threadIdx.x + 256 * u;
    b[u] = i < n ? __ldg(rp + i) : 0;
    e[u] = i < n ? __ldg(rp + i + 1) : 1;
  }
#pragma unroll
  for (int u = 0; u < NA_FIX_ROWS; ++u) {
    if (b[u] == e[u]) y[b0 + threadIdx.x + 256 * u] = 0.0;
    if (b[u] > e[u]) status[1] = 1;
  }
}

// Above this many chunks the rows are searched beforehand (three launches
// instead of two): a chunk kernel of a few waves hides its own search, and a
// launch costs about 2 us.  us a call without and with the search: binary32
// values 660 chunks 72 and 74, 1,380 89 and 91, 2,100 103 and 103, 4,500 164 and 155,
// 18,000 514 and 445; binary64 660 63 and 68, from 2,100 to 18,000 within 3 %.
constexpr int64_t NA_SEARCH_CHUNKS = 2048;

// one call's launches; the chunk kernel's shared memory (above the 48 KB
// that need no opt-in) is allowed on this device by na_prepare
template <int P>
static cudaError_t na_launch(const te_csr* A, const void* x, double* y, int64_t nchunks,
                             unsigned char* scratch, int* status, cudaStream_t s) {
  constexpr int CH = NaTr<P>::CHUNK;
  const int chunk_blocks = (int)((nchunks + 7) / 8);
  if (nchunks > 0) {
    const int searched = nchunks > NA_SEARCH_CHUNKS;
    if (searched)
      noalloc_search_kernel<<<(unsigned)chunk_blocks, 256, 0, s>>>(A->row_ptr, A->n, A->nnz, CH,
                                                                   nchunks, scratch);
    const bool vec = ((reinterpret_cast<uintptr_t>(A->col_idx) |
                       reinterpret_cast<uintptr_t>(A->values)) & 15) == 0;
    auto* k = vec ? noalloc_chunk_kernel<P, true> : noalloc_chunk_kernel<P, false>;
    k<<<(unsigned)nchunks, NOALLOC_THREADS, sizeof(NaSmem<P>), s>>>(
        A->row_ptr, A->col_idx, A->values, x, y, A->n, A->nnz, searched, scratch, status);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int64_t row_blocks = (A->n + 256 * NA_FIX_ROWS - 1) / (256 * NA_FIX_ROWS);
  noalloc_fixup_kernel<P><<<(unsigned)(chunk_blocks + row_blocks), 256, 0, s>>>(
      A->row_ptr, y, A->n, A->nnz, nchunks, chunk_blocks, scratch, status);
  return cudaGetLastError();
}

template <int P>
static cudaError_t na_prepare() {
  const cudaError_t e = cudaFuncSetAttribute(noalloc_chunk_kernel<P, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(NaSmem<P>));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(noalloc_chunk_kernel<P, false>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(NaSmem<P>));
}

namespace {
// Per device: the scratch array's address and the calls in flight.  A call's
// status words (bad column, malformed row_ptr) lie in managed memory, which the
// kernels write straight into, only when something is wrong.  The host clears
// them before the call and reads them after its synchronisation, so a call is
// two launches and a wait: a status word on the device took a memset and a copy
// more (53 us against 32 us a call at 600 k entries).  Every call in flight has
// a slot of its own.
struct NaDevice {
  void* scratch = nullptr;
  uint64_t busy = 0;  // one bit per slot
};
std::mutex g_na_mu;
std::condition_variable g_na_cv;
NaDevice g_na[NOALLOC_MAX_DEVICES];

// a call's slot, given back when the call returns
struct NaSlot {
  NaDevice& g;
  int i;
  explicit NaSlot(NaDevice& dev) : g(dev) {
    std::unique_lock<std::mutex> lk(g_na_mu);
    g_na_cv.wait(lk, [&] { return g.busy != ~0ull; });
    for (i = 0; (g.busy >> i) & 1u; ++i) {}
    g.busy |= 1ull << i;
  }
  ~NaSlot() {
    {
      std::lock_guard<std::mutex> lk(g_na_mu);
      g.busy &= ~(1ull << i);
    }
    g_na_cv.notify_one();
  }
};
static_assert(NA_SLOTS == 64, "one bit of `busy` per slot");
static_assert(NA_DEVICES >= NOALLOC_MAX_DEVICES, "status words for every device");
}  // namespace

}  // namespace te

using namespace te;

extern "C" te_status te_spmv_noalloc(const te_csr* A, te_precision p, const void* x, double* y,
                                     void* stream);

// Defined here (not in te_solver.cu) so that the scratch symbol and its device
// address stay in one translation unit.
extern "C" te_status te_spmv_noalloc(const te_csr* A, te_precision p, const void* x, double* y,
                                     void* stream) {
  auto fail = [](te_status s, const std::string& m) {
    set_last_error(m);
    return s;
  };
  if (!A || !x || !y) return fail(TE_ERR_INVALID_ARG, "te_spmv_noalloc: NULL argument");
  if (A->where != TE_DEVICE)
    return fail(TE_ERR_INVALID_ARG, "te_spmv_noalloc: the matrix must be in device memory");
  if (A->n < 1 || A->n >= (int64_t)1 << 31 || A->nnz < 0 || !A->row_ptr ||
      (A->nnz > 0 && (!A->col_idx || !A->values)))
    return fail(TE_ERR_INVALID_ARG, "te_spmv_noalloc: bad CSR sizes or pointers");
  if (A->row_scale) return fail(TE_ERR_UNSUPPORTED, "te_spmv_noalloc: row_scale must be NULL");
  int prec = -1;
  if (p.values == TE_F64 && p.arithmetic == TE_F64 && p.vectors == TE_F64) prec = PREC_DDD;
  if (p.values == TE_F32 && p.arithmetic == TE_F64 && p.vectors == TE_F32) prec = PREC_FDF;
  if (prec < 0) return fail(TE_ERR_UNSUPPORTED, "te_spmv_noalloc: precision must be DDD or FDF");
  if (A->values_f64 && prec != PREC_DDD)
    return fail(TE_ERR_INVALID_ARG,
                "te_spmv_noalloc: values must already have the precision's type (values_f64 = 0)");
  const int chunk = prec == PREC_DDD ? NaTr<PREC_DDD>::CHUNK : NaTr<PREC_FDF>::CHUNK;
  const int64_t nchunks = (A->nnz + chunk - 1) / chunk;
  if (nchunks > NOALLOC_MAX_CHUNKS)
    return fail(TE_ERR_INVALID_ARG,
                "te_spmv_noalloc: nnz = " + std::to_string(A->nnz) + " exceeds the maximum " +
                    std::to_string((int64_t)NOALLOC_MAX_CHUNKS * chunk) +
                    " of the fixed scratch array for this precision");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(TE_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES)
    return fail(TE_ERR_UNSUPPORTED, "te_spmv_noalloc: device index too large");
  // once per device, with that device current: the scratch array's device
  // address (kept for the life of the process; a device reset invalidates it)
  // and the chunk kernels' shared memory
  NaDevice& g = g_na[dev];
  {
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g.scratch) {
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
      if (e != cudaSuccess)
        return fail(TE_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      e = na_prepare<PREC_DDD>();
      if (e == cudaSuccess) e = na_prepare<PREC_FDF>();
      if (e != cudaSuccess)
        return fail(TE_ERR_CUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e));
      g.scratch = ptr;
    }
  }
  NaSlot slot(g);
  unsigned char* scratch = static_cast<unsigned char*>(g.scratch);
  int* words = noalloc_status_words() + (dev * NA_SLOTS + slot.i) * 2;
  volatile int* status = words;
  status[0] = 0;
  status[1] = 0;
  e = prec == PREC_DDD ? na_launch<PREC_DDD>(A, x, y, nchunks, scratch, words, s)
                       : na_launch<PREC_FDF>(A, x, y, nchunks, scratch, words, s);
  // also after a launch that failed: a kernel queued before it may still set the
  // slot's words, which the next call to take the slot would read
  const cudaError_t es = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = es;
  if (e != cudaSuccess) return fail(TE_ERR_CUDA, std::string("te_spmv_noalloc: ") + cudaGetErrorString(e));
  if (status[1]) return fail(TE_ERR_INVALID_ARG, "te_spmv_noalloc: malformed row_ptr");
  if (status[0]) return fail(TE_ERR_INVALID_ARG, "te_spmv_noalloc: a column index is outside [0, n)");
  return TE_OK;
}
