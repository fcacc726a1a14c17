// te_jacobi.cu - the Jacobi phase (Section III, Fig. 1): eigen-decomposition
// of the small tridiagonal T produced by the Lanczos phase, the selection of
// the K eigenvalues largest in modulo (Section I), and the coefficients of the
// Ritz-vector contraction.
//
// The paper ran this step on the CPU because one 24x24 matrix cannot fill a
// GPU; here it stays on the device so that a solve needs no host round trip
// before the Ritz contraction.  Cyclic Jacobi with the parallel (round-robin,
// "circle method") ordering of Brent & Luk: every round rotates m/2 disjoint
// index pairs at once, T <- J^T T J (on 2x2 blocks of the upper triangle),
// Y <- Y J.  A pair is rotated when |t_pq| > 1e-16 ||T||_F and the sweeps stop
// after one without rotations (which is skipped when no off-diagonal element
// left after a sweep exceeds that threshold: it could rotate nothing).
// Arithmetic is binary64.
//
// Bound: the latency of a round.  A binary64 instruction holds its scheduler's
// binary64 unit for 64 cycles whatever the number of active lanes, a
// conversion to or from binary32 for about 84 (measured), while binary32 and
// integer instructions follow one another every 5.  So what counts is the
// number of binary64 instructions that one scheduler issues in a row:
//   - the rotation angles (one warp) take 15 binary64 instructions: the
//     tangent starts from binary32, gets one Newton step in double-float and
//     one in binary64, the cosine one third-order step; conversions and
//     comparisons are integer operations (jac_angle; about 1,150 cycles
//     against 3,000 with hypot, a division and a reciprocal square root);
//   - the blocks of T take a thread per element, which exchanges with its
//     neighbours by shuffles: four binary64 instructions per 32 elements,
//     spread over the schedulers (a thread per block took 16 in a row);
//   - Y is updated one round behind, by warps 5-7 while warp 0 computes the
//     next angles (and while a cluster's barrier is pending), so only the
//     blocks of T lie between two rounds' angles;
//   - T is held as the blocks of the round, two copies that the rounds
//     alternate between: each element is stored where the next round needs
//     it, a place that its thread works out while the angles are computed.
// For larger T the blocks and the rows of Y are spread over a cluster of CL
// CTAs, and the elements go straight into the next owner's copy through
// distributed shared memory: one store each (pushing every element into every
// CTA's full copy of T took seven), except that a pair's own element goes to
// every CTA, since each computes all angles.  One cluster barrier per round.
// Each element is computed by the same formula from the same inputs as on one
// CTA, so all forms give the same bits.
// te_tridiag_eigs, a whole call (about 50 us of it outside the kernel), before
// and now: m = 16 308 -> 172 us, 32 903 -> 407, 48 1767 -> 684, 64 3190 -> 1055.
#include "te_common.cuh"
#include "te_internal.h"

namespace te {

constexpr int JAC_THREADS = 256;
constexpr int JAC_Y_WARP = 5;    // warps 5-7 update Y (not warp 4: its scheduler is warp 0's)
constexpr int JAC_MAX_SWEEPS = 100;
constexpr int JLD = MAX_M + 1;   // padded row length of Y in shared memory
constexpr int JAC_HALF = MAX_M / 2;
// CTAs by the order of T, measured per call: one below 23 (m = 20: 257 us on one
// CTA, 262 on four; m = 24: 384 and 314), which is also what a thread per
// element allows (55 blocks); four below 37, where eight are no faster (m = 32:
// 435 us on either; m = 40: 562 on four, 534 on eight) and take the serving
// engine's SMs.  Eight hold the 62 blocks per CTA of m = 64.
constexpr int JAC_CLUSTER4_MIN_M = 23, JAC_CLUSTER8_MIN_M = 37;

TE_DEV uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the shared::cluster address of the same location in CTA `rank` of the cluster
TE_DEV uint32_t cluster_map(uint32_t saddr, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(saddr), "r"(rank));
  return d;
}
TE_DEV void st_cluster_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
// every thread of every CTA of the cluster; orders shared-memory writes
// (local and remote) before the arrival against reads after the wait
TE_DEV void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
TE_DEV void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
TE_DEV void cluster_barrier() {
  cluster_arrive();
  cluster_wait();
}

// position j of the round-robin schedule in round r < mm - 1 (player 0 stays put)
TE_DEV int rr_player(int j, int r, int mm) {
  const int x = j - 1 + r;  // < 2 (mm - 1)
  return j == 0 ? 0 : 1 + (x < mm - 1 ? x : x - (mm - 1));
}

// the position of player x in round r (rr_player's inverse)
TE_DEV int rr_position(int x, int r, int mm) {
  if (x == 0) return 0;
  const int d = x - 1 - r;
  return 1 + (d < 0 ? d + mm - 1 : d);
}
// the pair of player x in round r, and whether x is the larger of the two:
// pair * 2 + that
TE_DEV int rr_pair(int x, int r, int mm) {
  const int j = rr_position(x, r, mm), o = mm - 1 - j;
  return 2 * (j < o ? j : o) + (rr_player(o, r, mm) < x ? 1 : 0);
}

// A binary64 value's place in its order as an integer (zeros of either sign
// alike): the selection's m^2 comparisons stay off the binary64 unit, and any
// bit pattern has one, so the ranks are always distinct.
TE_DEV int64_t order_key(double a) {
  const int64_t b = __double_as_longlong(a);
  return b >= 0 ? b : b == INT64_MIN ? 0 : INT64_MIN - b;
}
TE_DEV bool sel_before(int64_t a, int ia, int64_t b, int ib, int which) {
  if (which != TE_WHICH_LARGEST_ALGEBRAIC) {
    const int64_t fa = a < 0 ? -a : a, fb = b < 0 ? -b : b;
    if (fa != fb) return fa > fb;
    if ((a > 0) != (b > 0)) return a > 0;
    return ia < ib;
  }
  if (a != b) return a > b;
  return ia < ib;
}

// |x| as an integer that orders like it
TE_DEV int64_t abs_bits(double x) { return __double_as_longlong(x) & INT64_MAX; }

// The rotation that annihilates t_pq: t = tan of the angle, c = 1 / sqrt(1 +
// t^2), s = t c.  With A = |t_pq| and D = |t_qq - t_pp|, |t| is the root of
// A t^2 + D t - A in (0, 1], and 2 A t + D = sqrt(D^2 + 4 A^2) there, the
// derivative that Newton's iteration divides by.  T is held scaled to a
// largest element in [1, 2), and A exceeds 1e-16 ||T||_F, so binary32 holds
// both.  The binary32 start is good to 2^-20; a step whose residual is taken
// in double-float brings it to 2^-41, one with a binary64 residual to the
// rounding of its last subtraction.  The cosine: y in binary32 with e = 1 -
// y^2 - (t y)^2, then 1 + e/2 + 3 e^2/8 times y and times t y.  (Refining y in
// double-float first saves three binary64 instructions, but its thirty binary32
// ones are issued in order before them: 3 % slower.)
// Against 113-bit arithmetic on 2.9 M pairs (|t_pq| from 1e-16 to 2, equal
// and nearly equal diagonals): t within 2.4, c 1.3, s 4.0 and c^2 + s^2 within
// 1.5 times 2^-53.
TE_DEV void jac_angle(double tpp, double tqq, double tpq, double& t, double& c, double& s) {
  const double d = tqq - tpp;
  const double A = fabs(tpq), D = fabs(d);
  const float Ah = f_head(A), Al = f_tail(A), Dh = f_head(D), Dl = f_tail(D);
  const float two = 2.0f * Ah;
  float ih, inv, fc;
  const float u = __fmaf_rn(Dh, Dh, two * two);
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ih) : "f"(u));  // 1 / sqrt(D^2 + 4 A^2)
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(__fmaf_rn(u, ih, Dh)));
  const float t0 = two * inv;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(fc) : "f"(__fmaf_rn(t0, t0, 1.0f)));
  // A (t0^2 - 1) + D t0 in double-float
  float pe, p = __fmul_rn(t0, t0);
  pe = __fmaf_rn(t0, t0, -p);
  float vh, vl;
  fast_two_sum(-1.0f, p, vh, vl);
  vl = __fadd_rn(vl, pe);
  float ah, al, qh, ql, sh, sl;
  two_prod(Ah, vh, ah, al);
  al = __fmaf_rn(Ah, vl, __fmaf_rn(Al, vh, al));
  two_prod(Dh, t0, qh, ql);
  ql = __fmaf_rn(Dl, t0, ql);
  two_sum(ah, qh, sh, sl);
  const float r0 = __fadd_rn(sh, __fadd_rn(sl, __fadd_rn(al, ql)));
  double tt = f_wide(t0) - f_wide(r0 * ih);
  const double r1 = fma(A, fma(tt, tt, -1.0), D * tt);
  tt -= f_wide(f_narrow(r1) * ih);
  const double y = f_wide(fc), y2 = fma(-y, y, 1.0);
  const double ty = tt * y;
  const double e = fma(-ty, ty, y2);
  const double g = e * fma(0.375, e, 0.5);
  c = fma(y, g, y);
  s = fma(ty, g, ty);
  // sgn(t) = sgn(d / t_pq), + for d = 0
  const int64_t db = __double_as_longlong(d);
  const int64_t sign =
      (db & INT64_MAX) == 0 ? 0 : ((db ^ __double_as_longlong(tpq)) & INT64_MIN);
  t = __longlong_as_double(__double_as_longlong(tt) ^ sign);
  s = __longlong_as_double(__double_as_longlong(s) ^ sign);
}

// off-diagonal blocks (a, b), a < b, of h pairs: row-major index, and how many
__host__ __device__ constexpr int jac_block(int a, int b, int h) {
  return a * (2 * h - a - 1) / 2 + (b - a - 1);
}
constexpr int JAC_BLOCKS = JAC_HALF * (JAC_HALF - 1) / 2;

// Shared memory of a CTA.  Whatever a round writes for the next goes into the
// other copy ([2]), so one barrier per round orders it: a CTA can be at most
// one round ahead, and then it writes the copy that the slower one has read.
template <int CL>
struct JacSmem {
  static constexpr int NB = (JAC_BLOCKS + CL - 1) / CL;
  double blk[2][NB][4];          // this CTA's off-diagonal blocks of T
  double offd[2][JAC_HALF];      // every pair's own off-diagonal element
  double diag[2][MAX_M];         // every diagonal element
  double Y[MAX_M * JLD];         // rows rank + i CL (CTA 0 collects all at the end)
  double rc[2][JAC_HALF], rs[2][JAC_HALF], rt[2][JAC_HALF];
  long long wmax[JAC_THREADS / 32];
  double cmax[2][CL];
  double thr;
  int64_t key[MAX_M];
  int pq[2][JAC_HALF];           // a pair's players p | q << 8, bit 16: rotated
  int any;                       // a rotation in this sweep
  int sel[MAX_M];
  unsigned char ba[JAC_BLOCKS], bb[JAC_BLOCKS];  // the pairs of a block
};

template <int CL>
__global__ void __launch_bounds__(JAC_THREADS, 1) jacobi_kernel(JacobiArgs a) {
  extern __shared__ __align__(16) unsigned char jsm[];
  JacSmem<CL>& sm = *reinterpret_cast<JacSmem<CL>*>(jsm);
  double* const Y = sm.Y;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int m = a.m;
  const int mm = m + (m & 1);  // even size; a dummy index never rotates
  const int half = mm / 2;
  const int nblk = half * (half - 1) / 2;
  // this CTA's share: blocks e = rank + i CL (i < nb_mine), rows of Y
  // r = rank + i CL (i < ny_rows); CL = 1: everything
  const int rank = CL > 1 ? (int)cluster_ctarank() : 0;
  const int nb_mine = (nblk - rank + CL - 1) / CL;
  const int ny_rows = (mm - rank + CL - 1) / CL;

  // the exponent of T's largest element: T is held divided by 2^texp (exact),
  // and the Ritz values are multiplied by it at the end
  int texp;
  {
    int ex = 0;
    for (int r = lane; r < m; r += 32) {
      ex = max(ex, (int)(__double_as_longlong(a.alpha[r]) >> 52) & 0x7ff);
      if (r > 0) ex = max(ex, (int)(__double_as_longlong(a.beta[r]) >> 52) & 0x7ff);
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    // (subnormal: the smallest one becomes 1; infinities and NaN: no rotations)
    texp = ex == 0x7ff ? 0 : ex == 0 ? -1074 : ex - 1023;
  }
  auto t_init = [&](int r, int c) {  // the tridiagonal T
    double v = 0.0;
    if (r < m && c < m) {
      if (r == c) v = a.alpha[r];
      else if (r - c == 1 || c - r == 1) v = a.beta[r > c ? r : c];
    }
    return scalbn(v, -texp);
  };
  // Where the element of players i and j goes after round `r`: the block
  // (4 e + place in it) that it belongs to in the next round, or -1 - k when
  // the two meet there as pair k.
  auto dest = [&](int i, int j, int r) {
    const int rn = r + 1 < mm - 1 ? r + 1 : 0;
    const int x = rr_pair(i, rn, mm), y = rr_pair(j, rn, mm);
    if ((x >> 1) == (y >> 1)) return -1 - (x >> 1);
    const int lo = min(x, y), hi = max(x, y);
    return 4 * jac_block(lo >> 1, hi >> 1, half) + 2 * (lo & 1) + (hi & 1);
  };
  // the same for element el & 3 of this CTA's block el >> 2
  auto dest_of = [&](int el, int r) {
    const int e = rank + (el >> 2) * CL, ka = sm.ba[e], kb = sm.bb[e];
    const int a0 = rr_player(ka, r, mm), a1 = rr_player(mm - 1 - ka, r, mm);
    const int b0 = rr_player(kb, r, mm), b1 = rr_player(mm - 1 - kb, r, mm);
    return dest((el & 2) ? max(a0, a1) : min(a0, a1), (el & 1) ? max(b0, b1) : min(b0, b1), r);
  };
  auto put = [&](int to, double v, int nbuf) {
    if (to < 0) {  // every CTA needs it for the angles
      if constexpr (CL > 1) {
        const uint32_t at = smem_addr(&sm.offd[nbuf][-1 - to]);
#pragma unroll
        for (int q = 0; q < CL; ++q) st_cluster_f64(cluster_map(at, (uint32_t)q), v);
      } else {
        sm.offd[nbuf][-1 - to] = v;
      }
      return;
    }
    const int e = to >> 2;
    double* at = &sm.blk[nbuf][e / CL][to & 3];
    if constexpr (CL > 1) st_cluster_f64(cluster_map(smem_addr(at), (uint32_t)(e % CL)), v);
    else *at = v;
  };

  for (int e = tid; e < mm * mm; e += JAC_THREADS) {
    const int r = e / mm, c = e - r * mm;
    Y[r * JLD + c] = (r == c) ? 1.0 : 0.0;
  }
  for (int i = tid; i < mm; i += JAC_THREADS) sm.diag[0][i] = t_init(i, i);
  for (int i = tid; i < half; i += JAC_THREADS) {
    sm.offd[0][i] = t_init(rr_player(i, 0, mm), rr_player(mm - 1 - i, 0, mm));
    for (int b = i + 1; b < half; ++b) {
      sm.ba[jac_block(i, b, half)] = (unsigned char)i;
      sm.bb[jac_block(i, b, half)] = (unsigned char)b;
    }
  }
  if (wid == 7) {  // ||T||_F
    double f = 0.0;
    for (int r = lane; r < m; r += 32) {
      const double al = t_init(r, r), be = r > 0 ? t_init(r, r - 1) : 0.0;
      f = fma(al, al, fma(2.0 * be, be, f));
    }
    f = sqrt(warp_sum(f));
    if (lane == 0) sm.thr = 1e-16 * f;
  }
  __syncthreads();
  for (int i = tid; i < nb_mine * 4; i += JAC_THREADS) {
    const int e = rank + (i >> 2) * CL, u = i & 3;
    const int ka = sm.ba[e], kb = sm.bb[e];
    const int a0 = rr_player(ka, 0, mm), a1 = rr_player(mm - 1 - ka, 0, mm);
    const int b0 = rr_player(kb, 0, mm), b1 = rr_player(mm - 1 - kb, 0, mm);
    const int ra = (u & 2) ? (a0 > a1 ? a0 : a1) : (a0 < a1 ? a0 : a1);
    const int cb = (u & 1) ? (b0 > b1 ? b0 : b1) : (b0 < b1 ? b0 : b1);
    sm.blk[0][i >> 2][u] = t_init(ra, cb);
  }
  __syncthreads();
  // every CTA's copies are initialised before another pushes into them
  if constexpr (CL > 1) cluster_barrier();
  const int64_t thr = abs_bits(sm.thr);

  int sweep = 0, buf = 0;
  // this thread's element of the blocks, and its pairs; warp 0 comes last
  const int el0 = wid > 0 ? tid - 32 : JAC_THREADS - 32 + lane;
  int ka0 = 0, kb0 = 0;
  if (el0 < nb_mine * 4) {
    ka0 = sm.ba[rank + (el0 >> 2) * CL];
    kb0 = sm.bb[rank + (el0 >> 2) * CL];
  }
  // Y <- Y J with the angles of copy `at`, one round behind
  auto update_y = [&](int at) {
    for (int i = tid - 32 * JAC_Y_WARP; i < half * ny_rows; i += JAC_THREADS - 32 * JAC_Y_WARP) {
      const int k = i / ny_rows, row = rank + (i - k * ny_rows) * CL;
      const int w = sm.pq[at][k];
      if (!(w >> 16)) continue;
      const int p = w & 0xff, q = (w >> 8) & 0xff;
      const double c = sm.rc[at][k], sn = sm.rs[at][k];
      const double gy = Y[row * JLD + p], hy = Y[row * JLD + q];
      Y[row * JLD + p] = c * gy - sn * hy;
      Y[row * JLD + q] = sn * gy + c * hy;
    }
  };
  for (; sweep < JAC_MAX_SWEEPS; ++sweep) {
    unsigned any = 0;  // (warp 0's)
    for (int round = 0; round < mm - 1; ++round, buf ^= 1) {
      const int nb = buf ^ 1;
      int to = 0;  // the place that it goes to
      if (wid == 0) {
        bool rot = false;
        if (lane < half) {
          const int j0 = rr_player(lane, round, mm), j1 = rr_player(mm - 1 - lane, round, mm);
          const int p = min(j0, j1), q = max(j0, j1);
          const double tpq = sm.offd[buf][lane];
          rot = abs_bits(tpq) > thr;
          sm.pq[buf][lane] = p | q << 8 | (rot ? 1 << 16 : 0);
          if (rot) {
            double t, c, s;
            jac_angle(sm.diag[buf][p], sm.diag[buf][q], tpq, t, c, s);
            sm.rt[buf][lane] = t;
            sm.rc[buf][lane] = c;
            sm.rs[buf][lane] = s;
          }
        }
        any |= __ballot_sync(0xffffffffu, rot);
        if (lane == 0) sm.any = any != 0;
      } else if (el0 < nb_mine * 4) {
        to = dest_of(el0, round);
      }
      __syncthreads();
      // T <- J^T T J: block (a, b) becomes J_a^T T[{p_a,q_a},{p_b,q_b}] J_b,
      // a lane per element (lanes 4 j ... 4 j + 3 hold one block, row-major)
      if (el0 - lane < nb_mine * 4) {  // uniform per warp
        const bool in = el0 < nb_mine * 4;
        if (wid == 0 && in) to = dest_of(el0, round);
        const bool ra = in && (sm.pq[buf][ka0] >> 16), rb = in && (sm.pq[buf][kb0] >> 16);
        double x = in ? sm.blk[buf][el0 >> 2][el0 & 3] : 0.0;
        const double xr = __shfl_xor_sync(0xffffffffu, x, 2);  // the other row
        if (ra) {  // J_a^T
          const double sn = sm.rs[buf][ka0];
          x = fma(sm.rc[buf][ka0], x, ((el0 & 2) ? sn : -sn) * xr);
        }
        const double xc = __shfl_xor_sync(0xffffffffu, x, 1);  // the other column
        if (rb) {  // J_b
          const double sn = sm.rs[buf][kb0];
          x = fma(sm.rc[buf][kb0], x, ((el0 & 1) ? sn : -sn) * xc);
        }
        if (in) put(to, x, nb);
      }
      if (wid == 0 && lane < half) {
        // the pairs' own elements: the diagonal, and the off-diagonal one
        // (zero once rotated; every CTA knows it and places what it owns)
        const int w = sm.pq[buf][lane], p = w & 0xff, q = (w >> 8) & 0xff;
        double v = sm.offd[buf][lane], tpp = sm.diag[buf][p], tqq = sm.diag[buf][q];
        if (w >> 16) {
          const double t = sm.rt[buf][lane];
          tpp = fma(-t, v, tpp);
          tqq = fma(t, v, tqq);
          v = 0.0;
        }
        sm.diag[nb][p] = tpp;
        sm.diag[nb][q] = tqq;
        const int at = dest(p, q, round);
        if (at < 0) sm.offd[nb][-1 - at] = v;  // (two players only: the same pair again)
        else if ((at >> 2) % CL == rank) sm.blk[nb][(at >> 2) / CL][at & 3] = v;
      }
      // the angles in copy `buf` stay for this round's Y, which runs until
      // the next round's angles are complete
      if constexpr (CL > 1) {
        cluster_arrive();
        if (wid >= JAC_Y_WARP) update_y(buf);
        cluster_wait();
      } else {
        __syncthreads();
        if (wid >= JAC_Y_WARP) update_y(buf);
      }
    }
    __syncthreads();
    if (!sm.any) break;
    // When no |t_pq| off the diagonal exceeds thr, the next sweep's first
    // round rotates nothing, so T stays as it is and no later round rotates
    // either: that sweep is skipped (same bits, and the same sweep count).
    // The CTAs of a cluster join their blocks' maxima: one decision.
    {
      long long mx = 0;
      for (int i = tid; i < nb_mine * 4; i += JAC_THREADS)
        mx = max(mx, (long long)abs_bits(sm.blk[buf][i >> 2][i & 3]));
      if (tid < half) mx = max(mx, (long long)abs_bits(sm.offd[buf][tid]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0) sm.wmax[wid] = mx;
      __syncthreads();
      mx = sm.wmax[0];
#pragma unroll
      for (int w = 1; w < JAC_THREADS / 32; ++w) mx = max(mx, sm.wmax[w]);
      if constexpr (CL > 1) {
        if (tid < CL)
          st_cluster_f64(cluster_map(smem_addr(&sm.cmax[sweep & 1][rank]), (uint32_t)tid),
                         __longlong_as_double(mx));
        cluster_barrier();
#pragma unroll
        for (int q = 0; q < CL; ++q)
          mx = max(mx, (long long)__double_as_longlong(sm.cmax[sweep & 1][q]));
      }
      if (mx <= thr) {
        ++sweep;
        break;
      }
    }
    __syncthreads();  // (wmax and any are written again)
  }
  __syncthreads();
  if constexpr (CL > 1) {
    // the rows of Y into CTA 0, which selects and writes the outputs
    const uint32_t Y0 = cluster_map(smem_addr(Y), 0u);
    if (rank != 0)
      for (int i = tid; i < ny_rows * mm; i += JAC_THREADS) {
        const int row = rank + (i / mm) * CL, c = i % mm;
        st_cluster_f64(Y0 + (uint32_t)(row * JLD + c) * 8u, Y[row * JLD + c]);
      }
    cluster_barrier();
    if (rank != 0) return;
  }
  // The Ritz values, unscaled.  Divided by 2^texp, a diagonal element below 2^-1022
  // of the largest has lost bits; a rotation would have moved it by at least
  // 1e-33 of ||T||, so that one still there (or lost entirely) is alpha itself.
  double* const theta = sm.diag[buf ^ 1];
  int* const sel = sm.sel;
  constexpr int64_t NORMAL = (int64_t)1 << 52;
  if (tid < m) {
    const double d = sm.diag[buf][tid];
    const bool lost = abs_bits(d) < NORMAL && abs_bits(t_init(tid, tid)) < NORMAL;
    theta[tid] = lost ? a.alpha[tid] : scalbn(d, texp);
  }

  // selection: rank of each Ritz value under the selection order
  if (tid < m) sm.key[tid] = order_key(theta[tid]);
  __syncthreads();
  if (tid < m) {
    const int64_t th = sm.key[tid];
    int before = 0;
    for (int l = 0; l < m; ++l)
      if (l != tid && sel_before(sm.key[l], l, th, tid, a.which)) ++before;
    sel[before] = tid;
  }
  __syncthreads();
  double* eigvals_dev = a.eigvals_dev;
  if (a.st != nullptr) eigvals_dev = a.st->eigvals_out;
  // one warp per selected pair: sign, outputs, Ritz coefficients
  for (int k = wid; k < a.K; k += JAC_THREADS / 32) {
    const int j = sel[k];
    // largest-magnitude entry of y (lowest index on ties)
    int64_t best = -1;
    int bi = m;
    for (int r = lane; r < m; r += 32) {
      const int64_t v = abs_bits(Y[r * JLD + j]);
      if (v > best) {
        best = v;
        bi = r;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const int64_t ob = __shfl_xor_sync(0xffffffffu, (long long)best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    const int64_t flip = __double_as_longlong(Y[bi * JLD + j]) & INT64_MIN;
    if (lane == 0) {
      const double th = theta[j];
      a.theta_out[k] = th;
      if (eigvals_dev) eigvals_dev[k] = th;
      if (a.resid_out) a.resid_out[k] = fabs(a.beta[m] * Y[(m - 1) * JLD + j]);
    }
    for (int r = lane; r < m; r += 32) {
      const double y = __longlong_as_double(__double_as_longlong(Y[r * JLD + j]) ^ flip);
      if (a.Y_out) a.Y_out[(size_t)k * m + r] = y;
      if (a.C_out) a.C_out[(size_t)r * a.K + k] = (a.s ? a.s[r] : 1.0) * y;
    }
  }
  if (tid == 0) {
    const int conv = sweep < JAC_MAX_SWEEPS;
    if (a.sweeps_out) *a.sweeps_out = sweep;
    if (a.status_out) *a.status_out = conv ? 0 : (int)TE_ERR_NOT_CONVERGED;
    if (a.st) {
      a.st->sweeps = sweep;
      if (!conv && a.st->status == 0) a.st->status = (int)TE_ERR_NOT_CONVERGED;
    }
  }
}

template <int CL>
static cudaError_t jacobi_prepare_t() {
  return cudaFuncSetAttribute(jacobi_kernel<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(JacSmem<CL>));
}

cudaError_t jacobi_prepare() {
  cudaError_t e = jacobi_prepare_t<1>();
  if (e == cudaSuccess) e = jacobi_prepare_t<4>();
  if (e == cudaSuccess) e = jacobi_prepare_t<8>();
  return e;
}

template <int CL>
static cudaError_t launch_jacobi_t(const JacobiArgs& a, cudaStream_t s) {
  if constexpr (CL == 1) {
    jacobi_kernel<1><<<1, JAC_THREADS, sizeof(JacSmem<1>), s>>>(a);
    return cudaGetLastError();
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL, 1, 1);
    cfg.blockDim = dim3(JAC_THREADS, 1, 1);
    cfg.dynamicSmemBytes = sizeof(JacSmem<CL>);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, jacobi_kernel<CL>, a);
  }
}

cudaError_t launch_jacobi(const JacobiArgs& a, cudaStream_t s) {
  if (a.m < JAC_CLUSTER4_MIN_M) return launch_jacobi_t<1>(a, s);
  if (a.m < JAC_CLUSTER8_MIN_M) return launch_jacobi_t<4>(a, s);
  return launch_jacobi_t<8>(a, s);
}

}  // namespace te
