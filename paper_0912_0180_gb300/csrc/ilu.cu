// ilu.cu -- ILU(0) smoothing on 1D and 2D multigrid levels (Section 6.1: the smoother of the
// paper's experiments).
//
// The factors: L (unit lower) and U (upper) keep the sparsity pattern of the level matrix M
// (unknowns in lexicographic order, x fastest) and L U agrees with M on that pattern -- the
// row-wise form of Gaussian elimination with every fill entry outside the pattern dropped.  The
// pattern is the level's stencil: the Shortley-Weller cross (3 points in 1D, 5 in 2D) or the
// 9-point box of a Galerkin coarse operator.  One smoothing step is the defect correction
// u <- u + (L U)^{-1} (f - M u).
//
// Both the factorisation and the two triangular solves are recurrences over the rows: the row of
// (i, j) needs rows (i-1, j-1), (i, j-1), (i+1, j-1) and (i-1, j) first (the solve with U the
// mirror image).  The factors are computed once, in FP64, at create by one block that walks the
// wavefronts t = i + 2j with a barrier between them, and then packed for the solve.
//
// The solve runs in one cluster.  A warp takes a strip of 32 rows, a lane per row, and walks the
// columns skewed: at step t lane l is at column i = t - K l (K = 2 for the 9-point box, whose row
// above must be one column ahead, 1 for the cross), so every neighbour in the row above is what the
// lane above computed one to three steps ago -- a shuffle, no barrier and no shared memory.  The
// strips form a pipeline: a strip's last row goes value by value to the block of the strip below, by
// asynchronous stores into its shared memory that count on an mbarrier per 8 steps (no fence stalls
// the sender), and a strip runs 72 (box) or 40 (cross) steps behind the one above.  L's strips run
// down, U's run up in the same launch, U's entries multiplied by the pivot's reciprocal at create.
// What bounds it: the chain of n0 + K n1 (and the pipeline's lag) dependent steps per solve, a step
// being one shuffle and two complex multiply-adds in FP32, and in FP64 the strip's 8 to 20 DFMAs at 2
// lanes a clock of its SM.  The factors and the right-hand side are stored in the order the lanes
// read them ([strip][step][entry][lane]) and fetched 16 to 24 steps ahead (cp.async), since nothing
// else runs on the SM to hide a load.  One block walking the wavefronts with a barrier each cost 1.1
// us a wavefront in FP32; a V(0,1) cycle of MP3's operators on 640^2 unknowns went from 8.40 to 0.99
// ms, 0.95 with the factors of eight steps read into registers at once (about 0.1 us a step, 54 instructions of
// which half wait on the one before).
//
// The waits for a hand-over are bounded (about a second).  One that runs out makes the rest NaN and sets a
// pinned host word; a cluster barrier at the end keeps every block until all have sent (no measurable cost: 951 us
// against 956 without it).  The cluster is as large as the device grants, 16 blocks on GB300.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "stencil.cuh"

namespace helm {

constexpr int ILU_FACTOR_THREADS = 512;  // the factorisation

// whether (i + di, j + dj) is in row (i, j)'s pattern: inside the grid and the 3 x 3 box (the
// elimination also produces offsets of 2, fill outside every pattern), on the cross unless box
__device__ __forceinline__ bool ilu_in_pattern(int n0, int n1, bool box, int i, int j, int di, int dj) {
  const int ii = i + di, jj = j + dj;
  if (ii < 0 || ii >= n0 || jj < 0 || jj >= n1) return false;
  if (di < -1 || di > 1 || dj < -1 || dj > 1) return false;
  return box || di == 0 || dj == 0;
}

// The factors of one level, FP64.  stg: the Galerkin weights [9][ntot] (box pattern), else the
// Shortley-Weller rows of op.  f64: the 9 entries of point p at [9p + s], slot s = 3 (dj + 1) + (di + 1)
// of the neighbour (i + di, j + dj): L at the lower slots 0..3, U at 5..8, the pivot's reciprocal at 4.
__global__ void __launch_bounds__(ILU_FACTOR_THREADS) k_ilu_factor(OpView<double> op, const double2* __restrict__ stg,
                                                            double2* __restrict__ f64) {
  const int n0 = op.n[0], n1 = op.n[1];
  const long ntot = (long)n0 * n1;
  const bool box = stg != nullptr;
  const int lo[4][2] = {{-1, -1}, {0, -1}, {1, -1}, {-1, 0}};  // lower neighbours, columns increasing
  const int up[4][2] = {{1, 0}, {-1, 1}, {0, 1}, {1, 1}};      // upper neighbours
  const int waves = n0 + 2 * (n1 - 1);
  for (int t = 0; t < waves; ++t) {
    for (int j = threadIdx.x; j < n1; j += blockDim.x) {
      const int i = t - 2 * j;
      if (i < 0 || i >= n0) continue;
      const long p = i + (long)n0 * j;
      double2 a[9];
#pragma unroll
      for (int s = 0; s < 9; ++s) a[s] = make_double2(0.0, 0.0);
      if (box) {
#pragma unroll
        for (int s = 0; s < 9; ++s)
          if (ilu_in_pattern(n0, n1, true, i, j, s % 3 - 1, s / 3 - 1)) a[s] = stg[(long)s * ntot + p];
      } else {
        double2 d = op.a0[0][i];
        if (n1 > 1) d = cadd<double>(d, op.a0[1][j]);
        const double ph = op.phi ? op.phi[p] : op.phi0;
        d = cadd<double>(d, somm_diag(op, i, j, 0, ph));
        a[4] = csub<double>(d, sigma64(op, p, ph));
        if (i > 0) a[3] = op.am[0][i];
        if (i < n0 - 1) a[5] = op.ap[0][i];
        if (j > 0) a[1] = op.am[1][j];
        if (j < n1 - 1) a[7] = op.ap[1][j];
      }
      // eliminate with the rows above, in increasing column order; fill outside the pattern is
      // dropped
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int di = lo[k][0], dj = lo[k][1];
        if (!ilu_in_pattern(n0, n1, box, i, j, di, dj)) continue;
        const double2* uk = f64 + 9 * (p + di + (long)n0 * dj);  // row k, factored on an earlier wavefront
        const int sk = 3 * (dj + 1) + (di + 1);
        const double2 l = cmul<double>(a[sk], uk[4]);  // uk[4]: 1 / row k's pivot
        a[sk] = l;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int ei = up[v][0], ej = up[v][1];
          if (!ilu_in_pattern(n0, n1, box, i + di, j + dj, ei, ej)) continue;
          const int ti = di + ei, tj = dj + ej;
          if (!ilu_in_pattern(n0, n1, box, i, j, ti, tj)) continue;
          const int st = 3 * (tj + 1) + (ti + 1);
          a[st] = csub<double>(a[st], cmul<double>(l, uk[3 * (ej + 1) + (ei + 1)]));
        }
      }
      a[4] = crecip<double>(a[4]);
#pragma unroll
      for (int s = 0; s < 9; ++s) f64[9 * p + s] = a[s];
    }
    __syncthreads();
  }
}

// ---- the solve's layout -----------------------------------------------------------------------
constexpr int ILU_CH = 8;       // steps per chunk (fetches and hand-overs)
constexpr int ILU_MAX_WARPS = 8;
constexpr int ILU_MAX_BLOCKS = 16;
template <bool BOX> struct IluShape {
  static constexpr int K = BOX ? 2 : 1;   // columns a lane lies behind the lane above
  static constexpr int NL = BOX ? 4 : 2;  // L's entries a point
  static constexpr int NU = BOX ? 5 : 3;  // U's, and the pivot's reciprocal first
};
// stored rows of a strip: a level of fewer than 32 rows (a 1D level has one) stores only those
__host__ __device__ inline int ilu_width(int n1) { return n1 < 32 ? n1 : 32; }
__host__ __device__ inline int ilu_steps(int n0, int n1, bool box) {  // a strip's steps, whole chunks
  return (n0 + (ilu_width(n1) - 1) * (box ? 2 : 1) + ILU_CH - 1) / ILU_CH * ILU_CH;
}
// place of point (i, j) in a skewed vector (entry e of `per` entries a point) of width w
__host__ __device__ inline long ilu_at(int i, int j, int steps, int k, int per, int e, int w) {
  const int l = j & 31;
  return (((long)(j >> 5) * steps + i + k * l) * per + e) * w + l;
}

// Packs the natural factors for the solve: lo = L's entries, up = 1 / u_pp and U's entries times it.
template <typename T, bool BOX>
__global__ void k_ilu_pack(const double2* __restrict__ f, int n0, int n1, int steps, cx<T>* __restrict__ lo,
                           cx<T>* __restrict__ up) {
  using S = IluShape<BOX>;
  const long p = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (p >= (long)n0 * n1) return;
  const int i = (int)(p % n0), j = (int)(p / n0);
  const double2* a = f + 9 * p;
  const int w = ilu_width(n1);
  const int sl[4] = {BOX ? 0 : 1, BOX ? 1 : 3, 2, 3}, su[4] = {5, BOX ? 6 : 7, 7, 8};
#pragma unroll
  for (int e = 0; e < S::NL; ++e) lo[ilu_at(i, j, steps, S::K, S::NL, e, w)] = cconv<T, double>(a[sl[e]]);
  up[ilu_at(i, j, steps, S::K, S::NU, 0, w)] = cconv<T, double>(a[4]);
#pragma unroll
  for (int e = 1; e < S::NU; ++e)
    up[ilu_at(i, j, steps, S::K, S::NU, e, w)] = cconv<T, double>(cmul<double>(a[4], a[su[e - 1]]));
}

// v = f - M u (or f, from the zero guess) in the skewed order of the solve.
template <typename T, int DIM, bool BOX>
__global__ void k_ilu_resid(OpView<T> op, const cx<T>* __restrict__ u, const cx<T>* __restrict__ f, int steps,
                            cx<T>* __restrict__ v, const int* skip) {
  pdl_entry();
  if (skip && *skip) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= op.n[0] || j >= op.n[1]) return;
  const long p = i + (long)op.n[0] * j;
  cx<T> r = f[p];
  if (u) {
    if constexpr (BOX) {
      cx<T> acc = mkc<T>(T(0), T(0));
#pragma unroll
      for (int s = 0; s < 9; ++s) {
        const int ii = i + s % 3 - 1, jj = j + s / 3 - 1;
        if (s == 4 || ii < 0 || ii >= op.n[0] || jj < 0 || jj >= op.n[1]) continue;
        acc = cfma<T>(op.stg[(long)s * op.ntot + p], u[ii + (long)jj * op.n[0]], acc);
      }
      r = csub<T>(r, cfma<T>(op.stg[4 * op.ntot + p], u[p], acc));
    } else {
      r = csub<T>(r, op_row<T, T, DIM>(op, u, i, j, 0, p));
    }
  }
  v[ilu_at(i, j, steps, IluShape<BOX>::K, 1, 0, ilu_width(op.n[1]))] = r;
}

// u += z (u = z from the zero guess), z skewed; wide: u also as complex128.
template <typename T, bool BOX>
__global__ void k_ilu_add(int n0, int n1, int steps, const cx<T>* __restrict__ z, cx<T>* __restrict__ u, int zero,
                          double2* __restrict__ wide, const int* skip) {
  pdl_entry();
  if (skip && *skip) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= n0 || j >= n1) return;
  const long p = i + (long)n0 * j;
  const cx<T> d = z[ilu_at(i, j, steps, IluShape<BOX>::K, 1, 0, ilu_width(n1))];
  const cx<T> r = zero ? d : cadd<T>(u[p], d);
  u[p] = r;
  if (wide) wide[p] = cconv<double, T>(r);
}

template <typename T> struct IluArgs {
  int n0, n1, steps;
  int s0, s1;    // strips of this launch, one after another over its blocks' warps
  int passes;    // bit 0: L, bit 1: U
  int rows;      // whether the strips hand their edge row over in shared memory
  long long wait;  // clock cycles after which a wait for a hand-over gives up
  int mute;        // the strip that hands nothing over (tests), or -1
  int* word;       // pinned host word, set when a wait gave up
  const cx<T>*lo, *up;
  cx<T>* v;      // right-hand side, y and z in turn
};

// ---- the hand-over ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned ilu_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned ilu_map(unsigned a, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// (predicated, not branched around: a branch a step costs its resolution; no memory clobber: the next
// steps' loads may move above it)
__device__ __forceinline__ void ilu_send(bool on, unsigned to, unsigned bar, float2 v) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 d;\n setp.ne.u32 p, %0, 0;\n mov.b64 d, {%2, %3};\n"
      " @p st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%1], d, [%4];\n}" ::"r"((unsigned)on),
      "r"(to), "f"(v.x), "f"(v.y), "r"(bar));
}
__device__ __forceinline__ void ilu_send(bool on, unsigned to, unsigned bar, double2 v) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n"
      " @p st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%1], {%2, %3}, [%4];\n}" ::"r"((unsigned)on),
      "r"(to), "l"(__double_as_longlong(v.x)), "l"(__double_as_longlong(v.y)), "r"(bar));
}
__device__ __forceinline__ void ilu_expect(unsigned bar, unsigned bytes) {
  asm volatile("{\n .reg .b64 t;\n mbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1;\n}" ::"r"(bar), "r"(bytes) : "memory");
}
// waits for the barrier's first phase, for `limit` clock cycles at most (default: about a second); false
// when that runs out
__device__ __forceinline__ bool ilu_wait(unsigned bar, long long limit) {
  const long long t0 = clock64();
  for (int tries = 0; tries < (1 << 24); ++tries) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(0u)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > limit) break;
  }
  return false;
}
__device__ __forceinline__ void ilu_fetch(float2* dst, const float2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ilu_smem(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void ilu_fetch(double2* dst, const double2* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ilu_smem(dst)), "l"(src) : "memory");
}
template <int N> __device__ __forceinline__ void ilu_landed() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// valid columns of the edge row among a chunk's steps [m CH, m CH + CH): the edge lane is `lag` columns
// behind the step
__device__ __forceinline__ int ilu_sent(int m, int lag, int n0) {
  const int lo = max(m * ILU_CH - lag, 0), hi = min(m * ILU_CH + ILU_CH - lag, n0);
  return max(hi - lo, 0);
}

// After a wait gave up, and once every strip has sent what it will: until what was sent to the `nc` chunks'
// barriers at `bars` has landed (bounded: a strip that never sent leaves its barriers open).
__device__ __forceinline__ void ilu_drain(unsigned bars, int nc, int lag, int n0) {
  const long long t0 = clock64();
  for (int m = threadIdx.x & 31; m < nc; m += 32) {
    if (ilu_sent(m, lag, n0) == 0) continue;
    unsigned ok = 0;
    for (int tries = 0; !ok && tries < (1 << 16); ++tries) {
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
          : "=r"(ok)
          : "r"(bars + m * 8), "r"(0u)
          : "memory");
      if (clock64() - t0 > (1 << 20)) return;
    }
  }
}

template <typename T>
__device__ __forceinline__ cx<T> ilu_shfl(cx<T> v, int lane) {
  return mkc<T>(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}

// One strip's solve with L (UP = false: chunks and rows ascending) or U (UP = true: both descending).
// ring: this warp's fetch ring; row, bars: the edge row it receives and the barriers of its chunks;
// to_row, to_bar: the same in the receiving strip (0: nobody); edge: where the edge row comes from (0
// nowhere, 1 the row in shared memory, 2 the other strip's values in v).
// FEW: the level's only strip, of fewer than 32 rows.
// Returns whether every hand-over arrived in time (uniform over the warp); if not, the values after the
// missing ones are NaN.
template <typename T, bool BOX, bool UP, int DEPTH, bool FEW>
__device__ __forceinline__ bool ilu_strip(const IluArgs<T>& g, int strip, cx<T>* ring, const cx<T>* row, unsigned bars,
                                          unsigned to_row, unsigned to_bar, int edge) {
  using S = IluShape<BOX>;
  constexpr int K = S::K, NE = UP ? S::NU : S::NL, SL = NE + 1, CH = ILU_CH;
  // lane 0 (31) takes the edge row, lane 31 (0) gives it; new value per step: one column ahead (box)
  constexpr int TAKE = UP ? 31 : 0, GIVE = UP ? 0 : 31, LAG = UP ? 0 : 31 * K, AHEAD = BOX ? 1 : 0;
  const int lane = threadIdx.x & 31;
  const int n0 = g.n0, steps = g.steps, nc = steps / CH;
  const bool has_row = strip * 32 + lane < g.n1;
  const cx<T> zero = mkc<T>(T(0), T(0));
  const int W = FEW ? g.n1 : 32;
  cx<T>* const v = g.v + (long)strip * steps * W + lane;
  const cx<T>* const fac = (UP ? g.up : g.lo) + (long)strip * steps * NE * W + lane;
  const cx<T>* const other = g.v + (long)(UP ? strip + 1 : strip - 1) * steps * 32 + GIVE;
  const bool gives = lane == GIVE && to_row != 0 && strip != g.mute;
  bool failed = false;
  int armed = 0;  // chunks of the edge row waited for
  auto chunk = [&](int c) { return UP ? nc - 1 - c : c; };  // c-th chunk in this direction
  auto fetch = [&](int c) {
    if (c < nc && (!FEW || has_row)) {
      cx<T>* const to = ring + (c % DEPTH) * CH * SL * 32 + lane;
      const long t0 = (long)chunk(c) * CH;
#pragma unroll
      for (int k = 0; k < CH; ++k) {
#pragma unroll
        for (int e = 0; e < NE; ++e) ilu_fetch(to + (k * SL + e) * 32, fac + ((t0 + k) * NE + e) * W);
        ilu_fetch(to + (k * SL + NE) * 32, v + (t0 + k) * W);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // column that the take lane's new value has at step t; its chunk is the giving lane's
  auto col_new = [&](int t) { return UP ? t - 31 * K - AHEAD : t + AHEAD; };
  auto ready = [&](int c) {  // the edge values of this direction's chunk c, and the column before
    if (edge != 1) return;
    // giving lane's chunk of the last column needed, in this direction's count: UP gives column t at
    // its step t, else column t - 31 K
    const int need = min(c + (BOX ? 8 : 4), nc - 1);
    while (armed <= need) {
      const int m = chunk(armed), n = ilu_sent(m, LAG, n0);
      if (n) {
        const unsigned b = bars + m * 8;
        if (lane == 0) ilu_expect(b, n * (unsigned)sizeof(cx<T>));
        __syncwarp();
        if (!failed) failed = !ilu_wait(b, g.wait);
      }
      ++armed;
    }
    failed = __any_sync(0xffffffffu, failed);
  };
  auto edge_at = [&](int col) -> cx<T> {
    if (edge == 0 || col < 0 || col >= n0) return zero;
    return edge == 1 ? row[col] : __ldcg(other + (long)(col + LAG) * 32);
  };
#pragma unroll
  for (int c = 0; c < DEPTH - 1; ++c) fetch(c);
  ready(0);
  // neighbours in the row above (below): a and b one and two columns behind the new value c (box)
  cx<T> a = zero, b = zero, prev = zero;
  if (BOX && lane == TAKE) b = edge_at(col_new(UP ? steps : -1));
  for (int c = 0; c < nc; ++c) {
    fetch(c + DEPTH - 1);
    ready(c);
    if (failed) prev = b = mkc<T>(T(NAN), T(NAN));  // a wait ran out
    const int m = chunk(c);
    // lane k holds the take lane's new value of the chunk's k-th step
    const cx<T> en = lane < CH ? edge_at(col_new(UP ? m * CH + CH - 1 - lane : m * CH + lane)) : zero;
    ilu_landed<DEPTH - 1>();
    const cx<T>* const at = ring + (c % DEPTH) * CH * SL * 32 + lane;
    // a few steps' factors and right-hand sides into registers at once: one warp has nobody to hide a
    // shared-memory load behind
    constexpr int BS = sizeof(T) == 4 ? 8 : 4;
#pragma unroll
    for (int kb = 0; kb < CH; kb += BS) {
      cx<T> q[BS][SL];
#pragma unroll
      for (int k = 0; k < BS; ++k)
#pragma unroll
        for (int e = 0; e < SL; ++e) q[k][e] = at[((UP ? CH - 1 - kb - k : kb + k) * SL + e) * 32];
#pragma unroll
      for (int k = 0; k < BS; ++k) {
        const int kk = UP ? CH - 1 - kb - k : kb + k, t = m * CH + kk, i = t - K * lane;
        const cx<T> x = q[k][NE];
        // the lane above's (below's) last value
        cx<T> nw = UP ? mkc<T>(__shfl_down_sync(0xffffffffu, prev.x, 1), __shfl_down_sync(0xffffffffu, prev.y, 1))
                      : mkc<T>(__shfl_up_sync(0xffffffffu, prev.x, 1), __shfl_up_sync(0xffffffffu, prev.y, 1));
        const cx<T> ek = ilu_shfl<T>(en, kb + k);
        if (lane == TAKE) nw = ek;
        cx<T> r;
        if (UP) {
          r = cmul<T>(q[k][0], x);
          if (BOX) r = cfms<T>(q[k][BOX ? 4 : 0], a, cfms<T>(q[k][BOX ? 3 : 0], b, r));  // (i+1, j+1), (i, j+1)
          r = cfms<T>(q[k][1], prev, r);                                                 // (i+1, j)
          r = cfms<T>(q[k][2], nw, r);                                                   // (i-1, j+1); cross (i, j+1)
        } else {
          r = x;
          if (BOX) r = cfms<T>(q[k][1], b, cfms<T>(q[k][0], a, r));  // (i-1, j-1), (i, j-1)
          r = cfms<T>(q[k][BOX ? 3 : 1], prev, r);                   // (i-1, j)
          r = cfms<T>(q[k][BOX ? 2 : 0], nw, r);                     // (i+1, j-1); cross (i, j-1)
        }
        const bool in = has_row && i >= 0 && i < n0;
        if (!in) r = zero;  // a point outside the grid is zero for the neighbours
        else v[(long)t * W] = r;
        ilu_send(gives && in, to_row + (unsigned)(i * (int)sizeof(cx<T>)), to_bar + m * 8, r);
        a = b;
        b = nw;
        prev = r;
      }
    }
  }
  ilu_landed<0>();
  return !failed;
}

template <typename T, bool BOX, int DEPTH, bool FEW>
__global__ void k_ilu_solve(const IluArgs<T> g, const int* skip) {
  pdl_entry();
  if (skip && *skip) return;
  using S = IluShape<BOX>;
  extern __shared__ __align__(16) unsigned char ilu_sm[];
  constexpr int RING = DEPTH * ILU_CH * (S::NU + 1) * 32;
  const int wpc = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31, nc = g.steps / ILU_CH;
  cx<T>* const ring = reinterpret_cast<cx<T>*>(ilu_sm) + w * RING;
  cx<T>* const rows0 = reinterpret_cast<cx<T>*>(ilu_sm) + wpc * RING;
  const int row_n = g.rows ? g.n0 : 0;
  cx<T>* const row = rows0 + w * row_n;
  const unsigned bars0 = ilu_smem(rows0 + wpc * row_n), rowb0 = ilu_smem(rows0);
  const int strip = g.s0 + (int)blockIdx.x * wpc + w;
  if (g.rows) {
    for (int m = lane; m < 2 * nc; m += 32)  // L's hand-overs, then U's
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars0 + (2 * w * nc + m) * 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
  auto row_of = [&](int st) {  // the edge row and barriers of strip st (0: not in this launch)
    const int q = st - g.s0, blk = q / wpc, ww = q % wpc;
    struct P { unsigned row, bar; } r{0u, 0u};
    if (g.rows && st >= g.s0 && st < g.s1) {
      r.row = ilu_map(rowb0 + (unsigned)(ww * row_n * sizeof(cx<T>)), blk);
      r.bar = ilu_map(bars0 + (unsigned)(2 * ww * nc * 8), blk);
    }
    return r;
  };
  const unsigned bars = bars0 + 2 * w * nc * 8;
  const int strips = (g.n1 + 31) / 32;
  const bool on = strip < g.s1;  // nothing is sent to the others
  const int edge_l = strip == 0 ? 0 : strip > g.s0 ? 1 : 2, edge_u = strip == strips - 1 ? 0 : strip < g.s1 - 1 ? 1 : 2;
  bool ok = true;
  if (on && (g.passes & 1)) {
    const auto to = row_of(strip + 1);
    ok = ilu_strip<T, BOX, false, DEPTH, FEW>(g, strip, ring, row, bars, to.row, to.bar, edge_l);
    __threadfence();  // the values of this pass are fetched asynchronously in the next
    __syncwarp();
  }
  if (on && (g.passes & 2)) {
    const auto to = row_of(strip - 1);
    ok = ilu_strip<T, BOX, true, DEPTH, FEW>(g, strip, ring, row, bars + nc * 8, to.row, to.bar ? to.bar + nc * 8 : 0u, edge_u) && ok;
  }
  if (!ok && lane == 0) *reinterpret_cast<volatile int*>(g.word) = 1;
  if (!g.rows) return;
  // A strip whose wait gave up did not wait for what came later, and a store into the shared memory of a
  // block that has left is undefined: every block stays until all strips have sent, and then until what
  // was sent to it has landed.
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  if (!ok) {
    if ((g.passes & 1) && edge_l == 1) ilu_drain(bars, nc, 31 * S::K, g.n0);
    if ((g.passes & 2) && edge_u == 1) ilu_drain(bars + nc * 8, nc, 0, g.n0);
  }
}

helm_status ilu_check(int dim, const int n[3], bool f32) {
  if (dim > 2) {
    set_error("ILU(0) smoothing runs on 1D and 2D levels");
    return HELM_ERR_ARG;
  }
  const int most = (int)(ILU_ROW_BYTES / (4 * (f32 ? sizeof(float2) : sizeof(double2))));
  if (n[1] > most) {
    set_error("ILU(0) smoothing takes at most " + std::to_string(most) + " rows in this precision");
    return HELM_ERR_ARG;
  }
  return HELM_OK;
}

namespace {

constexpr size_t ILU_SMEM_MAX = 224 * 1024;

// The plan for clusters of at most `most` blocks.  The fewest warps a block (a strip has its SM's loads and, in FP64, its FP64 pipe to itself) that put
// all strips into one cluster; where the edge rows do not fit, fewer strips a launch; a row too long
// for shared memory is handed over in memory, one strip a launch.
IluPlan ilu_plan(int n0, int n1, bool box, size_t esz, int most) {
  const int strips = (n1 + 31) / 32, nc = ilu_steps(n0, n1, box) / ILU_CH;
  auto bytes = [&](int wpc, int depth, int rows) {
    return wpc * (esz * depth * ILU_CH * ((box ? 5 : 3) + 1) * 32 + (rows ? esz * n0 + 16 * (size_t)nc : 0));
  };
  IluPlan p;
  if (strips > 1) {
    for (int wpc = std::min((strips + most - 1) / most, ILU_MAX_WARPS); wpc >= 1 && !p.rows; --wpc)
      for (int depth = 3; depth >= 2 && !p.rows; --depth)
        if (bytes(wpc, depth, 1) <= ILU_SMEM_MAX) p = IluPlan{wpc, 1, depth, 1, 0};
    if (p.rows)
      while (2 * p.blocks <= most && p.blocks * p.wpc < strips) p.blocks *= 2;
  }
  p.smem = bytes(p.wpc, p.depth, p.rows);
  return p;
}

template <typename T, bool BOX>
cudaError_t ilu_attrs() {
  cudaError_t e = cudaSuccess;
  auto one = [&](auto kern) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ILU_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  };
  one(k_ilu_solve<T, BOX, 2, false>);
  one(k_ilu_solve<T, BOX, 3, false>);
  one(k_ilu_solve<T, BOX, 3, true>);
  return e;
}

// the launch of a plan (attributes in at[2])
cudaLaunchConfig_t ilu_config(const IluPlan& p, cudaLaunchAttribute* at, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.blocks);
  cfg.blockDim = dim3(32 * p.wpc);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = p.blocks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = g_use_pdl ? 2 : 1;
  return cfg;
}

// The plan for the largest cluster that the device grants (the kernels' attributes are set).
template <typename T, bool BOX>
IluPlan ilu_choose(int n0, int n1) {
  for (int most = std::min(ILU_MAX_BLOCKS, g_limits.cluster);; most /= 2) {
    const IluPlan p = ilu_plan(n0, n1, BOX, sizeof(cx<T>), most);
    if (p.blocks == 1) return p;
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = ilu_config(p, at, nullptr);
    cfg.numAttrs = 1;
    int fit = 0;
    const cudaError_t e = p.depth == 3 ? cudaOccupancyMaxActiveClusters(&fit, k_ilu_solve<T, BOX, 3, false>, &cfg)
                                       : cudaOccupancyMaxActiveClusters(&fit, k_ilu_solve<T, BOX, 2, false>, &cfg);
    if (e == cudaSuccess && fit > 0) return p;
    cudaGetLastError();
  }
}

template <typename T, bool BOX>
void ilu_launch(const IluPlan& p, const IluArgs<T>& g, const int* skip, cudaStream_t st) {
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = ilu_config(p, at, st);
  if (g.n1 < 32) cudaLaunchKernelEx(&cfg, k_ilu_solve<T, BOX, 3, true>, g, skip);  // (one strip: depth 3)
  else if (p.depth == 3) cudaLaunchKernelEx(&cfg, k_ilu_solve<T, BOX, 3, false>, g, skip);
  else cudaLaunchKernelEx(&cfg, k_ilu_solve<T, BOX, 2, false>, g, skip);
}

template <typename T, bool BOX>
helm_status ilu_pack(helm_ctx* c, LevelHost& L, const double2* fac, cudaStream_t st) {
  using S = IluShape<BOX>;
  const int steps = ilu_steps(L.n[0], L.n[1], BOX), strips = (L.n[1] + 31) / 32;
  const size_t pts = (size_t)strips * steps * ilu_width(L.n[1]);
  helm_status rc;
  if ((rc = ctx_alloc(c, &L.ilu_lo, sizeof(cx<T>) * S::NL * pts)) != HELM_OK) return rc;
  if ((rc = ctx_alloc(c, &L.ilu_up, sizeof(cx<T>) * S::NU * pts)) != HELM_OK) return rc;
  if ((rc = ctx_alloc(c, &L.ilu_v, sizeof(cx<T>) * pts)) != HELM_OK) return rc;
  // the places outside the grid stay zero
  HELM_CUDA(cudaMemsetAsync(L.ilu_lo, 0, sizeof(cx<T>) * S::NL * pts, st));
  HELM_CUDA(cudaMemsetAsync(L.ilu_up, 0, sizeof(cx<T>) * S::NU * pts, st));
  HELM_CUDA(cudaMemsetAsync(L.ilu_v, 0, sizeof(cx<T>) * pts, st));
  k_ilu_pack<T, BOX><<<(int)((L.ntot + 255) / 256), 256, 0, st>>>(fac, L.n[0], L.n[1], steps, (cx<T>*)L.ilu_lo,
                                                                (cx<T>*)L.ilu_up);
  HELM_CUDA(cudaGetLastError());
  // (here, outside any stream capture)
  HELM_CUDA((ilu_attrs<T, BOX>()));
  L.ilu = ilu_choose<T, BOX>(L.n[0], L.n[1]);
  return HELM_OK;
}

template <typename T, bool BOX>
void ilu_smooth_t(const LevelHost& L, const cx<T>* f, cx<T>* u, bool zero, double2* wide, const int* skip, cudaStream_t st) {
  const int n0 = L.n[0], n1 = L.n[1], steps = ilu_steps(n0, n1, BOX), strips = (n1 + 31) / 32;
  cx<T>* const v = (cx<T>*)L.ilu_v;
  const dim3 b(32, 8), gr((n0 + 31) / 32, (n1 + 7) / 8);
  const cx<T>* u0 = zero ? nullptr : u;
  if (L.dim == 1) launch_pdl(k_ilu_resid<T, 1, BOX>, gr, b, 0, st, L.view<T>(), u0, f, steps, v, skip);
  else launch_pdl(k_ilu_resid<T, 2, BOX>, gr, b, 0, st, L.view<T>(), u0, f, steps, v, skip);
  const IluPlan& p = L.ilu;
  const int per = p.wpc * p.blocks;
  IluArgs<T> g{n0, n1, steps, 0, strips, 3, p.rows, L.ilu_wait, L.ilu_mute, L.ilu_word,
               (const cx<T>*)L.ilu_lo, (const cx<T>*)L.ilu_up, v};
  if (strips <= per) {
    ilu_launch<T, BOX>(p, g, skip, st);
  } else {  // groups of strips: L down, then U up
    const int groups = (strips + per - 1) / per;
    for (int q = 0; q < 2 * groups; ++q) {
      const int grp = q < groups ? q : 2 * groups - 1 - q;
      g.s0 = grp * per;
      g.s1 = std::min(g.s0 + per, strips);
      g.passes = q < groups ? 1 : 2;
      ilu_launch<T, BOX>(p, g, skip, st);
    }
  }
  launch_pdl(k_ilu_add<T, BOX>, gr, b, 0, st, n0, n1, steps, (const cx<T>*)v, u, zero ? 1 : 0, wide, skip);
}

}  // namespace

helm_status ilu_build(helm_ctx* c, LevelHost& L, bool f32, cudaStream_t st) {
  void* fac = nullptr;  // the natural factors, FP64, until they are packed
  std::vector<DevBlock> tmp(1);
  helm_status rc = dev_alloc(&fac, sizeof(double2) * 9 * L.ntot, st, &tmp[0]);
  if (rc != HELM_OK) return rc;
  k_ilu_factor<<<1, std::min(ILU_FACTOR_THREADS, (L.n[1] + 31) / 32 * 32), 0, st>>>(L.view<double>(), L.stg64,
                                                                                  (double2*)fac);
  rc = cuda_err(cudaGetLastError());
  const bool box = L.stg64 != nullptr;
  if (!c->wait_word) {
    if (!(c->wait_word = (int*)pinned_slot_get(sizeof(int)))) rc = cuda_check(cudaErrorMemoryAllocation, "cudaMallocHost");
    else *c->wait_word = 0;
  }
  L.ilu_word = c->wait_word;
  L.ilu_wait = g_limits.ilu_wait;
  L.ilu_mute = g_limits.ilu_mute;
  if (rc == HELM_OK) {
    if (f32) rc = box ? ilu_pack<float, true>(c, L, (double2*)fac, st) : ilu_pack<float, false>(c, L, (double2*)fac, st);
    else rc = box ? ilu_pack<double, true>(c, L, (double2*)fac, st) : ilu_pack<double, false>(c, L, (double2*)fac, st);
  }
  dev_free_all(tmp, st);
  return rc;
}

template <typename T>
void ilu_smooth(const LevelHost& L, const cx<T>* f, cx<T>* u, bool zero, double2* wide, const int* skip, cudaStream_t st) {
  if (L.stg64) ilu_smooth_t<T, true>(L, f, u, zero, wide, skip, st);
  else ilu_smooth_t<T, false>(L, f, u, zero, wide, skip, st);
}

template void ilu_smooth<float>(const LevelHost&, const float2*, float2*, bool, double2*, const int*, cudaStream_t);
template void ilu_smooth<double>(const LevelHost&, const double2*, double2*, bool, double2*, const int*, cudaStream_t);

}  // namespace helm
