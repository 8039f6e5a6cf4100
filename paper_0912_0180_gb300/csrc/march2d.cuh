// march2d.cuh -- the two halves of a 2D V(1,1) level with damped Jacobi, walking down the rows.
//
// The tile kernels of mg_fused.cu stage a tile and its halo in shared memory; at 160 (down) and 240
// (up) instructions a point they are bound by instruction issue and shared-memory traffic in FP32, and
// recompute a halo of 30 to 60 % in FP64, where the pipe is the bound.  Here a warp owns 60 columns (a
// lane two neighbouring ones; the outer lanes are its halo) and walks down the rows with the last three
// rows in registers: x neighbours are shuffles, y neighbours the rows before and after, and every
// element is loaded once, 16 bytes at a time in FP32, two rows ahead of its use.  86 instructions a
// point (down); the halo is 2 lanes of 32 and 3 rows of 2 CR + 3.  The arithmetic is the tile kernels',
// per point (FP64: the prolongation shares a row's sums between its two rows).  Few warps with long
// chains of rows: bound by the latency of the loads (half the copy bandwidth).  It pays on large FP32
// levels (2304^2 cycle 141 -> 123 us, its finest level's kernels 39 and 56 -> 42 and 33 us); the tuner
// takes the tile kernels on small levels and in FP64.
#pragma once
#include "stencil.cuh"

namespace helm {

constexpr int MARCH_THREADS = 128;               // four warps beside each other
constexpr int MARCH_COLS = 30;                   // coarse columns of a warp
constexpr int MARCH_LONG = 16, MARCH_SHORT = 4;  // coarse rows of a block
__host__ __device__ inline int march_strips(int pairs) {  // blocks along x for that many column pairs
  return (pairs + 4 * MARCH_COLS - 1) / (4 * MARCH_COLS);
}

template <typename T> struct Pair {
  cx<T> a, b;
};
// columns c0 (even) and c0 + 1 of a row; outside the grid zero.  vec: pairs of complex64 are 16-byte
// aligned and move as one access (32-byte loads of complex128 pairs were slower: the 2304^2 cycle 138
// us against 131).
template <typename T, typename TI>
__device__ __forceinline__ Pair<T> march_load(const cx<TI>* __restrict__ row, int c0, bool v0, bool v1, bool vec) {
  const cx<T> zero = mkc<T>(T(0), T(0));
  Pair<T> r{zero, zero};
  if constexpr (sizeof(TI) == 4) {
    if (vec) {
      if (v0) {
        const float4 q = *reinterpret_cast<const float4*>(row + c0);
        r.a = mkc<T>(q.x, q.y);
        r.b = mkc<T>(q.z, q.w);
      }
      return r;
    }
  }
  if (v0) r.a = cconv<T, TI>(row[c0]);
  if (v1) r.b = cconv<T, TI>(row[c0 + 1]);
  return r;
}
template <typename T, typename TO>
__device__ __forceinline__ void march_store(cx<TO>* __restrict__ row, int c0, bool v0, bool v1, bool vec, cx<T> a, cx<T> b) {
  if constexpr (sizeof(TO) == 4) {
    if (vec) {
      if (v0) *reinterpret_cast<float4*>(row + c0) = make_float4(a.x, a.y, b.x, b.y);
      return;
    }
  }
  if (v0) row[c0] = cconv<TO, T>(a);
  if (v1) row[c0 + 1] = cconv<TO, T>(b);
}
template <typename T> __device__ __forceinline__ cx<T> march_up1(cx<T> v) {
  return mkc<T>(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
template <typename T> __device__ __forceinline__ cx<T> march_down1(cx<T> v) {
  return mkc<T>(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}

// The off-diagonal sums of a lane's two points in row j, from the rows below, at and above.  FP32 holds
// the x tables of its columns in registers (off2d's form); FP64 takes off2d.
template <typename T> struct MarchX {
  cx<T> am0, ap0, am1, ap1;
};
template <typename T>
__device__ __forceinline__ MarchX<T> march_x(const OpView<T>& op, int c0, bool v0, bool v1) {
  const cx<T> zero = mkc<T>(T(0), T(0));
  MarchX<T> m{zero, zero, zero, zero};
  if constexpr (sizeof(T) == 4) {
    if (v0) m.am0 = op.am[0][c0], m.ap0 = op.ap[0][c0];
    if (v1) m.am1 = op.am[0][c0 + 1], m.ap1 = op.ap[0][c0 + 1];
  }
  return m;
}
template <typename T>
__device__ __forceinline__ Pair<T> march_off(const OpView<T>& op, const MarchX<T>& m, int c0, bool v0, bool v1, int j,
                                             const Pair<T>& s, const Pair<T>& c, const Pair<T>& n) {
  const cx<T> w = march_up1<T>(c.b), e = march_down1<T>(c.a);
  if constexpr (sizeof(T) == 4) {
    const cx<T> am = op.am[1][j], ap = op.ap[1][j];
    const cx<T> xa = cfma<T>(m.am0, w, cmul1<T>(m.ap0, c.b)), xb = cfma<T>(m.am1, c.a, cmul1<T>(m.ap1, e));
    const cx<T> ya = cfma<T>(am, s.a, cmul1<T>(ap, n.a)), yb = cfma<T>(am, s.b, cmul1<T>(ap, n.b));
    return Pair<T>{cadd<T>(xa, ya), cadd<T>(xb, yb)};
  } else {
    Pair<T> r{mkc<T>(T(0), T(0)), mkc<T>(T(0), T(0))};
    if (v0) r.a = off2d<T>(op, c0, j, w, c.b, s.a, n.a);
    if (v1) r.b = off2d<T>(op, c0 + 1, j, c.a, e, s.b, n.b);
    return r;
  }
}

// ---- down: zero-guess sweep, residual, full weighting ------------------------------------------
template <typename T, typename TI, int CR, bool KEEP>
__device__ __forceinline__ void march_down(int bx, int by, const OpView<T>& op, int nc0, int nc1,
                                           const cx<TI>* __restrict__ f, cx<T>* __restrict__ u_out, cx<T>* __restrict__ fc,
                                           T omega, bool vec) {
  const int lane = threadIdx.x & 31, strip = bx * 4 + (threadIdx.x >> 5);
  const int n0 = op.n[0], n1 = op.n[1];
  const int I = strip * MARCH_COLS + lane - 1, c0 = 2 * I;
  if (2 * strip * MARCH_COLS >= n0) return;  // the whole warp
  const int J0 = by * CR, J1 = min(J0 + CR, nc1);
  const bool v0 = c0 >= 0 && c0 < n0, v1 = c0 >= 0 && c0 + 1 < n0;
  const bool own = lane >= 1 && lane <= MARCH_COLS;
  const cx<T> zero = mkc<T>(T(0), T(0));
  const MarchX<T> mx = march_x<T>(op, c0, v0, v1);
  const T om1 = T(1) - omega;
  const int jb = 2 * J0 - 1, je = 2 * J1 + 1;  // rows of u
  const int own1 = J1 == nc1 ? n1 : 2 * J1;    // rows [2 J0, own1) of u are this block's
  auto get = [&](int j, Pair<T>& fv, Pair<T>& dv) {
    const bool in = j >= 0 && j < n1 && j <= je;
    const long at = (long)n0 * (in ? j : 0);
    fv = march_load<T, TI>(f + at, c0, v0 && in, v1 && in, vec);
    dv = march_load<T, T>(op.dinv + at, c0, v0 && in, v1 && in, vec);
  };
  Pair<T> fq[2], dq[2];  // the next two rows
  get(jb, fq[0], dq[0]);
  get(jb + 1, fq[1], dq[1]);
  Pair<T> us{zero, zero}, uc{zero, zero}, fcur{zero, zero};
  cx<T> rw0 = zero, rw1 = zero;
  auto row = [&](int j, int par) {  // par = (j - jb) & 1, a compile-time constant in the unrolled loop
    const Pair<T> fr = fq[par], dr = dq[par];
    get(j + 2, fq[par], dq[par]);
    const Pair<T> un{cmul1<T>(fr.a, dr.a), cmul1<T>(fr.b, dr.b)};
    if (KEEP && own && j >= 2 * J0 && j < own1) march_store<T, T>(u_out + (long)n0 * j, c0, v0, v1, vec, un.a, un.b);
    const int q = j - 1;  // the residual's row
    if (q >= 2 * J0) {
      Pair<T> r{zero, zero};
      if (q < n1) {  // (uniform over the warp)
        const Pair<T> o = march_off<T>(op, mx, c0, v0, v1, q, us, uc, un);
        if (v0) r.a = mkc<T>(fma(om1, fcur.a.x, -o.a.x), fma(om1, fcur.a.y, -o.a.y));
        if (v1) r.b = mkc<T>(fma(om1, fcur.b.x, -o.b.x), fma(om1, fcur.b.y, -o.b.y));
      }
      const cx<T> rc = march_down1<T>(r.a);
      const cx<T> rw = mkc<T>(fma(T(2), r.b.x, r.a.x + rc.x), fma(T(2), r.b.y, r.a.y + rc.y));
      if (!par) {  // q even
        if (q > 2 * J0) {
          const cx<T> acc = mkc<T>(fma(T(2), rw1.x, rw0.x + rw.x), fma(T(2), rw1.y, rw0.y + rw.y));
          if (own && I < nc0) fc[I + (long)nc0 * (q / 2 - 1)] = cscale<T>(T(0.0625), acc);
        }
        rw0 = rw;
      } else {
        rw1 = rw;
      }
    }
    us = uc;
    uc = un;
    fcur = fr;
  };
  // rows jb .. je: 2 (J1 - J0) + 3 of them
  row(jb, 0);
  for (int j = jb + 1; j < je; j += 2) {
    row(j, 1);
    row(j + 1, 0);
  }
}

// ---- up: prolongation, correction, post-smoothing sweep -------------------------------------------
template <typename T, typename TO, typename TI, int CR, bool KEEP>
__device__ __forceinline__ void march_up(int bx, int by, const OpView<T>& op, int nc0, int nc1,
                                         const cx<T>* __restrict__ u_in, const cx<T>* __restrict__ ec,
                                         const cx<TI>* __restrict__ f, cx<TO>* __restrict__ u_out, T omega, bool vec) {
  const int lane = threadIdx.x & 31, strip = bx * 4 + (threadIdx.x >> 5);
  const int n0 = op.n[0], n1 = op.n[1];
  const int I = strip * MARCH_COLS + lane - 1, c0 = 2 * I;
  if (2 * strip * MARCH_COLS >= n0) return;  // the whole warp
  const int j0 = by * 2 * CR, j1 = min(j0 + 2 * CR, n1);
  const bool v0 = c0 >= 0 && c0 < n0, v1 = c0 >= 0 && c0 + 1 < n0, ve = I >= 0 && I < nc0;
  const bool own = lane >= 1 && lane <= MARCH_COLS;
  const cx<T> zero = mkc<T>(T(0), T(0));
  const MarchX<T> mx = march_x<T>(op, c0, v0, v1);
  const T om1 = T(1) - omega;
  auto get = [&](int j, Pair<T>& fv, Pair<T>& dv, Pair<T>& uv) {
    const bool in = j >= 0 && j < n1 && j <= j1;
    const long at = (long)n0 * (in ? j : 0);
    fv = march_load<T, TI>(f + at, c0, v0 && in, v1 && in, vec);
    dv = march_load<T, T>(op.dinv + at, c0, v0 && in, v1 && in, vec);
    if (KEEP) uv = march_load<T, T>(u_in + at, c0, v0 && in, v1 && in, vec);
  };
  auto coarse = [&](int J) -> cx<T> { return ve && J >= 0 && J < nc1 ? ec[I + (long)nc0 * J] : zero; };
  Pair<T> fq[2], dq[2], uq[2];
  get(j0 - 1, fq[0], dq[0], uq[0]);
  get(j0, fq[1], dq[1], uq[1]);
  // x-sums of a coarse row for the lane's even and odd column
  auto sums = [&](cx<T> e) -> Pair<T> {
    const cx<T> el = march_up1<T>(e);
    return Pair<T>{cadd<T>(el, e), sizeof(T) == 4 ? cadd<T>(e, e) : e};
  };
  Pair<T> sc = sums(coarse(j0 / 2 - 1));
  cx<T> en = coarse(j0 / 2);
  Pair<T> vs{zero, zero}, vc{zero, zero}, fcur{zero, zero}, dcur{zero, zero};
  auto row = [&](int j, int par) {  // par = 0: j odd; 1: j even
    const Pair<T> fr = fq[par], dr = dq[par];
    Pair<T> ur{zero, zero};
    if (KEEP) ur = uq[par];
    else ur = Pair<T>{cmul1<T>(fr.a, dr.a), cmul1<T>(fr.b, dr.b)};
    get(j + 2, fq[par], dq[par], uq[par]);
    Pair<T> acc;
    T wa, wb;
    if (par) {  // between the coarse rows j / 2 - 1 and j / 2
      const Pair<T> sn = sums(en);
      en = coarse(j / 2 + 1);
      acc = Pair<T>{cadd<T>(sc.a, sn.a), cadd<T>(sc.b, sn.b)};
      sc = sn;
      wa = T(0.25);
      wb = sizeof(T) == 4 ? T(0.25) : T(0.5);
    } else if (sizeof(T) == 4) {
      acc = Pair<T>{cadd<T>(sc.a, sc.a), cadd<T>(sc.b, sc.b)};
      wa = wb = T(0.25);
    } else {
      acc = sc;
      wa = T(0.5);
      wb = T(1);
    }
    Pair<T> vn{zero, zero};
    if (j >= 0 && j < n1) {
      if (v0) vn.a = mkc<T>(fma(wa, acc.a.x, ur.a.x), fma(wa, acc.a.y, ur.a.y));
      if (v1) vn.b = mkc<T>(fma(wb, acc.b.x, ur.b.x), fma(wb, acc.b.y, ur.b.y));
    }
    const int q = j - 1;
    if (q >= j0) {
      const Pair<T> o = march_off<T>(op, mx, c0, v0, v1, q, vs, vc, vn);
      const cx<T> ga = cmul1<T>(csub<T>(fcur.a, o.a), dcur.a), gb = cmul1<T>(csub<T>(fcur.b, o.b), dcur.b);
      if (own)
        march_store<T, TO>(u_out + (long)n0 * q, c0, v0, v1, vec, mkc<T>(fma(om1, vc.a.x, ga.x), fma(om1, vc.a.y, ga.y)),
                           mkc<T>(fma(om1, vc.b.x, gb.x), fma(om1, vc.b.y, gb.y)));
    }
    vs = vc;
    vc = vn;
    fcur = fr;
    dcur = dr;
  };
  // rows j0 - 1 .. j1
  row(j0 - 1, 0);
  int j = j0;
  for (; j + 1 <= j1; j += 2) {
    row(j, 1);
    row(j + 1, 0);
  }
  if (j == j1) row(j, 1);
}

}  // namespace helm
