// mg_cluster.cu -- the coarse part of a 2D V(1,1) cycle in ONE launch of one thread-block cluster.
//
// Launched level by level, a small level costs its launches, not its work.  Here one cluster of 16
// blocks (8 where the device does not grant 16) walks the levels from the tail's first one down to
// the operator level and back.  Every level's rows are split over the blocks, each block's share stays
// in its shared memory for the whole descent and ascent, the rows it needs of its neighbours are read
// from theirs (distributed shared memory), and a cluster barrier stands where a launch boundary stood.
// A cluster (not one block) because one SM has 2 FP64 lanes and too little shared memory for a 160^2
// level, and not the whole grid because a software grid barrier costs 2 us, a cluster's 0.5 us.
//
// The operator level: below some level the rest of the cycle, a fixed linear map of that level's
// right-hand side, is applied as what it is, one dense matrix (built at create from the levels'
// operators in FP64 arithmetic, one block per column), split by rows over the blocks.  That replaces a
// chain of some twenty dependent phases of a few hundred points by one.  The level is the finest one with
// at most 600 unknowns in FP32 (166 KB of a block's shared memory; reading it there takes 1300 cycles,
// a level's descent and ascent 5000) and 150 in FP64 (n^2 / 8 cycles of a block's FP64 pipe), or a larger
// coarsest level itself.
//
// Measured (whole V-cycles, us, a launch per level / with this kernel, paired when it was made): 96^2 FP32
// red-black 33.5 / 17.1, 640^2 FP32 Jacobi 50.0 / 33.8, FP64 125 / 116, MP2's Galerkin levels in FP64 119 / 101.
// Now, from graphs of cycles: 12.3 and 31.9 in FP32; paired runs: 116 and 94 in FP64.
//
// What bounds the kernel is the chain of phases: two cluster barriers and five block barriers a level,
// and between them one or two points a thread, whose instructions count.
//
// Split of level k's points: its right-hand side f_k is made by the restriction, so block r holds
// the rows [a_k(r), a_k(r+1)), a_k(r) = n1 r / NC.  Smoothing, residual and correction of level k
// run on the fine rows of the coarse rows it makes, [2 a_{k+1}(r), 2 a_{k+1}(r+1)) (the last block
// also takes the fine row past the last coarse one), with a halo recomputed on both sides, so that
// a descent needs nothing but f's halo and an ascent nothing but the coarse correction's.
#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "mg_cluster.cuh"
#include "stencil.cuh"

namespace helm {

namespace {

constexpr int CT = CTAIL_THREADS;

__device__ __forceinline__ unsigned ct_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the address of this block's shared-memory location in block `rank` of the cluster
__device__ __forceinline__ unsigned ct_map(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float2 ct_ld(unsigned addr, float2) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ double2 ct_ld(unsigned addr, double2) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void ct_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void ct_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void ct_sync() {
  ct_arrive();
  ct_wait();
}

// e = y w + x by the magic number ceil(2^32 / w) (exact for e w < 2^32; w = 1 has none)
__device__ __forceinline__ void ct_div(int e, int w, unsigned magic, int& x, int& y) {
  y = w == 1 ? e : (int)__umulhi((unsigned)e, magic);
  x = e - y * w;
}

// rows [first, end) of an n-row level held by block r of 2^sh, and the block holding row j (m: the
// magic number of n)
__device__ __forceinline__ int ct_first(int n, int r, int sh) { return (n * r) >> sh; }
__device__ __forceinline__ int ct_owner(int j, int n, unsigned m, int sh) {
  int x, o;
  ct_div(((j + 1) << sh) - 1, n, m, x, o);
  return o;
}

// This block's share of level k: coarse rows [A, B), staged fine rows [lo, lo + rows), corrected and
// written fine rows [2A, pe).
struct Share {
  int n0, n1, m0, m1, A, B, lo, rows, pe;
};
template <typename T, bool RB>
__device__ __forceinline__ Share ct_share(const CTailArgs<T>& a, int k, int r) {
  Share s;
  s.n0 = a.n0[k];
  s.n1 = a.n1[k];
  s.m0 = a.n0[k + 1];
  s.m1 = a.n1[k + 1];
  s.A = ct_first(s.m1, r, a.sh);
  s.B = ct_first(s.m1, r + 1, a.sh);
  s.lo = 2 * s.A - (RB ? 3 : 1);
  s.rows = s.A < s.B ? 2 * (s.B - s.A) + (RB ? 6 : 3) : 0;
  s.pe = s.B == s.m1 ? s.n1 : 2 * s.B;
  return s;
}

template <typename T>
__device__ __forceinline__ cx<T> ct_off(const OpView<T>& op, const cx<T>* u, int w, int i, int j) {
  if (op.stg) return off9_staged<T>(op, u, w, i + (long)op.n[0] * j);
  return off2d<T>(op, i, j, u[-1], u[1], u[-w], u[w]);
}

__device__ __forceinline__ void ct_copy(float2* dst, const float2* src) {  // asynchronous, 8 bytes
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void ct_copy(double2* dst, const double2* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Pairs of floats in one register pair, two operations an instruction.
__device__ __forceinline__ unsigned long long f2_pack(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long f2_sub(unsigned long long a, unsigned long long b) {
  return f2_fma(b, 0xbf800000bf800000ull, a);  // a - b, rounded once
}
// Two sums, each kept as two floats hi + lo, lo holding what hi's additions round away (the rounding
// error of an addition of two floats is a float: Knuth's two-sum).
struct Sum2 {
  unsigned long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(unsigned long long v) {
    const unsigned long long s = f2_add(hi, v), b = f2_sub(s, hi);
    lo = f2_add(lo, f2_add(f2_sub(hi, f2_sub(s, b)), f2_sub(v, b)));
    hi = s;
  }
  __device__ __forceinline__ void add(const Sum2& v) {
    add(v.hi);
    lo = f2_add(lo, v.lo);
  }
  __device__ __forceinline__ Sum2 from(int o) const {  // lane ^ o's
    Sum2 r;
    r.hi = __shfl_xor_sync(0xffffffffu, hi, o);
    r.lo = __shfl_xor_sync(0xffffffffu, lo, o);
    return r;
  }
};
constexpr int SUM_TERMS = 4;  // complex products of a partial sum
// hi + lo; an overflowed sum stays infinite (its lo is not a number)
__device__ __forceinline__ float sum2_value(float hi, float lo) { return isinf(hi) ? hi : hi + lo; }

// The levels a.first .. coarsest of one instance's cycle, by one cluster.
// TI: the type of f_in (complex128 when the whole FP32 cycle of a complex128 vector runs here).
template <typename T, bool RB, typename TO, typename TI>
__device__ __forceinline__ void ctail_body(const CTailArgs<T>* __restrict__ ga, const cx<TI>* __restrict__ f_in,
                                           cx<TO>* __restrict__ out, const int* skip) {
  extern __shared__ __align__(16) unsigned char ct_smem[];
  // the arguments in shared memory: as kernel parameters, every level's first use of its operator
  // stood for a chain of constant-cache misses (500 to 700 cycles a phase)
  __shared__ CTailArgs<T> a;
  static_assert(sizeof(a) % 16 == 0, "copied in 16-byte pieces");
  for (int q = threadIdx.x; q < (int)(sizeof(a) / 16); q += CT)
    ct_copy(reinterpret_cast<double2*>(&a) + q, reinterpret_cast<const double2*>(ga) + q);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  cx<T>* const base = reinterpret_cast<cx<T>*>(ct_smem);
  const unsigned base32 = (unsigned)__cvta_generic_to_shared(base);
  const int tid = threadIdx.x;
  const int r = (int)ct_rank(), sh = a.sh, last = a.count - 1;
  const cx<T> zero = mkc<T>(T(0), T(0));
  cx<T>* const scr = base + a.scr;
  const T om1 = T(1) - a.omega;
  auto remote = [&](int at, int o) -> cx<T> {  // element `at` of block o
    return ct_ld(ct_map(base32 + (unsigned)(at * sizeof(cx<T>)), o), zero);
  };

  // Constants of the hierarchy, asynchronously and before the wait on the previous kernel: 1/D of the
  // staged rows, the axis tables, this block's rows of the dense operator; zero columns beside the staged
  // rows.
  for (int k = 0; k < last; ++k) {
    const Share s = ct_share<T, RB>(a, k, r);
    const int w = s.n0 + 2;
    cx<T>* const sd = base + a.d[k];
    cx<T>* const su = base + a.u[k];
    const cx<T>* __restrict__ dinv = a.op[k].dinv;
    const int ne = s.rows * s.n0;
    for (int e = tid; e < ne; e += CT) {
      int x, y;
      ct_div(e, s.n0, a.magic[k], x, y);
      const int j = s.lo + y;
      cx<T>* const q = sd + y * w + x + 1;
      if (j >= 0 && j < s.n1) ct_copy(q, dinv + x + s.n0 * j);
      else *q = zero;
    }
    for (int y = tid; y < s.rows; y += CT) su[y * w] = su[y * w + s.n0 + 1] = zero;
    cx<T>* tb = base + a.tab[k];
    for (int q = tid; q < s.n0; q += CT) {
      ct_copy(tb + q, a.op[k].am[0] + q);
      ct_copy(tb + s.n0 + q, a.op[k].ap[0] + q);
    }
    for (int q = tid; q < s.n1; q += CT) {
      ct_copy(tb + 2 * s.n0 + q, a.op[k].am[1] + q);
      ct_copy(tb + 2 * s.n0 + s.n1 + q, a.op[k].ap[1] + q);
    }
  }
  // operator level: this block's rows of the matrix, points [pa, pb)
  const int l0 = a.n0[last], l1 = a.n1[last], nop = l0 * l1;
  const int pa = ct_first(nop, r, sh), pb = ct_first(nop, r + 1, sh);
  cx<T>* const mat = base + a.mat;
  {  // 16 bytes a copy: the pitch makes every row start on 16 bytes
    const int n16 = (int)((pb - pa) * a.pitch * sizeof(cx<T>) / 16);
    double2* const to = reinterpret_cast<double2*>(mat);
    const double2* const from = reinterpret_cast<const double2*>(a.dense + (long)pa * a.pitch);
    for (int e = tid; e < n16; e += CT) ct_copy(to + e, from + e);
  }

  pdl_entry();
  if (skip && *skip) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    return;
  }

  auto level_op = [&](int k) {  // level k's operator, its axis tables in shared memory
    OpView<T> op = a.op[k];
    const cx<T>* tb = base + a.tab[k];
    op.am[0] = tb;
    op.ap[0] = tb + a.n0[k];
    op.am[1] = tb + 2 * a.n0[k];
    op.ap[1] = op.am[1] + a.n1[k];
    return op;
  };

  // ---- descent
  for (int k = 0; k < last; ++k) {
    const Share s = ct_share<T, RB>(a, k, r);
    const OpView<T> op = level_op(k);
    const int w = s.n0 + 2;
    cx<T>* const sf = base + a.f[k];
    cx<T>* const su = base + a.u[k];
    const cx<T>* const sd = base + a.d[k];
    {  // stage f; the zero-guess sweep (its red half): four loads in flight a thread
      const int ne = s.rows * s.n0;
      const unsigned m1 = a.magic1[k];
      for (int e0 = tid; e0 < ne; e0 += 4 * CT) {
        cx<T> v[4];
        int at[4];
        bool red[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int e = e0 + q * CT;
          int x, y;
          v[q] = zero;
          ct_div(e, s.n0, a.magic[k], x, y);
          const int j = s.lo + y;
          at[q] = y * w + x + 1;
          red[q] = !((x + j) & 1);
          if (e < ne && j >= 0 && j < s.n1) {
            if (k == 0) {
              v[q] = cconv<T, TI>(f_in[x + s.n0 * j]);
            } else {
              const int o = ct_owner(j, s.n1, m1, sh);
              v[q] = remote(a.c[k] + (j - ct_first(s.n1, o, sh)) * s.n0 + x, o);
            }
          }
        }
        if (k == 0 && e0 == tid) {  // 1/D is in place once every thread's copies are
          asm volatile("cp.async.wait_all;" ::: "memory");
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (e0 + q * CT >= ne) break;
          sf[at[q]] = v[q];
          su[at[q]] = RB && !red[q] ? zero : cmul1<T>(v[q], sd[at[q]]);
        }
      }
      if (k == 0) asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncthreads();
    if (RB) {  // black points from the red ones, staged rows 1 .. rows - 2
      const int P = (s.n0 + 1) >> 1, ne = s.rows ? (s.rows - 2) * P : 0;
#pragma unroll 2
      for (int e = tid; e < ne; e += CT) {
        int x, y;
        ct_div(e, P, a.magich[k], x, y);
        y += 1;
        const int j = s.lo + y;
        x = 2 * x + ((j + 1) & 1);
        if (x >= s.n0 || j < 0 || j >= s.n1) continue;
        cx<T>* const u = su + y * w + x + 1;
        const cx<T> acc = ct_off<T>(op, u, w, x, j);
        *u = cmul1<T>(csub<T>(sf[y * w + x + 1], acc), sd[y * w + x + 1]);
      }
      __syncthreads();
    }
    // residual on fine rows 2A .. 2B (red points only after red-black sweeps), zero outside the grid
    const int wr = s.n0 + 1, y0 = 2 * s.A - s.lo;
    {
      const int ne = s.rows ? (2 * (s.B - s.A) + 1) * wr : 0;
#pragma unroll 2
      for (int e = tid; e < ne; e += CT) {
        int x, y;
        ct_div(e, wr, a.magicr[k], x, y);
        const int j = 2 * s.A + y;
        cx<T> rv = zero;
        if (x < s.n0 && j < s.n1 && !(RB && ((x + j) & 1))) {
          const int at = (y + y0) * w + x + 1;
          const cx<T> acc = ct_off<T>(op, su + at, w, x, j);
          if (RB) rv = mkc<T>(-acc.x, -acc.y);
          else rv = mkc<T>(fma(om1, sf[at].x, -acc.x), fma(om1, sf[at].y, -acc.y));
        }
        scr[e] = rv;
      }
    }
    __syncthreads();
    {  // full weighting into this block's rows of f_{k+1}
      cx<T>* const fc = base + a.c[k + 1];
      const int ne = (s.B - s.A) * s.m0;
      for (int e = tid; e < ne; e += CT) {
        int x, y;
        ct_div(e, s.m0, a.magic[k + 1], x, y);
        cx<T> rw[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const cx<T>* q = scr + (2 * y + d) * wr + 2 * x;
          rw[d] = mkc<T>(fma(T(2), q[1].x, q[0].x + q[2].x), fma(T(2), q[1].y, q[0].y + q[2].y));
        }
        const cx<T> acc = mkc<T>(fma(T(2), rw[1].x, rw[0].x + rw[2].x), fma(T(2), rw[1].y, rw[0].y + rw[2].y));
        fc[e] = cscale<T>(T(0.0625), acc);
      }
    }
    ct_sync();
  }

  // ---- operator level: its f gathered, then one warp per row of the matrix
  cx<T>* const fl = scr;  // the residual's readers are behind a cluster barrier
  if (last == 0) asm volatile("cp.async.wait_all;" ::: "memory");
  for (int e = tid; e < nop; e += CT) {
    if (last == 0) {
      fl[e] = cconv<T, TI>(f_in[e]);
    } else {
      int x, y;
      ct_div(e, l0, a.magic[last], x, y);
      const int o = ct_owner(y, l1, a.magic1[last], sh);
      fl[e] = remote(a.c[last] + (y - ct_first(l1, o, sh)) * l0 + x, o);
    }
  }
  __syncthreads();
  {
    const int lane = tid & 31;
    cx<T>* const el = base + a.e;
    // a warp takes three rows at a time, so that f is read from shared memory once for them (the
    // phase is bound by that memory's 128 bytes a cycle)
    constexpr int NW = CT / 32;
    for (int q0 = tid >> 5; q0 < pb - pa; q0 += 3 * NW) {
      const bool two = q0 + NW < pb - pa, three = q0 + 2 * NW < pb - pa;
      const cx<T>* row = mat + q0 * a.pitch;
      const cx<T>* row2 = two ? row + NW * a.pitch : row;
      const cx<T>* row3 = three ? row + 2 * NW * a.pitch : row;
      if constexpr (sizeof(T) == 4) {
        // FP32: partial sums of SUM_TERMS products, added up in sums of two floats.  One chain over the 18 products
        // that a lane has made 4 times the rounding of the matrix and f (1.2e-7 of the result against 0.33e-7).  Over
        // 50 cycles of 63^2 to 420^2 unknowns the error against 64 bits falls by 5 % and in none rises by more than
        // 2 %, for 0.3 to 0.5 us (96^2 red-black 11.8 -> 12.3 us); one product at a time: 8 % for 1.6 us.
        Sum2 s[3];
        for (int c0 = lane; c0 < nop; c0 += 32 * SUM_TERMS) {
          cx<T> p[3] = {zero, zero, zero};
#pragma unroll
          for (int k = 0; k < SUM_TERMS; ++k) {
            const int c = c0 + 32 * k;
            if (k && c >= nop) break;
            const cx<T> f = fl[c];
            p[0] = cfma<T>(row[c], f, p[0]);
            if (two) p[1] = cfma<T>(row2[c], f, p[1]);
            if (three) p[2] = cfma<T>(row3[c], f, p[2]);
          }
          s[0].add(f2_pack(p[0].x, p[0].y));
          if (two) s[1].add(f2_pack(p[1].x, p[1].y));
          if (three) s[2].add(f2_pack(p[2].x, p[2].y));
        }
        // over the lanes, half of them summing rows 0 and 1, half row 2 (its partners a zero)
        const bool b4 = lane & 16, b3 = lane & 8;
        Sum2 h = b4 ? s[2] : s[0], g = b4 ? Sum2() : s[1];
        {
          const Sum2 g0 = b4 ? s[0] : s[2], g1 = b4 ? s[1] : Sum2();
          h.add(g0.from(16));
          g.add(g1.from(16));
        }
        const Sum2 give = b3 ? h : g;
        Sum2 r = b3 ? g : h;
        r.add(give.from(8));
        r.add(r.from(4));
        r.add(r.from(2));
        r.add(r.from(1));
        const int q = q0 + (b4 ? 2 : b3 ? 1 : 0) * NW;
        if (!(lane & 7) && !(b4 && b3) && q < pb - pa) {
          const float2 hi = f2_unpack(r.hi), lo = f2_unpack(r.lo);
          const cx<T> v = mkc<T>(sum2_value(hi.x, lo.x), sum2_value(hi.y, lo.y));
          if (last == 0) out[pa + q] = cconv<TO, T>(v);
          else el[q] = v;
        }
      } else {
        cx<T> acc[3] = {zero, zero, zero};
#pragma unroll 4
        for (int c = lane; c < nop; c += 32) {
          const cx<T> f = fl[c];
          acc[0] = cfma<T>(row[c], f, acc[0]);
          if (two) acc[1] = cfma<T>(row2[c], f, acc[1]);
          if (three) acc[2] = cfma<T>(row3[c], f, acc[2]);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const int q = q0 + m * NW;
          if (q >= pb - pa) break;
          for (int o = 16; o > 0; o >>= 1) {
            acc[m].x += __shfl_down_sync(0xffffffffu, acc[m].x, o);
            acc[m].y += __shfl_down_sync(0xffffffffu, acc[m].y, o);
          }
          if (lane == 0) {
            if (last == 0) out[pa + q] = cconv<TO, T>(acc[m]);
            else el[q] = acc[m];
          }
        }
      }
    }
  }
  if (last == 0) return;
  ct_sync();

  // ---- ascent
  for (int k = last - 1; k >= 0; --k) {
    const Share s = ct_share<T, RB>(a, k, r);
    const OpView<T> op = level_op(k);
    const int w = s.n0 + 2, HU = RB ? 2 : 1;
    cx<T>* const sf = base + a.f[k];
    cx<T>* const su = base + a.u[k];
    const cx<T>* const sd = base + a.d[k];
    // the coarse correction on coarse rows A - 2 .. B + 1 (pitch we, zero outside the grid); level
    // k + 1 wrote its result over its staged f
    const int we = s.m0 + 2, c0 = s.A - 2;
    {
      const int ne = s.rows ? (s.B - s.A + 4) * we : 0;
      const bool low = k + 1 == last;
      const int mm = low ? nop : a.n1[k + 2];
      const unsigned mg = low ? a.magicn : a.magic1[k + 2];
#pragma unroll 2
      for (int e = tid; e < ne; e += CT) {
        int x, y;
        ct_div(e, we, a.magice[k + 1], x, y);
        const int J = c0 + y;
        x -= 1;
        cx<T> v = zero;
        if (x >= 0 && x < s.m0 && J >= 0 && J < s.m1) {
          const int g = low ? J * s.m0 + x : min(J >> 1, mm - 1);  // a point, or a coarse row
          const int o = ct_owner(g, mm, mg, sh), b0 = ct_first(mm, o, sh);
          v = remote(low ? a.e + g - b0 : a.f[k + 1] + (J - (2 * b0 - (RB ? 3 : 1))) * we + x + 1, o);
        }
        scr[e] = v;
      }
    }
    if (k == 0) pdl_trigger();  // the next kernel's blocks may come up while this one finishes
    if (k == 0) ct_arrive();  // the last read of another block's shared memory
    __syncthreads();
    {  // corrected iterate on rows 2A - HU .. pe - 1 + HU, in place (red-black: its black points, all that
       // the red half-sweep reads)
      const int jb = 2 * s.A - HU, wi = RB ? (s.n0 + 1) >> 1 : s.n0, ne = s.rows ? (s.pe + HU - jb) * wi : 0;
#pragma unroll 2
      for (int e = tid; e < ne; e += CT) {
        int i, y;
        ct_div(e, wi, RB ? a.magich[k] : a.magic[k], i, y);
        const int j = jb + y;
        if (RB) i = 2 * i + ((j + 1) & 1);
        if (i >= s.n0 || j < 0 || j >= s.n1) continue;
        const int ia = (i - 1) >> 1, ja = (j - 1) >> 1;  // odd: the coarse node; even: the one before
        const cx<T>* ra = scr + (ja - c0) * we + 1 + ia;
        cx<T> acc;
        T wt;
        if constexpr (std::is_same<T, float>::value) {  // all four terms, without branches
          const int dx = 1 - (i & 1), dy = (1 - (j & 1)) * we;
          acc = cadd<T>(cadd<T>(ra[0], ra[dx]), cadd<T>(ra[dy], ra[dy + dx]));
          wt = T(0.25);
        } else {
          acc = ra[0];
          if (!(i & 1)) acc = cadd<T>(acc, ra[1]);
          if (!(j & 1)) {
            acc = cadd<T>(acc, ra[we]);
            if (!(i & 1)) acc = cadd<T>(acc, ra[we + 1]);
          }
          wt = ((i & 1) ? T(1) : T(0.5)) * ((j & 1) ? T(1) : T(0.5));
        }
        cx<T>* const u = su + (j - s.lo) * w + i + 1;
        const cx<T> uo = *u;
        *u = mkc<T>(fma(wt, acc.x, uo.x), fma(wt, acc.y, uo.y));
      }
    }
    __syncthreads();
    if (!RB) {
      const int ne = s.rows ? (s.pe - 2 * s.A) * s.n0 : 0;
#pragma unroll 2
      for (int e = tid; e < ne; e += CT) {
        int i, y;
        ct_div(e, s.n0, a.magic[k], i, y);
        const int j = 2 * s.A + y, at = (j - s.lo) * w + i + 1;
        const cx<T> acc = ct_off<T>(op, su + at, w, i, j);
        const cx<T> g = cmul1<T>(csub<T>(sf[at], acc), sd[at]);
        const cx<T> uc = su[at];
        const cx<T> v = mkc<T>(fma(om1, uc.x, g.x), fma(om1, uc.y, g.y));
        if (k == 0) out[i + s.n0 * j] = cconv<TO, T>(v);
        else sf[at] = v;
      }
    } else {
      // red points of the tile and one ring of rows around it, in place (they read black points
      // only), then the black ones; the red results go out with them
      const int P = (s.n0 + 1) >> 1;
      {
        const int jr = 2 * s.A - 1, ne = s.rows ? (s.pe + 1 - jr) * P : 0;
#pragma unroll 2
        for (int e = tid; e < ne; e += CT) {
          int x, y;
          ct_div(e, P, a.magich[k], x, y);
          const int j = jr + y;
          x = 2 * x + (j & 1);
          if (x >= s.n0 || j < 0 || j >= s.n1) continue;
          const int at = (j - s.lo) * w + x + 1;
          const cx<T> acc = ct_off<T>(op, su + at, w, x, j);
          su[at] = cmul1<T>(csub<T>(sf[at], acc), sd[at]);
        }
      }
      __syncthreads();
      const int nq = s.rows ? (s.pe - 2 * s.A) * P : 0;
      for (int e = tid; e < nq; e += CT) {  // a black point and the red one beside it
        int x, y;
        ct_div(e, P, a.magich[k], x, y);
        const int j = 2 * s.A + y, row = (j - s.lo) * w + 1;
        const int xb = 2 * x + ((j + 1) & 1), xr = 2 * x + (j & 1);
        if (xr < s.n0) {
          const cx<T> v = su[row + xr];
          if (k == 0) out[xr + s.n0 * j] = cconv<TO, T>(v);
          else sf[row + xr] = v;
        }
        if (xb < s.n0) {
          const cx<T> acc = ct_off<T>(op, su + row + xb, w, xb, j);
          const cx<T> v = cmul1<T>(csub<T>(sf[row + xb], acc), sd[row + xb]);
          if (k == 0) out[xb + s.n0 * j] = cconv<TO, T>(v);
          else sf[row + xb] = v;
        }
      }
    }
    if (k == 0) ct_wait();
    else ct_sync();
  }
}

template <typename T, bool RB, typename TO, typename TI>
__global__ void __launch_bounds__(CT, 1) k_ctail(const CTailArgs<T>* __restrict__ a, const cx<TI>* __restrict__ f_in,
                                                 cx<TO>* __restrict__ out, const int* skip) {
  ctail_body<T, RB, TO, TI>(a, f_in, out, skip);
}

// The tails of a group's instances in one launch: virtual block w of the work list is cluster w.
template <typename T, bool RB, typename TO>
__global__ void __launch_bounds__(CT, 1) kg_ctail(const GCTail<T>* __restrict__ A, const GroupList* __restrict__ LT,
                                                  int li) {
  pdl_entry();
  const GroupList& L = LT[li];
  unsigned nc;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nc));
  const int w = (int)(blockIdx.x / nc);
  if (w >= L.first[L.nd]) return;  // the whole cluster
  const GCTail<T>& g = A[L.map[w]];
  ctail_body<T, RB, TO, T>(g.a, g.f, (cx<TO>*)g.out, g.skip);
}

template <typename K>
cudaError_t ct_prepare(K kern) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CTAIL_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}
template <typename T>
cudaError_t ct_prepare_all() {
  cudaError_t e = cudaSuccess;
  auto one = [&](auto kern) {
    if (e == cudaSuccess) e = ct_prepare(kern);
  };
  one(k_ctail<T, false, T, T>);
  one(k_ctail<T, true, T, T>);
  one(kg_ctail<T, false, T>);
  one(kg_ctail<T, true, T>);
  if (!std::is_same<T, double>::value) {
    one(k_ctail<T, false, double, T>);
    one(k_ctail<T, true, double, T>);
    one(k_ctail<T, false, T, double>);
    one(k_ctail<T, true, T, double>);
    one(k_ctail<T, false, double, double>);
    one(k_ctail<T, true, double, double>);
    one(kg_ctail<T, false, double>);
    one(kg_ctail<T, true, double>);
  }
  return e;
}

// Blocks per cluster on the current device, with the kernels' attributes set (outside any capture:
// the hierarchy's setup asks first): 16 where a cluster of 16 such blocks fits, else the portable 8.
int ct_granted() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  static std::mutex mu;
  static int known[64];
  std::lock_guard<std::mutex> lk(mu);
  if (known[dev]) return known[dev] > 0 ? known[dev] : 0;
  known[dev] = -1;
  if (ct_prepare_all<float>() != cudaSuccess || ct_prepare_all<double>() != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  for (int nc : {16, 8}) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3(CT);
    cfg.dynamicSmemBytes = CTAIL_SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int fit32 = 0, fit64 = 0;
    if (cudaOccupancyMaxActiveClusters(&fit32, k_ctail<float, true, double, double>, &cfg) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&fit64, k_ctail<double, true, double, double>, &cfg) == cudaSuccess && fit32 > 0 &&
        fit64 > 0) {
      known[dev] = nc;
      return nc;
    }
    cudaGetLastError();
  }
  return 0;
}

// the same under the thread's test limit
int ct_blocks() {
  const int nc = ct_granted();
  return nc <= g_limits.cluster ? nc : g_limits.cluster >= 8 ? 8 : 0;
}

template <typename... KArgs, typename... Args>
void launch_cluster(void (*kernel)(KArgs...), int grid, int nc, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(CT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = g_use_pdl ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

unsigned ct_magic(int w) { return w > 1 ? (unsigned)(((1ull << 32) + w - 1) / w) : 0u; }

// row pitch of the dense operator: rows of a multiple of 16 bytes
template <typename T> int ct_pitch(int n) { return std::is_same<T, double>::value ? n : (n + 1) & ~1; }

// Arguments and dynamic shared memory of the levels first.. operator level of c; 0 bytes when they
// do not fit.
template <typename T>
size_t ct_args(const helm_ctx* c, int first, int nc, CTailArgs<T>& a) {
  a = CTailArgs<T>{};
  a.count = c->ctail_op - first + 1;
  for (a.sh = 0; (1 << a.sh) < nc; ++a.sh) {}
  if (a.count < 1 || a.count > CTAIL_MAX_LEVELS) return 0;
  const bool rb = c->pc.smoother == HELM_SM_RBGS;
  const LevelHost& O = c->lv[c->ctail_op];
  long off = 0, scr = O.ntot;
  for (int k = 0; k < a.count; ++k) {
    const LevelHost& L = c->lv[first + k];
    if (L.ntot > (1 << 17)) return 0;
    a.op[k] = L.view<T>();
    a.n0[k] = L.n[0];
    a.n1[k] = L.n[1];
    a.magic[k] = ct_magic(L.n[0]);
    a.magich[k] = ct_magic((L.n[0] + 1) / 2);
    a.magicr[k] = ct_magic(L.n[0] + 1);
    a.magice[k] = ct_magic(L.n[0] + 2);
    a.magic1[k] = ct_magic(L.n[1]);
    if (k > 0) {  // the f rows the restriction of level k - 1 makes here
      a.c[k] = (int)off;
      off += (long)((L.n[1] + nc - 1) / nc) * L.n[0];
    }
    if (k == a.count - 1) break;
    const LevelHost& C = c->lv[first + k + 1];
    const long mc = (C.n[1] + nc - 1) / nc;
    const long rows = 2 * mc + (rb ? 6 : 3), staged = rows * (L.n[0] + 2);
    a.f[k] = (int)off;
    a.u[k] = (int)(off + staged);
    a.d[k] = (int)(off + 2 * staged);
    off += 3 * staged;
    a.tab[k] = (int)off;
    off += 2 * (L.n[0] + L.n[1]);
    scr = std::max(scr, (2 * mc + 1) * (L.n[0] + 1));
    scr = std::max(scr, (mc + 4) * (C.n[0] + 2));
  }
  const long prow = (O.ntot + nc - 1) / nc;
  a.magicn = ct_magic((int)O.ntot);
  a.e = (int)off;
  off += prow;
  off = (off + 1) & ~1L;
  a.pitch = ct_pitch<T>((int)O.ntot);
  a.mat = (int)off;
  off += prow * a.pitch;
  a.scr = (int)off;
  off += scr;
  a.dense = (const cx<T>*)c->ctail_dense;
  a.omega = (T)c->pc.omega;
  const size_t bytes = sizeof(cx<T>) * (size_t)off;
  return bytes <= CTAIL_SMEM ? bytes : 0;
}

// ---- the dense operator ----------------------------------------------------------------------
// Column q of the rest of the cycle below (and with) level 0 of `a`: the cycle of the unit vector q,
// in FP64 and in one block, by the definitions (a level's vectors u, f, r in shared memory).
// Also in FP32 from the FP64 tables: made of the rounded ones, its error partly cancels that of the
// rounded levels above it or adds to it (96^2 red-black 2.10 -> 1.62e-7, but 97 x 95 red-black 1.47 -> 1.88e-7; 2 % more
// over 50 problems).
constexpr int COL_MAX_LEVELS = 8;
constexpr int COL_THREADS = 128;
struct ColArgs {
  int count;
  OpView<double> op[COL_MAX_LEVELS];
  int at[COL_MAX_LEVELS];  // place of the level's vectors
  double omega;
};

__device__ __forceinline__ double2 col_diag(const OpView<double>& op, int i, int j) {
  const long p = i + (long)op.n[0] * j;
  if (op.stg) return op.stg[4 * op.ntot + p];
  const double ph = op.phi ? op.phi[p] : op.phi0;
  const double2 d = cadd<double>(cadd<double>(op.a0[0][i], op.a0[1][j]), somm_diag(op, i, j, 0, ph));
  return csub<double>(d, sigma64(op, p, ph));
}
__device__ double2 col_off(const OpView<double>& op, const double2* u, int i, int j) {
  const int n0 = op.n[0], n1 = op.n[1];
  const long p = i + (long)n0 * j;
  double2 acc = make_double2(0.0, 0.0);
  for (int dj = -1; dj <= 1; ++dj)
    for (int di = -1; di <= 1; ++di) {
      if ((di == 0 && dj == 0) || i + di < 0 || i + di >= n0 || j + dj < 0 || j + dj >= n1) continue;
      if (!op.stg && di != 0 && dj != 0) continue;
      const double2 wt = op.stg ? op.stg[(long)(3 * (dj + 1) + di + 1) * op.ntot + p]
                                : (dj == 0 ? (di < 0 ? op.am[0][i] : op.ap[0][i]) : (dj < 0 ? op.am[1][j] : op.ap[1][j]));
      acc = cfma<double>(wt, u[p + di + (long)dj * n0], acc);
    }
  return acc;
}

template <bool RB>
__global__ void __launch_bounds__(COL_THREADS) k_ctail_columns(const __grid_constant__ ColArgs a,
                                                               const double2* __restrict__ inv, int nco,
                                                               double2* __restrict__ o64, float2* __restrict__ o32, int pitch) {
  extern __shared__ __align__(16) unsigned char ct_smem[];
  double2* const base = reinterpret_cast<double2*>(ct_smem);
  const int tid = threadIdx.x, last = a.count - 1;
  const double2 zero = make_double2(0.0, 0.0);
  auto vec = [&](int k, int which) { return base + a.at[k] + which * (int)a.op[k].ntot; };
  for (int p = tid; p < a.op[0].ntot; p += COL_THREADS) vec(0, 1)[p] = make_double2(p == (int)blockIdx.x ? 1.0 : 0.0, 0.0);
  __syncthreads();
  auto points = [&](int k, auto&& fn) {
    const int n0 = a.op[k].n[0], n = (int)a.op[k].ntot;
    for (int p = tid; p < n; p += COL_THREADS) fn(p, p % n0, p / n0);
    __syncthreads();
  };
  for (int k = 0; k < last; ++k) {
    const OpView<double>& op = a.op[k];
    double2 *u = vec(k, 0), *f = vec(k, 1), *r = vec(k, 2);
    points(k, [&](int p, int i, int j) {
      u[p] = RB && ((i + j) & 1) ? zero : cscale<double>(RB ? 1.0 : a.omega, cdiv<double>(f[p], col_diag(op, i, j)));
    });
    if (RB)
      points(k, [&](int p, int i, int j) {
        if ((i + j) & 1) u[p] = cdiv<double>(csub<double>(f[p], col_off(op, u, i, j)), col_diag(op, i, j));
      });
    points(k, [&](int p, int i, int j) {
      r[p] = csub<double>(f[p], cfma<double>(col_diag(op, i, j), u[p], col_off(op, u, i, j)));
    });
    double2* fc = vec(k + 1, 1);
    points(k + 1, [&](int p, int I, int J) {
      double2 acc = zero;
      for (int b = 0; b < 3; ++b)
        for (int c = 0; c < 3; ++c) {
          const int i = 2 * I + c, j = 2 * J + b;
          if (i >= op.n[0] || j >= op.n[1]) continue;
          acc = cadd<double>(acc, cscale<double>((b == 1 ? 0.5 : 0.25) * (c == 1 ? 0.5 : 0.25), r[i + op.n[0] * j]));
        }
      fc[p] = acc;
    });
  }
  {
    const double2* f = vec(last, 1);
    double2* u = vec(last, 0);
    points(last, [&](int p, int, int) {
      double2 acc = zero;
      for (int c = 0; c < nco; ++c) acc = cfma<double>(inv[(long)p * nco + c], f[c], acc);
      u[p] = acc;
    });
  }
  for (int k = last - 1; k >= 0; --k) {
    const OpView<double>&op = a.op[k], &oc = a.op[k + 1];
    double2 *u = vec(k, 0), *f = vec(k, 1), *r = vec(k, 2);
    const double2* e = vec(k + 1, 0);
    points(k, [&](int p, int i, int j) {
      double2 acc = zero;
      for (int b = 0; b < ((j & 1) ? 1 : 2); ++b)
        for (int c = 0; c < ((i & 1) ? 1 : 2); ++c) {
          const int I = (i - 1) / 2 * (i > 0) - (i == 0) + c, J = (j - 1) / 2 * (j > 0) - (j == 0) + b;
          if (I < 0 || I >= oc.n[0] || J < 0 || J >= oc.n[1]) continue;
          acc = cadd<double>(acc, cscale<double>(((i & 1) ? 1.0 : 0.5) * ((j & 1) ? 1.0 : 0.5), e[I + oc.n[0] * J]));
        }
      r[p] = cadd<double>(u[p], acc);
    });
    if (!RB) {
      points(k, [&](int p, int i, int j) {
        const double2 g = cscale<double>(a.omega, cdiv<double>(csub<double>(f[p], col_off(op, r, i, j)), col_diag(op, i, j)));
        u[p] = cadd<double>(cscale<double>(1.0 - a.omega, r[p]), g);
      });
    } else {
      for (int colour = 0; colour < 2; ++colour)
        points(k, [&](int p, int i, int j) {
          if (((i + j) & 1) == colour) r[p] = cdiv<double>(csub<double>(f[p], col_off(op, r, i, j)), col_diag(op, i, j));
        });
      points(k, [&](int p, int, int) { u[p] = r[p]; });
    }
  }
  const double2* u = vec(0, 0);
  for (int p = tid; p < a.op[0].ntot; p += COL_THREADS) {
    const long at = p * (long)pitch + blockIdx.x;
    if (o64) o64[at] = u[p];
    else o32[at] = cconv<float, double>(u[p]);
  }
}

}  // namespace

// The cluster kernel takes 2D V(1,1) hierarchies with point smoothing, coarsening offset 1 and a
// dense coarsest inverse, 5-point or (Galerkin) 9-point levels.
bool ctail_applies(const helm_ctx* c) {
  return c->grid.dim == 2 && c->pc.nu1 == 1 && c->pc.nu2 == 1 && !(c->pc.flags & HELM_PF_UNFUSED) &&
         (c->pc.smoother == HELM_SM_JACOBI || c->pc.smoother == HELM_SM_RBGS) && !c->lv.empty() &&
         !c->lv[0].any_offset0() && !c->fdm.on && c->ctail_blocks > 0;
}

int ctail_first_level(const helm_ctx* c, long points) {
  const int nl = (int)c->ctail_smem.size();
  for (int l = 0; l < nl; ++l)
    if (c->lv[l].ntot <= points && c->ctail_smem[l]) return l;
  return (int)c->lv.size();
}

// Whether a block's shared memory holds its rows of an operator level of n unknowns, f and the result.
template <typename T> bool ct_op_fits(long n, int nc) {
  const long rows = (n + nc - 1) / nc;
  return sizeof(cx<T>) * (size_t)(rows + 1 + rows * ct_pitch<T>((int)n) + n) <= CTAIL_SMEM;
}

// Once, at create: the dense operator of the finest level small enough for it (see the top), from
// the coarsest inverse, and the arguments for every level the tail can begin at.
template <typename T> helm_status ctail_build(helm_ctx* c, const double2* inv, cudaStream_t st) {
  c->ctail_blocks = ct_blocks();
  if (!ctail_applies(c)) return HELM_OK;
  constexpr bool f64 = std::is_same<T, double>::value;
  const int nl = (int)c->lv.size(), nc = c->ctail_blocks;
  // (a coarsest level above `most` is the operator level itself: its dense inverse has to be applied anyway.  Up
  // to CTAIL_COARSEST unknowns: 4 us of the FP64 pipe, about the launch it replaces)
  const long most = f64 ? 150 : 600;
  ColArgs ca{};
  int l = nl;
  while (l > 0 && c->lv[l - 1].ntot <= (l == nl ? std::max(most, CTAIL_COARSEST) : most) &&
         ct_op_fits<T>(c->lv[l - 1].ntot, nc) && nl - (l - 1) <= COL_MAX_LEVELS)
    --l;
  if (l == nl) return HELM_OK;  // the coarsest level alone is too large
  ca.count = nl - l;
  ca.omega = c->pc.omega;
  int off = 0;
  for (int k = 0; k < ca.count; ++k) {
    ca.op[k] = c->lv[l + k].view<double>();
    ca.at[k] = off;
    off += 3 * (int)c->lv[l + k].ntot;
  }
  const int nop = (int)c->lv[l].ntot;
  helm_status s = ctx_alloc(c, &c->ctail_dense, sizeof(cx<T>) * nop * ct_pitch<T>(nop));
  if (s != HELM_OK) return s;
  const size_t smem = sizeof(double2) * off;  // at most 3 * 600 * 4 / 3 vectors' elements: 38 KB
  double2* o64 = f64 ? (double2*)c->ctail_dense : nullptr;
  float2* o32 = f64 ? nullptr : (float2*)c->ctail_dense;
  auto kern = c->pc.smoother == HELM_SM_RBGS ? k_ctail_columns<true> : k_ctail_columns<false>;
  HELM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
  kern<<<nop, COL_THREADS, smem, st>>>(ca, inv, c->nco, o64, o32, ct_pitch<T>(nop));
  HELM_CUDA(cudaGetLastError());
  c->ctail_op = l;
  std::vector<CTailArgs<T>> all(l + 1);
  std::vector<size_t> need(l + 1);
  for (int k = 0; k <= l; ++k) need[k] = ct_args<T>(c, k, nc, all[k]);
  if ((s = ctx_alloc(c, &c->ctail_dev, sizeof(CTailArgs<T>) * (l + 1))) != HELM_OK) return s;
  HELM_CUDA(cudaMemcpyAsync(c->ctail_dev, all.data(), sizeof(CTailArgs<T>) * (l + 1), cudaMemcpyHostToDevice, st));
  HELM_CUDA(cudaStreamSynchronize(st));
  c->ctail_smem = need;
  return HELM_OK;
}

template <typename T> size_t ctail_args(const helm_ctx* c, int first, const CTailArgs<T>** a) {
  *a = (const CTailArgs<T>*)c->ctail_dev + first;
  return first < (int)c->ctail_smem.size() ? c->ctail_smem[first] : 0;
}

template <typename T, typename TI>
helm_status ctail_vcycle(const helm_ctx* c, int first, const cx<TI>* f, void* out, bool out_f64, const int* skip,
                         cudaStream_t st) {
  const CTailArgs<T>* a;
  const size_t smem = ctail_args<T>(c, first, &a);
  if (!smem) {
    set_error("the one-cluster tail does not fit this hierarchy");
    return HELM_ERR_ARG;
  }
  const bool rb = c->pc.smoother == HELM_SM_RBGS;
  const int nc = c->ctail_blocks;
  if (out_f64) {
    if (rb) launch_cluster(k_ctail<T, true, double, TI>, nc, nc, smem, st, a, f, (double2*)out, skip);
    else launch_cluster(k_ctail<T, false, double, TI>, nc, nc, smem, st, a, f, (double2*)out, skip);
  } else {
    if (rb) launch_cluster(k_ctail<T, true, T, TI>, nc, nc, smem, st, a, f, (cx<T>*)out, skip);
    else launch_cluster(k_ctail<T, false, T, TI>, nc, nc, smem, st, a, f, (cx<T>*)out, skip);
  }
  HELM_CUDA(cudaGetLastError());
  return HELM_OK;
}

template <typename T>
void ctail_group(const GCTail<T>* args, const GroupList* LT, int li, int instances, int nc, bool rb, bool out_f64,
                 size_t smem, cudaStream_t st) {
  const int grid = instances * nc;
  if (out_f64) {
    if (rb) launch_cluster(kg_ctail<T, true, double>, grid, nc, smem, st, args, LT, li);
    else launch_cluster(kg_ctail<T, false, double>, grid, nc, smem, st, args, LT, li);
  } else {
    if (rb) launch_cluster(kg_ctail<T, true, T>, grid, nc, smem, st, args, LT, li);
    else launch_cluster(kg_ctail<T, false, T>, grid, nc, smem, st, args, LT, li);
  }
}

template helm_status ctail_build<float>(helm_ctx*, const double2*, cudaStream_t);
template helm_status ctail_build<double>(helm_ctx*, const double2*, cudaStream_t);
template size_t ctail_args<float>(const helm_ctx*, int, const CTailArgs<float>**);
template size_t ctail_args<double>(const helm_ctx*, int, const CTailArgs<double>**);
template helm_status ctail_vcycle<float, double>(const helm_ctx*, int, const double2*, void*, bool, const int*, cudaStream_t);
template helm_status ctail_vcycle<float, float>(const helm_ctx*, int, const float2*, void*, bool, const int*, cudaStream_t);
template helm_status ctail_vcycle<double, double>(const helm_ctx*, int, const double2*, void*, bool, const int*, cudaStream_t);
template void ctail_group<float>(const GCTail<float>*, const GroupList*, int, int, int, bool, bool, size_t, cudaStream_t);
template void ctail_group<double>(const GCTail<double>*, const GroupList*, int, int, int, bool, bool, size_t, cudaStream_t);

}  // namespace helm
