// mg_cluster.cuh -- the one-cluster tail of 2D V(1,1) cycles (mg_cluster.cu), shared with the lone
// and grouped cycles of mg_fused.cu.
#pragma once
#include "helm_internal.cuh"

namespace helm {

constexpr int CTAIL_MAX_LEVELS = 10;
constexpr int CTAIL_THREADS = 512;
constexpr long CTAIL_COARSEST = 256;  // FP64: the largest coarsest level that a tail ends in
constexpr size_t CTAIL_SMEM = 216 * 1024;  // a block's dynamic shared memory, beside the operator views

// Arguments of one instance's tail: its levels (the last one applies the dense operator) and the places (in
// elements of the block's dynamic shared memory, the same in every block) of their arrays.
template <typename T> struct alignas(16) CTailArgs {
  int count, sh;  // levels; log2 of the blocks
  OpView<T> op[CTAIL_MAX_LEVELS];
  int n0[CTAIL_MAX_LEVELS], n1[CTAIL_MAX_LEVELS];
  int f[CTAIL_MAX_LEVELS], u[CTAIL_MAX_LEVELS], d[CTAIL_MAX_LEVELS];  // staged rows of f, u, 1/D
  int c[CTAIL_MAX_LEVELS];                                           // f as the restriction made it
  int tab[CTAIL_MAX_LEVELS];                                         // axis tables am, ap (x, then y)
  int e, mat, scr;  // the operator level's result and matrix rows, residual / correction scratch
  unsigned magic[CTAIL_MAX_LEVELS], magich[CTAIL_MAX_LEVELS], magicr[CTAIL_MAX_LEVELS], magice[CTAIL_MAX_LEVELS],
      magic1[CTAIL_MAX_LEVELS];  // for divisions by n0, (n0 + 1) / 2, n0 + 1, n0 + 2, n1
  unsigned magicn;     // for divisions by the operator level's unknowns
  const cx<T>* dense;  // its matrix, rows of `pitch` elements
  int pitch;
  T omega;
};

template <typename T> struct GCTail {
  const CTailArgs<T>* a;
  const cx<T>* f;
  void* out;
  const int* skip;
};

bool ctail_applies(const helm_ctx* c);
// the finest level of at most `points` unknowns that a tail can begin at; the level count if none
int ctail_first_level(const helm_ctx* c, long points);
template <typename T> helm_status ctail_build(helm_ctx* c, const double2* inv, cudaStream_t st);
// the device arguments of a tail from level `first`, and its dynamic shared memory (0: does not fit)
template <typename T> size_t ctail_args(const helm_ctx* c, int first, const CTailArgs<T>** a);
template <typename T, typename TI>
helm_status ctail_vcycle(const helm_ctx* c, int first, const cx<TI>* f, void* out, bool out_f64, const int* skip,
                         cudaStream_t st);
template <typename T>
void ctail_group(const GCTail<T>* args, const GroupList* LT, int li, int instances, int nc, bool rb, bool out_f64,
                 size_t smem, cudaStream_t st);

}  // namespace helm
