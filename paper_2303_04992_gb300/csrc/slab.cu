// Launchers of the three-kernel FP32 Schur CG iteration (slab.cuh).
#include <cuda_runtime.h>

#include "slab.cuh"
#include "slab.h"

namespace kfbim {

size_t slab_reduce_slots(int N) {
  switch (N) {
    case 256: return slab::ZShape<256>::REDUCE;
    case 128: return slab::ZShape<128>::REDUCE;
    case 96: return slab::ZShape<96>::REDUCE;
    case 64: return slab::ZShape<64>::REDUCE;
    case 32: return slab::ZShape<32>::REDUCE;
    default: return 0;
  }
}

bool slab_supported(int N) { return N == 32 || N == 64 || N == 96 || N == 128 || N == 256; }

namespace {

template <typename K>
cudaError_t raise(K kern, size_t bytes) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int N, int MAXB>
cudaError_t prepare_nb() {
  cudaError_t e;
  if constexpr (plane::Shape<N>::CL > 1) e = raise(slab::k_cg_terms_cl<N, MAXB>, plane::Smem<N>::bytes);
  else e = raise(slab::k_cg_terms<N, MAXB>, plane::Smem<N>::bytes);
  if (e == cudaSuccess) e = raise(slab::k_cg_zfwd<N, MAXB>, slab::ZShape<N>::bytes);
  if (e == cudaSuccess) e = raise(slab::k_cg_zinv<N, MAXB>, slab::ZShape<N>::bytes);
  if (e == cudaSuccess) e = raise(slab::k_cg_start<N, MAXB>, slab::Conv<N>::bytes);
  if (e == cudaSuccess) e = raise(slab::k_cg_fin<N, MAXB>, slab::Conv<N>::bytes);
  return e;
}

template <int N>
cudaError_t prepare_n() {
  cudaError_t e = prepare_nb<N, 1>();
  if (e == cudaSuccess) e = prepare_nb<N, kSlabBatchMax>();
  if (e == cudaSuccess) e = raise(slab::k_to_slab<N>, slab::Conv<N>::bytes);
  if (e == cudaSuccess) e = raise(slab::k_from_slab<N>, slab::Conv<N>::bytes);
  return e;
}

template <int MAXB>
slab::SlabArgs<MAXB> make_args(const SlabCg* runs, int nrun) {
  slab::SlabArgs<MAXB> a{};
  for (int k = 0; k < nrun; ++k) {
    a.x[k] = runs[k].x;
    a.xs[k] = runs[k].xs;
    a.r[k] = runs[k].r;
    a.d[k] = runs[k].d;
    a.q[k] = runs[k].q;
    a.z1[k] = runs[k].z1;
    a.z3[k] = runs[k].z3;
    a.w1[k] = runs[k].w1;
    a.w2[k] = runs[k].w2;
    a.s[k] = runs[k].s;
    a.partial[k] = runs[k].partial;
  }
  return a;
}

// Launches that overlap the kernel before them: where the measurements in overlap.cuh
// show a gain.
template <int N>
constexpr bool kOverlap = N <= 128;

// Kernel `which` of the iteration: 0 k_cg_zfwd, 1 k_cg_terms, 2 k_cg_zinv; 3 is
// k_cg_fin, the end of a run.
template <int N, int MAXB>
void launch_nb(int which, const slab::SlabArgs<MAXB>& args, const SlabCg& t, int nrun, const CgLoop& loop,
               cudaStream_t st) {
  using Z = slab::ZShape<N>;
  using V = slab::Conv<N>;
  switch (which) {
    case 0:
      slab::k_cg_zfwd<N, MAXB><<<dim3(Z::BLOCKS, nrun), Z::THREADS, Z::bytes, st>>>(args, t.tw, t.qN, loop);
      break;
    case 1:
      if constexpr (plane::Shape<N>::CL > 1)
        (void)launch_overlapped(kOverlap<N>, slab::k_cg_terms_cl<N, MAXB>, dim3(plane::Shape<N>::CL * 3 * N, nrun),
                                plane::Shape<N>::THREADS, plane::Smem<N>::bytes, st, args, t.tw, t.qN, t.s2,
                                t.inv_mu);
      else
        (void)launch_overlapped(kOverlap<N>, slab::k_cg_terms<N, MAXB>, dim3(3 * N, nrun), plane::Shape<N>::THREADS,
                                plane::Smem<N>::bytes, st, args, t.tw, t.qN, t.s2, t.inv_mu);
      break;
    case 2:
      (void)launch_overlapped(kOverlap<N>, slab::k_cg_zinv<N, MAXB>, dim3(Z::BLOCKS, nrun), Z::THREADS, Z::bytes, st, args, t.tw,
                              t.qN);
      break;
    default:
      slab::k_cg_fin<N, MAXB><<<dim3(V::BLOCKS, nrun), V::THREADS, V::bytes, st>>>(args);
  }
}

// `count` kernels of the iteration from `first` on, for nrun runs.
template <int N>
void launch_n(int first, int count, const SlabCg* runs, int nrun, const CgLoop& loop, cudaStream_t st) {
  if (nrun == 1) {
    const slab::SlabArgs<1> args = make_args<1>(runs, 1);
    for (int k = first; k < first + count; ++k) launch_nb<N, 1>(k, args, runs[0], 1, loop, st);
  } else {
    const slab::SlabArgs<kSlabBatchMax> args = make_args<kSlabBatchMax>(runs, nrun);
    for (int k = first; k < first + count; ++k) launch_nb<N, kSlabBatchMax>(k, args, runs[0], nrun, loop, st);
  }
}

template <int N, int MAXB>
void start_nb(const SlabCg* runs, int nrun, const SlabRhs* rhs, double rank1, double cdiag, int* active,
              cudaStream_t st) {
  using V = slab::Conv<N>;
  slab::StartArgs<MAXB> a{};
  for (int k = 0; k < nrun; ++k) {
    a.g[k] = rhs[k].g;
    a.gm[k] = rhs[k].gm;
    a.b1[k] = rhs[k].b1;
    a.b2[k] = rhs[k].b2;
    a.b3[k] = rhs[k].b3;
    a.tol2[k] = rhs[k].tol2;
  }
  slab::k_cg_start<N, MAXB><<<dim3(V::BLOCKS, nrun), V::THREADS, V::bytes, st>>>(make_args<MAXB>(runs, nrun), a, rank1,
                                                                                 cdiag, active);
}

template <int N>
void start_n(const SlabCg* runs, int nrun, const SlabRhs* rhs, double rank1, double cdiag, int* active,
             cudaStream_t st) {
  if (nrun == 1) start_nb<N, 1>(runs, 1, rhs, rank1, cdiag, active, st);
  else start_nb<N, kSlabBatchMax>(runs, nrun, rhs, rank1, cdiag, active, st);
}

template <int N>
void schur_n(const SlabCg& a, const float* d, float* q, cudaStream_t st) {
  using V = slab::Conv<N>;
  slab::k_to_slab<N><<<V::BLOCKS, V::THREADS, V::bytes, st>>>(d, a.r);
  launch_n<N>(0, 3, &a, 1, CgLoop{}, st);
  slab::k_from_slab<N><<<V::BLOCKS, V::THREADS, V::bytes, st>>>(a.q, q);
}

// CALL(N) for a supported grid size, returning n; else 0.
#define KFBIM_SLAB_SWITCH(N_, CALL, n) \
  switch (N_) {                        \
    case 256: CALL(256); return n;     \
    case 128: CALL(128); return n;     \
    case 96: CALL(96); return n;       \
    case 64: CALL(64); return n;       \
    case 32: CALL(32); return n;       \
    default: return 0;                 \
  }

}  // namespace

cudaError_t slab_prepare(int N) {
  switch (N) {
    case 256: return prepare_n<256>();
    case 128: return prepare_n<128>();
    case 96: return prepare_n<96>();
    case 64: return prepare_n<64>();
    case 32: return prepare_n<32>();
    default: return cudaErrorInvalidValue;
  }
}

int slab_cg_start(const SlabCg* runs, int nrun, const SlabRhs* rhs, double rank1, double cdiag, int* active,
                  cudaStream_t st) {
  if (nrun < 1 || nrun > kSlabBatchMax) return 0;
#define KFBIM_CALL(N) start_n<N>(runs, nrun, rhs, rank1, cdiag, active, st)
  KFBIM_SLAB_SWITCH(runs[0].N, KFBIM_CALL, 1)
#undef KFBIM_CALL
}

int slab_cg_iteration(const SlabCg* runs, int nrun, const CgLoop& loop, cudaStream_t st) {
  if (nrun < 1 || nrun > kSlabBatchMax) return 0;
#define KFBIM_CALL(N) launch_n<N>(0, 3, runs, nrun, loop, st)
  KFBIM_SLAB_SWITCH(runs[0].N, KFBIM_CALL, 3)
#undef KFBIM_CALL
}

int slab_cg_finish(const SlabCg* runs, int nrun, cudaStream_t st) {
  if (nrun < 1 || nrun > kSlabBatchMax) return 0;
#define KFBIM_CALL(N) launch_n<N>(3, 1, runs, nrun, CgLoop{}, st)
  KFBIM_SLAB_SWITCH(runs[0].N, KFBIM_CALL, 1)
#undef KFBIM_CALL
}

int slab_launch(int which, const SlabCg& a, cudaStream_t st) {
  if (which < 0 || which > 3) return 0;
#define KFBIM_CALL(N) launch_n<N>(which, 1, &a, 1, CgLoop{}, st)
  KFBIM_SLAB_SWITCH(a.N, KFBIM_CALL, 1)
#undef KFBIM_CALL
}

int slab_schur_apply(const SlabCg& a, const float* d, float* q, cudaStream_t st) {
#define KFBIM_CALL(N) schur_n<N>(a, d, q, st)
  KFBIM_SLAB_SWITCH(a.N, KFBIM_CALL, 5)
#undef KFBIM_CALL
}

}  // namespace kfbim
