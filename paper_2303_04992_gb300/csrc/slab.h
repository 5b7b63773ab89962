// Host entry of the three-kernel FP32 Schur CG iteration of slab.cuh
// (Sec. 4.2, Eq. linearS1), compiled in its own translation unit.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace kfbim {

struct CGScalars;
struct CgLoop;
template <typename T>
struct C2;

// One CG run's buffers: the solution x in natural order; xs, r, d, q (slab order), the
// z-transformed fields z1, z3 and the term results w1, w2 (N^3 floats each); the FP32 transform tables (full-circle
// twiddles exp(-2 pi i t / 2N), t < 2N; post-twiddles exp(-i pi k / 2N), k < N;
// the eigenvalue table 4 sin^2 of the DCT (N) and DST (N) modes), 1/mu, the
// device scalars and the reduction memory (slab_reduce_slots(N) slots of eight
// bytes).
struct SlabCg {
  int N;
  float *x, *xs, *r, *d, *q, *z1, *z3, *w1, *w2;
  const C2<float>* tw;
  const C2<float>* qN;
  const float* s2;
  float inv_mu;
  CGScalars* s;
  double* partial;
};

// Largest number of CG runs one launch of the iteration's kernels serves.
constexpr int kSlabBatchMax = 64;

// Grids the slab iteration covers: N / 2 complex lines of N numbers (a whole
// plane) fit in the shared memory of one CTA, at N = 256 of a cluster of four.
bool slab_supported(int N);
size_t slab_reduce_slots(int N);
// Raises the kernels' dynamic shared-memory limits on the current device.
cudaError_t slab_prepare(int N);

// Every call below returns the number of kernels it enqueued.
//
// The right-hand side of a run, in natural order: b = g - gm[0] + b1 + b2 + b3 (gm
// nullable: no shift; g FP64, rounded once); the run stops at |r|^2 <= tol2 |b|^2.
struct SlabRhs {
  const double* g;
  const double* gm;
  const float *b1, *b2, *b3;
  double tol2;
};
// Start of `nrun` independent runs on one grid (blockIdx.y = run; only
// runs[0]'s N, tables and inv_mu are read): r = b, scalars of
// (S + rank1 1 1^T + cdiag I) x = b; *active (nullable)
// counts the runs that iterate.  The memory of the scalars and of *active must
// have been zeroed.
int slab_cg_start(const SlabCg* runs, int nrun, const SlabRhs* rhs, double rank1, double cdiag, int* active,
                  cudaStream_t st);
// One CG iteration of the runs (a no-op on the device for a run whose s->done is
// set); each run's arithmetic and reduction order are those of a single run.
// Each iteration leaves its own vector update (x += alpha d, r -= alpha q), its
// stopping test and its scalars for the next one's first kernel, so a run ends in
// an iteration that does nothing more.
// loop: the device-side loop the iteration is the body of (captured graphs).
int slab_cg_iteration(const SlabCg* runs, int nrun, const CgLoop& loop, cudaStream_t st);
// x in natural order, with the update still pending when the host stopped
// launching iterations, if any.
int slab_cg_finish(const SlabCg* runs, int nrun, cudaStream_t st);
// One kernel of the iteration (0 k_cg_zfwd, 1 k_cg_terms, 2 k_cg_zinv; 3 the
// finishing update) of a single run, for per-kernel timing.
int slab_launch(int which, const SlabCg& a, cudaStream_t st);
// Algorithmic bytes each kernel moves: 9, 6, 6 and 2 N^3 floats read and written (the
// last reads d as well where the host stopped the run with an update pending).
constexpr int kSlabValues[4] = {9, 6, 6, 2};
// q = S d (the three spectral terms plus s->cdiag d plus s->rank1 sum(d)), d and
// q in natural order, with s->iters = 0, s->beta = 0 and s->done = 0.  At N = 256 the
// tickets in the reduction memory must be zero, as slab_cg_start leaves them.
int slab_schur_apply(const SlabCg& a, const float* d, float* q, cudaStream_t st);

}  // namespace kfbim
