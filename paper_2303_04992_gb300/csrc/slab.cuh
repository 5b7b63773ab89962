// FP32 Schur-complement CG iteration in three kernels (Sec. 4.2, Eq. linearS1
// and items i-iii), for N = 32, 64, 96, 128, 256.
//
// The Schur operator is applied in spectral form,
//   S d = (1/mu) sum_c B_c^-1 Lambda_c B_c d (+ rank-one / c d terms),
// B_c = DCT-II along axis c and DST-II along the other two axes, Lambda_c =
// sin^2(a_c) / sum_b sin^2(a_b).  The transforms along z come first: terms 1
// and 2 share DST-II along z (Z1), term 3 takes DCT-II along z (Z3).  After that
// every (x, y) plane of every term is independent: one CTA per term and plane
// does the rest in shared memory (plane.cuh).  The inverse z transforms of the
// three results are summed into q.
//
// The vector update of iteration k waits for alpha_k, which is known only
// once the reduction of d.q over the whole grid is done, so it is carried
// into the first kernel of iteration k + 1, which touches every element
// anyway (and whose CTAs each merge the blocks' sums of iteration k while their
// vectors load: a last block that merged them took 4 us at the end of every
// iteration); the next r.r (for beta and the stopping test) then comes from its
// expansion
//   |r - alpha q|^2 = r.r - 2 alpha r.q + alpha^2 q.q
// with r.r, r.q and q.q summed beside d.q over the stored vectors.  r.r is
// that of the stored r, never the previous expansion: the expansion carries
// an absolute error of the FP32 rounding times the r.r it started from, and
// carried on from one iteration to the next those errors would add up to
// about 1e-7 of the first r.r, far above a stopping level of 1e-11 of it.
// One CG iteration:
//   k_cg_zfwd   alpha, the next r.r, beta; x += alpha d, r -= alpha q (pending
//               update), d = r + beta d, Z1 = S_z d, Z3 = C_z d, sum(d)
//                                                       (4 reads, 5 writes)
//   k_cg_terms  W1, W2 from Z1, W3 from Z3             (3 reads, 3 writes)
//   k_cg_zinv   q = S_z^-1 (W1 + W2) + C_z^-1 W3 + c d + rank-one; the blocks'
//               sums of d.q, r.r, r.q, q.q              (5 reads, 1 write)
// i.e. 21 N^3 values moved per iteration, against 28 for the transform
// passes of Schur apply run one axis at a time plus 14 for the CG vectors.  The
// k_cg_zfwd that finds the run converged applies the pending update of x and marks
// it done; the kernels after it do nothing.
//
// Orders.  Along every axis position n is Makhoul's (v_n = x_2n, v_(N-1-n) =
// x_(2n+1)), so a line's FFT input is contiguous and DST-II is DCT-II with the
// second half of the positions negated.  A plane's positions are numbered as in
// plane.cuh ("column" = [y / YB][x][y mod YB]).  The CG vectors hold element z
// of column c at ((z / M) N^2 + c) M + z mod M, M = lanes per FFT: the 32 lanes of
// a warp read the M-strided inputs of their 32 / M FFTs as one 128-byte line,
// straight into the FFT registers, and write q's outputs the same way.  The
// z-transformed fields are stored plane by plane (mode index k of the DCT in
// both: DST-II mode a = N - 1 - k).  k_cg_start and k_cg_fin convert from and to
// the natural order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "cg_common.cuh"
#include "fastcvt.h"
#include "overlap.cuh"
#include "plane.cuh"

namespace kfbim {
namespace slab {

// Columns per CTA of the z kernels: 128-byte rows of the plane fields; 64-byte
// ones on the small grids, which have few columns (N = 64: 256 CTAs, N = 32: 64).
template <int N>
struct ZShape {
  using S = plane::Shape<N>;
  static constexpr int TILE = N <= 64 ? 16 : 32;
  static constexpr int THREADS = TILE * S::M;
  static constexpr int BLOCKS = N * N / TILE;
  // two float tiles (N x TILE), over which the FFTs exchange, then the tables
  static constexpr size_t tile = sizeof(float) * N * TILE;
  static constexpr size_t bytes = 2 * tile + sizeof(C2<float>) * (2 * N + S::LINES);
  // blocks whose sums of k_cg_zinv are merged into one part by the last of them,
  // so that no CTA of k_cg_zfwd reads more than 16 KB of parts
  static constexpr int GROUP = BLOCKS > 512 ? BLOCKS / 256 : 1;
  static constexpr int PARTS = BLOCKS / GROUP;
  // a run's reduction memory, in float2: the parts (of four sums), the blocks' sums of d,
  // the blocks' sums of a group, the groups' tickets
  static constexpr int SUMD = 4 * PARTS, BLOCK_SUMS = SUMD + BLOCKS;
  static constexpr int TICKETS = BLOCK_SUMS + (GROUP > 1 ? 4 * BLOCKS : 0);
  static constexpr int REDUCE = TICKETS + (GROUP > 1 ? PARTS : 0);
  // resident CTAs per SM asked of the compiler (64 registers; 100 at N = 96, 24 values per lane;
  // 128 on the small grids, which have few CTAs)
  static constexpr int OCC = THREADS == 512 ? 2 : (THREADS == 256 ? 4 : (N == 96 ? 5 : 4));
};

// Element (z mode k, column l) of a tile at k TILE + (l ^ tile_sw(k)): the lanes of
// a warp (32 / M columns times M consecutive modes) fall on distinct banks, and
// groups of four columns stay together for 16-byte accesses.
template <int N>
__device__ __forceinline__ int tile_at(int k, int l) {
  constexpr int M = plane::Shape<N>::M, TILE = ZShape<N>::TILE;
  const int sw = M == 16 ? ((k >> 1) & 7) * 4   // modes 2i, 2i + 1 share banks (two-way): groups of four stay whole
                 : TILE == 32 ? (k & (M - 1)) * (32 / M) : ((k >> 1) & (M / 2 - 1)) * (32 / M);
  return k * TILE + (l ^ sw);
}

// The exchange slots of a z line: position c of line t at t N + (c ^ sw), sw such
// that the teams of a half warp (adjacent lines) use distinct banks.
template <int N>
__device__ __forceinline__ plane::YSlots<N> z_slots(int t) {
  return {t * N, plane::Shape<N>::M == 16 ? 0 : (plane::Shape<N>::M == 8 ? (t & 1) << 3 : (t & 3) << 2)};
}

// The buffers of up to MAXB independent CG runs on one grid (blockIdx.y
// selects the run): each run's blocks reduce exactly as a single run's, so a
// run's arithmetic does not depend on the batch it is part of.
template <int MAXB>
struct SlabArgs {
  float* x[MAXB];         // solution, natural order (k_cg_fin)
  float* xs[MAXB];        // x, r, d, q in slab order
  float* r[MAXB];
  float* d[MAXB];
  float* q[MAXB];
  float* z1[MAXB];
  float* z3[MAXB];        // W3 replaces Z3 in place
  float* w1[MAXB];
  float* w2[MAXB];
  CGScalars* s[MAXB];
  double* partial[MAXB];
};

// Tables of a z kernel: FFT twiddles [s][m] and [m][s] and post-twiddles q_k, k < N/2.
template <int N>
__device__ __forceinline__ void z_tables(C2<float>* tws, C2<float>* twr, C2<float>* qN,
                                         const C2<float>* __restrict__ twg, const C2<float>* __restrict__ qg) {
  using S = plane::Shape<N>;
  for (int e = threadIdx.x; e < N; e += ZShape<N>::THREADS) {
    tws[e] = twg[2 * (e / S::M) * (e % S::M)];
    twr[e] = twg[2 * (e / S::R) * (e % S::R)];
  }
  for (int e = threadIdx.x; e < S::LINES; e += ZShape<N>::THREADS) qN[e] = qg[e];
}

// Sign of a column block in the fields a term shares: -1 where the axis's
// Makhoul position lies in the second half (the block's columns agree).
template <int N>
__device__ __forceinline__ void col_signs(int col0, float& sx, float& sy) {
  constexpr int YB = plane::Shape<N>::YB;
  const int x = (col0 / YB) % N, y = col0 / (YB * N) * YB;
  sx = x >= N / 2 ? -1.f : 1.f;
  sy = y >= N / 2 ? -1.f : 1.f;
}

// The scalars of an iteration from the parts of the k_cg_zinv before it (PARTS each
// of d.q, r.r, r.q, q.q), merged in a fixed order: every CTA computes the same
// values.  One warp per sum, and one thread for the FP64 arithmetic (by all threads
// of a CTA it alone took 6 us per iteration at N = 128).
struct CgStep {
  double alpha, rr;     // rr: |r - alpha q|^2 by its expansion
  float a, beta;        // alpha, beta in FP32
};
template <int N, int THREADS>
__device__ __forceinline__ void cg_step(const float2* __restrict__ part, double* sums, CgStep* c) {
  constexpr int WARPS = THREADS / 32, P = ZShape<N>::PARTS;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int j = w; j < 4; j += WARPS) {
    CgAcc<float> g;
#pragma unroll 8
    for (int e = lane; e < P; e += 32) {
      const float2 p = part[j * P + e];
      g.merge(p.x, p.y);
    }
    warp_merge(g);
    if (lane == 0) sums[j] = g.value();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double dq = sums[0], rr = sums[1];
    const double alpha = (dq != 0.0) ? rr / dq : 0.0;
    const double r1 = rr - 2.0 * alpha * sums[2] + alpha * alpha * sums[3];
    c->alpha = alpha;
    c->rr = r1;
    c->a = float(alpha);
    c->beta = (rr != 0.0) ? float(r1 / rr) : 0.f;
  }
  __syncthreads();
}

// alpha, beta and the stopping test of the iteration before; its update x += alpha
// d, r -= alpha q (nothing pending in the first iteration; x starts at zero and is
// read from the third on); d = r + beta d; Z1 = DST-II_z d (negated at odd y), Z3 =
// DCT-II_z d (negated at odd x and at odd y); sum d.  A run that has converged or
// reached its cap only gets the update of x.  One column per team of M lanes.
// Bound by the loads' latency (the fields live in the L2 at N <= 128): no
// barrier stands between the loads and the FFT, whose inputs they are.
template <int N, int MAXB>
__global__ void __launch_bounds__(ZShape<N>::THREADS, ZShape<N>::OCC)
k_cg_zfwd(const __grid_constant__ SlabArgs<MAXB> args, const C2<float>* __restrict__ twg,
          const C2<float>* __restrict__ qg, const CgLoop loop) {
  using S = plane::Shape<N>;
  using Z = ZShape<N>;
  constexpr int M = S::M, R = S::R, H = S::H, TILE = Z::TILE;
  __shared__ float2 sh[32];
  __shared__ double sums[4];
  __shared__ CgStep step;
  const int b = blockIdx.y;
  CGScalars* s = args.s[b];
  overlap_trigger();
  // idle: done before this iteration (set by k_cg_start and k_cg_zinv; `done` is
  // written by this kernel and may be seen half-way)
  if (s->idle) {
    if (blockIdx.x == 0 && threadIdx.x == 0) loop_idle(loop);
    return;
  }
  extern __shared__ __align__(16) unsigned char smz[];
  C2<float>* P = reinterpret_cast<C2<float>*>(smz);
  float* O3 = reinterpret_cast<float*>(smz);
  float* O1 = O3 + N * TILE;
  C2<float>* tws = P + N * TILE;
  C2<float>* twr = tws + N;
  C2<float>* qN = twr + N;
  const int t = threadIdx.x / M, m = threadIdx.x % M, lane = threadIdx.x & 31;
  const int partner = (lane & ~(M - 1)) | ((M - m) & (M - 1));
  const int col0 = blockIdx.x * TILE;
  const int its = s->iters;
  const int64_t e0 = (int64_t)(col0 + t) * M + m;
  constexpr int64_t ES = (int64_t)N * N * M;   // from one element of a lane to the next
  float* __restrict__ x = args.xs[b] + e0;
  float* __restrict__ r = args.r[b] + e0;
  float* __restrict__ d = args.d[b] + e0;
  const float* __restrict__ q = args.q[b] + e0;
  CgAcc<float> acc[1];
  C2<float> v[R];
  constexpr int HALF = R > 8 ? R / 2 : R;   // loads in flight per array
  float a = 0.f, beta = 0.f;
  bool stop = false;
#pragma unroll
  for (int h = 0; h < R; h += HALF) {
    float rv[HALF], dv[HALF], xv[HALF], qv[HALF];
#pragma unroll
    for (int j = 0; j < HALF; ++j) {
      rv[j] = r[(h + j) * ES];
      dv[j] = its ? d[(h + j) * ES] : 0.f;
      xv[j] = its > 1 ? x[(h + j) * ES] : 0.f;
      qv[j] = its ? q[(h + j) * ES] : 0.f;
    }
    if (h == 0 && its) {   // while the vectors load
      cg_step<N, Z::THREADS>(reinterpret_cast<const float2*>(args.partial[b]), sums, &step);
      a = step.a;
      beta = step.beta;
      const bool done = !(step.rr > s->stop), cap = loop.maxit > 0 && its >= loop.maxit;
      stop = done || cap;
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        s->alpha = step.alpha;
        s->rr = step.rr;
        if (stop) s->done = done ? 1 : 2;
        loop_step(loop, done, its);
      }
    }
#pragma unroll
    for (int j = 0; j < HALF; ++j) {
      if (its) {
        rv[j] -= a * qv[j];
        x[(h + j) * ES] = xv[j] + a * dv[j];
        r[(h + j) * ES] = rv[j];
      }
      const float nv = rv[j] + beta * dv[j];
      if (!stop) d[(h + j) * ES] = nv;
      acc[0].add(nv);
      // the DCT-II (real) and DST-II (imaginary) inputs of one line
      v[h + j] = {nv, h + j < H ? nv : -nv};
    }
  }
  if (stop) return;
  z_tables<N>(tws, twr, qN, twg, qg);
  __syncthreads();
  plane::fft_to_pairs<N, float>(v, P, z_slots<N>(t), tws, m);
  float sx, sy;
  col_signs<N>(col0, sx, sy);
  const float s3 = sx * sy;
  // C + i S packed: q_k V_k = X_k - i X_(N-k) of both lines, k < N/2
  C2<float> oc[H], os[H];
  plane::for_pairs<N, true, false>(v, m, partner, [&](int i, int k, bool self, C2<float> z, C2<float> g) {
    const C2<float> q0 = plane::ldc(qN + k);
    const C2<float> qc = {0.5f * s3 * q0.x, 0.5f * s3 * q0.y}, qs = {0.5f * sy * q0.x, 0.5f * sy * q0.y};
    oc[i] = cmul(qc, C2<float>{z.x + g.x, z.y - g.y});
    os[i] = cmul(qs, C2<float>{z.y + g.y, g.x - z.x});
    if (self) {   // modes 0 and N/2 are real
      constexpr float c4 = 0.70710678118654752440f;
      oc[i] = {s3 * z.x, -(s3 * c4 * g.x)};
      os[i] = {sy * z.y, -(sy * c4 * g.y)};
    }
  });
  __syncthreads();   // every team is through its exchange, which the tiles overlay
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const int k = plane::pair_index<N>(i, m), kn = k ? N - k : N / 2;
    O3[tile_at<N>(k, t)] = oc[i].x;
    O3[tile_at<N>(kn, t)] = -oc[i].y;
    O1[tile_at<N>(k, t)] = os[i].x;
    O1[tile_at<N>(kn, t)] = -os[i].y;
  }
  __syncthreads();
  float* __restrict__ z1 = args.z1[b];
  float* __restrict__ z3 = args.z3[b];
  for (int e4 = threadIdx.x; e4 < N * (TILE / 4); e4 += Z::THREADS) {
    const int k = e4 / (TILE / 4), c4 = (e4 % (TILE / 4)) * 4;
    const int64_t g = (int64_t)k * N * N + col0 + c4;
    *reinterpret_cast<float4*>(z1 + g) = *reinterpret_cast<const float4*>(O1 + tile_at<N>(k, c4));
    *reinterpret_cast<float4*>(z3 + g) = *reinterpret_cast<const float4*>(O3 + tile_at<N>(k, c4));
  }
  // the block's part of sum(d); k_cg_terms merges the parts
  block_merge<1>(acc, sh);
  if (threadIdx.x == 0)
    (reinterpret_cast<float2*>(args.partial[b]) + Z::SUMD)[blockIdx.x] = make_float2(acc[0].s, acc[0].c);
}

// sum(d) from the blocks' parts of k_cg_zfwd, in block order, by one CTA.
template <int N, int THREADS>
__device__ __forceinline__ void merge_sumd(const float2* __restrict__ part, CGScalars* s) {
  __shared__ float2 sh[32];
  CgAcc<float> g[1];
  for (int e = threadIdx.x; e < ZShape<N>::BLOCKS; e += THREADS) g[0].merge(part[e].x, part[e].y);
  block_merge<1>(g, sh);
  if (threadIdx.x == 0) s->sumd = g[0].value();
}

// One term of the Schur operator on one plane (plane.cuh), plane-major so that
// terms 1 and 2 of a plane read Z1 close in time.  Z1 carries the signs of the
// DST-II along y, Z3 those along x and y.
template <int N, int MAXB>
__device__ __forceinline__ void terms_body(const SlabArgs<MAXB>& args, int unit, int rank,
                                           const C2<float>* __restrict__ twg, const C2<float>* __restrict__ qg,
                                           const float* __restrict__ s2g, float inv_mu) {
  const int b = blockIdx.y;
  extern __shared__ __align__(16) unsigned char smx[];
  plane::term_tables<N>(reinterpret_cast<C2<float>*>(smx), twg, qg, s2g);
  overlap_wait();
  overlap_trigger();
  if (args.s[b]->done) return;
  if (unit == 3 * N - 1 && rank == 0)
    merge_sumd<N, plane::Shape<N>::THREADS>(reinterpret_cast<const float2*>(args.partial[b]) + ZShape<N>::SUMD, args.s[b]);
  const int term = unit % 3, k = unit / 3;
  const int64_t off = (int64_t)k * N * N;
  const float* in = (term == 2 ? args.z3[b] : args.z1[b]) + off;
  float* out = (term == 0 ? args.w1[b] : (term == 1 ? args.w2[b] : args.z3[b])) + off;
  // 4 sin^2 along z: DCT-II mode k (term 3), DST-II mode N - 1 - k (terms 1, 2)
  const float az = term == 2 ? s2g[k] : s2g[2 * N - 1 - k];
  // 1 / N per inverse transform, as the one-axis passes scale: at N = 96 the rounding of
  // 1 / 96 offsets part of the FFT constants' (operator error 2.1e-7 with 1 / N^2 rounded once)
  constexpr float invN = 1.0f / N;
  plane::term_plane<N>(in, out, plane::term_of(term), plane::term_of(term == 2 ? 2 : 0), az,
                              inv_mu * (invN * invN), reinterpret_cast<C2<float>*>(smx), rank);
}
template <int N, int MAXB>
__global__ void __launch_bounds__(plane::Shape<N>::THREADS, 2)
k_cg_terms(const __grid_constant__ SlabArgs<MAXB> args, const C2<float>* __restrict__ twg,
           const C2<float>* __restrict__ qg, const float* __restrict__ s2g, float inv_mu) {
  terms_body<N, MAXB>(args, blockIdx.x, 0, twg, qg, s2g, inv_mu);
}
// The same with a plane on a cluster (N = 256): 235 us as four CTAs of 256 threads,
// two clusters' CTAs per SM (272 us as two CTAs of 512); issue 42 %, shared memory
// 38 % busy, the rest the waits of 16 warps per SM.  The five one-axis stages it
// replaces took 1.16 ms of a staged CG iteration of 1.32 ms (now 0.42 ms).
template <int N, int MAXB>
__global__ void __cluster_dims__(plane::Shape<N>::CL, 1, 1) __launch_bounds__(plane::Shape<N>::THREADS, 2)
k_cg_terms_cl(const __grid_constant__ SlabArgs<MAXB> args, const C2<float>* __restrict__ twg,
              const C2<float>* __restrict__ qg, const float* __restrict__ s2g, float inv_mu) {
  terms_body<N, MAXB>(args, blockIdx.x / plane::Shape<N>::CL, blockIdx.x % plane::Shape<N>::CL, twg, qg, s2g, inv_mu);
}

// q = DST-III_z (W1 + W2) + DCT-III_z W3 + cdiag d + rank1 sumd; the blocks' sums of
// d.q, r.r, r.q and q.q.  Columns as k_cg_zfwd; W1 comes negated at odd y, W2 at odd x, W3 at both.
template <int N, int MAXB>
__global__ void __launch_bounds__(ZShape<N>::THREADS, ZShape<N>::OCC)
k_cg_zinv(const __grid_constant__ SlabArgs<MAXB> args, const C2<float>* __restrict__ twg,
          const C2<float>* __restrict__ qg) {
  using S = plane::Shape<N>;
  using Z = ZShape<N>;
  constexpr int M = S::M, R = S::R, H = S::H, TILE = Z::TILE;
  __shared__ float2 sh[4 * 32];
  const int b = blockIdx.y;
  CGScalars* s = args.s[b];
  extern __shared__ __align__(16) unsigned char smi[];
  C2<float>* P = reinterpret_cast<C2<float>*>(smi);
  float* O3 = reinterpret_cast<float*>(smi);
  float* O1 = O3 + N * TILE;
  C2<float>* tws = P + N * TILE;
  C2<float>* twr = tws + N;
  C2<float>* qN = twr + N;
  z_tables<N>(tws, twr, qN, twg, qg);
  overlap_wait();
  if (s->done) {
    if (blockIdx.x == 0 && threadIdx.x == 0) s->idle = 1;
    return;
  }
  const int t = threadIdx.x / M, m = threadIdx.x % M, lane = threadIdx.x & 31;
  const int partner = (lane & ~(M - 1)) | ((M - m) & (M - 1));
  const int col0 = blockIdx.x * TILE;
  float sx, sy;
  col_signs<N>(col0, sx, sy);
  {
    const float* __restrict__ w1 = args.w1[b] + col0;
    const float* __restrict__ w2 = args.w2[b] + col0;
    const float* __restrict__ w3 = args.z3[b] + col0;
    constexpr int PER = N * (TILE / 4) / Z::THREADS;   // float4 groups per thread (R / 4)
    static_assert(PER * Z::THREADS == N * (TILE / 4), "whole groups");
    float4 f1[PER], f2[PER], f3[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int e4 = threadIdx.x + j * Z::THREADS;
      const int64_t g = (int64_t)(e4 / (TILE / 4)) * N * N + (e4 % (TILE / 4)) * 4;
      f1[j] = *reinterpret_cast<const float4*>(w1 + g);
      f2[j] = *reinterpret_cast<const float4*>(w2 + g);
      f3[j] = *reinterpret_cast<const float4*>(w3 + g);
    }
    const float s3 = sx * sy;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int e4 = threadIdx.x + j * Z::THREADS;
      const int at = tile_at<N>(e4 / (TILE / 4), (e4 % (TILE / 4)) * 4);
      *reinterpret_cast<float4*>(O1 + at) =
          make_float4(sy * f1[j].x + sx * f2[j].x, sy * f1[j].y + sx * f2[j].y, sy * f1[j].z + sx * f2[j].z,
                      sy * f1[j].w + sx * f2[j].w);
      *reinterpret_cast<float4*>(O3 + at) = make_float4(s3 * f3[j].x, s3 * f3[j].y, s3 * f3[j].z, s3 * f3[j].w);
    }
  }
  __syncthreads();
  // both inverse transforms of a column in one FFT: conj Z_k = q conj(A + i B),
  // conj Z_(N-k) = conj(q) (A - i B) with A = X_k - i X_(N-k) of the DCT-III input,
  // B of the DST-III input
  C2<float> v[R];
  plane::for_pairs<N, false, true>(v, m, partner, [&](int, int k, bool self, C2<float>& lo, C2<float>& hi) {
    const int kn = k ? N - k : N / 2;
    const float ax = O3[tile_at<N>(k, t)], ay = -O3[tile_at<N>(kn, t)];
    const float bx = O1[tile_at<N>(k, t)], by = -O1[tile_at<N>(kn, t)];
    const C2<float> q0 = plane::ldc(qN + k);
    lo = cmul(q0, C2<float>{ax - by, -(ay + bx)});
    hi = cmul(plane::conjg(q0), C2<float>{ax + by, ay - bx});
    if (self) {
      constexpr float c2 = 1.41421356237309504880f;
      lo = {ax, -bx};
      hi = {-(c2 * ay), c2 * by};
    }
  });
  __syncthreads();   // the tiles are read; the exchange overlays them
  plane::fft_from_pairs<N, float>(v, P, z_slots<N>(t), tws, twr, m);
  // q = the two inverse transforms + c d + rank-one; d.q, r.r, r.q and q.q for
  // alpha and the expansion of the next r.r.  d.q and r.r (alpha, the stopping
  // test) exact to about 2^-48: every product split by FMA, all sums compensated;
  // r.q and q.q (only in the expansion) sum four products by FMA first (within 3
  // roundings of their magnitudes) and those sums compensated
  const int64_t e0 = (int64_t)(col0 + t) * M + m;
  constexpr int64_t ES = (int64_t)N * N * M;
  const float* __restrict__ d = args.d[b] + e0;
  const float* __restrict__ r = args.r[b] + e0;
  float* __restrict__ q = args.q[b] + e0;
  const float cd = float(s->cdiag), c1 = float(s->sumd * s->rank1);
  constexpr float invN = 1.0f / N;
  CgAcc<float> acc[4];
#pragma unroll
  for (int h = 0; h < R; h += H) {
    float dv[H], rv[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      dv[j] = d[(h + j) * ES];
      rv[j] = r[(h + j) * ES];
    }
#pragma unroll
    for (int j = 0; j < H; j += 4) {
      float rq = 0.f, qq = 0.f;
#pragma unroll
      for (int i = j; i < j + 4; ++i) {
        // C line + S line (its second half negated); v holds the conjugate
        const float sum = h + i < H ? v[h + i].x - v[h + i].y : v[h + i].x + v[h + i].y;
        const float qv = invN * sum + (cd * dv[i] + c1);
        q[(h + i) * ES] = qv;
        acc[0].add_prod(dv[i], qv);
        acc[1].add_prod(rv[i], rv[i]);
        rq = fmaf(rv[i], qv, rq);
        qq = fmaf(qv, qv, qq);
      }
      acc[2].add(rq);
      acc[3].add(qq);
    }
  }
  // the block's (or its group's) part
  float2* part = reinterpret_cast<float2*>(args.partial[b]);
  block_merge<4>(acc, sh);
  if constexpr (Z::GROUP == 1) {
    if (threadIdx.x == 0) {
#pragma unroll
      for (int j = 0; j < 4; ++j) part[j * Z::PARTS + blockIdx.x] = make_float2(acc[j].s, acc[j].c);
    }
  } else {
    if (threadIdx.x == 0) {
      float2* own = part + Z::BLOCK_SUMS + 4 * blockIdx.x;
#pragma unroll
      for (int j = 0; j < 4; ++j) own[j] = make_float2(acc[j].s, acc[j].c);
      __threadfence();
      const int g = blockIdx.x / Z::GROUP;
      unsigned int* ticket = reinterpret_cast<unsigned int*>(part + Z::TICKETS + g);
      if (atomicAdd(ticket, 1u) == Z::GROUP - 1) {   // the group's last block: its blocks in order
        __threadfence();
        CgAcc<float> m[4];
        for (int k = 0; k < Z::GROUP; ++k)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 p = __ldcg(part + Z::BLOCK_SUMS + 4 * (g * Z::GROUP + k) + j);
            m[j].merge(p.x, p.y);
          }
#pragma unroll
        for (int j = 0; j < 4; ++j) part[j * Z::PARTS + g] = make_float2(m[j].s, m[j].c);
        *ticket = 0u;
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) s->iters += 1;
}

// ------------------------------------------------ natural <-> slab order
// A CTA converts the YB y positions x M z positions of one block of rows: in
// natural order YB M rows of N numbers, in slab order one contiguous run of
// YB M N, element (x, yy, zz) at (x YB + yy) M + zz.
template <int N>
struct Conv {
  using S = plane::Shape<N>;
  static constexpr int ROWS = S::YB * S::M;              // 64
  static constexpr int BLOCKS = (N / S::YB) * (N / S::M);
  static constexpr int THREADS = 256;
  static constexpr int RS = N + 1;                       // padded row in shared memory
  static constexpr size_t bytes = sizeof(float) * ROWS * RS;
  __device__ static int nat(int n) { return n < N / 2 ? 2 * n : 2 * (N - 1 - n) + 1; }
  // the natural offset of row (yy, zz) of block blk, and the slab offset of the block
  __device__ static int64_t row(int blk, int rw) {
    const int y = (blk % (N / S::YB)) * S::YB + rw / S::M, z = (blk / (N / S::YB)) * S::M + rw % S::M;
    return ((int64_t)nat(z) * N + nat(y)) * N;
  }
  __device__ static int64_t base(int blk) {
    return ((int64_t)(blk / (N / S::YB)) * N * N + (int64_t)(blk % (N / S::YB)) * N * S::YB) * S::M;
  }
};

// out (slab order) = in (natural order), or the reverse.
template <int N>
__global__ void __launch_bounds__(Conv<N>::THREADS) k_to_slab(const float* __restrict__ in, float* __restrict__ out) {
  using V = Conv<N>;
  extern __shared__ float smc[];
  const int blk = blockIdx.x;
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) smc[(e / N) * V::RS + e % N] = in[V::row(blk, e / N) + e % N];
  __syncthreads();
  float* o = out + V::base(blk);
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) o[e] = smc[(e % V::ROWS) * V::RS + V::nat(e / V::ROWS)];
}
template <int N>
__global__ void __launch_bounds__(Conv<N>::THREADS) k_from_slab(const float* __restrict__ in, float* __restrict__ out) {
  using V = Conv<N>;
  extern __shared__ float smc[];
  const int blk = blockIdx.x;
  const float* i = in + V::base(blk);
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) smc[(e % V::ROWS) * V::RS + V::nat(e / V::ROWS)] = i[e];
  __syncthreads();
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) out[V::row(blk, e / N) + e % N] = smc[(e / N) * V::RS + e % N];
}

// Right-hand sides b = g - gm[0] + b1 + b2 + b3 (natural order; gm nullable) and
// squared relative tolerances of up to MAXB runs.
template <int MAXB>
struct StartArgs {
  const double* g[MAXB];
  const double* gm[MAXB];
  const float *b1[MAXB], *b2[MAXB], *b3[MAXB];
  double tol2[MAXB];
};

// Start of a run on (S + rank one) x = b from x = 0: r = b in slab order, and
// the scalars rr = b.b, stop = tol2 b.b (compensated FP32 sums, cg_common.cuh);
// *active counts the runs that iterate.
// x and d need no start values: the first iterations do not read them.
template <int N, int MAXB>
__global__ void __launch_bounds__(Conv<N>::THREADS)
k_cg_start(const __grid_constant__ SlabArgs<MAXB> args, const __grid_constant__ StartArgs<MAXB> st, double rank1,
           double cdiag, int* active) {
  using V = Conv<N>;
  extern __shared__ float smc[];
  __shared__ float2 sh[32];
  const int run = blockIdx.y, blk = blockIdx.x;
  CGScalars* s = args.s[run];
  const double* __restrict__ g = st.g[run];
  const double* __restrict__ gm = st.gm[run];
  const float *__restrict__ b1 = st.b1[run], *__restrict__ b2 = st.b2[run], *__restrict__ b3 = st.b3[run];
  CgAcc<float> acc[1];
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) {
    const int64_t at = V::row(blk, e / N) + e % N;
    // FP32 sums of the FP64 g rounded once (by integer operations)
    const float v = f64_to_f32(gm ? g[at] - gm[0] : g[at]) + b1[at] + b2[at] + b3[at];
    smc[(e / N) * V::RS + e % N] = v;
    acc[0].add_prod(v, v);
  }
  __syncthreads();
  float* __restrict__ o = args.r[run] + V::base(blk);
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) o[e] = smc[(e % V::ROWS) * V::RS + V::nat(e / V::ROWS)];
  if constexpr (ZShape<N>::GROUP > 1) {   // the tickets of k_cg_zinv's groups
    if (blk == 0)
      for (int e = threadIdx.x; e < ZShape<N>::PARTS; e += V::THREADS)
        *reinterpret_cast<unsigned int*>(reinterpret_cast<float2*>(args.partial[run]) + ZShape<N>::TICKETS + e) = 0u;
  }
  double sum[1];
  if (last_block_merge<1>(acc, reinterpret_cast<float2*>(args.partial[run]), &s->ticket[1], sh, sum) &&
      threadIdx.x == 0) {
    s->rr = sum[0];
    s->bb = sum[0];
    s->stop = st.tol2[run] * sum[0];
    s->rank1 = rank1;
    s->cdiag = cdiag;
    s->iters = 0;
    s->done = s->idle = (sum[0] > s->stop) ? 0 : 1;
    if (active && !s->done) atomicAdd(active, 1);
  }
}

// End of a run: x in natural order (0 when no iteration ran); a run that the host
// stopped before k_cg_zfwd saw its end still has an update pending.
template <int N, int MAXB>
__global__ void __launch_bounds__(Conv<N>::THREADS) k_cg_fin(const __grid_constant__ SlabArgs<MAXB> args) {
  using V = Conv<N>;
  extern __shared__ float smc[];
  __shared__ double sums[4];
  __shared__ CgStep step;
  const int run = blockIdx.y, blk = blockIdx.x;
  const CGScalars* s = args.s[run];
  const int its = s->iters;
  const float* __restrict__ xs = args.xs[run] + V::base(blk);
  float a = 0.f;
  const bool pending = its && !s->done;
  if (pending) {
    cg_step<N, V::THREADS>(reinterpret_cast<const float2*>(args.partial[run]), sums, &step);
    a = step.a;
  }
  const float* __restrict__ d = args.d[run] + V::base(blk);
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) {
    float x0 = its > (pending ? 1 : 0) ? xs[e] : 0.f;
    if (pending) x0 += a * d[e];
    smc[(e % V::ROWS) * V::RS + V::nat(e / V::ROWS)] = x0;
  }
  __syncthreads();
  float* __restrict__ x = args.x[run];
#pragma unroll 8
  for (int e = threadIdx.x; e < V::ROWS * N; e += V::THREADS) x[V::row(blk, e / N) + e % N] = smc[(e / N) * V::RS + e % N];
}

}  // namespace slab
}  // namespace kfbim
