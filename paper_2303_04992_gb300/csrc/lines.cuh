// One-axis transform pass: the real transforms of transforms.cuh (DCT-II/III,
// DST-II/III, DST-I) of every line of an N^3 field along one axis, optionally
// followed by the spectral weight and an inverse transform along the same axis
// in the same registers.  N = 32, 64, 96, 128, 256; FP32 and FP64.
//
// A team of M lanes (plane.cuh) transforms a pair of adjacent lines: DCT-II and
// DST-II of the two real lines as one complex FFT in Makhoul's order (a DST-II is
// the DCT-II with the odd elements negated, its mode a at DCT index N - 1 - a),
// DST-I one line at a time: the odd extension y of the line (length 2N) packed as
// z_n = y_2n + i y_(2n+1) is one complex FFT of length N, and with
// a, b = (Z_k +- conj Z_(N-k)) / 2, w = exp(-i pi k / N) its modes are
//   X_k, X_(N-k) = (Re(w b) -+ Im a) / 2;
// backwards Z_k = (c s, s' s + d), Z_(N-k) = (-c s, s' s - d) with c + i s' =
// exp(i pi k / N), s = X_k + X_(N-k), d = X_(N-k) - X_k, and the inverse FFT is
// z_n = x_2n + i x_(2n+1).  A lane ends a forward transform holding modes k and
// N - k of its lines (plane::for_pairs), which is what the inverse starts from, so
// the weight of a fused pass costs no exchange.
//
// Lines go from global memory straight into the FFT registers and back: along y
// and z a pair of lines is one vector per element and a warp's teams fill 32- to
// 64-byte sectors; along x a lane reads (x_2n, x_(2n+1)) as one vector and hands
// the odd element to its mirror lane by a shuffle.  Shared memory holds the FFT
// exchange (N complex numbers per team) and the twiddles; the teams of a CTA do
// not wait for one another.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fastcvt.h"
#include "overlap.cuh"
#include "plane.cuh"
#include "transforms.cuh"

namespace kfbim {
namespace lines {

// What a pass does.  F2, I2: forward / inverse of the DCT-II and DST-II family;
// F1, I1: DST-I; the others forward, weight, inverse.
enum Op : int { OP_F2 = 0, OP_I2, OP_F1, OP_I1, OP_F2I2, OP_F1I1, OP_F1I2 };
__host__ __device__ constexpr bool op_fwd1(int op) { return op == OP_F1 || op == OP_F1I1 || op == OP_F1I2; }
__host__ __device__ constexpr bool op_fwd2(int op) { return op == OP_F2 || op == OP_F2I2; }
__host__ __device__ constexpr bool op_inv1(int op) { return op == OP_I1 || op == OP_F1I1; }
__host__ __device__ constexpr bool op_inv2(int op) { return op == OP_I2 || op == OP_F2I2 || op == OP_F1I2; }

// One pass of one field.  vec: in and out are aligned for vectors of two numbers.
template <typename Tin, typename Tout>
struct Job {
  const Tin* in;
  Tout* out;
  const int* skip;   // nullable: the pass does nothing when *skip != 0
  int8_t axis;       // 0 x, 1 y, 2 z
  int8_t dst;        // F2, I2: 1 for the DST-II family
  int8_t wmode, wc;  // weight mode (transforms.cuh), component axis of the weight
  int8_t vec;
  int8_t acc;        // FP64 output of an FP32 inverse pass: added to `out` instead of stored
};
template <typename Tin, typename Tout, int MAXJ>
struct Jobs {
  Job<Tin, Tout> j[MAXJ];
};

template <int N, typename T>
struct LShape {
  using S = plane::Shape<N>;
  // FP64: the 512 CTAs of 128 threads of one field at N = 128 are 3.4 per SM, which
  // the FP64 pipe (two lanes per SM and cycle) works through as four; 64 threads
  static constexpr int THREADS = sizeof(T) == 8 ? 64 : 128;
  static constexpr int TEAMS = THREADS / S::M;             // line pairs per CTA
  static constexpr int BLOCKS = (N * N / 2 + TEAMS - 1) / TEAMS;
  // FP32 at N = 256: a team of 16 lanes reads 16 rows of a pair at once, 16 bytes in
  // each of 16 cache lines, and the L1's tag stage bounds the pass (85 % busy, 79 us
  // per field along y or z against 30 along x); its CTA stages 64-byte rows instead
  static constexpr bool STAGED = sizeof(T) == 4 && S::M == 16;
  static constexpr int COLS = 2 * TEAMS;                   // lines per CTA
  static constexpr size_t tile = STAGED ? sizeof(T) * N * COLS : 0;
  static constexpr size_t bytes = sizeof(C2<T>) * ((size_t)TEAMS * N + 2 * N) + tile;
  // CTAs per SM asked of the compiler.  FP32: 96 registers, 128 where two lines' modes are
  // held beside the FFT (168 at N = 96, 24 values per lane).  FP64: 128 registers for a plain
  // pass (the 1024 CTAs of one field at N = 128 resident at once), 168 and 255.
  static constexpr int occ(int op) {
    if (sizeof(T) == 8) return N == 96 || op == OP_F1I2 ? 4 : (op == OP_F2 || op == OP_I2 ? 8 : 6);
    return N == 96 ? 3 : (op == OP_F1I2 ? 4 : 5);
  }
};

template <typename T, typename Tin>
__device__ __forceinline__ T to_work(Tin v) {
  if constexpr (sizeof(T) == 4 && sizeof(Tin) == 8) return f64_to_f32(v);   // integer operations: fastcvt.h
  else return T(v);
}

// Two adjacent numbers p[0], p[1].
template <typename T, typename Tin>
__device__ __forceinline__ C2<T> ld2(const Tin* p, bool vec) {
  if (vec) {
    if constexpr (sizeof(Tin) == 4) {
      const float2 v = *reinterpret_cast<const float2*>(p);
      return {to_work<T>(v.x), to_work<T>(v.y)};
    } else {
      const double2 v = *reinterpret_cast<const double2*>(p);
      return {to_work<T>(v.x), to_work<T>(v.y)};
    }
  }
  return {to_work<T>(p[0]), to_work<T>(p[1])};
}
template <typename T, typename Tout>
__device__ __forceinline__ void st2(Tout* p, T a, T b, bool vec, bool acc = false) {
  if constexpr (sizeof(Tout) == 8 && sizeof(T) == 4) {   // exact widening by integer operations
    double2 v = make_double2(f32_to_f64(a), f32_to_f64(b));
    double2* q = reinterpret_cast<double2*>(p);          // a field of the library: aligned
    if (acc) {
      const double2 o = *q;
      v.x += o.x;
      v.y += o.y;
    }
    *q = v;
  } else if (vec) {
    if constexpr (sizeof(Tout) == 4) *reinterpret_cast<float2*>(p) = make_float2(a, b);
    else *reinterpret_cast<double2*>(p) = make_double2(a, b);
  } else {
    p[0] = a;
    p[1] = b;
  }
}

// a, negated where `neg` (by its sign bits: no FP64 instruction).
template <typename T>
__device__ __forceinline__ T flip(T a, bool neg) {
  if constexpr (sizeof(T) == 4) return __uint_as_float(__float_as_uint(a) ^ (neg ? 0x80000000u : 0u));
  else return __hiloint2double(__double2hiint(a) ^ (neg ? (int)0x80000000 : 0), __double2loint(a));
}

// The exchange slots of a team: as plane.cuh's along y, each team its own line.
template <int N>
__device__ __forceinline__ plane::YSlots<N> slots(int t) {
  constexpr int M = plane::Shape<N>::M;
  return {t * N, M == 16 ? 0 : (M == 8 ? (t & 1) << 3 : (t & 3) << 2)};
}

// The constant factors of the spectral weights, each rounded once from FP64: 1 / mu
// (W_SCHUR), h^2 / mu (W_POISSON), -h / mu (W_RHS).
template <typename T>
struct Scales {
  T schur, poisson, rhs;
};

// Weights of a pass (the factors of spectral_weight2): 4 sin^2 of the line's two
// other modes, of the mode along the pass's axis, and the numerator.
template <typename T, int N>
struct Weights {
  const T* __restrict__ s2;
  T rest;       // 4 sin^2 of the modes across the line, summed
  T num;        // numerator, where it is not that of the pass's axis
  int kind;     // 0: the pass's axis takes DCT / DST-I modes, 1: DST-II modes
  int wmode;
  bool own;     // the weight's component axis is the pass's axis
  Scales<T> sc;
  // numerator for component mode value v = 4 sin^2 (zero for mode 0 of a face basis)
  __device__ __forceinline__ T numer(T v, bool zero) const {
    if (wmode == W_SCHUR) return v * sc.schur;
    if (zero) return T(0);
    if (wmode == W_POISSON) return sc.poisson;
    return sc.rhs * sqrt(v);   // -2 h sin(a), v = 4 sin^2(a)
  }
  __device__ __forceinline__ T at(int a, T& den) const {
    const T v = s2[kind * N + a];
    den = rest + v;
    return own ? numer(v, a == 0) : num;
  }
};

// The staged tile of a CTA: element i of line c at i COLS + (c ^ sw(i)) (pairs stay
// together; rows 2 i and 2 i + 2 of a team's accesses on distinct banks).
template <int COLS>
__device__ __forceinline__ int tile_at(int i, int c) {
  return i * COLS + (c ^ (2 * ((i >> 1) & (COLS / 2 - 1))));
}
template <int N, int COLS, int THREADS, typename T, typename Tin>
__device__ __forceinline__ void tile_load(T* tile, const Tin* in, int64_t es) {
  constexpr int Q = COLS / 4;
  const bool wide = reinterpret_cast<uintptr_t>(in) % 16 == 0;   // a caller's field may not be
#pragma unroll 8
  for (int e = threadIdx.x; e < N * Q; e += THREADS) {
    const int i = e / Q, c = (e % Q) * 4;
    const Tin* p = in + (int64_t)i * es + c;
    T v[4];
    if (wide && sizeof(Tin) == 4) {
      const float4 f = *reinterpret_cast<const float4*>(p);
      v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    } else if (wide) {
      const double2 f = reinterpret_cast<const double2*>(p)[0], g = reinterpret_cast<const double2*>(p)[1];
      v[0] = to_work<T>(f.x); v[1] = to_work<T>(f.y); v[2] = to_work<T>(g.x); v[3] = to_work<T>(g.y);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = to_work<T>(p[k]);
    }
    *reinterpret_cast<float2*>(tile + tile_at<COLS>(i, c)) = make_float2(v[0], v[1]);
    *reinterpret_cast<float2*>(tile + tile_at<COLS>(i, c + 2)) = make_float2(v[2], v[3]);
  }
}
template <int N, int COLS, int THREADS, typename T, typename Tout>
__device__ __forceinline__ void tile_store(const T* tile, Tout* out, int64_t es, bool acc) {
  constexpr int Q = COLS / 4;
  const bool wide = reinterpret_cast<uintptr_t>(out) % 16 == 0;
#pragma unroll 4
  for (int e = threadIdx.x; e < N * Q; e += THREADS) {
    const int i = e / Q, c = (e % Q) * 4;
    Tout* p = out + (int64_t)i * es + c;
    const float2 a = *reinterpret_cast<const float2*>(tile + tile_at<COLS>(i, c));
    const float2 b = *reinterpret_cast<const float2*>(tile + tile_at<COLS>(i, c + 2));
    if constexpr (sizeof(Tout) == 8) {
      st2<T>(p, a.x, a.y, true, acc);
      st2<T>(p + 2, b.x, b.y, true, acc);
    } else if (wide) {
      *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
    } else {
      p[0] = a.x;
      p[1] = a.y;
      p[2] = b.x;
      p[3] = b.y;
    }
  }
}

template <typename Tin, typename T, typename Tout, int N, int OP, int MAXJ>
__global__ void __launch_bounds__((LShape<N, T>::THREADS), (LShape<N, T>::occ(OP)))
k_lines(const __grid_constant__ Jobs<Tin, Tout, MAXJ> jobs, const Scales<T> scales, const C2<T>* __restrict__ twg,
        const C2<T>* __restrict__ qg, const T* __restrict__ s2) {
  using S = plane::Shape<N>;
  using L = LShape<N, T>;
  constexpr int M = S::M, R = S::R, H = S::H;
  const Job<Tin, Tout>& job = jobs.j[blockIdx.y];
  extern __shared__ __align__(16) unsigned char sml[];
  C2<T>* P = reinterpret_cast<C2<T>*>(sml);
  C2<T>* tws = P + L::TEAMS * N;
  C2<T>* twr = tws + N;
  constexpr bool pairs = plane::PairShape<N>::in_lane;
  for (int e = threadIdx.x; e < N; e += L::THREADS) {
    if (op_fwd1(OP) || op_fwd2(OP) || !pairs) tws[e] = twg[2 * (e / M) * (e % M)];
    if ((op_inv1(OP) || op_inv2(OP)) && pairs) twr[e] = twg[2 * (e / R) * (e % R)];
  }
  overlap_wait();
  overlap_trigger();
  if (job.skip && *job.skip) return;
  __syncthreads();
  const int t = threadIdx.x / M, m = threadIdx.x % M, lane = threadIdx.x & 31;
  const int partner = (lane & ~(M - 1)) | ((M - m) & (M - 1));
  const int pair = blockIdx.x * L::TEAMS + t;   // N^2 / 2 is a multiple of the CTA's teams
  const int line = 2 * pair;
  const int axis = job.axis;
  const bool vec = job.vec, dst = job.dst, acc = job.acc;
  // lines: x: line = k N + j (contiguous); y: (k, i); z: (j, i); ls, es: strides of lines and elements
  const int64_t base = axis == 0 ? (int64_t)line * N : (axis == 1 ? (int64_t)(line / N) * N * N + line % N : line);
  const int64_t ls = axis == 0 ? N : 1, es = axis == 0 ? 1 : (axis == 1 ? N : (int64_t)N * N);
  const Tin* in = job.in + base;
  Tout* out = job.out + base;
  // along y and z at N = 256 the CTA's lines go through shared memory
  constexpr bool STAGED = L::STAGED;
  T* tile = reinterpret_cast<T*>(twr + N);
  auto tp = [&](int i) { return tile + tile_at<L::COLS>(i, 2 * t); };   // element i of the pair
  if constexpr (STAGED) {
    if (axis != 0) {
      tile_load<N, L::COLS, L::THREADS>(tile, in - 2 * t, es);
      __syncthreads();
    }
  }
  const auto X = slots<N>(t);
  constexpr T half = T(0.5), r2 = T(1.41421356237309504880), ir2 = T(0.70710678118654752440);
  // the lane's modes (k, N - k), k = k1(i); slot (0, N/2) for k = 0
  auto k1 = [&](int i) { return plane::pair_index<N>(i, m); };
  auto k2 = [&](int i) { return (i == 0 && m == 0) ? N / 2 : N - k1(i); };
  auto mode = [&](int k) { return dst ? N - 1 - k : k; };   // array index of DCT index k (F2, I2)
  constexpr bool fused = OP == OP_F2I2 || OP == OP_F1I1 || OP == OP_F1I2;

  // ---- the steps of a pass; A, B: modes (k, N - k) of the two lines
  auto load2 = [&](C2<T>(&v)[R]) {   // both lines, Makhoul's order
    if (axis == 0) {
#pragma unroll
      for (int r = 0; r < H; ++r) {
        const int n = m + M * r;
        const C2<T> a = ld2<T>(in + 2 * n, vec), b = ld2<T>(in + N + 2 * n, vec);
        v[r] = {a.x, b.x};
        // element 2n + 1 is position N - 1 - n: lane M - 1 - m, register R - 1 - r
        v[R - 1 - r] = {flip(__shfl_xor_sync(0xffffffffu, a.y, M - 1), dst),
                        flip(__shfl_xor_sync(0xffffffffu, b.y, M - 1), dst)};
      }
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int n = m + M * r;
        const int i = r < H ? 2 * n : 2 * (N - 1 - n) + 1;
        if constexpr (STAGED) v[r] = plane::ldc(reinterpret_cast<const C2<T>*>(tp(i)));
        else v[r] = ld2<T>(in + (int64_t)i * es, vec);
        if (r >= H) v[r] = {flip(v[r].x, dst), flip(v[r].y, dst)};
      }
    }
  };
  auto load1 = [&](C2<T>(&v)[R], int ab) {   // one line, packed odd extension
    const Tin* x = in + ab * ls;
    // z_n = x_2n + i x_(2n+1) (x_0 is the wall: 0), z_(N-n) = -x_2n - i x_(2n-1)
#pragma unroll
    for (int r = 0; r < H; ++r) {
      const int n = m + M * r;
      C2<T> a;
      if (axis == 0) a = ld2<T>(x + 2 * n, vec);
      else if (STAGED) a = {tp(2 * n)[ab], tp(2 * n + 1)[ab]};
      else a = {to_work<T>(x[(int64_t)(2 * n) * es]), to_work<T>(x[(int64_t)(2 * n + 1) * es])};
      if (r == 0 && m == 0) a.x = T(0);
      v[r] = a;
    }
#pragma unroll
    for (int r = 0; r < H; ++r) {
      // position n = m + M (R - 1 - r): x_2n' of n' = N - n at lane M - m, register r (lane 0:
      // register r + 1, zero for n' = N/2), x_(2n'-1) at lane M - 1 - m, register r
      const T nx = r + 1 < H ? v[r + 1].x : T(0);
      const T re = __shfl_sync(0xffffffffu, m ? v[r].x : nx, partner);
      const T im = __shfl_xor_sync(0xffffffffu, v[r].y, M - 1);
      v[R - 1 - r] = {-re, -im};
    }
  };
  auto modes2 = [&](int k, bool self, C2<T> z, C2<T> g, C2<T>& A, C2<T>& B) {
    const C2<T> q0 = qg[k];
    const C2<T> q = {half * q0.x, half * q0.y};
    C2<T> a = cmul(q, C2<T>{z.x + g.x, z.y - g.y}), b = cmul(q, C2<T>{z.y + g.y, g.x - z.x});
    if (self) {
      a = {z.x, -(ir2 * g.x)};
      b = {z.y, -(ir2 * g.y)};
    }
    A = {a.x, -a.y};   // X_k, X_(N-k)
    B = {b.x, -b.y};
  };
  auto modes1 = [&](int k, bool self, C2<T> z, C2<T> g) {
    const C2<T> w = twg[k];
    // four times Im a and Re(w b) over two: a = (.., z.y - g.y), b = (z.x - g.x, z.y + g.y)
    const T ia = T(0.25) * (z.y - g.y), wb = T(0.25) * (w.x * (z.x - g.x) - w.y * (z.y + g.y));
    C2<T> f = {wb - ia, wb + ia};
    if (self) f = {T(0), half * g.y};   // modes 0 and N/2
    return f;
  };
  // the inverse FFT's input, conjugated: conj Z_k = q conj(a + i b), conj Z_(N-k) = conj(q) (a - i b)
  // with a = X_k - i X_(N-k) of line A, b of line B
  auto back2 = [&](int k, bool self, C2<T> A, C2<T> B, C2<T>& lo, C2<T>& hi) {
    const C2<T> a = {A.x, -A.y}, b = {B.x, -B.y}, q = qg[k];
    lo = cmul(q, C2<T>{a.x - b.y, -(a.y + b.x)});
    hi = cmul(plane::conjg(q), C2<T>{a.x + b.y, a.y - b.x});
    if (self) {
      lo = {a.x, -b.x};
      hi = {r2 * A.y, -(r2 * B.y)};
    }
  };
  auto back1 = [&](int k, bool self, C2<T> f, C2<T>& lo, C2<T>& hi) {
    const C2<T> w = twg[k];   // exp(-i pi k / N)
    const T s = f.x + f.y, d = f.y - f.x, cs = w.x * s, ss = -(w.y * s);
    lo = {cs, -(ss + d)};
    hi = {-cs, d - ss};
    if (self) {
      lo = {T(0), T(0)};
      hi = {T(0), T(-2) * f.y};
    }
  };
  // weights of line ln
  auto weights = [&](int ln) {
    Weights<T, N> w;
    w.s2 = s2;
    w.sc = scales;
    w.wmode = job.wmode;
    w.own = job.wc == axis;
    w.kind = w.own ? 0 : 1;
    // the two other axes' mode indices and their kinds (component axis 0, else 1)
    const int hi = ln / N, lo = ln % N;
    const int ax1 = axis == 0 ? 1 : 0, ax2 = axis == 2 ? 1 : 2;   // lo runs along ax1, hi along ax2
    const T v1 = s2[(job.wc == ax1 ? 0 : 1) * N + lo], v2 = s2[(job.wc == ax2 ? 0 : 1) * N + hi];
    w.rest = v1 + v2;
    w.num = w.own ? T(0) : (job.wc == ax1 ? w.numer(v1, lo == 0) : w.numer(v2, hi == 0));
    return w;
  };
  // a mode pair (array indices ka, kb) times its weights, the reciprocals correctly rounded.
  // FP64: one reciprocal of the product of the two denominators is 1 % of an FP64 matvec
  // faster and adds 3 % to the error of a Poisson solve (N = 64: 5.96e-16 against 5.80e-16)
  auto weigh = [&](const Weights<T, N>& W, int ka, int kb, C2<T>& f) {
    T d1, d2;
    const T n1 = W.at(ka, d1), n2 = W.at(kb, d2);
    if constexpr (sizeof(T) == 4) f = {f.x * (n1 * __frcp_rn(d1)), f.y * (n2 * __frcp_rn(d2))};
    else f = {f.x * (n1 * __drcp_rn(d1)), f.y * (n2 * __drcp_rn(d2))};
  };
  auto store2 = [&](const C2<T>(&v)[R]) {
    // v holds the conjugate: line A in the real, minus line B in the imaginary part; element
    // 2n here, element 2n + 1 at position N - 1 - n
    const T sc = T(1) / T(N);
    const bool neg = OP != OP_F1I2 && dst;
    const bool weighted = OP == OP_I2 && job.wmode != W_NONE;
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int n = m + M * j;
      // along x the odd element comes from the mirror lane: A and B of elements 2n, 2n + 1
      const int io = axis == 0 ? 2 * n + 1 : 2 * ((M - 1 - m) + M * j) + 1;
      C2<T> o = v[R - 1 - j];
      if (axis == 0) o = {__shfl_xor_sync(0xffffffffu, o.x, M - 1), __shfl_xor_sync(0xffffffffu, o.y, M - 1)};
      C2<T> fa = {sc * v[j].x, flip(sc * o.x, neg)}, fb = {-(sc * v[j].y), flip(sc * o.y, !neg)};
      if (weighted) {
        weigh(weights(line), 2 * n, io, fa);
        weigh(weights(line + 1), 2 * n, io, fb);
      }
      if (axis == 0) {
        st2<T>(out + 2 * n, fa.x, fa.y, vec, acc);
        st2<T>(out + N + 2 * n, fb.x, fb.y, vec, acc);
      } else if constexpr (STAGED) {
        plane::stc(reinterpret_cast<C2<T>*>(tp(2 * n)), C2<T>{fa.x, fb.x});
        plane::stc(reinterpret_cast<C2<T>*>(tp(io)), C2<T>{fa.y, fb.y});
      } else {
        st2<T>(out + (int64_t)(2 * n) * es, fa.x, fb.x, vec, acc);
        st2<T>(out + (int64_t)io * es, fa.y, fb.y, vec, acc);
      }
    }
  };
  auto store1 = [&](const C2<T>(&v)[R], int ab) {
    Tout* x = out + ab * ls;
    const T sc = T(1) / T(N);
    const bool weighted = OP == OP_I1 && job.wmode != W_NONE;
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int n = m + M * j;
      C2<T> f = {sc * v[j].x, -(sc * v[j].y)};
      if (j == 0 && m == 0) f.x = T(0);
      if (weighted) weigh(weights(line + ab), 2 * n, 2 * n + 1, f);
      if (axis == 0) {
        st2<T>(x + 2 * n, f.x, f.y, vec);
      } else if (STAGED) {
        tp(2 * n)[ab] = f.x;
        tp(2 * n + 1)[ab] = f.y;
      } else {
        x[(int64_t)(2 * n) * es] = f.x;
        x[(int64_t)(2 * n + 1) * es] = f.y;
      }
    }
  };
  auto fwd_store = [&](int i, C2<T> a, C2<T> b, int ka, int kb) {   // modes of both lines to memory
    if (job.wmode != W_NONE) {
      weigh(weights(line), ka, kb, a);
      weigh(weights(line + 1), ka, kb, b);
    }
    if (axis == 0) {
      out[ka] = a.x;
      out[kb] = a.y;
      out[N + ka] = b.x;
      out[N + kb] = b.y;
    } else if constexpr (STAGED) {
      plane::stc(reinterpret_cast<C2<T>*>(tp(ka)), C2<T>{a.x, b.x});
      plane::stc(reinterpret_cast<C2<T>*>(tp(kb)), C2<T>{a.y, b.y});
    } else {
      st2<T>(out + (int64_t)ka * es, a.x, b.x, vec);
      st2<T>(out + (int64_t)kb * es, a.y, b.y, vec);
    }
  };
  auto load_modes = [&](int ka, int kb, C2<T>& a, C2<T>& b) {
    if (axis == 0) {
      a = {to_work<T>(in[ka]), to_work<T>(in[kb])};
      b = {to_work<T>(in[N + ka]), to_work<T>(in[N + kb])};
    } else {
      C2<T> e, f;
      if constexpr (STAGED) {
        e = plane::ldc(reinterpret_cast<const C2<T>*>(tp(ka)));
        f = plane::ldc(reinterpret_cast<const C2<T>*>(tp(kb)));
      } else {
        e = ld2<T>(in + (int64_t)ka * es, vec);
        f = ld2<T>(in + (int64_t)kb * es, vec);
      }
      a = {e.x, f.x};
      b = {e.y, f.y};
    }
  };

  // ---- the passes
  C2<T> v[R];
  if constexpr (OP == OP_F2) {
    load2(v);
    plane::fft_to_pairs<N, T>(v, P, X, tws, m);
    plane::for_pairs<N, true, false>(v, m, partner, [&](int i, int k, bool self, C2<T> z, C2<T> g) {
      C2<T> A, B;
      modes2(k, self, z, g, A, B);
      fwd_store(i, A, B, mode(k), mode(self ? N / 2 : N - k));
    });
  } else if constexpr (OP == OP_F2I2) {
    load2(v);
    plane::fft_to_pairs<N, T>(v, P, X, tws, m);
    const Weights<T, N> WA = weights(line), WB = weights(line + 1);
    plane::for_pairs<N, true, true>(v, m, partner, [&](int, int k, bool self, C2<T>& z, C2<T>& g) {
      C2<T> A, B;
      modes2(k, self, z, g, A, B);
      const int ka = mode(k), kb = mode(self ? N / 2 : N - k);
      weigh(WA, ka, kb, A);
      weigh(WB, ka, kb, B);
      back2(k, self, A, B, z, g);
    });
    plane::fft_from_pairs<N, T>(v, P, X, tws, twr, m);
    store2(v);
  } else if constexpr (OP == OP_I2) {
    C2<T> A[H], B[H];   // every mode is read before any output is written (in place)
#pragma unroll
    for (int i = 0; i < H; ++i) load_modes(mode(k1(i)), mode(k2(i)), A[i], B[i]);
    plane::for_pairs<N, false, true>(v, m, partner, [&](int i, int k, bool self, C2<T>& lo, C2<T>& hi) {
      back2(k, self, A[i], B[i], lo, hi);
    });
    plane::fft_from_pairs<N, T>(v, P, X, tws, twr, m);
    store2(v);
  } else if constexpr (OP == OP_F1I1) {
#pragma unroll 1
    for (int ab = 0; ab < 2; ++ab) {
      load1(v, ab);
      plane::fft_to_pairs<N, T>(v, P, X, tws, m);
      const Weights<T, N> W = weights(line + ab);
      plane::for_pairs<N, true, true>(v, m, partner, [&](int, int k, bool self, C2<T>& z, C2<T>& g) {
        C2<T> f = modes1(k, self, z, g);
        weigh(W, k, self ? N / 2 : N - k, f);
        back1(k, self, f, z, g);
      });
      plane::fft_from_pairs<N, T>(v, P, X, tws, twr, m);
      store1(v, ab);
    }
  } else {
    // A, B: the lines' modes, the first line's moving on to A when the second's arrive in B
    C2<T> A[H], B[H];
    if constexpr (OP == OP_I1) {
#pragma unroll
      for (int i = 0; i < H; ++i) {
        load_modes(k1(i), k2(i), A[i], B[i]);
        if (i == 0 && m == 0) A[i].x = B[i].x = T(0);   // DST-I has no mode 0
      }
    } else {
#pragma unroll
      for (int i = 0; i < H; ++i) B[i] = {T(0), T(0)};
#pragma unroll 1
      for (int ab = 0; ab < 2; ++ab) {
        load1(v, ab);
        plane::fft_to_pairs<N, T>(v, P, X, tws, m);
        plane::for_pairs<N, true, false>(v, m, partner, [&](int i, int k, bool self, C2<T> z, C2<T> g) {
          A[i] = B[i];
          B[i] = modes1(k, self, z, g);
        });
      }
    }
    if constexpr (OP == OP_F1) {
#pragma unroll
      for (int i = 0; i < H; ++i) fwd_store(i, A[i], B[i], k1(i), k2(i));
    } else if constexpr (OP == OP_F1I2) {
      const Weights<T, N> WA = weights(line), WB = weights(line + 1);
      plane::for_pairs<N, false, true>(v, m, partner, [&](int i, int k, bool self, C2<T>& lo, C2<T>& hi) {
        const int kb = self ? N / 2 : N - k;
        weigh(WA, k, kb, A[i]);
        weigh(WB, k, kb, B[i]);
        back2(k, self, A[i], B[i], lo, hi);
      });
      plane::fft_from_pairs<N, T>(v, P, X, tws, twr, m);
      store2(v);
    } else {
      static_assert(OP == OP_I1, "the seven operations");
#pragma unroll 1
      for (int ab = 0; ab < 2; ++ab) {
        plane::for_pairs<N, false, true>(v, m, partner, [&](int i, int k, bool self, C2<T>& lo, C2<T>& hi) {
          back1(k, self, A[i], lo, hi);
          A[i] = B[i];
        });
        plane::fft_from_pairs<N, T>(v, P, X, tws, twr, m);
        store1(v, ab);
      }
    }
  }
  if constexpr (STAGED) {
    if (axis != 0) {
      __syncthreads();
      tile_store<N, L::COLS, L::THREADS>(tile, out - 2 * t, es, acc);
    }
  }
}

}  // namespace lines
}  // namespace kfbim
