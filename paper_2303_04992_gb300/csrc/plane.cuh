// The (x, y) part of one spectral term of the Schur operator on one plane:
// (X_x Y_y)^-1 L (X_x Y_y) applied to an N x N plane of a field already
// transformed along z, one CTA per (term, plane).
//
// The plane never leaves the chip between the four axis transforms and no
// real transform is formed: with v the line in Makhoul's order (v_n = x_2n,
// v_(N-1-n) = x_(2n+1)) and V its complex FFT, q_k V_k = X_k - i X_(N-k) with
// q_k = exp(-i pi k / 2N) holds the DCT-II modes k and N-k, so the modes along
// x of one row are N/2 complex numbers, and the N/2 complex lines along y that
// they form (line l: x modes l and N-l; line 0: the two real modes 0 and N/2)
// go straight into the next FFT.  A DST-II is a DCT-II of the line with the
// second half of Makhoul's order negated, its mode a at DCT index N-1-a.
// Along y the transform, the weight and the inverse transform are
// one step in the FFT's registers: with w_k the weight at DCT index k,
//   V'_k = s_k V_k + t_k exp(i pi k / N) V_(N-k),  s, t = (w_k +- w_(N-k)) / 2
// for a real line, and for the two real lines A, B of a complex one
//   Z'_k = s Z_k + ds P* + c (t P + dt Z*),  P = Z_(N-k), c = exp(i pi k / N),
// with s = (s_A + s_B) / 2, ds = (s_A - s_B) / 2 and t, dt alike.  Where a lane
// holds several residues of the index, Z_k and Z_(N-k) lie in the same lane.
//
// Shared memory: N/2 lines of N complex numbers, element n of line l at
// l N + (n ^ line_sw(l)).  A team of M lanes computes one FFT, R = N / M values
// per lane: DFT_R in registers, a twiddle, an exchange in place (along x in the
// team's own two columns of the plane, along y in its own line), R / M
// DFT_M per lane.  The swizzle makes the exchange along x (M/2 lines x two
// columns x the teams of a half warp), the exchange along y (runs of M), the
// 16-byte column pairs (M lines) and the line accesses free of bank conflicts.
//
// What bounds it (N = 128, 384 CTAs, FP32): instruction issue (59 % of the slots
// of the average SM, the busiest of the 152 holds three of the 384 CTAs) and the
// shared-memory pipe (51 %); 16.5 M warp instructions against 37.5 M for a kernel
// that formed every real transform and transposed the plane between the axes.
// Between events, which add about 3 us: 25.3 us for the three terms at N = 128 (that
// kernel: 56.6), 9.5 at N = 64 (about 30), 7.2 at N = 32 (27), 13.4 at N = 96 (five
// one-axis passes there: 133).  Of that the pair-blocked order of the planes gave 2.1 at
// N = 128, index pairs within a lane instead of shuffles 2.0 (at N = 96 as much), a copy
// of the code per term cost 2 (the warps waited for instructions), and 80 registers with
// three resident CTAs ran as fast as 128 with two.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "transforms.cuh"
#include "transforms2.cuh"

namespace kfbim {
namespace plane {

// Orders of the fields.  Along each axis position n is Makhoul's.  A plane
// (the positions of one z) is stored as [y / YB][x][y mod YB]: a warp's YB / 2 row
// pairs at M consecutive x are one contiguous run of 64 numbers.
template <int N>
struct Shape {
  static constexpr int R = N >= 128 ? 16 : (N == 96 ? 24 : 8);   // values per lane
  static constexpr int M = N / R;                                // lanes per FFT
  static constexpr int NS = R / M;                               // DFT_M per lane
  static constexpr int H = R / 2;
  static constexpr int LINES = N / 2;
  // CTAs per plane: the 256 KB of a plane at N = 256 take the four CTAs of a
  // cluster, each with a quarter of the lines and of the row pairs and the others'
  // lines through distributed shared memory (two CTAs fit a plane as well, but only
  // one of them an SM, where nothing then runs during its waits)
  static constexpr int CL = N == 256 ? 4 : 1;
  static constexpr int LL = LINES / CL;                          // lines and row pairs per CTA
  static constexpr int ROUNDS = N >= 128 ? 2 : 1;                // FFTs per team and axis step
  static constexpr int TEAMS = LL / ROUNDS;
  static constexpr int THREADS = TEAMS * M;                      // N = 256: 256; 256, 192, 256, 64
  static constexpr int YB = 2 * (32 / M);                        // y positions of one warp's row pairs
  static_assert(R % M == 0, "four-step split");
};

// A complex number as one 8- or 16-byte access.
template <typename T>
__device__ __forceinline__ C2<T> ldc(const C2<T>* p) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    return {v.x, v.y};
  } else {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return {v.x, v.y};
  }
}
template <typename T>
__device__ __forceinline__ void stc(C2<T>* p, C2<T> v) {
  if constexpr (sizeof(T) == 4) *reinterpret_cast<float2*>(p) = make_float2(v.x, v.y);
  else *reinterpret_cast<double2*>(p) = make_double2(v.x, v.y);
}
template <typename T>
__device__ __forceinline__ C2<T> conjg(C2<T> a) { return {a.x, -a.y}; }
// Complex sum and difference: FP32 as one packed instruction (the same
// pipe time as two scalar ones, half the issue slots; a - b as b (-1) + a,
// which is exact in the product).
template <typename T>
__device__ __forceinline__ C2<T> cadd(C2<T> a, C2<T> b) {
  if constexpr (sizeof(T) == 4) {
    const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    return {r.x, r.y};
  } else {
    return {a.x + b.x, a.y + b.y};
  }
}
template <typename T>
__device__ __forceinline__ C2<T> csub(C2<T> a, C2<T> b) {
  if constexpr (sizeof(T) == 4) {
    const float2 r = __ffma2_rn(make_float2(b.x, b.y), make_float2(-1.f, -1.f), make_float2(a.x, a.y));
    return {r.x, r.y};
  } else {
    return {a.x - b.x, a.y - b.y};
  }
}
// a s, packed
__device__ __forceinline__ C2<float> cscale(C2<float> a, float s) {
  const float2 r = __fmul2_rn(make_float2(a.x, a.y), make_float2(s, s));
  return {r.x, r.y};
}

// b exp(-2 pi i j / L) for a compile-time j (forward twiddles): quarter turns
// are swaps and eighth turns one scaling, neither a full product.
template <int L, typename T>
__device__ __forceinline__ C2<T> rot(C2<T> b, int j) {
  constexpr double s8 = 0.70710678118654752440;
  if (j == 0) return b;
  if (4 * j == L) return {b.y, -b.x};
  if (8 * j == L) return {T(s8) * (b.x + b.y), T(s8) * (b.y - b.x)};
  if (8 * j == 3 * L) return {T(s8) * (b.y - b.x), T(-s8) * (b.x + b.y)};
  const T c = L == 24 ? T(cos24(j)) : T(cos16(j * (16 / L)));
  const T s = L == 24 ? T(sin24(j)) : T(sin16(j * (16 / L)));
  return {c * b.x + s * b.y, c * b.y - s * b.x};
}

template <typename T>
__device__ __forceinline__ void dft4(C2<T>& a, C2<T>& b, C2<T>& c, C2<T>& d) {
  const C2<T> s0 = cadd(a, c), d0 = csub(a, c), s1 = cadd(b, d), d1 = csub(b, d);
  a = cadd(s0, s1);
  c = csub(s0, s1);
  b = {d0.x + d1.y, d0.y - d1.x};
  d = {d0.x - d1.y, d0.y + d1.x};
}

// Forward DFT of L = 4, 8, 16 or 24 points in registers, natural order in and
// out, as radix-4 steps (radix 2 for the last of 8, radix 3 first for 24).
template <int L, typename T>
__device__ __forceinline__ void dft(C2<T>* v) {
  if constexpr (L == 4) {
    dft4(v[0], v[1], v[2], v[3]);
  } else if constexpr (L == 8) {
    // n = 2 n1 + n2: two DFT4 over n1, twiddle, radix 2 over n2
    dft4(v[0], v[2], v[4], v[6]);
    dft4(v[1], v[3], v[5], v[7]);
    C2<T> o[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const C2<T> t = rot<8>(v[2 * k + 1], k);
      o[k] = cadd(v[2 * k], t);
      o[k + 4] = csub(v[2 * k], t);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = o[k];
  } else if constexpr (L == 16) {
    // n = 4 n1 + n2: DFT4 over n1, twiddle, DFT4 over n2
    C2<T> o[16];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      C2<T> a = v[4 * k1], b = rot<16>(v[4 * k1 + 1], k1), c = rot<16>(v[4 * k1 + 2], 2 * k1),
            d = v[4 * k1 + 3];
      // exp(-2 pi i 9 / 16) = -exp(-2 pi i / 16)
      if (k1 == 3) {
        d = rot<16>(d, 1);
        d = {-d.x, -d.y};
      } else {
        d = rot<16>(d, 3 * k1);
      }
      dft4(a, b, c, d);
      o[k1] = a;
      o[k1 + 4] = b;
      o[k1 + 8] = c;
      o[k1 + 12] = d;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = o[k];
  } else {
    static_assert(L == 24, "4, 8, 16 or 24 points");
    // n = 8 n1 + n2: DFT3 over n1, twiddle, DFT8 over n2
    const T h = T(0.86602540378443864676);   // sin 60 degrees
    C2<T> a[3][8];
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) {
      const C2<T> x0 = v[n2], s = cadd(v[8 + n2], v[16 + n2]), d = csub(v[8 + n2], v[16 + n2]);
      a[0][n2] = cadd(x0, s);
      const C2<T> m = {x0.x - T(0.5) * s.x, x0.y - T(0.5) * s.y};
      a[1][n2] = rot<24>(C2<T>{m.x + h * d.y, m.y - h * d.x}, n2);
      a[2][n2] = rot<24>(C2<T>{m.x - h * d.y, m.y + h * d.x}, 2 * n2);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      dft<8>(a[k1]);
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) v[k1 + 3 * k2] = a[k1][k2];
    }
  }
}

// ------------------------------------------------------------ addressing
// Swizzle of line l (complex units, added by XOR to the position in the line;
// within aligned groups of 16).  Teams of 8 lanes: a half warp is two teams,
// which need lines 0..3 (times two columns) on distinct 16-byte pairs and
// lines 0..7 of a column pair on distinct 16-byte units.  Teams of 4: four
// teams, lines 0 and 1 of an exchange, lines 0..3 of a column pair.
template <int M>
__device__ __forceinline__ int line_sw(int l) {
  if constexpr (M == 16) return (l & 7) << 1;   // a half warp is one team: 8 lines of a column pair
  else if constexpr (M == 8) return ((l & 3) << 2) | ((l >> 1) & 2);
  else return ((l & 1) << 3) | ((l & 2) << 1);
}

// Exchange slot of logical index c = s M + v (v < M), of the team: along x slots
// are the two columns 2p, 2p+1 of lines c / 2, along y the positions of the
// team's line.  Index c is stored at s M + (v ^ (s mod M)).
template <int N>
struct XSlots {   // along x
  using S = Shape<N>;
  int col;   // 2p
  __device__ __forceinline__ int at(int s, int v) const {
    const int w = v ^ (s & (S::M - 1));
    const int line = s * (S::M / 2) + (w >> 1);
    return line * N + ((col + (w & 1)) ^ line_sw<S::M>(line));
  }
};
template <int N>
struct XScratch {   // along x on a cluster, whose CTAs' columns are not whole: a buffer of the team
  using S = Shape<N>;
  int base;
  __device__ __forceinline__ int at(int s, int v) const { return base + s * S::M + (v ^ (s & (S::M - 1))); }
};
template <int N>
struct YSlots {   // along y
  using S = Shape<N>;
  int base, sw;   // line * N and its swizzle
  __device__ __forceinline__ int at(int s, int v) const {
    return base + ((s * S::M + (v ^ (s & (S::M - 1)))) ^ sw);
  }
};

// Forward complex FFT of length N by a team: lane m holds z[m + M r] in v[r] on
// entry and Z[m + M j] in v[j] on return.  tws[s M + m] = exp(-2 pi i m s / N).
// The exchange slots hold nothing the team still needs on entry.
template <int N, typename T, class Slots>
__device__ __forceinline__ void team_fft(C2<T> (&v)[Shape<N>::R], C2<T>* P, const Slots& X, const C2<T>* tws,
                                         int m) {
  using S = Shape<N>;
  constexpr int M = S::M, R = S::R, NS = S::NS;
  dft<R>(v);
  __syncwarp();   // the team has read its inputs from the slots
#pragma unroll
  for (int s = 0; s < R; ++s) {
    C2<T> y = v[s];
    if (s != 0) y = cmul(y, ldc(tws + s * M + m));
    stc(P + X.at(s, m), y);
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    C2<T> w[M];
#pragma unroll
    for (int k = 0; k < M; ++k) w[k] = ldc(P + X.at(q * M + m, k));
    dft<M>(w);
    // Z[s + R k], s = q M + m, i.e. index j = q + NS k of m + M j
#pragma unroll
    for (int k = 0; k < M; ++k) v[q + NS * k] = w[k];
  }
  __syncwarp();   // the slots may be written again
}

// The upper half of a team's FFT indices by lane pairs: for k = m + M j < N/2,
// mirror_fetch returns the value at index N - k (for k = 0: at N/2) out of the
// registers v[j] (index m + M j).  mirror_put stores values g[j] that the partner
// lane made for its indices N - k into the upper registers v[H..R-1].
template <int N, typename T>
__device__ __forceinline__ C2<T> mirror_fetch(const C2<T> (&v)[Shape<N>::R], int j, int m, int partner) {
  using S = Shape<N>;
  const C2<T> a = v[S::R - 1 - j], b = j ? v[S::R - j] : v[S::H];
  const C2<T> snd = m ? a : b;
  return {__shfl_sync(0xffffffffu, snd.x, partner), __shfl_sync(0xffffffffu, snd.y, partner)};
}
template <int N, typename T>
__device__ __forceinline__ void mirror_put(C2<T> (&v)[Shape<N>::R], const C2<T> (&g)[Shape<N>::H], int m) {
  using S = Shape<N>;
#pragma unroll
  for (int r = S::H; r < S::R; ++r) {
    const C2<T> a = g[S::R - 1 - r], b = g[(S::R - r) % S::H];
    v[r] = m ? a : b;
  }
}

// ------------------------------------------------------- mode pairs (k, N - k)
// The transforms of real lines need FFT indices k and N - k together.  Where a
// lane does an even number of DFT_M (NS), it takes residues s and R - s of the
// index k = s + R k', so that every pair lies in one lane's registers and no
// shuffle is needed: group g holds Z[s + R k'] in v[2 M g + k'] and Z[s' + R k'] in
// v[2 M g + M + k'], s = g M + m, s' = R - s (lane 0, group 0: s = 0 and s' = R/2,
// their own mirrors; pair_swap then puts each index's mirror where the other
// lanes have it).  The inverse FFT starts from that layout with the DFT_M and
// ends with the DFT_R, at index m + M j.  Where NS is odd, the natural layout and
// shuffles between lanes m and M - m.
template <int N>
struct PairShape {
  using S = Shape<N>;
  static constexpr bool in_lane = S::NS % 2 == 0;
  __device__ __forceinline__ static int s0(int g, int m) { return g * S::M + m; }
  __device__ __forceinline__ static int s1(int g, int m) { return g == 0 && m == 0 ? S::R / 2 : S::R - g * S::M - m; }
};
// Lane 0, group 0, of in-lane pairs: a[k'] = Z[R k'], b[k'] = Z[R/2 + R k'].
// Forward: upper half of a <- upper half of b; b[M-1-j] <- a[M-j], b[M-1] <- a[M/2].
template <int M, typename T>
__device__ __forceinline__ void pair_swap(C2<T>* a, C2<T>* b, bool lane0, bool back) {
  C2<T> na[M / 2], nb[M / 2];
#pragma unroll
  for (int i = 0; i < M / 2; ++i) {
    const int u = M / 2 + i;
    if (!back) {
      na[i] = b[u];
      nb[i] = u + 1 < M ? a[u + 1] : a[M / 2];
    } else {
      na[i] = u == M / 2 ? b[M - 1] : b[u - 1];
      nb[i] = a[u];
    }
  }
#pragma unroll
  for (int i = 0; i < M / 2; ++i) {
    const int u = M / 2 + i;
    a[u] = {lane0 ? na[i].x : a[u].x, lane0 ? na[i].y : a[u].y};
    b[u] = {lane0 ? nb[i].x : b[u].x, lane0 ? nb[i].y : b[u].y};
  }
}

// Forward FFT, z[m + M r] in v[r] -> the pair layout.
template <int N, typename T, class Slots>
__device__ __forceinline__ void fft_to_pairs(C2<T> (&v)[Shape<N>::R], C2<T>* P, const Slots& X, const C2<T>* tws,
                                             int m) {
  using S = Shape<N>;
  constexpr int M = S::M, R = S::R;
  if constexpr (!PairShape<N>::in_lane) {
    team_fft<N, T>(v, P, X, tws, m);
  } else {
    dft<R>(v);
    __syncwarp();
#pragma unroll
    for (int s = 0; s < R; ++s) {
      C2<T> y = v[s];
      if (s != 0) y = cmul(y, ldc(tws + s * M + m));
      stc(P + X.at(s, m), y);
    }
    __syncwarp();
#pragma unroll
    for (int g = 0; g < S::NS / 2; ++g) {
      const int s0 = PairShape<N>::s0(g, m), s1 = PairShape<N>::s1(g, m);
      C2<T>* a = v + 2 * M * g;
      C2<T>* b = a + M;
#pragma unroll
      for (int k = 0; k < M; ++k) {
        a[k] = ldc(P + X.at(s0, k));
        b[k] = ldc(P + X.at(s1, k));
      }
      dft<M>(a);
      dft<M>(b);
      if (g == 0) pair_swap<M>(a, b, m == 0, false);
    }
    __syncwarp();
  }
}
// Forward FFT from the pair layout -> index m + M j in v[j].  twr[k R + s] =
// exp(-2 pi i k s / N).
template <int N, typename T, class Slots>
__device__ __forceinline__ void fft_from_pairs(C2<T> (&v)[Shape<N>::R], C2<T>* P, const Slots& X, const C2<T>* tws,
                                               const C2<T>* twr, int m) {
  using S = Shape<N>;
  constexpr int M = S::M, R = S::R;
  if constexpr (!PairShape<N>::in_lane) {
    team_fft<N, T>(v, P, X, tws, m);
  } else {
    __syncwarp();
#pragma unroll
    for (int g = 0; g < S::NS / 2; ++g) {
      const int s0 = PairShape<N>::s0(g, m), s1 = PairShape<N>::s1(g, m);
      C2<T>* a = v + 2 * M * g;
      C2<T>* b = a + M;
      if (g == 0) pair_swap<M>(a, b, m == 0, true);
      dft<M>(a);
      dft<M>(b);
#pragma unroll
      for (int k = 0; k < M; ++k) {
        C2<T> x = a[k], y = b[k];
        if (k != 0) {
          x = cmul(x, ldc(twr + k * R + s0));
          y = cmul(y, ldc(twr + k * R + s1));
        }
        stc(P + X.at(s0, k), x);
        stc(P + X.at(s1, k), y);
      }
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < R; ++s) v[s] = ldc(P + X.at(s, m));
    __syncwarp();
    dft<R>(v);
  }
}
// The lane's i-th index k < N/2 in the order of for_pairs, i < H.
template <int N>
__device__ __forceinline__ int pair_index(int i, int m) {
  using S = Shape<N>;
  if constexpr (PairShape<N>::in_lane) {
    const int g = i / S::M, j = i % S::M;
    return (j % 2 ? PairShape<N>::s1(g, m) : PairShape<N>::s0(g, m)) + S::R * (j / 2);
  } else {
    return m + S::M * i;
  }
}
// f(i, k, self, Z_k, Z_(N-k)) for the lane's indices k < N/2; self: k = 0, with
// Z_(N/2) in the place of Z_(N-k).  READ: the values come from v; WRITE: those
// that f leaves go back to v.
template <int N, bool READ, bool WRITE, typename T, class F>
__device__ __forceinline__ void for_pairs(C2<T> (&v)[Shape<N>::R], int m, int partner, F&& f) {
  using S = Shape<N>;
  constexpr int M = S::M, R = S::R, H = S::H;
  if constexpr (PairShape<N>::in_lane) {
#pragma unroll
    for (int g = 0; g < S::NS / 2; ++g) {
      const int s0 = PairShape<N>::s0(g, m), s1 = PairShape<N>::s1(g, m);
      C2<T>* a = v + 2 * M * g;
      C2<T>* b = a + M;
#pragma unroll
      for (int j = 0; j < M / 2; ++j) {
        f(g * M + 2 * j, s0 + R * j, g == 0 && j == 0 && m == 0, a[j], b[M - 1 - j]);
        f(g * M + 2 * j + 1, s1 + R * j, false, b[j], a[M - 1 - j]);
      }
    }
  } else {
    C2<T> up[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      C2<T> z{}, g{};
      if constexpr (READ) {
        z = v[j];
        g = mirror_fetch<N, T>(v, j, m, partner);
      }
      f(j, m + M * j, j == 0 && m == 0, z, g);
      if constexpr (WRITE) {
        v[j] = z;
        up[j] = {__shfl_sync(0xffffffffu, g.x, partner), __shfl_sync(0xffffffffu, g.y, partner)};
      }
    }
    if constexpr (WRITE) mirror_put<N, T>(v, up, m);
  }
}

// 1 / d for a sum d of three 4 sin^2, in [1e-4, 12]: the hardware reciprocal (within 1 ulp)
__device__ __forceinline__ float rcp(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}

// One term of the Schur operator, uniform over a CTA.  The axis `term` takes
// DCT-II, the other two DST-II; the weight is 4 sin^2 of the DCT axis over the
// sum of the three, times 1 / (mu N^2).
struct Term {
  bool xs, ys;   // DST-II along x, y
  bool nx, ny;   // the weight's numerator is the x / the y (else the z) value
};
__device__ __forceinline__ Term term_of(int term) { return {term != 0, term != 1, term == 0, term == 1}; }

// Weights of one complex y line (real lines A and B: two x modes) at DCT index
// k < N/2 along y and its mirror N - k: s, ds, t, dt of the header comment.
// eX = ax + az; nX: the numerator's part that does not depend on y; cy: where the
// numerator is ay; both with a quarter of the weight's factor.  A reciprocal per
// weight: one for the product of two denominators is half a percent of a matvec
// faster and leaves the weights less exact; correctly rounded ones take 4 % longer
// and change nothing below.  The operator's error against 64 bits, relative in the
// 2-norm on white noise (mu = 0.7): 1.89e-7, 2.04e-7, 1.87e-7, 2.15e-7, 2.44e-7 at
// N = 32, 64, 96, 128, 256; real transforms with correctly rounded reciprocals, one
// axis at a time: 2.12e-7, 2.12e-7, 1.94e-7, 2.21e-7, 2.62e-7.
struct LineW {
  float eA, eB, nA, nB, cy;
  // ay, ay2: 4 sin^2 at k and N - k
  __device__ __forceinline__ void pair(float ay, float ay2, float& s, float& ds, float& t, float& dt) const {
    const float y1 = cy * ay, y2 = cy * ay2;
    // the weights (a quarter) of A and B at k and N - k
    const float u1 = (nA + y1) * rcp(eA + ay), u2 = (nA + y2) * rcp(eA + ay2);
    const float v1 = (nB + y1) * rcp(eB + ay), v2 = (nB + y2) * rcp(eB + ay2);
    const float sA = u1 + u2, sB = v1 + v2, tA = u1 - u2, tB = v1 - v2;
    s = sA + sB;
    ds = sA - sB;
    t = tA + tB;
    dt = tA - tB;
  }
  // the weights of A and B at an index that is its own mirror (k = 0 and N/2)
  __device__ __forceinline__ void self(float ay, float& wA, float& wB) const {
    wA = 4.f * (nA + cy * ay) * rcp(eA + ay);
    wB = 4.f * (nB + cy * ay) * rcp(eB + ay);
  }
};

template <int N>
struct Smem {
  using S = Shape<N>;
  static constexpr size_t scratch = S::CL > 1 ? sizeof(C2<float>) * S::TEAMS * N : 0;
  static constexpr size_t field = sizeof(C2<float>) * S::LL * N + scratch;
  static constexpr size_t tables = sizeof(C2<float>) * (2 * N + 2 * S::LINES) + sizeof(float) * S::LINES;
  static constexpr size_t bytes = field + tables;
};

// The tables of term_plane behind the field in shared memory.
// twg: exp(-pi i t / N), t < 2N; qg: exp(-pi i k / 2N); s2: 4 sin^2(pi a / 2N), a < N.
template <int N>
__device__ __forceinline__ void term_tables(C2<float>* P, const C2<float>* __restrict__ twg,
                                            const C2<float>* __restrict__ qg, const float* __restrict__ s2) {
  using S = Shape<N>;
  constexpr int M = S::M, R = S::R;
  C2<float>* tws = P + Smem<N>::field / sizeof(C2<float>);   // FFT twiddles [s][m]
  C2<float>* twr = tws + N;                 // the same by [m][s]
  C2<float>* qh = twr + N;                  // q_k / 2, k < N/2
  C2<float>* cy = qh + S::LINES;            // exp(i pi k / N), k < N/2
  float* sg = reinterpret_cast<float*>(cy + S::LINES);   // 4 sin^2(pi k / 2N), k < N/2
  for (int e = threadIdx.x; e < N; e += S::THREADS) {
    tws[e] = twg[2 * (e / M) * (e % M)];
    twr[e] = twg[2 * (e / R) * (e % R)];
  }
  for (int e = threadIdx.x; e < S::LINES; e += S::THREADS) {
    const C2<float> q = qg[e];
    qh[e] = {0.5f * q.x, 0.5f * q.y};
    cy[e] = conjg(twg[e]);
    sg[e] = s2[e];
  }
}

// One term on one plane: `in` and `out` are planes in the slab order (below;
// they may be the same).  Where an axis takes DST-II
// the field's odd nodes along it are negated in `in` and in `out`; `in` carries
// instead the signs of `signs` (so that two terms can share an input).
// az: the plane's 4 sin^2 along z; sc: 1 / (mu N^2).
// P: Smem<N>, its tables filled (term_tables; a barrier follows here).
// Called by all threads of the CTA (of every CTA of the cluster; rank: this one's).
template <int N>
__device__ __forceinline__ void term_plane(const float* in, float* out, const Term term, const Term signs, float az,
                                           float sc, C2<float>* P, int rank = 0) {
  using S = Shape<N>;
  constexpr int M = S::M, R = S::R, H = S::H;
  C2<float>* tws = P + Smem<N>::field / sizeof(C2<float>);   // FFT twiddles [s][m]
  C2<float>* twr = tws + N;                 // the same by [m][s]
  C2<float>* qh = twr + N;                  // q_k / 2, k < N/2
  C2<float>* cy = qh + S::LINES;            // exp(i pi k / N), k < N/2
  float* sg = reinterpret_cast<float*>(cy + S::LINES);   // 4 sin^2(pi k / 2N), k < N/2
  const int t = threadIdx.x / M, m = threadIdx.x % M;
  const int lane = threadIdx.x & 31;
  const int partner = (lane & ~(M - 1)) | ((M - m) & (M - 1));
  // the lines of CTA c of the cluster (all lines without one)
  C2<float>* lines[S::CL];
  if constexpr (S::CL > 1) {
#pragma unroll
    for (int c = 0; c < S::CL; ++c) lines[c] = cooperative_groups::this_cluster().map_shared_rank(P, c);
  } else {
    lines[0] = P;
  }
  auto sync = [] {
    if constexpr (S::CL > 1) cooperative_groups::this_cluster().sync();
    else __syncthreads();
  };
  // the column pair n0, n0 + 1 of line l, the lane's i-th index
  auto pair_at = [&](int i, int l, int n0) -> C2<float>* {
    static_assert(S::CL == 1 || !PairShape<N>::in_lane, "i gives the owner of line m + M i");
    if constexpr (S::CL > 1) return lines[M * i / S::LL] + ((l % S::LL) * N + (n0 ^ line_sw<M>(l)));
    else return P + (l * N + (n0 ^ line_sw<M>(l)));
  };
  C2<float> v[R];
  // ---- along x: the rows of Makhoul positions 2p, 2p + 1 along y -> columns 2p, 2p + 1
#pragma unroll 1
  for (int rd = 0; rd < S::ROUNDS; ++rd) {
    const int n0 = 2 * (rank * S::LL + t + S::TEAMS * rd);
    const C2<float>* ra =
        reinterpret_cast<const C2<float>*>(in + (int64_t)(n0 / S::YB) * (N * S::YB) + m * S::YB + n0 % S::YB);
    const float fl = (n0 >= N / 2 && term.ys != signs.ys) ? -1.f : 1.f, fh = term.xs != signs.xs ? -fl : fl;
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = cscale(ldc(ra + r * (M * S::YB / 2)), r < H ? fl : fh);
    if (rd == 0) sync();   // tables (and the others run before their lines are written)
    if constexpr (S::CL > 1) fft_to_pairs<N, float>(v, P, XScratch<N>{S::LL * N + t * N}, tws, m);
    else fft_to_pairs<N, float>(v, P, XSlots<N>{n0}, tws, m);
    for_pairs<N, true, false>(v, m, partner, [&](int i, int l, bool self, C2<float> z, C2<float> g) {
      const C2<float> q = ldc(qh + l);
      C2<float> a = cmul(q, C2<float>{z.x + g.x, z.y - g.y}), b = cmul(q, C2<float>{z.y + g.y, g.x - z.x});
      if (self) {   // the real modes 0 and N/2
        a = {z.x, g.x};
        b = {z.y, g.y};
      }
      C2<float>* at = pair_at(i, l, n0);   // the swizzle keeps pairs 2p, 2p + 1 together
      *reinterpret_cast<float4*>(at) = make_float4(a.x, a.y, b.x, b.y);
    });
  }
  sync();
  // ---- along y: transform, weight and inverse transform of line l in place
#pragma unroll 1
  for (int rd = 0; rd < S::ROUNDS; ++rd) {
    const int tt = t + S::TEAMS * rd;
    // the two teams of 8 lanes of a half warp take lines that differ in bit 1
    const int ll = M == 8 ? ((tt & ~3) | ((tt & 1) << 1) | ((tt >> 1) & 1)) : tt, l = rank * S::LL + ll;
    const YSlots<N> Y{ll * N, line_sw<M>(l)};
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ldc(P + (Y.base + ((m + M * r) ^ Y.sw)));
    fft_to_pairs<N, float>(v, P, Y, tws, m);
    // 4 sin^2 of the line's x modes l and N - l (line 0: 0 and N/2)
    const float sl = sg[l];
    const float axA = term.xs ? 4.f - sl : sl, axB = l ? (term.xs ? sl : 4.f - sl) : 2.f;
    LineW W;
    W.eA = axA + az;
    W.eB = axB + az;
    const float f = 0.5f * sc;   // twice a quarter: the inverse along x takes q / 2
    W.nA = f * (term.nx ? axA : (term.ny ? 0.f : az));
    W.nB = f * (term.nx ? axB : (term.ny ? 0.f : az));
    W.cy = term.ny ? f : 0.f;
    for_pairs<N, true, true>(v, m, partner, [&](int, int k, bool self, C2<float>& z, C2<float>& p) {
      const C2<float> c = ldc(cy + k);
      const float sk = sg[k], sm = 4.f - sk;
      float s, ds, tt2, dt;
      W.pair(term.ys ? sm : sk, term.ys ? sk : sm, s, ds, tt2, dt);
      // Z'_k = s Z + ds P* + c (t P + dt Z*), Z'_(N-k) = s P + ds Z* + c* (t Z + dt P*),
      // conjugated for the inverse by a forward FFT
      const C2<float> g = {tt2 * p.x + dt * z.x, tt2 * p.y - dt * z.y};
      const C2<float> h = {tt2 * z.x + dt * p.x, tt2 * z.y - dt * p.y};
      C2<float> lo = {s * z.x + ds * p.x + (c.x * g.x - c.y * g.y), ds * p.y - s * z.y - (c.x * g.y + c.y * g.x)};
      C2<float> hi = {s * p.x + ds * z.x + (c.x * h.x + c.y * h.y), ds * z.y - s * p.y - (c.x * h.y - c.y * h.x)};
      if (self) {   // indices 0 and N/2, each its own mirror
        float wA, wB;
        W.self(term.ys ? 4.f : 0.f, wA, wB);
        lo = {wA * z.x, -(wB * z.y)};
        W.self(2.f, wA, wB);
        hi = {wA * p.x, -(wB * p.y)};
      }
      z = lo;
      p = hi;
    });
    fft_from_pairs<N, float>(v, P, Y, tws, twr, m);
#pragma unroll
    for (int j = 0; j < R; ++j) stc(P + (Y.base + ((m + M * j) ^ Y.sw)), conjg(v[j]));
  }
  sync();
  // ---- along x back: columns 2p, 2p + 1 -> rows
#pragma unroll 1
  for (int rd = 0; rd < S::ROUNDS; ++rd) {
    const int n0 = 2 * (rank * S::LL + t + S::TEAMS * rd);
    // conj Z'_k = q conj(A + i B), conj Z'_(N-k) = conj(q) (A - i B)
    for_pairs<N, false, true>(v, m, partner, [&](int i, int l, bool self, C2<float>& lo, C2<float>& hi) {
      const C2<float>* at = pair_at(i, l, n0);
      const float4 f = *reinterpret_cast<const float4*>(at);
      const C2<float> a = {f.x, f.y}, b = {f.z, f.w};
      const C2<float> q = ldc(qh + l);
      lo = cmul(q, C2<float>{a.x - b.y, -(a.y + b.x)});
      hi = cmul(conjg(q), C2<float>{a.x + b.y, a.y - b.x});
      if (self) {
        lo = {0.5f * a.x, -0.5f * b.x};
        hi = {0.5f * a.y, -0.5f * b.y};
      }
    });
    if constexpr (S::CL > 1) fft_from_pairs<N, float>(v, P, XScratch<N>{S::LL * N + t * N}, tws, twr, m);
    else fft_from_pairs<N, float>(v, P, XSlots<N>{n0}, tws, twr, m);
    C2<float>* ra =
        reinterpret_cast<C2<float>*>(out + (int64_t)(n0 / S::YB) * (N * S::YB) + m * S::YB + n0 % S::YB);
#pragma unroll
    for (int j = 0; j < R; ++j) stc(ra + j * (M * S::YB / 2), conjg(v[j]));
  }
  if constexpr (S::CL > 1) sync();   // the others may still read this CTA's lines
}

}  // namespace plane
}  // namespace kfbim
