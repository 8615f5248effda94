// Complex64 warp transforms of N = V S points (V = 24 values a lane in physical space), the sides
// m = 384 and 768 = 3/4 of 512 and 1024 on which the 2/3-rule step of these grids is evaluated; and
// the twiddles and small DFTs that kd_fused.cuh shares.
//
// Why three quarters.  The kept set is |k| <= K = n / 3 and both flows hold only the
// wavenumbers +-1, so u x b has |k| <= K + 1 and m >= 2K + 2 points resolve its kept modes
// without aliasing: the kept modes of the pseudo-spectral step on m points are those of the
// step on n points (fine_fft_grid in kd_fine.h).  For n = 2^p, m = 3n/4 >= 2K + 2 always
// holds, and the mixed fields and the row transforms shrink by 1/4, the column pass (fewer
// and shorter transforms) by 7/16.
//
// A warp owns C = 32 / S transforms of one kind (columns or rows) at a time:
//   physical layout: lane l = c S + m1 holds X_c[m1 + S m2], m2 < V          (all 32 lanes)
//   spectral layout: lane a < 24 (the rest repeat lane 23), transform r < C: register r S + k holds
//                    x_r[a + V k], k < S
// spectral -> physical (n = a + V k, m = m1 + S m2): an S-point DFT over k in the lane, the
// twiddle w_N^(a m1), a transpose through the warp's shared buffer, a V-point DFT over a.
// physical -> spectral is the transposed sequence.  One transpose a transform; the S-point
// side runs on 24 of 32 lanes, which is the cheaper side (S <= 32 radix-2 points, and all of
// its twiddles depend on the lane only).  Both directions compute
// X[m] = sum_n x[n] exp(DIR 2 pi i n m / N), no normalisation.
#pragma once
#include "kd_fft2.cuh"

namespace kd {

// w_768^e = exp(-2 pi i e / 768), e < 768, evaluated by the compiler: one octant by the
// Taylor series (arguments up to pi / 4; the remainder after these terms is below 1e-20),
// the rest by symmetry, so multiples of pi / 4 are exact or correctly placed.  Every side
// here divides 768: w_N^e is entry e 768 / N, and its real and minus its imaginary part are
// the cos and sin of the collocation points.
struct W768 {
  double re[768], im[768];
};
constexpr double wt_cos_taylor(double x) {
  const double y = x * x;
  double s = 1.0;
  for (int k = 12; k >= 1; --k) s = 1.0 - s * y / ((2.0 * k - 1.0) * (2.0 * k));
  return s;
}
constexpr double wt_sin_taylor(double x) {
  const double y = x * x;
  double s = 1.0;
  for (int k = 12; k >= 1; --k) s = 1.0 - s * y / ((2.0 * k) * (2.0 * k + 1.0));
  return s * x;
}
constexpr W768 wt_make_w768() {
  W768 t{};
  constexpr double pi = 3.14159265358979323846;
  for (int e = 0; e < 768; ++e) {
    const int q = e / 192, r = e - 192 * q;           // quadrant and angle r pi / 384 in it
    double c = 0.0, s = 0.0;
    if (r <= 96) {
      c = wt_cos_taylor(r * pi / 384.0);
      s = wt_sin_taylor(r * pi / 384.0);
    } else {
      c = wt_sin_taylor((192 - r) * pi / 384.0);
      s = wt_cos_taylor((192 - r) * pi / 384.0);
    }
    const double cc = q == 0 ? c : (q == 1 ? -s : (q == 2 ? -c : s));
    const double ss = q == 0 ? s : (q == 1 ? c : (q == 2 ? -s : -c));
    t.re[e] = cc;
    t.im[e] = -ss;
  }
  return t;
}
__device__ constexpr W768 g_w768 = wt_make_w768();

template <int N, typename T>
__device__ __forceinline__ cx<T> wt_tw(int e) {       // w_N^e, 0 <= e < N
  static_assert(768 % N == 0, "sides that divide 768");
  const int i = e * (768 / N);
  return mk((T)g_w768.re[i], (T)g_w768.im[i]);
}

// a s + b on both components; complex64: one packed FP32x2 instruction (each component rounds
// once, as a scalar fused multiply-add does).
__device__ __forceinline__ cx<float> wt_fma(cx<float> a, float s, cx<float> b) {
  const float2 r = __ffma2_rn(make_float2(a.x, a.y), make_float2(s, s), make_float2(b.x, b.y));
  return mk(r.x, r.y);
}
__device__ __forceinline__ cx<double> wt_fma(cx<double> a, double s, cx<double> b) {
  return mk(__fma_rn(a.x, s, b.x), __fma_rn(a.y, s, b.y));
}
__device__ __forceinline__ cx<float> wt_add(cx<float> a, cx<float> b) {
  const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
  return mk(r.x, r.y);
}
__device__ __forceinline__ cx<double> wt_add(cx<double> a, cx<double> b) { return a + b; }

// 3-point DFT in place; (a, b, c) -> X[0], X[1], X[2].
template <typename T, int DIR>
__device__ __forceinline__ void wt_dft3(cx<T>& a, cx<T>& b, cx<T>& c) {
  constexpr T h = (T)(DIR * 0.86602540378443864676);
  const cx<T> x0 = a;
  cx<T> t = b, d = c;
  bfly(t, d);                                          // t = b + c, d = b - c
  a = wt_add(x0, t);
  const cx<T> m = wt_fma(t, T(-0.5), x0);
  b = mk(m.x - h * d.y, m.y + h * d.x);
  c = mk(m.x + h * d.y, m.y - h * d.x);
}

// DFT of 24 = 3 x 8 points (coprime factors: no twiddles between them).  In: v[n] natural
// order; out: X[k] at v[wt_pos(k)].  Input n = (8 n1 + 3 n2) mod 24, output k = k1 mod 3 = k2 mod 8.
__host__ __device__ constexpr int wt_pos(int k) { return (8 * (k % 3) + 3 * bitrev<8>(k % 8)) % 24; }
template <int DIR>
__device__ __forceinline__ void wt_dft24(cx<float> (&v)[24]) {
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2)
    wt_dft3<float, DIR>(v[(3 * n2) % 24], v[(8 + 3 * n2) % 24], v[(16 + 3 * n2) % 24]);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cx<float> u[8];
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) u[n2] = v[(8 * k1 + 3 * n2) % 24];
    dft_dif<float, 8, DIR>(u);                         // residue k2 at u[bitrev(k2)]
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) v[(8 * k1 + 3 * n2) % 24] = u[n2];
  }
}

template <int S_>
struct WT {
  static_assert(S_ == 32 || S_ == 16, "lanes a transform");
  static constexpr int V = 24, S = S_, N = V * S;
  static constexpr int C = 32 / S;                     // transforms of a warp
  static constexpr int SV = C * S;                     // spectral values a lane
  // transpose buffer: [c][m1][a], rows of PITCH complex: the 16-byte row accesses of a quarter
  // warp are conflict-free
  static constexpr int PITCH = V + 2;
  static constexpr int CST = S * PITCH;                // complex per transform
  static constexpr int BUF = C * CST;
  // twiddles of a lane: w_N^(a m1) from the table s_tw[m1 * V + a] (m1 < S)
  static constexpr int TAB = S * V;

  static __device__ __forceinline__ void table(cx<float>* s_tw) {
    for (int i = threadIdx.x; i < TAB; i += blockDim.x) s_tw[i] = wt_tw<N, float>(((i / V) * (i % V)) % N);
  }
  // The spectral lane of lane l: lanes 24..31 read and compute what lane 23 does (their values are
  // not stored), which costs no more than idling them and keeps the code free of divergence.
  static __device__ __forceinline__ int slane(int l) { return l < 24 ? l : 23; }
  static __device__ __forceinline__ int phys_c(int l) { return l / S; }
  static __device__ __forceinline__ int phys_m1(int l) { return l % S; }

  template <int DIR>
  static __device__ __forceinline__ cx<float> tw_mul(cx<float> v, cx<float> w) {
    return DIR < 0 ? mk(v.x * w.x - v.y * w.y, v.x * w.y + v.y * w.x) : mk(v.x * w.x + v.y * w.y, v.y * w.x - v.x * w.y);
  }

  // Spectral registers s -> physical registers v.  B: the warp's buffer (BUF complex), free on
  // entry; free again on return for accesses after a __syncwarp.
  template <int DIR>
  static __device__ __forceinline__ void s2p(cx<float> (&s)[SV], cx<float> (&v)[V], int l, cx<float>* B,
                                             const cx<float>* s_tw) {
    const int a = slane(l);
#pragma unroll
    for (int r = 0; r < C; ++r) {
      dft_dif<float, S, DIR>(&s[r * S]);               // X[m1] at bitrev(m1)
      cx<float>* row = B + r * CST + a;
#pragma unroll
      for (int m1 = 0; m1 < S; ++m1) {
        cx<float> y = s[r * S + bitrev<S>(m1)];
        if (m1 != 0) y = tw_mul<DIR>(y, s_tw[m1 * V + a]);
        if (l < 24) row[m1 * PITCH] = y;
      }
    }
    __syncwarp();
    const cx<float>* row = B + phys_c(l) * CST + phys_m1(l) * PITCH;
#pragma unroll
    for (int i = 0; i < V; i += 2) {
      const float4 q = *(const float4*)&row[i];
      v[i] = mk(q.x, q.y);
      v[i + 1] = mk(q.z, q.w);
    }
    __syncwarp();
    wt_dft24<DIR>(v);
    cx<float> t[V];
#pragma unroll
    for (int k = 0; k < V; ++k) t[k] = v[wt_pos(k)];
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = t[k];
  }

  // Physical registers v (destroyed) -> spectral registers s.
  template <int DIR>
  static __device__ __forceinline__ void p2s(cx<float> (&v)[V], cx<float> (&s)[SV], int l, cx<float>* B,
                                             const cx<float>* s_tw) {
    wt_dft24<DIR>(v);                                  // residue a at v[wt_pos(a)]
    cx<float>* to = B + phys_c(l) * CST + phys_m1(l) * PITCH;
#pragma unroll
    for (int i = 0; i < V; i += 2) {
      const cx<float> y0 = v[wt_pos(i)], y1 = v[wt_pos(i + 1)];
      *(float4*)&to[i] = make_float4(y0.x, y0.y, y1.x, y1.y);
    }
    __syncwarp();
    const int a = slane(l);
#pragma unroll
    for (int r = 0; r < C; ++r) {
      const cx<float>* row = B + r * CST + a;
#pragma unroll
      for (int m1 = 0; m1 < S; ++m1) {
        cx<float> y = row[m1 * PITCH];
        if (m1 != 0) y = tw_mul<DIR>(y, s_tw[m1 * V + a]);
        s[r * S + m1] = y;
      }
      dft_dif<float, S, DIR>(&s[r * S]);
      cx<float> t[S];
#pragma unroll
      for (int k = 0; k < S; ++k) t[k] = s[r * S + bitrev<S>(k)];
#pragma unroll
      for (int k = 0; k < S; ++k) s[r * S + k] = t[k];
    }
    __syncwarp();
  }
};

}  // namespace kd
