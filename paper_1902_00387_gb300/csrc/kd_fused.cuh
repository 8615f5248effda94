// Persistent fine propagator for the grids whose mixed field fits the shared memory of a
// thread-block cluster (kept sets K <= 95: n <= 286), RK443, both precisions: every step of a
// field in one launch.
//
// The step runs on N = L R = 24, 48, 96, 128 or 192 points, the smallest of them with
// N >= 2K + 2 (alias-free for the kept set, fine_fft_grid in kd_fine.h).  A cluster of CS
// blocks holds one field; block r owns the x columns [r XH, (r + 1) XH), XH = N / CS, of the
// mixed field B[c][ky][x] and the ky rows [r RH, (r + 1) RH).  A stage is
//   column pass (own columns, local): kept ky -> inverse y transform -> u x b -> forward y
//     transform -> kept ky, in place in B; cluster barrier;
//   row pass (own rows, x from every block through distributed shared memory): forward x
//     transform -> curl and IMEX update (stage arrays in global memory, L2-resident) -> inverse
//     x transform -> back into B; cluster barrier.
// A column or row is L lanes with R values a lane of all three components, transformed by an
// R-point DFT in the lane and an L-point DFT across the lanes (shuffles), so u x b, the curl
// and the update need no exchange, no shared memory is spent on transposes (B alone decides
// how few blocks a field needs) and 12 to 16 warps an SM fit.
//
// Why one launch: with two kernels a stage (kd_fine2.cuh and the others) these grids were bound by
// the launches, by few warps in flight and by L2 round trips of the mixed field.  Bound now: the
// instruction issue of the passes (90% in the column pass, 870 instructions a 96-point column)
// for a batch, the chain of a stage (~11 k cycles at 128^2, two cluster barriers among them) for
// a few fields.  Measured, us a step, against the two-kernel plans: 128^2 complex64, 64 fields 72
// (137), one 23 (39); 64^2 x 64 22 (81); 32^2 x 8 14 (62); 160^2 x 10 on 128 points 43 (82); 192^2
// x 100 425 (889); 256^2 x 128 745 (931); complex128 32^2 x 8 57 (314), 128^2 x 64 1970 (2508).
// In complex64 stage 0 stores its explicit term alone, and stage 1 forms the accumulators from it
// and the state: 14 compact arrays a step instead of 17 (128^2 x 64 72.1 us instead of 75.6, 256^2 x
// 128 745 instead of 777).  Complex128 is bound by FP64 arithmetic and keeps the accumulators.
// Tried and slower: 12 or 24 values a lane with one transpose through shared memory, which
// executes fewer instructions but fits fewer and longer chains of warps (80 and 100 us at 128^2
// x 64); x in q + R rev(l), whose accesses to other blocks split into three times the sectors.
//
// The arithmetic of a field does not depend on CS or on the batch (one instantiation, every
// transform owned by one group of lanes), so results are the same bit for bit however a batch
// is cut.
#pragma once
#include "kd_stage.cuh"
#include "kd_wt.cuh"

namespace kd {

// Transform of N = L R points by L lanes, R values a lane:
//   spectral layout: lane l holds x[l + L k], k < R
//   physical layout: lane l holds x[q + R rev(l)], q < R (rev: bit reversal of l < L)
// a_to_b (spectral -> physical): R-point DFT, twiddle w_N^(l q), L-point DFT across the lanes,
// decimation in frequency with the twiddles of two stages merged after the second (a quarter
// turn between them); b_to_a: the transposed sequence.  X[m] = sum_n x[n] exp(DIR 2 pi i n m / N).
template <typename T, int L, int R>
struct LaneFFT {
  static_assert((L == 8 || L == 16 || L == 32) && (R == 1 || R == 3 || R == 4 || R == 6), "lane transforms");
  static constexpr int N = L * R, LB = L == 32 ? 5 : (L == 16 ? 4 : 3);
  cx<T> w1, w2;      // merged twiddles of the lane: w_L^..., w_8^... (L = 32)
  cx<T> wq[R];       // w_N^(l q)
  T sg[LB];          // +1 / -1: the lane is the lower / upper one of the pair that differs in this bit
  bool rot1, rot2;   // quarter turns

  __device__ __forceinline__ explicit LaneFFT(int l) {
    constexpr int H = LB - 1;                       // highest lane bit
    const int top = (l >> H) & 1, nxt = (l >> (H - 1)) & 1, m = l & (L / 4 - 1);
    w1 = wt_tw<N, T>(R * m * (top + 2 * nxt) % N);  // w_L^(m (top + 2 next))
    rot1 = top && nxt;
    if (L == 32) {
      w2 = wt_tw<N, T>(4 * R * ((l & 1) * (((l >> 2) & 1) + 2 * ((l >> 1) & 1))) % N);   // w_8^...
      rot2 = ((l >> 2) & 1) && ((l >> 1) & 1);
    } else {
      w2 = mk(T(1), T(0));
      rot2 = (l & 3) == 3;                          // L = 16
    }
#pragma unroll
    for (int q = 0; q < R; ++q) wq[q] = wt_tw<N, T>(l * q % N);
#pragma unroll
    for (int b = 0; b < LB; ++b) sg[b] = (l >> b) & 1 ? T(-1) : T(1);
  }

  // physical index of register q
  static __device__ __forceinline__ int phys(int l, int q) { return q + R * (int)(__brev((unsigned)l) >> (32 - LB)); }

  template <int DIR>
  static __device__ __forceinline__ cx<T> mul(cx<T> v, cx<T> w) {
    return DIR < 0 ? mk(v.x * w.x - v.y * w.y, v.x * w.y + v.y * w.x) : mk(v.x * w.x + v.y * w.y, v.y * w.x - v.x * w.y);
  }
  template <int DIR>
  static __device__ __forceinline__ cx<T> turn(cx<T> v, bool on) {   // times DIR i
    return mk(on ? (DIR > 0 ? -v.y : v.y) : v.x, on ? (DIR > 0 ? v.x : -v.x) : v.y);
  }
  // Butterflies of every value with the lane that differs in bit BIT.  The three components go
  // through a stage together: shuffles keep their program order, so a value at a time would be
  // one long dependent chain.
  template <int BIT>
  __device__ __forceinline__ void bf(cx<T> (&v)[3][R]) const {
    cx<T> p[3][R];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < R; ++q)
        p[c][q] = mk(__shfl_xor_sync(0xffffffffu, v[c][q].x, 1 << BIT), __shfl_xor_sync(0xffffffffu, v[c][q].y, 1 << BIT));
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < R; ++q) v[c][q] = wt_fma(v[c][q], sg[BIT], p[c][q]);
  }
  template <int DIR>
  static __device__ __forceinline__ void mul3(cx<T> (&v)[3][R], cx<T> w) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < R; ++q) v[c][q] = mul<DIR>(v[c][q], w);
  }
  template <int DIR>
  static __device__ __forceinline__ void turn3(cx<T> (&v)[3][R], bool on) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < R; ++q) v[c][q] = turn<DIR>(v[c][q], on);
  }
  template <int DIR>
  static __device__ __forceinline__ void dft_r(cx<T> (&v)[R]) {
    if constexpr (R == 1) {
    } else if constexpr (R == 3) {
      wt_dft3<T, DIR>(v[0], v[1], v[2]);
    } else if constexpr (R == 4) {
      dft_dif<T, 4, DIR>(v);
      const cx<T> t = v[1];
      v[1] = v[2];
      v[2] = t;
    } else {                                        // 6 = 2 x 3, coprime: no twiddles
#pragma unroll
      for (int n2 = 0; n2 < 3; ++n2) bfly(v[(2 * n2) % 6], v[(3 + 2 * n2) % 6]);
      wt_dft3<T, DIR>(v[0], v[2], v[4]);
      wt_dft3<T, DIR>(v[3], v[5], v[1]);
      const cx<T> t[6] = {v[0], v[1], v[2], v[3], v[4], v[5]};
#pragma unroll
      for (int k = 0; k < 6; ++k) v[k] = t[(3 * (k % 2) + 2 * (k % 3)) % 6];
    }
  }
  template <int DIR>
  __device__ __forceinline__ void a_to_b(cx<T> (&v)[3][R]) const {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      dft_r<DIR>(v[c]);
#pragma unroll
      for (int q = 1; q < R; ++q) v[c][q] = mul<DIR>(v[c][q], wq[q]);
    }
    bf<LB - 1>(v);
    turn3<DIR>(v, rot1);
    bf<LB - 2>(v);
    mul3<DIR>(v, w1);
    bf<LB - 3>(v);
    if constexpr (L >= 16) {
      turn3<DIR>(v, rot2);
      bf<LB - 4>(v);
    }
    if constexpr (L == 32) {
      mul3<DIR>(v, w2);
      bf<0>(v);
    }
  }
  template <int DIR>
  __device__ __forceinline__ void b_to_a(cx<T> (&v)[3][R]) const {
    if constexpr (L == 32) {
      bf<0>(v);
      mul3<DIR>(v, w2);
    }
    if constexpr (L >= 16) {
      bf<LB - 4>(v);
      turn3<DIR>(v, rot2);
    }
    bf<LB - 3>(v);
    mul3<DIR>(v, w1);
    bf<LB - 2>(v);
    turn3<DIR>(v, rot1);
    bf<LB - 1>(v);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int q = 1; q < R; ++q) v[c][q] = mul<DIR>(v[c][q], wq[q]);
      dft_r<DIR>(v[c]);
    }
  }
};

template <typename T, int L, int R>
struct FusedStep {
  static constexpr int N = L * R, TPW = 32 / L;        // transforms a warp takes at once
  static constexpr int MAXW = sizeof(T) == 4 ? (R <= 4 ? 16 : 12) : (R <= 3 ? 12 : 8);
  __host__ __device__ static constexpr int xp(int XH) { return XH | 1; }   // odd pitch: conflict-free columns
  __host__ __device__ static constexpr int field(int P, int CS) { return (3 * P * xp(N / CS) + 1) & ~1; }
  static size_t smem(int P, int CS) { return ((size_t)field(P, CS) + N) * sizeof(cx<T>); }
  // warps of a block: the passes' tasks in as few rounds as the largest block needs, evenly
  static int warps(int P, int CS) {
    const int ct = (N / CS + TPW - 1) / TPW, rt = ((P + CS - 1) / CS + TPW - 1) / TPW;
    const int t = ct > rt ? ct : rt, rounds = (t + MAXW - 1) / MAXW;
    return (t + rounds - 1) / rounds;
  }
};

__device__ __forceinline__ uint32_t fused_peer(uint32_t addr, int rank) {
  uint32_t o;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(addr), "r"(rank));
  return o;
}
// Loads and stores of a value at a shared address of this block (near) or of a cluster address.
__device__ __forceinline__ cx<float> fused_ld(uint32_t addr, bool near, float) {
  cx<float> v;
  if (near)
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
  else
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ cx<double> fused_ld(uint32_t addr, bool near, double) {
  cx<double> v;
  if (near)
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr));
  else
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ void fused_st(uint32_t addr, bool near, cx<float> v) {
  if (near)
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
  else
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void fused_st(uint32_t addr, bool near, cx<double> v) {
  if (near)
    asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(addr), "d"(v.x), "d"(v.y) : "memory");
  else
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(addr), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void fused_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Element at a 32-bit byte offset of a (uniform) base.
template <typename T>
__device__ __forceinline__ const cx<T>& fused_at(const cx<T>* p, unsigned o) {
  return *(const cx<T>*)((const char*)p + o);
}
template <typename T>
__device__ __forceinline__ cx<T>& fused_at(cx<T>* p, unsigned o) {
  return *(cx<T>*)((char*)p + o);
}

// One component of one IMEX RK443 stage (the expressions of stage_update, kd_stage.cuh): f =
// F_c(X_j); r the arrays read: X (stage 0), R2 R3 R4 (1), R3 R4 (2), R4 X Xlo (3); o: where the
// arrays written go: R2 R3 R4; R3 R4; R4; X Xlo; stored where `on`.  In complex64 stage 0 writes
// f to R2 only and stage 1 reads X and f.  Returns X_{j+1}.
template <int MODE, typename T>
__device__ __forceinline__ cx<T> fused_update(cx<T>* o0, cx<T>* o1, cx<T>* o2, bool on, T dt, T g, T dl, cx<T> f,
                                              const cx<T>* r) {
  if constexpr (MODE == 0) {
    const cx<T> t = wt_fma(f, dt * T(0.5), r[0]), x = wt_fma(t, -g, t);
    if constexpr (sizeof(T) == 4) {
      if (on) *o0 = f;
      return x;
    }
    if (on) {
      *o0 = wt_fma(x, dl * T(-1.0 / 6.0), wt_fma(f, dt * T(11.0 / 18.0), r[0]));
      *o1 = wt_fma(x, dl * T(0.5), wt_fma(f, dt * T(5.0 / 6.0), r[0]));
      *o2 = wt_fma(x, dl * T(-1.5), f * (dt * T(0.25)));
    }
    return x;
  } else if constexpr (MODE == 1 && sizeof(T) == 4) {   // r: X, the explicit term of stage 0
    const cx<T> t0 = wt_fma(r[1], dt * T(0.5), r[0]), x1 = wt_fma(t0, -g, t0);
    const cx<T> a[3] = {wt_fma(x1, dl * T(-1.0 / 6.0), wt_fma(r[1], dt * T(11.0 / 18.0), r[0])),
                        wt_fma(x1, dl * T(0.5), wt_fma(r[1], dt * T(5.0 / 6.0), r[0])),
                        wt_fma(x1, dl * T(-1.5), r[1] * (dt * T(0.25)))};
    const cx<T> t = wt_fma(f, dt * T(1.0 / 18.0), a[0]), x = wt_fma(t, -g, t);
    if (on) {
      *o0 = wt_fma(x, dl * T(-0.5), wt_fma(f, dt * T(-5.0 / 6.0), a[1]));
      *o1 = wt_fma(x, dl * T(1.5), wt_fma(f, dt * T(1.75), a[2]));
    }
    return x;
  } else if constexpr (MODE == 1) {
    const cx<T> t = wt_fma(f, dt * T(1.0 / 18.0), r[0]), x = wt_fma(t, -g, t);
    if (on) {
      *o0 = wt_fma(x, dl * T(-0.5), wt_fma(f, dt * T(-5.0 / 6.0), r[1]));
      *o1 = wt_fma(x, dl * T(1.5), wt_fma(f, dt * T(1.75), r[2]));
    }
    return x;
  } else if constexpr (MODE == 2) {
    const cx<T> t = wt_fma(f, dt * T(0.5), r[0]), x = wt_fma(t, -g, t);
    if (on) *o0 = wt_fma(x, dl * T(-0.5), wt_fma(f, dt * T(0.75), r[1]));
    return x;
  } else {
    const cx<T> e = final_increment(r[1], wt_fma(f, dt * T(-1.75), r[0]), g);
    if constexpr (sizeof(T) == 8) {
      const cx<T> x = r[1] + e;
      if (on) *o0 = x;
      return x;
    } else {                                        // the state as a pair (state_add, kd_stage.cuh)
      T s0, e0, s1, e1;
      cx<T> hi, lo;
      two_sum(r[1].x, e.x, s0, e0);
      two_sum(r[1].y, e.y, s1, e1);
      two_sum(s0, r[2].x + e0, hi.x, lo.x);
      two_sum(s1, r[2].y + e1, hi.y, lo.y);
      if (on) {
        *o0 = hi;
        *o1 = lo;
      }
      return hi;
    }
  }
}

// FUSED_CLUSTER: steps [s0, s0 + nsteps) of every field b = blockIdx.x / CS, from the state X (and
// Xlo when s0 > 0) back to X (Xlo).
//
// A few fields of the largest complex128 sets leave most of the GPU idle in clusters, 16 SMs each at
// most, and FP64 arithmetic bounds them.  For them (LaneKernel::SPREAD in kd_fused.cu, with the
// times of both) the same passes run as launches over the whole GPU, a warp a block, so that every
// quarter of an SM has one task, with the mixed field in global memory (a.W, L2).  FUSED_COLS: column
// pass of stage nsteps of step s0, field blockIdx.y; FUSED_ROWS: row pass of stage nsteps (4: before the
// first stage), CS: whether another stage follows.  The arithmetic is this one source's, so the
// values are the same bits.
enum { FUSED_CLUSTER = 0, FUSED_COLS = 1, FUSED_ROWS = 2 };

template <typename T, int L, int R, int MODE = FUSED_CLUSTER>
__global__ void __launch_bounds__(MODE == FUSED_CLUSTER ? 32 * FusedStep<T, L, R>::MAXW : 32, 1)
    fused_kernel(FineArgs a, int CS, int s0, int nsteps) {
  using F = FusedStep<T, L, R>;
  constexpr bool CL = MODE == FUSED_CLUSTER;
  constexpr int N = F::N, TPW = F::TPW;
  // registers of the row whose stage arrays are in flight ahead of their use
  constexpr int AHEAD = sizeof(T) == 4 ? (R == 6 ? 3 : R) : (R == 1 ? 1 : 2);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int K = a.K, P = a.P;
  const int XH = CL ? N / CS : N, XP = CL ? F::xp(XH) : N, RH = CL ? (P + CS - 1) / CS : P;
  const int rank = CL ? (int)(blockIdx.x % CS) : 0;
  const long b = CL ? blockIdx.x / CS : blockIdx.y;
  const int x0 = rank * XH, y0 = rank * RH, rows = max(0, min(RH, P - y0));
  // the warp index as the uniform value that it is: the loops over a warp's tasks then need no
  // re-convergence before each shuffle (a third of the instructions otherwise)
  const int warp = CL ? __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0) : blockIdx.x;
  const int nw = CL ? blockDim.x >> 5 : gridDim.x;
  const int l = threadIdx.x & (L - 1), grp = (threadIdx.x & 31) / L;   // lane and transform of the warp's TPW
  cx<T>* B = CL ? (cx<T>*)smem_raw : (cx<T>*)a.W + b * 3 * P * N;   // [3][P][XP]
  cx<T>* s_cs = CL ? B + F::field(P, CS) : (cx<T>*)smem_raw;        // (cos, sin)(2 pi j / N)
  if (MODE != FUSED_ROWS)
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const cx<T> w = wt_tw<N, T>(i);
      s_cs[i] = mk(w.x, -w.y);
    }
  const LaneFFT<T, L, R> fft(l);
  const StageCoef<T> sc = stage_coef<T>(a, b);
  const T A = flow_amp<T>(a, b);
  const T inv_n2 = T(1) / (T(N) * T(N));
  const int rl = fft.phys(l, 0);                   // R rev(l)

  // Columns keep ky in the lane layout l + L k and y in q + R rev(l); rows keep x in l + L q, so
  // that the lanes of an access to another block's shared memory are consecutive (a request is
  // split by block and 32-byte sector), and kx in k + R rev(l).
  // The stage arrays R2..R4, Xlo and the kernel's own copy of the state (in a.M, which the
  // two-kernel step uses) hold a row's P kept values in that order: those of k = 0, then 1, ...,
  // ascending in rev(l), so that an access is consecutive too.
  bool kk[R], kx_on[R];                            // ky, kx of register k kept
  int ky_at[R], kx[R], slot[R];                    // row offset in B, kx, place in a stage array's row
  uint32_t at_q[R];                                // cluster address of (row 0, x of register q)
  bool near[R];                                    // ... in this block: off the network between the SMs
  {
    int first = 0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const int ky = l + L * k < N / 2 ? l + L * k : l + L * k - N;
      kk[k] = ky >= -K && ky <= K;
      ky_at[k] = (K + ky) * XP;
      const int i = k + rl, m = rl / R, nlow = K >= k ? (K - k) / R + 1 : 0, mhigh = (N - K - k + R - 1) / R;
      kx[k] = i < N / 2 ? i : i - N;
      kx_on[k] = i <= K || i >= N - K;
      slot[k] = first + (i <= K ? m : nlow + m - mhigh);
      first += nlow + L - mhigh;
      if (CL) {
        const int x = l + L * k, own = x / XH;
        near[k] = own == rank;
        at_q[k] = (uint32_t)__cvta_generic_to_shared(B + x - own * XH);
        if (!near[k]) at_q[k] = fused_peer(at_q[k], own);
      }
    }
  }
  const uint32_t row_b = (uint32_t)(XP * (int)sizeof(cx<T>));   // bytes of a row of B
  const long PP = (long)P * P, fld = b * 3 * PP;   // a component, the field in the stage arrays
  cx<T>* X = (cx<T>*)a.X + fld;                    // the caller's state [3][P][P], kx ascending
  cx<T>* Xp = (cx<T>*)a.M + fld;                   // the kernel's copy
  cx<T>* Xl = a.Xlo ? (cx<T>*)a.Xlo + fld : nullptr;
  cx<T>*R2 = (cx<T>*)a.R2 + fld, *R3 = (cx<T>*)a.R3 + fld, *R4 = (cx<T>*)a.R4 + fld;

  // Row pass of a stage (4: the inverse x transform of X only); more: another stage follows.  The
  // stage arrays are loaded before the transform, which covers their latency (L2), those of AHEAD
  // registers at a time.
  auto row_pass = [&](int stage, bool more, bool lo_valid) {
    constexpr bool f0 = sizeof(T) == 4;            // stage 0 leaves its explicit term in R2
    const cx<T>* p0 = stage == 0 || (stage == 1 && f0) ? Xp : (stage == 1 ? R2 : (stage == 2 ? R3 : R4));
    const cx<T>* p1 = stage == 1 ? (f0 ? R2 : R3) : (stage == 2 ? R4 : (stage == 3 ? Xp : nullptr));
    const cx<T>* p2 = stage == 1 && !f0 ? R4 : (stage == 3 && lo_valid ? Xl : nullptr);
    for (int t = warp; t * TPW < rows; t += nw) {
      const bool ok = t * TPW + grp < rows;
      const int iy = y0 + min(t * TPW + grp, rows - 1);
      cx<T> v[3][R], r[3][AHEAD][3];
      auto load = [&](int k, int to) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const unsigned at = (unsigned)((int)(c * PP) + iy * P + slot[k]) * (unsigned)sizeof(cx<T>);
          const bool on = ok && kx_on[k];
          r[c][to][0] = on ? fused_at(p0, at) : mk(T(0), T(0));
          r[c][to][1] = on && p1 ? fused_at(p1, at) : mk(T(0), T(0));
          r[c][to][2] = on && p2 ? fused_at(p2, at) : mk(T(0), T(0));
        }
      };
      if (stage < 4) {
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) load(k, k);
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int q = 0; q < R; ++q)
            v[c][q] = CL ? fused_ld(at_q[q] + (uint32_t)(c * P + iy) * row_b, near[q], T(0)) : B[(c * P + iy) * N + l + L * q];
        fft.template a_to_b<-1>(v);                // x -> kx
        const T fky = (T)(iy - K), kz = sc.kz, ly = fky * fky + kz * kz;
        auto update = [&](auto mode_c) {
          constexpr int MODE = decltype(mode_c)::value;
#pragma unroll
          for (int k = 0; k < R; ++k) {
            const bool on = ok && kx_on[k];
            const T fkx = (T)kx[k], lam = (fkx * fkx + ly) * sc.inv_rm;
            const T gain = fused_gain(sc.dt * T(0.5) * lam), dl = sc.dt * lam;
            const T ax = fkx * inv_n2, ay = fky * inv_n2, az = kz * inv_n2;
            const cx<T> w0 = v[0][k], w1 = v[1][k], w2 = v[2][k];
            const cx<T> f[3] = {mul_i(wt_fma(w2, ay, w1 * -az)), mul_i(wt_fma(w0, az, w2 * -ax)),
                                mul_i(wt_fma(w1, ax, w0 * -ay))};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const unsigned at = (unsigned)((int)(c * PP) + iy * P + slot[k]) * (unsigned)sizeof(cx<T>);
              cx<T>* o0 = MODE == 0 ? R2 : (MODE == 1 ? R3 : (MODE == 2 ? R4 : Xp));
              cx<T>* o1 = MODE == 0 ? R3 : (MODE == 1 ? R4 : Xl);
              const cx<T> x = fused_update<MODE, T>(&fused_at(o0, at), &fused_at(o1, at), &fused_at(R4, at), on, sc.dt, gain, dl, f[c], r[c][k % AHEAD]);
              if (MODE == 3 && !more && on) X[(int)(c * PP) + iy * P + K + kx[k]] = x;   // the step's result
              v[c][k] = on ? x : mk(T(0), T(0));
            }
            if (k + AHEAD < R) load(k + AHEAD, k % AHEAD);
          }
        };
        if (stage == 0) update(std::integral_constant<int, 0>());
        else if (stage == 1) update(std::integral_constant<int, 1>());
        else if (stage == 2) update(std::integral_constant<int, 2>());
        else update(std::integral_constant<int, 3>());
        if (!more) continue;
      } else {
#pragma unroll
        for (int k = 0; k < R; ++k)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const bool on = ok && kx_on[k];
            v[c][k] = on ? X[(int)(c * PP) + iy * P + K + kx[k]] : mk(T(0), T(0));
            if (on) Xp[(int)(c * PP) + iy * P + slot[k]] = v[c][k];
          }
      }
      fft.template b_to_a<+1>(v);                  // kx -> x
      if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (CL)
              fused_st(at_q[q] + (uint32_t)(c * P + iy) * row_b, near[q], v[c][q]);
            else
              B[(c * P + iy) * N + l + L * q] = v[c][q];
      }
    }
  };

  auto col_pass = [&](int step, int stage) {
    const Phase<T> ph = load_phase<T>(a, b, step, stage);
    // u at the lane's y: u_x and the y part of u_z
    T ux[R], uzy[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const cx<T> cs = s_cs[q + rl];
      ux[q] = A * (cs.x * ph.cpy - cs.y * ph.spy);
      uzy[q] = cs.y * ph.cpy + cs.x * ph.spy;
    }
    for (int t = warp; t * TPW < XH; t += nw) {
      const bool ok = t * TPW + grp < XH;
      const int xl = min(t * TPW + grp, XH - 1);
      cx<T>* col = B + xl;
      cx<T> v[3][R];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < R; ++k) v[c][k] = kk[k] ? col[c * P * XP + ky_at[k]] : mk(T(0), T(0));
      fft.template a_to_b<+1>(v);                  // ky -> y
      const cx<T> csx = s_cs[x0 + xl];
      const T uy = A * (csx.y * ph.cpx + csx.x * ph.spx), uzx = csx.x * ph.cpx - csx.y * ph.spx;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const T uz = A * (uzx + uzy[q]);
        const cx<T> bx = v[0][q], by = v[1][q], bz = v[2][q];
        v[0][q] = wt_fma(bz, uy, by * -uz);
        v[1][q] = wt_fma(bx, uz, bz * -ux[q]);
        v[2][q] = wt_fma(by, ux[q], bx * -uy);
      }
      fft.template b_to_a<-1>(v);                  // y -> ky
      if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int k = 0; k < R; ++k)
            if (kk[k]) col[c * P * XP + ky_at[k]] = v[c][k];
      }
    }
  };

  if constexpr (CL) {
    griddep_wait();                                // X comes from the predecessor
    fused_cluster_sync();                          // tables; every block of the cluster runs
    // one copy of each pass: the prologue is the row pass before the first stage
#pragma unroll 1
    for (int it = -1; it < 4 * nsteps; ++it) {
      const int s = s0 + (it >> 2), j = it & 3;
      if (it >= 0) {
        col_pass(s, j);
        fused_cluster_sync();
      }
      row_pass(it < 0 ? 4 : j, it + 1 < 4 * nsteps, s > 0);
      fused_cluster_sync();   // B is complete; after the last stage: no peer reads it any more
    }
  } else {
    griddep_launch_dependents();                   // the next pass waits for this one's end itself
    __syncwarp();                                  // table
    griddep_wait();
    if constexpr (MODE == FUSED_COLS)
      col_pass(s0, nsteps);
    else
      row_pass(nsteps, CS != 0, s0 > 0);
  }
}

}  // namespace kd
