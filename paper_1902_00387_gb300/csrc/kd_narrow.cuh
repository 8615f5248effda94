// Fine-step kernels of the complex64 grids n = 1024 and 512 evaluated on N = 3n/4 = 768 and
// 384 points (kd_wt.cuh: alias-free for the kept set), RK443.
//
// Two kernels a stage as on the other grids (kd_fine.cu): a column kernel (one warp per C
// adjacent columns with all three components in registers) and a row kernel (one warp per
// component of C ky rows), both persistent.  What bounds them at 1024^2 x 256: the column
// kernel the shared-memory data pipe (71% of its wavefronts by the counters; transposes,
// twiddles, staging), the row kernel HBM (4.7 TB/s on its bytes) and the latency of its loads.
// A step measured against the 1024-point kernels (column 3.13 ms, row 3.97 a launch): 23.0 ms
// (30.2), the column kernel 2.30 a launch; a step of 45 fields of 512^2 1.02 ms (1.38).  With all
// the stage arrays of a row staged in shared memory (three blocks an SM instead of five at stages
// 1 and 3) and three accumulators stored by stage 0 the steps took 25.3 and 1.15 ms.  Two column groups
// a block (8 warps, 255 registers) took 2.32 ms, so a third (12 warps, 168 registers, 140
// bytes of spills) gains little; the components in rolled loops (38 instead of 92 KB of
// code) 2.85 ms, for the register moves and the lost overlap.
#pragma once
#include "kd_fine4.cuh"
#include "kd_wt.cuh"

namespace kd {

template <int N>
struct NarrowGrid {
  static_assert(N == 768 || N == 384, "3/4 of 1024 and 512");
  using W = WT<N / 24>;
  static constexpr int FULL = N / 3 * 4;               // the problem's grid side
  static constexpr int K = FULL / 3, P = 2 * K + 1;
  static_assert(N >= 2 * K + 2, "no aliasing onto the kept set");
  // Element lane + 24 q of a transform (lane < 24, wavenumber itself or itself - N) has the kept
  // index j = lane + K + kofs(q); keeps(q, lane) says whether it is kept.  Both fold to
  // constants but for the one or two q whose range straddles an end of the kept set.
  __host__ __device__ static constexpr int kofs(int q) { return 24 * q <= K ? 24 * q : 24 * q - N; }
  __host__ __device__ static constexpr bool keeps(int q, int lane) {
    return 24 * q <= K ? (24 * q + 23 <= K || lane + 24 * q <= K)
                       : (24 * q >= N - K || (24 * q + 23 >= N - K && lane + 24 * q >= N - K));
  }
};

// ------------------------------------------------------------------ column kernel
// A group of 4 warps owns XG = 4 C adjacent columns (32- or 64-byte runs of a row); GR groups
// a block with their own buffers and named barriers, so that one group copies while another
// transforms.  Input rows arrive a component at a time through two staging buffers (16-byte
// cp.async, two components ahead; 16-byte chunks swizzled by row bits that adding a multiple
// of 24 rows leaves alone, so a lane's accesses differ by constants); the output goes through
// a staging area that overlays the group's transpose buffers (odd pitch: conflict-free column
// writes).
template <int N, int GR_>
struct ColN {
  using G = NarrowGrid<N>;
  using W = typename G::W;
  static constexpr int GR = GR_, GW = 4, GT = 32 * GW, XG = GW * W::C, BLOCK = GT * GR;
  static constexpr int P = G::P, H = XG / 2;           // 16-byte chunks of a staged row
  static constexpr int OP = XG + 1;                    // pitch of the output staging (complex)
  static constexpr int TB = (GW * W::BUF > P * OP ? GW * W::BUF : P * OP) + 1 & ~1;
  static constexpr int GSM = TB + 2 * P * XG;          // complex per group
  static_assert(TB % 2 == 0 && (P * XG) % 2 == 0, "16-byte aligned buffers");
  static constexpr size_t smem = ((size_t)GR * GSM + W::TAB) * sizeof(cx<float>) + (size_t)N * sizeof(float2);
  static constexpr int SH = XG == 8 ? 1 : 2;           // rows per 128 bytes: 2 or 4
  __device__ __forceinline__ static int in_at(int j, int xi) {
    return j * XG + ((((xi >> 1) ^ (j >> SH)) & (H - 1)) << 1) + (xi & 1);
  }
};

template <int N, int GR>
__global__ void __launch_bounds__(ColN<N, GR>::BLOCK, 1) coln_kernel(FineArgs a, int step, int stage) {
  using CN = ColN<N, GR>;
  using NG = typename CN::G;
  using W = typename CN::W;
  constexpr int K = NG::K, P = CN::P, XG = CN::XG, GT = CN::GT, H = CN::H, OP = CN::OP, GPF = N / XG;
  constexpr int C = W::C, S = W::S, V = W::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sl = W::slane(lane);
  const int grp = warp / CN::GW, wl = warp - grp * CN::GW, gtid = threadIdx.x - grp * GT;
  cx<float>* Out = (cx<float>*)smem_raw + grp * CN::GSM;   // output staging / transpose buffers
  cx<float>* B = Out + wl * W::BUF;
  cx<float>* In = Out + CN::TB;                            // [2][P][XG]
  cx<float>* s_tw = (cx<float>*)smem_raw + GR * CN::GSM;
  float2* s_cs = (float2*)(s_tw + W::TAB);                 // (cos, sin)(2 pi j / N)
  W::table(s_tw);
  for (int i = threadIdx.x; i < N; i += CN::BLOCK) {
    const cx<float> w = wt_tw<N, float>(i);
    s_cs[i] = make_float2(w.x, -w.y);
  }
  __syncthreads();
  const long groups = (long)a.batch * GPF;
  // neighbouring groups on different SMs, so that a few fields use all of them
  const long first = blockIdx.x + (long)grp * gridDim.x, stride = (long)gridDim.x * GR;
  const long mine = groups > first ? (groups - 1 - first) / stride + 1 : 0;
  const cx<float>* M = (const cx<float>*)a.M;
  cx<float>* Wo = (cx<float>*)a.W;
  // load k of this group: component k % 3 of its column group k / 3 into buffer k % 2
  auto load = [&](long k) {
    if (k < 3 * mine) {
      const long g = first + (k / 3) * stride;
      const int c = (int)(k % 3);
      const long b = g / GPF;
      const int x0 = (int)(g - b * GPF) * XG;
      const cx<float>* src = M + ((b * 3 + c) * (long)P) * N + x0;
      cx<float>* dst = In + (k & 1) * P * XG;
      for (int i = gtid; i < P * H; i += GT) {
        const int h = i % H, j = i / H;
        cp_async16(dst + CN::in_at(j, 2 * h), src + (long)j * N + 2 * h, true);
      }
    }
    cp_async_commit();   // possibly empty: keeps one group per load for the waits
  };
  griddep_wait();    // M is the predecessor's output
  load(0);
  load(1);
  for (long jg = 0; jg < mine; ++jg) {
    const long g = first + jg * stride;
    const long b = g / GPF;
    const int x0 = (int)(g - b * GPF) * XG;
    const Phase<float> ph = load_phase<float>(a, b, step, stage);
    const float A = flow_amp<float>(a, b);
    cx<float> v0[V], v1[V], v2[V];
    // component c: staged ky rows -> spectral registers -> inverse FFT in y
    auto fetch = [&](cx<float>(&v)[V], int c) {
      const long k = 3 * jg + c;
      cp_async_wait_group1();
      named_bar(1 + grp, GT);   // load k visible to the group; every warp is done with the output staging
      const cx<float>* buf = In + (k & 1) * P * XG;
      cx<float> s[W::SV];
#pragma unroll
      for (int r = 0; r < W::C; ++r) {
        const cx<float>* col = buf + CN::in_at(sl + K, wl * C + r);
#pragma unroll
        for (int q = 0; q < S; ++q) s[r * S + q] = NG::keeps(q, sl) ? col[NG::kofs(q) * XG] : mk(0.f, 0.f);
      }
      named_bar(1 + grp, GT);   // the buffer is read: it takes load k + 2
      load(k + 2);
      W::template s2p<+1>(s, v, lane, B, s_tw);
    };
    fetch(v0, 0);
    fetch(v1, 1);
    fetch(v2, 2);
    // w = u x b at (x, y = m1 + S m2)
    {
      const int m1 = W::phys_m1(lane);
      const float2 csx = s_cs[x0 + wl * C + W::phys_c(lane)];
      const float uy = A * (csx.y * ph.cpx + csx.x * ph.spx);
      const float uzx = csx.x * ph.cpx - csx.y * ph.spx;
#pragma unroll
      for (int p = 0; p < V; ++p) {
        const float2 csy = s_cs[m1 + S * p];
        const float ux = A * (csy.x * ph.cpy - csy.y * ph.spy);
        const float uz = A * (uzx + (csy.y * ph.cpy + csy.x * ph.spy));
        const cx<float> bx = v0[p], by = v1[p], bz = v2[p];
        v0[p] = bz * uy - by * uz;
        v1[p] = bx * uz - bz * ux;
        v2[p] = by * ux - bx * uy;
      }
    }
    // component c: forward FFT in y -> kept ky rows -> staging -> W
    auto emit = [&](cx<float>(&v)[V], int c) {
      cx<float> s[W::SV];
      W::template p2s<-1>(v, s, lane, B, s_tw);
      named_bar(1 + grp, GT);   // the group's transposes are done: their buffers take the output
#pragma unroll
      for (int r = 0; r < W::C; ++r) {
        cx<float>* col = Out + (sl + K) * OP + wl * C + r;
#pragma unroll
        for (int q = 0; q < S; ++q)
          if (NG::keeps(q, sl)) col[NG::kofs(q) * OP] = s[r * S + q];
      }
      named_bar(1 + grp, GT);
      cx<float>* dst = Wo + ((b * 3 + c) * (long)P) * N + x0;
      for (int i = gtid; i < P * H; i += GT) {
        const int h = i % H, j = i / H;
        const cx<float> e0 = Out[j * OP + 2 * h], e1 = Out[j * OP + 2 * h + 1];
        *(float4*)(dst + (long)j * N + 2 * h) = make_float4(e0.x, e0.y, e1.x, e1.y);
      }
      named_bar(1 + grp, GT);   // the staging is read before the next transposes
    };
    emit(v0, 0);
    emit(v1, 1);
    emit(v2, 2);
  }
  cp_async_wait_all();
}

// --------------------------------------------------------------------- row kernel
// A block of three warps owns C ky rows, one warp per component.  The forward transform's
// kept values go to the warp's buffer in wavenumber order, where the curl reads the other
// two components and the stage update runs over consecutive kx on all 32 lanes (22 slots),
// with coalesced accesses of the stage arrays.  The first of them is copied to shared memory by
// cp.async while the row is transformed (its place takes the new stage value), the others are
// brought into L2 meanwhile and loaded by the update.
//
// Stage arrays: stage 0 stores its explicit term f0 alone (in R2's place) and stage 1 forms X1 and
// the accumulators from X and f0 again, the same operations in the same order: a step moves 14
// compact fields through HBM instead of 17 (X | f0; X f0 | R3 R4; R3 R4 | R4; R4 X Xlo | X Xlo).
constexpr int rown_reads(int mode) { return mode == 3 ? 3 : (mode == 4 ? 0 : (mode == 0 ? 1 : 2)); }

template <int MODE>
__device__ __forceinline__ cx<float> rown_update(const StageCoef<float>& q, const StageArrays<float>& sa, long s,
                                                 float g, float dl, const cx<float>* r, cx<float> f,
                                                 cx<float>* xout) {
  const float dt = q.dt;
  if (MODE == 0) {
    sa.R2[s] = f;
    return implicit_solve(r[0] + f * (dt * 0.5f), g);
  }
  if (MODE == 1) {
    const cx<float> x0 = r[0], f0 = r[1], x1 = implicit_solve(x0 + f0 * (dt * 0.5f), g);
    const cx<float> r2 = x0 + f0 * (dt * float(11.0 / 18.0)) - x1 * (dl * float(1.0 / 6.0));
    const cx<float> r3 = x0 + f0 * (dt * float(5.0 / 6.0)) + x1 * (dl * 0.5f);
    const cx<float> r4 = f0 * (dt * 0.25f) - x1 * (dl * 1.5f);
    const cx<float> a[3] = {r2, r3, r4};
    return stage_update_1<1>(q, sa, s, g, dl, a, f, nullptr);
  }
  return stage_update_1<MODE>(q, sa, s, g, dl, r, f, xout);
}

template <int N, int MODE>
struct RowN {
  using G = NarrowGrid<N>;
  using W = typename G::W;
  static constexpr int BLOCK = 96, P = G::P;
  static constexpr int NPRE = rown_reads(MODE), NST = NPRE < 1 ? 0 : 1;   // arrays read, of them staged
  static constexpr int ELEMS = W::C * P, SLOTS = (ELEMS + 31) / 32;
  static_assert(ELEMS <= W::BUF, "the kept values fit the transpose buffer");
  static constexpr int WSM = W::BUF + NST * SLOTS * 32;    // complex per warp
  static constexpr size_t smem = ((size_t)3 * WSM + W::TAB) * sizeof(cx<float>);
  static constexpr int FIT = (int)(233472 / (smem + 1024));
  static constexpr int MINB = FIT > 5 ? 5 : FIT;           // 5: 128 registers a thread
};

template <int N, int MODE>
__global__ void __launch_bounds__(RowN<N, MODE>::BLOCK, RowN<N, MODE>::MINB) rown_kernel(FineArgs a, int store_m) {
  using RN = RowN<N, MODE>;
  using NG = typename RN::G;
  using W = typename RN::W;
  constexpr int K = NG::K, P = NG::P, FULL = NG::FULL, NPRE = RN::NPRE, C = W::C, S = W::S, V = W::V;
  constexpr int SLOTS = RN::SLOTS, ELEMS = RN::ELEMS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1, sl = W::slane(lane);
  cx<float>* Sm = (cx<float>*)smem_raw;
  cx<float>* B = Sm + c * RN::WSM;
  cx<float>* Q = B + W::BUF;                               // [NST][SLOTS][32]: the staged array, then the stage value
  cx<float>* s_tw = Sm + 3 * RN::WSM;
  W::table(s_tw);
  __syncthreads();
  const StageArrays<float> sa = stage_arrays<float>(a);
  const cx<float>* src[3] = {MODE <= 1 ? sa.X : (MODE == 2 ? sa.R3 : sa.R4),
                             MODE == 1 ? sa.R2 : (MODE == 2 ? sa.R4 : sa.X), sa.Xlo};
  // the array holding the state X among src (stages 0, 1 and 3), read from the caller's layout
  // [batch][3][FULL][FULL] in the first step when x_in_full is set
  constexpr int XSRC = MODE <= 1 ? 0 : (MODE == 3 ? 1 : -1);
  const cx<float>* xin = (const cx<float>*)a.x_in_full;
  cx<float>* xout = MODE == 3 ? (cx<float>*)a.x_out_full : nullptr;
  const int npre = MODE == 3 && !sa.lo_valid ? 2 : NPRE;   // before the first step the low part is zero
  const long rows = (long)a.batch * P;
  griddep_wait();    // W (and the stage arrays) come from the predecessors
  for (long r0 = (long)blockIdx.x * C; r0 < rows; r0 += (long)gridDim.x * C) {
    // row i of the block's C rows: field, ky index, offsets of its kept kx = -K in the compact
    // arrays and in the caller's layout, and of its x = 0 in the mixed arrays
    long cb[C], fb[C], mb[C];
    int iy[C];
    long fld[C];
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const long row = r0 + i < rows ? r0 + i : rows - 1;
      fld[i] = row / P;
      iy[i] = (int)(row - fld[i] * P);
      cb[i] = ((fld[i] * 3 + c) * P + iy[i]) * (long)P;
      mb[i] = ((fld[i] * 3 + c) * P + iy[i]) * (long)N;
      fb[i] = ((fld[i] * 3 + c) * FULL + (iy[i] < K ? iy[i] - K + FULL : iy[i] - K)) * (long)FULL;
    }
    const bool last_ok = C == 1 || r0 + C <= rows;         // false: the block's last row is past the end
    // kept element e of the block's rows (slot q, lane): row i and index j of kx = j - K
    auto row_of = [&](int e) { return C == 1 || e < P ? 0 : 1; };
    auto at = [&](const auto& t, int i) { return C == 1 || i == 0 ? t[0] : t[C - 1]; };
    auto valid = [&](int e) { return e < ELEMS && (last_ok || e < P); };
    auto full_at = [&](int i, int j) { return at(fb, i) + (j < K ? j - K + FULL : j - K); };
    cx<float> s[W::SV], v[V];
    if (MODE == 4) {
#pragma unroll
      for (int q = 0; q < SLOTS; ++q) {
        const int e = lane + 32 * q;
        if (valid(e)) {
          const int i = row_of(e), j = e - i * P;
          B[e] = xin ? xin[full_at(i, j)] : sa.X[at(cb, i) + j];
        }
      }
    } else {
      auto addr = [&](int t, int i, int j) {
        return t == XSRC && xin ? xin + full_at(i, j) : src[t] + at(cb, i) + j;
      };
#pragma unroll
      for (int q = 0; q < SLOTS; ++q) {
        const int e = lane + 32 * q;
        if (valid(e)) cp_async8(Q + e, addr(0, row_of(e), e - row_of(e) * P));
      }
      cp_async_commit();
      // the other arrays into L2 meanwhile, a lane a 128-byte line
#pragma unroll
      for (int t = 1; t < NPRE; ++t)
        if (t < npre)
#pragma unroll
          for (int q = 0; q < (ELEMS + 511) / 512; ++q) {
            const int e = 16 * (lane + 32 * q);
            if (valid(e)) prefetch_l2(addr(t, row_of(e), e - row_of(e) * P));
          }
      const cx<float>* Wr = (const cx<float>*)a.W + at(mb, W::phys_c(lane)) + W::phys_m1(lane);
#pragma unroll
      for (int p = 0; p < V; ++p) v[p] = Wr[S * p];
      W::template p2s<-1>(v, s, lane, B, s_tw);            // x -> kx
#pragma unroll
      for (int r = 0; r < W::C; ++r)
#pragma unroll
        for (int k = 0; k < S; ++k)
          if (NG::keeps(k, sl)) B[r * P + sl + K + NG::kofs(k)] = s[r * S + k];
      __syncthreads();                                     // the rows' three components are in place
      cp_async_wait_all();                                 // this lane's staged values
      const float inv_n2 = 1.f / ((float)N * (float)N);
      const cx<float>* B1 = Sm + c1 * RN::WSM;
      const cx<float>* B2 = Sm + c2 * RN::WSM;
      StageCoef<float> sc[C];
      float ky[C], ly[C];
#pragma unroll
      for (int i = 0; i < C; ++i) {
        sc[i] = stage_coef<float>(a, fld[i]);
        ky[i] = (float)(iy[i] - K);
        ly[i] = ky[i] * ky[i] + sc[i].kz * sc[i].kz;
      }
      // the new stage value replaces the staged array, element by element; the others come from L2,
      // a chunk of slots ahead of their use
      constexpr int CH = 6;
      cx<float> nx[2][CH][2];
      auto fetch = [&](int q0, cx<float>(&d)[CH][2]) {
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
          for (int t = 1; t < NPRE; ++t) {
            const int e = lane + 32 * (q0 + k);
            d[k][t - 1] = q0 + k < SLOTS && valid(e) && t < npre ? *addr(t, row_of(e), e - row_of(e) * P) : mk(0.f, 0.f);
          }
      };
      fetch(0, nx[0]);
#pragma unroll
      for (int q0 = 0; q0 < SLOTS; q0 += CH) {
        fetch(q0 + CH, nx[(q0 / CH + 1) & 1]);
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const int q = q0 + k, e = lane + 32 * q;
          if (q < SLOTS && valid(e)) {
            const int i = row_of(e), j = e - i * P;
            const float fkx = (float)(j - K), fky = at(ky, i);
            const StageCoef<float> cf = at(sc, i);
            const float kz = cf.kz;
            const float k1 = (c == 0 ? fky : (c == 1 ? kz : fkx)) * inv_n2;
            const float k2 = (c == 0 ? kz : (c == 1 ? fkx : fky)) * inv_n2;
            const cx<float> f = mul_i(B2[e] * k1 - B1[e] * k2);
            const float lam = (fkx * fkx + at(ly, i)) * cf.inv_rm;
            const float g = fused_gain(cf.dt * 0.5f * lam);
            const cx<float> r[3] = {Q[e], nx[(q0 / CH) & 1][k][0], nx[(q0 / CH) & 1][k][1]};
            Q[e] = rown_update<MODE>(cf, sa, at(cb, i) + j, g, cf.dt * lam, r, f, xout ? xout + full_at(i, j) : nullptr);
          }
        }
      }
      __syncthreads();                                     // the curl is read before B is rewritten
      if (!store_m) continue;                              // uniform over the grid
    }
    __syncwarp();
    const cx<float>* X = MODE == 4 ? B : Q;                // the new stage value in wavenumber order
#pragma unroll
    for (int r = 0; r < W::C; ++r)
#pragma unroll
      for (int k = 0; k < S; ++k)
        s[r * S + k] = NG::keeps(k, sl) ? X[r * P + sl + K + NG::kofs(k)] : mk(0.f, 0.f);
    __syncwarp();
    W::template s2p<+1>(s, v, lane, B, s_tw);              // kx -> x
    const int pc = W::phys_c(lane);
    cx<float>* Mr = (cx<float>*)a.M + at(mb, pc) + W::phys_m1(lane);
    if (last_ok || pc < C - 1) {
#pragma unroll
      for (int p = 0; p < V; ++p) Mr[S * p] = v[p];
    }
  }
}

}  // namespace kd
