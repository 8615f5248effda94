// Launches of the persistent fused fine propagator (kd_fused.cuh).
#include <mutex>

#include "kd_fine.h"
#include "kd_fused.cuh"

namespace kd {

bool fused_covers(int K, int scheme) { return scheme == SCHEME_RK443 && K >= 1 && 2 * K + 2 <= 192; }

namespace {

constexpr int kShapes[] = {1, 2, 3, 4, 6, 8, 12, 16};   // blocks a cluster
constexpr int kNShapes = 8;
constexpr size_t kMaxSmem = 232448;                     // shared memory a block may opt in to

template <typename T, int L, int R>
int run_spread(const FineArgs& a, const StepCfg& cfg, int s, int e);

// A kernel with the threads (0: the shape does not fit) and shared memory of its blocks.
template <typename T, int L, int R>
struct LaneKernel {
  using F = FusedStep<T, L, R>;
  static constexpr auto kernel = fused_kernel<T, L, R>;
  // Fields for which the passes run as launches of their own (0: never).  An SM has few FP64 units
  // and a field has 16 SMs at most in a cluster, so that up to seven fields take what one takes.  192^2
  // complex128, us a step of 1, 4, 8, 12, 24 fields, clusters | launches: 1070 1072 1323 2071 4131 |
  // 640 776 1007 1334 2616.  More fields gain less (40: 4934 | 4140), for room in W that grows with them.
  // In complex64 the launches' latencies take what the units would give (54 55 75 88 141 | 49 56 81
  // 114 198).
  static constexpr int SPREAD = L * R == 192 && sizeof(T) == 8 ? kSpreadFields : 0;
  static int spread(const FineArgs& a, const StepCfg& cfg, int s, int e) { return run_spread<T, L, R>(a, cfg, s, e); }
  static int threads(int P, int CS) { return F::N % CS == 0 && F::smem(P, CS) <= kMaxSmem ? 32 * F::warps(P, CS) : 0; }
  static size_t smem(int P, int CS) { return F::smem(P, CS); }
};
cudaLaunchConfig_t config(int CS, int clusters, int threads, size_t smem, cudaStream_t st, bool pdl,
                          cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(CS * clusters), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)CS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cfg;
}

// Clusters of the shape that the current device runs at once (0: it does not fit), asked of the
// runtime once per device, kept set and shape.
template <class KT>
int active_clusters(int P, int shape) {
  static std::mutex m;
  static short cache[16][96][kNShapes];          // [device][K][shape], 0: not asked yet, else clusters + 1
  int dev = 0;
  cudaGetDevice(&dev);
  const int K = (P - 1) / 2, CS = kShapes[shape];
  std::lock_guard<std::mutex> lock(m);
  if (dev < 16 && cache[dev][K][shape]) return cache[dev][K][shape] - 1;
  int n = 0;
  const int th = KT::threads(P, CS);
  if (th > 0) {
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t cfg = config(CS, 1, th, KT::smem(P, CS), nullptr, false, at);
    if (cudaOccupancyMaxActiveClusters(&n, KT::kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
  }
  if (dev < 16) cache[dev][K][shape] = (short)(n < 32000 ? n + 1 : 32000);
  return n;
}

// Steps [s, e) of the fields of a, a launch a pass (fused_kernel); returns the launches, negative on failure.
template <typename T, int L, int R>
int run_spread(const FineArgs& a, const StepCfg& cfg, int s, int e) {
  constexpr int N = L * R;
  cudaLaunchAttribute at[2];
  auto pass = [&](int kid, int tasks, auto kernel, size_t smem, int step, int stage, bool more) {
    cudaLaunchConfig_t lc = config(1, 1, 32, smem, cfg.st, cfg.pdl, at);
    lc.gridDim = dim3((unsigned)tasks, (unsigned)a.batch, 1);
    if (cfg.probe) cfg.probe->before(cfg.probe->user, kid);
    if (cudaLaunchKernelEx(&lc, kernel, a, (int)more, step, stage) != cudaSuccess) return false;
    if (cfg.probe) cfg.probe->after(cfg.probe->user, kid);
    return true;
  };
  auto cols = fused_kernel<T, L, R, FUSED_COLS>;
  auto rows = fused_kernel<T, L, R, FUSED_ROWS>;
  if (!pass(1, a.P, rows, 0, s, 4, true)) return -1;
  for (int st = s; st < e; ++st)
    for (int j = 0; j < 4; ++j)
      if (!pass(0, N, cols, N * sizeof(cx<T>), st, j, true) || !pass(1, a.P, rows, 0, st, j, st + 1 < e || j < 3))
        return -1;
  return 1 + 8 * (e - s);
}

// Blocks a cluster for a batch: the shape with the least waves (co / CS + 1/8 + co CS / 400), co
// blocks sharing an SM.  A step of one field takes about that part of a constant: its work splits
// over the blocks, its barriers and latencies do not, and the barriers grow with the blocks
// (128^2 complex64, us a step: 141, 75, 47, 29, 23 for CS = 1, 2, 4, 8, 16).  So a few fields take
// the largest clusters, a large batch the smallest that hold the field (64 fields of 128^2: 75 us
// at CS = 2; 95 at 4, two blocks an SM; 142 at 8, four waves; 64 of 64^2: 22 at 2, 24 at 4, 36 at 16).
template <class KT>
int shape_for(int P, int batch) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 148;
  int best = 0;
  double best_t = 0.0;
  for (int i = 0; i < kNShapes; ++i) {
    const int CS = kShapes[i], cap = active_clusters<KT>(P, i);
    if (cap <= 0) continue;
    const int at_once = batch < cap ? batch : cap, co = (at_once * CS + sms - 1) / sms;
    const double t = (double)((batch + cap - 1) / cap) * ((double)co / CS + 0.125 + co * CS / 400.0);
    if (!best || t < best_t) {
      best = CS;
      best_t = t;
    }
  }
  return best;
}

template <class KT>
cudaError_t prepare_one() {
  cudaError_t e = cudaFuncSetAttribute(KT::kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(KT::kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <class KT>
int run_one(const FineArgs& a0, const StepCfg& cfg) {
  int launches = 0;
  FineArgs a = a0;
  // fields leave the batch as their steps run out (cfg.active: a shrinking prefix): one launch
  // for every run of steps with the same fields
  for (int s = 0; s < cfg.nsteps;) {
    int e = cfg.nsteps;
    if (cfg.active) {
      a.batch = cfg.active[s];
      if (a.batch <= 0) break;
      e = s + 1;
      while (e < cfg.nsteps && cfg.active[e] == a.batch) ++e;
    }
    if constexpr (KT::SPREAD > 0) {
      if (a.batch <= KT::SPREAD && a.w_len >= 3L * a.P * KT::F::N * a.batch) {
        const int r = KT::spread(a, cfg, s, e);
        if (r < 0) return -1;
        launches += r;
        s = e;
        continue;
      }
    }
    const int CS = shape_for<KT>(a.P, a.batch);
    if (CS == 0) return -1;
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t lc = config(CS, a.batch, KT::threads(a.P, CS), KT::smem(a.P, CS), cfg.st, cfg.pdl, at);
    if (cfg.probe) cfg.probe->before(cfg.probe->user, 1);
    if (cudaLaunchKernelEx(&lc, KT::kernel, a, CS, s, e - s) != cudaSuccess) return -1;
    if (cfg.probe) cfg.probe->after(cfg.probe->user, 1);
    ++launches;
    s = e;
  }
  return launches;
}

// f(kernel) for the kernel of the kept set K: the smallest N >= 2K + 2 points.  complex128 takes
// 16 x 1 and 32 x 1 instead of 8 x 3 points for the smallest sets: an FP64 instruction costs an SM's
// quarter 64 cycles whatever its lanes do, so a third of the values a lane is a third of the time for
// the few fields of such a grid (8 fields of 32^2: 57 us a step against 142; 16^2 on 16 | 32 points: 1
// field 46 | 57, 100 59 | 201, 300 131 | 459, which the kernels of kd_fine2.cuh take in 129, 145, 198).
template <typename T, class Fn>
auto with_kernel(int K, Fn&& f) {
  const int m = 2 * K + 2;
  if constexpr (sizeof(T) == 8) {
    if (m <= 16) return f(LaneKernel<T, 16, 1>());
    if (m <= 32) return f(LaneKernel<T, 32, 1>());
  } else {
    if (m <= 24) return f(LaneKernel<T, 8, 3>());
  }
  if (m <= 48) return f(LaneKernel<T, 16, 3>());
  if (m <= 96) return f(LaneKernel<T, 32, 3>());
  if (m <= 128) return f(LaneKernel<T, 32, 4>());
  return f(LaneKernel<T, 32, 6>());
}

template <typename T>
cudaError_t prepare_T(int K) {
  auto prep = [](auto k) { return prepare_one<decltype(k)>(); };
  if (K > 0) return 2 * K + 2 <= 192 ? with_kernel<T>(K, prep) : cudaSuccess;
  for (int k : {5, 10, 20, 40, 60, 90}) {
    const cudaError_t e = with_kernel<T>(k, prep);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
int run_T(const FineArgs& a, const StepCfg& cfg) {
  return with_kernel<T>(a.K, [&](auto k) { return run_one<decltype(k)>(a, cfg); });
}

}  // namespace

cudaError_t fused_prepare(int prec, int K) { return prec == 0 ? prepare_T<float>(K) : prepare_T<double>(K); }

int fused_run(int prec, const FineArgs& a, const StepCfg& cfg) {
  return prec == 0 ? run_T<float>(a, cfg) : run_T<double>(a, cfg);
}

}  // namespace kd
