// AsymSpec per-step fuse-and-verify on GB300 (sm_103a): host side of the C ABI
// declared in include/asymspec.h, and the launch of its kernels.
//
//   fuse_verify_tma      (kernel_tma.cuh) one cluster per row, each CTA's
//                        slice brought in by chunked 1-D bulk copies, per-row
//                        programs; 16-byte aligned rows where the streaming
//                        kernels do not apply (the row tokens alone, another
//                        delta source).  Its rows are decided, and Algorithm
//                        1's scan run, by decide_rows, a second launch.
//   fuse_verify_row      (kernel_row.cuh) the same decomposition with no
//                        slice in shared memory (pass 1 from HBM, four CTAs
//                        per SM; a second pass from the L2 only for rows whose
//                        decision needs it): the production programs (no
//                        per-row outputs, delta = a - b), also for rows off
//                        the 16-byte boundaries.  Its rows are decided by
//                        decide_blocks.
//   fuse_verify_full     (kernel_full.cuh) the same for the steps that record
//                        row statistics or log-probabilities; decide_full.
//   fuse_verify_xrow     (kernel_xrow.cuh) the cross-family step on the rows
//                        as they are; decide_xrow.
//   fuse_verify_generic  (kernel_generic.cuh) one cluster per row, any
//                        element-aligned input; folds the scan into the same
//                        launch through a per-element ticket in the workspace.
//
// Each reads every logit row from HBM once.
#include <algorithm>
#include <mutex>

#include "device_common.cuh"
#include "kernel_generic.cuh"
#include "kernel_tma.cuh"
#include "kernel_row.cuh"
#include "kernel_full.cuh"
#include "kernel_draft.cuh"
#include "kernel_xvocab.cuh"
#include "kernel_xrow.cuh"
#include "kernels.h"

namespace {

using namespace asymspec_impl;

thread_local int g_last_cuda_error = 0;

int cuda_fail(cudaError_t e) {
  g_last_cuda_error = static_cast<int>(e);
  return ASYMSPEC_ERR_CUDA;
}

constexpr int kTmaPreferredSmem = 113 * 1024;  // two CTAs per SM

struct Plan {
  int kernel;  // ASYMSPEC_KERNEL_*
  int C, W, VE, sh_off, smem;
  int group_stride;  // TMA kernels: floats per row and CTA of group masses
  long long rows;
  long long ctas;  // grid size
  bool vector_path;
  bool row;          // the production row kernel (fuse_verify_row) runs
  bool stoch, edge;  // its mode; its form for rows off the 16-byte boundaries
  bool full;         // the recording row kernel (fuse_verify_full) instead
  int nt;            // threads per CTA (kRowThreads or kTThreads)
};

const void* row_kernel(int dtype, bool stoch, bool edge, bool full) {
  if (full) return dtype == ASYMSPEC_FP32 ? full_kernel_f32(stoch, edge) : full_kernel_bf16(stoch, edge);
  return dtype == ASYMSPEC_FP32 ? row_kernel_f32(stoch, edge) : row_kernel_bf16(stoch, edge);
}


int elt_size(int dtype) { return dtype == ASYMSPEC_FP32 ? 4 : 2; }

long long round_up_ll(long long x, long long a) { return (x + a - 1) / a * a; }

// Cluster sizes tried, in order of preference (8 packs GB300's GPCs best).
constexpr int kClusterOrder[] = {1, 2, 4, 8, 10, 12, 16};

// Generic kernel: first C whose slice fits the preferred size, else C=16.
bool plan_generic(int V, int elt, int VE, int forced_C, Plan* pl) {
  const int shared_bytes = static_cast<int>(sizeof(SharedGeneric));
  auto fill = [&](int C) {
    const long long per = (static_cast<long long>(V) + C - 1) / C;
    const long long W = round_up_ll(per, VE);
    const long long sh_off = round_up_ll(3 * W * elt, 16);
    pl->C = C;
    pl->W = static_cast<int>(W);
    pl->sh_off = static_cast<int>(sh_off);
    pl->smem = static_cast<int>(sh_off + shared_bytes);
    return sh_off + shared_bytes <= kMaxSmem;
  };
  if (forced_C > 0) return fill(forced_C);
  for (int C : kClusterOrder)
    if (fill(C) && pl->sh_off <= kPreferredSliceBytes) return true;
  return fill(16);
}

// TMA kernel: first C whose slice (and shared state) fits two CTAs per SM,
// else the first that fits one; a slice holds at most kMaxRounds vectors
// per thread.
bool plan_tma(int V, int elt, int forced_C, Plan* pl) {
  const int VE = 16 / elt;
  auto fill = [&](int C) {
    const long long per = (static_cast<long long>(V) + C - 1) / C;
    const long long W = round_up_ll(per, VE);
    const int shared_bytes = shared_tma_bytes(C);
    const long long sh_off = round_up_ll(3 * W * elt, 128);
    pl->C = C;
    pl->W = static_cast<int>(W);
    pl->sh_off = static_cast<int>(sh_off);
    pl->smem = static_cast<int>(sh_off + shared_bytes);
    pl->group_stride = kGroupsMax;
    return sh_off + shared_bytes <= kMaxSmem &&
           W / VE <= static_cast<long long>(kMaxRounds) * kTThreads;
  };
  if (forced_C > 0) return fill(forced_C);
  for (int C : kClusterOrder)
    if (fill(C) && pl->smem <= kTmaPreferredSmem) return true;
  for (int C : kClusterOrder)
    if (fill(C)) return true;
  return false;
}

// The production row kernel.  A second pass re-reads its row from the L2, so
// the rows in flight (one per resident cluster) must stay well inside it, while
// fewer CTAs per row give each warp a longer block over which the fixed
// costs of a CTA (its launch, the first loads, the exchange of the pass-1
// records) are spread.  With at least one wave of clusters of 8 (rows x 8 >=
// 4 CTAs x SMs): the smallest C of kRowClusters whose resident clusters
// hold at most kRowL2Budget of rows and whose CTAs fill the chip.  us a step,
// rows in flight:
//   B=64, K=7, V=128256 bf16 stochastic: C=4 70.8, C=5 67.9 (90 MB), C=6 66.5 (75 MB), C=7 67.8,
//     C=8 69.0 (57 MB), C=10 73.6; greedy: C=4 62.1, C=5 60.8, C=6 60.6, C=7 60.8, C=8 62.6
//   B=256, K=4, V=151936 fp32 stochastic: C=10 347, C=12 332 (84 MB), C=16 351 (60 MB)
//   too few CTAs for the chip against enough, K=4, stochastic / greedy: V=128256 bf16 B=16 C=4
//     23.3 / 16.9, C=8 20.6 / 16.5; B=19 C=4 23.8 / 20.2, C=7 21.7 / 18.3; B=22 C=4 25.6 / 22.0,
//     C=6 23.1 / 20.5; V=64000 fp32 B=16 19.6 / 15.3, 18.2 / 14.9 and (the worst of 20) B=22
//     C=4 22.8 / 18.0, C=6 23.5 / 18.6
// (The recording kernel is not held to that: B=12, K=4, V=128256 bf16 greedy C=4 26.6, C=8 30.1.)
// Smaller batches take C = 8: no size is best there, and 8 within 5 % of the best
// where several are measured (us a step):
//   B=8, K=5, V=151936 bf16 stochastic: C=5 18.2, 6 17.6, 7 18.3, 8 17.8, 10 18.0, 12 18.3, 16 17.4;
//     greedy 13.8, 13.6, 14.4, 14.4, 15.1, 14.3, 14.9; recorded (greedy) 23.3, 26.8, 24.9, 23.9,
//     27.0, 27.8, 31.1
//   B=1, K=4, V=32000 fp32 greedy: C=4 5.3, 6 5.3, 8 5.1, 12 5.1, 16 5.1
//   B=4, K=4, V=128256 bf16 stochastic: C=4 12.8, 6 10.9, 8 11.5, 12 10.7, 16 10.2 (the one it loses)
// Rows too wide for C = 8 take the largest that fits (V=151936 fp32, B=4, K=4 stochastic: C=10
// 14.8, 12 14.3, 16 14.9).  The rule does not count how full the last wave is.
// A warp's block takes at most kWalkRounds steps (the decision kernel's draw takes one
// vector of a block per thread).  Only the pass-1 records live in shared memory.
// forced_C: the caller's asymspec_launch_opts.
constexpr int kRowClusters[] = {4, 5, 6, 7, 8, 10, 12, 16};
constexpr double kRowL2Budget = 86.0e6;

struct DeviceShape {
  int device, sms;
  bool ok;
};
DeviceShape device_shape() {
  DeviceShape d{0, 152, false};  // GB300 when no device answers
  int n = 0;
  if (cudaGetDevice(&d.device) == cudaSuccess &&
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d.device) == cudaSuccess && n > 0) {
    d.sms = n;
    d.ok = true;
  }
  cudaGetLastError();
  return d;
}

cudaError_t prepare_kernel(const void* fn, int device);
cudaError_t active_clusters(const void* fn, const Plan& pl, int device, int* out);

bool plan_row(int V, int dtype, bool stoch, bool edge, bool full, int forced_C, long long rows,
              Plan* pl) {
  const int elt = elt_size(dtype);
  const int VE = 16 / elt;
  // (a row off the 16-byte boundaries may touch one vector more than it fills)
  const long long span = edge ? static_cast<long long>(V) + VE - 1 : V;
  auto width = [&](int C) { return round_up_ll((span + C - 1) / C, VE); };
  auto fits = [&](int C) {
    return width(C) / VE <= static_cast<long long>(kWalkRounds) * kRowThreads;
  };
  auto smem = [&](int C) {
    // the warps' rings follow the fixed state and the pushed records
    return (full ? full_shared_bytes(C) : row_shared_bytes(C)) + kRingBytes;
  };
  int C = 0;
  if (forced_C) {
    if (fits(forced_C)) C = forced_C;
  } else {
    const DeviceShape dev = device_shape();
    const long long slots = static_cast<long long>(dev.sms) * (full ? kFullMinBlocks : kRowMinBlocks);
    const double row_bytes = 3.0 * V * elt;
    if (rows * 8 < slots) {
      if (fits(8)) C = 8;
    } else {
      const void* fn = row_kernel(dtype, stoch, edge, full);
      const bool query = dev.ok && prepare_kernel(fn, dev.device) == cudaSuccess;
      for (int c : kRowClusters) {
        if (!fits(c) || (!full && rows * c < slots)) continue;
        // the clusters the device holds at once (an estimate without a device)
        long long resident = slots / c;
        Plan q = *pl;
        q.C = c;
        q.smem = smem(c);
        q.nt = kRowThreads;
        q.kernel = ASYMSPEC_KERNEL_TMA;
        int n = 0;
        if (query && active_clusters(fn, q, dev.device, &n) == cudaSuccess && n > 0) resident = n;
        cudaGetLastError();
        if (static_cast<double>(std::min(rows, resident)) * row_bytes <= kRowL2Budget) {
          C = c;
          break;
        }
      }
    }
    if (!C) {  // nothing within the budget (or no full wave): the largest cluster that fits
      for (int c : kRowClusters)
        if (fits(c)) C = c;
    }
  }
  if (!C) return false;
  pl->C = C;
  pl->W = static_cast<int>(width(C));
  pl->smem = smem(C);
  pl->sh_off = pl->smem - kRingBytes;
  pl->group_stride = kGroupsMax;
  pl->nt = kRowThreads;
  pl->stoch = stoch;
  pl->edge = edge;
  pl->full = full;
  return true;
}

size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

size_t ws_records_bytes(int B, int K) {
  return round_up(static_cast<size_t>(B) * (K + 1) * sizeof(int4), 256);
}

size_t cluster_ws_bytes(int B, int K) {
  return ws_records_bytes(B, K) + round_up(static_cast<size_t>(B) * sizeof(unsigned), 256);
}

// Workspace of the cluster kernels for clusters of C CTAs: the records and
// tickets first (same offsets), then what each row leaves for the decision
// kernel: the row's pass-1 results, one pass-2 record per CTA (staged) or warp
// (streaming) and, from the staged kernel, each CTA's inverse-CDF group masses.
// A workspace may serve calls of other sizes, and of other kernels, whose parts
// lie over these: a call reads nothing but what it wrote itself.  The tickets,
// which have to start at zero, are cleared by the call that uses them
// (asymspec_fuse_verify_ex; fuse_verify_full clears its own).
struct TmaLayout {
  size_t stat, p2rec, groups, total;
};

// group_stride: floats of group masses per row and CTA.
TmaLayout tma_layout(int B, int K, int C, int group_stride = kGroupsMax) {
  TmaLayout L;
  const size_t R = static_cast<size_t>(B) * (K + 1);
  size_t off = cluster_ws_bytes(B, K);
  L.stat = off;
  off += round_up(R * sizeof(RowStat), 256);
  L.p2rec = off;
  // one record per CTA (fuse_verify_tma) or per warp (fuse_verify_row)
  off += round_up(R * C * kRowMaxWarps * sizeof(X2), 256);
  L.groups = off;
  off += round_up(R * C * static_cast<size_t>(group_stride) * sizeof(float), 256);
  L.total = off;
  return L;
}

// What the streaming row kernels could take of a call: delta = a - b, and no
// per-row outputs (fuse_verify_row) or all of what they need (fuse_verify_full);
// the row tokens alone stay with the staged kernel.
struct RowProgram {
  bool ok, stoch, full;
};

// KParams::tail_first: no element's in a grid of one wave (per_sm CTAs an SM),
// else the last ones', as many as the chip holds clusters.
int tail_first(const Plan& pl, int B, int per_sm) {
  const int slots = device_shape().sms * per_sm;
  return pl.ctas > slots ? std::max(0, B - slots / pl.C) : B;
}

// The streaming kernels' grid: a cluster per row (cluster_row); B up to 65535.
dim3 row_grid(const Plan& pl, int B, int K) {
  return dim3(static_cast<unsigned>(pl.C * (K + 1)), static_cast<unsigned>(B));
}

RowProgram row_program(const asymspec_gate_params& gp, bool full, bool tokens) {
  return {(gp.flags & ASYMSPEC_FLAG_DELTA_MASK) == ASYMSPEC_DELTA_AB && (full || !tokens),
          gp.mode == ASYMSPEC_MODE_STOCHASTIC, full};
}

// Rows off the 16-byte boundaries stream too: the generic kernel reads them
// element by element (greedy bf16, K=4: 98 us at B=32, V=100003 against 23
// streaming; 16 against 7 at B=8, V=16385).  That is the shortest row measured, not
// where the two cross: shorter rows keep the generic kernel, unmeasured.
constexpr int kEdgeMinV = 16384;

// How a call's rows lie in memory: every row on a 16-byte boundary; a, b and t
// at the same offset from one; or neither.
enum RowAlign { kRowsAligned, kRowsShifted, kRowsScattered };

int make_plan(int B, int K, int V, int dtype, const asymspec_launch_opts* opts, RowAlign align,
              size_t ws_bytes, RowProgram prog, Plan* pl) {
  const int elt = elt_size(dtype);
  const int forced_C = (opts && opts->cluster_size > 0) ? opts->cluster_size : 0;
  const int forced_kernel = opts ? opts->kernel : 0;
  if (forced_C < 0 || forced_C > 16) return ASYMSPEC_ERR_INVALID_ARG;
  if (forced_kernel != 0 && forced_kernel != ASYMSPEC_KERNEL_GENERIC &&
      forced_kernel != ASYMSPEC_KERNEL_TMA)
    return ASYMSPEC_ERR_INVALID_ARG;
  const bool vec_ok = align == kRowsAligned;
  pl->rows = static_cast<long long>(B) * (K + 1);
  pl->vector_path = vec_ok;
  pl->row = false;
  pl->nt = kTThreads;
  if (ws_bytes < cluster_ws_bytes(B, K)) return ASYMSPEC_ERR_WORKSPACE;
  bool ok = false;
  // (decide_full's grid is (K+1, B): B up to 65535)
  // Greedy and recorded steps stream too (B=64, K=7, V=128256 bf16 greedy:
  // 114 us of staged kernel against 59 us; B=8, K=5, V=151936 bf16 greedy with
  // every row recorded: 48 us a step against 28).  The staged kernel's copy waits are
  // what the test hook shortens, so such calls that set it, or ask for
  // ASYMSPEC_KERNEL_TMA, keep the staged kernel.
  const bool edge = align == kRowsShifted && V >= kEdgeMinV && !forced_kernel;
  const bool streams = prog.ok && ((prog.stoch && !prog.full) ||
                                   (!forced_kernel && !(opts && opts->test_flags)));
  if (forced_kernel != ASYMSPEC_KERNEL_GENERIC && (vec_ok || edge) && streams && B <= 65535 &&
      plan_row(V, dtype, prog.stoch, edge, prog.full, forced_C, pl->rows, pl)) {
    if (ws_bytes >= tma_layout(B, K, pl->C).total) {
      pl->kernel = ASYMSPEC_KERNEL_TMA;
      pl->VE = 16 / elt;
      pl->row = true;
      ok = true;
    } else if (forced_kernel == ASYMSPEC_KERNEL_TMA) {
      return ASYMSPEC_ERR_WORKSPACE;
    }
  }
  if (ok) {
    // the streaming row kernel
  } else if (forced_kernel != ASYMSPEC_KERNEL_GENERIC && vec_ok && plan_tma(V, elt, forced_C, pl)) {
    // the TMA kernel leaves each row's results in the workspace; the generic
    // kernel, which needs only the records and tickets, runs when it is short
    if (ws_bytes >= tma_layout(B, K, pl->C).total) {
      pl->kernel = ASYMSPEC_KERNEL_TMA;
      pl->VE = 16 / elt;
      ok = true;
    } else if (forced_kernel == ASYMSPEC_KERNEL_TMA) {
      return ASYMSPEC_ERR_WORKSPACE;
    }
  } else if (forced_kernel == ASYMSPEC_KERNEL_TMA) {
    return vec_ok ? ASYMSPEC_ERR_TOO_LARGE : ASYMSPEC_ERR_UNSUPPORTED;
  }
  if (!ok) {
    pl->kernel = ASYMSPEC_KERNEL_GENERIC;
    pl->VE = vec_ok ? 16 / elt : 1;
    if (!plan_generic(V, elt, pl->VE, forced_C, pl)) return ASYMSPEC_ERR_TOO_LARGE;
  }
  pl->ctas = pl->rows * pl->C;
  if (pl->ctas > INT_MAX) return ASYMSPEC_ERR_TOO_LARGE;
  return ASYMSPEC_OK;
}

using KernelFn = const void*;  // a __global__ function taking KParams (or SParams)

// sel: the TMA kernel's program set (tma_program_set; 0 = run-time dispatch)
KernelFn pick_kernel(const Plan& pl, int dtype, bool stoch, int sel = 0) {
  if (pl.row) return row_kernel(dtype, pl.stoch, pl.edge, pl.full);
  if (pl.kernel == ASYMSPEC_KERNEL_TMA)
    return dtype == ASYMSPEC_FP32 ? tma_kernel_f32(stoch, sel) : tma_kernel_bf16(stoch, sel);
  return generic_kernel(dtype, pl.vector_path, stoch);
}

KernelFn pick_decide(const Plan& pl, int dtype, bool stoch) {
  if (pl.row && pl.full)
    return dtype == ASYMSPEC_FP32 ? decide_full_f32(stoch, pl.edge)
                                  : decide_full_bf16(stoch, pl.edge);
  if (pl.row)
    return dtype == ASYMSPEC_FP32 ? decide_blocks_f32(stoch, pl.edge)
                                  : decide_blocks_bf16(stoch, pl.edge);
  return dtype == ASYMSPEC_FP32 ? decide_kernel_f32(stoch) : decide_kernel_bf16(stoch);
}

// Per (kernel, device): attributes set once; cluster occupancy cached per
// (cluster size, shared memory size).
std::mutex g_mu;
struct AttrEntry {
  const void* fn;
  int device;
};
AttrEntry g_attr_done[64];
int g_attr_count = 0;
struct OccEntry {
  const void* fn;
  int device, C, smem, clusters;
};
OccEntry g_occ[128];
int g_occ_count = 0;

cudaError_t prepare_kernel(KernelFn fn, int device) {
  std::lock_guard<std::mutex> lock(g_mu);
  const void* f = fn;
  for (int i = 0; i < g_attr_count; ++i)
    if (g_attr_done[i].fn == f && g_attr_done[i].device == device) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  if (g_attr_count < 64) g_attr_done[g_attr_count++] = {f, device};
  return cudaSuccess;
}

// A kernel without clusters whose dynamic shared memory may reach max_bytes
// (the gather's restricted row of t).
cudaError_t prepare_plain_kernel(KernelFn fn, int device, int max_bytes) {
  std::lock_guard<std::mutex> lock(g_mu);
  const void* f = fn;
  for (int i = 0; i < g_attr_count; ++i)
    if (g_attr_done[i].fn == f && g_attr_done[i].device == device) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_bytes);
  if (e != cudaSuccess) return e;
  if (g_attr_count < 64) g_attr_done[g_attr_count++] = {f, device};
  return cudaSuccess;
}

cudaLaunchConfig_t launch_config(const Plan& pl, long long ctas, cudaStream_t stream,
                                 cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = pl.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(pl.kernel == ASYMSPEC_KERNEL_GENERIC ? kThreads : pl.nt);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Clusters of this shape the device holds at once (0 if it cannot).
cudaError_t active_clusters(KernelFn fn, const Plan& pl, int device, int* out) {
  const void* f = fn;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    for (int i = 0; i < g_occ_count; ++i)
      if (g_occ[i].fn == f && g_occ[i].device == device && g_occ[i].C == pl.C &&
          g_occ[i].smem == pl.smem) {
        *out = g_occ[i].clusters;
        return cudaSuccess;
      }
  }
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = launch_config(pl, pl.C, nullptr, attr);  // a grid of one cluster
  int n = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(g_mu);
  if (g_occ_count < 128) g_occ[g_occ_count++] = {f, device, pl.C, pl.smem, n};
  *out = n;
  return cudaSuccess;
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

int check_params(const asymspec_gate_params* gp) {
  if (!(gp->gamma > 0.f && gp->gamma <= 1.f)) return ASYMSPEC_ERR_INVALID_ARG;
  if (!(std::isfinite(gp->beta) && gp->beta >= 0.f)) return ASYMSPEC_ERR_INVALID_ARG;
  if (gp->mode != ASYMSPEC_MODE_GREEDY && gp->mode != ASYMSPEC_MODE_STOCHASTIC)
    return ASYMSPEC_ERR_UNSUPPORTED;
  if (gp->divergence < ASYMSPEC_DIV_JSD || gp->divergence > ASYMSPEC_DIV_LAMBDA)
    return ASYMSPEC_ERR_UNSUPPORTED;
  if (gp->divergence == ASYMSPEC_DIV_LAMBDA && !std::isfinite(gp->lambda))
    return ASYMSPEC_ERR_INVALID_ARG;
  // flags: bits 0-1 the delta source, every other bit reserved
  if ((gp->flags & ~ASYMSPEC_FLAG_DELTA_MASK) != 0) return ASYMSPEC_ERR_INVALID_ARG;
  const int ds = gp->flags & ASYMSPEC_FLAG_DELTA_MASK;
  if (ds != ASYMSPEC_DELTA_AB && ds != ASYMSPEC_DELTA_A && ds != ASYMSPEC_DELTA_TB)
    return ASYMSPEC_ERR_INVALID_ARG;
  return ASYMSPEC_OK;
}

int check_opts(const asymspec_launch_opts* opts) {
  // every kernel runs 256-thread CTAs
  if (opts && opts->block_threads != 0 && opts->block_threads != 256)
    return ASYMSPEC_ERR_INVALID_ARG;
  if (opts && (opts->test_flags & ~ASYMSPEC_TEST_COPY_GIVE_UP) != 0) return ASYMSPEC_ERR_INVALID_ARG;
  if (opts && ((opts->timing_begin == nullptr) != (opts->timing_end == nullptr)))
    return ASYMSPEC_ERR_INVALID_ARG;
  return ASYMSPEC_OK;
}

// The call's inputs and gate.
void set_inputs(KParams* P, const void* a, const void* b, const void* t, const int32_t* tokens,
                const float* probs, const float* unif, int B, int K, int V,
                const asymspec_gate_params& gp) {
  P->a = a;
  P->b = b;
  P->t = t;
  P->tokens = tokens;
  P->dprobs = probs;
  P->unif = unif;
  P->B = B;
  P->K = K;
  P->V = V;
  P->gamma = gp.gamma;
  P->beta = gp.beta;
  P->lambda = gp.lambda;
  P->ln_gamma = logf(gp.gamma);
  P->divergence = gp.divergence;
  P->delta_src = gp.flags & ASYMSPEC_FLAG_DELTA_MASK;
  P->fuse_bonus = gp.fuse_bonus ? 1 : 0;
}

// The caller's timing events around the fused row kernel (asymspec_launch_opts).
cudaError_t record_timing(const asymspec_launch_opts* opts, bool begin, cudaStream_t s) {
  if (!opts || !opts->timing_begin) return cudaSuccess;
  return cudaEventRecord(static_cast<cudaEvent_t>(begin ? opts->timing_begin : opts->timing_end), s);
}

// Scratch of asymspec_fuse_verify_static, used as asymspec_fuse_verify_ex
// uses any workspace.  The generic kernel needs records for
// ASYMSPEC_STATIC_MAX_ROWS rows and tickets for the largest batch that can
// have that many rows (K >= 1, so B <= ASYMSPEC_STATIC_MAX_ROWS / 2): 144 KiB.
// 4 MiB also holds the cluster kernels' per-row results (48 + 576 C bytes a
// row for clusters of C: about 890 rows at C = 8, 1190 at C = 6); larger
// batches take the generic kernel.
constexpr size_t kStaticScratchBytes = ASYMSPEC_STATIC_SCRATCH_BYTES;
static_assert(kStaticScratchBytes >= static_cast<size_t>(ASYMSPEC_STATIC_MAX_ROWS) * sizeof(int4) +
                                         static_cast<size_t>(ASYMSPEC_STATIC_MAX_ROWS / 2) *
                                             sizeof(unsigned),
              "the static scratch holds the generic kernel's records and tickets");
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Device address of g_static_scratch in the current device's context, looked
// up on every call: a cached address would outlive a context that
// cudaDeviceReset tore down (the module, and the array, are loaded again in
// the next context).  Once the module is loaded the lookup is a host-side
// table read; the first lookup in a context may load the module.
constexpr int kMaxDevices = 64;

int static_scratch(void** out) {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
  if (e != cudaSuccess) return cuda_fail(e);
  *out = p;
  return ASYMSPEC_OK;
}

// asymspec_fuse_verify_host: the scratch layout (each part 256-byte aligned)
// and the chunking of the batch.
struct HostLayout {
  int P, Bc;  // chunks, batch elements per chunk (the last may have fewer)
  size_t a, b, t, tok, prob, unif, len, next, ws, ws_each, total;
};

HostLayout host_layout(int B, int K, int V, int dtype) {
  HostLayout L;
  L.Bc = (B + ASYMSPEC_HOST_CHUNKS - 1) / ASYMSPEC_HOST_CHUNKS;
  L.P = (B + L.Bc - 1) / L.Bc;
  const size_t R = static_cast<size_t>(B) * (K + 1);
  const size_t row = static_cast<size_t>(V) * elt_size(dtype);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += round_up(bytes, 256);
    return o;
  };
  L.a = take(R * row);
  L.b = take(R * row);
  L.t = take(R * row);
  L.tok = take(static_cast<size_t>(B) * K * sizeof(int32_t));
  L.prob = take(static_cast<size_t>(B) * K * sizeof(float));
  L.unif = take(R * sizeof(float));
  L.len = take(static_cast<size_t>(B) * sizeof(int32_t));
  L.next = take(static_cast<size_t>(B) * sizeof(int32_t));
  L.ws_each = round_up(asymspec_workspace_bytes(L.Bc, K, V), 256);
  L.ws = take(L.ws_each * L.P);
  L.total = off;
  return L;
}

// Per device: the copy stream and its per-chunk events (created on first use).
struct HostRes {
  cudaStream_t copy;
  cudaEvent_t start;
  cudaEvent_t chunk[ASYMSPEC_HOST_CHUNKS];
  bool ready;
};
std::mutex g_host_mu;
HostRes g_host[kMaxDevices] = {};

int host_resources(HostRes** out) {
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return cuda_fail(e);
  if (device < 0 || device >= kMaxDevices) return ASYMSPEC_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_host_mu);
  HostRes& r = g_host[device];
  if (!r.ready) {
    e = cudaStreamCreateWithFlags(&r.copy, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_fail(e);
    e = cudaEventCreateWithFlags(&r.start, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(e);
    for (int c = 0; c < ASYMSPEC_HOST_CHUNKS; ++c) {
      e = cudaEventCreateWithFlags(&r.chunk[c], cudaEventDisableTiming);
      if (e != cudaSuccess) return cuda_fail(e);
    }
    r.ready = true;
  }
  *out = &r;
  return ASYMSPEC_OK;
}

}  // namespace

extern "C" {

void asymspec_default_gate_params(asymspec_gate_params* p) {
  if (!p) return;
  p->gamma = 0.5f;
  p->beta = 1.0f;
  p->lambda = 0.1f;
  p->mode = ASYMSPEC_MODE_GREEDY;
  p->divergence = ASYMSPEC_DIV_JSD;
  p->fuse_bonus = 0;
  p->flags = 0;
}

size_t asymspec_workspace_bytes(int B, int K, int V) {
  (void)V;
  if (B < 1 || K < 1) return 0;
  // the TMA kernel's layout for the largest cluster
  return tma_layout(B, K, 16).total;
}

int asymspec_workspace_reset(void* workspace, size_t workspace_bytes, void* stream) {
  if (!workspace) return ASYMSPEC_ERR_INVALID_ARG;
  const cudaError_t e =
      cudaMemsetAsync(workspace, 0, workspace_bytes, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ASYMSPEC_OK : cuda_fail(e);
}

int asymspec_plan(int B, int K, int V, int dtype, const asymspec_gate_params* gate_params,
                  const asymspec_launch_opts* opts, asymspec_launch_info* out) {
  if (!out || B < 1 || K < 1 || V < 2) return ASYMSPEC_ERR_INVALID_ARG;
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return ASYMSPEC_ERR_UNSUPPORTED;
  int st = check_opts(opts);
  if (st) return st;
  asymspec_gate_params gp;
  asymspec_default_gate_params(&gp);
  if (gate_params) gp = *gate_params;
  st = check_params(&gp);
  if (st) return st;
  const bool vec_ok = (static_cast<long long>(V) * elt_size(dtype)) % 16 == 0;
  Plan pl = {};
  st = make_plan(B, K, V, dtype, opts, vec_ok ? kRowsAligned : kRowsShifted,
                 asymspec_workspace_bytes(B, K, V), row_program(gp, false, false), &pl);
  if (st) return st;
  out->cluster_size = pl.C;
  out->block_threads = pl.kernel == ASYMSPEC_KERNEL_GENERIC ? kThreads : pl.nt;
  out->slice_elems = pl.W;
  out->smem_bytes = pl.smem;
  out->ctas = pl.ctas;
  out->vector_path = vec_ok ? 1 : 0;
  out->max_active_clusters = 0;
  out->kernel = pl.kernel;
  out->launches = pl.kernel == ASYMSPEC_KERNEL_TMA ? 2 : 1;
  out->row_kernel = pl.row && pl.stoch ? 1 : 0;
  int device = 0;
  if (cudaGetDevice(&device) == cudaSuccess) {
    const bool st_mode = gp.mode == ASYMSPEC_MODE_STOCHASTIC;
    KernelFn fn = pick_kernel(pl, dtype, st_mode,
                              tma_program_set(st_mode, gp.divergence, gp.fuse_bonus != 0, false,
                                              false, gp.flags & ASYMSPEC_FLAG_DELTA_MASK));
    int ncl = 0;
    if (fn && prepare_kernel(fn, device) == cudaSuccess &&
        active_clusters(fn, pl, device, &ncl) == cudaSuccess)
      out->max_active_clusters = ncl;
  }
  cudaGetLastError();
  return ASYMSPEC_OK;
}

int asymspec_fuse_verify_ex(const void* logits_full, const void* logits_comp,
                            const void* logits_ver, const int32_t* draft_tokens,
                            const float* draft_probs, const float* uniforms, int B, int K,
                            int V, int dtype, const asymspec_gate_params* gate_params,
                            int32_t* out_accept_len, int32_t* out_next_token,
                            void* workspace, size_t workspace_bytes, float* out_row_stats,
                            int32_t* out_row_tokens, float* out_fused_logprobs,
                            uint32_t* out_error_word, const asymspec_launch_opts* opts,
                            void* stream) {
  if (B < 1 || K < 1 || V < 2) return ASYMSPEC_ERR_INVALID_ARG;
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return ASYMSPEC_ERR_UNSUPPORTED;
  int st = check_opts(opts);
  if (st) return st;
  asymspec_gate_params gp;
  asymspec_default_gate_params(&gp);
  if (gate_params) gp = *gate_params;
  st = check_params(&gp);
  if (st) return st;
  const bool stoch = gp.mode == ASYMSPEC_MODE_STOCHASTIC;
  if (!logits_full || !logits_comp || !logits_ver || !draft_tokens || !out_accept_len ||
      !out_next_token)
    return ASYMSPEC_ERR_INVALID_ARG;
  if (stoch && (!draft_probs || !uniforms)) return ASYMSPEC_ERR_INVALID_ARG;
  const int elt = elt_size(dtype);
  if (!aligned(logits_full, elt) || !aligned(logits_comp, elt) || !aligned(logits_ver, elt) ||
      !aligned(draft_tokens, 4) || !aligned(out_accept_len, 4) || !aligned(out_next_token, 4) ||
      (draft_probs && !aligned(draft_probs, 4)) || (uniforms && !aligned(uniforms, 4)) ||
      (out_row_stats && !aligned(out_row_stats, 4)) ||
      (out_row_tokens && !aligned(out_row_tokens, 4)) ||
      (out_fused_logprobs && !aligned(out_fused_logprobs, 4)) ||
      (out_error_word && !aligned(out_error_word, 4)))
    return ASYMSPEC_ERR_MISALIGNED;
  if (!workspace || !aligned(workspace, 16)) return ASYMSPEC_ERR_WORKSPACE;
  const auto offset = [](const void* p) { return reinterpret_cast<uintptr_t>(p) % 16; };
  const RowAlign align =
      offset(logits_full) != offset(logits_comp) || offset(logits_full) != offset(logits_ver)
          ? kRowsScattered
      : (static_cast<long long>(V) * elt) % 16 == 0 && !offset(logits_full) ? kRowsAligned
                                                                            : kRowsShifted;
  Plan pl = {};
  st = make_plan(B, K, V, dtype, opts, align, workspace_bytes,
                 row_program(gp, out_row_stats || out_fused_logprobs, out_row_tokens), &pl);
  if (st) return st;

  KParams P = {};
  set_inputs(&P, logits_full, logits_comp, logits_ver, draft_tokens, draft_probs, uniforms, B, K, V,
             gp);
  P.C = pl.C;
  P.W = pl.W;
  P.sh_off = pl.sh_off;
  P.need_lse_s = (stoch || out_fused_logprobs || out_row_stats) ? 1 : 0;
  P.need_pass2 = (stoch || out_fused_logprobs || gp.divergence == ASYMSPEC_DIV_JSD ||
                  gp.divergence == ASYMSPEC_DIV_KL)
                     ? 1
                     : 0;
  P.full = (out_row_stats || out_fused_logprobs) ? 1 : 0;
  P.want_tokens = out_row_tokens ? 1 : 0;
  P.rows = pl.rows;
  P.out_len = out_accept_len;
  P.out_next = out_next_token;
  P.row_stats = out_row_stats;
  P.row_tokens = out_row_tokens;
  P.logprobs = out_fused_logprobs;
  P.err_word = out_error_word;
  P.recs = static_cast<int4*>(workspace);
  P.tma_threads = pl.nt;
  P.head0 = static_cast<int>(offset(logits_full) / elt);
  P.tail_first = pl.row ? tail_first(pl, B, pl.full ? kFullMinBlocks : kRowMinBlocks) : B;
  P.lp_vec = P.head0 == 0 && aligned(out_fused_logprobs, 16) ? 1 : 0;
  // the chunk waits of the TMA kernel: bounded, or (test hook) giving up at once
  P.copy_wait_ns =
      (opts && (opts->test_flags & ASYMSPEC_TEST_COPY_GIVE_UP)) ? 0ull : kCopyTimeoutNs;
  P.tickets = reinterpret_cast<unsigned int*>(static_cast<char*>(workspace) +
                                              ws_records_bytes(B, K));

  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return cuda_fail(e);
  KernelFn fn = pick_kernel(pl, dtype, stoch,
                            tma_program_set(stoch, gp.divergence, gp.fuse_bonus != 0, P.full != 0,
                                            P.want_tokens != 0, P.delta_src));
  if (!fn) return ASYMSPEC_ERR_UNSUPPORTED;
  e = prepare_kernel(fn, device);
  if (e != cudaSuccess) return cuda_fail(e);
  const long long ctas = pl.ctas;  // one cluster of C CTAs per row
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = launch_config(pl, ctas, static_cast<cudaStream_t>(stream), attr);
  if (pl.row) cfg.gridDim = row_grid(pl, B, K);
  void* args[] = {&P};
  P.group_stride = pl.group_stride;
  if (pl.kernel == ASYMSPEC_KERNEL_TMA) {
    char* base = static_cast<char*>(workspace);
    const TmaLayout L = tma_layout(B, K, pl.C, pl.group_stride);
    P.row_stat = base + L.stat;
    P.pass2_rec = reinterpret_cast<float*>(base + L.p2rec);
    P.group_mass = reinterpret_cast<float*>(base + L.groups);
  } else {
    // Cleared by every call: another call's results may lie there.  (us a greedy
    // step in calls, before -> after: B=1, K=4, V=4099 bf16 14.4 -> 15.1, B=8, K=5,
    // V=1001 10.4 -> 12.4; 3 us in a graph.)
    e = cudaMemsetAsync(P.tickets, 0, static_cast<size_t>(B) * sizeof(unsigned), cfg.stream);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  e = record_timing(opts, true, cfg.stream);
  if (e == cudaSuccess) e = cudaLaunchKernelExC(&cfg, fn, args);
  if (e == cudaSuccess) e = record_timing(opts, false, cfg.stream);
  if (e != cudaSuccess) return cuda_fail(e);
  if (pl.kernel == ASYMSPEC_KERNEL_TMA) {
    // the rows' decisions and Algorithm 1's scan: one CTA per batch element
    // (per row after the recording kernel), as a programmatic dependent launch: its launch overlaps the row
    // kernel's last CTAs, and it waits (griddepcontrol.wait) for that kernel
    const int threads = !pl.row              ? 32 * std::min(K + 1, kDecideThreads / 32)
                        : pl.full && !stoch ? 32
                                            : kDrawThreads;
    const KernelFn dfn = pick_decide(pl, dtype, stoch);
    cudaLaunchConfig_t dcfg = {};
    cudaLaunchAttribute dattr[1];
    dattr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    dattr[0].val.programmaticStreamSerializationAllowed = 1;
    dcfg.gridDim = pl.row && pl.full ? dim3(static_cast<unsigned>(K + 1), static_cast<unsigned>(B))
                                     : dim3(static_cast<unsigned>(B));
    dcfg.blockDim = dim3(threads);
    dcfg.stream = static_cast<cudaStream_t>(stream);
    dcfg.attrs = dattr;
    dcfg.numAttrs = 1;
    e = cudaLaunchKernelExC(&dcfg, dfn, args);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  return ASYMSPEC_OK;
}

int asymspec_fuse_verify(const void* logits_full, const void* logits_comp,
                         const void* logits_ver, const int32_t* draft_tokens,
                         const float* draft_probs, const float* uniforms, int B, int K,
                         int V, int dtype, const asymspec_gate_params* gate_params,
                         int32_t* out_accept_len, int32_t* out_next_token, void* stream) {
  if (B < 1 || K < 1 || V < 2) return ASYMSPEC_ERR_INVALID_ARG;
  const size_t bytes = asymspec_workspace_bytes(B, K, V);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  void* ws = nullptr;
  cudaError_t e = cudaMallocAsync(&ws, bytes, s);
  if (e != cudaSuccess) return cuda_fail(e);
  const int st = asymspec_fuse_verify_ex(logits_full, logits_comp, logits_ver, draft_tokens,
                                         draft_probs, uniforms, B, K, V, dtype, gate_params,
                                         out_accept_len, out_next_token, ws, bytes, nullptr,
                                         nullptr, nullptr, nullptr, nullptr, stream);
  e = cudaFreeAsync(ws, s);
  if (st != ASYMSPEC_OK) return st;
  if (e != cudaSuccess) return cuda_fail(e);
  return ASYMSPEC_OK;
}

int asymspec_fuse_verify_static(const void* logits_full, const void* logits_comp,
                                const void* logits_ver, const int32_t* draft_tokens,
                                const float* draft_probs, const float* uniforms, int B, int K,
                                int V, int dtype, const asymspec_gate_params* gate_params,
                                int32_t* out_accept_len, int32_t* out_next_token,
                                void* stream) {
  if (B < 1 || K < 1 || V < 2) return ASYMSPEC_ERR_INVALID_ARG;
  if (static_cast<long long>(B) * (K + 1) > ASYMSPEC_STATIC_MAX_ROWS)
    return ASYMSPEC_ERR_SCRATCH_LIMIT;
  void* scratch = nullptr;
  int st = static_scratch(&scratch);
  if (st) return st;
  return asymspec_fuse_verify_ex(logits_full, logits_comp, logits_ver, draft_tokens,
                                 draft_probs, uniforms, B, K, V, dtype, gate_params,
                                 out_accept_len, out_next_token, scratch, kStaticScratchBytes,
                                 nullptr, nullptr, nullptr, nullptr, nullptr, stream);
}

size_t asymspec_host_scratch_bytes(int B, int K, int V, int dtype) {
  if (B < 1 || K < 1 || V < 2) return 0;
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return 0;
  return host_layout(B, K, V, dtype).total;
}

int asymspec_fuse_verify_host(const void* h_logits_full, const void* h_logits_comp,
                              const void* h_logits_ver, const int32_t* h_draft_tokens,
                              const float* h_draft_probs, const float* h_uniforms, int B, int K,
                              int V, int dtype, const asymspec_gate_params* gate_params,
                              int32_t* h_out_accept_len, int32_t* h_out_next_token,
                              void* d_scratch, size_t scratch_bytes, void* stream) {
  if (B < 1 || K < 1 || V < 2) return ASYMSPEC_ERR_INVALID_ARG;
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return ASYMSPEC_ERR_UNSUPPORTED;
  asymspec_gate_params gp;
  asymspec_default_gate_params(&gp);
  if (gate_params) gp = *gate_params;
  int st = check_params(&gp);
  if (st) return st;
  const bool stoch = gp.mode == ASYMSPEC_MODE_STOCHASTIC;
  if (!h_logits_full || !h_logits_comp || !h_logits_ver || !h_draft_tokens ||
      !h_out_accept_len || !h_out_next_token)
    return ASYMSPEC_ERR_INVALID_ARG;
  if (stoch && (!h_draft_probs || !h_uniforms)) return ASYMSPEC_ERR_INVALID_ARG;
  const HostLayout L = host_layout(B, K, V, dtype);
  if (!d_scratch || !aligned(d_scratch, 256) || scratch_bytes < L.total)
    return ASYMSPEC_ERR_WORKSPACE;
  HostRes* r = nullptr;
  st = host_resources(&r);
  if (st) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* base = static_cast<char*>(d_scratch);
  const size_t row = static_cast<size_t>(V) * elt_size(dtype);
  const int K1 = K + 1;
  // the copies start after everything already on `stream` (which may still
  // read this scratch), then run back to back on the copy stream
  cudaError_t e = cudaEventRecord(r->start, s);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(r->copy, r->start, 0);
  if (e != cudaSuccess) return cuda_fail(e);
  auto h2d = [&](size_t dst, const void* src, size_t off, size_t bytes) {
    return cudaMemcpyAsync(base + dst + off, static_cast<const char*>(src) + off, bytes,
                           cudaMemcpyHostToDevice, r->copy);
  };
  for (int c = 0; c < L.P && e == cudaSuccess; ++c) {
    const int b0 = c * L.Bc, nb = std::min(L.Bc, B - b0);
    const size_t r0 = static_cast<size_t>(b0) * K1, nr = static_cast<size_t>(nb) * K1;
    e = h2d(L.a, h_logits_full, r0 * row, nr * row);
    if (e == cudaSuccess) e = h2d(L.b, h_logits_comp, r0 * row, nr * row);
    if (e == cudaSuccess) e = h2d(L.t, h_logits_ver, r0 * row, nr * row);
    if (e == cudaSuccess)
      e = h2d(L.tok, h_draft_tokens, static_cast<size_t>(b0) * K * 4, static_cast<size_t>(nb) * K * 4);
    if (stoch && e == cudaSuccess)
      e = h2d(L.prob, h_draft_probs, static_cast<size_t>(b0) * K * 4, static_cast<size_t>(nb) * K * 4);
    if (stoch && e == cudaSuccess) e = h2d(L.unif, h_uniforms, r0 * 4, nr * 4);
    if (e == cudaSuccess) e = cudaEventRecord(r->chunk[c], r->copy);
  }
  if (e != cudaSuccess) {
    cudaStreamSynchronize(r->copy);
    return cuda_fail(e);
  }
  // each chunk's step on `stream` once its copies have landed
  for (int c = 0; c < L.P; ++c) {
    const int b0 = c * L.Bc, nb = std::min(L.Bc, B - b0);
    const size_t r0 = static_cast<size_t>(b0) * K1;
    char* ws = base + L.ws + static_cast<size_t>(c) * L.ws_each;
    e = cudaStreamWaitEvent(s, r->chunk[c], 0);
    if (e != cudaSuccess) {
      cudaStreamSynchronize(r->copy);
      return cuda_fail(e);
    }
    int32_t* d_len = reinterpret_cast<int32_t*>(base + L.len) + b0;
    int32_t* d_next = reinterpret_cast<int32_t*>(base + L.next) + b0;
    st = asymspec_fuse_verify_ex(
        base + L.a + r0 * row, base + L.b + r0 * row, base + L.t + r0 * row,
        reinterpret_cast<const int32_t*>(base + L.tok) + static_cast<size_t>(b0) * K,
        stoch ? reinterpret_cast<const float*>(base + L.prob) + static_cast<size_t>(b0) * K : nullptr,
        stoch ? reinterpret_cast<const float*>(base + L.unif) + r0 : nullptr, nb, K, V, dtype, &gp,
        d_len, d_next, ws, L.ws_each, nullptr, nullptr, nullptr, nullptr, nullptr, stream);
    if (st != ASYMSPEC_OK) {
      cudaStreamSynchronize(r->copy);
      return st;
    }
    e = cudaMemcpyAsync(h_out_accept_len + b0, d_len, static_cast<size_t>(nb) * 4,
                        cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(h_out_next_token + b0, d_next, static_cast<size_t>(nb) * 4,
                          cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) {
      cudaStreamSynchronize(r->copy);
      return cuda_fail(e);
    }
  }
  return ASYMSPEC_OK;
}

int asymspec_draft_sample(const void* logits, int rows, int V, int dtype, int mode,
                          const float* uniforms, int32_t* out_tokens, float* out_probs,
                          int cluster_size, void* stream) {
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return ASYMSPEC_ERR_UNSUPPORTED;
  if (mode != ASYMSPEC_MODE_GREEDY && mode != ASYMSPEC_MODE_STOCHASTIC)
    return ASYMSPEC_ERR_UNSUPPORTED;
  if (rows < 0 || V < 2) return ASYMSPEC_ERR_INVALID_ARG;
  if (cluster_size != 0 && cluster_size != 1 && cluster_size != 2 && cluster_size != 4 &&
      cluster_size != kDMaxCluster)
    return ASYMSPEC_ERR_INVALID_ARG;
  if (V > ASYMSPEC_DRAFT_MAX_V || rows > (1 << 27)) return ASYMSPEC_ERR_TOO_LARGE;
  if (rows == 0) return ASYMSPEC_OK;
  const bool stoch = mode == ASYMSPEC_MODE_STOCHASTIC;
  if (!logits || !out_tokens || !out_probs || (stoch && !uniforms)) return ASYMSPEC_ERR_INVALID_ARG;
  const int elt = elt_size(dtype);
  if (!aligned(logits, elt) || !aligned(out_tokens, 4) || !aligned(out_probs, 4) ||
      (stoch && !aligned(uniforms, 4)))
    return ASYMSPEC_ERR_MISALIGNED;
  const bool edge = (static_cast<long long>(V) * elt) % 16 != 0 || !aligned(logits, 16);
  const int VE = 16 / elt;
  // (a row off the 16-byte boundaries may touch one vector more than it fills)
  const int nv = edge ? (V + 2 * VE - 2) / VE : V / VE;
  int C = cluster_size;
  if (C == 0) {
    int device = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return cuda_fail(e);
    // the smallest C that gives every SM three CTAs (of the four it holds): a
    // CTA's start and its reductions cost about 5 us, so more, smaller ones
    // lose.  Measured (us, bf16 V=128256, sampling; C = 1, 2, 4, 8): 512 rows
    // 28.5 29.6 30.8 39.0, 256 rows 17.8 17.0 18.7 22.2, 64 rows 13.3 9.2 7.9
    // 8.0; 128 rows of fp32 V=151936 25.4 19.2 18.8 19.6
    C = 1;
    while (C < kDMaxCluster && static_cast<long long>(rows) * C < 3LL * sms &&
           (nv + 2 * C - 1) / (2 * C) >= 512)
      C *= 2;
  }
  DParams P;
  P.logits = logits;
  P.unif = stoch ? uniforms : nullptr;
  P.tokens = out_tokens;
  P.probs = out_probs;
  P.rows = rows;
  P.V = V;
  P.head0 = static_cast<int>(reinterpret_cast<uintptr_t>(logits) % 16) / elt;
  P.W = (nv + C - 1) / C;
  // sampling: one float of group mass per warp and round of a slice
  const size_t smem =
      kDRingBytes +
      (stoch ? static_cast<size_t>((P.W + kDThreads - 1) / kDThreads) * kDWarps * sizeof(float) : 0);
  const void* fn = draft_kernel_ptr(dtype, edge, stoch);
  cudaError_t e = cudaSuccess;
  if (smem > 47 * 1024)  // (beside the static shared memory: 48 KB without it)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return cuda_fail(e);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(static_cast<long long>(rows) * C));
  cfg.blockDim = dim3(kDThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = static_cast<cudaStream_t>(stream);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {&P};
  e = cudaLaunchKernelExC(&cfg, fn, args);
  return e == cudaSuccess ? ASYMSPEC_OK : cuda_fail(e);
}

}  // extern "C"

// ------------------------------------------------- cross-family vocabularies

namespace {

// Scratch of asymspec_xvocab_gather, each part 256-byte aligned: inv_d[V_d],
// inv_v[V_v] (int32) and the map-error word.
struct XScratch {
  size_t inv_d, inv_v, err, total;
};

XScratch xvocab_scratch_layout(int V_d, int V_v) {
  XScratch L;
  L.inv_d = 0;
  L.inv_v = round_up(static_cast<size_t>(V_d) * sizeof(int32_t), 256);
  L.err = L.inv_v + round_up(static_cast<size_t>(V_v) * sizeof(int32_t), 256);
  L.total = L.err + 256;
  return L;
}

// Workspace of asymspec_fuse_verify_xvocab, each part 256-byte aligned: the
// restricted rows a', b', t' ([B, K+1, S] each), the emitted pair indices
// ([B] int32), the gather's scratch, then the step's own workspace for a
// vocabulary of S entries.
struct XLayout {
  size_t ga, gb, gt, idx, scratch, scratch_bytes, step, step_bytes, total;
};

XLayout xvocab_layout(int B, int K, int S, int V_d, int V_v, int dtype) {
  XLayout L;
  const size_t plane = round_up(static_cast<size_t>(B) * (K + 1) * S * elt_size(dtype), 256);
  L.ga = 0;
  L.gb = plane;
  L.gt = 2 * plane;
  L.idx = 3 * plane;
  L.scratch = L.idx + round_up(static_cast<size_t>(B) * sizeof(int32_t), 256);
  L.scratch_bytes = xvocab_scratch_layout(V_d, V_v).total;
  L.step = L.scratch + L.scratch_bytes;
  L.step_bytes = asymspec_workspace_bytes(B, K, S);
  L.total = L.step + L.step_bytes;
  return L;
}

// The map check: inverse maps built with atomicCAS, the map-error word.
cudaError_t map_check(const int32_t* md, const int32_t* mv, int S, int Vd, int Vv, char* scratch,
                      uint32_t* ew, cudaStream_t st) {
  const XScratch XL = xvocab_scratch_layout(Vd, Vv);
  int* inv_d = reinterpret_cast<int*>(scratch + XL.inv_d);
  int* inv_v = reinterpret_cast<int*>(scratch + XL.inv_v);
  unsigned* merr = reinterpret_cast<unsigned*>(scratch + XL.err);
  void* fargs[] = {&inv_d, &Vd, &inv_v, &Vv, &merr};
  const int vmax = std::max(Vd, Vv);
  const cudaError_t e =
      cudaLaunchKernel(xvocab_inv_fill_ptr(), dim3((vmax + 255) / 256), dim3(256), fargs, 0, st);
  if (e != cudaSuccess) return e;
  void* bargs[] = {&md, &mv, &S, &inv_d, &Vd, &inv_v, &Vv, &merr, &ew};
  return cudaLaunchKernel(xvocab_inv_build_ptr(), dim3((S + 255) / 256), dim3(256), bargs, 0, st);
}

// The one-kernel cross-family step: clusters of C <= 4 CTAs (128 warp records
// a row), one CTA an SM, each with its share of a restricted row of t in
// shared memory.  C by the time of rows C CTAs in waves of one an SM: a CTA's
// is about 0.4 + 0.6 / C of a whole row's (every CTA reads the whole row of t
// and the inverse map), and 1.4 times that when its share leaves the L1 less
// than about 60 KB.  Measured (us a step; C = 1, 2, 3, 4):
//   512 rows, S=109568 bf16: 215 187 247 285    160 rows, S=93793 bf16: 79 83 94 100
//   320 rows, S=105622 fp32: - 185 144 157       80 rows: - 94 60 67
//    20 rows, S=93793 bf16: 41 29 26 25           5 rows, S=64000: 27 21 20 19
// False: the gather and the step on its output run instead.
bool plan_xrow(int S, int elt, long long rows, int sms, Plan* pl) {
  double best = 0.0;
  for (int C = 1; C <= 4; ++C) {
    const int W = static_cast<int>(round_up_ll((static_cast<long long>(S) + C - 1) / C, kXVec));
    const long long smem = xrow_shared_bytes(C) + static_cast<long long>(W) * elt;
    // (a warp's block of pairs is at most what the decision kernel's draw takes)
    if (smem > kMaxSmem ||
        row_block_vectors(W / kXVec, kXRowWarps) > kDrawThreads)
      continue;
    const double waves = static_cast<double>((rows * C + sms - 1) / sms);
    const double cost = waves * (0.4 + 0.6 / C) * (smem > 160 * 1024 ? 1.4 : 1.0);
    if (best > 0.0 && cost >= best) continue;
    best = cost;
    pl->C = C;
    pl->W = W;
    pl->sh_off = xrow_shared_bytes(C);
    pl->smem = static_cast<int>(smem);
    pl->nt = kXRowThreads;
  }
  pl->ctas = rows * pl->C;
  return best > 0.0;
}

// The map check, the row kernel (a programmatic dependent: it fetches its
// rows into the L2 meanwhile) and the decision kernel.  step_ws: a workspace
// of the step for S entries.
int run_xrow(const Plan& pl, const void* a, const void* b, int V_d, const void* t, int V_v,
             const int32_t* map_d, const int32_t* map_v, int S, const int32_t* draft_index,
             const float* probs, const float* unif, int B, int K, int dtype,
             const asymspec_gate_params& gp, int32_t* out_len, int32_t* out_next, int32_t* out_index,
             char* scratch, char* step_ws, uint32_t* err_word, cudaStream_t st) {
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return cuda_fail(e);
  const bool stoch = gp.mode == ASYMSPEC_MODE_STOCHASTIC;
  const KernelFn fn =
      dtype == ASYMSPEC_FP32 ? xrow_kernel_f32(stoch) : xrow_kernel_bf16(stoch);
  const KernelFn dfn = dtype == ASYMSPEC_FP32 ? decide_xrow_f32(stoch) : decide_xrow_bf16(stoch);
  e = prepare_kernel(fn, device);
  if (e != cudaSuccess) return cuda_fail(e);
  const TmaLayout TL = tma_layout(B, K, 16);
  const XScratch XL = xvocab_scratch_layout(V_d, V_v);
  KParams P = {};
  set_inputs(&P, a, b, t, draft_index, probs, unif, B, K, S, gp);
  P.C = pl.C;
  P.W = pl.W;
  P.sh_off = pl.sh_off;
  const long long rows = static_cast<long long>(B) * (K + 1);
  P.rows = rows;
  P.tail_first = tail_first(pl, B, 1);
  P.out_len = out_len;
  P.out_next = out_next;
  P.err_word = err_word;
  P.recs = reinterpret_cast<int4*>(step_ws);
  P.row_stat = step_ws + TL.stat;
  P.pass2_rec = reinterpret_cast<float*>(step_ws + TL.p2rec);
  XRowParams X;
  X.map_d = map_d;
  X.map_v = map_v;
  X.inv_v = reinterpret_cast<const int*>(scratch + XL.inv_v);
  X.map_err = reinterpret_cast<const unsigned*>(scratch + XL.err);
  X.out_index = out_index;
  X.V_d = V_d;
  X.V_v = V_v;
  X.t_vec = aligned(t, 16) && (static_cast<size_t>(V_v) * elt_size(dtype)) % 16 == 0 ? 1 : 0;
  X.idx2 = aligned(map_d, 8) ? 1 : 0;
  e = map_check(map_d, map_v, S, V_d, V_v, scratch, err_word, st);
  if (e != cudaSuccess) return cuda_fail(e);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = pl.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = row_grid(pl, B, K);
  cfg.blockDim = dim3(pl.nt);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  void* args[] = {&P, &X};
  e = cudaLaunchKernelExC(&cfg, fn, args);
  if (e != cudaSuccess) return cuda_fail(e);
  cudaLaunchConfig_t dcfg = {};
  dcfg.gridDim = dim3(static_cast<unsigned>(B));
  dcfg.blockDim = dim3(kDrawThreads);
  dcfg.stream = st;
  dcfg.attrs = attr + 1;
  dcfg.numAttrs = 1;
  e = cudaLaunchKernelExC(&dcfg, dfn, args);
  return e == cudaSuccess ? ASYMSPEC_OK : cuda_fail(e);
}

}  // namespace

extern "C" {

size_t asymspec_xvocab_gather_scratch_bytes(int V_d, int V_v) {
  if (V_d < 1 || V_v < 1) return 0;
  return xvocab_scratch_layout(V_d, V_v).total;
}

size_t asymspec_xvocab_workspace_bytes(int B, int K, int S, int V_d, int V_v, int dtype) {
  if (B < 1 || K < 1 || S < 2 || V_d < 1 || V_v < 1) return 0;
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return 0;
  return xvocab_layout(B, K, S, V_d, V_v, dtype).total;
}

int asymspec_xvocab_gather(const void* logits_full, const void* logits_comp, int V_d,
                           const void* logits_ver, int V_v, const int32_t* map_d,
                           const int32_t* map_v, int S, int rows, int dtype, void* out_full,
                           void* out_comp, void* out_ver, uint32_t* out_error_word,
                           void* scratch, size_t scratch_bytes, void* stream) {
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return ASYMSPEC_ERR_UNSUPPORTED;
  if (rows < 0 || S < 2 || V_d < 1 || V_v < 1) return ASYMSPEC_ERR_INVALID_ARG;
  if (rows == 0) return ASYMSPEC_OK;
  if (!logits_full || !logits_comp || !logits_ver || !map_d || !map_v || !out_full ||
      !out_comp || !out_ver)
    return ASYMSPEC_ERR_INVALID_ARG;
  const int elt = elt_size(dtype);
  if (!aligned(logits_full, elt) || !aligned(logits_comp, elt) || !aligned(logits_ver, elt) ||
      !aligned(out_full, elt) || !aligned(out_comp, elt) || !aligned(out_ver, elt) ||
      !aligned(map_d, 4) || !aligned(map_v, 4) || (out_error_word && !aligned(out_error_word, 4)))
    return ASYMSPEC_ERR_MISALIGNED;
  const XScratch XL = xvocab_scratch_layout(V_d, V_v);
  if (scratch && (!aligned(scratch, 256) || scratch_bytes < XL.total)) return ASYMSPEC_ERR_WORKSPACE;
  const long long ycount = (static_cast<long long>(rows) + kXRows - 1) / kXRows;
  if (ycount > 65535) return ASYMSPEC_ERR_TOO_LARGE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  if (scratch) {
    e = map_check(map_d, map_v, S, V_d, V_v, static_cast<char*>(scratch), out_error_word, st);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  XGatherParams P;
  P.inv_v = scratch ? reinterpret_cast<const int*>(static_cast<char*>(scratch) + XL.inv_v) : nullptr;
  P.map_err =
      scratch ? reinterpret_cast<const unsigned*>(static_cast<char*>(scratch) + XL.err) : nullptr;
  P.a = logits_full;
  P.b = logits_comp;
  P.t = logits_ver;
  P.map_d = map_d;
  P.map_v = map_v;
  P.ga = out_full;
  P.gb = out_comp;
  P.gt = out_ver;
  P.err_word = out_error_word;
  P.rows = rows;
  P.V_d = V_d;
  P.V_v = V_v;
  P.S = S;
  const dim3 grid(static_cast<unsigned>((S + kXThreads * kXJ - 1) / (kXThreads * kXJ)),
                  static_cast<unsigned>(ycount));
  void* args[] = {&P};
  // t built in shared memory through the inverse map (its map may be in any
  // order) when the caller gave the scratch (where the map check builds the
  // inverse map), every row of t starts on a 16-byte boundary and a
  // restricted row fits in one CTA's shared memory; a and b (and otherwise
  // t) through global memory
  // (one CTA per row; a restricted row larger than a CTA's shared memory is
  // cut into parts, each CTA reading the whole row of t for its part)
  int parts = 1;
  while (parts < 16 && ((static_cast<size_t>(S) + parts - 1) / parts + 8) * elt >
                           static_cast<size_t>(kMaxSmem))
    ++parts;
  const size_t row_out = ((static_cast<size_t>(S) + parts - 1) / parts + 8) * elt;
  const bool inv_t = scratch && row_out <= static_cast<size_t>(kMaxSmem) &&
                     aligned(logits_ver, 16) && (static_cast<size_t>(V_v) * elt) % 16 == 0;
  e = cudaLaunchKernel(xvocab_gather_ptr(dtype, !inv_t), grid, dim3(kXThreads), args, 0, st);
  if (e != cudaSuccess) return cuda_fail(e);
  if (inv_t) {
    const KernelFn fn = xvocab_gather_inv_ptr(dtype);
    int device = 0;
    e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = prepare_plain_kernel(fn, device, kMaxSmem);
    if (e == cudaSuccess) {
      // a programmatic dependent of the a/b gather, which it does not read:
      // the two gathers overlap (the map check before them is complete)
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.gridDim = dim3(static_cast<unsigned>(rows), static_cast<unsigned>(parts));
      cfg.blockDim = dim3(kXInvThreads);
      cfg.dynamicSmemBytes = round_up(row_out, 16);
      cfg.stream = st;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      e = cudaLaunchKernelExC(&cfg, fn, args);
    }
  }
  return e == cudaSuccess ? ASYMSPEC_OK : cuda_fail(e);
}

int asymspec_fuse_verify_xvocab(const void* logits_full, const void* logits_comp, int V_d,
                                const void* logits_ver, int V_v, const int32_t* map_d,
                                const int32_t* map_v, int S, const int32_t* draft_index,
                                const float* draft_probs, const float* uniforms, int B, int K,
                                int dtype, const asymspec_gate_params* gate_params,
                                int32_t* out_accept_len, int32_t* out_next_token,
                                int32_t* out_next_index, void* workspace,
                                size_t workspace_bytes, uint32_t* out_error_word, void* stream) {
  if (B < 1 || K < 1 || S < 2 || V_d < 1 || V_v < 1) return ASYMSPEC_ERR_INVALID_ARG;
  if (dtype != ASYMSPEC_FP32 && dtype != ASYMSPEC_BF16) return ASYMSPEC_ERR_UNSUPPORTED;
  asymspec_gate_params gp;
  asymspec_default_gate_params(&gp);
  if (gate_params) gp = *gate_params;
  int st = check_params(&gp);
  if (st) return st;
  if (!draft_index || !out_accept_len || !out_next_token) return ASYMSPEC_ERR_INVALID_ARG;
  if (gp.mode == ASYMSPEC_MODE_STOCHASTIC && (!draft_probs || !uniforms))
    return ASYMSPEC_ERR_INVALID_ARG;
  if (!aligned(out_next_token, 4) || !aligned(out_accept_len, 4) ||
      (out_next_index && !aligned(out_next_index, 4)))
    return ASYMSPEC_ERR_MISALIGNED;
  const XLayout L = xvocab_layout(B, K, S, V_d, V_v, dtype);
  if (!workspace || !aligned(workspace, 256) || workspace_bytes < L.total)
    return ASYMSPEC_ERR_WORKSPACE;
  char* base = static_cast<char*>(workspace);
  int32_t* idx = out_next_index ? out_next_index : reinterpret_cast<int32_t*>(base + L.idx);
  const long long rows = static_cast<long long>(B) * (K + 1);
  const int elt = elt_size(dtype);
  Plan pl = {};
  if ((gp.flags & ASYMSPEC_FLAG_DELTA_MASK) == ASYMSPEC_DELTA_AB &&
      B <= 65535 && rows <= 8LL * 65535 &&
      plan_xrow(S, elt, rows, device_shape().sms, &pl)) {
    if (!logits_full || !logits_comp || !logits_ver || !map_d || !map_v) return ASYMSPEC_ERR_INVALID_ARG;
    if (!aligned(logits_full, elt) || !aligned(logits_comp, elt) || !aligned(logits_ver, elt) ||
        !aligned(map_d, 4) || !aligned(map_v, 4) || (out_error_word && !aligned(out_error_word, 4)) ||
        !aligned(draft_index, 4) || (draft_probs && !aligned(draft_probs, 4)) ||
        (uniforms && !aligned(uniforms, 4)))
      return ASYMSPEC_ERR_MISALIGNED;
    return run_xrow(pl, logits_full, logits_comp, V_d, logits_ver, V_v, map_d, map_v, S,
                    draft_index, draft_probs, uniforms, B, K, dtype, gp, out_accept_len,
                    out_next_token, idx, base + L.scratch, base + L.step, out_error_word,
                    static_cast<cudaStream_t>(stream));
  }
  st = asymspec_xvocab_gather(logits_full, logits_comp, V_d, logits_ver, V_v, map_d, map_v, S,
                              B * (K + 1), dtype, base + L.ga, base + L.gb, base + L.gt,
                              out_error_word, base + L.scratch, L.scratch_bytes, stream);
  if (st) return st;
  st = asymspec_fuse_verify_ex(base + L.ga, base + L.gb, base + L.gt, draft_index, draft_probs,
                               uniforms, B, K, S, dtype, &gp, out_accept_len, idx,
                               base + L.step, L.step_bytes, nullptr, nullptr, nullptr,
                               out_error_word, nullptr, stream);
  if (st) return st;
  int32_t* next = out_next_token;
  int32_t* len = out_accept_len;
  const int32_t* mv = map_v;
  const unsigned* merr =
      reinterpret_cast<const unsigned*>(base + L.scratch + xvocab_scratch_layout(V_d, V_v).err);
  int S_ = S, B_ = B;
  void* args[] = {&idx, &mv, &S_, &B_, &merr, &len, &next};
  const cudaError_t e = cudaLaunchKernel(xvocab_emit_ptr(), dim3((B + 255) / 256), dim3(256),
                                         args, 0, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? ASYMSPEC_OK : cuda_fail(e);
}

const char* asymspec_status_string(int status) {
  switch (status) {
    case ASYMSPEC_OK: return "ok";
    case ASYMSPEC_ERR_INVALID_ARG: return "invalid argument";
    case ASYMSPEC_ERR_UNSUPPORTED: return "unsupported dtype, mode, divergence or kernel";
    case ASYMSPEC_ERR_MISALIGNED: return "pointer not aligned to its element size";
    case ASYMSPEC_ERR_WORKSPACE: return "workspace missing or too small";
    case ASYMSPEC_ERR_CUDA: return "CUDA error (see asymspec_last_cuda_error)";
    case ASYMSPEC_ERR_TOO_LARGE: return "problem too large for the on-chip row slices";
    case ASYMSPEC_ERR_SCRATCH_LIMIT:
      return "B*(K+1) exceeds ASYMSPEC_STATIC_MAX_ROWS (8192), the static scratch of "
             "asymspec_fuse_verify_static; use asymspec_fuse_verify_ex with a workspace";
    default: return "unknown status";
  }
}

int asymspec_last_cuda_error(void) { return g_last_cuda_error; }

int asymspec_version(void) { return 200; }

}  // extern "C"
