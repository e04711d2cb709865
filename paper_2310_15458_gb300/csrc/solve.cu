// Applying the factorization (Section 2.5): x = W_1 .. W_K A_top^{-1} V_K .. V_1 b.
//
// Upward sweep, boxes in factor order (each colour class in one launch):
//   b_R <- L_R^{-1} P_R (b_R - T^* b_S);  b_C -= E b_R                 (apply V)
// dense top solve, then the downward sweep in reverse order:
//   y_R <- U_R^{-1} (y_R - F y_C);  y_S -= T y_R                       (apply W)
// Boxes of one colour class touch disjoint entries of x, so a class is one
// launch; the right-hand sides are split into chunks of RC columns.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <sstream>
#include <type_traits>

#include <cooperative_groups.h>

#include "internal.h"
#include "tw_common.cuh"
#include "tw_plan.h"

namespace {

constexpr int NT = 256;

#include "sweep.cuh"

// The working copy of the right-hand sides: point g (tree order), column q at
// x[g * ldx + q], so that whatever gathers the points of a box reads whole lines.
// Tiles of 32 points x 32 columns go through shared memory (one column: straight).
template <typename T>
__global__ void __launch_bounds__(NT) k_perm_in(const T* __restrict__ b, int64_t ldb, T* __restrict__ x, int64_t n,
                                                int nrhs, const int* __restrict__ u2t) {
  __shared__ __align__(16) unsigned char s_raw[sizeof(T) * 32 * 33];
  T* tile = reinterpret_cast<T*>(s_raw);
  pdl_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (nrhs == 1) {
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n; i += (int64_t)gridDim.x * NT) x[u2t[i]] = b[i];
    return;
  }
  const int64_t ct = (nrhs + 31) / 32, tiles = ((n + 31) / 32) * ct;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t i0 = (t / ct) * 32;
    const int j0 = (int)(t % ct) * 32, jw = min(32, nrhs - j0);
    __syncthreads();
    for (int j = warp; j < jw; j += NT / 32)
      if (i0 + lane < n) tile[lane * 33 + j] = b[i0 + lane + (int64_t)(j0 + j) * ldb];
    __syncthreads();
    for (int i = warp; i < 32; i += NT / 32)
      if (i0 + i < n && lane < jw) x[(int64_t)u2t[i0 + i] * nrhs + j0 + lane] = tile[i * 33 + lane];
  }
}

template <typename T>
__global__ void __launch_bounds__(NT) k_perm_out(T* __restrict__ b, int64_t ldb, const T* __restrict__ x, int64_t n,
                                                 int nrhs, const int* __restrict__ u2t, const int* __restrict__ err) {
  __shared__ __align__(16) unsigned char s_raw[sizeof(T) * 32 * 33];
  T* tile = reinterpret_cast<T*>(s_raw);
  pdl_wait();
  // a wait of the sweeps that ran out (*err != 0) voids the result: every entry
  // becomes NaN rather than a silently wrong number
  const bool bad = err != nullptr && *(const volatile int*)err != 0;
  const T nan = from_re<T>(__longlong_as_double(0x7FF8000000000000LL));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (nrhs == 1) {
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n; i += (int64_t)gridDim.x * NT)
      b[i] = bad ? nan : ld_l2(x + u2t[i]);
    return;
  }
  const int64_t ct = (nrhs + 31) / 32, tiles = ((n + 31) / 32) * ct;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t i0 = (t / ct) * 32;
    const int j0 = (int)(t % ct) * 32, jw = min(32, nrhs - j0);
    __syncthreads();
    for (int i = warp; i < 32; i += NT / 32)
      if (i0 + i < n && lane < jw) tile[i * 33 + lane] = ld_l2(x + (int64_t)u2t[i0 + i] * nrhs + j0 + lane);
    __syncthreads();
    for (int j = warp; j < jw; j += NT / 32)
      if (i0 + lane < n) b[i0 + lane + (int64_t)(j0 + j) * ldb] = bad ? nan : tile[lane * 33 + j];
  }
}

#include "sweep_tc.cuh"

// Right-hand sides from which a call takes the tensor-core sweeps.  16 complex columns at
// 256^2: 6.9 ms against 14.7 in FP64; 16 real ones: 3.2 ms against 4.1 (with the classes
// of fewer than TCMIN boxes, where four launches of the products take longer than one of
// the FP64 sweep, left to the latter; at 64^2 every class).  From TCB on a real factor
// keeps its digits, which a first call builds, and the classes that fit take the products,
// below TCL columns but the smallest (tw_takes).
constexpr int TCN = 16, TCB = 32, TCL = 64, TCMIN = 16;

// Top block: x_top <- A_top^{-1} x_top with the inverse formed at factor time.
template <typename T>
__global__ void k_top_gather(const int* __restrict__ idx, int n, const T* __restrict__ x, int64_t ldx, int nrhs,
                             T* __restrict__ z) {
  pdl_launch();
  pdl_wait();
  const long long tot = (long long)n * nrhs;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e % n);
    const long long q = e / n;
    z[e] = ld_l2(x + idx[i] * ldx + q);
  }
}

// 32 rows per CTA, the columns in SW_NT / 32 consecutive parts (one warp each)
// whose sums are added in order
template <typename T, int RC>
__global__ void __launch_bounds__(SW_NT) k_top_gemv(const T* __restrict__ Ainv, const int* __restrict__ idx, int n,
                                                    const T* __restrict__ z, T* __restrict__ x, int64_t ldx, int nrhs) {
  constexpr int W = SW_NT / 32;
  __shared__ __align__(16) unsigned char s_ps[sizeof(T) * W * 32 * RC];
  T* ps = reinterpret_cast<T*>(s_ps);
  pdl_launch();
  const int q0 = blockIdx.y * RC, nq = min(RC, nrhs - q0);
  const int lane = threadIdx.x % 32, w = threadIdx.x / 32, i = blockIdx.x * 32 + lane;
  const int nw = (n + W - 1) / W, j1 = min(n, (w + 1) * nw);
  pdl_wait();
  T acc[RC];
#pragma unroll
  for (int q = 0; q < RC; ++q) acc[q] = zero<T>();
  if (i < n) {
#pragma unroll 8
    for (int j = w * nw; j < j1; ++j) {
      const T av = Ainv[i + (size_t)j * n];
#pragma unroll
      for (int q = 0; q < RC; ++q)
        if (q < nq) acc[q] = mad(acc[q], av, ld_l2(z + j + (int64_t)(q0 + q) * n));
    }
  }
#pragma unroll
  for (int q = 0; q < RC; ++q) ps[(w * RC + q) * 32 + lane] = acc[q];
  __syncthreads();
  for (int e = threadIdx.x; e < RC * 32; e += SW_NT) {
    const int l = e % 32, q = e / 32, row = blockIdx.x * 32 + l;
    T s = ps[q * 32 + l];
#pragma unroll
    for (int p = 1; p < W; ++p) s = s + ps[(p * RC + q) * 32 + l];
    if (row < n && q < nq) x[idx[row] * ldx + q0 + q] = s;
  }
}

// Workspace of the sweeps for nrhs right-hand sides in chunks of rc columns: four
// ints at bar_off (grid barrier counters and the timeout flag of the persistent
// sweeps) and the gathered top block.
struct SweepWs {
  size_t bar_off = 0, topz_off = 0, bytes = 0;
};

template <typename T> SweepWs sweep_ws(const rss_factorization* f, int64_t nrhs, int rc) {
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  SweepWs w;
  w.topz_off = w.bar_off + al(sizeof(int) * 4);
  w.bytes = w.topz_off + al(sizeof(T) * (size_t)f->ntop * cdiv(nrhs, rc) * rc);
  return w;
}

// A launch that may start while the launch before it on the stream still runs; its
// kernel waits for that one (pdl_wait) before it touches the right-hand sides.
// cluster > 1: that many CTAs along x form a thread-block cluster.
template <typename... KA, typename... A>
cudaError_t launch_pdl(void (*kern)(KA...), dim3 grid, int threads, size_t smem, cudaStream_t st, int cluster, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KA>(args)...);
}

// Slices of C of a colour class in the downward sweep, and the most CTAs a box gets:
// a property of the class alone, so that sums do not depend on the call.
int sweep_slices(int nrec) {
  int q = 1;
  while (q < SW_QMAX && nrec * q <= 8 * 152) q *= 2;
  return q;
}

int rhs_chunk(int64_t nrhs) { return nrhs == 1 ? 1 : nrhs <= 4 ? 4 : 8; }

// Top block: x_top <- A_top^{-1} x_top (gathered, one product, scattered back).
template <typename T, int RC>
rss_status top_apply(const rss_factorization* f, T* x, int64_t ldx, int nrhs, cudaStream_t st, T* topz) {
  if (f->ntop <= 0) return RSS_OK;
  const unsigned nz = cdiv(nrhs, RC);
  const unsigned g = std::min<long long>(cdiv((long long)f->ntop * nrhs, 256), 152LL * 8);
  RSS_CUDA(launch_pdl(k_top_gather<T>, dim3(g), 256, 0, st, 1, f->d_top_idx, f->ntop, x, ldx, nrhs, topz));
  RSS_CUDA(launch_pdl(k_top_gemv<T, RC>, dim3(cdiv(f->ntop, 32), nz), SW_NT, 0, st, 1,
                      static_cast<const T*>(f->d_top_inv), f->d_top_idx, f->ntop, topz, x, ldx, nrhs));
  return RSS_OK;
}

// The two persistent launches of the FP64 sweeps (k_sweep) around the top
// block.  Shared memory: the most any class needs without staging its matrices, at
// least 48 KB, so that small boxes stage theirs (16, 32, 48, 100 KB: one column at 1024^2
// 4.64, 4.56, 4.50, 5.32 ms); the grid: as many clusters as fit on the device at once (a
// cooperative launch needs all of them resident).
constexpr int SWP_POLLS = 1 << 24;

template <typename T, int RC> size_t sweep_persistent_smem(const rss_factorization* f, int k0) {
  size_t need = 0;
  for (size_t i = k0; i < f->batches.size(); ++i) {
    const Batch& b = f->batches[i];
    const int qc = sweep_slices(b.nrec), Q = qc == SW_QMAX ? SW_QMAX : 1;
    need = std::max({need, sweep_sm_up<T, RC>(b.max_n, b.max_r, b.max_c, Q).need,
                     sweep_sm_down<T, RC>(b.max_n, b.max_r, b.max_c, Q, qc).need});
  }
  const size_t smem = std::max(need * sizeof(T), size_t(48) << 10);
  return (smem + 1023) & ~size_t(1023);
}

// One persistent launch (k_sweep) over the colour classes k0 .. end of the
// factor order: upward in that order, or downward in reverse.
template <typename T, int RC>
rss_status sweep_persistent_launch(const rss_factorization* f, T* x, int64_t ldx, int nrhs, cudaStream_t st,
                                   unsigned* bar, int k0, bool up) {
  const size_t smem = sweep_persistent_smem<T, RC>(f, k0);
  int dev = 0, sms = 0;
  RSS_CUDA(cudaGetDevice(&dev));
  RSS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SwpArgs<T> a;
  a.cls = static_cast<const SwpClass<T>*>(f->d_swp) + k0;
  a.ncls = (int)f->batches.size() - k0;
  a.x = x;
  a.ldx = ldx;
  a.nrhs = nrhs;
  a.bar = bar;
  a.err = reinterpret_cast<int*>(bar + 2);
  a.polls = wait_limit(f->params.wait_polls, SWP_POLLS);
  a.sm_cap = (int)(smem / sizeof(T));
  void* args[] = {&a};
  const void* fn = up ? reinterpret_cast<const void*>(k_sweep<T, RC, true>)
                      : reinterpret_cast<const void*>(k_sweep<T, RC, false>);
  RSS_CUDA(allow_smem(fn));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(SW_QMAX);
  cfg.blockDim = dim3(SWP_NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = SW_QMAX;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  int clusters = 0;
  RSS_CUDA(cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg));
  if (f->swp_ctas > 0) clusters = std::min(clusters, f->swp_ctas * sms / SW_QMAX);
  if (clusters < 1) {
    rss_set_error("rss_solve: the persistent sweep kernel does not fit an SM");
    return RSS_ECUDA;
  }
  cfg.gridDim = dim3(clusters * SW_QMAX);
  RSS_CUDA(cudaLaunchKernelExC(&cfg, fn, args));
  return RSS_OK;
}

// First colour class of the persistent part of the sweeps: the whole factor
// (form 2), the tail of classes with fewer than f->swp_tail_boxes boxes each
// (form 3), or none (per-class kernels; also when the device or the factor's
// box sizes do not allow the cooperative launch).
template <typename T, int RC> int sweep_persistent_start(const rss_factorization* f) {
  const int nb = (int)f->batches.size();
  if (!f->d_swp || nb == 0 || (f->swp_launch != 2 && f->swp_launch != 3)) return nb;
  int k0 = 0;
  if (f->swp_launch == 3) {
    k0 = nb;
    while (k0 > 0 && f->batches[k0 - 1].nrec < f->swp_tail_boxes) --k0;
  }
  if (k0 == nb || sweep_persistent_smem<T, RC>(f, k0) > (size_t(200) << 10)) return nb;
  int dev = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return nb;
  }
  return k0;
}

// One colour class of the FP64 sweeps: Q CTAs per box, at most as many as the class
// has slices.  Fewer boxes (times column chunks) than SMs: a cluster per box, at most
// two CTAs to an SM, its matrices staged.  More: CTAs that stage nothing, many to an SM,
// since the memory latency is then hidden by their number (one column at 1024^2: 4.0 ms so,
// 4.9 with the same classes staged; at 64^2, where every class is small, 0.26 ms staged and
// 0.40 not).  Boxes too large for either matrix to be staged count as many: alone on their
// SMs for nothing, such CTAs took 5.5 instead of 3.0 ms (one column, 512^2, leaf 256).
// Unstaged CTAs of 256 threads, so that a box is shared by fewer, but of 128 where boxes
// hold at most 40 points (128 threads everywhere, then this, ms: 15 columns, 512^2, leaf 256
// 24.8, 23.1; 1024^2 32.9, 31.7; one column, 1024^2 4.0, 3.7; 256 threads everywhere, 15
// columns, 512^2, leaf 4: 8.2 instead of 7.9).  The columns are taken in smaller chunks
// where a box's vectors would not fit (the sums do not depend on any of this).
template <typename T, int RC, bool UP>
rss_status sweep_class(const Batch& b, T* x, int64_t ldx, int nrhs, cudaStream_t st) {
  constexpr size_t MOST = 220 * 1024 / sizeof(T);   // scalars
  const long long nz = cdiv(nrhs, RC);
  const int qc = sweep_slices(b.nrec);
  const bool large = b.max_n > 40;
  bool staged = b.nrec * nz <= 152;
  int Q = 1;
  auto split = [&](int per_sm) {
    while (Q < qc && b.nrec * nz * Q * 2 <= per_sm * 152) Q *= 2;
    return UP ? sweep_sm_up<T, RC>(b.max_n, b.max_r, b.max_c, Q) : sweep_sm_down<T, RC>(b.max_n, b.max_r, b.max_c, Q, qc);
  };
  SweepSm s = {};
  if (staged) {
    s = split(2);
    staged = s.one <= MOST;
  }
  if (!staged) s = split(!large ? 12 : RC == 1 ? 4 : 8);
  if (s.need > MOST) {
    if constexpr (RC > 1) {
      return sweep_class<T, RC == 8 ? 4 : 1, UP>(b, x, ldx, nrhs, st);
    } else {
      rss_set_error("rss_solve: a box's sweep needs more shared memory than an SM has");
      return RSS_EINVAL;
    }
  }
  const size_t smem = (staged ? std::min(s.full, MOST) : s.need) * sizeof(T);
  RSS_CUDA(allow_smem(k_sweep_cl<T, RC, UP>));
  RSS_CUDA(launch_pdl(k_sweep_cl<T, RC, UP>, dim3(b.nrec * Q, (unsigned)nz), staged || large ? SW_NT : 128, smem, st, Q,
                      static_cast<const BoxRec<T>*>(b.d_recs), x, ldx, nrhs, Q, qc, (int)(smem / sizeof(T))));
  return RSS_OK;
}

template <typename T, int RC>
rss_status sweeps(const rss_factorization* f, T* x, int64_t ldx, int nrhs, cudaStream_t st, void* ws) {
  const SweepWs w = sweep_ws<T>(f, nrhs, RC);
  char* wb = static_cast<char*>(ws);
  T* topz = reinterpret_cast<T*>(wb + w.topz_off);
  // classes k0 .. end go through the persistent launches (none, all, or the
  // coarse tail), the others through the per-class kernels
  const int nb = (int)f->batches.size();
  const int k0 = sweep_persistent_start<T, RC>(f);
  unsigned* bar = reinterpret_cast<unsigned*>(wb + w.bar_off);
  for (int bi = 0; bi < k0; ++bi) {
    const rss_status s = sweep_class<T, RC, true>(f->batches[bi], x, ldx, nrhs, st);
    if (s != RSS_OK) return s;
  }
  if (k0 < nb) {
    const rss_status sp = sweep_persistent_launch<T, RC>(f, x, ldx, nrhs, st, bar, k0, true);
    if (sp != RSS_OK) return sp;
  }
  {
    const rss_status stp = top_apply<T, RC>(f, x, ldx, nrhs, st, topz);
    if (stp != RSS_OK) return stp;
  }
  if (k0 < nb) {
    const rss_status sp = sweep_persistent_launch<T, RC>(f, x, ldx, nrhs, st, bar, k0, false);
    if (sp != RSS_OK) return sp;
  }
  for (int bi = k0 - 1; bi >= 0; --bi) {
    const rss_status s = sweep_class<T, RC, false>(f->batches[bi], x, ldx, nrhs, st);
    if (s != RSS_OK) return s;
  }
  return RSS_OK;
}

// The digits of a real factor's matrices for the tensor-core sweeps: built once per
// factor by the first solve that needs them (on its stream, which it then waits for),
// kept until the factor is freed.  They take more than twice the matrices' bytes; where the
// device has not that much left (RSS_ENOMEM), a solve cuts them per call.
bool tw_fits(const Batch& b, bool real) { return tw_shape_fits(b.max_n, b.max_r, b.max_c, real); }
// whether a class takes the tensor-core products in a call with nrhs right-hand sides
// (real classes of at most four boxes of 129 to 192 points: FP64 below TCL; 128^2, eps
// 1e-9: 32 columns 2.64 ms so, 2.77 with products; boxes of 256 points, 64^2: 1.83 and 1.51)
bool tw_takes(const Batch& b, int64_t nrhs, bool real) {
  if (!tw_fits(b, real)) return false;
  if (!real || nrhs >= TCL) return true;
  if (b.nrec <= 4 && b.max_n > TW_M && b.max_n <= 192) return false;
  return nrhs >= TCB || b.nrec >= TCMIN;
}
struct SliceSize {
  size_t dig[4], eb[4];
};
SliceSize slice_size(const BoxRec<double>& R, int kx) {   // kx: entries of K of a stretch
  auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
  const int n = R.k + R.r, rows[4] = {R.r, R.c, R.r, n}, inner[4] = {n, R.r, R.c, R.r};
  SliceSize s;
  for (int op = 0; op < 4; ++op) {
    s.dig[op] = al(tw_cache_bytes(rows[op], inner[op]));
    s.eb[op] = al(sizeof(int) * rows[op] * ((inner[op] + kx - 1) / kx));
  }
  return s;
}

size_t slice_total(const rss_factorization* f) {
  auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
  size_t total = 0;
  for (size_t bi = 0; bi < f->batches.size(); ++bi) {
    const Batch& b = f->batches[bi];
    const BoxRec<double>* hr = static_cast<const BoxRec<double>*>(f->rec_host[bi]);
    total += al(sizeof(SliceRec) * b.nrec);
    if (!tw_fits(b, true)) continue;
    for (int q = 0; q < b.nrec; ++q) {
      const SliceSize z = slice_size(hr[q], TW_K * tw_stages(true, b.max_n));
      for (int op = 0; op < 4; ++op) total += z.dig[op] + z.eb[op];
    }
  }
  return total;
}

rss_status ensure_slices(rss_factorization* f, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(f->slice_mu);
  if (f->slices_ready) return RSS_OK;
  auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t total = slice_total(f);
  char* base = nullptr;
  const cudaError_t em = pool_malloc(reinterpret_cast<void**>(&base), total, st);
  if (em == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    rss_set_error("rss_solve: no device memory for the digits of the factor");
    return RSS_ENOMEM;
  }
  RSS_CUDA(em);
  char* p = base;
  auto take = [&](size_t b) {
    char* q = p;
    p += al(b);
    return q;
  };
  std::vector<SliceRec*> recs(f->batches.size());
  std::vector<std::vector<SliceRec>> hs(f->batches.size());   // alive until the copies are done
  cudaError_t e = cudaSuccess;
  for (size_t bi = 0; bi < f->batches.size() && e == cudaSuccess; ++bi) {
    const Batch& b = f->batches[bi];
    const BoxRec<double>* hr = static_cast<const BoxRec<double>*>(f->rec_host[bi]);
    recs[bi] = reinterpret_cast<SliceRec*>(take(sizeof(SliceRec) * b.nrec));
    if (!tw_fits(b, true)) continue;
    hs[bi].assign(b.nrec, SliceRec{});
    for (int q = 0; q < b.nrec; ++q) {
      const SliceSize z = slice_size(hr[q], TW_K * tw_stages(true, b.max_n));
      for (int op = 0; op < 4; ++op) {
        hs[bi][q].dig[op] = reinterpret_cast<unsigned char*>(take(z.dig[op]));
        hs[bi][q].eb[op] = reinterpret_cast<int*>(take(z.eb[op]));
      }
    }
    e = cudaMemcpyAsync(recs[bi], hs[bi].data(), sizeof(SliceRec) * b.nrec, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) break;
    const BoxRec<double>* dr = static_cast<const BoxRec<double>*>(b.d_recs);
    const unsigned tr = cdiv(b.max_r, TW_M), tc = std::max(1u, cdiv(b.max_c, TW_M)), tn = cdiv(b.max_n, TW_M);
    auto cut = [&](auto sx) {
      constexpr int SX = decltype(sx)::value;
      auto z = [](int k) { return std::max(1u, cdiv(k, SX * TW_K)); };
      k_tw_cache<TW_UPW, SX><<<dim3(tr, b.nrec, z(b.max_n)), TW_NT, 0, st>>>(dr, recs[bi]);
      k_tw_cache<TW_UPE, SX><<<dim3(tc, b.nrec, z(b.max_r)), TW_NT, 0, st>>>(dr, recs[bi]);
      k_tw_cache<TW_DNF, SX><<<dim3(tr, b.nrec, z(b.max_c)), TW_NT, 0, st>>>(dr, recs[bi]);
      k_tw_cache<TW_DNW, SX><<<dim3(tn, b.nrec, z(b.max_r)), TW_NT, 0, st>>>(dr, recs[bi]);
    };
    if (tw_stages(true, b.max_n) == TW_SX) cut(std::integral_constant<int, TW_SX>{});
    else cut(std::integral_constant<int, TW_SX_LONG>{});
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // other streams may use the digits from here on
  else cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    pool_free(base, st);
    rss_set_error(std::string("rss_solve: slice cache: ") + cudaGetErrorString(e));
    return RSS_ECUDA;
  }
  f->slice_bytes = total;
  f->d_slice_mem = base;
  f->d_slices = recs;
  f->slices_ready = true;
  return RSS_OK;
}

template <typename T, int OP, bool CACHE, int GW, int SX>
cudaError_t launch_tw_gw(const Batch& b, const SliceRec* sl, T* x, int64_t ldx, int nrhs, int* err, int polls,
                         cudaStream_t st) {
  constexpr bool real = sizeof(T) == sizeof(double);
  const int mr = OP == TW_UPE ? std::max(1, b.max_c) : OP == TW_DNW ? b.max_n : b.max_r;
  const int mk = OP == TW_UPW ? b.max_n : OP == TW_DNF ? b.max_c : b.max_r;
  const TwPlan p = tw_plan_op(OP, b.max_n, b.max_r, b.max_c, GW, real);
  const int tiles = cdiv(mr, TW_M);
  const cudaError_t e = allow_smem(k_tw<T, OP, CACHE, GW, SX>);
  if (e != cudaSuccess) return e;
  // a property of the class alone, so that a column's bits do not depend on the others
  int spl = 1;
  if (OP == TW_DNF)
    while (spl < 8 && b.nrec * tiles * spl <= 76 && mk >= 16 * spl * (real ? TW_K : TW_K / 2)) spl *= 2;
  return launch_pdl(k_tw<T, OP, CACHE, GW, SX>, dim3(spl * tiles, cdiv(nrhs, real ? 2 * GW : GW), b.nrec), TW_NT,
                    p.smem, st, OP == TW_UPW || OP == TW_DNW ? tiles : spl, static_cast<const BoxRec<T>*>(b.d_recs), sl, x, ldx, nrhs, p.rows8, p.nst, p.nstr, err,
                    polls);
}

// 16 columns to a group where 32 would leave half of the SMs without a CTA, or do not fit.
// Real classes of more than 128 points take stretches of 64 entries: a panel's error against
// quadruple precision is then 3.65e-16 (96^2, leaf 144; FP64 columns 4.03e-16, stretches of
// 384 4.56e-16) and 3.61e-16 (64^2, leaf 256; 4.47e-16 and 5.41e-16).
template <typename T, int OP, bool CACHE>
cudaError_t launch_tw(const Batch& b, const SliceRec* sl, T* x, int64_t ldx, int nrhs, int* err, int polls,
                      cudaStream_t st) {
  constexpr bool real = sizeof(T) == sizeof(double);
  const long long tiles = cdiv(OP == TW_UPE ? std::max(1, b.max_c) : OP == TW_DNW ? b.max_n : b.max_r, TW_M);
  const bool few = tiles * b.nrec * cdiv(nrhs, real ? TW_NC : TW_NC / 2) <= 76;
  const bool g16 = few || nrhs <= 16 || tw_group(OP, b.max_n, b.max_r, b.max_c, real) == 16;
  auto go = [&](auto sx) {
    constexpr int SX = decltype(sx)::value;
    return g16 ? launch_tw_gw<T, OP, CACHE, 16, SX>(b, sl, x, ldx, nrhs, err, polls, st)
               : launch_tw_gw<T, OP, CACHE, 32, SX>(b, sl, x, ldx, nrhs, err, polls, st);
  };
  if constexpr (!real) return go(std::integral_constant<int, TW_SXZ>{});
  else if (tw_stages(true, b.max_n) == TW_SX) return go(std::integral_constant<int, TW_SX>{});
  else return go(std::integral_constant<int, TW_SX_LONG>{});
}

// The tensor-core sweeps for the colour classes that take them, the FP64 sweeps for the
// others.  may_build: the
// caller allows the one-time allocation of a real factor's digits (rss_solve_noalloc
// does not; it uses them only when they already exist, and cuts them per call else).
// large: the products in classes of many boxes only.
template <typename T>
rss_status sweeps_tc(const rss_factorization* f, T* x, int64_t ldx, int nrhs, cudaStream_t st, void* ws, bool may_build,
                     bool large) {
  constexpr int RC = 8;
  constexpr bool real = sizeof(T) == sizeof(double);
  bool sl = real && nrhs >= TCB;
  if (sl && may_build) {
    const rss_status s = ensure_slices(const_cast<rss_factorization*>(f), st);
    if (s != RSS_OK && s != RSS_ENOMEM) return s;
    sl = s == RSS_OK;   // (no memory for the digits: cut per call)
  } else if (sl) {
    std::lock_guard<std::mutex> lk(const_cast<rss_factorization*>(f)->slice_mu);
    sl = f->slices_ready;
  }
  const SweepWs w = sweep_ws<T>(f, nrhs, RC);
  T* topz = reinterpret_cast<T*>(static_cast<char*>(ws) + w.topz_off);
  int* err = reinterpret_cast<int*>(static_cast<char*>(ws) + w.bar_off + 2 * sizeof(unsigned));
  const int polls = wait_limit(f->params.wait_polls, TW_POLLS);
  auto takes = [&](const Batch& b) {
    return tw_takes(b, nrhs, real) && (!large || (long long)b.nrec * cdiv(nrhs, TCB) >= 152);
  };
  auto product = [&](size_t bi, auto op) -> cudaError_t {
    constexpr int OP = decltype(op)::value;
    const Batch& b = f->batches[bi];
    if constexpr (real)
      if (sl) return launch_tw<T, OP, true>(b, f->d_slices[bi], x, ldx, nrhs, err, polls, st);
    return launch_tw<T, OP, false>(b, nullptr, x, ldx, nrhs, err, polls, st);
  };
  for (size_t bi = 0; bi < f->batches.size(); ++bi) {
    if (!takes(f->batches[bi])) {
      const rss_status s = sweep_class<T, RC, true>(f->batches[bi], x, ldx, nrhs, st);
      if (s != RSS_OK) return s;
      continue;
    }
    RSS_CUDA(product(bi, std::integral_constant<int, TW_UPW>{}));
    RSS_CUDA(product(bi, std::integral_constant<int, TW_UPE>{}));
  }
  const rss_status stp = top_apply<T, RC>(f, x, ldx, nrhs, st, topz);
  if (stp != RSS_OK) return stp;
  for (size_t bi = f->batches.size(); bi-- > 0;) {
    if (!takes(f->batches[bi])) {
      const rss_status s = sweep_class<T, RC, false>(f->batches[bi], x, ldx, nrhs, st);
      if (s != RSS_OK) return s;
      continue;
    }
    RSS_CUDA(product(bi, std::integral_constant<int, TW_DNF>{}));
    RSS_CUDA(product(bi, std::integral_constant<int, TW_DNW>{}));
  }
  return RSS_OK;
}

bool use_tc(const rss_factorization* f, int64_t nrhs) {
  return nrhs >= TCN && (f->params.schur_path == 0 || f->params.schur_path == 2);
}

template <typename T>
rss_status run_sweeps(const rss_factorization* f, T* x, int64_t ldx, int64_t nrhs, cudaStream_t st, void* ws,
                      bool may_build = true, Sweeps how = Sweeps::by_columns) {
  if (how != Sweeps::fp64 && use_tc(f, nrhs))
    return sweeps_tc<T>(f, x, ldx, (int)nrhs, st, ws, may_build, how == Sweeps::large_classes);
  const int rc = rhs_chunk(nrhs);
  return rc == 1 ? sweeps<T, 1>(f, x, ldx, (int)nrhs, st, ws)
         : rc == 4 ? sweeps<T, 4>(f, x, ldx, (int)nrhs, st, ws)
                   : sweeps<T, 8>(f, x, ldx, (int)nrhs, st, ws);
}

}  // namespace

template <typename T>
rss_status solve_impl(const rss_factorization* f, T* b, int64_t nrhs, int64_t ldb, cudaStream_t st, Sweeps how) {
  const int64_t N = f->n;
  const SweepWs w = sweep_ws<T>(f, nrhs, rhs_chunk(nrhs));
  const size_t xb = (sizeof(T) * (size_t)N * nrhs + 255) & ~size_t(255);
  char* mem = nullptr;
  RSS_CUDA(pool_malloc(reinterpret_cast<void**>(&mem), xb + w.bytes, st));
  T* x = reinterpret_cast<T*>(mem);
  const int* err = reinterpret_cast<const int*>(mem + xb + w.bar_off + 2 * sizeof(unsigned));
  RSS_CUDA(cudaMemsetAsync(mem + xb + w.bar_off, 0, 4 * sizeof(int), st));
  const unsigned grid = std::min<long long>(cdiv((long long)N * nrhs, NT), 152LL * 16);
  k_perm_in<T><<<grid, NT, 0, st>>>(b, ldb, x, N, (int)nrhs, f->d_user_to_tree);
  rss_status s = RSS_OK;
  if (cudaGetLastError() != cudaSuccess) {
    rss_set_error("rss_solve: launch failed");
    s = RSS_ECUDA;
  }
  if (s == RSS_OK) s = run_sweeps<T>(f, x, nrhs, nrhs, st, mem + xb, true, how);
  if (s == RSS_OK) {
    if (launch_pdl(k_perm_out<T>, dim3(grid), NT, 0, st, 1, b, ldb, x, N, (int)nrhs, f->d_user_to_tree, err) !=
        cudaSuccess) {
      cudaGetLastError();
      rss_set_error("rss_solve: launch failed");
      s = RSS_ECUDA;
    }
  }
  pool_free(mem, st);
  return s;
}

template rss_status solve_impl<double>(const rss_factorization*, double*, int64_t, int64_t, cudaStream_t, Sweeps);

template <typename T> rss_status build_sweep_classes(rss_factorization* f, cudaStream_t st) {
  if (f->batches.empty()) return RSS_OK;
  std::vector<SwpClass<T>> h(f->batches.size());
  for (size_t i = 0; i < h.size(); ++i) {
    const Batch& b = f->batches[i];
    h[i] = SwpClass<T>{static_cast<const BoxRec<T>*>(b.d_recs), b.nrec, sweep_slices(b.nrec)};
  }
  void* d = f->arena.get(sizeof(SwpClass<T>) * h.size());
  if (!d) {
    rss_set_error("rss_factor: device arena allocation failed");
    return RSS_ENOMEM;
  }
  RSS_CUDA(cudaMemcpyAsync(d, h.data(), sizeof(SwpClass<T>) * h.size(), cudaMemcpyHostToDevice, st));
  RSS_CUDA(cudaStreamSynchronize(st));   // h is a host temporary
  f->d_swp = d;
  return RSS_OK;
}

template rss_status build_sweep_classes<double>(rss_factorization*, cudaStream_t);
template rss_status build_sweep_classes<zd>(rss_factorization*, cudaStream_t);

size_t solve_device_bytes(const rss_factorization* f, int64_t nrhs) {
  const size_t esz = f->is_complex ? 16 : 8;
  const size_t xb = (esz * (size_t)f->n * (size_t)nrhs + 255) & ~size_t(255);
  return xb + (f->is_complex ? sweep_ws<zd>(f, nrhs, rhs_chunk(nrhs)).bytes
                             : sweep_ws<double>(f, nrhs, rhs_chunk(nrhs)).bytes);
}

// Requests of TCN columns take the products alone, so also in a panel; smaller ones, whose
// solves take the FP64 sweeps, do so in panels of TCB columns: on real factors in every
// class, on complex ones in the classes whose products fill the GPU.  (Requests of one
// column in panels of 64, Helmholtz 2048^2: 45 RHS/s, with FP64 sweeps in all classes 21;
// 256^2: 1868 and 1329.)
Sweeps panel_sweeps(const rss_factorization* f, int64_t cols, int64_t smallest) {
  if (smallest >= TCN) return Sweeps::by_columns;
  return cols < TCB ? Sweeps::fp64 : f->is_complex ? Sweeps::large_classes : Sweeps::by_columns;
}

size_t solve_cache_bytes(const rss_factorization* f, int64_t max_nrhs) {
  return !f->is_complex && max_nrhs >= TCB && use_tc(f, max_nrhs) ? slice_total(f) : 0;
}

rss_status prepare_solve_caches(const rss_factorization* f, int64_t max_nrhs, cudaStream_t st) {
  if (f->is_complex || max_nrhs < TCB || !use_tc(f, max_nrhs)) return RSS_OK;
  return ensure_slices(const_cast<rss_factorization*>(f), st);
}
template rss_status solve_impl<zd>(const rss_factorization*, zd*, int64_t, int64_t, cudaStream_t, Sweeps);

// ---------------------------------------------------------------------------
// rss_solve_noalloc: the same sweeps as rss_solve, with the working copy of
// the right-hand sides in a fixed device array instead of memory obtained at
// call time.  Some callers cannot allocate device memory: a process whose
// framework allocator has already reserved the device's free memory, a
// latency-bound serving loop that may not take the synchronisation a fresh
// allocation can cost, or a host that budgets device memory up front.  For
// them the scratch is a file-scope array that exists on every GPU that loads
// the library, for the life of the process.

namespace {

constexpr size_t kNoAllocScratchBytes = size_t(16) << 20;   // 16 MiB per device
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device, looked up once
// per device (the symbol's host-side name is not a device address).
rss_status noalloc_scratch(void** out) {
  int dev = -1;
  RSS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    rss_set_error("rss_solve_noalloc: device ordinal out of range");
    return RSS_EINVAL;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    RSS_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return RSS_OK;
}

template <typename T>
rss_status solve_in_scratch(const rss_factorization* f, T* b, int64_t nrhs, int64_t ldb, cudaStream_t st,
                            T* x) {
  const int64_t N = f->n;
  const unsigned grid = std::min<long long>(cdiv((long long)N * nrhs, NT), 152LL * 16);
  // every entry of x is written here, so nothing left from an earlier call is read
  k_perm_in<T><<<grid, NT, 0, st>>>(b, ldb, x, N, (int)nrhs, f->d_user_to_tree);
  RSS_LAUNCHED();
  const size_t xb = (sizeof(T) * (size_t)N * nrhs + 255) & ~size_t(255);
  char* ws = reinterpret_cast<char*>(x) + xb;
  const SweepWs w = sweep_ws<T>(f, nrhs, rhs_chunk(nrhs));
  RSS_CUDA(cudaMemsetAsync(ws + w.bar_off, 0, 4 * sizeof(int), st));   // barrier words of the last call
  const rss_status s = run_sweeps<T>(f, x, nrhs, nrhs, st, ws, false);
  if (s != RSS_OK) return s;
  RSS_CUDA(launch_pdl(k_perm_out<T>, dim3(grid), NT, 0, st, 1, b, ldb, x, N, (int)nrhs, f->d_user_to_tree,
                      reinterpret_cast<const int*>(ws + w.bar_off + 2 * sizeof(unsigned))));
  return RSS_OK;
}

}  // namespace

extern "C" rss_status rss_solve_noalloc(const rss_factorization* f, void* b, int64_t nrhs, int64_t ldb,
                                        void* stream) {
  if (!f || f->tag != RSS_TAG_FACTOR) {
    rss_set_error("rss_solve_noalloc: not a factor handle");
    return RSS_EINVAL;
  }
  if (!b || nrhs <= 0 || ldb < f->n) {
    rss_set_error("rss_solve_noalloc: b must be non-NULL with nrhs > 0 and ldb >= n");
    return RSS_EINVAL;
  }
  const size_t esz = f->is_complex ? 16 : 8;
  const size_t need = ((esz * (size_t)f->n * (size_t)nrhs + 255) & ~size_t(255)) +
                      (f->is_complex ? sweep_ws<zd>(f, nrhs, rhs_chunk(nrhs)).bytes
                                     : sweep_ws<double>(f, nrhs, rhs_chunk(nrhs)).bytes);
  if (need > kNoAllocScratchBytes) {
    rss_set_error("rss_solve_noalloc: n * nrhs (with the sweep workspace) needs " + std::to_string(need) +
                  " bytes of scratch; the fixed maximum is " + std::to_string(kNoAllocScratchBytes) +
                  " bytes (use rss_solve, or fewer right-hand sides per call)");
    return RSS_EINVAL;
  }
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, b) != cudaSuccess) {
    cudaGetLastError();
    attr.type = cudaMemoryTypeUnregistered;
  }
  if (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged) {
    rss_set_error("rss_solve_noalloc: b must be device memory (staging host data would allocate)");
    return RSS_EINVAL;
  }
  void* scratch = nullptr;
  rss_status s = noalloc_scratch(&scratch);
  if (s != RSS_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return f->is_complex
             ? solve_in_scratch<zd>(f, static_cast<zd*>(b), nrhs, ldb, st, static_cast<zd*>(scratch))
             : solve_in_scratch<double>(f, static_cast<double*>(b), nrhs, ldb, st, static_cast<double*>(scratch));
}

// ---------------------------------------------------------------------------
// rss_tune_solve: the launch form of the sweeps, chosen by measurement.  Every form
// adds the same products in the same order, so the choice changes the time of a
// solve, never its result.  (The table has eleven candidates, as its readers expect; their
// `spread` has no effect, so six forms are timed.)
extern "C" rss_status rss_tune_solve(rss_factorization* f, int64_t nrhs, void* stream, char* json, size_t len) {
  if (!f || f->tag != RSS_TAG_FACTOR || nrhs <= 0 || nrhs >= 1 << 20) {
    rss_set_error("rss_tune_solve: needs a factor handle and 0 < nrhs < 2^20");
    return RSS_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t esz = f->is_complex ? 16 : 8;
  // (from TCN to TCB - 1 columns: the forms are timed with that many, for the calls with fewer)
  const bool fp64_path = nrhs < TCB || !use_tc(f, nrhs);
  std::ostringstream o;
  o << "{\"nrhs\": " << nrhs;
  if (!fp64_path || !f->d_swp) {
    o << ", \"path\": \"tensor-core sweeps (nothing to tune)\"}";
  } else {
    const size_t bytes = esz * (size_t)f->n * (size_t)nrhs;
    void* b = nullptr;
    RSS_CUDA(pool_malloc(&b, bytes, st));
    RSS_CUDA(cudaMemsetAsync(b, 0, bytes, st));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    RSS_CUDA(cudaEventCreate(&e0));
    RSS_CUDA(cudaEventCreate(&e1));
    struct Cand {
      int launch, spread, ctas, tail;
    };
    const Cand cands[] = {{1, 0, 0, 0},   {2, 1, 4, 0},   {2, 1, 0, 0},   {2, 4, 4, 0},
                          {2, 4, 0, 0},   {3, 1, 0, 32},  {3, 4, 0, 32},  {3, 1, 0, 128},
                          {3, 4, 0, 128}, {3, 1, 0, 512}, {3, 4, 0, 512}};
    constexpr int ncand = (int)(sizeof(cands) / sizeof(cands[0]));
    float ms[ncand];   // (candidates that differ in `spread` alone are one launch form, timed once)
    const int keep = f->swp_spread, keep_c = f->swp_ctas, keep_l = f->swp_launch, keep_t = f->swp_tail_boxes;
    Cand best{1, 0, 0, 0};
    float best_ms = 1e30f;
    rss_status s = RSS_OK;
    o << ", \"path\": \"FP64 sweeps\", \"candidates\": [";
    for (int ci = 0; ci < ncand && s == RSS_OK; ++ci) {
      const Cand& c = cands[ci];
      f->swp_launch = c.launch;
      f->swp_spread = c.spread;
      f->swp_ctas = c.ctas;
      f->swp_tail_boxes = c.tail;
      int same = 0;
      while (same < ci && (cands[same].launch != c.launch || cands[same].ctas != c.ctas || cands[same].tail != c.tail)) ++same;
      if (same < ci) {
        ms[ci] = ms[same];
      } else {
        float t[3];
        for (int rep = -1; rep < 3 && s == RSS_OK; ++rep) {   // one untimed run first
          cudaEventRecord(e0, st);
          s = f->is_complex ? solve_impl<zd>(f, static_cast<zd*>(b), nrhs, f->n, st, Sweeps::fp64)
                            : solve_impl<double>(f, static_cast<double*>(b), nrhs, f->n, st, Sweeps::fp64);
          cudaEventRecord(e1, st);
          if (cudaEventSynchronize(e1) != cudaSuccess) s = RSS_ECUDA;
          if (rep >= 0 && s == RSS_OK) cudaEventElapsedTime(&t[rep], e0, e1);
        }
        if (s != RSS_OK) break;
        std::sort(t, t + 3);
        ms[ci] = t[1];
      }
      o << (ci ? ", " : "") << "{\"launch\": \"" << (c.launch == 1 ? "per_class" : c.launch == 2 ? "persistent" : "hybrid")
        << "\"";
      if (c.launch != 1) o << ", \"spread\": " << c.spread << ", \"ctas_per_sm\": " << c.ctas;
      if (c.launch == 3) o << ", \"tail_boxes\": " << c.tail;
      o << ", \"ms\": " << ms[ci] << "}";
      if (ms[ci] < best_ms) {
        best_ms = ms[ci];
        best = c;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    pool_free(b, st);
    if (s != RSS_OK) {
      f->swp_spread = keep;
      f->swp_ctas = keep_c;
      f->swp_launch = keep_l;
      f->swp_tail_boxes = keep_t;
      return s;
    }
    f->swp_launch = best.launch;
    f->swp_spread = best.spread;
    f->swp_ctas = best.ctas;
    f->swp_tail_boxes = best.tail;
    o << "], \"launch\": \"" << (best.launch == 1 ? "per_class" : best.launch == 2 ? "persistent" : "hybrid")
      << "\"";
    if (best.launch != 1) o << ", \"spread\": " << best.spread << ", \"ctas_per_sm\": " << best.ctas;
    if (best.launch == 3) o << ", \"tail_boxes\": " << best.tail;
    o << ", \"ms\": " << best_ms << "}";
  }
  const std::string js = o.str();
  if (json && len) {
    if (js.size() + 1 > len) {
      rss_set_error("rss_tune_solve: json buffer too small");
      return RSS_EINVAL;
    }
    std::memcpy(json, js.c_str(), js.size() + 1);
  }
  return RSS_OK;
}
