// The FP64 sweeps.  Per box, with v = [b_S; b_R] and the matrices W_E, W_F of the
// factorization (n x r, columns of B in pivot order):
//   up:    y = W_F^T v (= L^{-1} P (b_R - T^* b_S)), b_R <- y, b_C -= E y;
//   down:  z = y_R - F y_C, [y_S; y_R] <- [y_S; 0] + W_E z (= y_S - T U^{-1} z; U^{-1} z).
// One launch per colour class and sweep: a cluster of Q CTAs owns a box and RC
// columns.  CTA q owns a slice of the rows of every product; y (up) and the partial
// sums of F y_C (down) go through distributed shared memory.  A class too small to
// fill the GPU is bound by latency: its CTAs stage every factor entry they need by
// cp.async before they wait for the previous launch (programmatic dependent
// launch), so neither the memory latency nor the launch latency is on the path from
// class to class.  A class that fills the GPU is bound by the FP64 pipe (one FMA per
// factor entry and column, two FMAs per clock and SM): its CTAs read the factor
// straight from global memory, many to an SM.
//
// Every sum has a fixed order that depends on neither Q, RC nor the launch form:
//   W_F^T v: four sums over l = p, p + 4, .. (p = 0 .. 3), added as a tree;
//   E y, W_E z: four sums over consecutive quarters of r, added as a tree;
//   F y_C: per slice of C (qc slices, a property of the class) four sums over the
//   rows i = p, p + 4, .. of the slice, added as a tree; the slices added in order.
constexpr int SW_NT = 256;
constexpr int SW_QMAX = 8;
constexpr int SW_PF = 4, SW_PE = 4, SW_PC = 4;

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// scalars of shared memory: always, with the smaller and with both matrices staged
struct SweepSm {
  size_t need, one, full;
};
template <typename T, int RC> inline SweepSm sweep_sm_up(int n, int r, int c, int Q) {
  const size_t rows = (c + Q - 1) / Q, js = (r + Q - 1) / Q;
  const size_t need = ((size_t)n + r) * RC;
  const size_t w = js * (n | 1), e = (rows | 1) * r;
  return SweepSm{need, need + std::min(w, e), need + w + e};
}
template <typename T, int RC> inline SweepSm sweep_sm_down(int n, int r, int c, int Q, int qc) {
  const size_t rows = (c + Q - 1) / Q, ls = (n + Q - 1) / Q, sl = qc / Q;
  const size_t need = (rows + r + sl * r) * RC;
  const size_t f = (rows | 1) * r, w = (ls | 1) * r;
  return SweepSm{need, need + std::min(f, w), need + f + w};
}

// W lanes that hold the parts of one sum: their tree sum, in every lane
template <int W, typename T> __device__ __forceinline__ T part_sum(T v) {
#pragma unroll
  for (int d = 1; d < W; d <<= 1) v = v + shfl_xor(v, d);
  return v;
}

// The same for the sums of RC columns (RC a multiple of 4, four lanes, p = lane % 4): lane
// p ends with the sums of columns own_column(p) .. + RC / 4 - 1 in acc[0 ..].  6 additions
// for 8 columns instead of 16, which counts where a lane has about ten products a column:
// 15 columns, Laplace 896^2, leaf 49 30.0 -> 26.5 ms, 1024^2 36.8 -> 32.9 ms.
template <int RC> __device__ __forceinline__ int own_column(int p) { return (p & 1) * (RC / 2) + (p >> 1) * (RC / 4); }
template <int RC, typename T> __device__ __forceinline__ void part_scatter(T (&acc)[RC], int p) {
#pragma unroll
  for (int q = 0; q < RC / 2; ++q) {
    const T give = (p & 1) ? acc[q] : acc[q + RC / 2];
    const T keep = (p & 1) ? acc[q + RC / 2] : acc[q];
    acc[q] = keep + shfl_xor(give, 1);
  }
#pragma unroll
  for (int q = 0; q < RC / 4; ++q) {
    const T give = (p & 2) ? acc[q] : acc[q + RC / 4];
    const T keep = (p & 2) ? acc[q + RC / 4] : acc[q];
    acc[q] = keep + shfl_xor(give, 2);
  }
}

// (entry (g, q) of the right-hand sides at x[g * ldx + q]: the columns of a point
// side by side)
// x_g(i) = [keep(i)] x_g(i) +- sum_j M(i, j) w_j (+: add) for the rows i < rows of M (ld
// scalars between columns) and the columns j >= lo(i) (M is zero before), w in shared
// memory (RC scalars per j): four lanes per row, or, for one column when the rows fill
// half the CTA, one thread per row (no shuffles); the same sums either way.
template <typename T, int RC, typename LO, typename GI, typename KP>
__device__ __forceinline__ void row_products(int rows, int r, int nq, int tid, int nt, const T* w, const T* M, size_t ld,
                                             LO lo, GI gidx, KP keep, bool add, T* xq, int64_t ldx) {
  const int L4 = (r + SW_PE - 1) / SW_PE;
  if constexpr (RC == 1) {
    if (rows * 2 >= nt) {
      for (int i = tid; i < rows; i += nt) {
        T* g = xq + gidx(i) * ldx;
        const int a = lo(i);
        const T* m = M + i;
        T acc[SW_PE];
#pragma unroll
        for (int p = 0; p < SW_PE; ++p) acc[p] = zero<T>();
#pragma unroll 4
        for (int t = 0; t < L4; ++t)   // the four sums together
#pragma unroll
          for (int p = 0; p < SW_PE; ++p) {
            const int j = p * L4 + t;
            if (j >= a && j < r) acc[p] = mad(acc[p], m[(size_t)j * ld], w[j]);
          }
        const T s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
        *g = !keep(i) ? s : add ? ld_l2(g) + s : ld_l2(g) - s;
      }
      return;
    }
  }
  for (int e = tid; e < ((rows * SW_PE + 31) & ~31); e += nt) {
    const int p = e % SW_PE, i = e / SW_PE;
    constexpr int OW = (RC + SW_PE - 1) / SW_PE;   // columns that a lane stores: c0 ..
    const int c0 = RC == 1 ? 0 : own_column<RC>(p);
    const bool own = RC > 1 || p == 0;
    T acc[RC], old[OW];
#pragma unroll
    for (int q = 0; q < RC; ++q) acc[q] = zero<T>();
    int64_t gi = 0;
    if (i < rows) {
      gi = gidx(i);
      const bool kp = keep(i);
#pragma unroll
      for (int q = 0; q < OW; ++q)
        if (own && c0 + q < nq) old[q] = kp ? ld_l2(xq + gi * ldx + c0 + q) : zero<T>();
      const int j1 = min(r, (p + 1) * L4);
      const T* m = M + i;
#pragma unroll 4
      for (int j = max(p * L4, lo(i)); j < j1; ++j) {
        const T mv = m[(size_t)j * ld];
#pragma unroll
        for (int q = 0; q < RC; ++q) acc[q] = mad(acc[q], mv, w[j * RC + q]);
      }
    }
    if constexpr (RC == 1) acc[0] = part_sum<SW_PE>(acc[0]);
    else part_scatter<RC>(acc, p);
    if (i < rows) {
#pragma unroll
      for (int q = 0; q < OW; ++q)
        if (own && c0 + q < nq) xq[gi * ldx + c0 + q] = add ? old[q] + acc[q] : old[q] - acc[q];
    }
  }
}

// How the CTAs of a box meet: every thread arrives at a barrier before it waits.
struct SoloCta {
  __device__ void arrive() const {}
  __device__ void wait() const { __syncthreads(); }
  template <typename T> __device__ T* peer(T* p, int) const { return p; }
};
struct ClusterCta {
  __device__ void arrive() const { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
  __device__ void wait() const { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
  template <typename T> __device__ T* peer(T* p, int q) const {
    return cooperative_groups::this_cluster().map_shared_rank(p, q);
  }
};

// CTA `rank` of Q on one box; peer(p, q): the address of shared scalar p in CTA q.
// Every thread calls it.
template <typename T, int RC, typename CL>
__device__ void up_box(const BoxRec<T>& R, T* xq, int64_t ldx, int nq, T* sm, size_t sm_cap, int rank, int Q,
                       bool wait_prev, CL cl) {
  cl.arrive();   // this CTA runs: its peers may write its y
  const int k = R.k, r = R.r, c = R.c, n = k + r, tid = threadIdx.x, nt = blockDim.x;
  const int j0 = r * rank / Q, j1 = r * (rank + 1) / Q;
  const int i0 = (int)((long long)c * rank / Q), i1 = (int)((long long)c * (rank + 1) / Q), rows = i1 - i0;
  const int ldw = n | 1, lde = rows | 1;
  T* v = sm;                          // n x RC
  T* y = v + (size_t)n * RC;          // r x RC
  T* Ws = y + (size_t)r * RC;         // columns j0 .. j1 of W_F, ld n|1
  const bool stw = (size_t)(Ws - sm) + (size_t)(j1 - j0) * ldw <= sm_cap;
  T* Es = Ws + (stw ? (size_t)(j1 - j0) * ldw : 0);   // rows i0 .. i1 of E, ld rows|1
  const bool ste = (size_t)(Es - sm) + (size_t)lde * r <= sm_cap;
  if (stw) {
    for (int j = j0 + tid / 32; j < j1; j += nt / 32)
      for (int l = tid % 32; l < n; l += 32) cp_async_el(Ws + (size_t)(j - j0) * ldw + l, R.Wf + (size_t)j * n + l);
  }
  cp_async_commit();
  if (ste) {
    for (int j = tid / 32; j < r; j += nt / 32)
      for (int i = tid % 32; i < rows; i += 32) cp_async_el(Es + (size_t)j * lde + i, R.E + i0 + i + (size_t)j * c);
  }
  cp_async_commit();
  if (wait_prev) pdl_wait();
  for (int e = tid; e < n * RC; e += nt) {
    const int l = e / RC, q = e % RC;
    v[e] = q < nq ? ld_l2(xq + (l < k ? R.idxC[l] : R.idxR[l - k]) * ldx + q) : zero<T>();
  }
  cp_async_wait_group<1>();
  __syncthreads();
  cl.wait();
  for (int e = tid; e < (((j1 - j0) * SW_PF + 31) & ~31); e += nt) {
    const int p = e % SW_PF, j = j0 + e / SW_PF;
    T acc[RC];
#pragma unroll
    for (int q = 0; q < RC; ++q) acc[q] = zero<T>();
    if (j < j1) {
      const T* w = stw ? Ws + (size_t)(j - j0) * ldw : R.Wf + (size_t)j * n;
#pragma unroll 8
      for (int l = p; l < n; l += SW_PF) {
        const T wv = w[l];
#pragma unroll
        for (int q = 0; q < RC; ++q) acc[q] = mad(acc[q], wv, v[l * RC + q]);
      }
    }
    if constexpr (RC == 1) {
      acc[0] = part_sum<SW_PF>(acc[0]);
      if (j < j1)
        for (int t = p; t < Q; t += SW_PF) *cl.peer(y + j, t) = acc[0];
    } else {
      part_scatter<RC>(acc, p);
      if (j < j1)
        for (int t = 0; t < Q; ++t) {
          T* d = cl.peer(y + (size_t)j * RC + own_column<RC>(p), t);
#pragma unroll
          for (int q = 0; q < RC / 4; ++q) d[q] = acc[q];
        }
    }
  }
  cp_async_wait_group<0>();
  __syncthreads();
  cl.arrive();
  cl.wait();   // y is complete, and every CTA has read its copy of v
  for (int e = tid; e < (j1 - j0) * RC; e += nt) {
    const int j = j0 + e / RC, q = e % RC;
    if (q < nq) xq[R.idxR[j] * ldx + q] = y[j * RC + q];
  }
  row_products<T, RC>(rows, r, nq, tid, nt, y, ste ? Es : R.E + i0, ste ? lde : c, [](int) { return 0; },
                      [&](int i) { return (int64_t)R.idxC[i0 + i]; }, [](int) { return true; }, false, xq, ldx);
}

template <typename T, int RC, typename CL>
__device__ void down_box(const BoxRec<T>& R, T* xq, int64_t ldx, int nq, T* sm, size_t sm_cap, int rank, int Q, int qc,
                         bool wait_prev, CL cl) {
  const int k = R.k, r = R.r, c = R.c, n = k + r, tid = threadIdx.x, nt = blockDim.x;
  const int sl = qc / Q;   // slices of C of this CTA: rank sl ..
  auto row0 = [&](int s) { return (int)((long long)c * s / qc); };
  const int i0 = row0(rank * sl), rows = row0((rank + 1) * sl) - i0;
  const int l0 = n * rank / Q, lw = n * (rank + 1) / Q - l0;
  const int ldf = rows | 1, ldw = lw | 1;
  T* gp = sm;                                   // sl x r x RC: this CTA's slices' sums (the same place in every CTA)
  T* z = gp + (size_t)sl * r * RC;              // r x RC
  T* yc = z + (size_t)r * RC;                   // rows x RC
  T* Fs = yc + (size_t)rows * RC;               // rows i0 .. of F^T, ld rows|1
  const bool stf = (size_t)(Fs - sm) + (size_t)ldf * r <= sm_cap;
  T* Ws = Fs + (stf ? (size_t)ldf * r : 0);     // rows l0 .. of W_E, ld lw|1
  const bool stw = (size_t)(Ws - sm) + (size_t)ldw * r <= sm_cap;
  if (stf) {
    for (int j = tid / 32; j < r; j += nt / 32)
      for (int i = tid % 32; i < rows; i += 32) cp_async_el(Fs + (size_t)j * ldf + i, R.Ft + i0 + i + (size_t)j * c);
  }
  cp_async_commit();
  if (stw) {
    for (int j = tid / 32; j < r; j += nt / 32)
      for (int l = tid % 32; l < lw; l += 32) cp_async_el(Ws + (size_t)j * ldw + l, R.We + l0 + l + (size_t)j * n);
  }
  cp_async_commit();
  if (wait_prev) pdl_wait();
  for (int e = tid; e < rows * RC; e += nt) {
    const int i = e / RC, q = e % RC;
    yc[e] = q < nq ? ld_l2(xq + R.idxC[i0 + i] * ldx + q) : zero<T>();
  }
  for (int e = tid; e < r * RC; e += nt) {
    const int j = e / RC, q = e % RC;
    z[e] = q < nq ? ld_l2(xq + R.idxR[j] * ldx + q) : zero<T>();
  }
  cp_async_wait_group<1>();
  __syncthreads();
  for (int e = tid; e < ((sl * r * SW_PC + 31) & ~31); e += nt) {
    const int p = e % SW_PC, t = e / SW_PC, j = t % r, s = t / r;
    T acc[RC];
#pragma unroll
    for (int q = 0; q < RC; ++q) acc[q] = zero<T>();
    if (s < sl) {
      const int a0 = row0(rank * sl + s) - i0, a1 = row0(rank * sl + s + 1) - i0;
      const T* f = stf ? Fs + (size_t)j * ldf : R.Ft + i0 + (size_t)j * c;
#pragma unroll 8
      for (int i = a0 + p; i < a1; i += SW_PC) {
        const T fv = f[i];
#pragma unroll
        for (int q = 0; q < RC; ++q) acc[q] = mad(acc[q], fv, yc[i * RC + q]);
      }
    }
    if constexpr (RC == 1) {
      acc[0] = part_sum<SW_PC>(acc[0]);
      if (s < sl && p == 0) gp[(size_t)s * r + j] = acc[0];
    } else {
      part_scatter<RC>(acc, p);
      if (s < sl) {
#pragma unroll
        for (int q = 0; q < RC / 4; ++q) gp[((size_t)s * r + j) * RC + own_column<RC>(p) + q] = acc[q];
      }
    }
  }
  cp_async_wait_group<0>();
  __syncthreads();
  cl.arrive();
  cl.wait();   // the slices' sums are complete, and every CTA has read y_C and y_R
  for (int e = tid; e < r * RC; e += nt) {
    T s = zero<T>();
    for (int g = 0; g < qc; g += 4) {   // four loads issued together, added in order
      T t[4];
#pragma unroll
      for (int h = 0; h < 4; ++h)
        if (g + h < qc) t[h] = cl.peer(gp + (size_t)((g + h) % sl) * r * RC + e, (g + h) / sl)[0];
#pragma unroll
      for (int h = 0; h < 4; ++h)
        if (g + h < qc) s = s + t[h];
    }
    z[e] = z[e] - s;
  }
  __syncthreads();
  cl.arrive();   // this CTA has read its peers' sums
  row_products<T, RC>(lw, r, nq, tid, nt, z, stw ? Ws : R.We + l0, stw ? ldw : n,
                      [&](int l) { return max(0, l0 + l - k); },   // rows of U^{-1} are zero left of the diagonal
                      [&](int l) { return (int64_t)(l0 + l < k ? R.idxC[l0 + l] : R.idxR[l0 + l - k]); },
                      [&](int l) { return l0 + l < k; }, true, xq, ldx);
  cl.wait();   // no CTA ends while its sums are read
}

// One colour class: cluster of Q CTAs per (box, RC columns).
template <typename T, int RC, bool UP>
__global__ void __launch_bounds__(SW_NT) k_sweep_cl(const BoxRec<T>* __restrict__ recs, T* __restrict__ x, int64_t ldx,
                                                    int nrhs, int Q, int qc, int sm_cap) {
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);
  pdl_launch();
  const int rank = blockIdx.x % Q, q0 = blockIdx.y * RC, nq = min(RC, nrhs - q0);
  const BoxRec<T> R = recs[blockIdx.x / Q];
  T* xq = x + q0;
  if (Q == 1) {
    if (UP) up_box<T, RC>(R, xq, ldx, nq, sm, sm_cap, 0, 1, true, SoloCta{});
    else down_box<T, RC>(R, xq, ldx, nq, sm, sm_cap, 0, 1, qc, true, SoloCta{});
  } else {
    if (UP) up_box<T, RC>(R, xq, ldx, nq, sm, sm_cap, rank, Q, true, ClusterCta{});
    else down_box<T, RC>(R, xq, ldx, nq, sm, sm_cap, rank, Q, qc, true, ClusterCta{});
  }
}

// ------------------------------------------------------------------ one persistent launch per sweep
// The sweeps as two cooperative launches of clusters of SW_QMAX CTAs: they walk the
// colour classes in factor order (upward) or reverse order (downward) and meet at a grid
// barrier between classes.  A class whose boxes have SW_QMAX slices of C, one too small to
// fill the GPU, takes a cluster per box (and RC columns), the others a CTA per box.  The
// same sums in the same order as the launches per class.  (One column, one CTA per box in
// every class, then this: Laplace 64^2 1.20, 0.42 ms, 1024^2 11.7, 4.5; Helmholtz 256^2 13.3,
// 2.3.)
constexpr int SWP_NT = 256;

// One colour class as the persistent sweeps see it (device array in factor order).
template <typename T> struct SwpClass {
  const BoxRec<T>* recs;
  int nrec, qc;
};

template <typename T> struct SwpArgs {
  const SwpClass<T>* cls;   // colour classes in factor order
  int ncls;
  T* x;
  int64_t ldx;
  int nrhs;
  unsigned* bar;            // grid barrier counters (zeroed before the launch)
  int* err;                 // RSS_ETIMEOUT when a barrier wait runs out
  long long polls;
  int sm_cap;               // scalars of dynamic shared memory
};

// whether v holds in every CTA of the cluster: its CTAs leave the sweep together (one that
// left alone would take the shared memory along that its peers write)
__device__ inline bool cluster_all(bool v) {
  __shared__ int s_v;
  namespace cg = cooperative_groups;
  if (threadIdx.x == 0) s_v = v;
  cg::this_cluster().sync();
  int all = 1;
  for (int q = 0; q < SW_QMAX; ++q) all &= *cg::this_cluster().map_shared_rank(&s_v, q);
  cg::this_cluster().sync();
  return all != 0;
}

template <typename T, int RC, bool UP> __global__ void __launch_bounds__(SWP_NT) k_sweep(SwpArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);
  const int nz = (a.nrhs + RC - 1) / RC;
  for (int step = 0; step < a.ncls; ++step) {
    const SwpClass<T> C = a.cls[UP ? step : a.ncls - 1 - step];
    const int Q = C.qc == SW_QMAX ? SW_QMAX : 1, rank = blockIdx.x % Q;
    for (int it = blockIdx.x / Q; it < C.nrec * nz; it += gridDim.x / Q) {
      const int q0 = (it / C.nrec) * RC, nq = min(RC, a.nrhs - q0);
      const BoxRec<T> R = C.recs[it % C.nrec];
      T* xq = a.x + q0;
      if (Q == 1) {
        if (UP) up_box<T, RC>(R, xq, a.ldx, nq, sm, a.sm_cap, 0, 1, false, SoloCta{});
        else down_box<T, RC>(R, xq, a.ldx, nq, sm, a.sm_cap, 0, 1, C.qc, false, SoloCta{});
      } else {
        if (UP) up_box<T, RC>(R, xq, a.ldx, nq, sm, a.sm_cap, rank, Q, false, ClusterCta{});
        else down_box<T, RC>(R, xq, a.ldx, nq, sm, a.sm_cap, rank, Q, C.qc, false, ClusterCta{});
      }
      __syncthreads();
    }
    if (step + 1 < a.ncls && !cluster_all(grid_barrier(a.bar, a.polls, a.err))) return;
  }
}
