// A_top^{-1} by in-place Gauss-Jordan elimination with partial pivoting, NB columns
// per step, two launches each: k_gj_panel (one CTA) picks the step's pivots by an
// LU of the panel's unused rows and inverts the pivot block, k_gj_update (the whole
// GPU) applies the step to every row and column, from one buffer to the other, with
// the row exchanges as an index list.  The solve needs the inverse only, so no LU is
// kept.  Bound by the FP64 pipe of one SM in the panel and by launch latency; an LU
// followed by triangular solves on the identity, which this replaces, was bound by
// one CTA's panel reads from L2.  445 real points: 5.7 -> 1.6 ms, 576: 6.8 -> 2.6,
// 500 complex: 11.9 -> 4.7.
template <typename T> constexpr int gj_nb() { return sizeof(T) == sizeof(double) ? 16 : 8; }

// Pivots of columns jb .. je from rows jb .. n: piv (absolute rows), src (the row of
// the input buffer that the exchanges bring to each place), D = (pivot block)^{-1}.
// The panel sits in shared memory, or in `scratch` when it does not fit.
template <typename T, int NB>
__global__ void __launch_bounds__(512) k_gj_panel(const T* __restrict__ in, int n, int jb, T* D, int* src, int* piv,
                                                  int* err, T* scratch) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int w = min(NB, n - jb), m = n - jb;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  int* ord = reinterpret_cast<int*>(smraw);   // m: the panel's rows in their new order
  T* A = scratch ? scratch : reinterpret_cast<T*>(smraw + (((size_t)m * sizeof(int) + 15) & ~size_t(15)));
  __shared__ int s_piv[2], s_zero[2];
  __shared__ __align__(16) unsigned char s_inv[NB * NB * sizeof(T)];
  for (int e = tid; e < m * w; e += blockDim.x) A[e] = in[jb + e % m + (size_t)(jb + e / m) * n];
  for (int i = tid; i < m; i += blockDim.x) ord[i] = jb + i;
  for (int i = tid; i < jb; i += blockDim.x) src[i] = i;
  __syncthreads();
  // as k_elim_lu2: warp 0 runs one column ahead of the others
  auto pivot = [&](int j) {
    T* col = A + (size_t)j * m;
    unsigned long long key = 0;
    int row = INT_MAX;
    for (int i = j + lane; i < m; i += 32) {
      const unsigned long long v = mod_key(col[i]);
      if (row == INT_MAX || v > key) {
        key = v;
        row = i;
      }
    }
    warp_argmax(key, row);
    if (key != 0) {
      const T p = col[row], t = col[j];
      __syncwarp();
      if (lane == 0) {
        col[row] = t;
        col[j] = p;
        const int o = ord[j];
        ord[j] = ord[row];
        ord[row] = o;
        piv[jb + j] = jb + row;
      }
      __syncwarp();
      const T d = dv(from_re<T>(1.0), p);
      for (int i = j + 1 + lane; i < m; i += 32) col[i] = col[i] * d;
    }
    if (lane == 0) {
      s_piv[j & 1] = row;
      s_zero[j & 1] = key == 0;
    }
  };
  auto update = [&](int j, int p, int jj) {
    T* col = A + (size_t)jj * m;
    const T* l = A + (size_t)j * m;
    const T u = col[p], v = col[j];
    __syncwarp();
    for (int i = j + lane; i < m; i += 32) {
      const T x = i == p ? v : col[i];
      col[i] = i == j ? u : msb(x, l[i], u);
    }
  };
  if (warp == 0) pivot(0);
  for (int j = 0; j < w; ++j) {
    __syncthreads();
    if (s_zero[j & 1]) {   // the inverse does not exist: every index stays within bounds
      if (tid == 0) set_error(err, RSS_ENUMERIC);
      for (int i = j + tid; i < w; i += blockDim.x) piv[jb + i] = jb + i;
      break;
    }
    const int p = s_piv[j & 1];
    if (warp == 0) {
      if (j + 1 < w) {
        update(j, p, j + 1);
        __syncwarp();
        pivot(j + 1);
      }
    } else {
      for (int jj = j + 1 + warp; jj < w; jj += nw - 1) update(j, p, jj);
      if (warp == nw - 1 && p != j && lane < j) {
        T* col = A + (size_t)lane * m;
        const T t = col[j];
        col[j] = col[p];
        col[p] = t;
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < m; i += blockDim.x) src[jb + i] = ord[i];
  // D = U^{-1} L^{-1}: one column per half warp, lane = row
  T* X = reinterpret_cast<T*>(s_inv);
  if (warp < NB / 2) {
    const int c = 2 * warp + (lane >> 4), i = lane & 15, base = lane & 16;
    const bool on = i < w && c < w;
    T x = (on && i == c) ? from_re<T>(1.0) : zero<T>();
    for (int s = 0; s < w; ++s) {
      const T y = shfl_idx(x, base + s);
      if (on && i > s) x = msb(x, A[i + (size_t)s * m], y);
    }
    T rec = from_re<T>(1.0);
    if (i < w) rec = dv(rec, A[i + (size_t)i * m]);
    for (int s = w - 1; s >= 0; --s) {
      if (i == s) x = x * rec;
      const T y = shfl_idx(x, base + s);
      if (on && i < s) x = msb(x, A[i + (size_t)s * m], y);
    }
    if (i < NB && c < NB) X[i + c * NB] = on ? x : zero<T>();
  }
  __syncthreads();
  for (int e = tid; e < NB * NB; e += blockDim.x) D[e] = X[e];
}

// One 32-row x 64-column tile of the step on columns jb .. je = J:
// rows outside J: x - (A_iJ D) A_J*, rows J: D A_J*, columns J: -A_iJ D and D.
template <typename T, int NB>
__global__ void __launch_bounds__(256) k_gj_update(const T* __restrict__ in, T* __restrict__ out, int n, int jb,
                                                   const T* __restrict__ D, const int* __restrict__ src) {
  const int w = min(NB, n - jb), i0 = blockIdx.y * 32, c0 = blockIdx.x * 64;
  __shared__ __align__(16) unsigned char s_raw[sizeof(T) * (NB * NB + 2 * 32 * (NB + 1) + NB * 64)];
  T* Ds = reinterpret_cast<T*>(s_raw);
  T* Ai = Ds + NB * NB;              // 32 x (NB + 1)
  T* Cp = Ai + 32 * (NB + 1);        // 32 x (NB + 1)
  T* Bt = Cp + 32 * (NB + 1);        // NB x 64
  const int tid = threadIdx.x, li = tid & 31, gi = tid >> 5;
  for (int e = tid; e < NB * NB; e += 256) Ds[e] = D[e];
  const int i = i0 + li, si = i < n ? src[i] : 0;
  for (int q = gi; q < NB; q += 8) Ai[li * (NB + 1) + q] = (i < n && q < w) ? in[si + (size_t)(jb + q) * n] : zero<T>();
  for (int e = tid; e < NB * 64; e += 256) {
    const int q = e % NB, c = c0 + e / NB;
    T v = zero<T>();
    if (q < w && c < n)
      v = (c >= jb && c < jb + w) ? (c - jb == q ? from_re<T>(1.0) : zero<T>()) : in[src[jb + q] + (size_t)c * n];
    Bt[q * 64 + e / NB] = v;
  }
  __syncthreads();
  const bool inJ = i >= jb && i < jb + w;
  for (int q = gi; q < NB; q += 8) {
    T x = zero<T>();
    if (inJ) {
      x = -Ds[(i - jb) + q * NB];
    } else {
#pragma unroll
      for (int s = 0; s < NB; ++s) x = mad(x, Ai[li * (NB + 1) + s], Ds[s + q * NB]);
    }
    Cp[li * (NB + 1) + q] = x;
  }
  __syncthreads();
  if (i >= n) return;
  T acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int c = c0 + gi * 8 + e;
    acc[e] = (c < n && !inJ && !(c >= jb && c < jb + w)) ? in[si + (size_t)c * n] : zero<T>();
  }
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const T cv = Cp[li * (NB + 1) + q];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = msb(acc[e], cv, Bt[q * 64 + gi * 8 + e]);
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int c = c0 + gi * 8 + e;
    if (c < n) out[i + (size_t)c * n] = acc[e];
  }
}

// Column c of the inverse: the row exchanges undone as column exchanges, last first.
template <typename T>
__global__ void __launch_bounds__(128) k_gj_columns(const T* __restrict__ in, T* __restrict__ out, int n,
                                                    const int* __restrict__ piv) {
  __shared__ int s_c;
  const int c = blockIdx.x;
  if (threadIdx.x == 0) {
    int pos = c;
#pragma unroll 8
    for (int j = 0; j < n; ++j) {
      const int p = piv[j];
      pos = pos == j ? p : pos == p ? j : pos;
    }
    s_c = pos;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) out[i + (size_t)c * n] = in[i + (size_t)s_c * n];
}

// inv = (the n x n matrix in buf[0])^{-1}; buf[1], D, src, piv and (for panels that
// do not fit on chip) scratch are workspace.  Returns the launches made, or a
// negative value on a launch failure.
template <typename T>
int gj_inverse(T* const buf[2], T* inv, int n, T* D, int* src, int* piv, int* err, T* scratch, cudaStream_t st) {
  constexpr int NB = gj_nb<T>();
  const size_t ib = ((size_t)n * sizeof(int) + 15) & ~size_t(15);
  const size_t full = ib + sizeof(T) * (size_t)n * NB;
  if (ib > 200 * 1024) return -1;
  const bool onchip = full <= 200 * 1024;
  const size_t smem = onchip ? full : ib;
  if (allow_smem(k_gj_panel<T, NB>) != cudaSuccess) return -1;
  int cur = 0, launches = 0;
  for (int jb = 0; jb < n; jb += NB) {
    k_gj_panel<T, NB><<<1, 512, smem, st>>>(buf[cur], n, jb, D, src, piv, err, onchip ? nullptr : scratch);
    k_gj_update<T, NB><<<dim3((n + 63) / 64, (n + 31) / 32), 256, 0, st>>>(buf[cur], buf[cur ^ 1], n, jb, D, src);
    cur ^= 1;
    launches += 2;
  }
  k_gj_columns<T><<<n, 128, 0, st>>>(buf[cur], inv, n, piv);
  return cudaGetLastError() == cudaSuccess ? launches + 1 : -1;
}
