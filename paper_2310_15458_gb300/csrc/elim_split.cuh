// Sparsification, LU and inverses of a colour class's boxes (Eqs. 7, 8) in three
// kernels, so that a box is shared by many CTAs wherever its work is independent:
//   k_elim_x   X_RR, a group of columns per CTA (and the box's index lists);
//   k_elim_lu2 P X_RR = L U, one CTA per box, one block barrier per column;
//   k_elim_inv U^{-1}, L^{-1} P and from them W_E, W_F, a group of columns per CTA.
// All are bound by the FP64 pipe (two FMAs per clock and SM): one CTA alone
// needs 0.3 ms for a real box of 112 points and 1.1 ms for a complex one, and the
// coarse colour classes hold one to nine boxes.  Elimination phase, one kernel per box
// before, this after: Helmholtz 256^2 86.9 -> 41.3 ms, Laplace 64^2 (eps 1e-8)
// 10.3 -> 4.2, 256^2 16.3 -> 10.4, 1024^2 70.9 -> 60.1.

// CT columns per thread, two threads per row: 2 CT columns of X_RR per CTA.
// V = A_BB [-T; I] restricted to the group: V_S = X_SR, then
// X_RR = V_R - T^* V_S (Eq. 7).
template <typename T, int CT> __global__ void __launch_bounds__(256) k_elim_x(ElimArgs<T> a) {
  constexpr int JC = 2 * CT;
  extern __shared__ __align__(16) unsigned char smraw[];
  const LevelDev<T>& L = a.L;
  const BoxRec<T> R = a.recs[blockIdx.y];
  const int nmax = L.nmax, g = L.g, B = R.box, k = R.k, r = R.r, c = R.c, n = k + r;
  const int j0 = blockIdx.x * JC;
  if (j0 >= r) return;
  const size_t nn = (size_t)nmax * nmax;
  const int* perm = a.perm_in + (size_t)a.cls_idx[blockIdx.y] * nmax;
  const T* __restrict__ Tw = a.T_ws + (size_t)a.cls_idx[blockIdx.y] * nn;
  const T* __restrict__ Abb = L.blk + ((size_t)B * 25 + 12) * nn;
  const int tid = threadIdx.x, jw = min(JC, r - j0);
  T* Ts = reinterpret_cast<T*>(smraw);   // k x JC: T(:, group)
  T* Vs = Ts + (size_t)k * JC;           // k x JC: X_SR(:, group)
  int* sp = reinterpret_cast<int*>(Vs + (size_t)k * JC);   // n: B's points in pivot order
  for (int i = tid; i < n; i += 256) sp[i] = perm[i];
  for (int e = tid; e < k * JC; e += 256) {
    const int q = e % k, j = e / k;
    Ts[q * JC + j] = j < jw ? Tw[(size_t)(j0 + j) * nmax + q] : zero<T>();
  }
  __syncthreads();
  for (int e = tid; e < k * jw; e += 256) {
    const int i = e % k, j = e / k;
    T x = Abb[(size_t)sp[k + j0 + j] * nmax + sp[i]];
    for (int q = 0; q < k; ++q) x = msb(x, Abb[(size_t)sp[q] * nmax + sp[i]], Ts[q * JC + j]);
    Vs[i * JC + j] = x;
    R.Tm[(size_t)(j0 + j) * k + i] = Ts[i * JC + j];
  }
  if (blockIdx.x == 0) {   // the box's index lists
    __shared__ int nb[9], coff[10], ord[9];
    if (tid == 0) {
      const int o9[9] = {4, 0, 1, 2, 3, 5, 6, 7, 8};
      int off = 0;
      for (int q = 0; q < 9; ++q) {
        const int s = o9[q];
        ord[q] = s;
        nb[s] = nbr_box(B, g, s % 3 - 1, s / 3 - 1);
        coff[q] = off;
        off += s == 4 ? k : (nb[s] >= 0 ? L.nact[nb[s]] : 0);
      }
      coff[9] = off;
    }
    __syncthreads();
    for (int i = tid; i < c; i += 256) {
      int q = 0;
      while (coff[q + 1] <= i) ++q;
      const int s = ord[q], ii = i - coff[q], u = nb[s];
      const int pos = s == 4 ? sp[ii] : L.act[u * nmax + ii];
      R.cmap[i] = (s << 16) | pos;
      R.idxC[i] = L.pts[u * nmax + pos];
    }
    for (int j = tid; j < r; j += 256) R.idxR[j] = L.pts[B * nmax + sp[k + j]];
    // B keeps only its skeleton
    for (int q = tid; q < k; q += 256) L.act[B * nmax + q] = sp[q];
    if (tid == 0) L.nact[B] = k;
  }
  __syncthreads();
  const int row = tid >> 1, h = (tid & 1) * CT;
  for (int i = row; i < r; i += 128) {
    const int pi = sp[k + i];
    T x[CT];
#pragma unroll
    for (int j = 0; j < CT; ++j) x[j] = h + j < jw ? Abb[(size_t)sp[k + j0 + h + j] * nmax + pi] : zero<T>();
    const T* ti = Tw + (size_t)i * nmax;
#pragma unroll 4
    for (int q = 0; q < k; ++q) {
      const T av = Abb[(size_t)sp[q] * nmax + pi];
#pragma unroll
      for (int j = 0; j < CT; ++j) x[j] = msb(x[j], av, Ts[q * JC + h + j]);
    }
#pragma unroll 4
    for (int q = 0; q < k; ++q) {
      const T tv = ti[q];
#pragma unroll
      for (int j = 0; j < CT; ++j) x[j] = msbc(x[j], tv, Vs[q * JC + h + j]);
    }
#pragma unroll
    for (int j = 0; j < CT; ++j)
      if (h + j < jw) R.LU[i + (size_t)(j0 + h + j) * r] = x[j];
  }
}
template <typename T> size_t elim_x_bytes(int CT, int k, int n) {
  return sizeof(T) * 4 * (size_t)CT * k + sizeof(int) * (size_t)n;
}

__device__ __forceinline__ double shfl_idx(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ zd shfl_idx(zd v, int l) { return zd{shfl_idx(v.x, l), shfl_idx(v.y, l)}; }

// largest |x| of a warp's lanes and its lowest row: key an ordered non-negative
// integer, row < 2^31 (lanes without an entry: key 0, row INT_MAX)
__device__ __forceinline__ void warp_argmax(unsigned long long& key, int& row) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(key >> 32));
  const bool a = (uint32_t)(key >> 32) == hi;
  const uint32_t lo = __reduce_max_sync(0xffffffffu, a ? (uint32_t)key : 0u);
  const bool b = a && (uint32_t)key == lo;
  row = (int)__reduce_min_sync(0xffffffffu, b ? (uint32_t)row : (uint32_t)INT_MAX);
  key = ((unsigned long long)hi << 32) | lo;
}
// |x| (complex: |x|^2) as such a key; a NaN is never the pivot
__device__ __forceinline__ unsigned long long mod_key(double x) {
  const unsigned long long b = oz_abs_bits(x);
  return b > 0x7FF0000000000000ull ? 0ull : b;
}
__device__ __forceinline__ unsigned long long mod_key(zd x) { return mod_key(abs2(x)); }

// P X_RR = L U by the whole CTA, partial pivoting (largest modulus, lowest row on
// ties).  Warp 0 runs one column ahead: it updates column j + 1, finds its pivot
// and scales it while the other warps finish step j, so a step has one block
// barrier.  A row exchange is applied by the warp that updates the column; the
// columns left of the pivot are exchanged by the last warp.  The exchange order
// pos (P e_m = e_pos[m]) goes to R.pos.
template <typename T> __global__ void __launch_bounds__(256) k_elim_lu2(ElimArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<T> R = a.recs[blockIdx.x];
  const int r = R.r, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const bool onchip = (size_t)r * (r | 1) <= (size_t)a.smem_cap;
  const int ld = onchip ? r | 1 : r;
  T* A = onchip ? reinterpret_cast<T*>(smraw) : R.LU;
  __shared__ int s_piv[2], s_zero[2];
  if (onchip)
    for (int e = tid; e < r * r; e += blockDim.x) A[e % r + (size_t)(e / r) * ld] = R.LU[e];
  __syncthreads();
  // pivot of column j (rows j ..), exchanged and scaled inside the column (warp 0)
  auto pivot = [&](int j) {
    T* col = A + (size_t)j * ld;
    unsigned long long key = 0;
    int row = INT_MAX;
    for (int i = j + lane; i < r; i += 32) {
      const unsigned long long v = mod_key(col[i]);
      if (row == INT_MAX || v > key) {
        key = v;
        row = i;
      }
    }
    warp_argmax(key, row);
    const bool zero_piv = key == 0;
    if (!zero_piv) {
      const T p = col[row], t = col[j];
      __syncwarp();
      if (lane == 0) {
        col[row] = t;
        col[j] = p;
      }
      __syncwarp();
      const T d = dv(from_re<T>(1.0), p);
      for (int i = j + 1 + lane; i < r; i += 32) col[i] = col[i] * d;
    }
    if (lane == 0) {
      s_piv[j & 1] = row;
      s_zero[j & 1] = zero_piv;
      if (!zero_piv) R.piv[j] = row;
    }
  };
  // column jj of step j: rows j and p exchanged, then the rank-1 update
  auto update = [&](int j, int p, int jj) {
    T* col = A + (size_t)jj * ld;
    const T* l = A + (size_t)j * ld;
    const T u = col[p], v = col[j];
    __syncwarp();
    for (int i = j + lane; i < r; i += 32) {
      const T x = i == p ? v : col[i];
      col[i] = i == j ? u : msb(x, l[i], u);
    }
  };
  if (warp == 0) pivot(0);
  for (int j = 0; j < r; ++j) {
    __syncthreads();
    if (s_zero[j & 1]) {   // every later kernel of the level still indexes within bounds
      if (tid == 0) set_error(a.err, RSS_ENUMERIC);
      for (int i = j + tid; i < r; i += blockDim.x) R.piv[i] = i;
      break;
    }
    const int p = s_piv[j & 1];
    if (warp == 0) {
      if (j + 1 < r) {
        update(j, p, j + 1);
        __syncwarp();
        pivot(j + 1);
      }
    } else {
      for (int jj = j + 1 + warp; jj < r; jj += nw - 1) update(j, p, jj);
      if (warp == nw - 1 && p != j)
        for (int q = lane; q < j; q += 32) {
          T* col = A + (size_t)q * ld;
          const T t = col[j];
          col[j] = col[p];
          col[p] = t;
        }
    }
  }
  __syncthreads();
  if (onchip)
    for (int e = tid; e < r * r; e += blockDim.x) R.LU[e] = A[e % r + (size_t)(e / r) * ld];
  __syncthreads();
  int* sig = reinterpret_cast<int*>(smraw);   // the rows of the identity through the exchanges, then its inverse
  for (int i = tid; i < r; i += blockDim.x) sig[i] = i;
  __syncthreads();
  if (tid == 0)
    for (int i = 0; i < r; ++i) {
      const int q = R.piv[i];
      if (q != i) {
        const int t = sig[i];
        sig[i] = sig[q];
        sig[q] = t;
      }
    }
  __syncthreads();
  for (int i = tid; i < r; i += blockDim.x) R.pos[sig[i]] = i;
}

// One group of NBC columns of M^{-1} for M = U (blockIdx.y = 0) or M = L^T (1, so
// a column is a row of L^{-1}), both upper triangular, by 16-row blocks from the
// diagonal up: X_I = -M_II^{-1} sum_{I < l} M_Il X_l.  Thread (i, c) = (tid / NBC,
// tid % NBC) owns entry (i, c) of a block.  Then the group's columns of W_E or W_F.
template <typename T, int NBC> __global__ void __launch_bounds__(16 * NBC) k_elim_inv(ElimArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<T> R = a.recs[blockIdx.z];
  const int k = R.k, r = R.r, n = k + r, which = blockIdx.y, c0 = blockIdx.x * NBC;
  if (c0 >= r) return;
  constexpr int NTH = 16 * NBC;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cw = min(NBC, r - c0), nbk = (c0 + cw + 15) / 16;   // row blocks of the group
  T* X = reinterpret_cast<T*>(smraw);               // 16 nbk x NBC
  T* S = X + (size_t)16 * nbk * NBC;                // 16 x NBC
  T* D = S + 16 * NBC;                              // nbk blocks of 16 x 17: M_II^{-1}, column-major
  const T* __restrict__ LU = R.LU;
  const size_t si = which ? r : 1, sl = which ? 1 : r;   // M(i, l) = LU[i si + l sl], l > i
  // inverses of the diagonal blocks: lane (column c of 16, half h); a column is
  // eliminated from the bottom, the halves share the rows above
  for (int b = warp; b < nbk; b += NTH / 32) {
    const int r0 = 16 * b, rw = min(16, r - r0), cc = lane & 15, h = lane >> 4;
    T* d = D + (size_t)b * 16 * 17 + cc * 17;
    for (int i = h; i < 16; i += 2) d[i] = (i == cc && i < rw) ? from_re<T>(1.0) : zero<T>();
    T rec = from_re<T>(1.0);
    if (which == 0 && cc < rw) rec = dv(rec, LU[(size_t)(r0 + cc) * (r + 1)]);
    __syncwarp();
    for (int i = rw - 1; i >= 0; --i) {
      T x = d[i];
      if (which == 0) x = x * shfl_idx(rec, i);
      __syncwarp();
      if (h == 0) d[i] = x;
      if (cc >= i)
        for (int l = h; l < i; l += 2) d[l] = msb(d[l], LU[(size_t)(r0 + l) * si + (size_t)(r0 + i) * sl], x);
      __syncwarp();
    }
  }
  __syncthreads();
  const int ti = tid / NBC, tc = tid % NBC;
  for (int I = nbk - 1; I >= 0; --I) {
    const int i0 = 16 * I, i = i0 + ti, cg = c0 + tc;   // entry (i, cg); the group's own rows start the recursion
    T s = (i == cg && cg < r) ? from_re<T>(1.0) : zero<T>();
    const T* mr = LU + (size_t)min(i, r - 1) * si;
    const int l1 = min(16 * nbk, r);
#pragma unroll 4
    for (int l = i0 + 16; l < l1; ++l) s = msb(s, mr[(size_t)l * sl], X[l * NBC + tc]);
    S[ti * NBC + tc] = s;
    __syncthreads();
    T x = zero<T>();
    const T* d = D + (size_t)I * 16 * 17;
#pragma unroll 4
    for (int l = ti; l < 16; ++l) x = mad(x, d[l * 17 + ti], S[l * NBC + tc]);
    X[i * NBC + tc] = i < r ? x : zero<T>();
    __syncthreads();
  }
  const int rows = min(16 * nbk, r);   // rows past the group's are zero
  if (which == 0) {
    for (int e = tid; e < r * cw; e += NTH) {
      const int i = e % r, j = e / r;
      const T x = i < rows ? X[i * NBC + j] : zero<T>();
      if (R.Ui) R.Ui[i + (size_t)(c0 + j) * r] = x;
      R.We[(size_t)(c0 + j) * n + k + i] = x;
    }
    for (int e = tid; e < k * cw; e += NTH) {   // W_E = [-T U^{-1}; U^{-1}]
      const int l = e % k, j = e / k;
      T x = zero<T>();
#pragma unroll 4
      for (int m = 0; m < rows; ++m) x = msb(x, R.Tm[l + (size_t)m * k], X[m * NBC + j]);
      R.We[(size_t)(c0 + j) * n + l] = x;
    }
  } else {
    // row c0 + j of L^{-1} P: entry m is entry pos(m) of the row of L^{-1}
    const int* pos = R.pos;
    if (R.Li)
      for (int e = tid; e < r * NBC; e += NTH) {
        const int j = e % NBC, m = e / NBC;
        if (j < cw) R.Li[(c0 + j) + (size_t)m * r] = m < rows ? X[m * NBC + j] : zero<T>();
      }
    // W_F = [-(L^{-1} P T^*)^T; (L^{-1} P)^T]
    for (int e = tid; e < r * cw; e += NTH) {
      const int m = e % r, j = e / r, pm = pos[m];
      R.Wf[(size_t)(c0 + j) * n + k + m] = pm < rows ? X[pm * NBC + j] : zero<T>();
    }
    for (int e = tid; e < k * cw; e += NTH) {
      const int l = e % k, j = e / k;
      T x = zero<T>();
#pragma unroll 4
      for (int m = 0; m < r; ++m) {
        const int pm = pos[m];
        if (pm < rows) x = msb(x, X[pm * NBC + j], cj(R.Tm[l + (size_t)m * k]));
      }
      R.Wf[(size_t)(c0 + j) * n + l] = x;
    }
  }
}
template <typename T> size_t elim_inv_bytes(int NBC, int r) {
  const size_t nbk = (size_t)(r + 15) / 16;
  return sizeof(T) * (16 * nbk * NBC + 16 * (size_t)NBC + nbk * 16 * 17);
}
