// RS-S factorization on the device (Algorithm 1), batched by colour class.
//
// Per level (box grid side g >= 4) and per colour class (ix mod 3, iy mod 3),
// all boxes of the class are pairwise more than distance 2 apart (Section 3),
// so each phase handles the whole class in one launch:
//   k_id      : proxy stack Y = [A_MB; K_PB; A_BM^*; K_BP^*] (Eqs. 4-6) and its
//               column-pivoted Householder QR, truncated at eps (Definition 1);
//   k_elim    : sparsification (Eq. 7), LU of X_RR, E = X_CR U^{-1} and
//               F = L^{-1} P X_RC (Eq. 8);
//   k_schur   : A_CC -= E F scattered into the stencil blocks (Remark 2);
// then the merge to the parent level (Section 2.4) and a dense LU at the top.
//
// Matrix storage: for each box u of a level, 25 blocks A(u, v), v = u + (dx, dy),
// |dx|, |dy| <= 2, each nmax x nmax column-major over the level-start point
// lists of u and v.  A box's active points are a position list into its
// level-start list (the skeleton after elimination); far pairs (distance > 2)
// are never stored because they are never modified (Theorem 1).
#include <algorithm>
#include <chrono>
#include <climits>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "internal.h"
#include "tw_common.cuh"

namespace {

// Pivot ties: remaining squared norms within TIE_REL n_max + TIE_ABS sqrt(n_max y2max)
// of the maximum n_max (y2max: largest initial squared column norm) are rounding
// noise apart and count as tied; the lowest original column wins.
constexpr double TIE_REL = 1e-6;
constexpr double TIE_ABS = 1e-12;
// A downdated squared norm is re-accumulated once it falls below sqrt(unit
// roundoff) of its last accumulated value (LAPACK geqp3's rule); between
// re-accumulations it is accurate to a few 1e-8 relative, inside the tie window.
constexpr double RECOMPUTE_REL = 1.4901161193847656e-08;
constexpr int NT = 256;                 // threads per CTA for the per-box kernels

template <typename T> struct LevelDev {
  int g, nbox, nmax;
  int* pts;    // nbox x nmax tree indices (level-start points)
  int* n;      // nbox
  int* act;    // nbox x nmax active positions
  int* nact;   // nbox
  T* blk;      // nbox x 25 x nmax x nmax
};

__device__ __forceinline__ int nbr_box(int u, int g, int dx, int dy) {
  int bx = u % g + dx, by = u / g + dy;
  return (bx < 0 || by < 0 || bx >= g || by >= g) ? -1 : by * g + bx;
}
__device__ __forceinline__ int off_index(int u, int v, int g) {
  return (v / g - u / g + 2) * 5 + (v % g - u % g + 2);
}
__device__ __forceinline__ int cheb(int u, int v, int g) {
  return max(abs(u % g - v % g), abs(u / g - v / g));
}

template <typename T> __device__ T block_sum(T v, T* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < nw ? sh[lane] : zero<T>();
    v = warp_sum(v);
    if (lane == 0) sh[0] = v;
  }
  __syncthreads();
  return sh[0];
}

__device__ inline double warp_max(double v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}

// ------------------------------------------------------------------ kernel table
// tab[(dy + s - 1) (2s - 1) + (dx + s - 1)] = K at grid displacement (dx, dy) != 0.
template <typename T> __global__ void k_ktab(T* tab, int side, KParams kp, Geo geo) {
  const long long w = 2 * side - 1, tot = w * w;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    const int dx = (int)(e % w) - (side - 1), dy = (int)(e / w) - (side - 1);
    tab[e] = (dx == 0 && dy == 0) ? zero<T>() : kval(kp, dx * geo.hg, dy * geo.hg, 0.0, 0.0, T{});
  }
}

// Lippmann-Schwinger weights w = kappa sqrt(b(x)) = kappa exp(-bump_a |x - c|^2 / 2)
// at each grid point (iy * side + ix)   (Eq. 19)
__global__ void k_ls_weights(double* w, int side, Geo geo, double kappa, double cx, double cy, double a) {
  const long long n = (long long)side * side;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const double x = geo.x0 + (e % side) * geo.hg - cx, y = geo.y0 + (e / side) * geo.hg - cy;
    w[e] = kappa * exp(-0.5 * a * (x * x + y * y));
  }
}

// ------------------------------------------------------------------ leaf generation
template <typename T>
__global__ void __launch_bounds__(NT) k_gen_blocks(LevelDev<T> L, const int2* __restrict__ ixy,
                                                   const T* __restrict__ tab, KParams kp, int side) {
  const int u = blockIdx.x / 25, o = blockIdx.x % 25;
  const int v = nbr_box(u, L.g, o % 5 - 2, o / 5 - 2);
  if (v < 0) return;
  const int nu = L.n[u], nv = L.n[v];
  // grid coordinates of both boxes' points, read once (leaf boxes: at most 256 points)
  __shared__ int2 gu[256], gv[256];
  for (int i = threadIdx.x; i < nu; i += blockDim.x) gu[i] = ixy[L.pts[u * L.nmax + i]];
  for (int j = threadIdx.x; j < nv; j += blockDim.x) gv[j] = ixy[L.pts[v * L.nmax + j]];
  __syncthreads();
  T* A = L.blk + ((size_t)u * 25 + o) * L.nmax * L.nmax;
  if (nu == 0) return;
  // entry e = i + j nu, stepped by the block size without a division per entry
  const int di = (int)blockDim.x % nu, dj = (int)blockDim.x / nu;
  int i = (int)threadIdx.x % nu, j = (int)threadIdx.x / nu;
  for (; j < nv; i += di, j += dj) {
    if (i >= nu) {
      i -= nu;
      ++j;
      if (j >= nv) break;
    }
    A[(size_t)j * L.nmax + i] = aval_tab<T>(kp, tab, side, gu[i], gv[j]);
  }
}

// ------------------------------------------------------------------ ID (Definition 1, Eq. 6)
// One CTA per box.  Y = [A_MB; K_PB; A_BM^*; K_BP^*] is assembled once and then
// only read: the Householder reflectors H_l = I - tau_l v_l v_l^H are kept as
// V (m x k) and G (n x k) with H_{j-1}..H_0 Y = Y - V G^T (column c of G holds
// tau_l v_l^H (H_{l-1}..H_0 Y)[:, c]), so a step costs one product v^H Y over
// the remaining columns plus O((m + n) j) corrections, the pivot column and row j
// of R are formed on demand, and Y is never rewritten.  In exact arithmetic this
// is the same sequence of reflectors and pivots as updating Y in place.
constexpr int NT_ID = 256;
// Cluster ID (small colour classes): up to CL_QMAX CTAs per box (above 8 a
// non-portable cluster size), NTC threads per CTA: 512 when every CTA of the
// launch gets an SM of its own (more warps share the per-step dot products of
// the reflector with the owned rows), else 256, two CTAs per SM.
constexpr int CL_QMAX = 16;
constexpr int CL_QDEF = 8;   // the largest size the default policy takes
// stride of one of the two partial-sum buffers of the cluster ID: a vector of up
// to 2 nmax sums, or 2 scalars plus one partial per warp
template <int NTC> __host__ __device__ inline int cl_part_stride(int nmax) {
  return 2 * nmax > 2 + NTC / 32 ? 2 * nmax : 2 + NTC / 32;
}

// T: arithmetic of the ID; S: scalar of the matrix.  T = double with S = zd is
// the complex symmetric case (Helmholtz): there A_BM^* = conj(A_MB) and
// K_BP^* = conj(K_PB) hold through the eliminations (T stays real, so the
// Schur updates keep A complex symmetric), the stack is [X; conj X] with
// X = [A_MB; K_PB], and its Gram matrix 2 Re(X^H X) is that of the real matrix
// sqrt(2) [Re X; Im X].  Column-pivoted QR sees Y only through its Gram matrix
// (norms, pivots, R up to unimodular row scales, ||R22||, T = R11^{-1} R12), so
// the real stack [Re X; Im X] gives the same ID with T real, at a quarter of
// the arithmetic.
template <typename T, typename S = T> struct IdArgs {
  LevelDev<S> L;
  const int* boxes;   // colour class
  int base;           // first box of this chunk within the class
  T* ws;              // chunk workspace: per box Y (ldY x nmax), V (ldY x nmax), G, Rr (nmax x nmax)
  int ldY;
  int half;           // 1: rows [A_MB; K_PB] only (real symmetric kernel)
  int* k_out;         // per class box
  int* perm_out;      // class x nmax
  S* T_ws;            // class x nmax x nmax (k x r, ld nmax)
  const int2* ixy;
  KParams kp;
  Geo geo;
  double eps;
  int P;              // proxy points
  double rho;         // proxy radius
  double Lbox;        // box side
  int g_sm;           // 1: G (nmax x nmax) and row k of V are kept in shared memory
  const S* ptab;      // proxy rows K(y_p, x) by the point's place in its box (null: evaluated here)
  int lsz;            // grid points per box side at this level
};

template <typename T, typename S> __device__ inline S id_store(T v) {
  if constexpr (std::is_same<T, S>::value) return v;
  else return S{v, 0.0};
}
template <typename T, typename S> __device__ inline T id_load(S v) {
  if constexpr (std::is_same<T, S>::value) return v;
  else return v.x;
}

// Entry (i, j) of the proxy stack of box B (Eq. 6): rows [A_MB; K_PB] then
// [A_BM^*; K_BP^*]; with T real and S complex, [Re X; Im X] for X = [A_MB; K_PB].
// Mbox/Moff: the distance-2 boxes and their row offsets, mh = their active rows,
// (cx, cy) the box centre; column j is point j of B (identity active list).
template <typename T, typename S>
__device__ __forceinline__ T id_entry(const IdArgs<T, S>& a, int B, int i, int j, int mh, const int* Mbox,
                                      const int* Moff, double cx, double cy) {
  const LevelDev<S>& L = a.L;
  const int nmax = L.nmax, g = L.g, P = a.P;
  const size_t nn = (size_t)nmax * nmax;
  constexpr bool split = !std::is_same<T, S>::value;
  bool second = i >= mh + P;                // conjugate half (or imaginary parts)
  const int ii = second ? i - mh - P : i;   // row of X
  S v;
  if (ii < mh) {
    int q = 0;
    while (Moff[q + 1] <= ii) ++q;
    const int mb = Mbox[q];
    const int pm = L.act[mb * nmax + (ii - Moff[q])];
    if (split || !second)
      v = L.blk[((size_t)mb * 25 + off_index(mb, B, g)) * nn + (size_t)j * nmax + pm];
    else
      v = cj(L.blk[((size_t)B * 25 + off_index(B, mb, g)) * nn + (size_t)pm * nmax + j]);
  } else {
    const int p = ii - mh;
    const int2 q = a.ixy[L.pts[B * nmax + j]];
    if (a.ptab != nullptr && (split || !second)) {   // K(y_p, x_j) from the level's table
      const int local = (q.y - (B / g) * a.lsz) * a.lsz + (q.x - (B % g) * a.lsz);
      v = a.ptab[(size_t)p * a.lsz * a.lsz + local];
    } else {
      double sn, cs;
      sincospi(2.0 * p / P, &sn, &cs);
      const double px = cx + a.rho * cs, py = cy + a.rho * sn;
      const double xj = a.geo.x0 + q.x * a.geo.hg, yj = a.geo.y0 + q.y * a.geo.hg;
      v = (!split && second) ? cj(kval(a.kp, xj, yj, px, py, S{})) : kval(a.kp, px, py, xj, yj, S{});
    }
    if (a.kp.kind == RSS_HELMHOLTZ_LS)   // proxy weight kappa, column weight w_j
      v = (a.kp.kappa * a.kp.w[q.y * a.geo.side + q.x]) * v;
  }
  if constexpr (split) return second ? v.y : v.x;
  else return v;
}

// Proxy rows by place (Eq. 6): on the uniform grid the box centre, the proxy
// circle and the box's grid points move together from box to box, and every
// kernel kind depends only on x - y, so K(y_p, x) for a point x of box B is a
// function of p and of x's place (ox, oy) inside B (lsz x lsz places): one table
// per level, tab[p * lsz^2 + oy * lsz + ox], serves the proxy rows of every box.
// The coordinates are taken relative to the box centre, y_p - x =
// rho (cos, sin)(2 pi p / P) - ((ox, oy) + 1/2 - lsz/2) hg.
template <typename S>
__global__ void __launch_bounds__(NT) k_proxy_tab(S* __restrict__ tab, int lsz, int P, double rho, double hg,
                                                  KParams kp) {
  const long long nloc = (long long)lsz * lsz, tot = nloc * P;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int p = (int)(e / nloc), o = (int)(e % nloc), ox = o % lsz, oy = o / lsz;
    double sn, cs;
    sincospi(2.0 * p / P, &sn, &cs);
    const double xr = (ox + 0.5 - 0.5 * lsz) * hg, yr = (oy + 0.5 - 0.5 * lsz) * hg;
    tab[e] = kval(kp, rho * cs - xr, rho * sn - yr, 0.0, 0.0, S{});
  }
}

template <typename T, typename S = T> __global__ void __launch_bounds__(NT_ID, 4) k_id(IdArgs<T, S> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const LevelDev<S>& L = a.L;
  const int nmax = L.nmax, g = L.g, ldY = a.ldY;
  T* vbuf = reinterpret_cast<T*>(smraw);          // ldY: current reflector
  T* u = vbuf + ldY;                              // nmax: V^H v
  T* beta = u + nmax;                             // nmax: R diagonal
  double* norms2 = reinterpret_cast<double*>(beta + nmax);
  double* ref = norms2 + nmax;
  double* taus = ref + nmax;
  int* perm = reinterpret_cast<int*>(taus + nmax);
  int* flag = perm + nmax;
  T* Gs = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(smraw) +
                               ((reinterpret_cast<unsigned char*>(flag + nmax) - smraw + 15) & ~size_t(15)));
  T* vrow = Gs + (size_t)nmax * nmax;             // row k of V (a.g_sm)
  __shared__ int Mbox[16], Moff[17], s_nM, s_piv, s_stop;
  __shared__ double s_thresh, s_y2max, s_redd[32];
  __shared__ T s_scale;

  const int bi = a.base + blockIdx.x;
  const int B = a.boxes[bi];
  const size_t nn = (size_t)nmax * nmax;
  const int n = L.n[B];
  const size_t slot = 2 * (size_t)ldY * nmax + 2 * nn;
  const T* Y = a.ws + (size_t)blockIdx.x * slot;
  T* Yw = a.ws + (size_t)blockIdx.x * slot;
  T* V = Yw + (size_t)ldY * nmax;
  T* G = a.g_sm ? Gs : V + (size_t)ldY * nmax;   // G[l * nmax + c]
  T* Rr = V + (size_t)ldY * nmax + nn;            // Rr[i * nmax + c]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;

  if (tid == 0) {
    int cnt = 0, off = 0;
    for (int dy = -2; dy <= 2; ++dy)
      for (int dx = -2; dx <= 2; ++dx) {
        if (max(abs(dx), abs(dy)) != 2) continue;
        const int mb = nbr_box(B, g, dx, dy);
        if (mb < 0) continue;
        Mbox[cnt] = mb;
        Moff[cnt] = off;
        off += L.nact[mb];
        ++cnt;
      }
    Moff[cnt] = off;
    s_nM = cnt;
  }
  __syncthreads();
  const int nM = s_nM, mh = Moff[nM], P = a.P;
  const int m = a.half ? mh + P : 2 * (mh + P);
  const int bx = B % g, by = B / g;
  const double cx = a.geo.x0 - 0.5 * a.geo.hg + (bx + 0.5) * a.Lbox;
  const double cy = a.geo.y0 - 0.5 * a.geo.hg + (by + 0.5) * a.Lbox;

  // Y, column-major; column j = point j of B (not yet eliminated: identity active list)
  for (long long e = tid; e < (long long)m * n; e += blockDim.x) {
    const int i = (int)(e % m), j = (int)(e / m);
    Yw[(size_t)j * ldY + i] = id_entry(a, B, i, j, mh, Mbox, Moff, cx, cy);
  }
  __syncthreads();
  for (int c = warp; c < n; c += nwarp) {
    double s = 0.0;
    for (int i = lane; i < m; i += 32) s += abs2(Y[(size_t)c * ldY + i]);
    s = warp_sum(s);
    if (lane == 0) {
      norms2[c] = s;
      ref[c] = s;
      perm[c] = c;
    }
  }
  __syncthreads();
  if (warp == 0) {
    double s = 0.0, mx = 0.0;
    for (int c = lane; c < n; c += 32) {
      s += norms2[c];
      mx = fmax(mx, norms2[c]);
    }
    s = warp_sum(s);
    mx = warp_max(mx);
    if (lane == 0) {
      s_thresh = a.eps * a.eps * s;
      s_y2max = mx;
    }
  }
  __syncthreads();

  int k = 0;
  const int kmax = min(m, n);
  while (k < kmax) {
    // stop test and pivot: largest remaining norm, lowest original column among ties
    if (warp == 0) {
      double s = 0.0, mx = -1.0;
      for (int c = k + lane; c < n; c += 32) {
        s += norms2[c];
        mx = fmax(mx, norms2[c]);
      }
      s = warp_sum(s);
      mx = warp_max(mx);
      const double thr = mx - (TIE_REL * mx + TIE_ABS * sqrt(mx * s_y2max));
      int bp = INT_MAX, bc = -1;
      for (int c = k + lane; c < n; c += 32)
        if (norms2[c] >= thr && perm[c] < bp) {
          bp = perm[c];
          bc = c;
        }
      for (int d = 16; d > 0; d >>= 1) {
        const int op = __shfl_xor_sync(0xffffffffu, bp, d), oc = __shfl_xor_sync(0xffffffffu, bc, d);
        if (op < bp) {
          bp = op;
          bc = oc;
        }
      }
      if (lane == 0) {
        s_stop = (s <= s_thresh) || bc < 0;   // bc < 0 only if every norm is NaN
        s_piv = bc;
        if (!s_stop && bc != k) {
          int ti = perm[k]; perm[k] = perm[bc]; perm[bc] = ti;
          double td = norms2[k]; norms2[k] = norms2[bc]; norms2[bc] = td;
          td = ref[k]; ref[k] = ref[bc]; ref[bc] = td;
        }
      }
    }
    __syncthreads();
    if (s_stop) break;
    const int q = perm[k];
    // pivot column after k reflectors, rows k..m-1
    double s2 = 0.0;
    for (int i = k + tid; i < m; i += blockDim.x) {
      T x = Y[(size_t)q * ldY + i];
      for (int l = 0; l < k; ++l) x = msb(x, V[(size_t)l * ldY + i], G[(size_t)l * nmax + q]);
      vbuf[i] = x;
      s2 += abs2(x);
    }
    const double alpha2 = block_sum(s2, s_redd);
    if (tid == 0) {
      const T x0 = vbuf[k];
      const double alpha = sqrt(alpha2);
      if (alpha == 0.0) {
        s_stop = 1;
      } else {
        const double ax0 = sqrt(abs2(x0));
        T phase = from_re<T>(1.0);
        if (ax0 != 0.0) phase = scl(1.0 / ax0, x0);
        const T bt = scl(-alpha, phase);
        beta[k] = bt;
        s_scale = dv(from_re<T>(1.0), x0 - bt);   // 1 / (x0 - beta), one division
        taus[k] = (alpha + ax0) / alpha;
      }
    }
    __syncthreads();
    if (s_stop) break;
    {
      const T d = s_scale;
      for (int i = k + 1 + tid; i < m; i += blockDim.x) {
        const T v = vbuf[i] * d;
        vbuf[i] = v;
        V[(size_t)k * ldY + i] = v;
      }
      if (tid == 0) {
        vbuf[k] = from_re<T>(1.0);
        V[(size_t)k * ldY + k] = from_re<T>(1.0);
      }
    }
    __syncthreads();
    // u_l = v^H V[:, l] (l < k) and raw g_c = v^H Y[:, c] for the remaining columns,
    // four columns per warp: one accumulator per column and lane, then a transposing
    // butterfly that sums the four columns with six additions instead of twenty
    // (an FP64 instruction costs the same with one lane or 32)
    const int nc = n - k - 1, ncol = k + nc;
    for (int gi = warp; 4 * gi < ncol; gi += nwarp) {
      const T* col[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int w = 4 * gi + c;
        col[c] = w >= ncol ? nullptr : w < k ? V + (size_t)w * ldY : Y + (size_t)perm[k + 1 + (w - k)] * ldY;
      }
      T d[4] = {zero<T>(), zero<T>(), zero<T>(), zero<T>()};
      if (col[3] != nullptr) {
        for (int i = k + lane; i < m; i += 32) {
          const T x = vbuf[i];
#pragma unroll
          for (int c = 0; c < 4; ++c) d[c] = madc(d[c], x, col[c][i]);
        }
      } else {
        for (int i = k + lane; i < m; i += 32) {
          const T x = vbuf[i];
#pragma unroll
          for (int c = 0; c < 3; ++c)
            if (col[c] != nullptr) d[c] = madc(d[c], x, col[c][i]);
        }
      }
      // lanes 0-15 keep columns 0, 1 and lanes 16-31 columns 2, 3; then each group of
      // eight lanes keeps one column (lanes 8c .. 8c + 7: column c) and sums it
      const bool hi = lane >= 16;
      T a0 = hi ? d[2] : d[0], a1 = hi ? d[3] : d[1];
      a0 = a0 + shfl_xor(hi ? d[0] : d[2], 16);
      a1 = a1 + shfl_xor(hi ? d[1] : d[3], 16);
      const bool odd = (lane & 8) != 0;
      T t = odd ? a1 : a0;
      t = t + shfl_xor(odd ? a0 : a1, 8);
      t = t + shfl_xor(t, 4);
      t = t + shfl_xor(t, 2);
      t = t + shfl_xor(t, 1);
      const int w = 4 * gi + (lane >> 3);
      if ((lane & 7) == 0 && w < ncol) {
        if (w < k) u[w] = t;
        else G[(size_t)k * nmax + perm[k + 1 + (w - k)]] = t;
      }
    }
    if (a.g_sm)
      for (int l = tid; l <= k; l += blockDim.x) vrow[l] = V[(size_t)l * ldY + k];
    __syncthreads();
    // g_c, row k of R, norm downdate
    const double tau = taus[k];
    for (int pos = k + 1 + tid; pos < n; pos += blockDim.x) {
      const int c = perm[pos];
      T gc = G[(size_t)k * nmax + c];
      for (int l = 0; l < k; ++l) gc = msb(gc, G[(size_t)l * nmax + c], u[l]);
      gc = scl(tau, gc);
      G[(size_t)k * nmax + c] = gc;
      T r = Y[(size_t)c * ldY + k];
      if (a.g_sm)
        for (int l = 0; l <= k; ++l) r = msb(r, vrow[l], G[(size_t)l * nmax + c]);
      else
        for (int l = 0; l <= k; ++l) r = msb(r, V[(size_t)l * ldY + k], G[(size_t)l * nmax + c]);
      Rr[(size_t)k * nmax + c] = r;
      const double nv = norms2[pos] - abs2(r);
      flag[pos] = nv < RECOMPUTE_REL * ref[pos];
      norms2[pos] = nv;
    }
    __syncthreads();
    for (int pos = k + 1 + warp; pos < n; pos += nwarp) {
      if (!flag[pos]) continue;
      const int c = perm[pos];
      double t = 0.0;
      int i = k + 1 + lane;
      for (; i + 96 < m; i += 128) {   // four rows per lane in flight
        T x0 = Y[(size_t)c * ldY + i], x1 = Y[(size_t)c * ldY + i + 32];
        T x2 = Y[(size_t)c * ldY + i + 64], x3 = Y[(size_t)c * ldY + i + 96];
        for (int l = 0; l <= k; ++l) {
          const T gl = G[(size_t)l * nmax + c];
          const T* vl = V + (size_t)l * ldY + i;
          x0 = msb(x0, vl[0], gl);
          x1 = msb(x1, vl[32], gl);
          x2 = msb(x2, vl[64], gl);
          x3 = msb(x3, vl[96], gl);
        }
        t += (abs2(x0) + abs2(x1)) + (abs2(x2) + abs2(x3));
      }
      for (; i < m; i += 32) {
        T x = Y[(size_t)c * ldY + i];
        for (int l = 0; l <= k; ++l) x = msb(x, V[(size_t)l * ldY + i], G[(size_t)l * nmax + c]);
        t += abs2(x);
      }
      t = warp_sum(t);
      if (lane == 0) {
        norms2[pos] = t;
        ref[pos] = t;
      }
    }
    __syncthreads();
    ++k;
  }
  __syncthreads();
  // T = R11^{-1} R12 (back substitution), k x r with ld nmax
  const int r = n - k;
  S* Tw = a.T_ws + (size_t)bi * nn;
  for (int c = tid; c < r; c += blockDim.x) {
    const int oc = perm[k + c];
    for (int i = k - 1; i >= 0; --i) {
      T x = Rr[(size_t)i * nmax + oc];
      for (int l = i + 1; l < k; ++l)
        x = msb(x, Rr[(size_t)i * nmax + perm[l]], id_load<T, S>(Tw[(size_t)c * nmax + l]));
      Tw[(size_t)c * nmax + i] = id_store<T, S>(dv(x, beta[i]));
    }
  }
  for (int c = tid; c < n; c += blockDim.x) a.perm_out[(size_t)bi * nmax + c] = perm[c];
  if (tid == 0) a.k_out[bi] = k;
}

// ------------------------------------------------------------------ ID on a thread-block cluster
// For colour classes too small to fill the GPU: a cluster of Q CTAs works on one
// box, CTA q owning a contiguous slice of the rows of Y (and of V).  Every CTA
// keeps an identical copy of the small state (norms, permutation, G, rows of R)
// and makes the same decisions; the sums over rows (column norms, the pivot
// column's norm, v^H Y, v^H V, re-accumulated norms) are formed per CTA and
// added through distributed shared memory in rank order, so all CTAs see the
// same bits.  Every CTA reaches every cluster barrier the same number of times.
template <typename T, typename S, int NTC>
__global__ void __launch_bounds__(NTC, (sizeof(T) == sizeof(double) && NTC == 256) ? 2 : 1) k_id_cl(IdArgs<T, S> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int Q = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const LevelDev<S>& L = a.L;
  const int nmax = L.nmax, g = L.g, ldY = a.ldY;
  const int rp = (ldY + Q - 1) / Q;                // rows per CTA (upper bound)
  T* vbuf = reinterpret_cast<T*>(smraw);           // rp: owned rows of the reflector
  T* u = vbuf + rp;                                // nmax
  T* beta = u + nmax;                              // nmax
  const int pst = cl_part_stride<NTC>(nmax);
  T* part = beta + nmax;                           // 2 x pst: partial sums, double buffered
  double* norms2 = reinterpret_cast<double*>(part + 2 * pst);
  double* ref = norms2 + nmax;
  double* taus = ref + nmax;
  int* perm = reinterpret_cast<int*>(taus + nmax);
  int* flag = perm + nmax;
  T* Gs = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(smraw) +
                               ((reinterpret_cast<unsigned char*>(flag + nmax) - smraw + 15) & ~size_t(15)));
  T* vrow = Gs + (size_t)nmax * nmax;              // row k of V (a.g_sm)
  __shared__ int Mbox[16], Moff[17], s_nM, s_stop;
  __shared__ double s_thresh, s_y2max;
  __shared__ T s_scale;

  const int box_local = blockIdx.x / Q;
  const int bi = a.base + box_local;
  const int B = a.boxes[bi];
  const size_t nn = (size_t)nmax * nmax;
  const int n = L.n[B];
  const size_t slot = 2 * (size_t)ldY * nmax + 2 * nn * Q;
  T* Yw = a.ws + (size_t)box_local * slot;
  const T* Y = Yw;
  T* V = Yw + (size_t)ldY * nmax;
  T* G = a.g_sm ? Gs : V + (size_t)ldY * nmax + 2 * nn * rank;   // this CTA's copy: G[l * nmax + c]
  T* Rr = V + (size_t)ldY * nmax + 2 * nn * rank + nn;            // Rr[i * nmax + c]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  int pb = 0;                                       // partial-sum buffer in use

  // sum the Q CTAs' partial vectors part[pb][0..len) in rank order into out[]
  auto cluster_sum = [&](int len, T* out) {
    cl.sync();
    for (int e = tid; e < len; e += blockDim.x) {
      T s = zero<T>();
      for (int q0 = 0; q0 < Q; q0 += 8) {
        T v[8];   // eight remote loads issued together, then added in rank order
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q0 + q < Q) v[q] = cl.map_shared_rank(part + pb * pst, q0 + q)[e];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q0 + q < Q) s = s + v[q];
      }
      out[e] = s;
    }
    pb ^= 1;
    __syncthreads();
  };

  if (tid == 0) {
    int cnt = 0, off = 0;
    for (int dy = -2; dy <= 2; ++dy)
      for (int dx = -2; dx <= 2; ++dx) {
        if (max(abs(dx), abs(dy)) != 2) continue;
        const int mb = nbr_box(B, g, dx, dy);
        if (mb < 0) continue;
        Mbox[cnt] = mb;
        Moff[cnt] = off;
        off += L.nact[mb];
        ++cnt;
      }
    Moff[cnt] = off;
    s_nM = cnt;
  }
  __syncthreads();
  const int nM = s_nM, mh = Moff[nM], P = a.P;
  const int m = a.half ? mh + P : 2 * (mh + P);
  const int r0 = min(m, rank * rp), r1 = min(m, r0 + rp);
  const int bx = B % g, by = B / g;
  const double cx = a.geo.x0 - 0.5 * a.geo.hg + (bx + 0.5) * a.Lbox;
  const double cy = a.geo.y0 - 0.5 * a.geo.hg + (by + 0.5) * a.Lbox;
  // owned rows of Y
  const int mr = r1 - r0;
  for (long long e = tid; e < (long long)mr * n; e += blockDim.x) {
    const int i = r0 + (int)(e % mr), j = (int)(e / mr);
    Yw[(size_t)j * ldY + i] = id_entry(a, B, i, j, mh, Mbox, Moff, cx, cy);
  }
  __syncthreads();
  // column norms: partials over owned rows, summed across the cluster
  for (int c = warp; c < n; c += nwarp) {
    double s = 0.0;
    for (int i = r0 + lane; i < r1; i += 32) s += abs2(Y[(size_t)c * ldY + i]);
    s = warp_sum(s);
    if (lane == 0) part[pb * pst + c] = from_re<T>(s);
  }
  cluster_sum(n, u);   // (u used as scratch)
  for (int c = tid; c < n; c += blockDim.x) {
    norms2[c] = re(u[c]);
    ref[c] = norms2[c];
    perm[c] = c;
  }
  __syncthreads();
  if (warp == 0) {
    double s = 0.0, mx = 0.0;
    for (int c = lane; c < n; c += 32) {
      s += norms2[c];
      mx = fmax(mx, norms2[c]);
    }
    s = warp_sum(s);
    mx = warp_max(mx);
    if (lane == 0) {
      s_thresh = a.eps * a.eps * s;
      s_y2max = mx;
    }
  }
  __syncthreads();

  int k = 0;
  const int kmax = min(m, n);
  while (k < kmax) {
    if (warp == 0) {   // stop test and pivot (identical in every CTA)
      double s = 0.0, mx = -1.0;
      for (int c = k + lane; c < n; c += 32) {
        s += norms2[c];
        mx = fmax(mx, norms2[c]);
      }
      s = warp_sum(s);
      mx = warp_max(mx);
      const double thr = mx - (TIE_REL * mx + TIE_ABS * sqrt(mx * s_y2max));
      int bp = INT_MAX, bc = -1;
      for (int c = k + lane; c < n; c += 32)
        if (norms2[c] >= thr && perm[c] < bp) {
          bp = perm[c];
          bc = c;
        }
      for (int d = 16; d > 0; d >>= 1) {
        const int op = __shfl_xor_sync(0xffffffffu, bp, d), oc = __shfl_xor_sync(0xffffffffu, bc, d);
        if (op < bp) {
          bp = op;
          bc = oc;
        }
      }
      if (lane == 0) {
        s_stop = (s <= s_thresh) || bc < 0;
        if (!s_stop && bc != k) {
          int ti = perm[k]; perm[k] = perm[bc]; perm[bc] = ti;
          double td = norms2[k]; norms2[k] = norms2[bc]; norms2[bc] = td;
          td = ref[k]; ref[k] = ref[bc]; ref[bc] = td;
        }
      }
    }
    __syncthreads();
    if (s_stop) break;
    const int q = perm[k];
    // owned rows of the pivot column after k reflectors; partial norm and x0
    double s2 = 0.0;
    for (int i = max(k, r0) + tid; i < r1; i += blockDim.x) {
      T x = Y[(size_t)q * ldY + i];
      for (int l = 0; l < k; ++l) x = msb(x, V[(size_t)l * ldY + i], G[(size_t)l * nmax + q]);
      vbuf[i - r0] = x;
      s2 += abs2(x);
    }
    s2 = warp_sum(s2);
    if (lane == 0) part[pb * pst + 2 + warp] = from_re<T>(s2);
    if (tid == 0) part[pb * pst + 0] = zero<T>();
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < nwarp; ++w) t += re(part[pb * pst + 2 + w]);
      part[pb * pst + 0] = from_re<T>(t);
      part[pb * pst + 1] = (k >= r0 && k < r1) ? vbuf[k - r0] : zero<T>();
    }
    cluster_sum(2, u + nmax - 2);   // u[nmax-2] = alpha^2, u[nmax-1] = x0
    if (tid == 0) {
      const T x0 = u[nmax - 1];
      const double alpha = sqrt(re(u[nmax - 2]));
      if (alpha == 0.0) {
        s_stop = 1;
      } else {
        const double ax0 = sqrt(abs2(x0));
        T phase = from_re<T>(1.0);
        if (ax0 != 0.0) phase = scl(1.0 / ax0, x0);
        const T bt = scl(-alpha, phase);
        beta[k] = bt;
        s_scale = dv(from_re<T>(1.0), x0 - bt);   // 1 / (x0 - beta), one division
        taus[k] = (alpha + ax0) / alpha;
      }
    }
    __syncthreads();
    if (s_stop) break;
    {
      const T d = s_scale;
      for (int i = max(k + 1, r0) + tid; i < r1; i += blockDim.x) {
        const T v = vbuf[i - r0] * d;
        vbuf[i - r0] = v;
        V[(size_t)k * ldY + i] = v;
      }
      if (tid == 0 && k >= r0 && k < r1) {
        vbuf[k - r0] = from_re<T>(1.0);
        V[(size_t)k * ldY + k] = from_re<T>(1.0);
      }
    }
    __syncthreads();
    // partials of u_l = v^H V[:, l] (l < k) and g_c = v^H Y[:, c] over owned rows
    const int nc = n - k - 1;
    const int ib = max(k, r0);
    for (int w = warp; w < k + nc; w += nwarp) {
      const T* col = w < k ? V + (size_t)w * ldY : Y + (size_t)perm[k + 1 + (w - k)] * ldY;
      T d0 = zero<T>(), d1 = zero<T>(), d2 = zero<T>(), d3 = zero<T>();
      int i = ib + lane;
      for (; i + 96 < r1; i += 128) {
        d0 = madc(d0, vbuf[i - r0], col[i]);
        d1 = madc(d1, vbuf[i + 32 - r0], col[i + 32]);
        d2 = madc(d2, vbuf[i + 64 - r0], col[i + 64]);
        d3 = madc(d3, vbuf[i + 96 - r0], col[i + 96]);
      }
      for (; i < r1; i += 32) d0 = madc(d0, vbuf[i - r0], col[i]);
      const T d = warp_sum((d0 + d1) + (d2 + d3));
      if (lane == 0) part[pb * pst + w] = d;
    }
    if (a.g_sm)   // row k of V may belong to another CTA: read through L2
      for (int l = tid; l <= k; l += blockDim.x) vrow[l] = ld_l2(V + (size_t)l * ldY + k);
    cluster_sum(k + nc, u);   // u[0..k): v^H V, u[k..k+nc): raw g for positions k+1..
    // g_c, row k of R, norm downdate (identical in every CTA; own copies of G, Rr)
    const double tau = taus[k];
    int anyf = 0;
    for (int pos = k + 1 + tid; pos < n; pos += blockDim.x) {
      const int c = perm[pos];
      T gc = u[k + (pos - k - 1)];
      for (int l = 0; l < k; ++l) gc = msb(gc, G[(size_t)l * nmax + c], u[l]);
      gc = scl(tau, gc);
      G[(size_t)k * nmax + c] = gc;
      T r = ld_l2(Y + (size_t)c * ldY + k);   // row k may belong to another CTA
      if (a.g_sm)
        for (int l = 0; l <= k; ++l) r = msb(r, vrow[l], G[(size_t)l * nmax + c]);
      else
        for (int l = 0; l <= k; ++l) r = msb(r, ld_l2(V + (size_t)l * ldY + k), G[(size_t)l * nmax + c]);
      Rr[(size_t)k * nmax + c] = r;
      const double nv = norms2[pos] - abs2(r);
      flag[pos] = nv < RECOMPUTE_REL * ref[pos];
      anyf |= flag[pos];
      norms2[pos] = nv;
    }
    // the flags are the same in every CTA of the cluster (same data, same
    // operations), so all of them skip the re-accumulation together
    if (!__syncthreads_or(anyf)) {
      ++k;
      continue;
    }
    // re-accumulation of flagged norms: partials over owned rows
    for (int pos = k + 1 + warp; pos < n; pos += nwarp) {
      double t = 0.0;
      if (flag[pos]) {
        const int c = perm[pos];
        for (int i = max(k + 1, r0) + lane; i < r1; i += 32) {
          T x = Y[(size_t)c * ldY + i];
          for (int l = 0; l <= k; ++l) x = msb(x, V[(size_t)l * ldY + i], G[(size_t)l * nmax + c]);
          t += abs2(x);
        }
        t = warp_sum(t);
      }
      if (lane == 0) part[pb * pst + pos] = from_re<T>(t);
    }
    cluster_sum(n, u);
    for (int pos = k + 1 + tid; pos < n; pos += blockDim.x)
      if (flag[pos]) {
        norms2[pos] = re(u[pos]);
        ref[pos] = norms2[pos];
      }
    __syncthreads();
    ++k;
  }
  cl.sync();   // every CTA is done reading its peers' shared memory
  if (rank != 0) return;
  // T = R11^{-1} R12 (back substitution), k x r with ld nmax
  const int r = n - k;
  S* Tw = a.T_ws + (size_t)bi * nn;
  for (int c = tid; c < r; c += blockDim.x) {
    const int oc = perm[k + c];
    for (int i = k - 1; i >= 0; --i) {
      T x = Rr[(size_t)i * nmax + oc];
      for (int l = i + 1; l < k; ++l)
        x = msb(x, Rr[(size_t)i * nmax + perm[l]], id_load<T, S>(Tw[(size_t)c * nmax + l]));
      Tw[(size_t)c * nmax + i] = id_store<T, S>(dv(x, beta[i]));
    }
  }
  for (int c = tid; c < n; c += blockDim.x) a.perm_out[(size_t)bi * nmax + c] = perm[c];
  if (tid == 0) a.k_out[bi] = k;
}

// ------------------------------------------------------------------ tensor-core helpers

// ------------------------------------------------------------------ digit slices
// A row x_0..x_{r-1} with max |x_l| = m 2^e (m in [0.5, 1)) is written as
// x_l = 2^e sum_{p=0}^{OZ_S-1} d_{p,l} 2^{-7(p+1)}, with signed digits
// |d_0| <= 128 and |d_p| <= 64 (p >= 1), all exact in bf16; the truncation error
// is below 2^(e-57), the rounding of x 2^(56-e) to an integer.
__device__ inline uint16_t bf16_of_small_int(int d) {
  const __nv_bfloat16 h = __float2bfloat16_rn((float)d);
  return __bfloat16_as_ushort(h);
}

__device__ void oz_split_row(const double* __restrict__ src, int stride, int r, int kp, uint16_t* dst, int* eout) {
  double mx = 0.0;
  for (int l = 0; l < r; ++l) mx = fmax(mx, fabs(src[(size_t)l * stride]));
  int e = 0;
  if (mx > 0.0) frexp(mx, &e);
  *eout = e;
  const double scale = ldexp(1.0, 56 - e);
  for (int l = 0; l < kp; l += 2) {
    long long X0 = l < r ? llrint(src[(size_t)l * stride] * scale) : 0;
    long long X1 = l + 1 < r ? llrint(src[(size_t)(l + 1) * stride] * scale) : 0;
    int d0[OZ_S], d1[OZ_S];
#pragma unroll
    for (int p = OZ_S - 1; p >= 1; --p) {
      d0[p] = (int)(((X0 + 64) & 127) - 64);
      X0 = (X0 - d0[p]) >> OZ_BITS;
      d1[p] = (int)(((X1 + 64) & 127) - 64);
      X1 = (X1 - d1[p]) >> OZ_BITS;
    }
    d0[0] = (int)X0;
    d1[0] = (int)X1;
#pragma unroll
    for (int p = 0; p < OZ_S; ++p)
      *reinterpret_cast<uint32_t*>(dst + (size_t)p * kp + l) =
          (uint32_t)bf16_of_small_int(d0[p]) | ((uint32_t)bf16_of_small_int(d1[p]) << 16);
  }
}

// ------------------------------------------------------------------ sparsify + LU (Eqs. 7, 8)
template <typename T> struct ElimArgs {
  LevelDev<T> L;
  const BoxRec<T>* recs;
  const int* cls_idx;       // class index of each record's box (row into perm/T_ws)
  const int* perm_in;
  const T* T_ws;
  int* err;
  int smem_cap;             // scalars of dynamic shared memory available
};

constexpr int PKC = 16;     // rows of a panel product's right operand staged per chunk

// Register-blocked panel product: out(i, j) = init(i, j) + sum_l A_l[i] B(l, j)
// for the rows i < rows of a panel of 16 MA rows and the columns j of the block
// [j0, min(r, j0 + 16 NB)).  arow(l) points at row l of the left operand (16 MA
// scalars in shared memory); B(l, j) is read through bfun in chunks of PKC rows
// staged in Bs (PKC x (16 NB + 1)).  Thread (tx, ty) owns rows tx + 16 a and
// columns j0 + ty + 16 b.  TRI: B is upper triangular (B(l, j) = 0 for l > j).
// Every thread of the block calls it; out() runs after a barrier, so it may
// overwrite what init() reads.
template <typename T, int MA, int NB, bool TRI, typename AR, typename BF, typename IF, typename OF>
__device__ __forceinline__ void panel_gemm(AR arow, int nl, int rows, int j0, int r, T* Bs, BF bfun, IF init,
                                           OF out) {
  constexpr int RB = 16 * NB + 1;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  T acc[MA][NB];
#pragma unroll
  for (int a = 0; a < MA; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int i = tx + 16 * a, j = j0 + ty + 16 * b;
      acc[a][b] = (i < rows && j < r) ? init(i, j) : zero<T>();
    }
  const int jw = min(16 * NB, r - j0);                              // columns in the block
  const int lend = TRI ? min(nl, j0 + jw) : nl;                     // rows of B that can be nonzero
  const int tend = TRI ? min(lend, j0 + ty + 16 * (NB - 1) + 1) : lend;   // this thread's last row
  for (int l0 = 0; l0 < lend; l0 += PKC) {
    __syncthreads();
    for (int e = threadIdx.x; e < PKC * 16 * NB; e += blockDim.x) {
      const int ll = e % PKC, jj = e / PKC, l = l0 + ll, j = j0 + jj;
      Bs[ll * RB + jj] = (l < lend && jj < jw && (!TRI || l <= j)) ? bfun(l, j) : zero<T>();
    }
    __syncthreads();
    const int le = min(PKC, tend - l0);
    for (int ll = 0; ll < le; ++ll) {
      const T* ar = arow(l0 + ll);
      T av[MA], bv[NB];
#pragma unroll
      for (int a = 0; a < MA; ++a) av[a] = ar[tx + 16 * a];
#pragma unroll
      for (int b = 0; b < NB; ++b) bv[b] = Bs[ll * RB + ty + 16 * b];
#pragma unroll
      for (int a = 0; a < MA; ++a)
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[a][b] = mad(acc[a][b], av[a], bv[b]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int a = 0; a < MA; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int i = tx + 16 * a, j = j0 + ty + 16 * b;
      if (i < rows && j < r) out(i, j, acc[a][b]);
    }
}

// Calls f(std::integral_constant<int, NB>) for every 16 NBMAX-column block of
// [0, r), NB = the block's column groups of 16.
template <int NBMAX, typename F> __device__ __forceinline__ void for_col_blocks(int r, F f) {
  for (int j0 = 0; j0 < r; j0 += 16 * NBMAX) {
    const int nb = (min(r - j0, 16 * NBMAX) + 15) / 16;
    switch (nb) {
      case 1: f(j0, std::integral_constant<int, 1>{}); break;
      case 2: if constexpr (NBMAX >= 2) f(j0, std::integral_constant<int, 2>{}); break;
      case 3: if constexpr (NBMAX >= 3) f(j0, std::integral_constant<int, 3>{}); break;
      case 4: if constexpr (NBMAX >= 4) f(j0, std::integral_constant<int, 4>{}); break;
      case 5: if constexpr (NBMAX >= 5) f(j0, std::integral_constant<int, 5>{}); break;
      case 6: if constexpr (NBMAX >= 6) f(j0, std::integral_constant<int, 6>{}); break;
      case 7: if constexpr (NBMAX >= 7) f(j0, std::integral_constant<int, 7>{}); break;
      default: if constexpr (NBMAX >= 8) f(j0, std::integral_constant<int, 8>{}); break;
    }
  }
}

// Complex rows: real and imaginary parts share the row scale (the largest |Re|,
// |Im| of the row) and are split into OZ_S slices each; a row holds the OZ_S
// real slices followed by the OZ_S imaginary slices.
__device__ void oz_split_row(const zd* __restrict__ src, int stride, int r, int kp, uint16_t* dst, int* eout) {
  double mx = 0.0;
  for (int l = 0; l < r; ++l) {
    const zd v = src[(size_t)l * stride];
    mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
  }
  int e = 0;
  if (mx > 0.0) frexp(mx, &e);
  *eout = e;
  const double scale = ldexp(1.0, 56 - e);
  for (int part = 0; part < 2; ++part)
    for (int l = 0; l < kp; l += 2) {
      const zd v0 = l < r ? src[(size_t)l * stride] : zd{0.0, 0.0};
      const zd v1 = l + 1 < r ? src[(size_t)(l + 1) * stride] : zd{0.0, 0.0};
      long long X0 = llrint((part ? v0.y : v0.x) * scale);
      long long X1 = llrint((part ? v1.y : v1.x) * scale);
      int d0[OZ_S], d1[OZ_S];
#pragma unroll
      for (int p = OZ_S - 1; p >= 1; --p) {
        d0[p] = (int)(((X0 + 64) & 127) - 64);
        X0 = (X0 - d0[p]) >> OZ_BITS;
        d1[p] = (int)(((X1 + 64) & 127) - 64);
        X1 = (X1 - d1[p]) >> OZ_BITS;
      }
      d0[0] = (int)X0;
      d1[0] = (int)X1;
#pragma unroll
      for (int p = 0; p < OZ_S; ++p)
        *reinterpret_cast<uint32_t*>(dst + (size_t)(part * OZ_S + p) * kp + l) =
            (uint32_t)bf16_of_small_int(d0[p]) | ((uint32_t)bf16_of_small_int(d1[p]) << 16);
    }
}

// LU with partial pivoting of the r x r matrix LU (ld r) by the whole CTA:
// largest modulus, lowest row on ties; the exchanges go to piv.  Returns false
// (after flagging RSS_ENUMERIC) on a zero pivot; piv then holds no exchange for
// the remaining steps, so kernels that still read it index within 0 .. r-1.
template <typename T> __device__ bool lu_pp_block(T* LU, int r, int* piv, int* err) {
  __shared__ int s_piv, s_zero;
  __shared__ __align__(16) double s_dinv[2];   // 1 / pivot, computed once per step (T = double or zd)
  const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, warp = tid >> 5;
  for (int j = 0; j < r; ++j) {
    if (warp == 0) {
      double mx = -1.0;
      int mi = INT_MAX;
      for (int i = j + lane; i < r; i += 32) {
        const double v = abs2(LU[i + (size_t)j * r]);
        if (v > mx) { mx = v; mi = i; }
      }
      for (int d = 16; d > 0; d >>= 1) {
        const double om = __shfl_xor_sync(0xffffffffu, mx, d);
        const int oi = __shfl_xor_sync(0xffffffffu, mi, d);
        if (om > mx || (om == mx && oi < mi)) { mx = om; mi = oi; }
      }
      if (lane == 0) {
        s_piv = mi;
        s_zero = !(mx > 0.0);
        if (mx > 0.0) *reinterpret_cast<T*>(s_dinv) = dv(from_re<T>(1.0), LU[mi + (size_t)j * r]);
      }
    }
    __syncthreads();
    if (s_zero) {
      if (tid == 0) set_error(err, RSS_ENUMERIC);
      for (int i = j + tid; i < r; i += bs) piv[i] = i;
      __syncthreads();
      return false;
    }
    const int p = s_piv;
    if (p != j)
      for (int col = tid; col < r; col += bs) {
        const T t = LU[j + (size_t)col * r];
        LU[j + (size_t)col * r] = LU[p + (size_t)col * r];
        LU[p + (size_t)col * r] = t;
      }
    if (tid == 0) piv[j] = p;
    __syncthreads();
    const T d = *reinterpret_cast<const T*>(s_dinv);
    for (int i = j + 1 + tid; i < r; i += bs) LU[i + (size_t)j * r] = LU[i + (size_t)j * r] * d;
    __syncthreads();
    const int w = r - j - 1;
    for (int e = tid; e < w * w; e += bs) {
      const int ii = j + 1 + e % w, jj = j + 1 + e / w;
      LU[ii + (size_t)jj * r] = msb(LU[ii + (size_t)jj * r], LU[ii + (size_t)j * r], LU[j + (size_t)jj * r]);
    }
    __syncthreads();
  }
  return true;
}

// ------------------------------------------------------------------ sparsify + LU (Eqs. 7, 8)
// k_elim_lu (one CTA per box): C map, X_SR, X_RR, P X_RR = L U, U^{-1}, L^{-1}
// and L^{-1} P.  k_elim_panels (one CTA per 16-, 32- or 64-row panel of C): X_CR, X_RC and
// E = X_CR U^{-1}, F = L^{-1} P X_RC (kept as F^T), from shared-memory panels.
// Boxes too large for the panel kernel's shared memory get E and F here, row by
// row from global memory.
template <typename T> __global__ void __launch_bounds__(NT, 4) k_elim_lu(ElimArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const LevelDev<T>& L = a.L;
  const BoxRec<T> R = a.recs[blockIdx.x];
  const int nmax = L.nmax, g = L.g, B = R.box, k = R.k, r = R.r, c = R.c;
  const size_t nn = (size_t)nmax * nmax;
  const int* perm = a.perm_in + (size_t)a.cls_idx[blockIdx.x] * nmax;
  const T* Tw = a.T_ws + (size_t)a.cls_idx[blockIdx.x] * nn;
  const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, warp = tid >> 5;
  // on chip: LU (r x r), then one region holding T until X_RR is formed and
  // the inverses while they are built
  int* sperm = reinterpret_cast<int*>(smraw);   // 2 r: exchange order and its inverse
  unsigned char* smT = smraw + ((2 * r * sizeof(int) + 15) & ~size_t(15));
  const bool onchip = (size_t)r * r + (size_t)max(k * r, r * r) <= (size_t)a.smem_cap;
  T* LU = onchip ? reinterpret_cast<T*>(smT) : R.LU;
  T* Ts = onchip ? LU + (size_t)r * r : R.Tm;
  T* Wb = onchip ? Ts : nullptr;
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
  for (int i = tid; i < c; i += bs) {
    int q = 0;
    while (coff[q + 1] <= i) ++q;
    const int s = ord[q], ii = i - coff[q], u = nb[s];
    const int pos = s == 4 ? perm[ii] : L.act[u * nmax + ii];
    R.cmap[i] = (s << 16) | pos;
    R.idxC[i] = L.pts[u * nmax + pos];
  }
  for (int j = tid; j < r; j += bs) R.idxR[j] = L.pts[B * nmax + perm[k + j]];
  for (int e = tid; e < k * r; e += bs) {
    const T t = Tw[(size_t)(e / k) * nmax + e % k];
    R.Tm[e] = t;
    if (onchip) Ts[e] = t;
  }
  __syncthreads();
  const T* Abb = L.blk + ((size_t)B * 25 + 12) * nn;
  // X_SR = A_SR - A_SS T into E's first k rows (the rows of S in C)
  for (int e = tid; e < k * r; e += bs) {
    const int si = e % k, j = e / k;
    T x = Abb[(size_t)perm[k + j] * nmax + perm[si]];
    for (int q = 0; q < k; ++q) x = msb(x, Abb[(size_t)perm[q] * nmax + perm[si]], Ts[q + (size_t)j * k]);
    R.E[si + (size_t)j * c] = x;
  }
  __syncthreads();
  // X_RR = A_RR - A_RS T - T^* X_SR
  for (int e = tid; e < r * r; e += bs) {
    const int ai = e % r, bj = e / r;
    T x = Abb[(size_t)perm[k + bj] * nmax + perm[k + ai]];
    for (int q = 0; q < k; ++q) x = msb(x, Abb[(size_t)perm[q] * nmax + perm[k + ai]], Ts[q + (size_t)bj * k]);
    for (int q = 0; q < k; ++q) x = msbc(x, Ts[q + (size_t)ai * k], R.E[q + (size_t)bj * c]);
    LU[ai + (size_t)bj * r] = x;
  }
  __syncthreads();
  // P X_RR = L U, partial pivoting (largest modulus, lowest row on ties)   (Eq. 8)
  if (!lu_pp_block(LU, r, R.piv, a.err)) return;
  // U^{-1} and L^{-1}, one column per thread (built in shared memory when it
  // fits, then copied out); L^{-1} P is L^{-1} with its columns permuted:
  // P e_j = e_{pos(j)} for pos the inverse of the exchange order sig (P v = v[sig])
  for (int which = 0; which < 2; ++which) {
    T* dst = which == 0 ? R.Ui : R.Li;
    T* W = onchip ? Wb : dst;
    for (int j = tid; j < r; j += bs) {
      T* w = W + (size_t)j * r;
      if (which == 0) {               // U^{-1} e_j
        for (int i = j + 1; i < r; ++i) w[i] = zero<T>();
        for (int i = j; i >= 0; --i) {
          T x = i == j ? from_re<T>(1.0) : zero<T>();
          for (int l = i + 1; l <= j; ++l) x = msb(x, LU[i + (size_t)l * r], w[l]);
          w[i] = dv(x, LU[i + (size_t)i * r]);
        }
      } else {                        // L^{-1} e_j
        for (int i = 0; i < j; ++i) w[i] = zero<T>();
        w[j] = from_re<T>(1.0);
        for (int i = j + 1; i < r; ++i) {
          T x = zero<T>();
          for (int l = j; l < i; ++l) x = msb(x, LU[i + (size_t)l * r], w[l]);
          w[i] = x;
        }
      }
    }
    __syncthreads();
    if (onchip)
      for (int e = tid; e < r * r; e += bs) dst[e] = Wb[e];
    if (which == 1) {
      if (tid == 0) {
        for (int i = 0; i < r; ++i) sperm[i] = i;
        for (int i = 0; i < r; ++i) {
          const int p = R.piv[i], t = sperm[i];
          sperm[i] = sperm[p];
          sperm[p] = t;
        }
        for (int i = 0; i < r; ++i) sperm[r + sperm[i]] = i;
      }
      __syncthreads();
      for (int e = tid; e < r * r; e += bs) {
        const int i = e % r, j = e / r;
        R.LiP[e] = W[i + (size_t)sperm[r + j] * r];
      }
    }
    __syncthreads();
  }
  if (onchip)
    for (int e = tid; e < r * r; e += bs) R.LU[e] = LU[e];
  __syncthreads();
  {
    // W_E = [-T U^{-1}; U^{-1}] and W_F = [-(L^{-1} P T^*)^T; (L^{-1} P)^T], n x r, ld n:
    // E = X_CR U^{-1} = A_CB W_E and F^T = (L^{-1} P X_RC)^T = A_BC^T W_F (Eqs. 7, 8)
    const int n = k + r;
    for (int e = tid; e < n * r; e += bs) {
      const int l = e % n, j = e / n;
      T we, wf;
      if (l < k) {
        we = zero<T>();
        for (int m = 0; m <= j; ++m) we = msb(we, R.Tm[l + (size_t)m * k], R.Ui[m + (size_t)j * r]);
        wf = zero<T>();
        for (int m = 0; m < r; ++m) wf = msb(wf, R.LiP[j + (size_t)m * r], cj(R.Tm[l + (size_t)m * k]));
      } else {
        we = l - k <= j ? R.Ui[(l - k) + (size_t)j * r] : zero<T>();
        wf = R.LiP[j + (size_t)(l - k) * r];
      }
      R.We[e] = we;
      R.Wf[e] = wf;
    }
  }
  if (!R.panels && !R.ozp) {
    // E and F^T row by row from global memory
    for (long long e = tid; e < (long long)c * r; e += bs) {
      const int i = (int)(e % c), j = (int)(e / c);
      const int cm = R.cmap[i], s = cm >> 16, pos = cm & 0xffff, u = nb[s];
      const T* Aub = L.blk + ((size_t)u * 25 + off_index(u, B, g)) * nn;
      const T* Abu = L.blk + ((size_t)B * 25 + off_index(B, u, g)) * nn;
      const int rj = perm[k + j];
      T x = Aub[(size_t)rj * nmax + pos];
      T y = Abu[(size_t)pos * nmax + rj];
      for (int q = 0; q < k; ++q) {
        const T t = R.Tm[q + (size_t)j * k];
        x = msb(x, Aub[(size_t)perm[q] * nmax + pos], t);
        y = msbc(y, t, Abu[(size_t)pos * nmax + perm[q]]);
      }
      R.E[i + (size_t)j * c] = x;
      R.Ft[i + (size_t)j * c] = y;
    }
    __syncthreads();
    for (int i = tid; i < c; i += bs) {
      T* e = R.E + i;
      for (int j = r - 1; j >= 0; --j) {
        T x = zero<T>();
        for (int l = 0; l <= j; ++l) x = mad(x, e[(size_t)l * c], R.Ui[l + (size_t)j * r]);
        e[(size_t)j * c] = x;
      }
      T* f = R.Ft + i;
      for (int j = 0; j < r; ++j) {
        const int p = R.piv[j];
        if (p != j) {
          const T t = f[(size_t)j * c];
          f[(size_t)j * c] = f[(size_t)p * c];
          f[(size_t)p * c] = t;
        }
      }
      for (int j = 1; j < r; ++j) {
        T x = f[(size_t)j * c];
        for (int l = 0; l < j; ++l) x = msb(x, R.LU[j + (size_t)l * r], f[(size_t)l * c]);
        f[(size_t)j * c] = x;
      }
    }
    __syncthreads();
    if (R.Esl != nullptr) {
      const int ns = sizeof(T) == sizeof(double) ? OZ_S : 2 * OZ_S;   // slices per row
      for (int i = tid; i < 2 * c; i += bs) {
        const bool isE = i < c;
        const int row = isE ? i : i - c;
        oz_split_row((isE ? R.E : R.Ft) + row, c, r, R.kp,
                     (isE ? R.Esl : R.Fsl) + (size_t)row * ns * R.kp, (isE ? R.Eexp : R.Fexp) + row);
      }
    }
  }
  // B keeps only its skeleton
  for (int q = tid; q < k; q += bs) L.act[B * nmax + q] = perm[q];
  if (tid == 0) L.nact[B] = k;
}

#include "elim_split.cuh"

// One panel of 16 MA rows of C.  The rows of A(u, B) (columns of B in pivot
// order) sit in shared memory as [column][row]; X_CR overwrites the R columns in
// place, then E = X_CR U^{-1} goes to global memory; the same buffer then takes
// the columns of A(B, u) for X_RC and F^T = (L^{-1} P_R X_RC)^T.  The right
// operands (T, U^{-1}, L^{-1}) are staged from global memory in chunks, so any
// rank fits.
template <typename T, int MA, int NBMAX>
__device__ void elim_panel_body(const ElimArgs<T>& a, const BoxRec<T>& R, unsigned char* smraw, int p0, int rows) {
  constexpr int EPR = 16 * MA;
  const LevelDev<T>& L = a.L;
  const int nmax = L.nmax, g = L.g, B = R.box, k = R.k, r = R.r, c = R.c, n = k + r;
  const size_t nn = (size_t)nmax * nmax;
  const int* perm = a.perm_in + (size_t)a.cls_idx[blockIdx.y] * nmax;
  const int tid = threadIdx.x, bs = blockDim.x;
  T* As = reinterpret_cast<T*>(smraw);                 // n x EPR
  T* Bs = As + (size_t)n * EPR;                        // PKC x (16 NBMAX + 1)
  int* sig = reinterpret_cast<int*>(Bs + PKC * (16 * NBMAX + 1));   // r
  const T* __restrict__ Tm = R.Tm;
  const T* __restrict__ Ui = R.Ui;
  const T* __restrict__ Li = R.Li;
  for (int e = tid; e < rows * n; e += bs) {   // rows of A(u, B), columns of B in pivot order
    const int ii = e % rows, col = e / rows;
    const int cm = R.cmap[p0 + ii], s = cm >> 16, pos = cm & 0xffff;
    const int u = nbr_box(B, g, s % 3 - 1, s / 3 - 1);
    As[col * EPR + ii] = L.blk[((size_t)u * 25 + off_index(u, B, g)) * nn + (size_t)perm[col] * nmax + pos];
  }
  if (tid == 0) {   // P_R v = v[sig]: the row exchanges applied to the identity
    for (int i = 0; i < r; ++i) sig[i] = i;
    for (int i = 0; i < r; ++i) {
      const int p = R.piv[i], t = sig[i];
      sig[i] = sig[p];
      sig[p] = t;
    }
  }
  __syncthreads();
  auto plain = [&](int l) { return As + (size_t)l * EPR; };
  auto rcol = [&](int l) { return As + (size_t)(k + l) * EPR; };
  // X_CR = A_CR - A_CS T, in place
  for_col_blocks<NBMAX>(r, [&](int j0, auto nbc) {
    panel_gemm<T, MA, decltype(nbc)::value, false>(
        plain, k, rows, j0, r, Bs, [&](int q, int j) { return -Tm[q + (size_t)j * k]; },
        [&](int i, int j) { return As[(k + j) * EPR + i]; }, [&](int i, int j, T v) { As[(k + j) * EPR + i] = v; });
  });
  // E = X_CR U^{-1}
  for_col_blocks<NBMAX>(r, [&](int j0, auto nbc) {
    panel_gemm<T, MA, decltype(nbc)::value, true>(
        rcol, r, rows, j0, r, Bs, [&](int l, int j) { return Ui[l + (size_t)j * r]; },
        [&](int, int) { return zero<T>(); }, [&](int i, int j, T v) { R.E[p0 + i + (size_t)j * c] = v; });
  });
  __syncthreads();
  for (int e = tid; e < rows * n; e += bs) {   // columns of A(B, u), rows of B in pivot order
    const int row = e % n, ii = e / n;
    const int cm = R.cmap[p0 + ii], s = cm >> 16, pos = cm & 0xffff;
    const int u = nbr_box(B, g, s % 3 - 1, s / 3 - 1);
    As[row * EPR + ii] = L.blk[((size_t)B * 25 + off_index(B, u, g)) * nn + (size_t)pos * nmax + perm[row]];
  }
  __syncthreads();
  // X_RC^T = A_RC^T - A_SC^T conj(T), in place
  for_col_blocks<NBMAX>(r, [&](int j0, auto nbc) {
    panel_gemm<T, MA, decltype(nbc)::value, false>(
        plain, k, rows, j0, r, Bs, [&](int q, int j) { return -cj(Tm[q + (size_t)j * k]); },
        [&](int i, int j) { return As[(k + j) * EPR + i]; }, [&](int i, int j, T v) { As[(k + j) * EPR + i] = v; });
  });
  // F^T = (P_R X_RC)^T (L_R^{-1})^T: row l of P_R X_RC is row sig[l] of X_RC;
  // (L^{-1})^T is upper triangular
  auto prow = [&](int l) { return As + (size_t)(k + sig[l]) * EPR; };
  for_col_blocks<NBMAX>(r, [&](int j0, auto nbc) {
    panel_gemm<T, MA, decltype(nbc)::value, true>(
        prow, r, rows, j0, r, Bs, [&](int l, int j) { return Li[j + (size_t)l * r]; },
        [&](int, int) { return zero<T>(); }, [&](int i, int j, T v) { R.Ft[p0 + i + (size_t)j * c] = v; });
  });
  __syncthreads();
  if (R.Esl != nullptr) {   // digit slices of this panel's rows of E and F^T
    const int ns = sizeof(T) == sizeof(double) ? OZ_S : 2 * OZ_S;
    for (int e = tid; e < 2 * rows; e += bs) {
      const bool isE = e < rows;
      const int row = p0 + (isE ? e : e - rows);
      oz_split_row((isE ? R.E : R.Ft) + row, c, r, R.kp,
                   (isE ? R.Esl : R.Fsl) + (size_t)row * ns * R.kp, (isE ? R.Eexp : R.Fexp) + row);
    }
  }
}

template <typename T> constexpr int panel_nbmax() { return sizeof(T) == sizeof(double) ? 6 : 4; }

// shared memory of one panel CTA of 16 MA rows for a box with n = k + r points
template <typename T> size_t panel_smem_bytes(int MA, int n, int r) {
  return sizeof(T) * ((size_t)n * 16 * MA + (size_t)PKC * (16 * panel_nbmax<T>() + 1)) + sizeof(int) * (size_t)r;
}

template <typename T, int MA> __global__ void __launch_bounds__(NT, 2) k_elim_panels(ElimArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<T> R = a.recs[blockIdx.y];
  if (!R.panels || R.ozp) return;
  const int p0 = blockIdx.x * 16 * MA;
  if (p0 >= R.c) return;
  elim_panel_body<T, MA, panel_nbmax<T>()>(a, R, smraw, p0, min(16 * MA, R.c - p0));
}


#include "elim_panels.cuh"

// ------------------------------------------------------------------ Schur update A_CC -= E F
template <typename T> __global__ void __launch_bounds__(NT) k_schur(LevelDev<T> L, const BoxRec<T>* recs) {
  constexpr int TM = 64, KC = 16;
  const BoxRec<T> R = recs[blockIdx.y];
  const int c = R.c, r = R.r, nt = (c + TM - 1) / TM;
  if ((int)blockIdx.x >= nt * nt) return;
  const int i0 = (blockIdx.x % nt) * TM, j0 = (blockIdx.x / nt) * TM;
  const int nmax = L.nmax, g = L.g;
  const long long nn = (long long)nmax * nmax;
  __shared__ T Es[KC][TM], Fs[KC][TM];
  __shared__ long long rowb[TM], colb[TM];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  if (tid < TM) {
    const int i = i0 + tid;
    if (i < c) {
      const int cm = R.cmap[i], s = cm >> 16, pos = cm & 0xffff;
      const int u = nbr_box(R.box, g, s % 3 - 1, s / 3 - 1);
      rowb[tid] = (long long)u * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
    }
  } else if (tid < 2 * TM) {
    const int j = j0 + tid - TM;
    if (j < c) {
      const int cm = R.cmap[j], s = cm >> 16, pos = cm & 0xffff;
      colb[tid - TM] = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
    }
  }
  T acc[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int w = 0; w < 4; ++w) acc[q][w] = zero<T>();
  for (int l0 = 0; l0 < r; l0 += KC) {
    __syncthreads();
    for (int e = tid; e < KC * TM; e += NT) {
      const int ii = e % TM, ll = e / TM, l = l0 + ll;
      Es[ll][ii] = (i0 + ii < c && l < r) ? R.E[i0 + ii + (size_t)l * c] : zero<T>();
      Fs[ll][ii] = (j0 + ii < c && l < r) ? R.Ft[j0 + ii + (size_t)l * c] : zero<T>();
    }
    __syncthreads();
#pragma unroll 4
    for (int ll = 0; ll < KC; ++ll) {
      T av[4], bv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { av[q] = Es[ll][tx + 16 * q]; bv[q] = Fs[ll][ty + 16 * q]; }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int w = 0; w < 4; ++w) acc[q][w] = mad(acc[q][w], av[q], bv[w]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int i = i0 + tx + 16 * q, j = j0 + ty + 16 * w;
      if (i < c && j < c) {
        T* p = L.blk + rowb[tx + 16 * q] + colb[ty + 16 * w];
        *p = *p - acc[q][w];
      }
    }
}

// ------------------------------------------------------------------ Schur update on tensor cores
// A_CC -= E F for real factors with E and F^T split into OZ_S digit slices.
// (E F)_ij = 2^(e_i + f_j) sum_u 2^(-7(u+2)) G_u with G_u = sum_{p+q=u} D_p D'_q^T:
// each G_u is a sum of integer products below 2^24, so bf16 MMAs with FP32
// accumulation compute it exactly; groups u <= OZ_S-1 are kept (the rest lie
// below 2^-56 of the row/column scale, the order of an FP64 product's rounding).
// The groups are gathered in one int64 W = sum_u G_u 2^(39-7u) (the last two by
// rounding right shifts, an error below 2^-53 of the scale), so
// (E F)_ij = W 2^(e_i + f_j - 53): one conversion and one scaling per entry.
// 64 x 32 tile per CTA, 8 warps of 16 x 16.  All eight group sums of a warp's
// tile stay in FP32 registers over the whole K: each is an integer below
// 10 2^12 K, exact for K <= 384, so the groups are combined into W once per
// tile (and once per 384 entries of K beyond that) instead of once per chunk.
// Per K step of 16 the B fragments are loaded once, four slices at a time, and
// the A slices that pair with them, for the 36 products p + q <= 7.  K is staged in chunks of
// 32, double-buffered with cp.async.
constexpr int SRK = 32, SRSA = OZ_S * SRK + 8;   // real Schur: K chunk and slice-row stride
constexpr int SR_M = 64, SR_N = 32;              // CTA tile
constexpr int SR_BUF = (SR_M + SR_N) * SRSA;     // one stage of slices (uint16)
constexpr int SR_FLUSH = OZ_KX / SRK;            // chunks between int64 gathers (12 x 32 = 384)

__global__ void __launch_bounds__(NT, 2) k_schur_oz(LevelDev<double> L, const BoxRec<double>* recs, int sym) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<double> R = recs[blockIdx.y];
  const int c = R.c, kp = R.kp, ntr = (c + SR_M - 1) / SR_M, ntc = (c + SR_N - 1) / SR_N;
  if ((int)blockIdx.x >= ntr * ntc) return;
  const int i0 = (blockIdx.x % ntr) * SR_M, j0 = (blockIdx.x / ntr) * SR_N;
  if (sym && j0 + SR_N <= i0) return;   // symmetric A: entries j >= i, stored to both triangles
  const int SA = SRSA;
  uint16_t* stage = reinterpret_cast<uint16_t*>(smraw);   // two stages: A rows then B rows
  __shared__ long long rowb[SR_M], colb[SR_N], coli[SR_M], rowj[SR_N];
  __shared__ int rexp[SR_M], cexp[SR_N];
  const int nmax = L.nmax, g = L.g;
  const long long nn = (long long)nmax * nmax;
  const int tid = threadIdx.x;
  if (tid < SR_M) {
    const int i = i0 + tid;
    if (i < c) {
      const int cm = R.cmap[i], s = cm >> 16, pos = cm & 0xffff;
      const int u = nbr_box(R.box, g, s % 3 - 1, s / 3 - 1);
      rowb[tid] = (long long)u * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
      coli[tid] = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
      rexp[tid] = R.Eexp[i];
    }
  } else if (tid < SR_M + SR_N) {
    const int j = j0 + tid - SR_M;
    if (j < c) {
      const int cm = R.cmap[j], s = cm >> 16, pos = cm & 0xffff;
      colb[tid - SR_M] = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
      rowj[tid - SR_M] = (long long)nbr_box(R.box, g, s % 3 - 1, s / 3 - 1) * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
      cexp[tid - SR_M] = R.Fexp[j];
    }
  }
  const int warp = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
  const int m0 = (warp >> 1) * 16, n0 = (warp & 1) * 16;
  const int a_row = lane & 15, a_k = (lane >> 4) * 8;
  const int b_row = ((lane >> 4) << 3) + (lane & 7), b_k = ((lane >> 3) & 1) * 8;
  // slices of rows i0.. of E and j0.. of F^T, entries kc .. kc + kl of K
  auto load = [&](int buf, int kc) {
    const int kl = min(SRK, kp - kc), cpr = OZ_S * (kl / 8);   // 16-byte chunks per row
    uint16_t* As = stage + buf * SR_BUF;
    for (int e = tid; e < (SR_M + SR_N) * cpr; e += NT) {
      const int row = e / cpr, rem = e % cpr, sl = rem / (kl / 8), ch = rem % (kl / 8);
      const bool isA = row < SR_M;
      const int gi = isA ? i0 + row : j0 + row - SR_M;
      uint16_t* d = As + row * SA + sl * SRK + ch * 8;
      if (gi < c)
        cp_async16(d, (isA ? R.Esl : R.Fsl) + (size_t)gi * OZ_S * kp + (size_t)sl * kp + kc + ch * 8);
      else
        *reinterpret_cast<uint4*>(d) = make_uint4(0, 0, 0, 0);
    }
    cp_async_commit();
  };
  float acc[OZ_S][2][4];
  long long W[2][4];
#pragma unroll
  for (int ni = 0; ni < 2; ++ni)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      W[ni][e] = 0;
#pragma unroll
      for (int u = 0; u < OZ_S; ++u) acc[u][ni][e] = 0.f;
    }
  // W += the sums of the `entries` of K since the last gather; they restart from zero
  auto gather = [&](int entries) {
#pragma unroll
    for (int ni = 0; ni < 2; ++ni)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        W[ni][e] += oz_join_k(entries, [&](int u) { return acc[u][ni][e]; });
#pragma unroll
        for (int u = 0; u < OZ_S; ++u) acc[u][ni][e] = 0.f;
      }
  };
  const int nch = (kp + SRK - 1) / SRK;
  // the tile of A_CC, prefetched into the idle stage while the last chunk is multiplied
  double* Cs = reinterpret_cast<double*>(stage + (nch & 1) * SR_BUF);   // SR_M x SR_N, ld SR_M
  load(0, 0);
  for (int ci = 0; ci < nch; ++ci) {
    if (ci + 1 < nch) {
      load((ci + 1) & 1, (ci + 1) * SRK);
    } else {
      if (ci == 0) __syncthreads();   // rowb and colb
      for (int e = tid; e < SR_M * SR_N; e += NT) {
        const int row = e % SR_M, col = e / SR_M;
        if (i0 + row < c && j0 + col < c) cp_async8(Cs + e, L.blk + rowb[row] + colb[col]);
      }
      cp_async_commit();
    }
    cp_async_wait_group<1>();
    __syncthreads();
    const uint16_t* As = stage + (ci & 1) * SR_BUF;
    const uint16_t* Bs = As + SR_M * SA;
    const int kl = min(SRK, kp - ci * SRK);
    for (int kk = 0; kk < kl; kk += 16) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // slices q = 4h .. 4h + 3 of B, then every A slice p <= 7 - q
        uint32_t bq[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) ldsm_x4(bq[q], Bs + (n0 + b_row) * SA + (4 * h + q) * SRK + kk + b_k);
#pragma unroll
        for (int p = 0; p + 4 * h < OZ_S; ++p) {
          uint32_t af[4];
          ldsm_x4(af, As + (m0 + a_row) * SA + p * SRK + kk + a_k);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (p + 4 * h + q < OZ_S) {
              mma_bf16(acc[p + 4 * h + q][0], af, bq[q]);
              mma_bf16(acc[p + 4 * h + q][1], af, bq[q] + 2);
            }
        }
      }
    }
    if ((ci + 1) % SR_FLUSH == 0 && ci + 1 < nch) gather(SR_FLUSH * SRK);
    __syncthreads();   // the stage read here is refilled by the next iteration's load
  }
  gather(kp - (nch - 1) / SR_FLUSH * (SR_FLUSH * SRK));
  cp_async_wait_group<0>();
  __syncthreads();
#pragma unroll
  for (int ni = 0; ni < 2; ++ni)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int row = m0 + gq + (e >= 2 ? 8 : 0);
      const int col = n0 + ni * 8 + 2 * t4 + (e & 1);
      if (i0 + row < c && j0 + col < c && (!sym || j0 + col >= i0 + row)) {
        const double v = Cs[row + col * SR_M] - oz_ldexp_int(W[ni][e], rexp[row] + cexp[col] - 53);
        L.blk[rowb[row] + colb[col]] = v;
        if (sym && j0 + col > i0 + row) L.blk[rowj[col] + coli[row]] = v;
      }
    }
}

// The same update on the 5th-generation tensor cores (tcgen05): one thread
// issues the slice products into tensor memory.  A CTA of 256 threads owns 128
// rows (of E) x 32 columns (rows of F^T) of A_CC; group sum G_u (u = p + q)
// accumulates in TMEM columns 32u .. 32u + 31 (256 columns, two CTAs per SM) in
// FP32 over the whole K (exact for kp <= OZ_KX, checked by the host); per K step
// of 16 it takes eight products, A slice p against the stacked B slices
// 0 .. 7 - p (N = 32 (8 - p)).  K is staged
// in chunks of 32 in the no-swizzle K-major layout of 8-row x 16-byte core
// matrices: slice p, row m, entries 8g .. 8g + 7 of the chunk at
// p * rows * 64 + ((m / 8) * 4 + g) * 128 + (m % 8) * 16 bytes (LBO 128, SBO 512).
// After the last chunk every thread reads the eight groups of 16 columns of its
// row (warps w and w + 4 share TMEM lanes 32 (w % 4) ..) with
// tcgen05.ld, gathers each entry into one int64 as k_schur_oz does (same integer
// arithmetic, same result) and subtracts it from the entries of A_CC, which it
// loaded while the last products ran.  A barrier wait that runs out (after
// `polls` polls) sets RSS_ETIMEOUT in *err; the CTA then waits, with the much
// longer limit ST_DRAIN_POLLS, for the products it already issued to finish
// (they write its tensor memory), frees its tensor memory and returns.
constexpr int ST_M = 128, ST_N = 32, ST_KC = 32, ST_NT = 256;
constexpr int ST_A = OZ_S * ST_M * ST_KC * 2;   // bytes of one chunk of A slices (64 KB)
constexpr int ST_B = OZ_S * ST_N * ST_KC * 2;   // 16 KB
constexpr uint32_t ST_TMEM_COLS = OZ_S * ST_N;  // 256
constexpr int ST_POLLS = 1 << 22;
constexpr int ST_DRAIN_POLLS = 1 << 26;

__global__ void __launch_bounds__(ST_NT, 2) k_schur_tc(LevelDev<double> L, const BoxRec<double>* recs, int* err,
                                                        int polls, int sym) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t s_tmem;
  __shared__ long long colb[ST_N], rowj[ST_N];
  __shared__ int cexp[ST_N];
  const BoxRec<double> R = recs[blockIdx.y];
  const int c = R.c, kp = R.kp, ntr = (c + ST_M - 1) / ST_M, ntc = (c + ST_N - 1) / ST_N;
  if ((int)blockIdx.x >= ntr * ntc) return;
  const int i0 = (blockIdx.x % ntr) * ST_M, j0 = (blockIdx.x / ntr) * ST_N;
  if (sym && j0 + ST_N <= i0) return;   // (its entries come from the tile across the diagonal)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quarter = warp & 3, half = warp >> 2;   // TMEM lanes 32 quarter .., columns 16 half ..
  unsigned char* As = smraw;
  unsigned char* Bs = smraw + ST_A;
  const int nmax = L.nmax, g = L.g;
  const long long nn = (long long)nmax * nmax;
  const int i = i0 + 32 * quarter + lane;   // this thread's row of the tile (TMEM lane)
  long long rowb = 0, coli = 0;
  int rexp = 0;
  if (i < c) {
    const int cm = R.cmap[i], s = cm >> 16, pos = cm & 0xffff;
    const int u = nbr_box(R.box, g, s % 3 - 1, s / 3 - 1);
    rowb = (long long)u * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
    coli = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
    rexp = R.Eexp[i];
  }
  if (tid < ST_N) {
    const int j = j0 + tid;
    colb[tid] = rowj[tid] = 0;
    cexp[tid] = 0;
    if (j < c) {
      const int cm = R.cmap[j], s = cm >> 16, pos = cm & 0xffff;
      colb[tid] = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
      rowj[tid] = (long long)nbr_box(R.box, g, s % 3 - 1, s / 3 - 1) * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
      cexp[tid] = R.Fexp[j];
    }
  }
  if (tid == 0) mbar_init(&mbar, 1);
  if (warp == 0) tmem_alloc(&s_tmem, ST_TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int nch = (kp + ST_KC - 1) / ST_KC;
  constexpr int CH = ST_N / 2;   // columns of the tile per thread
  double cv[CH];
#pragma unroll
  for (int j = 0; j < CH; ++j) cv[j] = 0.0;
  int ok = 1;
  uint32_t parity = 0;   // phase of the barrier for the chunk in flight
  for (int ci = 0; ci < nch && ok; ++ci) {
    parity = ci & 1;
    const int kc = ci * ST_KC, kl = min(ST_KC, kp - kc), ng = kl / 8;   // 16-byte pieces per slice row
    const int lg = ng == 4 ? 2 : 1;                                        // kl is 16 or 32
    for (int e = tid; e < (ST_M + ST_N) * OZ_S * ng; e += ST_NT) {
      const int row = e >> (3 + lg), rem = e & (OZ_S * ng - 1), p = rem >> lg, gg = rem & (ng - 1);
      const bool isA = row < ST_M;
      const int rr = isA ? row : row - ST_M, gi = (isA ? i0 : j0) + rr;
      unsigned char* d = (isA ? As + p * (ST_M * ST_KC * 2) : Bs + p * (ST_N * ST_KC * 2)) +
                         ((rr / 8) * 4 + gg) * 128 + (rr % 8) * 16;
      if (gi < c)
        cp_async16(d, (isA ? R.Esl : R.Fsl) + (size_t)gi * OZ_S * kp + (size_t)p * kp + kc + gg * 8);
      else
        *reinterpret_cast<uint4*>(d) = make_uint4(0, 0, 0, 0);
    }
    if (ci + 1 == nch && i < c) {   // the entries of A_CC this thread updates, loaded under the last products
#pragma unroll
      for (int j = 0; j < CH; ++j)
        if (j0 + CH * half + j < c) cv[j] = L.blk[rowb + colb[CH * half + j]];
    }
    cp_async_wait_all();
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      // the B slices are stacked along N (slice q = rows 32q .. 32q + 31, SBO 512
      // throughout), so one product of A slice p with slices 0 .. 7 - p written at
      // TMEM column 32p puts A_p B_q^T into the columns of group p + q
      tc_fence_after();
      for (int s = 0; s < kl / 16; ++s) {
        const uint64_t bd = umma_desc(smem_u32(Bs + s * 256), 128, 512);
#pragma unroll
        for (int p = 0; p < OZ_S; ++p) {
          const uint64_t ad = umma_desc(smem_u32(As + p * (ST_M * ST_KC * 2) + s * 256), 128, 512);
          umma_bf16(tmem + ST_N * p, ad, bd, umma_idesc_bf16(ST_M, ST_N * (OZ_S - p)),
                    (ci > 0 || s > 0 || p > 0) ? 1u : 0u);
        }
      }
      umma_commit(&mbar);
    }
    // one warp polls the barrier; the others wait at the block barrier without issuing
    int got = 1;
    if (warp == 0) got = mbar_wait(&mbar, parity, polls) ? 1 : 0;
    ok = __syncthreads_and(got);
  }
  tc_fence_after();
  if (ok) {
    const uint32_t lane_base = tmem + ((uint32_t)(32 * quarter) << 16) + CH * half;
#pragma unroll
    for (int c0 = 0; c0 < CH; c0 += 8) {
      uint32_t gr[OZ_S][8];
#pragma unroll
      for (int u = 0; u < OZ_S; ++u) tmem_ld8(gr[u], lane_base + ST_N * u + c0);
      tmem_ld_wait();
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const long long w = oz_join_k(kp, [&](int u) { return __uint_as_float(gr[u][jj]); });
        const int j = CH * half + c0 + jj;
        if (i < c && j0 + j < c && (!sym || j0 + j >= i)) {
          const double x = cv[c0 + jj] - oz_ldexp_int(w, rexp + cexp[j] - 53);
          L.blk[rowb + colb[j]] = x;
          if (sym && j0 + j > i) L.blk[rowj[j] + coli] = x;
        }
      }
    }
  } else {
    if (tid == 0) set_error(err, RSS_ETIMEOUT);
    if (warp == 0) mbar_wait(&mbar, parity, ST_DRAIN_POLLS);   // products in flight finish before the TMEM is freed
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, ST_TMEM_COLS);
}

// The same update with one CTA per 128-row block of A_CC that walks the
// 32-column tiles of its rows (kp <= 64): the A slices of the block are staged
// once and stay in shared memory, and the group sums alternate between two
// 256-column halves of tensor memory, so the gathering and read-modify-write of
// tile t - 1 run while the products of tile t are in flight.  The B slices of
// tile t + 1 are staged while tile t - 1 is gathered (its products, the last
// reader of that buffer, are done), and the entries of A_CC of a tile are
// loaded one tile ahead.  Every warp polls the products' barrier itself; one
// block barrier ends each step.  Per tile the same slice products, the same
// exact FP32 group sums and the same integer gathering as k_schur_tc: the same
// bits.  A barrier wait that runs out sets RSS_ETIMEOUT; the CTA then drains
// the products it issued (up to two tiles, the long limit), frees its tensor
// memory and returns.
// Symmetric A (sym; E F = X_CR X_RR^{-1} X_RC is symmetric to rounding): only the entries
// j >= i are formed, and stored to A_CC(j, i) too, four entries of a row of the mirror
// block side by side.  Half the products and FP64 arithmetic: Schur phase at Laplace
// 1024^2 34 -> 28 ms, 448^2 (leaf 49) 58.8 -> 56.0 ms a factorization.
constexpr int SRW_KP = 64;                  // largest kp of the row-block form
constexpr uint32_t SRW_TMEM_COLS = 2 * ST_TMEM_COLS;
constexpr int SRW_NT = 512;   // four warps per 32 TMEM lanes, 8 columns of a tile per thread
constexpr int SRW_XB = 32 * 5 * 8;   // bytes of a warp's transposition

__global__ void __launch_bounds__(SRW_NT, 1) k_schur_tc_rows(LevelDev<double> L, const BoxRec<double>* recs, int* err,
                                                             int polls, int sym) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t s_tmem;
  __shared__ long long colb[3][ST_N], rowj[3][ST_N];   // column data of tile t in buffer t % 3
  __shared__ long long coli[ST_M];      // the rows' places as columns
  __shared__ int cexp[3][ST_N];
  const BoxRec<double> R = recs[blockIdx.y];
  const int c = R.c, kp = R.kp, ntr = (c + ST_M - 1) / ST_M;
  if ((int)blockIdx.x >= ntr) return;
  const int i0 = blockIdx.x * ST_M;
  const int tb = sym ? i0 / ST_N : 0, ntc = (c + ST_N - 1) / ST_N - tb;   // first tile, tiles
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quarter = warp & 3, half = warp >> 2;   // TMEM lanes 32 quarter .., columns CH half ..
  const int nch = (kp + ST_KC - 1) / ST_KC;   // 1 or 2
  unsigned char* As = smraw;                   // nch chunks of ST_A
  unsigned char* Bs = smraw + nch * ST_A;      // two buffers of nch chunks of ST_B
  const int nmax = L.nmax, g = L.g;
  const long long nn = (long long)nmax * nmax;
  const int i = i0 + 32 * quarter + lane;
  double* xb = reinterpret_cast<double*>(smraw + nch * (ST_A + 2 * ST_B)) + warp * (SRW_XB / 8);   // 32 x 5 of the warp
  long long rowb = 0;
  int rexp = 0;
  if (i < c) {
    const int cm = R.cmap[i], s = cm >> 16, pos = cm & 0xffff;
    const int u = nbr_box(R.box, g, s % 3 - 1, s / 3 - 1);
    rowb = (long long)u * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
    if (half == 0) coli[32 * quarter + lane] = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
    rexp = R.Eexp[i];
  }
  // stage the B slices of tile t into buffer t & 1 and its column data into buffer t % 3
  auto stage_b = [&](int t) {
    const int j0 = (tb + t) * ST_N;
    unsigned char* Bb = Bs + (t & 1) * nch * ST_B;
    for (int ci = 0; ci < nch; ++ci) {
      const int kc = ci * ST_KC, kl = min(ST_KC, kp - kc), ng = kl / 8, lg = ng == 4 ? 2 : 1;
      for (int e = tid; e < ST_N * OZ_S * ng; e += SRW_NT) {
        const int rr = e >> (3 + lg), rem = e & (OZ_S * ng - 1), p = rem >> lg, gg = rem & (ng - 1);
        unsigned char* d = Bb + ci * ST_B + p * (ST_N * ST_KC * 2) + ((rr / 8) * 4 + gg) * 128 + (rr % 8) * 16;
        if (j0 + rr < c)
          cp_async16(d, R.Fsl + (size_t)(j0 + rr) * OZ_S * kp + (size_t)p * kp + kc + gg * 8);
        else
          *reinterpret_cast<uint4*>(d) = make_uint4(0, 0, 0, 0);
      }
    }
    if (tid < ST_N) {
      const int j = j0 + tid;
      long long cb = 0, rj = 0;
      int ce = 0;
      if (j < c) {
        const int cm = R.cmap[j], s = cm >> 16, pos = cm & 0xffff;
        cb = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
        rj = (long long)nbr_box(R.box, g, s % 3 - 1, s / 3 - 1) * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
        ce = R.Fexp[j];
      }
      colb[t % 3][tid] = cb;
      rowj[t % 3][tid] = rj;
      cexp[t % 3][tid] = ce;
    }
  };
  // A slices of the row block, all chunks
  for (int ci = 0; ci < nch; ++ci) {
    const int kc = ci * ST_KC, kl = min(ST_KC, kp - kc), ng = kl / 8, lg = ng == 4 ? 2 : 1;
    for (int e = tid; e < ST_M * OZ_S * ng; e += SRW_NT) {
      const int rr = e >> (3 + lg), rem = e & (OZ_S * ng - 1), p = rem >> lg, gg = rem & (ng - 1);
      unsigned char* d = As + ci * ST_A + p * (ST_M * ST_KC * 2) + ((rr / 8) * 4 + gg) * 128 + (rr % 8) * 16;
      if (i0 + rr < c)
        cp_async16(d, R.Esl + (size_t)(i0 + rr) * OZ_S * kp + (size_t)p * kp + kc + gg * 8);
      else
        *reinterpret_cast<uint4*>(d) = make_uint4(0, 0, 0, 0);
    }
  }
  stage_b(0);
  if (ntc > 1) stage_b(1);
  if (tid == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
  }
  if (warp == 0) tmem_alloc(&s_tmem, SRW_TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int uwarp = __shfl_sync(0xffffffffu, warp, 0);   // (uniform)
  const uint32_t lead = uwarp == 0 ? elect_one() : 0u;   // issues the products, always the same lane
  constexpr int CH = ST_N / (SRW_NT / 128);
  double cv[CH], cvn[CH];
#pragma unroll
  for (int j = 0; j < CH; ++j) cv[j] = cvn[j] = 0.0;
  int ok = 1, failed_at = -1;
  for (int t = 0; t <= ntc && ok; ++t) {
    if (t == 0) {
      cp_async_wait_all();
      fence_async_smem();
      __syncthreads();   // A slices and the B slices of tiles 0 and 1 staged
    }
    // from tile 1 on, the barrier at the end of the previous step stands here:
    // the B slices of tile t staged, tensor memory half t & 1 drained (tile t - 2)
    if (t < ntc) {
      if (uwarp == 0) {
        tc_fence_after();
        const uint32_t bl = umma_lo(smem_u32(Bs + (t & 1) * nch * ST_B)), al = umma_lo(smem_u32(As));
        const uint32_t dcol = tmem + (uint32_t)(t & 1) * ST_TMEM_COLS;
        for (int ci = 0; ci < nch; ++ci) {
          const int kl = min(ST_KC, kp - ci * ST_KC);
          for (int s = 0; s < kl / 16; ++s)
#pragma unroll
            for (int p = 0; p < OZ_S; ++p)
              umma_bf16_w(dcol + ST_N * p, al + (uint32_t)(ci * (ST_A / 16) + p * (ST_M * ST_KC / 8) + s * 16),
                          bl + (uint32_t)(ci * (ST_B / 16) + s * 16), umma_idesc_bf16(ST_M, ST_N * (OZ_S - p)),
                          (ci > 0 || s > 0 || p > 0) ? 1u : 0u, lead);
        }
        umma_commit_w(&mbar[t & 1], lead);
        __syncwarp();
      }
      // the entries of A_CC of tile t, read while its products run
      const int j0 = (tb + t) * ST_N;
      if (i < c) {
#pragma unroll
        for (int j = 0; j < CH; ++j)
          if (j0 + CH * half + j < c) cvn[j] = L.blk[rowb + colb[t % 3][CH * half + j]];
      }
    }
    if (t >= 1) {   // tile t - 1: wait for its products, gather, update A_CC
      // every warp polls the barrier itself, so the warps that issued no products
      // start gathering while thread 0 is still issuing those of tile t
      const int tp = t - 1, b = tp & 1;
      const int got = __all_sync(0xffffffffu, mbar_wait(&mbar[b], (uint32_t)(tp >> 1) & 1u, polls) ? 1 : 0);
      if (got) {
        // the products of tile t - 1 are done, so its B buffer takes tile t + 1
        // while this tile is gathered
        if (t + 1 < ntc) stage_b(t + 1);
        tc_fence_after();
        const int j0 = (tb + tp) * ST_N, cb3 = tp % 3;
        const uint32_t lane_base = tmem + (uint32_t)b * ST_TMEM_COLS + ((uint32_t)(32 * quarter) << 16) + CH * half;
#pragma unroll
        for (int c0 = 0; c0 < CH; c0 += 8) {
          uint32_t gr[OZ_S][8];
#pragma unroll
          for (int u = 0; u < OZ_S; ++u) tmem_ld8(gr[u], lane_base + ST_N * u + c0);
          tmem_ld_wait();
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const long long w = oz_join([&](int u) { return __uint_as_float(gr[u][jj]); });
            const int j = CH * half + c0 + jj;
            const double x = cv[c0 + jj] - oz_ldexp_int(w, rexp + cexp[cb3][j] - 53);
            if (i < c && j0 + j < c && (!sym || j0 + j >= i)) L.blk[rowb + colb[cb3][j]] = x;
            // across the diagonal: four columns at a time through shared memory, so that
            // a warp stores the four entries of a row of the mirror block side by side
            if (sym) {
              if (jj % 4 == 0) __syncwarp();
              xb[lane * 5 + jj % 4] = x;
              if (jj % 4 == 3) {
                __syncwarp();
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const int ii = 8 * q + (lane >> 2), jm = j - 3 + (lane & 3), im = i0 + 32 * quarter + ii;
                  if (im < c && j0 + jm < c && j0 + jm > im)
                    L.blk[rowj[cb3][jm] + coli[32 * quarter + ii]] = xb[ii * 5 + (lane & 3)];
                }
              }
            }
          }
        }
      }
      cp_async_wait_all();   // the B slices of tile t + 1, for the products issued after this barrier
      fence_async_smem();
      tc_fence_before();
      // column data of tile t - 1 read; tensor memory half (t - 1) & 1 drained
      ok = __syncthreads_and(got);
      if (!ok) {
        failed_at = tp;
        break;
      }
    }
#pragma unroll
    for (int j = 0; j < CH; ++j) cv[j] = cvn[j];
  }
  if (!ok) {
    if (tid == 0) set_error(err, RSS_ETIMEOUT);
    if (warp == 0) {   // products in flight (tiles failed_at and failed_at + 1) finish before the TMEM is freed
      mbar_wait(&mbar[failed_at & 1], (uint32_t)(failed_at >> 1) & 1u, ST_DRAIN_POLLS);
      if (failed_at + 1 < ntc)
        mbar_wait(&mbar[(failed_at + 1) & 1], (uint32_t)((failed_at + 1) >> 1) & 1u, ST_DRAIN_POLLS);
    }
  }
  cp_async_wait_all();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, SRW_TMEM_COLS);
}

#include "schur_z.cuh"

// Complex factors: Re(E F) = Er Fr^T - Ei Fi^T and Im(E F) = Er Fi^T + Ei Fr^T
// (F^T rows split as Fr, Fi), each group sum exact as in the real case; the
// sign of -Ei is flipped on the bf16 fragment bits.  64 x 32 tile per CTA,
// 8 warps of 16 x 16; K (the slices' length kp) in chunks of 32.  Row and
// column scales are fixed per row, so the int64 sums of the chunks add exactly
// (|W| <= kp 2^53).
constexpr int SCK = 32, SCSA = 2 * OZ_S * SCK + 8;

__global__ void __launch_bounds__(NT) k_schur_oz_c(LevelDev<zd> L, const BoxRec<zd>* recs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<zd> R = recs[blockIdx.y];
  const int c = R.c, kp = R.kp;
  const int ntr = (c + 63) / 64, ntc = (c + 31) / 32;
  if ((int)blockIdx.x >= ntr * ntc) return;
  const int i0 = (blockIdx.x % ntr) * 64, j0 = (blockIdx.x / ntr) * 32;
  const int SA = SCSA;                          // row: 8 real then 8 imaginary slices of one chunk
  uint16_t* As = reinterpret_cast<uint16_t*>(smraw);
  uint16_t* Bs = As + 64 * SA;
  __shared__ long long rowb[64], colb[32];
  __shared__ int rexp[64], cexp[32];
  const int nmax = L.nmax, g = L.g;
  const long long nn = (long long)nmax * nmax;
  const int tid = threadIdx.x;
  if (tid < 64) {
    const int i = i0 + tid;
    if (i < c) {
      const int cm = R.cmap[i], s = cm >> 16, pos = cm & 0xffff;
      const int u = nbr_box(R.box, g, s % 3 - 1, s / 3 - 1);
      rowb[tid] = (long long)u * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
      rexp[tid] = R.Eexp[i];
    }
  } else if (tid < 96) {
    const int j = j0 + tid - 64;
    if (j < c) {
      const int cm = R.cmap[j], s = cm >> 16, pos = cm & 0xffff;
      colb[tid - 64] = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
      cexp[tid - 64] = R.Fexp[j];
    }
  }
  const int warp = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
  const int m0 = (warp >> 1) * 16, n0 = (warp & 1) * 16;
  const int a_row = lane & 15, a_k = (lane >> 4) * 8;
  const int b_row = ((lane >> 4) << 3) + (lane & 7), b_k = ((lane >> 3) & 1) * 8;
  long long Wr[2][4], Wi[2][4];
#pragma unroll
  for (int ni = 0; ni < 2; ++ni)
#pragma unroll
    for (int e = 0; e < 4; ++e) { Wr[ni][e] = 0; Wi[ni][e] = 0; }
  for (int kc = 0; kc < kp; kc += SCK) {
    const int kl = min(SCK, kp - kc), cpr = 2 * OZ_S * (kl / 8);   // 16-byte chunks per row
    __syncthreads();
    for (int e = tid; e < 96 * cpr; e += NT) {
      const int row = e / cpr, rem = e % cpr, sl = rem / (kl / 8), ch = rem % (kl / 8);
      const bool isA = row < 64;
      const int rr = isA ? row : row - 64;
      uint16_t* d = (isA ? As : Bs) + rr * SA + sl * SCK + ch * 8;
      const int gi = (isA ? i0 : j0) + rr;
      if (gi < c)
        cp_async16(d, (isA ? R.Esl : R.Fsl) + (size_t)gi * 2 * OZ_S * kp + (size_t)sl * kp + kc + ch * 8);
      else
        *reinterpret_cast<uint4*>(d) = make_uint4(0, 0, 0, 0);
    }
    cp_async_wait_all();
    __syncthreads();
    // groups u and u + 1 together, combined exactly in int32 (|G| < 2^22)
#pragma unroll 1
    for (int u = 0; u < OZ_S; u += 2) {
      float cr0[2][4], ci0[2][4], cr1[2][4], ci1[2][4];
#pragma unroll
      for (int ni = 0; ni < 2; ++ni)
#pragma unroll
        for (int e = 0; e < 4; ++e) cr0[ni][e] = ci0[ni][e] = cr1[ni][e] = ci1[ni][e] = 0.f;
      for (int p = 0; p <= u + 1; ++p) {
        const uint16_t* Ar = As + p * SCK;
        const uint16_t* Ai = As + (OZ_S + p) * SCK;
        for (int kk = 0; kk < kl; kk += 16) {
          uint32_t ar[4], ai[4], ain[4], br[4], bi[4];
          ldsm_x4(ar, Ar + (m0 + a_row) * SA + kk + a_k);
          ldsm_x4(ai, Ai + (m0 + a_row) * SA + kk + a_k);
#pragma unroll
          for (int i = 0; i < 4; ++i) ain[i] = ai[i] ^ 0x80008000u;
          ldsm_x4(br, Bs + (u + 1 - p) * SCK + (n0 + b_row) * SA + kk + b_k);
          ldsm_x4(bi, Bs + (OZ_S + u + 1 - p) * SCK + (n0 + b_row) * SA + kk + b_k);
#pragma unroll
          for (int ni = 0; ni < 2; ++ni) {
            mma_bf16(cr1[ni], ar, br + 2 * ni);
            mma_bf16(cr1[ni], ain, bi + 2 * ni);
            mma_bf16(ci1[ni], ar, bi + 2 * ni);
            mma_bf16(ci1[ni], ai, br + 2 * ni);
          }
          if (p <= u) {
            ldsm_x4(br, Bs + (u - p) * SCK + (n0 + b_row) * SA + kk + b_k);
            ldsm_x4(bi, Bs + (OZ_S + u - p) * SCK + (n0 + b_row) * SA + kk + b_k);
#pragma unroll
            for (int ni = 0; ni < 2; ++ni) {
              mma_bf16(cr0[ni], ar, br + 2 * ni);
              mma_bf16(cr0[ni], ain, bi + 2 * ni);
              mma_bf16(ci0[ni], ar, bi + 2 * ni);
              mma_bf16(ci0[ni], ai, br + 2 * ni);
            }
          }
        }
      }
      const int sh = 32 - OZ_BITS * u;
#pragma unroll
      for (int ni = 0; ni < 2; ++ni)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const long long gr = (long long)(oz_fint(cr0[ni][e]) * 128 + oz_fint(cr1[ni][e]));
          const long long gi = (long long)(oz_fint(ci0[ni][e]) * 128 + oz_fint(ci1[ni][e]));
          if (sh >= 0) {
            Wr[ni][e] += gr << sh;
            Wi[ni][e] += gi << sh;
          } else {
            Wr[ni][e] += (gr + (1LL << (-sh - 1))) >> (-sh);
            Wi[ni][e] += (gi + (1LL << (-sh - 1))) >> (-sh);
          }
        }
    }
  }
#pragma unroll
  for (int ni = 0; ni < 2; ++ni)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int row = m0 + gq + (e >= 2 ? 8 : 0);
      const int col = n0 + ni * 8 + 2 * t4 + (e & 1);
      if (i0 + row < c && j0 + col < c) {
        const int sx = rexp[row] + cexp[col] - 53;
        zd* ptr = L.blk + rowb[row] + colb[col];
        const zd o = *ptr;
        *ptr = zd{o.x - oz_ldexp_int(Wr[ni][e], sx), o.y - oz_ldexp_int(Wi[ni][e], sx)};
      }
    }
}

#include "id_gram.cuh"

// ------------------------------------------------------------------ merge (Section 2.4)
template <typename T> __global__ void __launch_bounds__(NT) k_merge_pts(LevelDev<T> C, LevelDev<T> P) {
  const int Pb = blockIdx.x, gp = P.g, px = Pb % gp, py = Pb / gp;
  __shared__ int ch[4], off[5];
  if (threadIdx.x == 0) {
    int o = 0;
    for (int q = 0; q < 4; ++q) {
      ch[q] = (2 * py + q / 2) * C.g + 2 * px + q % 2;   // SW, SE, NW, NE
      off[q] = o;
      o += C.nact[ch[q]];
    }
    off[4] = o;
    P.n[Pb] = o;
    P.nact[Pb] = o;
  }
  __syncthreads();
  for (int q = 0; q < 4; ++q)
    for (int i = threadIdx.x; i < off[q + 1] - off[q]; i += blockDim.x)
      P.pts[Pb * P.nmax + off[q] + i] = C.pts[ch[q] * C.nmax + C.act[ch[q] * C.nmax + i]];
  for (int i = threadIdx.x; i < off[4]; i += blockDim.x) P.act[Pb * P.nmax + i] = i;
}

template <typename T>
__global__ void __launch_bounds__(NT) k_merge_blk(LevelDev<T> C, LevelDev<T> P, const int2* __restrict__ ixy,
                                                  const T* __restrict__ tab, KParams kp, int side) {
  // dynamic: the source (child slot << 16 | position in the child) and the grid
  // coordinates of every row and every column of the parent block
  extern __shared__ __align__(16) int msm[];
  const int u = blockIdx.x / 25, o = blockIdx.x % 25;
  const int v = nbr_box(u, P.g, o % 5 - 2, o / 5 - 2);
  if (v < 0) return;
  __shared__ int cu[4], cv[4], ou[5], ov[5];
  __shared__ long long pbase[16];   // child pair (qa, qb): start of its stored block, or -1 (never stored)
  if (threadIdx.x == 0) {
    int a = 0, b = 0;
    for (int q = 0; q < 4; ++q) {
      cu[q] = (2 * (u / P.g) + q / 2) * C.g + 2 * (u % P.g) + q % 2;
      cv[q] = (2 * (v / P.g) + q / 2) * C.g + 2 * (v % P.g) + q % 2;
      ou[q] = a; a += C.nact[cu[q]];
      ov[q] = b; b += C.nact[cv[q]];
    }
    ou[4] = a; ov[4] = b;
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    const int a = cu[threadIdx.x >> 2], b = cv[threadIdx.x & 3];
    pbase[threadIdx.x] = cheb(a, b, C.g) <= 2 ? ((long long)a * 25 + off_index(a, b, C.g)) * C.nmax * C.nmax : -1;
  }
  const int nr = ou[4], ncl = ov[4];
  int* rsrc = msm;
  int* csrc = msm + P.nmax;
  int2* rxy = reinterpret_cast<int2*>(msm + 2 * P.nmax);
  int2* cxy = rxy + P.nmax;
  for (int ip = threadIdx.x; ip < nr; ip += blockDim.x) {
    int q = 0;
    while (ou[q + 1] <= ip) ++q;
    const int pos = C.act[cu[q] * C.nmax + ip - ou[q]];
    rsrc[ip] = (q << 16) | pos;
    rxy[ip] = ixy[C.pts[cu[q] * C.nmax + pos]];
  }
  for (int jp = threadIdx.x; jp < ncl; jp += blockDim.x) {
    int q = 0;
    while (ov[q + 1] <= jp) ++q;
    const int pos = C.act[cv[q] * C.nmax + jp - ov[q]];
    csrc[jp] = (q << 16) | pos;
    cxy[jp] = ixy[C.pts[cv[q] * C.nmax + pos]];
  }
  __syncthreads();
  T* A = P.blk + ((size_t)u * 25 + o) * P.nmax * P.nmax;
  // the 4 x 4 child pairs in one pass over the parent block, rows fastest; entry
  // e = ip + jp nr stepped by the block size without a division per entry
  if (nr == 0) return;
  const int di = (int)blockDim.x % nr, dj = (int)blockDim.x / nr;
  int ip = (int)threadIdx.x % nr, jp = (int)threadIdx.x / nr;
  for (; jp < ncl; ip += di, jp += dj) {
    if (ip >= nr) {
      ip -= nr;
      ++jp;
      if (jp >= ncl) break;
    }
    const int rs = rsrc[ip], cs = csrc[jp];
    const long long base = pbase[((rs >> 16) << 2) | (cs >> 16)];
    T val;
    if (base >= 0)   // a pair the child level stored (and may have modified)
      val = C.blk[base + (long long)(cs & 0xffff) * C.nmax + (rs & 0xffff)];
    else             // never modified: kernel evaluation (Theorem 1)
      val = aval_tab<T>(kp, tab, side, rxy[ip], cxy[jp]);
    A[(size_t)jp * P.nmax + ip] = val;
  }
}

// Child level kept for the merge only: its blocks restricted to the active
// points (the merge reads nothing else), so the full blocks can be freed
// before the parent level is allocated.  out: nbox x 25 x kmax x kmax.
template <typename T>
__global__ void __launch_bounds__(NT) k_compact_blk(LevelDev<T> C, T* __restrict__ out, int* __restrict__ pts_out,
                                                    int kmax) {
  const int u = blockIdx.x / 25, o = blockIdx.x % 25;
  const int v = nbr_box(u, C.g, o % 5 - 2, o / 5 - 2);
  const int nu = C.nact[u];
  if (o == 0)
    for (int i = threadIdx.x; i < nu; i += blockDim.x) pts_out[(size_t)u * kmax + i] = C.pts[u * C.nmax + C.act[u * C.nmax + i]];
  if (v < 0) return;
  const int nv = C.nact[v];
  const T* S = C.blk + ((size_t)u * 25 + o) * C.nmax * C.nmax;
  T* D = out + ((size_t)u * 25 + o) * kmax * kmax;
  const int* au = C.act + u * C.nmax;
  const int* av = C.act + v * C.nmax;
  for (int e = threadIdx.x; e < nu * nv; e += blockDim.x) {
    const int i = e % nu, j = e / nu;
    D[(size_t)j * kmax + i] = S[(size_t)av[j] * C.nmax + au[i]];
  }
}

// Grid coordinates of every tree index (box-major, row-major inside a leaf box)
// and the grid index iy * side + ix of every user point.
__global__ void k_grid_coords(int2* ixy, int32_t* u2g, const int32_t* u2t, long long n, int gL, int ls,
                              int side) {
  const int leaf = ls * ls;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(t / leaf), l = (int)(t % leaf);
    ixy[t] = make_int2((b % gL) * ls + l % ls, (b / gL) * ls + l / ls);
  }
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long t = u2t[i];
    const int b = (int)(t / leaf), l = (int)(t % leaf);
    u2g[i] = ((b / gL) * ls + l / ls) * side + (b % gL) * ls + l % ls;
  }
}

// Leaf level: box b holds tree indices b * leaf + i, all active.
__global__ void k_leaf_init(int* pts, int* act, int* n, int* nact, int nbox, int leaf) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)nbox * leaf;
       e += (long long)gridDim.x * blockDim.x) {
    pts[e] = (int)e;
    act[e] = (int)(e % leaf);
    if (e % leaf == 0) n[e / leaf] = nact[e / leaf] = leaf;
  }
}

__global__ void k_iota_rows(int* act, int nbox, int kmax) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)nbox * kmax;
       e += (long long)gridDim.x * blockDim.x)
    act[e] = (int)(e % kmax);
}

// ------------------------------------------------------------------ dense top
template <typename T>
__global__ void __launch_bounds__(NT) k_top_assemble(LevelDev<T> L, T* D, int ntop, int* top_idx, int4 offs_lo,
                                                     int offs_hi) {
  const int offs[5] = {offs_lo.x, offs_lo.y, offs_lo.z, offs_lo.w, offs_hi};
  const int u = blockIdx.x / L.nbox, v = blockIdx.x % L.nbox;
  const int nu = L.n[u], nv = L.n[v];
  const T* A = L.blk + ((size_t)u * 25 + off_index(u, v, L.g)) * L.nmax * L.nmax;
  for (int e = threadIdx.x; e < nu * nv; e += blockDim.x) {
    const int i = e % nu, j = e / nu;
    D[(size_t)(offs[v] + j) * ntop + offs[u] + i] = A[(size_t)j * L.nmax + i];
  }
  if (v == 0)
    for (int i = threadIdx.x; i < nu; i += blockDim.x) top_idx[offs[u] + i] = L.pts[u * L.nmax + i];
}

#include "top_inv.cuh"

// ------------------------------------------------------------------ host helpers
template <typename T> struct HostLevel {
  LevelDev<T> d{};
  std::vector<int32_t> n, nact;
};

// Level memory is stream-ordered: freeing it needs no device synchronisation.
template <typename T> void free_level(HostLevel<T>& L, cudaStream_t st) {
  pool_free(L.d.pts, st); pool_free(L.d.n, st); pool_free(L.d.act, st); pool_free(L.d.nact, st);
  pool_free(L.d.blk, st);
  L.d = LevelDev<T>{};
}

template <typename T>
rss_status alloc_level(HostLevel<T>& L, int g, int nmax, size_t& transient, cudaStream_t st) {
  L.d = LevelDev<T>{};
  L.d.g = g;
  L.d.nbox = g * g;
  L.d.nmax = nmax;
  const size_t nb = (size_t)g * g;
  auto get = [&](auto** p, size_t bytes) { return pool_malloc(reinterpret_cast<void**>(p), bytes, st); };
  const size_t bytes = sizeof(T) * nb * 25 * (size_t)nmax * nmax;
  if (get(&L.d.pts, sizeof(int) * nb * nmax) != cudaSuccess || get(&L.d.n, sizeof(int) * nb) != cudaSuccess ||
      get(&L.d.act, sizeof(int) * nb * nmax) != cudaSuccess || get(&L.d.nact, sizeof(int) * nb) != cudaSuccess ||
      get(&L.d.blk, bytes) != cudaSuccess) {
    free_level(L, st);
    rss_set_error("rss_factor: out of device memory for the stencil blocks of the " + std::to_string(g) + " x " +
                  std::to_string(g) + " level (" + std::to_string(bytes >> 20) + " MiB, " + std::to_string(nmax) +
                  " points per box)");
    return RSS_ENOMEM;
  }
  transient += bytes;
  return RSS_OK;
}

// Frees the level it watches when the factorization returns early.
template <typename T> struct LevelGuard {
  HostLevel<T>& L;
  cudaStream_t st;
  ~LevelGuard() { free_level(L, st); }
};

// Device time of a phase: events recorded on the factor's stream around it.
struct Ev {
  cudaEvent_t a = nullptr, b = nullptr;
  Ev() { cudaEventCreate(&a); cudaEventCreate(&b); }
  ~Ev() { cudaEventDestroy(a); cudaEventDestroy(b); }
  void start(cudaStream_t st) { cudaEventRecord(a, st); }
  void stop(cudaStream_t st) { cudaEventRecord(b, st); }
  double ms() {   // call after the stream has been synchronised
    float t = 0.f;
    cudaEventElapsedTime(&t, a, b);
    return t;
  }
};

// Grow-only device buffer (freed with the factorization's host frame), in the
// order of the factor's stream: the old buffer is released after the launches
// already queued that read it.
struct GrowBuf {
  cudaStream_t st;
  void* p = nullptr;
  size_t cap = 0;
  explicit GrowBuf(cudaStream_t s) : st(s) {}
  bool ensure(size_t bytes) {
    if (bytes <= cap) return true;
    pool_free(p, st);
    p = nullptr;
    cap = 0;
    if (pool_malloc(&p, bytes, st) != cudaSuccess) return false;
    cap = bytes;
    return true;
  }
  ~GrowBuf() { pool_free(p, st); }
};

struct Timer {
  std::chrono::steady_clock::time_point t0 = std::chrono::steady_clock::now();
  double ms() const {
    return std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  }
};

}  // namespace

template <typename T>
rss_status factor_impl(const rss_tree* tree, const rss_params* prm, cudaStream_t st, rss_factorization* f) {
  Timer total;
  f->n = tree->n;
  f->side = tree->side;
  f->leaf = tree->leaf;
  f->gL = tree->gL;
  f->geo = tree->geo;
  f->tree_to_user = tree->tree_to_user;
  const int P = f->params.proxy_n;
  const double ratio = f->params.proxy_radius_over_side;
  const double extent = tree->side * tree->geo.hg;
  const int64_t N = tree->n;

  f->arena.st = st;
  f->d_user_to_tree = static_cast<int32_t*>(f->arena.get(sizeof(int32_t) * N));
  if (!f->d_user_to_tree) { rss_set_error("rss_factor: device arena allocation failed"); return RSS_ENOMEM; }
  RSS_CUDA(cudaMemcpyAsync(f->d_user_to_tree, tree->user_to_tree.data(), sizeof(int32_t) * N,
                           cudaMemcpyHostToDevice, st));
  int2* d_ixy = static_cast<int2*>(f->arena.get(sizeof(int2) * N));
  int* d_err = static_cast<int*>(f->arena.get(sizeof(int)));
  f->d_user_to_grid = static_cast<int32_t*>(f->arena.get(sizeof(int32_t) * N));
  if (!d_ixy || !d_err || !f->d_user_to_grid) {
    rss_set_error("rss_factor: device arena allocation failed");
    return RSS_ENOMEM;
  }
  RSS_CUDA(cudaMemsetAsync(d_err, 0, sizeof(int), st));
  k_grid_coords<<<152 * 8, NT, 0, st>>>(d_ixy, f->d_user_to_grid, f->d_user_to_tree, N, tree->gL, tree->ls,
                                        tree->side);
  RSS_LAUNCHED();
  f->launches += 1;
  if (prm->kind == RSS_HELMHOLTZ_LS) {   // w = kappa sqrt(b) per grid point (Eq. 19)
    f->d_w = static_cast<double*>(f->arena.get(sizeof(double) * N));
    if (!f->d_w) { rss_set_error("rss_factor: device arena allocation failed"); return RSS_ENOMEM; }
    k_ls_weights<<<cdiv(N, NT), NT, 0, st>>>(f->d_w, tree->side, f->geo, f->kp.kappa, f->params.bump_cx,
                                             f->params.bump_cy, f->params.bump_a);
    RSS_LAUNCHED();
    f->kp.w = f->d_w;
    f->launches += 1;
  }
  // kernel values by displacement, for the leaf blocks and the never-modified far blocks
  const int side = tree->side;
  T* d_tab = nullptr;
  RSS_CUDA(pool_malloc(reinterpret_cast<void**>(&d_tab), sizeof(T) * (size_t)(2 * side - 1) * (2 * side - 1), st));
  struct TabFree {
    T* p;
    cudaStream_t st;
    ~TabFree() { pool_free(p, st); }
  } tab_free{d_tab, st};
  Ev span;
  span.start(st);
  k_ktab<T><<<152 * 8, NT, 0, st>>>(d_tab, side, f->kp, f->geo);
  RSS_LAUNCHED();
  f->launches += 1;

  // workspaces reused across colour classes and levels
  GrowBuf gb_cls(st), gb_k(st), gb_perm(st), gb_clsidx(st), gb_Tws(st), gb_Y(st), gb_oz(st), gb_w(st), gb_inv(st);
  // leaf level
  size_t transient = 0;
  HostLevel<T> cur;
  LevelGuard<T> cur_guard{cur, st};
  int g = tree->gL;
  {
    rss_status s = alloc_level(cur, g, tree->leaf, transient, st);
    if (s != RSS_OK) return s;
    const int nbox = g * g, leaf = tree->leaf;
    std::vector<int> hn(nbox, leaf);
    k_leaf_init<<<152 * 8, NT, 0, st>>>(cur.d.pts, cur.d.act, cur.d.n, cur.d.nact, nbox, leaf);
    RSS_LAUNCHED();
    f->launches += 1;
    cur.n = hn;
    cur.nact = hn;
    Timer tg;
    Ev ev;
    ev.start(st);
    k_gen_blocks<T><<<nbox * 25, NT, 0, st>>>(cur.d, d_ixy, d_tab, f->kp, side);
    RSS_LAUNCHED();
    ev.stop(st);
    RSS_CUDA(cudaStreamSynchronize(st));
    f->t_gen += tg.ms();
    f->g_gen += ev.ms();
    f->launches += 1;
  }

  // A real symmetric kernel (Laplace, real diagonal) keeps A symmetric through the
  // eliminations, so the conjugate half of the proxy stack repeats the first half
  // and the ID of [A_MB; K_PB] alone is the same ID.
  const int half = (prm->id_rows == 0 && prm->kind == RSS_LAPLACE && prm->diag_im == 0.0) ? 1 : 0;
  // poll limits of the Schur update's waits on tcgen05 and of the ID's and the panels'
  const int polls = wait_limit(prm->wait_polls, ST_POLLS);
  const int tc_polls = prm->schur_path == 0 ? polls : ST_POLLS;
  // status of the kernels so far (waits for them)
  auto device_status = [&]() -> rss_status {
    int herr = 0;
    RSS_CUDA(cudaMemcpy(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (herr == RSS_ETIMEOUT) {
      rss_set_error("rss_factor: a tensor-core barrier wait of the ID, the panels or the Schur update ran out");
      return RSS_ETIMEOUT;
    }
    if (herr) {
      rss_set_error("rss_factor: zero pivot in the LU of a redundant block");
      return RSS_ENUMERIC;
    }
    return RSS_OK;
  };
  // A complex symmetric kernel (Helmholtz): the ID of the real stack
  // [Re X; Im X], X = [A_MB; K_PB], which is the ID of the full stack (T real).
  const bool split = std::is_same<T, zd>::value && prm->id_rows == 0 &&
                     (prm->kind == RSS_HELMHOLTZ || prm->kind == RSS_HELMHOLTZ_LS);
  while (g >= 4) {
    const int nbox = g * g, nmax = cur.d.nmax;
    const size_t nn = (size_t)nmax * nmax;
    const double Lbox = extent / g;
    LevelInfo info;
    info.side = g;
    info.n = cur.n;
    info.k = cur.n;
    // colour classes
    std::vector<int> cls;
    std::vector<int> coff(10, 0);
    for (int col = 0; col < 9; ++col) {
      coff[col] = (int)cls.size();
      for (int by = col / 3; by < g; by += 3)
        for (int bx = col % 3; bx < g; bx += 3) cls.push_back(by * g + bx);
    }
    coff[9] = (int)cls.size();
    if (prm->class_order != 0) {   // a seeded permutation of every class (Fisher-Yates, 64-bit LCG)
      uint64_t st64 = (uint64_t)(uint32_t)prm->class_order * 0x9E3779B97F4A7C15ull + (uint64_t)g;
      for (int col = 0; col < 9; ++col)
        for (int i = coff[col + 1] - 1; i > coff[col]; --i) {
          st64 = st64 * 6364136223846793005ull + 1442695040888963407ull;
          const int j = coff[col] + (int)((st64 >> 33) % (uint64_t)(i - coff[col] + 1));
          std::swap(cls[i], cls[j]);
        }
    }
    int maxcls = 0;
    for (int col = 0; col < 9; ++col) maxcls = std::max(maxcls, coff[col + 1] - coff[col]);
    // proxy rows from one table per level where the boxes' points outnumber the
    // table's places (the fine levels); the coarse levels evaluate them per box
    const int lsz = side / g;
    T* d_ptab = nullptr;
    if ((long long)nbox * nmax >= 2LL * lsz * lsz) {
      const size_t pb = sizeof(T) * (size_t)P * lsz * lsz;
      RSS_CUDA(pool_malloc(reinterpret_cast<void**>(&d_ptab), pb, st));
      f->peak_transient = std::max(f->peak_transient, transient + pb);
      Ev evp;
      evp.start(st);
      k_proxy_tab<T><<<std::min<long long>(cdiv((long long)P * lsz * lsz, NT), 152LL * 8), NT, 0, st>>>(
          d_ptab, lsz, P, ratio * Lbox, f->geo.hg, f->kp);
      RSS_LAUNCHED();
      evp.stop(st);
      RSS_CUDA(cudaStreamSynchronize(st));
      f->g_id += evp.ms();
      info.g_id += evp.ms();
      f->launches += 1;
    }
    struct PtabFree {
      T* p;
      cudaStream_t st;
      ~PtabFree() { pool_free(p, st); }
    } ptab_free{d_ptab, st};
    if (!gb_cls.ensure(sizeof(int) * cls.size()) || !gb_k.ensure(sizeof(int) * maxcls) ||
        !gb_perm.ensure(sizeof(int) * (size_t)maxcls * nmax) || !gb_clsidx.ensure(sizeof(int) * maxcls) ||
        !gb_Tws.ensure(sizeof(T) * (size_t)maxcls * nn)) {
      rss_set_error("rss_factor: device workspace allocation failed");
      return RSS_ENOMEM;
    }
    int* d_cls = static_cast<int*>(gb_cls.p);
    int* d_k = static_cast<int*>(gb_k.p);
    int* d_perm = static_cast<int*>(gb_perm.p);
    int* d_clsidx = static_cast<int*>(gb_clsidx.p);
    T* d_Tws = static_cast<T*>(gb_Tws.p);
    RSS_CUDA(cudaMemcpyAsync(d_cls, cls.data(), sizeof(int) * cls.size(), cudaMemcpyHostToDevice, st));
    std::vector<int> hk(maxcls);
    std::vector<std::pair<int, std::unique_ptr<Ev>>> evs;   // phase (0 id, 1 elim, 2 schur), events

    // launch segments: the nine colour classes, or (the plain per-box form, kept
    // to measure what batching gains) one box per launch in the same order
    std::vector<int> segs;
    if (prm->per_box) {
      for (int i = 0; i <= (int)cls.size(); ++i) segs.push_back(i);
    } else {
      segs = coff;
    }
    for (size_t sgi = 0; sgi + 1 < segs.size(); ++sgi) {
      const int seg0 = segs[sgi];
      const int nb = segs[sgi + 1] - seg0;
      if (nb == 0) continue;
      const int* boxes = cls.data() + seg0;
      // rows of Y per box, from the host copy of the active counts
      int mmax = 0;
      std::vector<int> mrows(nb);
      for (int q = 0; q < nb; ++q) {
        const int B = boxes[q], bx = B % g, by = B / g;
        int mh = 0;
        for (int dy = -2; dy <= 2; ++dy)
          for (int dx = -2; dx <= 2; ++dx) {
            if (std::max(std::abs(dx), std::abs(dy)) != 2) continue;
            const int x = bx + dx, y = by + dy;
            if (x < 0 || y < 0 || x >= g || y >= g) continue;
            mh += cur.nact[y * g + x];
          }
        mrows[q] = half ? mh + P : 2 * (mh + P);
        mmax = std::max(mmax, mrows[q]);
      }
      const int ldY = (mmax + 1) & ~1;
      // cluster of Q CTAs per box when the class is too small to fill the GPU
      int Q = 1;
      if (prm->id_cluster >= 0) {
        const int qcap = prm->id_cluster > 0 ? std::min(prm->id_cluster, CL_QMAX) : CL_QDEF;
        while (Q < qcap && (long long)nb * Q * 2 <= 2 * 152) Q *= 2;
        Q = std::min(Q, qcap);
      }
      Timer tid_;
      evs.emplace_back(0, std::make_unique<Ev>());
      evs.back().second->start(st);
      // TC: arithmetic of the ID (double for the complex symmetric real stack)
      auto run_id = [&](auto tag) -> rss_status {
        using TC = decltype(tag);
        const size_t slot = (2 * (size_t)ldY * nmax + 2 * nn * Q) * sizeof(TC);
        const size_t ybudget = size_t(2) << 30;
        const int cap = (int)std::max<size_t>(1, std::min<size_t>(nb, ybudget / slot));
        const int nchunks = (nb + cap - 1) / cap;
        const int chunk = (nb + nchunks - 1) / nchunks;   // balanced chunks
        if (!gb_Y.ensure(slot * chunk)) {
          rss_set_error("rss_factor: device workspace allocation failed");
          return RSS_ENOMEM;
        }
        TC* d_Y = static_cast<TC*>(gb_Y.p);
        size_t smem_id =
            sizeof(TC) * ((size_t)ldY + 2 * nmax) + (size_t)nmax * (3 * sizeof(double) + 2 * sizeof(int));
        // 512 threads per CTA when every CTA of the class gets an SM of its own
        const int ntc = (sizeof(TC) == sizeof(double) && (long long)nb * Q <= 152) ? 512 : 256;
        const int pst = ntc == 512 ? cl_part_stride<512>(nmax) : cl_part_stride<256>(nmax);
        size_t smem_cl = sizeof(TC) * ((size_t)(ldY + Q - 1) / Q + 2 * (size_t)nmax + 2 * (size_t)pst) +
                         (size_t)nmax * (3 * sizeof(double) + 2 * sizeof(int));
        // G and row k of V on chip when they fit
        const size_t gsm = 16 + sizeof(TC) * ((size_t)nmax * nmax + nmax);
        const int g_sm = (Q > 1 ? smem_cl : smem_id) + gsm <= 200 * 1024 ? 1 : 0;
        if (g_sm) {
          smem_id += gsm;
          smem_cl += gsm;
        }
        if (smem_id > 220 * 1024) {
          rss_set_error("rss_factor: proxy stack of a box too tall for the on-chip reflector buffer");
          return RSS_EINVAL;
        }
        RSS_CUDA(allow_smem(k_id<TC, T>));
        auto kcl = k_id_cl<TC, T, 256>;
        if constexpr (sizeof(TC) == sizeof(double))
          if (ntc == 512) kcl = k_id_cl<TC, T, 512>;
        if (Q > 1) {
          RSS_CUDA(allow_smem(kcl));
          if (Q > 8) RSS_CUDA(cudaFuncSetAttribute(kcl, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        }
        f->peak_transient = std::max(f->peak_transient, transient + slot * chunk);
        for (int c0 = 0; c0 < nb; c0 += chunk) {
          IdArgs<TC, T> a;
          a.L = cur.d;
          a.boxes = d_cls + seg0;
          a.base = c0;
          a.ws = d_Y;
          a.ldY = ldY;
          a.half = half;
          a.k_out = d_k;
          a.perm_out = d_perm;
          a.T_ws = d_Tws;
          a.ixy = d_ixy;
          a.kp = f->kp;
          a.geo = f->geo;
          a.eps = f->params.eps;
          a.P = P;
          a.rho = ratio * Lbox;
          a.Lbox = Lbox;
          a.g_sm = g_sm;
          a.ptab = d_ptab;
          a.lsz = lsz;
          const int cnt = std::min(chunk, nb - c0);
          if (Q > 1) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(cnt * Q);
            cfg.blockDim = dim3(ntc);
            cfg.dynamicSmemBytes = smem_cl;
            cfg.stream = st;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = Q;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            RSS_CUDA(cudaLaunchKernelEx(&cfg, kcl, a));
          } else {
            k_id<TC, T><<<cnt, NT_ID, smem_id, st>>>(a);
          }
          RSS_LAUNCHED();
          f->launches += 1;
          f->n_id += 1;
        }
        return RSS_OK;
      };
      // the ID from the exact Gram matrix of a real stack: where its fixed-point
      // error is below the reflectors' (eps >= IDG_EPS) and G fits on chip; a
      // cluster policy asks for the reflector kernels
      const bool gram = (half || split) && f->params.eps >= IDG_EPS && prm->id_cluster == 0 && mmax < 65536 &&
                        idg_chol_bytes(nmax) <= GI_CHOL_SM && idg_tsolve_bytes(nmax) <= GI_CHOL_SM;
      auto run_gram = [&]() -> rss_status {
        auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
        GramWs w;
        w.nch = (mmax + GI_K - 1) / GI_K;
        w.ch = ((mmax + w.nch - 1) / w.nch + GI_B - 1) / GI_B * GI_B;
        w.J = (nmax + GI_B - 1) / GI_B;
        w.o_part = (size_t)w.nch * (w.ch / GI_B) * OZ_S * w.J * GI_BLK;
        w.o_R = w.o_part + (size_t)w.nch * w.J * w.J * GI_B * GI_B * sizeof(uint4);
        w.o_ex = w.o_R + up(sizeof(double) * (nn + nmax));
        w.o_m = w.o_ex + up(sizeof(int) * (size_t)w.nch * w.J * GI_B);
        w.slot = w.o_m + 256;
        const int cap = (int)std::max<size_t>(1, std::min<size_t>({(size_t)nb, (size_t(2) << 30) / w.slot, size_t(32768)}));
        const int nchunks = (nb + cap - 1) / cap;
        const int chunk = (nb + nchunks - 1) / nchunks;
        if (!gb_Y.ensure(w.slot * chunk)) {
          rss_set_error("rss_factor: device workspace allocation failed");
          return RSS_ENOMEM;
        }
        w.p = static_cast<unsigned char*>(gb_Y.p);
        f->peak_transient = std::max(f->peak_transient, transient + w.slot * chunk);
        const size_t smc = idg_chol_bytes(nmax), smt = idg_tsolve_bytes(nmax);
        RSS_CUDA(allow_smem(k_idg_gram));
        RSS_CUDA(allow_smem(k_idg_chol<T>));
        RSS_CUDA(allow_smem(k_idg_tsolve<T>));
        IdArgs<double, T> a{};
        a.L = cur.d;
        a.boxes = d_cls + seg0;
        a.half = half;
        a.k_out = d_k;
        a.perm_out = d_perm;
        a.T_ws = d_Tws;
        a.ixy = d_ixy;
        a.kp = f->kp;
        a.geo = f->geo;
        a.eps = f->params.eps;
        a.P = P;
        a.rho = ratio * Lbox;
        a.Lbox = Lbox;
        a.ptab = d_ptab;
        a.lsz = lsz;
        for (int c0 = 0; c0 < nb; c0 += chunk) {
          const int cnt = std::min(chunk, nb - c0);
          a.base = c0;
          const int ntc = cnt <= 152 ? (nmax > 64 ? 1024 : 512) : nmax > 72 ? 512 : nmax > 32 ? 256 : 128;
          k_idg_split<T><<<dim3(w.J * (GI_B / 8), w.nch, cnt), 256, 0, st>>>(a, w);
          RSS_LAUNCHED();
          k_idg_gram<<<dim3(idg_items(w.J), w.nch, cnt), 256, GI_ST, st>>>(cur.d.n, d_cls + seg0 + c0, w, d_err, tc_polls);
          RSS_LAUNCHED();
          k_idg_chol<T><<<cnt, ntc, smc, st>>>(a, w, d_err);
          RSS_LAUNCHED();
          k_idg_tsolve<T><<<dim3((nmax + 31) / 32, cnt), 128, smt, st>>>(a, w);
          RSS_LAUNCHED();
          f->launches += 4;
          f->n_id += 4;
        }
        return RSS_OK;
      };
      {
        const rss_status s_id = gram ? run_gram() : split ? run_id(double{}) : run_id(T{});
        if (s_id != RSS_OK) return s_id;
      }
      evs.back().second->stop(st);
      RSS_CUDA(cudaMemcpyAsync(hk.data(), d_k, sizeof(int) * nb, cudaMemcpyDeviceToHost, st));
      RSS_CUDA(cudaStreamSynchronize(st));
      if (nb > 0 && *std::min_element(hk.begin(), hk.begin() + nb) < 0) return device_status();
      f->t_id += tid_.ms();
      const double cf = (sizeof(T) == sizeof(double) || split) ? 1.0 : 4.0;
      for (int q = 0; q < nb; ++q) {   // k steps of Householder QR on the m x n stack
        const double m = mrows[q], n = cur.n[boxes[q]], k = hk[q];
        f->f_id += cf * (4.0 * m * n * k - 2.0 * k * k * (m + n) + 2.0 * k * k * k / 3.0);
      }

      // records for the boxes that have redundant points
      std::vector<BoxRec<T>> recs;
      std::vector<int> clsidx;
      int max_k = 0, max_r = 0, max_c = 0;
      for (int q = 0; q < nb; ++q) {
        const int B = boxes[q], bx = B % g, by = B / g;
        const int k = hk[q], n = cur.n[B], r = n - k;
        info.k[B] = k;
        if (r <= 0) continue;
        int c = k;
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx) {
            if (!dx && !dy) continue;
            const int x = bx + dx, y = by + dy;
            if (x < 0 || y < 0 || x >= g || y >= g) continue;
            c += cur.nact[y * g + x];
          }
        BoxRec<T> R{};
        R.box = B; R.k = k; R.r = r; R.c = c;
        R.Tm = static_cast<T*>(f->arena.get(sizeof(T) * (size_t)k * r));
        R.LU = static_cast<T*>(f->arena.get(sizeof(T) * (size_t)r * r));
        R.piv = static_cast<int*>(f->arena.get(sizeof(int) * r));
        R.We = static_cast<T*>(f->arena.get(sizeof(T) * (size_t)n * r));
        R.Wf = static_cast<T*>(f->arena.get(sizeof(T) * (size_t)n * r));
        R.E = static_cast<T*>(f->arena.get(sizeof(T) * (size_t)c * r));
        R.Ft = static_cast<T*>(f->arena.get(sizeof(T) * (size_t)c * r));
        R.idxR = static_cast<int*>(f->arena.get(sizeof(int) * r));
        R.idxC = static_cast<int*>(f->arena.get(sizeof(int) * c));
        R.cmap = static_cast<int*>(f->arena.get(sizeof(int) * c));
        if (!R.Tm || !R.LU || !R.piv || !R.We || !R.Wf || !R.E || !R.Ft || !R.idxR || !R.idxC ||
            !R.cmap) {
          rss_set_error("rss_factor: device arena allocation failed");
          return RSS_ENOMEM;
        }
        recs.push_back(R);
        clsidx.push_back(q);
        {
          const double cf = sizeof(T) == sizeof(double) ? 1.0 : 4.0;
          const double K = k, Rr = r, Cc = c;
          f->f_elim += cf * (4.0 * Cc * K * Rr + 4.0 * Rr * Rr * K + 2.0 * Rr * Rr * Rr / 3.0 + 2.0 * Cc * Rr * Rr);
          f->f_schur += cf * 2.0 * Cc * Cc * Rr;
        }
        max_k = std::max(max_k, k); max_r = std::max(max_r, r); max_c = std::max(max_c, c);
      }
      for (int q = 0; q < nb; ++q)
        if (cur.n[boxes[q]] - hk[q] > 0) cur.nact[boxes[q]] = hk[q];
      if (recs.empty()) continue;
      // a box may have c = 0 (rank 0 and no active neighbour: a far field that is
      // exactly zero); grids are sized for at least one row chunk, and the kernels
      // skip the chunks past each box's own c
      max_c = std::max(max_c, 1);
      const int nrec = (int)recs.size();
      // panel kernel shape: the widest panel (16 MA rows) whose shared memory
      // leaves room for two CTAs per SM; boxes beyond 200 KB take the row path
      int pan_ma = 1;
      size_t pan_max = 0;
      {
        int max_n = 0;
        for (const BoxRec<T>& R : recs) max_n = std::max(max_n, R.k + R.r);
        for (int ma : {4, 2, 1})
          if (panel_smem_bytes<T>(ma, max_n, max_r) <= 110 * 1024) { pan_ma = ma; break; }
        for (BoxRec<T>& R : recs) {
          const size_t pb = panel_smem_bytes<T>(pan_ma, R.k + R.r, R.r);
          R.panels = pb <= 200 * 1024 ? 1 : 0;
        }
      }
      // E = A_CB W_E and F^T = A_BC^T W_F on the tensor cores (elim_panels.cuh): real
      // boxes up to the n whose digits stay in shared memory, complex ones up to the n
      // whose rows' exponents do
      const bool sym = sizeof(T) == sizeof(double) && prm->kind == RSS_LAPLACE;
      EpArgs<T> ep = {};
      int ep_r = 0, ep_n = 0;
      if (prm->schur_path == 0 || prm->schur_path == 2) {
        constexpr int ozp_nmax = sizeof(T) == sizeof(double) ? 4 * TW_K : 3840;
        for (BoxRec<T>& R : recs) {
          if (R.k + R.r > ozp_nmax) continue;
          R.ozp = 1;
          ep_r = std::max(ep_r, R.r);
          ep_n = std::max(ep_n, R.k + R.r);
        }
      }
      if (ep_n > 0) {
        ep.sets = sym ? 1 : 2;
        ep.ns = cdiv(ep_n, ep_ks<T>());
        ep.ng = cdiv(sym ? 2 * ep_r : ep_r, 32);
        ep.nstr = cdiv(ep.ns, ep_smax<T>());
        ep.o_ew = (size_t)ep.sets * ep.ng * ep.ns * ep_parts<T>() * EP_GB;
        ep.slot = (ep.o_ew + (size_t)ep.sets * ep.ng * ep.nstr * 32 * sizeof(int) + 255) & ~size_t(255);
        if (!gb_w.ensure(ep.slot * nrec)) {
          rss_set_error("rss_factor: device workspace allocation failed");
          return RSS_ENOMEM;
        }
        ep.ws = static_cast<unsigned char*>(gb_w.p);
        f->peak_transient = std::max(f->peak_transient, transient + ep.slot * nrec);
        // real: the tile's digits over all of K, complex: two stages of them, beside
        // two or three stages of W and the rows' exponents
        ep.rows = sizeof(T) == sizeof(double) && ep.ns > 3 ? 96 : TW_M;
        ep.ad = sizeof(T) == sizeof(double) ? std::max(2, ep.ns) : 2;
        ep.wd = sizeof(T) == sizeof(double) && ep.ns <= 2 ? 3 : 2;
        ep.spn = TW_M;
      }
      for (const BoxRec<T>& R : recs)
        if (R.panels && !R.ozp) pan_max = std::max(pan_max, panel_smem_bytes<T>(pan_ma, R.k + R.r, R.r));
      // tensor-core Schur update for any r (K taken in chunks of 32)
      const bool oz = prm->schur_path == 0 || prm->schur_path == 2;
      const int ns = sizeof(T) == sizeof(double) ? OZ_S : 2 * OZ_S;   // slices per row
      int kp_max = 0;
      // complex, tcgen05: the slices in the layout of its stages, F's twice
      bool staged = sizeof(T) != sizeof(double) && prm->schur_path == 0;
      for (const BoxRec<T>& R : recs) staged = staged && R.ozp && R.r <= 16 * SZ_NS;
      auto slice_bytes = [&](const BoxRec<T>& R, int forms) {
        return forms * (size_t)(staged ? (R.c + 7) & ~7 : R.c) * ns * ((R.r + 15) & ~15) * sizeof(uint16_t);
      };
      const int fforms = staged ? 2 : 1;
      if (oz) {
        size_t bytes = 0;
        for (const BoxRec<T>& R : recs)
          bytes += slice_bytes(R, 1 + fforms) + 512 + 2 * ((size_t)R.c * sizeof(int) + 256);
        if (!gb_oz.ensure(bytes)) {
          rss_set_error("rss_factor: device workspace allocation failed");
          return RSS_ENOMEM;
        }
        char* p = static_cast<char*>(gb_oz.p);
        auto take = [&](size_t b) {
          char* q = p;
          p += (b + 255) & ~size_t(255);
          return q;
        };
        for (BoxRec<T>& R : recs) {
          R.kp = (R.r + 15) & ~15;
          kp_max = std::max(kp_max, R.kp);
          R.Esl = reinterpret_cast<uint16_t*>(take(slice_bytes(R, 1)));
          R.Fsl = reinterpret_cast<uint16_t*>(take(slice_bytes(R, fforms)));
          R.Eexp = reinterpret_cast<int*>(take((size_t)R.c * sizeof(int)));
          R.Fexp = reinterpret_cast<int*>(take((size_t)R.c * sizeof(int)));
        }
        f->peak_transient = std::max(f->peak_transient, transient + bytes);
      }
      // the column-group kernels, for boxes that fit them and take E and F from the
      // panel kernels; the FP64 panels read U^{-1} and L^{-1}, k_elim_lu also L^{-1} P
      int max_n = 0;
      bool ef_later = true;
      for (const BoxRec<T>& R : recs) {
        max_n = std::max(max_n, R.k + R.r);
        ef_later = ef_later && (R.panels || R.ozp);
      }
      const bool elim_cols =
          ef_later && std::max(elim_x_bytes<T>(8, max_k, max_n), elim_inv_bytes<T>(16, max_r)) <= 200 * 1024;
      {
        auto rr = [](const BoxRec<T>& R) { return ((size_t)R.r * R.r * sizeof(T) + 255) & ~size_t(255); };
        auto rp = [](const BoxRec<T>& R) { return ((size_t)R.r * sizeof(int) + 255) & ~size_t(255); };
        size_t bytes = 0;
        for (const BoxRec<T>& R : recs) bytes += rp(R) + (!elim_cols || !R.ozp ? 3 * rr(R) : 0);
        if (!gb_inv.ensure(bytes)) {
          rss_set_error("rss_factor: device workspace allocation failed");
          return RSS_ENOMEM;
        }
        f->peak_transient = std::max(f->peak_transient, transient + bytes);
        char* p = static_cast<char*>(gb_inv.p);
        for (BoxRec<T>& R : recs) {
          R.pos = reinterpret_cast<int*>(p);
          p += rp(R);
          if (elim_cols && R.ozp) continue;
          R.Ui = reinterpret_cast<T*>(p);
          R.Li = reinterpret_cast<T*>(p + rr(R));
          R.LiP = reinterpret_cast<T*>(p + 2 * rr(R));
          p += 3 * rr(R);
        }
      }
      BoxRec<T>* d_recs = static_cast<BoxRec<T>*>(f->arena.get(sizeof(BoxRec<T>) * nrec));
      if (!d_recs) { rss_set_error("rss_factor: device arena allocation failed"); return RSS_ENOMEM; }
      RSS_CUDA(cudaMemcpyAsync(d_recs, recs.data(), sizeof(BoxRec<T>) * nrec, cudaMemcpyHostToDevice, st));
      RSS_CUDA(cudaMemcpyAsync(d_clsidx, clsidx.data(), sizeof(int) * nrec, cudaMemcpyHostToDevice, st));
      ElimArgs<T> ea;
      ea.L = cur.d;
      ea.recs = d_recs;
      ea.cls_idx = d_clsidx;
      ea.perm_in = d_perm;
      ea.T_ws = d_Tws;
      ea.err = d_err;
      // shared memory of the per-box kernel: T and the LU of the largest box that fits
      const size_t ints = (2 * (size_t)max_r * sizeof(int) + 15) & ~size_t(15);
      const size_t want =
          sizeof(T) * ((size_t)max_r * max_r + std::max((size_t)max_k * max_r, (size_t)max_r * max_r)) + ints;
      const size_t ecap = std::min<size_t>(want, 200 * 1024);
      ea.smem_cap = (int)((ecap - ints) / sizeof(T));
      evs.emplace_back(1, std::make_unique<Ev>());
      evs.back().second->start(st);
      if (elim_cols) {
        // columns per CTA: as many as still give every SM two CTAs
        auto launch_x = [&](auto kern, int jc, size_t smem) -> cudaError_t {
          cudaError_t e = allow_smem(kern);
          if (e != cudaSuccess) return e;
          kern<<<dim3((max_r + jc - 1) / jc, nrec), 256, smem, st>>>(ea);
          return cudaGetLastError();
        };
        auto launch_inv = [&](auto kern, int nbc) -> cudaError_t {
          const size_t smem = elim_inv_bytes<T>(nbc, max_r);
          cudaError_t e = allow_smem(kern);
          if (e != cudaSuccess) return e;
          kern<<<dim3((max_r + nbc - 1) / nbc, 2, nrec), 16 * nbc, smem, st>>>(ea);
          return cudaGetLastError();
        };
        const long long groups = (long long)nrec * ((max_r + 15) / 16);
        RSS_CUDA(groups < 2 * 152 ? launch_x(k_elim_x<T, 2>, 4, elim_x_bytes<T>(2, max_k, max_n))
                                  : launch_x(k_elim_x<T, 8>, 16, elim_x_bytes<T>(8, max_k, max_n)));
        const size_t lub = std::min<size_t>(sizeof(T) * (size_t)max_r * (max_r | 1), 224 * 1024) + sizeof(int) * (size_t)max_r;
        const size_t lus = std::min<size_t>(lub, 224 * 1024);
        ea.smem_cap = (int)(lus / sizeof(T));
        RSS_CUDA(allow_smem(k_elim_lu2<T>));
        k_elim_lu2<T><<<nrec, 256, lus, st>>>(ea);
        RSS_LAUNCHED();
        RSS_CUDA(2 * groups < 2 * 152 ? launch_inv(k_elim_inv<T, 8>, 8) : launch_inv(k_elim_inv<T, 16>, 16));
        f->launches += 2;
      } else {
        RSS_CUDA(allow_smem(k_elim_lu<T>));
        k_elim_lu<T><<<nrec, NT, ecap, st>>>(ea);
      }
      RSS_LAUNCHED();
      if (pan_max > 0) {
        auto launch_panels = [&](auto kern, int rows) -> cudaError_t {
          cudaError_t e = allow_smem(kern);
          if (e != cudaSuccess) return e;
          kern<<<dim3((max_c + rows - 1) / rows, nrec), NT, pan_max, st>>>(ea);
          return cudaGetLastError();
        };
        RSS_CUDA(pan_ma == 4   ? launch_panels(k_elim_panels<T, 4>, 64)
                 : pan_ma == 2 ? launch_panels(k_elim_panels<T, 2>, 32)
                               : launch_panels(k_elim_panels<T, 1>, 16));
        RSS_LAUNCHED();
        f->launches += 1;
      }
      if (ep_n > 0) {
        ep.L = cur.d;
        ep.recs = d_recs;
        ep.cls_idx = d_clsidx;
        ep.perm_in = d_perm;
        ep.err = d_err;
        ep.polls = tc_polls;
        ep.staged = staged;
        // the passes of a tile over as many CTAs as the tiles leave SMs
        const int tiles = cdiv(max_c, ep.rows);
        ep.psplit = std::max(1, std::min<int>(ep.ng, 152 / std::max<long long>(1, (long long)tiles * ep.sets * nrec)));
        const int smem = ep.ad * ep.rows * OZ_S * TW_K * 2 + ep.wd * ep_parts<T>() * EP_GB + (ep.spn + ep.nstr * TW_M) * (int)sizeof(int);
        RSS_CUDA(allow_smem(k_ep<T>, 225 * 1024));
        k_ep_cut_w<T><<<dim3(ep.ng, ep.sets, nrec), EP_WT, 0, st>>>(ep);
        RSS_LAUNCHED();
        k_ep<T><<<dim3(tiles, ep.sets * ep.psplit, nrec), EP_NT, smem, st>>>(ep);
        RSS_LAUNCHED();
        f->launches += 2;
        if (ep.psplit > 1 && oz) {
          k_ep_slices<T><<<dim3(cdiv(max_c, TW_M), 2, nrec), 512, 0, st>>>(d_recs, staged);
          RSS_LAUNCHED();
          f->launches += 1;
        }
      }
      evs.back().second->stop(st);
      const int ntile = (max_c + 63) / 64;
      evs.emplace_back(2, std::make_unique<Ev>());
      evs.back().second->start(st);
      if (oz) {
        if constexpr (sizeof(T) == sizeof(double)) {
          const int ntr_rows = (max_c + ST_M - 1) / ST_M;
          if (prm->schur_path == 0 && kp_max <= SRW_KP && (long long)nrec * ntr_rows >= 2 * 152) {
            // tcgen05, one CTA per 128-row block walking its column tiles (one CTA per SM)
            const int nchm = (kp_max + ST_KC - 1) / ST_KC;
            const int smem = std::max(nchm * (ST_A + 2 * ST_B) + SRW_NT / 32 * SRW_XB, 120 * 1024);
            RSS_CUDA(allow_smem(k_schur_tc_rows));
            k_schur_tc_rows<<<dim3(ntr_rows, nrec), SRW_NT, smem, st>>>(cur.d, d_recs, d_err, polls, sym);
          } else if (prm->schur_path == 0 && kp_max <= OZ_KX) {   // tcgen05: FP32 group sums over the whole K
            const int smem = ST_A + ST_B;
            RSS_CUDA(allow_smem(k_schur_tc));
            const int ntr = (max_c + ST_M - 1) / ST_M, ntc = (max_c + ST_N - 1) / ST_N;
            k_schur_tc<<<dim3(ntr * ntc, nrec), ST_NT, smem, st>>>(cur.d, d_recs, d_err, polls, sym);
          } else {
            const size_t smem = 2 * (size_t)SR_BUF * sizeof(uint16_t);
            RSS_CUDA(allow_smem(k_schur_oz));
            const int ntr = (max_c + SR_M - 1) / SR_M, ntc = (max_c + SR_N - 1) / SR_N;
            k_schur_oz<<<dim3(ntr * ntc, nrec), NT, smem, st>>>(cur.d, d_recs, sym);
          }
        } else {
          if (staged) {
            const int nst = cdiv(kp_max, 16), trows = nst > 2 ? 96 : TW_M, ntr = cdiv(max_c, trows);
            const int ad = nst > 2 ? 3 : 2, nb = ad == 3 ? 5 : 6;   // stages of rows, pieces of columns in shared memory
            const int smem = ad * trows * SZ_AST + nb * SZ_BP;
            const int csplit = std::max(1, std::min<int>(cdiv(max_c, 32), 152 / std::max(1, ntr * nrec)));
            RSS_CUDA(allow_smem(k_schur_z));
            k_schur_z<<<dim3(nrec, csplit, ntr), EP_NT, smem, st>>>(cur.d, d_recs, trows, ad, nb, csplit, split ? 1 : 0, d_err, polls);
          } else {
            const size_t smem = (64 + 32) * (size_t)SCSA * sizeof(uint16_t);
            RSS_CUDA(allow_smem(k_schur_oz_c));
            const int ntc = (max_c + 31) / 32;
            k_schur_oz_c<<<dim3(ntile * ntc, nrec), NT, smem, st>>>(cur.d, d_recs);
          }
        }
      } else {
        k_schur<T><<<dim3(ntile * ntile, nrec), NT, 0, st>>>(cur.d, d_recs);
      }
      RSS_LAUNCHED();
      evs.back().second->stop(st);
      for (BoxRec<T>& R : recs) R.Esl = R.Fsl = nullptr, R.Eexp = R.Fexp = nullptr, R.Ui = R.Li = R.LiP = nullptr, R.pos = nullptr;
      f->launches += 2;
      f->n_elim += 1;
      f->n_schur += 1;
      void* hcopy = std::malloc(sizeof(BoxRec<T>) * nrec);
      if (!hcopy) { rss_set_error("rss_factor: host allocation failed"); return RSS_ENOMEM; }
      std::memcpy(hcopy, recs.data(), sizeof(BoxRec<T>) * nrec);
      f->rec_host.push_back(hcopy);
      const int colour = (boxes[0] % g) % 3 + 3 * ((boxes[0] / g) % 3);
      f->batches.push_back(Batch{g, colour, nrec, d_recs, max_k, max_r, max_c, max_n});
    }
    RSS_CUDA(cudaStreamSynchronize(st));
    for (auto& pe : evs) {
      const double ms = pe.second->ms();
      (pe.first == 0 ? f->g_id : pe.first == 1 ? f->g_elim : f->g_schur) += ms;
      (pe.first == 0 ? info.g_id : pe.first == 1 ? info.g_elim : info.g_schur) += ms;
      (pe.first == 1 ? f->t_elim : pe.first == 2 ? f->t_schur : f->t_gen) += pe.first ? ms : 0.0;
    }
    const rss_status s_dev = device_status();
    if (s_dev != RSS_OK) return s_dev;
    f->levels.push_back(info);

    // merge to the parent level
    Timer tm;
    const int gp = g / 2;
    HostLevel<T> par;
    par.n.assign(gp * gp, 0);
    int pmax = 1;
    for (int Pb = 0; Pb < gp * gp; ++Pb) {
      const int px = Pb % gp, py = Pb / gp;
      int s = 0;
      for (int q = 0; q < 4; ++q) s += cur.nact[(2 * py + q / 2) * g + 2 * px + q % 2];
      par.n[Pb] = s;
      pmax = std::max(pmax, s);
    }
    if (pmax > 65535) { rss_set_error("rss_factor: box too large after merging"); return RSS_EINVAL; }
    par.nact = par.n;
    {
      // when the parent's blocks do not fit beside the child's, keep only the
      // child's active entries (all the merge reads) and free the rest first
      size_t fr = 0, tot = 0;
      RSS_CUDA(cudaMemGetInfo(&fr, &tot));
      fr += pool_idle_bytes();
      const size_t pbytes = sizeof(T) * (size_t)gp * gp * 25 * (size_t)pmax * pmax;
      if (pbytes + (size_t(4) << 30) > fr) {
        int kmax = 1;
        for (int b = 0; b < nbox; ++b) kmax = std::max(kmax, cur.nact[b]);
        const size_t cbytes = sizeof(T) * (size_t)nbox * 25 * (size_t)kmax * kmax;
        T* cblk = nullptr;
        int *cpts = nullptr, *cact = nullptr;
        if (pool_malloc(reinterpret_cast<void**>(&cblk), cbytes, st) != cudaSuccess ||
            pool_malloc(reinterpret_cast<void**>(&cpts), sizeof(int) * (size_t)nbox * kmax, st) != cudaSuccess ||
            pool_malloc(reinterpret_cast<void**>(&cact), sizeof(int) * (size_t)nbox * kmax, st) != cudaSuccess) {
          pool_free(cblk, st); pool_free(cpts, st); pool_free(cact, st);
          rss_set_error("rss_factor: out of device memory for the compacted child blocks");
          return RSS_ENOMEM;
        }
        k_compact_blk<T><<<nbox * 25, NT, 0, st>>>(cur.d, cblk, cpts, kmax);
        RSS_LAUNCHED();
        k_iota_rows<<<1024, NT, 0, st>>>(cact, nbox, kmax);
        RSS_LAUNCHED();
        RSS_CUDA(cudaStreamSynchronize(st));
        f->launches += 2;
        pool_free(cur.d.blk, st);
        pool_free(cur.d.pts, st);
        pool_free(cur.d.act, st);
        transient -= sizeof(T) * (size_t)nbox * 25 * nn;
        transient += cbytes;
        cur.d.blk = cblk;
        cur.d.pts = cpts;
        cur.d.act = cact;
        cur.d.nmax = kmax;
      }
    }
    LevelGuard<T> par_guard{par, st};
    {
      rss_status s = alloc_level(par, gp, pmax, transient, st);
      if (s != RSS_OK) return s;
    }
    f->peak_transient = std::max(f->peak_transient, transient);
    Ev evm;
    evm.start(st);
    k_merge_pts<T><<<gp * gp, NT, 0, st>>>(cur.d, par.d);
    RSS_LAUNCHED();
    {
      const size_t msmem = (size_t)par.d.nmax * (2 * sizeof(int) + 2 * sizeof(int2));
      if (msmem > 48 * 1024)
        RSS_CUDA(allow_smem(k_merge_blk<T>));
      k_merge_blk<T><<<gp * gp * 25, NT, msmem, st>>>(cur.d, par.d, d_ixy, d_tab, f->kp, side);
    }
    RSS_LAUNCHED();
    evm.stop(st);
    RSS_CUDA(cudaStreamSynchronize(st));
    f->g_merge += evm.ms();
    f->launches += 2;
    transient -= sizeof(T) * (size_t)nbox * 25 * (size_t)cur.d.nmax * cur.d.nmax;
    free_level(cur, st);
    cur = par;
    par.d = LevelDev<T>{};   // owned by cur from here
    g = gp;
    f->t_merge += tm.ms();
  }

  // dense LU of everything still active (box grid side <= 2)
  Timer tt;
  {
    const int nbox = g * g;
    int offs[5] = {0, 0, 0, 0, 0};
    for (int b = 0; b < nbox; ++b) offs[b + 1] = offs[b] + cur.n[b];
    for (int b = nbox + 1; b < 5; ++b) offs[b] = offs[nbox];
    const int ntop = offs[nbox];
    f->ntop = ntop;
    f->d_top_idx = static_cast<int*>(f->arena.get(sizeof(int) * ntop));
    f->d_top_inv = f->arena.get(sizeof(T) * (size_t)ntop * ntop);
    if (!f->d_top_idx || !f->d_top_inv) {
      rss_set_error("rss_factor: device arena allocation failed");
      return RSS_ENOMEM;
    }
    // two matrices, a panel, the pivot block's inverse and two index lists
    constexpr int NB = gj_nb<T>();
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t mb = up(sizeof(T) * (size_t)ntop * ntop), pb = up(sizeof(T) * (size_t)ntop * NB);
    const size_t ib = up(sizeof(int) * (size_t)ntop);
    GrowBuf gb_top(st);
    if (!gb_top.ensure(2 * mb + pb + up(sizeof(T) * NB * NB) + 2 * ib)) {
      rss_set_error("rss_factor: device workspace allocation failed");
      return RSS_ENOMEM;
    }
    char* tp = static_cast<char*>(gb_top.p);
    T* const tbuf[2] = {reinterpret_cast<T*>(tp), reinterpret_cast<T*>(tp + mb)};
    T* tpan = reinterpret_cast<T*>(tp + 2 * mb);
    T* tD = reinterpret_cast<T*>(tp + 2 * mb + pb);
    int* tsrc = reinterpret_cast<int*>(tp + 2 * mb + pb + up(sizeof(T) * NB * NB));
    int* tpiv = reinterpret_cast<int*>(reinterpret_cast<char*>(tsrc) + ib);
    Ev evt;
    evt.start(st);
    k_top_assemble<T><<<nbox * nbox, NT, 0, st>>>(cur.d, tbuf[0], ntop, f->d_top_idx,
                                                  make_int4(offs[0], offs[1], offs[2], offs[3]), offs[4]);
    RSS_LAUNCHED();
    if (ntop > 0) {
      const int nl = gj_inverse<T>(tbuf, static_cast<T*>(f->d_top_inv), ntop, tD, tsrc, tpiv, d_err, tpan, st);
      if (nl < 0) {
        RSS_LAUNCHED();
        rss_set_error("rss_factor: top inverse launch failed");
        return RSS_ECUDA;
      }
      f->launches += nl;
    }
    evt.stop(st);
    span.stop(st);
    f->launches += 1;
    RSS_CUDA(cudaStreamSynchronize(st));
    f->g_top += evt.ms();
    f->g_span = span.ms();
    f->f_top += (sizeof(T) == sizeof(double) ? 1.0 : 4.0) * (2.0 / 3.0 + 2.0) * (double)ntop * ntop * ntop;
    free_level(cur, st);
    int herr = 0;
    RSS_CUDA(cudaMemcpy(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (herr) { rss_set_error("rss_factor: zero pivot in the inverse of the dense top block"); return RSS_ENUMERIC; }
  }
  f->t_top += tt.ms();
  {
    const rss_status sb = build_sweep_classes<T>(f, st);
    if (sb != RSS_OK) return sb;
  }
  f->t_total = total.ms();
  return RSS_OK;
}

template rss_status factor_impl<double>(const rss_tree*, const rss_params*, cudaStream_t, rss_factorization*);
template rss_status factor_impl<zd>(const rss_tree*, const rss_params*, cudaStream_t, rss_factorization*);
