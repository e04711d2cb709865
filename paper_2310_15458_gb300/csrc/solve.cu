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
#include "tc_gemm.cuh"

namespace {

constexpr int NT = 256;

#include "sweep.cuh"

template <typename T>
__global__ void k_perm_in(const T* __restrict__ b, int64_t ldb, T* __restrict__ x, int64_t N, int nrhs,
                          const int* __restrict__ u2t) {
  pdl_launch();
  const long long tot = (long long)N * nrhs;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const long long i = e % N, j = e / N;
    x[u2t[i] + j * N] = b[i + j * ldb];
  }
}

template <typename T>
__global__ void k_perm_out(T* __restrict__ b, int64_t ldb, const T* __restrict__ x, int64_t N, int nrhs,
                           const int* __restrict__ u2t, const int* __restrict__ err) {
  pdl_wait();
  // a grid-barrier wait of the persistent sweeps that ran out (*err != 0) voids
  // the result: every entry becomes NaN rather than a silently wrong number
  const bool bad = err != nullptr && *err != 0;
  const T nan = from_re<T>(__longlong_as_double(0x7FF8000000000000LL));
  const long long tot = (long long)N * nrhs;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const long long i = e % N, j = e / N;
    b[i + j * ldb] = bad ? nan : ld_l2(x + u2t[i] + j * N);
  }
}

// ------------------------------------------------------------------ many right-hand sides on the tensor cores
// Real factors with at least TCN right-hand sides: every product of a sweep is a
// small GEMM (factor block) x (TCN columns of right-hand sides), formed exactly
// from 7-bit digit slices as in the factorization's products: the rows of the
// factor block and the columns of the right-hand sides are scaled by powers of
// two and cut into eight digits (integer operations), the slice products are
// summed exactly by bf16 MMAs with FP32 accumulation, gathered into one int64
// per entry and per K chunk of TCK, and the chunks are added in FP64.  One CTA
// owns one box and TCN columns, so each sweep is one launch per colour class
// with no cross-CTA dependency.
constexpr int TCN = 32, TCM = 64, TCK = 32, TSA = 8 * TCK + 8;   // TSA: bf16 per slice row (16-byte rows)
constexpr int TC_NT = 256;

// C(i, q) receives sum_l A(i, l) B(l, q) for i < M, q < TCN; A(i, l) = aval(i, l),
// B(l, q) = bval(l, q) (FP64).  Every thread of the CTA calls it.
template <typename AF, typename BF, typename OF>
__device__ void tc_gemm32(int M, int K, AF aval, BF bval, OF cout, uint16_t* As, uint16_t* Bs, int* rexp,
                          int* cexp) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
  const int m0 = (warp >> 1) * 16, n0 = (warp & 1) * 16;
  const int a_row = lane & 15, a_k = (lane >> 4) * 8;
  const int b_row = ((lane >> 4) << 3) + (lane & 7), b_k = ((lane >> 3) & 1) * 8;
  __syncthreads();   // the caller's shared operands are written (with K = 0 no chunk barrier follows)
  for (int mt = 0; mt < M; mt += TCM) {
    double acc[2][4];
#pragma unroll
    for (int ni = 0; ni < 2; ++ni)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[ni][e] = 0.0;
    for (int kc = 0; kc < K; kc += TCK) {
      const int kl = min(TCK, K - kc);
      __syncthreads();   // the previous chunk's slices are consumed
      {   // rows of A: 64 rows x 4 lanes
        const int row = tid >> 2, gl = tid & 3, i = mt + row;
        const bool act = i < M;
        unsigned long long mk = 0;
        if (act)
          for (int l = gl; l < kl; l += 4) mk = max(mk, oz_abs_bits(aval(i, kc + l)));
        mk = max(mk, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mk, 1));
        mk = max(mk, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mk, 2));
        const int eb = oz_emax_b(mk);
        if (gl == 0) rexp[row] = eb - 1022;
        uint16_t* dst = As + row * TSA;
        for (int l = 2 * gl; l < TCK; l += 8) {
          const long long X0 = (act && l < kl) ? oz_scaled_int(aval(i, kc + l), eb) : 0;
          const long long X1 = (act && l + 1 < kl) ? oz_scaled_int(aval(i, kc + l + 1), eb) : 0;
          uint32_t dg[8];
          oz_digits2(X0, X1, dg);
#pragma unroll
          for (int p = 0; p < 8; ++p) *reinterpret_cast<uint32_t*>(dst + p * TCK + l) = dg[p];
        }
      }
      {   // columns of B: 32 columns x 8 lanes
        const int col = tid >> 3, gl = tid & 7;
        unsigned long long mk = 0;
        for (int l = gl; l < kl; l += 8) mk = max(mk, oz_abs_bits(bval(kc + l, col)));
#pragma unroll
        for (int d = 1; d < 8; d <<= 1)
          mk = max(mk, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mk, d));
        const int eb = oz_emax_b(mk);
        if (gl == 0) cexp[col] = eb - 1022;
        uint16_t* dst = Bs + col * TSA;
        for (int l = 2 * gl; l < TCK; l += 16) {
          const long long X0 = l < kl ? oz_scaled_int(bval(kc + l, col), eb) : 0;
          const long long X1 = l + 1 < kl ? oz_scaled_int(bval(kc + l + 1, col), eb) : 0;
          uint32_t dg[8];
          oz_digits2(X0, X1, dg);
#pragma unroll
          for (int p = 0; p < 8; ++p) *reinterpret_cast<uint32_t*>(dst + p * TCK + l) = dg[p];
        }
      }
      __syncthreads();
      long long W[2][4];
#pragma unroll
      for (int ni = 0; ni < 2; ++ni)
#pragma unroll
        for (int e = 0; e < 4; ++e) W[ni][e] = 0;
#pragma unroll 1
      for (int u = 0; u < 8; u += 2) {   // groups u, u + 1 together (|G| < 2^22)
        float c0[2][4], c1[2][4];
#pragma unroll
        for (int ni = 0; ni < 2; ++ni)
#pragma unroll
          for (int e = 0; e < 4; ++e) c0[ni][e] = c1[ni][e] = 0.f;
        for (int p = 0; p <= u + 1; ++p) {
          const uint16_t* Ab = As + p * TCK + (m0 + a_row) * TSA + a_k;
#pragma unroll
          for (int kk = 0; kk < TCK; kk += 16) {
            uint32_t af[4], bq[4];
            ldsm_x4(af, Ab + kk);
            ldsm_x4(bq, Bs + (u + 1 - p) * TCK + (n0 + b_row) * TSA + b_k + kk);
            mma_bf16(c1[0], af, bq);
            mma_bf16(c1[1], af, bq + 2);
            if (p <= u) {
              ldsm_x4(bq, Bs + (u - p) * TCK + (n0 + b_row) * TSA + b_k + kk);
              mma_bf16(c0[0], af, bq);
              mma_bf16(c0[1], af, bq + 2);
            }
          }
        }
        const int sh = 32 - 7 * u;
#pragma unroll
        for (int ni = 0; ni < 2; ++ni)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const long long gv = (long long)(oz_fint(c0[ni][e]) * 128 + oz_fint(c1[ni][e]));
            W[ni][e] += sh >= 0 ? (gv << sh) : ((gv + (1LL << (-sh - 1))) >> (-sh));
          }
      }
#pragma unroll
      for (int ni = 0; ni < 2; ++ni)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int row = m0 + gq + (e >= 2 ? 8 : 0), col = n0 + ni * 8 + 2 * t4 + (e & 1);
          acc[ni][e] += oz_ldexp_int(W[ni][e], rexp[row] + cexp[col] - 53);
        }
    }
#pragma unroll
    for (int ni = 0; ni < 2; ++ni)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int row = m0 + gq + (e >= 2 ? 8 : 0), col = n0 + ni * 8 + 2 * t4 + (e & 1);
        if (mt + row < M) cout(mt + row, col, acc[ni][e]);
      }
  }
  __syncthreads();
}

__device__ __forceinline__ size_t tc_smem_head() {
  return (size_t)(TCM + TCN) * TSA * sizeof(uint16_t);
}

// Slices of the rows of E (K = r), 64 rows per CTA, four lanes per row.
__global__ void __launch_bounds__(TC_NT) k_slice_e(const BoxRec<double>* __restrict__ recs,
                                                   const SliceRec* __restrict__ sl) {
  const BoxRec<double> R = recs[blockIdx.x];
  const SliceRec S = sl[blockIdx.x];
  const int i = blockIdx.y * 64 + (int)threadIdx.x / 4, c = R.c, r = R.r;
  if (blockIdx.y * 64 >= c) return;
  const bool act = i < c;
  const double* E = R.E;
  oz_split_vec<4>([&](int l) { return E[i + (size_t)l * c]; }, act ? r : 0, S.kp,
                  S.Esl + (size_t)(act ? i : 0) * OZ_S * S.kp, S.kp, S.Eexp + (act ? i : 0), act);
}

// Slices of the rows of F (columns of F^T, K = c), one warp per row.
__global__ void __launch_bounds__(TC_NT) k_slice_f(const BoxRec<double>* __restrict__ recs,
                                                   const SliceRec* __restrict__ sl) {
  const BoxRec<double> R = recs[blockIdx.x];
  const SliceRec S = sl[blockIdx.x];
  const int j = blockIdx.y * (TC_NT / 32) + (int)threadIdx.x / 32, c = R.c, r = R.r;
  if (blockIdx.y * (TC_NT / 32) >= r) return;
  const bool act = j < r;
  const double* Fc = R.Ft + (size_t)(act ? j : 0) * c;
  oz_split_vec<32>([&](int l) { return Fc[l]; }, act ? c : 0, S.cp, S.Fsl + (size_t)(act ? j : 0) * OZ_S * S.cp,
                   S.cp, S.Fexp + (act ? j : 0), act);
}

// C(i, q) receives sum_l A(i, l) B(l, q) for i < M, q < TCN, with the rows of A
// given as precomputed slices (row i at Asl + i * OZ_S * ka, scale 2^Aexp[i],
// zero past K) and B(l, q) = bval(l, q) in FP64, cut here under one scale per
// column over the whole K.  With both scales fixed along K, the eight group
// sums stay exact in FP32 for 384 entries of K and are gathered into one int64
// per entry (|W| <= K 2^53, K < 1024); K is staged in chunks of TCK.  Every
// thread of the CTA calls it.
template <typename BF, typename OF>
__device__ void tc_gemm_sl(int M, int ka, const uint16_t* __restrict__ Asl, const int* __restrict__ Aexp, BF bval,
                           OF cout, uint16_t* As, uint16_t* Bs, int* rexp, int* cexp, int* ceb) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
  const int m0 = (warp >> 1) * 16, n0 = (warp & 1) * 16;
  const int a_row = lane & 15, a_k = (lane >> 4) * 8;
  const int b_row = ((lane >> 4) << 3) + (lane & 7), b_k = ((lane >> 3) & 1) * 8;
  {   // column scales of B over the whole K (zero past it)
    const int col = tid >> 3, gl = tid & 7;
    unsigned long long mk = 0;
    for (int l = gl; l < ka; l += 8) mk = max(mk, oz_abs_bits(bval(l, col)));
#pragma unroll
    for (int d = 1; d < 8; d <<= 1)
      mk = max(mk, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mk, d));
    const int eb = oz_emax_b(mk);
    if (gl == 0) {
      ceb[col] = eb;
      cexp[col] = mk ? eb - 1022 : 0;
    }
  }
  for (int mt = 0; mt < M; mt += TCM) {
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
    auto gather = [&]() {
#pragma unroll
      for (int ni = 0; ni < 2; ++ni)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          long long w = W[ni][e];
#pragma unroll
          for (int u = 0; u < OZ_S; u += 2) {
            const long long gv = (long long)(oz_fint(acc[u][ni][e]) * 128 + oz_fint(acc[u + 1][ni][e]));
            const int sh = 32 - OZ_BITS * u;
            w += sh >= 0 ? (gv << sh) : ((gv + (1LL << (-sh - 1))) >> (-sh));
            acc[u][ni][e] = acc[u + 1][ni][e] = 0.f;
          }
          W[ni][e] = w;
        }
    };
    for (int kc = 0; kc < ka; kc += TCK) {
      const int kl = min(TCK, ka - kc), cpr = OZ_S * (kl / 8);   // ka is a multiple of 16
      __syncthreads();   // the previous chunk is consumed (and the column scales are visible)
      for (int e = tid; e < TCM * cpr; e += TC_NT) {   // rows of A: slices p, entries kc .. kc + kl
        const int row = e / cpr, rem = e % cpr, p = rem / (kl / 8), ch = rem % (kl / 8);
        uint16_t* d = As + row * TSA + p * TCK + ch * 8;
        if (mt + row < M)
          cp_async16(d, Asl + (size_t)(mt + row) * OZ_S * ka + (size_t)p * ka + kc + ch * 8);
        else
          *reinterpret_cast<uint4*>(d) = make_uint4(0, 0, 0, 0);
      }
      {   // columns of B: 32 columns x 8 lanes, two entries per lane and step
        const int col = tid >> 3, gl = tid & 7, eb = ceb[col];
        uint16_t* dst = Bs + col * TSA;
        for (int l = 2 * gl; l < TCK; l += 16) {
          const long long X0 = l < kl ? oz_scaled_int(bval(kc + l, col), eb) : 0;
          const long long X1 = l + 1 < kl ? oz_scaled_int(bval(kc + l + 1, col), eb) : 0;
          uint32_t dg[8];
          oz_digits2(X0, X1, dg);
#pragma unroll
          for (int p = 0; p < 8; ++p) *reinterpret_cast<uint32_t*>(dst + p * TCK + l) = dg[p];
        }
      }
      cp_async_wait_all();
      __syncthreads();
      for (int kk = 0; kk < kl; kk += 16) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // slices q = 4h .. 4h + 3 of B, then every A slice p <= 7 - q
          uint32_t bq[4][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) ldsm_x4(bq[q], Bs + (n0 + b_row) * TSA + (4 * h + q) * TCK + kk + b_k);
#pragma unroll
          for (int p = 0; p + 4 * h < OZ_S; ++p) {
            uint32_t af[4];
            ldsm_x4(af, As + (m0 + a_row) * TSA + p * TCK + kk + a_k);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (p + 4 * h + q < OZ_S) {
                mma_bf16(acc[p + 4 * h + q][0], af, bq[q]);
                mma_bf16(acc[p + 4 * h + q][1], af, bq[q] + 2);
              }
          }
        }
      }
      if ((kc / TCK + 1) % 12 == 0 && kc + TCK < ka) gather();   // 12 chunks: 384 entries of K
    }
    gather();
    if (tid < TCM) rexp[tid] = mt + tid < M ? Aexp[mt + tid] : 0;
    __syncthreads();
#pragma unroll
    for (int ni = 0; ni < 2; ++ni)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int row = m0 + gq + (e >= 2 ? 8 : 0), col = n0 + ni * 8 + 2 * t4 + (e & 1);
        if (mt + row < M) cout(mt + row, col, oz_ldexp_int(W[ni][e], rexp[row] + cexp[col] - 53));
      }
  }
  __syncthreads();
}

// Upward sweep of one box for TCN right-hand-side columns:
// b_R = W_F^T [b_S; b_R], b_C -= E b_R.
__global__ void __launch_bounds__(TC_NT, 2) k_up_tc(const BoxRec<double>* __restrict__ recs,
                                                    const SliceRec* __restrict__ sl, double* __restrict__ x,
                                                    int64_t N, int nrhs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<double> R = recs[blockIdx.x];
  const int k = R.k, r = R.r, c = R.c;
  const int q0 = blockIdx.y * TCN, nq = min(TCN, nrhs - q0);
  uint16_t* As = reinterpret_cast<uint16_t*>(smraw);
  uint16_t* Bs = As + TCM * TSA;
  double* v = reinterpret_cast<double*>(smraw + tc_smem_head());    // n x TCN: b_S, b_R
  double* u = v + (size_t)(k + r) * TCN;                             // r x TCN
  __shared__ int rexp[TCM], cexp[TCN], ceb[TCN];
  const int tid = threadIdx.x, bs = blockDim.x;
  double* xq = x + (int64_t)q0 * N;
  for (int e = tid; e < k * TCN; e += bs) {
    const int s2 = e / TCN, q = e % TCN;
    v[e] = q < nq ? xq[R.idxC[s2] + (int64_t)q * N] : 0.0;
  }
  for (int e = tid; e < r * TCN; e += bs) {
    const int j = e / TCN, q = e % TCN;
    v[k * TCN + e] = q < nq ? xq[R.idxR[j] + (int64_t)q * N] : 0.0;
  }
  const double* __restrict__ Wf = R.Wf;
  const double* __restrict__ E = R.E;
  const int n = k + r;
  tc_gemm32(r, n, [&](int i, int l) { return Wf[l + (size_t)i * n]; }, [&](int l, int q) { return v[l * TCN + q]; },
            [&](int i, int q, double d) { u[i * TCN + q] = d; }, As, Bs, rexp, cexp);
  for (int e = tid; e < r * TCN; e += bs) {
    const int j = e / TCN, q = e % TCN;
    if (q < nq) xq[R.idxR[j] + (int64_t)q * N] = u[e];
  }
  auto sub_c = [&](int i, int q, double v) {
    if (q < nq) {
      const int64_t gi = R.idxC[i] + (int64_t)q * N;
      xq[gi] = xq[gi] - v;
    }
  };
  if (sl != nullptr) {
    const SliceRec S = sl[blockIdx.x];
    tc_gemm_sl(c, S.kp, S.Esl, S.Eexp, [&](int l, int q) { return l < r ? u[l * TCN + q] : 0.0; }, sub_c, As, Bs,
               rexp, cexp, ceb);
  } else {
    tc_gemm32(c, r, [&](int i, int l) { return E[i + (size_t)l * c]; }, [&](int l, int q) { return u[l * TCN + q]; },
              sub_c, As, Bs, rexp, cexp);
  }
}

// Downward sweep of one box for TCN columns: z = y_R - F y_C, [y_S; y_R] =
// [y_S; 0] + W_E z.
__global__ void __launch_bounds__(TC_NT, 2) k_down_tc(const BoxRec<double>* __restrict__ recs,
                                                      const SliceRec* __restrict__ sl, double* __restrict__ x,
                                                      int64_t N, int nrhs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<double> R = recs[blockIdx.x];
  const int k = R.k, r = R.r, c = R.c;
  const int q0 = blockIdx.y * TCN, nq = min(TCN, nrhs - q0);
  uint16_t* As = reinterpret_cast<uint16_t*>(smraw);
  uint16_t* Bs = As + TCM * TSA;
  double* z = reinterpret_cast<double*>(smraw + tc_smem_head());   // r x TCN
  __shared__ int rexp[TCM], cexp[TCN], ceb[TCN];
  const int tid = threadIdx.x, bs = blockDim.x;
  double* xq = x + (int64_t)q0 * N;
  for (int e = tid; e < r * TCN; e += bs) {
    const int j = e / TCN, q = e % TCN;
    z[e] = q < nq ? xq[R.idxR[j] + (int64_t)q * N] : 0.0;
  }
  const double* __restrict__ Ft = R.Ft;
  const double* __restrict__ We = R.We;
  const int* __restrict__ idxC = R.idxC;
  if (sl != nullptr) {
    const SliceRec S = sl[blockIdx.x];
    tc_gemm_sl(r, S.cp, S.Fsl, S.Fexp,
               [&](int i, int q) { return (i < c && q < nq) ? xq[idxC[i] + (int64_t)q * N] : 0.0; },
               [&](int j, int q, double v) { z[j * TCN + q] -= v; }, As, Bs, rexp, cexp, ceb);
  } else {
    tc_gemm32(r, c, [&](int j, int i) { return Ft[i + (size_t)j * c]; },
              [&](int i, int q) { return q < nq ? xq[idxC[i] + (int64_t)q * N] : 0.0; },
              [&](int j, int q, double v) { z[j * TCN + q] -= v; }, As, Bs, rexp, cexp);
  }
  const int n = k + r;
  tc_gemm32(n, r, [&](int l, int j) { return We[l + (size_t)j * n]; }, [&](int j, int q) { return z[j * TCN + q]; },
            [&](int l, int q, double d) {
              if (q < nq) {
                double* g = xq + (l < k ? idxC[l] : R.idxR[l - k]) + (int64_t)q * N;
                *g = l < k ? *g + d : d;
              }
            },
            As, Bs, rexp, cexp);
}

// Complex factors with at least ZCN right-hand sides: the products of both sweeps
// as complex digit-slice GEMMs on the tensor cores (tc_gemm_c), one CTA per box
// and ZCN columns; the vectors of the box stay in shared memory between them.
__device__ __forceinline__ size_t tcz_head() { return (size_t)(ZCM + ZCN) * ZSA * sizeof(uint16_t); }
inline size_t tcz_smem_up(int n, int r) { return (size_t)(ZCM + ZCN) * ZSA * 2 + sizeof(zd) * ((size_t)n + r) * ZCN; }
inline size_t tcz_smem_down(int r) { return (size_t)(ZCM + ZCN) * ZSA * 2 + sizeof(zd) * (size_t)r * ZCN; }
constexpr size_t TCZ_SMEM_MAX = 220 * 1024;

// b_R = W_F^T [b_S; b_R], b_C -= E b_R.
__global__ void __launch_bounds__(TC_NT) k_up_tcz(const BoxRec<zd>* __restrict__ recs, zd* __restrict__ x,
                                                  int64_t N, int nrhs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<zd> R = recs[blockIdx.x];
  const int k = R.k, r = R.r, c = R.c;
  const int q0 = blockIdx.y * ZCN, nq = min(ZCN, nrhs - q0);
  uint16_t* As = reinterpret_cast<uint16_t*>(smraw);
  uint16_t* Bs = As + ZCM * ZSA;
  zd* v = reinterpret_cast<zd*>(smraw + tcz_head());    // n x ZCN: b_S, b_R
  zd* u = v + (size_t)(k + r) * ZCN;                      // r x ZCN
  __shared__ int rexp[ZCM], cexp[ZCN];
  const int tid = threadIdx.x, bs = blockDim.x;
  zd* xq = x + (int64_t)q0 * N;
  for (int e = tid; e < k * ZCN; e += bs) {
    const int s2 = e / ZCN, q = e % ZCN;
    v[e] = q < nq ? xq[R.idxC[s2] + (int64_t)q * N] : zero<zd>();
  }
  for (int e = tid; e < r * ZCN; e += bs) {
    const int j = e / ZCN, q = e % ZCN;
    v[k * ZCN + e] = q < nq ? xq[R.idxR[j] + (int64_t)q * N] : zero<zd>();
  }
  __syncthreads();   // (tc_gemm_c synchronises per K chunk; K = k may be 0)
  const zd* __restrict__ Wf = R.Wf;
  const zd* __restrict__ E = R.E;
  const int n = k + r;
  tc_gemm_c(r, n, [&](int i, int l) { return Wf[l + (size_t)i * n]; }, [&](int l, int q) { return v[l * ZCN + q]; },
            [&](int i, int q, zd d) { u[i * ZCN + q] = d; }, As, Bs, rexp, cexp);
  for (int e = tid; e < r * ZCN; e += bs) {
    const int j = e / ZCN, q = e % ZCN;
    if (q < nq) xq[R.idxR[j] + (int64_t)q * N] = u[e];
  }
  tc_gemm_c(c, r, [&](int i, int l) { return E[i + (size_t)l * c]; }, [&](int l, int q) { return u[l * ZCN + q]; },
            [&](int i, int q, zd v) {
              if (q < nq) {
                const int64_t gi = R.idxC[i] + (int64_t)q * N;
                xq[gi] = xq[gi] - v;
              }
            },
            As, Bs, rexp, cexp);
}

// z = y_R - F y_C, [y_S; y_R] = [y_S; 0] + W_E z.
__global__ void __launch_bounds__(TC_NT) k_down_tcz(const BoxRec<zd>* __restrict__ recs, zd* __restrict__ x,
                                                    int64_t N, int nrhs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BoxRec<zd> R = recs[blockIdx.x];
  const int k = R.k, r = R.r, c = R.c;
  const int q0 = blockIdx.y * ZCN, nq = min(ZCN, nrhs - q0);
  uint16_t* As = reinterpret_cast<uint16_t*>(smraw);
  uint16_t* Bs = As + ZCM * ZSA;
  zd* z = reinterpret_cast<zd*>(smraw + tcz_head());   // r x ZCN
  __shared__ int rexp[ZCM], cexp[ZCN];
  const int tid = threadIdx.x, bs = blockDim.x;
  zd* xq = x + (int64_t)q0 * N;
  for (int e = tid; e < r * ZCN; e += bs) {
    const int j = e / ZCN, q = e % ZCN;
    z[e] = q < nq ? xq[R.idxR[j] + (int64_t)q * N] : zero<zd>();
  }
  __syncthreads();
  const zd* __restrict__ Ft = R.Ft;
  const zd* __restrict__ We = R.We;
  const int* __restrict__ idxC = R.idxC;
  tc_gemm_c(r, c, [&](int j, int i) { return Ft[i + (size_t)j * c]; },
            [&](int i, int q) { return q < nq ? xq[idxC[i] + (int64_t)q * N] : zero<zd>(); },
            [&](int j, int q, zd v) { z[j * ZCN + q] = z[j * ZCN + q] - v; }, As, Bs, rexp, cexp);
  const int n = k + r;
  tc_gemm_c(n, r, [&](int l, int j) { return We[l + (size_t)j * n]; }, [&](int j, int q) { return z[j * ZCN + q]; },
            [&](int l, int q, zd d) {
              if (q < nq) {
                zd* g = xq + (l < k ? idxC[l] : R.idxR[l - k]) + (int64_t)q * N;
                *g = l < k ? *g + d : d;
              }
            },
            As, Bs, rexp, cexp);
}

// Top block: x_top <- A_top^{-1} x_top with the inverse formed at factor time.
template <typename T>
__global__ void k_top_gather(const int* __restrict__ idx, int n, const T* __restrict__ x, int64_t N, int nrhs,
                             T* __restrict__ z) {
  pdl_launch();
  pdl_wait();
  const long long tot = (long long)n * nrhs;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e % n);
    const long long q = e / n;
    z[e] = ld_l2(x + idx[i] + q * N);
  }
}

// 32 rows per CTA, the columns in SW_NT / 32 consecutive parts (one warp each)
// whose sums are added in order
template <typename T, int RC>
__global__ void __launch_bounds__(SW_NT) k_top_gemv(const T* __restrict__ Ainv, const int* __restrict__ idx, int n,
                                                    const T* __restrict__ z, T* __restrict__ x, int64_t N, int nrhs) {
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
    if (row < n && q < nq) x[idx[row] + (int64_t)(q0 + q) * N] = s;
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
rss_status top_apply(const rss_factorization* f, T* x, int64_t N, int nrhs, cudaStream_t st, T* topz) {
  if (f->ntop <= 0) return RSS_OK;
  const unsigned nz = cdiv(nrhs, RC);
  const unsigned g = std::min<long long>(cdiv((long long)f->ntop * nrhs, 256), 152LL * 8);
  RSS_CUDA(launch_pdl(k_top_gather<T>, dim3(g), 256, 0, st, 1, f->d_top_idx, f->ntop, x, N, nrhs, topz));
  RSS_CUDA(launch_pdl(k_top_gemv<T, RC>, dim3(cdiv(f->ntop, 32), nz), SW_NT, 0, st, 1,
                      static_cast<const T*>(f->d_top_inv), f->d_top_idx, f->ntop, topz, x, N, nrhs));
  return RSS_OK;
}

// The two persistent launches of the FP64 sweeps (k_sweep) around the top
// block.  Shared memory: the most any class needs without staging its matrices
// (at least 16 KB; more room lets them be staged); the grid: as many CTAs as fit
// on the device at once (a cooperative launch needs all of them resident).
constexpr long long SWP_POLLS = 1LL << 24;

template <typename T, int RC> size_t sweep_persistent_smem(const rss_factorization* f, int k0) {
  size_t need = 0;
  for (size_t i = k0; i < f->batches.size(); ++i) {
    const Batch& b = f->batches[i];
    need = std::max({need, sweep_sm_up<T, RC>(b.max_n, b.max_r, b.max_c, 1).need,
                     sweep_sm_down<T, RC>(b.max_n, b.max_r, b.max_c, 1, sweep_slices(b.nrec)).need});
  }
  const size_t smem = std::max(need * sizeof(T), size_t(16) << 10);
  return (smem + 1023) & ~size_t(1023);
}

// One persistent launch (k_sweep) over the colour classes k0 .. end of the
// factor order: upward in that order, or downward in reverse.
template <typename T, int RC>
rss_status sweep_persistent_launch(const rss_factorization* f, T* x, int64_t N, int nrhs, cudaStream_t st,
                                   unsigned* bar, int k0, bool up) {
  const size_t smem = sweep_persistent_smem<T, RC>(f, k0);
  int dev = 0, sms = 0;
  RSS_CUDA(cudaGetDevice(&dev));
  RSS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SwpArgs<T> a;
  a.cls = static_cast<const SwpClass<T>*>(f->d_swp) + k0;
  a.ncls = (int)f->batches.size() - k0;
  a.x = x;
  a.N = N;
  a.nrhs = nrhs;
  a.bar = bar;
  a.err = reinterpret_cast<int*>(bar + 2);
  a.polls = f->params.wait_polls == 0 ? SWP_POLLS : f->params.wait_polls < 0 ? 0 : (long long)f->params.wait_polls;
  a.sm_cap = (int)(smem / sizeof(T));
  void* args[] = {&a};
  const void* fn = up ? reinterpret_cast<const void*>(k_sweep<T, RC, true>)
                      : reinterpret_cast<const void*>(k_sweep<T, RC, false>);
  RSS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  RSS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, SWP_NT, smem));
  if (per_sm < 1) {
    rss_set_error("rss_solve: the persistent sweep kernel does not fit an SM");
    return RSS_ECUDA;
  }
  if (f->swp_ctas > 0) per_sm = std::min(per_sm, f->swp_ctas);
  RSS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(per_sm * sms), dim3(SWP_NT), args, smem, st));
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

// tcz: complex factors with at least ZCN right-hand sides take the tensor-core
// sweeps (k_up_tcz, k_down_tcz) for every colour class whose boxes fit their
// shared memory and that gives at least one CTA per SM (boxes x column chunks);
// smaller classes, whose one-CTA-per-box chain of products would be latency
// bound, keep these FP64 kernels, which spread the rows of C over CTAs.
// One colour class of the FP64 sweeps: Q CTAs per box, at most as many as the class
// has slices.  Fewer boxes (times column chunks) than SMs: a cluster per box, at most
// two CTAs to an SM, every matrix staged.  More: 128-thread CTAs that stage nothing,
// up to twelve to an SM, since the memory latency is then hidden by their number (one
// column at 1024^2: 4.0 ms so, 4.9 with the same classes staged; at 64^2, where every
// class is small, 0.26 ms staged and 0.40 not).  The columns are taken in smaller
// chunks where a box's vectors would not fit (the sums do not depend on it).
template <typename T, int RC, bool UP>
rss_status sweep_class(const Batch& b, T* x, int64_t N, int nrhs, cudaStream_t st) {
  const long long nz = cdiv(nrhs, RC);
  const int qc = sweep_slices(b.nrec);
  int Q = 1;
  const bool fills = b.nrec * nz > 152;
  while (Q < qc && b.nrec * nz * Q * 2 <= (fills ? 12 : 2) * 152) Q *= 2;
  const SweepSm s = UP ? sweep_sm_up<T, RC>(b.max_n, b.max_r, b.max_c, Q)
                       : sweep_sm_down<T, RC>(b.max_n, b.max_r, b.max_c, Q, qc);
  if (s.need * sizeof(T) > 220 * 1024) {
    if constexpr (RC > 1) {
      return sweep_class<T, RC == 8 ? 4 : 1, UP>(b, x, N, nrhs, st);
    } else {
      rss_set_error("rss_solve: a box's sweep needs more shared memory than an SM has");
      return RSS_EINVAL;
    }
  }
  const size_t smem = fills ? s.need * sizeof(T) : std::min<size_t>(s.full * sizeof(T), 220 * 1024);
  RSS_CUDA(cudaFuncSetAttribute(k_sweep_cl<T, RC, UP>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  RSS_CUDA(launch_pdl(k_sweep_cl<T, RC, UP>, dim3(b.nrec * Q, (unsigned)nz), fills ? 128 : SW_NT, smem, st, Q,
                      static_cast<const BoxRec<T>*>(b.d_recs), x, N, nrhs, Q, qc, (int)(smem / sizeof(T))));
  return RSS_OK;
}

template <typename T, int RC>
rss_status sweeps(const rss_factorization* f, T* x, int64_t N, int nrhs, cudaStream_t st, void* ws,
                  bool tcz = false) {
  const unsigned nzc = cdiv(nrhs, ZCN);
  if constexpr (std::is_same<T, zd>::value) {
    if (tcz) {
      RSS_CUDA(cudaFuncSetAttribute(k_up_tcz, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TCZ_SMEM_MAX));
      RSS_CUDA(cudaFuncSetAttribute(k_down_tcz, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TCZ_SMEM_MAX));
    }
  }
  const SweepWs w = sweep_ws<T>(f, nrhs, RC);
  char* wb = static_cast<char*>(ws);
  T* topz = reinterpret_cast<T*>(wb + w.topz_off);
  // classes k0 .. end go through the persistent launches (none, all, or the
  // coarse tail), the others through the per-class kernels
  const int nb = (int)f->batches.size();
  const int k0 = tcz ? nb : sweep_persistent_start<T, RC>(f);
  unsigned* bar = reinterpret_cast<unsigned*>(wb + w.bar_off);
  // the classes that take the complex tensor-core kernels
  auto on_tc = [&](const Batch& b) {
    return tcz && tcz_smem_up(b.max_n, b.max_r) <= TCZ_SMEM_MAX && (long long)b.nrec * nzc >= 152;
  };
  for (int bi = 0; bi < k0; ++bi) {
    const Batch& b = f->batches[bi];
    if constexpr (std::is_same<T, zd>::value) {
      if (on_tc(b)) {
        k_up_tcz<<<dim3(b.nrec, nzc), TC_NT, tcz_smem_up(b.max_n, b.max_r), st>>>(
            static_cast<const BoxRec<T>*>(b.d_recs), x, N, nrhs);
        RSS_LAUNCHED();
        continue;
      }
    }
    const rss_status s = sweep_class<T, RC, true>(b, x, N, nrhs, st);
    if (s != RSS_OK) return s;
  }
  if (k0 < nb) {
    const rss_status sp = sweep_persistent_launch<T, RC>(f, x, N, nrhs, st, bar, k0, true);
    if (sp != RSS_OK) return sp;
  }
  {
    const rss_status stp = top_apply<T, RC>(f, x, N, nrhs, st, topz);
    if (stp != RSS_OK) return stp;
  }
  if (k0 < nb) {
    const rss_status sp = sweep_persistent_launch<T, RC>(f, x, N, nrhs, st, bar, k0, false);
    if (sp != RSS_OK) return sp;
  }
  for (int bi = k0 - 1; bi >= 0; --bi) {
    const Batch& b = f->batches[bi];
    if constexpr (std::is_same<T, zd>::value) {
      if (on_tc(b)) {
        k_down_tcz<<<dim3(b.nrec, nzc), TC_NT, tcz_smem_down(b.max_r), st>>>(
            static_cast<const BoxRec<T>*>(b.d_recs), x, N, nrhs);
        RSS_LAUNCHED();
        continue;
      }
    }
    const rss_status s = sweep_class<T, RC, false>(b, x, N, nrhs, st);
    if (s != RSS_OK) return s;
  }
  return RSS_OK;
}

// The digit slices of E and F for the tensor-core sweeps: built once per factor
// by the first solve that needs them (on its stream, which it then waits for),
// kept until the factor is freed.  Boxes with c >= 1024 keep the per-chunk
// products (the int64 sums of tc_gemm_sl need K < 1024).
bool slices_fit(const rss_factorization* f) {
  for (const Batch& b : f->batches)
    if (b.max_c >= 1024) return false;
  return true;
}

size_t slice_total(const rss_factorization* f) {
  auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
  size_t total = 0;
  for (size_t bi = 0; bi < f->batches.size(); ++bi) {
    const Batch& b = f->batches[bi];
    const BoxRec<double>* hr = static_cast<const BoxRec<double>*>(f->rec_host[bi]);
    total += al(sizeof(SliceRec) * b.nrec);
    for (int q = 0; q < b.nrec; ++q) {
      const size_t kp = (hr[q].r + 15) & ~15, cp = (hr[q].c + 15) & ~15;
      total += al(sizeof(uint16_t) * hr[q].c * OZ_S * kp) + al(sizeof(int) * hr[q].c) +
               al(sizeof(uint16_t) * hr[q].r * OZ_S * cp) + al(sizeof(int) * hr[q].r);
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
  RSS_CUDA(pool_malloc(reinterpret_cast<void**>(&base), total, st));
  char* p = base;
  auto take = [&](size_t b) {
    char* q = p;
    p += al(b);
    return q;
  };
  std::vector<SliceRec*> recs(f->batches.size());
  std::vector<SliceRec> hs;
  for (size_t bi = 0; bi < f->batches.size(); ++bi) {
    const Batch& b = f->batches[bi];
    const BoxRec<double>* hr = static_cast<const BoxRec<double>*>(f->rec_host[bi]);
    recs[bi] = reinterpret_cast<SliceRec*>(take(sizeof(SliceRec) * b.nrec));
    hs.assign(b.nrec, SliceRec{});
    for (int q = 0; q < b.nrec; ++q) {
      SliceRec& S = hs[q];
      S.kp = (hr[q].r + 15) & ~15;
      S.cp = (hr[q].c + 15) & ~15;
      S.Esl = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * hr[q].c * OZ_S * S.kp));
      S.Eexp = reinterpret_cast<int*>(take(sizeof(int) * hr[q].c));
      S.Fsl = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * hr[q].r * OZ_S * S.cp));
      S.Fexp = reinterpret_cast<int*>(take(sizeof(int) * hr[q].r));
    }
    cudaError_t e = cudaMemcpyAsync(recs[bi], hs.data(), sizeof(SliceRec) * b.nrec, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // hs is reused for the next batch
    if (e == cudaSuccess) {
      const BoxRec<double>* dr = static_cast<const BoxRec<double>*>(b.d_recs);
      k_slice_e<<<dim3(b.nrec, cdiv(b.max_c, 64)), TC_NT, 0, st>>>(dr, recs[bi]);
      k_slice_f<<<dim3(b.nrec, cdiv(b.max_r, TC_NT / 32)), TC_NT, 0, st>>>(dr, recs[bi]);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
      cudaStreamSynchronize(st);
      pool_free(base, st);
      rss_set_error(std::string("rss_solve: slice cache: ") + cudaGetErrorString(e));
      return RSS_ECUDA;
    }
  }
  RSS_CUDA(cudaStreamSynchronize(st));   // other streams may use the slices from here on
  f->slice_bytes = total;
  f->d_slice_mem = base;
  f->d_slices = recs;
  f->slices_ready = true;
  return RSS_OK;
}

// Real factors with at least TCN right-hand sides: the tensor-core sweeps; the
// top block as in sweeps<double, 8>.
// may_build: the caller allows the one-time allocation of the slice cache
// (rss_solve_noalloc does not; it uses the cache only when it already exists).
rss_status sweeps_tc(const rss_factorization* f, double* x, int64_t N, int nrhs, cudaStream_t st, void* ws,
                     bool may_build) {
  constexpr int RC = 8;
  bool sl = slices_fit(f);
  if (sl && may_build) {
    const rss_status s = ensure_slices(const_cast<rss_factorization*>(f), st);
    if (s != RSS_OK) return s;
  } else if (sl) {
    std::lock_guard<std::mutex> lk(const_cast<rss_factorization*>(f)->slice_mu);
    sl = f->slices_ready;
  }
  const unsigned nz = cdiv(nrhs, TCN);
  const SweepWs w = sweep_ws<double>(f, nrhs, RC);
  double* topz = reinterpret_cast<double*>(static_cast<char*>(ws) + w.topz_off);
  RSS_CUDA(cudaFuncSetAttribute(k_up_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  RSS_CUDA(cudaFuncSetAttribute(k_down_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  const size_t head = (size_t)(TCM + TCN) * TSA * sizeof(uint16_t);
  for (size_t bi = 0; bi < f->batches.size(); ++bi) {
    const Batch& b = f->batches[bi];
    const size_t sm = head + sizeof(double) * ((size_t)b.max_n + b.max_r) * TCN;
    if (sm > 220 * 1024) {
      rss_set_error("rss_solve: box too large for the tensor-core sweep");
      return RSS_EINVAL;
    }
    k_up_tc<<<dim3(b.nrec, nz), TC_NT, sm, st>>>(static_cast<const BoxRec<double>*>(b.d_recs),
                                                  sl ? f->d_slices[bi] : nullptr, x, N, nrhs);
    RSS_LAUNCHED();
  }
  const rss_status stp = top_apply<double, RC>(f, x, N, nrhs, st, topz);
  if (stp != RSS_OK) return stp;
  for (size_t bi = f->batches.size(); bi-- > 0;) {
    const Batch& b = f->batches[bi];
    const size_t sm = head + sizeof(double) * (size_t)b.max_r * TCN;
    k_down_tc<<<dim3(b.nrec, nz), TC_NT, sm, st>>>(static_cast<const BoxRec<double>*>(b.d_recs),
                                                    sl ? f->d_slices[bi] : nullptr, x, N, nrhs);
    RSS_LAUNCHED();
  }
  return RSS_OK;
}

bool use_tc(const rss_factorization* f, int64_t nrhs) {
  return !f->is_complex && nrhs >= TCN && (f->params.schur_path == 0 || f->params.schur_path == 2);
}

template <typename T>
rss_status run_sweeps(const rss_factorization* f, T* x, int64_t N, int64_t nrhs, cudaStream_t st, void* ws,
                      bool may_build = true) {
  if constexpr (sizeof(T) == sizeof(double))
    if (use_tc(f, nrhs)) return sweeps_tc(f, x, N, (int)nrhs, st, ws, may_build);
  const int rc = rhs_chunk(nrhs);
  const bool tcz = f->is_complex && nrhs >= ZCN && (f->params.schur_path == 0 || f->params.schur_path == 2);
  return rc == 1 ? sweeps<T, 1>(f, x, N, (int)nrhs, st, ws, tcz)
         : rc == 4 ? sweeps<T, 4>(f, x, N, (int)nrhs, st, ws, tcz)
                   : sweeps<T, 8>(f, x, N, (int)nrhs, st, ws, tcz);
}

}  // namespace

template <typename T>
rss_status solve_impl(const rss_factorization* f, T* b, int64_t nrhs, int64_t ldb, cudaStream_t st) {
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
  if (s == RSS_OK) s = run_sweeps<T>(f, x, N, nrhs, st, mem + xb);
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

template rss_status solve_impl<double>(const rss_factorization*, double*, int64_t, int64_t, cudaStream_t);

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

size_t solve_cache_bytes(const rss_factorization* f, int64_t max_nrhs) {
  return use_tc(f, max_nrhs) && slices_fit(f) ? slice_total(f) : 0;
}

rss_status prepare_solve_caches(const rss_factorization* f, int64_t max_nrhs, cudaStream_t st) {
  if (!use_tc(f, max_nrhs) || !slices_fit(f)) return RSS_OK;
  return ensure_slices(const_cast<rss_factorization*>(f), st);
}
template rss_status solve_impl<zd>(const rss_factorization*, zd*, int64_t, int64_t, cudaStream_t);

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
  const rss_status s = run_sweeps<T>(f, x, N, nrhs, st, ws, false);
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
// solve, never its result.  (A candidate's `spread` is kept in the table for readers
// of earlier ones; no form uses it.)
extern "C" rss_status rss_tune_solve(rss_factorization* f, int64_t nrhs, void* stream, char* json, size_t len) {
  if (!f || f->tag != RSS_TAG_FACTOR || nrhs <= 0 || nrhs >= 1 << 20) {
    rss_set_error("rss_tune_solve: needs a factor handle and 0 < nrhs < 2^20");
    return RSS_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t esz = f->is_complex ? 16 : 8;
  const bool fp64_path = f->is_complex ? nrhs < ZCN : !use_tc(f, nrhs);
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
    const int ncand = (int)(sizeof(cands) / sizeof(cands[0]));
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
      float t[3];
      for (int rep = -1; rep < 3 && s == RSS_OK; ++rep) {   // one untimed run first
        cudaEventRecord(e0, st);
        s = f->is_complex ? solve_impl<zd>(f, static_cast<zd*>(b), nrhs, f->n, st)
                          : solve_impl<double>(f, static_cast<double*>(b), nrhs, f->n, st);
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) s = RSS_ECUDA;
        if (rep >= 0 && s == RSS_OK) cudaEventElapsedTime(&t[rep], e0, e1);
      }
      if (s != RSS_OK) break;
      std::sort(t, t + 3);
      o << (ci ? ", " : "") << "{\"launch\": \"" << (c.launch == 1 ? "per_class" : c.launch == 2 ? "persistent" : "hybrid")
        << "\"";
      if (c.launch != 1) o << ", \"spread\": " << c.spread << ", \"ctas_per_sm\": " << c.ctas;
      if (c.launch == 3) o << ", \"tail_boxes\": " << c.tail;
      o << ", \"ms\": " << t[1] << "}";
      if (t[1] < best_ms) {
        best_ms = t[1];
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
