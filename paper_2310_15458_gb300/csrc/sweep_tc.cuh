// The sweeps with many right-hand sides on the 5th-generation tensor cores.  Per
// colour class two products up, y = W_F^T [b_S; b_R] into b_R and b_C -= E b_R, and
// two down, z = y_R - F y_C into y_R and [y_S; y_R] = [y_S; 0] + W_E y_R (see
// sweep.cuh), each a launch of one CTA per box, 128 rows of the matrix and TW_NC real
// columns.  Rows of the matrix and columns of the right-hand sides are scaled by powers of
// two over stretches of K (SX) and cut into eight signed 7-bit digits; the slice products
// of equal weight u = p + q <= 7 are summed exactly in FP32 in tensor memory over a
// stretch, gathered into one int64 per output and added in FP64: the accuracy of an FP64
// product.  A complex product is the real one with K doubled, [A_re A_im] times
// [B_re; -B_im] and [B_im; B_re]: the two column groups of a CTA are then the real and
// imaginary parts of 32 columns.
//
// The products with W_F and W_E write what they read: of a box of more than 128 points the
// row tiles form a cluster and meet between the two (64 columns, FP64 sweeps before, this
// after: Laplace 384^2, leaf 144 36.5 -> 6.5 ms, 512^2, leaf 256 112 -> 13.1; Helmholtz
// 192^2, leaf 144 31.6 -> 9.1).
//
// K is staged 32 at a time in two to four buffers, so the digits of one stage are cut
// while the products of the others run; the down sweep's F y_C (K = c, up to thousands)
// is split over a cluster of up to 8 CTAs where a class has few boxes, and the
// parts are added in order.  A column that holds an
// infinity or a NaN gives NaN.  Real factors keep the matrices' digits (SliceRec, built
// by the first call of 32 and more columns), which then come by bulk copies; with fewer
// columns and for complex factors they are cut on the fly.
//
// Bound by latency: one CTA of 16 warps on an SM gathers x, cuts, meets at a block barrier
// a stage and joins; in the leaf classes the tensor pipe is busy for 9 to 10 % of the time
// (about 70 clocks a product), no other unit for more than 25 %; in the coarse classes a
// launch takes about 20 us.  64 columns, against mma.sync products of one CTA per box
// (real) and the FP64 sweeps (complex): Laplace 512^2 23.3 -> 9.2 ms, Helmholtz 256^2
// 30.3 -> 11.9 ms; 16 columns, against the FP64 sweeps: 4.1 -> 3.2 ms (Laplace
// 256^2).
// Stages of K that share scales and sums (SX below; tw_stages).  Shorter stretches follow
// the entries' range more closely and cost a gather each.  Errors of a panel against the
// records applied in quadruple precision, and 64 columns' times:
//   complex (Helmholtz, 64^2, leaf 64): 9.8e-16 in stretches of 48 entries, of one-column
//     FP64 solves 1.00e-15; of 128, 192 and 384: 1.06e-15, 1.08e-15 and 1.14e-15, in 11.0,
//     10.7 and 10.2 ms instead of 11.9 (256^2);
//   real, n <= 128 (Laplace, 64^2, leaf 64): 3.36e-16 in stretches of 384, FP64 3.25e-16;
//   real, n > 128: see TW_SX_LONG in launch_tw.
static_assert(TW_M == 128 && TW_K == 32 && OZ_S == 8 && TW_SX == TW_KX / TW_K && TW_SXZ == TW_KN / TW_K, "");

// rows and inner dimension of a product
template <int OP, typename T> __host__ __device__ inline int tw_rows(const BoxRec<T>& R) {
  return OP == TW_UPE ? R.c : OP == TW_DNW ? R.k + R.r : R.r;
}
template <int OP, typename T> __host__ __device__ inline int tw_inner(const BoxRec<T>& R) {
  return OP == TW_UPW ? R.k + R.r : OP == TW_DNF ? R.c : R.r;
}
// the matrix: entry (i, l) at p[i * si + l * sl]
template <int OP, typename T> __device__ __forceinline__ const T* tw_mat(const BoxRec<T>& R, size_t& si, size_t& sl) {
  if (OP == TW_UPW) { si = R.k + R.r; sl = 1; return R.Wf; }
  if (OP == TW_UPE) { si = 1; sl = R.c; return R.E; }
  if (OP == TW_DNF) { si = R.c; sl = 1; return R.Ft; }
  si = 1; sl = R.k + R.r; return R.We;
}
constexpr bool tw_k_contiguous(int op) { return op == TW_UPW || op == TW_DNF; }

// Exponents (biased, at least 1) of the largest of the entries K0 .. K of the CTA's rows
// i0 .., for each stretch st of K (from the one of K0 on), into reb[st * TW_M + i], which
// holds 1s.  (A barrier must follow.)
template <int OP, int SX, typename T>
__device__ void tw_row_exps(const BoxRec<T>& R, int i0, int rows, int K0, int K, int* reb) {
  constexpr int KX = SX * (sizeof(T) == sizeof(double) ? TW_K : TW_K / 2);
  size_t si, sl;
  const T* A = tw_mat<OP>(R, si, sl);
  const int tid = threadIdx.x;
  for (int l0 = K0, st = 0; l0 < K; l0 = (l0 / KX + 1) * KX, ++st) {
    const int l1 = min(K, (l0 / KX + 1) * KX);
    if (tw_k_contiguous(OP)) {   // a warp per row
      for (int i = tid / 32; i < rows; i += TW_NT / 32) {
        unsigned long long mk = 0;
        for (int l = l0 + tid % 32; l < l1; l += 32) mk = max(mk, tw_key(A[(i0 + i) * si + l]));
        mk = shfl_max_u64(mk, 32);
        if (tid % 32 == 0) reb[st * TW_M + i] = oz_emax_b(mk);
      }
    } else {                     // four threads per row, lanes over rows
      const int i = tid % TW_M, part = tid / TW_M;
      unsigned long long mk = 0;
      if (i < rows) {
        for (int l = l0 + part; l < l1; l += TW_NT / TW_M) mk = max(mk, tw_key(A[(i0 + i) + (size_t)l * sl]));
        atomicMax(&reb[st * TW_M + i], oz_emax_b(mk));
      }
    }
  }
}

// One stage (K entries 32 s ..; complex: 16 entries) of the rows' digits at d, slices
// `stride` bytes apart.  Real: a thread cuts eight entries of a row; complex: eight
// real and eight imaginary parts (half the threads).
template <int OP, typename T>
__device__ __forceinline__ void tw_cut_a(const BoxRec<T>& R, int i0, int rows, int K, int s, const int* reb,
                                         unsigned char* d, size_t stride) {
  size_t si, sl;
  const T* A = tw_mat<OP>(R, si, sl);
  constexpr bool cplx = sizeof(T) != sizeof(double);
  constexpr int G = cplx ? 2 : 4;   // groups of eight entries of a stage
  const int tid = threadIdx.x;
  if (tid >= TW_M * G) return;
  const int i = tw_k_contiguous(OP) ? tid / G : tid % TW_M, kg = tw_k_contiguous(OP) ? tid % G : tid / TW_M;
  if (i >= ((rows + 7) & ~7)) return;
  const int l0 = s * 8 * G + kg * 8, eb = i < rows ? reb[i] : 1;
  const T* a = A + (size_t)(i0 + i) * si + (size_t)l0 * sl;
  T v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = (i < rows && l0 + e < K) ? a[(size_t)e * sl] : zero<T>();
  long long X[8];
  if constexpr (!cplx) {
#pragma unroll
    for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e], eb);
    tw_put8(X, d + tw_at(i, kg), stride, 0u);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].x, eb);
    tw_put8(X, d + tw_at(i, kg), stride, 0u);
#pragma unroll
    for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].y, eb);
    tw_put8(X, d + tw_at(i, 2 + kg), stride, 0u);
  }
}

// Digits of the four matrices of a real box, in the stages' layout: for the rows of
// tile t (128 rows, the last one rounded up to 8) and stage s, slice p at
// base + off(t) + (s * 8 + p) * rows8 * 64.
__host__ __device__ inline size_t tw_tile_off(int t, int K) { return (size_t)t * TW_M * ((K + TW_K - 1) / TW_K) * (OZ_S * TW_K * 2); }
inline size_t tw_cache_bytes(int rows, int K) {
  return (size_t)((rows + 7) & ~7) * ((K + TW_K - 1) / TW_K) * (OZ_S * TW_K * 2);
}
// One CTA per box, row tile and stretch of K: a long K in one CTA is a serial chain in the
// coarse classes (first call of 32 columns, 512^2, eps 1e-9: 19.6 ms so, 14.6 now).
template <int OP, int SX>
__global__ void __launch_bounds__(TW_NT) k_tw_cache(const BoxRec<double>* __restrict__ recs, const SliceRec* __restrict__ sl) {
  constexpr int KX = SX * TW_K;
  __shared__ int reb[TW_M];
  const BoxRec<double> R = recs[blockIdx.y];
  const SliceRec S = sl[blockIdx.y];
  const int M = tw_rows<OP>(R), K = tw_inner<OP>(R), i0 = blockIdx.x * TW_M, rows = min(TW_M, M - i0);
  const int st = blockIdx.z, l0 = st * KX, l1 = min(K, l0 + KX);
  if (rows <= 0 || l0 >= K) return;
  if (threadIdx.x < TW_M) reb[threadIdx.x] = 1;
  __syncthreads();
  tw_row_exps<OP, SX>(R, i0, rows, l0, l1, reb);
  __syncthreads();
  const int rows8 = (rows + 7) & ~7;
  unsigned char* base = S.dig[OP] + tw_tile_off(blockIdx.x, K);
  for (int s = st * SX; s * TW_K < l1; ++s)
    tw_cut_a<OP>(R, i0, rows, K, s, reb, base + (size_t)s * OZ_S * rows8 * 64, (size_t)rows8 * 64);
  for (int i = threadIdx.x; i < rows; i += TW_NT) S.eb[OP][(size_t)st * M + i0 + i] = reb[i];
}

// GW: columns of a group (32, or 16 for classes of few boxes: more and shorter CTAs)
template <typename T, int OP, bool CACHE, int GW, int SX>
__global__ void __launch_bounds__(TW_NT, 1) k_tw(const BoxRec<T>* __restrict__ recs, const SliceRec* __restrict__ sl,
                                                 T* __restrict__ x, int64_t ldx, int nrhs, int srows, int nst, int nstr, int* err,
                                                 int polls) {
  extern __shared__ __align__(1024) unsigned char sm[];
  constexpr bool cplx = sizeof(T) != sizeof(double);
  constexpr int KS = cplx ? TW_K / 2 : TW_K;       // entries of K per stage
  constexpr int NC = cplx ? GW : 2 * GW;           // right-hand sides per CTA
  constexpr int BG = OZ_S * GW * TW_K * 2;         // bytes of a group's stage
  constexpr int CT = GW / 4;                       // columns of a group per thread
  constexpr int LDO = NC + 1;
  __shared__ __align__(8) uint64_t mb_mma[4], mb_full[4];
  __shared__ uint32_t s_tmem;
  __shared__ int s_bad[2];
  const BoxRec<T> R = recs[blockIdx.z];
  const int M = tw_rows<OP>(R), Kall = tw_inner<OP>(R), k = R.k;
  // the down sweep's long inner dimension: a cluster of CTAs, each a range of stages
  const int spl = OP == TW_DNF ? (int)cooperative_groups::this_cluster().num_blocks() : 1;
  const int rank = OP == TW_DNF ? (int)cooperative_groups::this_cluster().block_rank() : 0;
  // the row tiles of a product that writes what the others read meet before they write
  const bool meet = (OP == TW_UPW || OP == TW_DNW) && gridDim.x > 1;
  const int tile0 = blockIdx.x / spl, i0 = tile0 * TW_M, rows = min(TW_M, M - i0);
  const int nsall = (Kall + KS - 1) / KS, s0 = nsall * rank / spl, ns = nsall * (rank + 1) / spl - s0;
  const int K0 = s0 * KS, K = min(Kall, (s0 + ns) * KS);   // this CTA's entries of K
  pdl_launch();
  // (a launch without a row, E where every box has c = 0, must not end before the launch
  // before it: the next launch waits for this one alone)
  if (rows <= 0) {
    pdl_wait();
    if (meet) cooperative_groups::this_cluster().sync();
    return;
  }
  const int q0 = blockIdx.y * NC, nq = min(NC, nrhs - q0);
  const int gn = cplx || nq > GW ? 2 : 1;   // groups that hold columns
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int uwarp = __shfl_sync(0xffffffffu, warp, 0);   // (uniform)
  T* xq = x + q0;
  const int ABYTES = srows * OZ_S * TW_K * 2, ST = ABYTES + 2 * BG;   // (srows: of the launch)
  int* reb = reinterpret_cast<int*>(sm + (size_t)nst * ST + (TW_M - srows) * 64);   // stretch st, row i: st * 128 + i
  int* ceb = reb + nstr * TW_M;                                                    // stretch st, column q: st * NC + q
  int* kx = ceb + nstr * 2 * GW - K0;                                              // entry l of this CTA's K
  auto stretch = [&](int s) { return (s0 + s) / SX - s0 / SX; };
  const unsigned char* dig = nullptr;
  const int rows8 = (rows + 7) & ~7;
  if (CACHE) {
    dig = sl[blockIdx.z].dig[OP] + tw_tile_off(tile0, Kall);
    for (int st = 0; st < nstr && (s0 / SX + st) * SX < nsall; ++st)
      for (int i = tid; i < rows; i += TW_NT)
        reb[st * TW_M + i] = sl[blockIdx.z].eb[OP][(size_t)(s0 / SX + st) * M + i0 + i];
  } else {
    for (int i = tid; i < nstr * TW_M; i += TW_NT) reb[i] = 1;
    __syncthreads();
    tw_row_exps<OP, SX>(R, i0, rows, K0, K, reb);
  }
  for (int i = tid; i < nstr * NC; i += TW_NT) ceb[i] = 1;
  if (tid < 4) {
    mbar_init(&mb_mma[tid], 1);
    mbar_init(&mb_full[tid], 1);
    if (tid < 2) s_bad[tid] = 0;
  }
  if (warp == 0) tmem_alloc(&s_tmem, 16 * GW);
  // where the entries of the right-hand side's K rows sit in x
  for (int l = K0 + tid; l < K; l += TW_NT)
    kx[l] = OP == TW_DNF ? R.idxC[l] : OP == TW_UPW ? (l < k ? R.idxC[l] : R.idxR[l - k]) : R.idxR[l];
  const int pd = nst > 2 ? nst - 2 : 1;   // stages fetched ahead
  auto fetch_a = [&](int s) {   // (thread 0)
    const int b = s % nst;
    mbar_expect_tx(&mb_full[b], (uint32_t)(OZ_S * rows8 * 64));
    for (int p = 0; p < OZ_S; ++p)
      bulk_g2s(sm + (size_t)b * ST + p * srows * 64, dig + ((size_t)(s0 + s) * OZ_S + p) * rows8 * 64, rows8 * 64, &mb_full[b]);
  };
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  int fetched = 0;
  if (CACHE && tid == 0)
    for (; fetched < min(ns, pd); ++fetched) fetch_a(fetched);
  pdl_wait();
  {   // column exponents of each stretch of K: lanes over columns
    constexpr int PT = TW_NT / NC;
    const int q = tid % NC, part = tid / NC;
    if (q < nq)
      for (int sa = 0, st = 0; sa < ns; sa = (s0 + sa) / SX * SX + SX - s0, ++st) {
        const int l1 = min(K, ((s0 + sa) / SX * SX + SX) * KS);
        unsigned long long mk = 0;
#pragma unroll 8
        for (int l = (s0 + sa) * KS + part; l < l1; l += PT) mk = max(mk, tw_key(ld_l2(xq + kx[l] * ldx + q)));
        atomicMax(&ceb[st * NC + q], oz_emax_b(mk));
      }
  }
  __syncthreads();
  // outputs: row 32 (warp % 4) + lane, columns CT (warp / 4) .. of both groups
  const int row = 32 * (warp & 3) + lane, cg = CT * (warp >> 2);
  const bool live = 32 * (warp & 3) < rows;   // (warps past the tile's rows have no outputs)
  double acc[2][CT];
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int e = 0; e < CT; ++e) acc[g][e] = 0.0;
  // the group sums of one stretch of K, scaled, into acc
  auto gather = [&](int st, auto narrow) {
    constexpr int XB = cplx || decltype(narrow)::value ? 2 : 1;   // (|W| <= K 2^(53 + XB))
    if (!live) return;
    const uint32_t base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + cg;
    const int re = row < rows ? reb[st * TW_M + row] - 1022 : 0;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      if (g >= gn) break;
      uint32_t gr[OZ_S][CT];
#pragma unroll
      for (int u = 0; u < OZ_S; ++u) tmem_ldn<CT>(gr[u], base + (OZ_S * GW) * g + GW * u);
      tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < CT; ++e) {
        const int col = cplx ? cg + e : GW * g + cg + e;
        const int ce = ceb[st * NC + col];
        double v = oz_ldexp_int(tw_join<XB>(gr, e, narrow), re + (ce - 1022) - 53 - XB);
        if (ce == 2047) v = __longlong_as_double(0x7FF8000000000000ll);   // an infinity or a NaN in the column
        acc[g][e] = st > 0 ? acc[g][e] + v : v;
      }
    }
  };
  // the threads that cut columns: (column, group of eight entries, complex: part)
  const int tb = tid - (TW_NT - NC * 4);
  const int bq = tb & (NC - 1), bg = (tb / NC) & (cplx ? 1 : 3), bim = cplx ? tb / (2 * NC) : 0;
  double bv[8];
  auto load_b = [&](int s) {
    const double* xc = reinterpret_cast<const double*>(xq + bq) + bim;
    const int l0 = (s0 + s) * KS + bg * 8;
#pragma unroll
    for (int e = 0; e < 8; ++e) bv[e] = (bq < nq && l0 + e < K) ? __ldcg(xc + (cplx ? 2 : 1) * (kx[l0 + e] * ldx)) : 0.0;
  };
  if (tb >= 0) load_b(0);
  // A wait that runs out ends the CTA's work at the next block barrier.  Barrier s reads
  // flag s & 1, which is written before it and again only after barrier s + 1: every
  // thread leaves it with the same verdict.
  volatile int* bad = s_bad;
  auto wait_mma = [&](int s, int at) {   // the products of stage s are done (each thread polls); verdict at barrier `at`
    const bool done = mbar_wait(&mb_mma[s % nst], (s / nst) & 1, polls);
    if (!done) bad[at & 1] = 1;
    return done;
  };
  int ok = 1, issued = 0;   // (issued: stages whose products were issued, known to warp 0)
  for (int s = 0; s < ns; ++s) {
    const int b = s % nst;
    unsigned char* As = sm + (size_t)b * ST;
    unsigned char* Bs = As + ABYTES;
    const bool fresh = s == 0 || (s0 + s) % SX == 0;   // the group sums start over
    if (s >= nst) wait_mma(s - nst, s);           // the products that read this buffer
    if (CACHE && tid == 0 && fetched < ns && s + pd < ns) {
      if (s + pd < nst || wait_mma(s + pd - nst, s)) {
        fetch_a(fetched);
        ++fetched;
      }
    }
    if (fresh && s > 0) {   // the sums of the stretch of K before this stage
      wait_mma(s - 1, s);
      __syncwarp();
      tc_fence_after();
      gather(stretch(s - 1), std::integral_constant<bool, !cplx && SX <= TW_KN / TW_K>{});
      tc_fence_before();
    }
    if (!CACHE) tw_cut_a<OP>(R, i0, rows, K, s0 + s, reb + stretch(s) * TW_M, As, srows * 64);
    // columns: eight entries of K per thread, those of the next stage loaded meanwhile
    if (tb >= 0) {
      const int beb = ceb[stretch(s) * NC + bq];
      long long X[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(bv[e], beb);
      load_b(s + 1);
      if constexpr (!cplx) {
        tw_put8(X, Bs + (bq / GW) * BG + tw_at(bq % GW, bg), GW * 64, 0u);
      } else if (!bim) {   // real parts: real outputs at the first half of the stage, imaginary ones at the second
        tw_put8(X, Bs + tw_at(bq, bg), GW * 64, 0u);
        tw_put8(X, Bs + BG + tw_at(bq, 2 + bg), GW * 64, 0u);
      } else {
        tw_put8(X, Bs + tw_at(bq, 2 + bg), GW * 64, 0x80008000u);
        tw_put8(X, Bs + BG + tw_at(bq, bg), GW * 64, 0u);
      }
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    ok = !bad[s & 1];
    if (!ok) break;
    if (uwarp == 0) {
      // (a copy that never lands leaves the stage without products)
      const bool got = __all_sync(0xffffffffu, !CACHE || mbar_wait(&mb_full[b], (s / nst) & 1, polls));
      if (!got) bad[(s + 1) & 1] = 1;
      issued += got;
      tc_fence_after();
      const uint32_t lead = got ? elect_one() : 0u;
      const uint32_t al = umma_lo(smem_u32(As)), bl = umma_lo(smem_u32(Bs));
#pragma unroll
      for (int h = 0; h < TW_K / 16; ++h)
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          if (g >= gn) break;
#pragma unroll
          for (int p = 0; p < OZ_S; ++p)
            umma_bf16_w(tmem + OZ_S * GW * g + GW * p, al + (uint32_t)(p * srows * 4 + h * 16),
                        bl + (uint32_t)(g * (BG / 16) + h * 16), umma_idesc_bf16(TW_M, GW * (OZ_S - p)),
                        (fresh && h == 0 && p == 0) ? 0u : 1u, lead);
        }
      umma_commit_w(&mb_mma[b], lead);
      __syncwarp();
    }
  }
  __syncthreads();
  ok = ok && !bad[ns & 1];
  if (ok && ns > 0) wait_mma(ns - 1, ns + 1);
  __syncthreads();
  ok = ok && !bad[(ns + 1) & 1];
  tc_fence_after();
  if (ok) {
    if (ns > 0) {
      const int st = stretch(ns - 1);
      if ((s0 + ns - 1) % SX < TW_KN / TW_K || ns <= TW_KN / TW_K) gather(st, std::true_type{});
      else gather(st, std::false_type{});
    }
    // through shared memory (the stages are free), so that a warp handles the columns
    // of one point side by side
    T* tile = reinterpret_cast<T*>(sm);
    if (live) {
#pragma unroll
      for (int e = 0; e < CT; ++e) {
        if constexpr (cplx) {
          tile[row * LDO + cg + e] = zd{acc[0][e], acc[1][e]};
        } else {
          tile[row * LDO + cg + e] = acc[0][e];
          tile[row * LDO + GW + cg + e] = acc[1][e];
        }
      }
    }
  } else if (tid == 0) {
    set_error(err, RSS_ETIMEOUT);
    // what is in flight (products, copies) ends before the buffers and the tensor memory go
    for (int q = max(0, issued - nst); q < issued; ++q) mbar_wait(&mb_mma[q % nst], (q / nst) & 1, TW_DRAIN);
    if (CACHE)
      for (int q = max(0, fetched - nst); q < fetched; ++q) mbar_wait(&mb_full[q % nst], (q / nst) & 1, TW_DRAIN);
  }
  if (spl > 1 || meet) cooperative_groups::this_cluster().sync();
  else __syncthreads();
  if (ok) {
    // (of a cluster: each CTA the sums of a share of the rows, parts added in order)
    const T* tile = reinterpret_cast<const T*>(sm);
    const int ra = rows * rank / spl, rb = rows * (rank + 1) / spl;
    constexpr int RPW = 32 / (NC < 32 ? NC : 32);   // rows of a warp at a time
    for (int i = ra + warp * RPW + lane / NC; i < rb; i += TW_NT / 32 * RPW) {
      const int o = i0 + i;
      const int64_t gi = OP == TW_UPE ? R.idxC[o] : OP == TW_DNW ? (o < k ? R.idxC[o] : R.idxR[o - k]) : R.idxR[o];
      const bool keep = OP == TW_UPE || OP == TW_DNF || (OP == TW_DNW && o < k);
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 32) {
        const int q = c0 + (lane & (NC - 1));
        if (q < nq) {
          T v = tile[i * LDO + q];
          if (spl > 1) {
            v = zero<T>();
            for (int j = 0; j < spl; ++j) v = v + cooperative_groups::this_cluster().map_shared_rank(tile, j)[i * LDO + q];
          }
          T* g = xq + gi * ldx + q;
          *g = !keep ? v : (OP == TW_UPE || OP == TW_DNF) ? ld_l2(g) - v : ld_l2(g) + v;
        }
      }
    }
  }
  if (spl > 1) cooperative_groups::this_cluster().sync();   // (the parts have been read)
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, 16 * GW);
}
