// E = A_CB W_E and F^T = A_BC^T W_F (Eqs. 7, 8) as exact digit products on tcgen05, for
// one row tile of C per CTA.  The columns of W are cut into digits once per box
// (k_ep_cut_w), in the layout of the products' stages; the rows of A by the CTA itself.
// Symmetric A: A_BC^T = A_CB, so the tile is cut once for the columns of [W_E W_F];
// else a CTA takes one of the two matrices.  Complex: K doubled, [A_re A_im] times
// [W_re; -W_im] and [W_im; W_re] (see sweep_tc.cuh), the real and imaginary parts of 32
// columns to a pass.
//
// Sixteen warps cut the rows, join the group sums into E and F^T and at last cut the
// rows of E and F^T for the Schur update; one more warp copies the stages of W and
// issues the products.  Real boxes (n <= 128) keep the tile's digits in shared memory
// over all columns, and the group sums of one pass of 32 columns are joined from one
// half of tensor memory while the products of the next fill the other.  Complex rows
// are cut again for each pass.
// A class of few boxes splits the passes over CTAs.
//
// Real: the same integers, so the same E and F^T, as the digits of whole rows and
// columns give in any other order.  Complex: 64 entries of K at a time under scales of
// their own, joined with two more bits and added in FP64: against long double on boxes
// of 16 to 256 points an error of 0.47 to 0.9 times that of 32 entries at a time
// joined at 53 bits, and 0.3 to 0.9 times that of FP64.
//
// Bound by latency: one CTA of 17 warps on an SM gathers rows of A, cuts and joins; in the
// first leaf class (512^2 real, 256^2 complex) the schedulers issue in 28 to 29 % of their
// cycles, the tensor pipe is busy for 9 to 10 % (70 clocks a product), ALU 26 to 29 %.
// Panels of a factorization against products on mma.sync with the rows and columns cut
// per 64-row CTA: Laplace 1024^2 34.3 -> 24.8 ms, Helmholtz 256^2 22.1 -> 9.3 ms (of which
// cutting W 2.0 and 0.6); a coarse complex class of one or two boxes 530 -> 100 us.
constexpr int EP_W = 16, EP_NT = 32 * (EP_W + 1);
constexpr int EP_GB = OZ_S * 32 * TW_K * 2;   // bytes of a stage of 32 columns of W (one part)

template <typename T> struct EpArgs {
  LevelDev<T> L;
  const BoxRec<T>* recs;
  const int* cls_idx;
  const int* perm_in;
  unsigned char* ws;   // per record: digits of W, exponents of its columns
  size_t slot, o_ew;
  int sets;            // 1: A is symmetric, one list of 2 r columns; 2: two lists of r
  int ns, ng, nstr;    // of the class: stages of K, groups of 32 columns of a list, stretches of K
  int rows, ad, wd;    // rows of a tile; stages of A and of W in shared memory
  int psplit;          // CTAs that share the passes of a tile
  int spn;             // entries of the pivot order kept in shared memory
  int staged;          // complex: the slices in the layout of k_schur_z
  int* err;
  int polls;           // of the waits that wait_polls governs
};
template <typename T> __host__ __device__ constexpr int ep_ks() { return sizeof(T) == sizeof(double) ? TW_K : TW_K / 2; }
// stages of K that share scales and sums
template <typename T> __host__ __device__ constexpr int ep_smax() { return sizeof(T) == sizeof(double) ? TW_KX / TW_K : 4; }
template <typename T> __host__ __device__ constexpr int ep_parts() { return sizeof(T) == sizeof(double) ? 1 : 2; }
// columns of group g of a list of nc, rounded up to what a product takes
__host__ __device__ inline int ep_cols(int nc, int g) { return nc - 32 * g > 16 ? 32 : 16; }

__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(mbar)) : "memory");
}

// 32 columns of a list: exponents, then digits, the stage s of group g at
// ((set * ng + g) * ns + s) * parts * EP_GB
constexpr int EP_WT = 512;
template <typename T> __global__ void __launch_bounds__(EP_WT) k_ep_cut_w(EpArgs<T> a) {
  constexpr bool cplx = sizeof(T) != sizeof(double);
  constexpr int PARTS = ep_parts<T>();
  const BoxRec<T> R = a.recs[blockIdx.z];
  const int r = R.r, n = R.k + R.r, set = blockIdx.y, g = blockIdx.x, nc = a.sets == 1 ? 2 * r : r;
  if (!R.ozp || 32 * g >= nc) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cw = ep_cols(nc, g);
  auto column = [&](int j) -> const T* {   // column j of the group (null past the list)
    const int cc = 32 * g + j;
    if (cc >= nc) return nullptr;
    return a.sets == 1 && cc >= r ? R.Wf + (size_t)(cc - r) * n : (set ? R.Wf : R.We) + (size_t)cc * n;
  };
  unsigned char* slot = a.ws + (size_t)blockIdx.z * a.slot;
  constexpr int SMAX = ep_smax<T>(), KX = SMAX * ep_ks<T>();   // a stretch
  int* ew = reinterpret_cast<int*>(slot + a.o_ew) + (size_t)(set * a.ng + g) * a.nstr * 32;
  for (int j = warp; j < cw; j += EP_WT / 32) {
    const T* w = column(j);
    for (int l0 = 0; l0 < n; l0 += KX) {
      unsigned long long mk = 0;
      if (w)
        for (int l = l0 + lane; l < min(n, l0 + KX); l += 32) mk = max(mk, tw_key(w[l]));
      mk = shfl_max_u64(mk, 32);
      if (lane == 0) ew[l0 / KX * 32 + j] = oz_emax_b(mk);
    }
  }
  __syncthreads();
  const int ns = (n + ep_ks<T>() - 1) / ep_ks<T>(), t = tid & 127, j = cplx ? (t >> 1) & 31 : t >> 2;
  if (j >= cw) return;
  const T* w = column(j);
  unsigned char* dst = slot + ((size_t)set * a.ng + g) * a.ns * (PARTS * EP_GB);
  for (int s = tid >> 7; s < ns; s += EP_WT / 128) {
    unsigned char* d = dst + (size_t)s * (PARTS * EP_GB);
    const int eb = ew[s / SMAX * 32 + j];
    long long X[8];
    if constexpr (!cplx) {
      const int kg = t & 3, l0 = s * 32 + kg * 8;
#pragma unroll
      for (int e = 0; e < 8; ++e) X[e] = (w && l0 + e < n) ? oz_scaled_int(w[l0 + e], eb) : 0;
      tw_put8(X, d + tw_at(j, kg), cw * 64, 0u);
    } else {
      const int hh = t & 1, im = t >> 6, l0 = s * 16 + hh * 8;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        double v = 0.0;
        if (w && l0 + e < n) v = im ? w[l0 + e].y : w[l0 + e].x;
        X[e] = oz_scaled_int(v, eb);
      }
      const int part = OZ_S * cw * 64;   // the imaginary outputs' columns
      if (!im) {
        tw_put8(X, d + tw_at(j, hh), cw * 64, 0u);
        tw_put8(X, d + part + tw_at(j, 2 + hh), cw * 64, 0u);
      } else {
        tw_put8(X, d + tw_at(j, 2 + hh), cw * 64, 0x80008000u);
        tw_put8(X, d + part + tw_at(j, hh), cw * 64, 0u);
      }
    }
  }
}

// Digit slices of rows i0 .. of E (or F^T) for the Schur update: row i at
// sl + i * S * kp, slice p at + p * kp (complex: 8 real slices, then 8 imaginary).  staged
// (complex): in the layout of k_schur_z, slice p of stage s at (s * 8 + p) * c8 * 64
// (c8: c rounded up to 8), rows as in a stage; of F^T two such forms, for real and for
// imaginary parts.  Four threads per row; scr: 512 keys, reb: 128 ints of shared memory.
// 512 threads.
template <typename T>
__device__ void ep_slices(const BoxRec<T>& R, int which, int i0, int rows, int staged, unsigned long long* scr, int* reb) {
  constexpr bool cplx = sizeof(T) != sizeof(double);
  const int c = R.c, r = R.r, kp = R.kp;
  const T* src = (which ? R.Ft : R.E) + i0;
  uint16_t* dst = (which ? R.Fsl : R.Esl) + (size_t)i0 * (cplx ? 2 : 1) * OZ_S * kp;
  int* ex = (which ? R.Fexp : R.Eexp) + i0;
  const int tid = threadIdx.x, i = tid % TW_M, part = tid / TW_M;
  const bool work = part < 4, on = work && i < rows;
  unsigned long long mk = 0;
  if (on) {
#pragma unroll 4
    for (int l = part; l < r; l += 4) mk = max(mk, tw_key(src[i + (size_t)l * c]));
  }
  if (work) scr[tid] = mk;
  __syncthreads();
  if (tid < TW_M) {
#pragma unroll
    for (int p = 1; p < 4; ++p) mk = max(mk, scr[tid + TW_M * p]);
    reb[tid] = oz_emax_b(mk);
    if (on) ex[tid] = mk ? reb[tid] - 1022 : 0;
  }
  __syncthreads();
  if (!on) return;
  const int eb = reb[i];
  if constexpr (cplx) {
    if (staged) {
      const size_t c8 = (size_t)((c + 7) & ~7) * 64, form = (size_t)((r + 15) / 16) * OZ_S * c8;
      unsigned char* b = reinterpret_cast<unsigned char*>(which ? R.Fsl : R.Esl);
      for (int q = part; q < (r + 15) / 16 * 2; q += 4) {   // stage q / 2, entries 8 (q % 2) ..
        T v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = q * 8 + e < r ? src[i + (size_t)(q * 8 + e) * c] : zero<T>();
        unsigned char* d = b + (size_t)(q / 2) * OZ_S * c8;
        const int at0 = tw_at(i0 + i, q % 2), at1 = tw_at(i0 + i, 2 + q % 2);
        long long X[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].x, eb);
        tw_put8(X, d + at0, c8, 0u);
        if (which) tw_put8(X, d + form + at1, c8, 0u);
#pragma unroll
        for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].y, eb);
        tw_put8(X, d + at1, c8, which ? 0x80008000u : 0u);
        if (which) tw_put8(X, d + form + at0, c8, 0u);
      }
      return;
    }
  }
  unsigned char* d = reinterpret_cast<unsigned char*>(dst + (size_t)i * (cplx ? 2 : 1) * OZ_S * kp);
  for (int kg = part; kg < kp / 8; kg += 4) {
    T v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = kg * 8 + e < r ? src[i + (size_t)(kg * 8 + e) * c] : zero<T>();
    long long X[8];
    if constexpr (!cplx) {
#pragma unroll
      for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e], eb);
      tw_put8(X, d + kg * 16, (size_t)kp * 2, 0u);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].x, eb);
      tw_put8(X, d + kg * 16, (size_t)kp * 2, 0u);
#pragma unroll
      for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].y, eb);
      tw_put8(X, d + (size_t)OZ_S * kp * 2 + kg * 16, (size_t)kp * 2, 0u);
    }
  }
}

// the slices alone, where the passes of a tile are shared by CTAs
template <typename T> __global__ void __launch_bounds__(512) k_ep_slices(const BoxRec<T>* __restrict__ recs, int staged) {
  __shared__ unsigned long long scr[512];
  __shared__ int reb[TW_M];
  const BoxRec<T> R = recs[blockIdx.z];
  const int i0 = blockIdx.x * TW_M;
  if (!R.ozp || i0 >= R.c || R.Esl == nullptr) return;
  ep_slices(R, blockIdx.y, i0, min(TW_M, R.c - i0), staged, scr, reb);
}

template <typename T> __global__ void __launch_bounds__(EP_NT, 1) k_ep(EpArgs<T> a) {
  extern __shared__ __align__(1024) unsigned char sm[];
  constexpr bool cplx = sizeof(T) != sizeof(double);
  constexpr int PARTS = ep_parts<T>(), NBUF = cplx ? 1 : 2, KS = ep_ks<T>(), G = KS / 8;
  constexpr int SMAX = ep_smax<T>();
  __shared__ __align__(8) uint64_t afull[4], afree[4], wfull[4], wfree[4], tdone[2], tfree[2], drained;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_ok;
  __shared__ long long base[TW_M];
  const BoxRec<T> R = a.recs[blockIdx.z];
  const LevelDev<T>& L = a.L;
  const int c = R.c, r = R.r, n = R.k + r, i0 = blockIdx.x * a.rows, rows = min(a.rows, c - i0);
  const int set = blockIdx.y % a.sets, p0 = blockIdx.y / a.sets;
  const int nc = a.sets == 1 ? 2 * r : r, np = (nc + 31) / 32;   // columns, passes
  if (!R.ozp || rows <= 0 || p0 >= np) return;
  const int ns = (n + KS - 1) / KS, ad = a.ad, wd = a.wd, np_mine = (np - p0 + a.psplit - 1) / a.psplit;
  const bool resident = ns <= ad;
  const int ABYTES = a.rows * OZ_S * TW_K * 2;
  // (the products of a short tile read, and ignore, up to 128 rows past each slice)
  unsigned char* wsm = sm + (size_t)ad * ABYTES;
  int* spsm = reinterpret_cast<int*>(wsm + (size_t)wd * PARTS * EP_GB);
  int* reb = spsm + a.spn;   // of stretch st, row i: at st * 128 + i
  unsigned long long* scr = reinterpret_cast<unsigned long long*>(sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int nmax = L.nmax, g = L.g, B = R.box;
  const unsigned char* slot = a.ws + (size_t)blockIdx.z * a.slot;
  {
    const long long nn = (long long)nmax * nmax;
    const int* perm = a.perm_in + (size_t)a.cls_idx[blockIdx.z] * nmax;
    if (n <= a.spn)
      for (int i = tid; i < n; i += EP_NT) spsm[i] = perm[i];
    if (tid < rows) {
      const int cm = R.cmap[i0 + tid], s = cm >> 16, pos = cm & 0xffff;
      const int u = nbr_box(B, g, s % 3 - 1, s / 3 - 1);
      base[tid] = set == 0 ? ((long long)u * 25 + off_index(u, B, g)) * nn + pos
                           : ((long long)B * 25 + off_index(B, u, g)) * nn + (long long)pos * nmax;
    }
    if (tid < 4) {
      mbar_init(&afull[tid], cplx ? EP_W / 2 : EP_W);
      mbar_init(&afree[tid], 1);
      mbar_init(&wfull[tid], 1);
      mbar_init(&wfree[tid], 1);
      if (tid < 2) {
        mbar_init(&tdone[tid], 1);
        mbar_init(&tfree[tid], EP_W);
      }
      if (tid == 0) {
        mbar_init(&drained, 1);
        s_ok = 1;
      }
    }
    if (warp == EP_W) tmem_alloc(&s_tmem, 512);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int* sp = n <= a.spn ? spsm : a.perm_in + (size_t)a.cls_idx[blockIdx.z] * nmax;
  const long long ls = set == 0 ? nmax : 1;
  // the rows' exponents over the whole K; real: the first two stages' entries stay in registers
  const int ci = tid % TW_M, cq = tid / TW_M;   // row, quarter
  const T* arow = warp < EP_W && ci < rows ? L.blk + base[ci] : nullptr;
  constexpr int KEEP = cplx ? 1 : 2;
  T keep[KEEP][8];
  {
    unsigned long long mk = 0;
    if constexpr (!cplx) {
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int l = s * 32 + cq * 8 + e;
          keep[s][e] = arow && l < n ? arow[sp[l] * ls] : 0.0;
        }
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int e = 0; e < 8; ++e) mk = max(mk, tw_key(keep[s][e]));
      if (arow)
        for (int l0 = 64 + cq * 8; l0 < n; l0 += 32)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (l0 + e < n) mk = max(mk, tw_key(arow[sp[l0 + e] * ls]));
    }
    for (int st = 0; st * SMAX < ns; ++st) {
      if (cplx && arow) {
        mk = 0;
#pragma unroll 8
        for (int l = st * SMAX * KS + cq; l < min(n, (st + 1) * SMAX * KS); l += 4) mk = max(mk, tw_key(arow[sp[l] * ls]));
      }
      if (warp < EP_W) scr[tid] = mk;
      __syncthreads();
      if (tid < TW_M) {
#pragma unroll
        for (int p = 1; p < 4; ++p) mk = max(mk, scr[tid + p * TW_M]);
        reb[st * TW_M + tid] = oz_emax_b(mk);
      }
      __syncthreads();
    }
  }
  const int srows8 = (rows + 7) & ~7;
  if (warp == EP_W) {
    // ---- stages of W by bulk copies, products
    const uint32_t lead = elect_one();
    const int nu = np_mine * ns;
    int loaded = 0;
    auto load_w = [&]() {
      const int p = p0 + a.psplit * (loaded / ns), s = loaded % ns, b = loaded % wd;
      const uint32_t bytes = (uint32_t)(PARTS * OZ_S * 64 * ep_cols(nc, p));
      if (lead) {
        mbar_expect_tx(&wfull[b], bytes);
        bulk_g2s(wsm + (size_t)b * PARTS * EP_GB, slot + (((size_t)set * a.ng + p) * a.ns + s) * (PARTS * EP_GB), bytes,
                 &wfull[b]);
      }
      ++loaded;
      __syncwarp();
    };
    while (loaded < min(wd, nu)) load_w();
    int t = 0, seq = 0, u = 0;   // stages of A, joins, stages of W
    // (a.polls governs the first wait; constants in the issuing loop, as in k_schur_z)
    bool ok = __all_sync(0xffffffffu, mbar_wait(&wfull[0], 0, a.polls));
    for (int q = 0; q < np_mine && ok; ++q) {
      const int cw = ep_cols(nc, p0 + a.psplit * q);
      for (int s = 0; s < ns && ok; ++s, ++u) {
        const bool fresh = s % SMAX == 0;
        const int ab = resident ? s : t % ad, wb = u % wd, h = seq % NBUF;
        ok = mbar_wait(&wfull[wb], (u / wd) & 1, TW_POLLS);
        if (ok && (!resident || q == 0)) ok = mbar_wait(&afull[ab], resident ? 0 : (t / ad) & 1, TW_POLLS);
        if (ok && fresh && seq >= NBUF) ok = mbar_wait(&tfree[h], (seq / NBUF - 1) & 1, TW_POLLS);
        ok = __all_sync(0xffffffffu, ok) && s_ok;
        if (!ok) break;
        tc_fence_after();
        const uint32_t al = umma_lo(smem_u32(sm + (size_t)ab * ABYTES));
        const uint32_t bl = umma_lo(smem_u32(wsm + (size_t)wb * PARTS * EP_GB));
#pragma unroll
        for (int hk = 0; hk < TW_K / 16; ++hk)
#pragma unroll
          for (int part = 0; part < PARTS; ++part)
#pragma unroll
            for (int p = 0; p < OZ_S; ++p)
              umma_bf16_w(tmem + 256 * (cplx ? part : h) + cw * p, al + (uint32_t)(p * a.rows * 4 + hk * 16),
                          bl + (uint32_t)(part * OZ_S * cw * 4 + hk * 16), umma_idesc_bf16(TW_M, cw * (OZ_S - p)),
                          (fresh && hk == 0 && p == 0) ? 0u : 1u, lead);
        umma_commit_w(&wfree[wb], lead);
        if (!resident) umma_commit_w(&afree[ab], lead);
        if (s % SMAX == SMAX - 1 || s == ns - 1) {
          umma_commit_w(&tdone[h], lead);
          ++seq;
        }
        ++t;
        __syncwarp();
        if (u > 0 && loaded < nu) {   // the buffer of the stage before
          ok = __all_sync(0xffffffffu, mbar_wait(&wfree[(u - 1) % wd], ((u - 1) / wd) & 1, TW_POLLS));
          if (!ok) break;
          load_w();
        }
      }
    }
    if (!ok) s_ok = 0;
    // everything issued has ended before the buffers and the tensor memory go
    umma_commit_w(&drained, lead);
    __syncwarp();
    mbar_wait(&drained, 0, ok ? TW_POLLS : TW_DRAIN);
    if (!ok)
      for (int v = max(0, loaded - wd); v < loaded; ++v) mbar_wait(&wfull[v % wd], (v / wd) & 1, TW_DRAIN);
  } else {
    // ---- digits of the rows, join of the group sums
    const int row = 32 * (warp & 3) + lane, cg = 8 * (warp >> 2);
    bool ok = true;
    int t = 0, seq = 0;
    double acc[PARTS][8];
    const int* wexp = reinterpret_cast<const int*>(slot + a.o_ew) + (size_t)set * a.ng * a.nstr * 32;
    constexpr int XB = cplx ? 2 : 0;   // (|W| <= K 2^(53 + XB), K of a stretch)
    // sums of join `sq`: pass p, the stages sa .. sb of its K
    auto join = [&](int sq, int p, int sa, int sb) {
      const int h = sq % NBUF, cw = ep_cols(nc, p);
      ok = ok && mbar_wait(&tdone[h], (sq / NBUF) & 1, a.polls);
      ok = __all_sync(0xffffffffu, ok) && s_ok;
      if (!ok) return;
      tc_fence_after();
      const bool live = cg < cw && 32 * (warp & 3) < rows;
      const uint32_t tb = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + cg;
      const int st = sa / SMAX, er = live ? reb[st * TW_M + row] - 2044 - 53 - XB : 0;
      const int* we = wexp + (p * a.nstr + st) * 32 + cg;
      // four columns at a time, for the registers' sake
#pragma unroll
      for (int c0 = 0; c0 < 8; c0 += 4)
#pragma unroll
        for (int part = 0; part < PARTS; ++part) {
          uint32_t gr[OZ_S][4];
          if (live) {
#pragma unroll
            for (int u = 0; u < OZ_S; ++u) tmem_ldn<4>(gr[u], tb + 256 * (cplx ? part : h) + cw * u + c0);
            tmem_ld_wait();
          }
          if (c0 == 4 && part == PARTS - 1) {   // all read: the products may overwrite them
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tfree[h]);
          }
          if (live) {
            auto put = [&](auto narrow) {
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const double v = oz_ldexp_int(tw_join<XB>(gr, e, narrow), er + __ldg(we + c0 + e));
                acc[part][c0 + e] = sa > 0 ? acc[part][c0 + e] + v : v;
              }
            };
            if (sb - sa <= TW_KN / TW_K) put(std::true_type{});
            else put(std::false_type{});
          }
        }
      if (live && sb == ns && row < rows) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int cc = 32 * p + cg + e;
          if (cc < nc) {
            T* m = a.sets == 1 ? (cc < r ? R.E : R.Ft) : set ? R.Ft : R.E;
            T* o = m + (size_t)(a.sets == 1 && cc >= r ? cc - r : cc) * c + i0 + row;
            if constexpr (cplx) *o = zd{acc[0][e], acc[1][e]};
            else *o = acc[0][e];
          }
        }
      }
    };
    for (int q = 0; q < np_mine && ok; ++q) {
      const int p = p0 + a.psplit * q;
      for (int sa = 0; sa < ns && ok; sa += SMAX, ++seq) {
        const int sb = min(ns, sa + SMAX);
        if (!resident || q == 0)
          for (int s = sa; s < sb && ok; ++s, ++t) {
            const int ab = resident ? s : t % ad;
            if (cplx && (t & 1) != cq >> 1) continue;   // complex: half of the warps a stage
            const int kg = cplx ? cq & 1 : cq, l0 = s * KS + kg * 8;
            T v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              if (!cplx && s < 2) v[e] = s == 0 ? keep[0][e] : keep[KEEP - 1][e];
              else v[e] = arow && l0 + e < n ? arow[sp[l0 + e] * ls] : zero<T>();
            }
            if (!resident && t >= ad) ok = mbar_wait(&afree[ab], (t / ad - 1) & 1, a.polls);
            ok = __all_sync(0xffffffffu, ok) && s_ok;
            if (!ok) break;
            if (ci < srows8) {
              const int eb = ci < rows ? reb[s / SMAX * TW_M + ci] : 1;
              unsigned char* d = sm + (size_t)ab * ABYTES;
              long long X[8];
              if constexpr (!cplx) {
#pragma unroll
                for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e], eb);
                tw_put8(X, d + tw_at(ci, kg), (size_t)a.rows * 64, 0u);
              } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].x, eb);
                tw_put8(X, d + tw_at(ci, kg), (size_t)a.rows * 64, 0u);
#pragma unroll
                for (int e = 0; e < 8; ++e) X[e] = oz_scaled_int(v[e].y, eb);
                tw_put8(X, d + tw_at(ci, 2 + kg), (size_t)a.rows * 64, 0u);
              }
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull[ab]);
          }
        if (!ok) break;
        if (NBUF == 1) join(seq, p, sa, sb);
        else if (seq > 0) join(seq - 1, p - a.psplit, 0, ns);   // (real: one stretch a pass)
      }
    }
    if (NBUF == 2 && ok) join(seq - 1, p0 + a.psplit * (np_mine - 1), 0, ns);
    if (!ok) s_ok = 0;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == EP_W) tmem_free(tmem, 512);
  if (!s_ok) {
    if (tid == 0) set_error(a.err, RSS_ETIMEOUT);
    return;
  }
  if (a.psplit == 1 && R.Esl != nullptr) {
    const int last = a.sets == 1 ? 1 : set;
    for (int w = a.sets == 1 ? 0 : set; w <= last; ++w) {
      ep_slices(R, w, i0, rows, a.staged, scr, reb);
      __syncthreads();
    }
  }
}
