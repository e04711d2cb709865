// The Schur update A_CC -= E F of complex factors on tcgen05: K doubled as in
// elim_panels.cuh, [E_re E_im] times [F_re; -F_im] and [F_im; F_re], exact group sums in
// tensor memory (eight for the real, eight for the imaginary parts of 32 columns), one
// int64 per part and output.  One CTA walks the 32-column tiles of a block of 128
// rows (96 where r > 32, for room to copy columns well ahead of their products):
// sixteen warps join the sums into A_CC, one more copies stages and issues products.
// ep_slices writes the digits in the stages' layout, F's in both forms, so that they come
// by bulk copies; those of the block's rows stay in shared memory where they fit (r <= 48).
//
// Symmetric A with a real T (X_RC = X_CR^T, so E F is symmetric to rounding): only the
// entries j >= i are formed, and stored to A_CC(j, i) as well; the row blocks with the
// most tiles of every box start first (60.2 -> 59.5 ms at Helmholtz 256^2).
//
// Bound by the entries of A_CC (DRAM 39 % of its peak, warps waiting for global loads) and
// the products (tensor pipe 32 %: 96 a tile at r = 48, about 70 clocks each); the join of
// the sums cannot overlap them (a tile's sums fill tensor memory), the FP64 arithmetic (a
// conversion and a subtraction take 32 clocks a warp) runs beside the next products.
// One tile per CTA, staged by cp.async and never overlapped, took 10.9 ms a
// factorization at Helmholtz 256^2 and 32 ms at Lippmann-Schwinger 512^2; now 7.6 ms and
// about 15 ms.
constexpr int SZ_AST = OZ_S * TW_K * 2;          // bytes of a stage per row
constexpr int SZ_BP = EP_GB;                     // ... of one form of 32 columns (16 KB)
constexpr int SZ_NS = 12;                        // stages whose sums stay exact: r <= 192

__global__ void __launch_bounds__(EP_NT, 1) k_schur_z(LevelDev<zd> L, const BoxRec<zd>* __restrict__ recs, int trows, int ad, int nb,
                                                      int csplit, int sym, int* err, int polls) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t afull[4], afree[4], bfull[8], bfree[8], tdone, tfree, drained;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_ok;
  const BoxRec<zd> R = recs[blockIdx.x];
  const int c = R.c, r = R.r, i0 = blockIdx.z * trows, rows = min(trows, c - i0), c8 = (c + 7) & ~7;
  const int ns = (r + 15) / 16;
  // tiles of this CTA: t0, t0 + csplit, ..
  const int tend = (c + 31) / 32, t0 = (sym ? i0 / 32 : 0) + blockIdx.y;
  if (rows <= 0 || r == 0 || t0 >= tend) return;
  const int nt = (tend - t0 + csplit - 1) / csplit;
  const bool resident = ns <= ad;
  // (the products of a short tile read, and ignore, up to 128 rows past each slice)
  unsigned char* bsm = sm + (size_t)ad * trows * SZ_AST;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  if (tid == 0) {
    for (int s = 0; s < 4; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&afree[s], 1);
    }
    for (int s = 0; s < 8; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bfree[s], 1);
    }
    mbar_init(&tdone, 1);
    mbar_init(&tfree, EP_W);
    mbar_init(&drained, 1);
    s_ok = 1;
  }
  if (warp == EP_W) tmem_alloc(&s_tmem, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  if (warp == EP_W) {
    const uint32_t lead = elect_one();
    const unsigned char* E = reinterpret_cast<const unsigned char*>(R.Esl);
    const unsigned char* F = reinterpret_cast<const unsigned char*>(R.Fsl);
    const uint32_t arow = (uint32_t)min(trows, c8 - i0) * 64;
    const int na = resident ? ns : nt * ns, nv = 2 * nt * ns;   // stages of rows, pieces of columns
    int la = 0, lb = 0;
    auto load_a = [&]() {
      const int s = la % ns, b = resident ? s : la % ad;
      if (lead) {
        mbar_expect_tx(&afull[b], OZ_S * arow);
        for (int p = 0; p < OZ_S; ++p)
          bulk_g2s(sm + (size_t)b * trows * SZ_AST + p * trows * 64, E + ((size_t)s * OZ_S + p) * c8 * 64 + (size_t)i0 * 64, arow,
                   &afull[b]);
      }
      ++la;
      __syncwarp();
    };
    auto load_b = [&]() {
      const int q = lb / (2 * ns), s = lb / 2 % ns, part = lb & 1, b = lb % nb, j0 = 32 * (t0 + q * csplit);
      const uint32_t bytes = (uint32_t)min(32, c8 - j0) * 64;
      if (lead) {
        mbar_expect_tx(&bfull[b], OZ_S * bytes);
        for (int p = 0; p < OZ_S; ++p)
          bulk_g2s(bsm + (size_t)b * SZ_BP + p * 32 * 64,
                   F + (((size_t)part * ns + s) * OZ_S + p) * c8 * 64 + (size_t)j0 * 64, bytes, &bfull[b]);
      }
      ++lb;
      __syncwarp();
    };
    while (la < min(na, ad)) load_a();
    while (lb < min(nv, nb)) load_b();
    // (`polls` governs the first wait; the limits of the others are constants, which keeps
    // the issuing loop on uniform registers: 7.3 -> 6.9 ms, Helmholtz 256^2)
    bool ok = __all_sync(0xffffffffu, mbar_wait(&bfull[0], 0, polls));
    int t = 0, v = 0;
    for (int q = 0; q < nt && ok; ++q)
      for (int s = 0; s < ns && ok; ++s, ++t) {
        const int ab = resident ? s : t % ad;
        if (!resident || q == 0) ok = mbar_wait(&afull[ab], resident ? 0 : (t / ad) & 1, TW_POLLS);
        if (ok && s == 0 && q > 0) ok = mbar_wait(&tfree, (q - 1) & 1, TW_POLLS);
        const uint32_t al = umma_lo(smem_u32(sm + (size_t)ab * trows * SZ_AST));
#pragma unroll
        for (int part = 0; part < 2; ++part, ++v) {
          if (ok) ok = mbar_wait(&bfull[v % nb], (v / nb) & 1, TW_POLLS);
          ok = __all_sync(0xffffffffu, ok) && s_ok;
          if (!ok) break;
          tc_fence_after();
          const uint32_t bl = umma_lo(smem_u32(bsm + (size_t)(v % nb) * SZ_BP));
#pragma unroll
          for (int hk = 0; hk < TW_K / 16; ++hk)
#pragma unroll
            for (int p = 0; p < OZ_S; ++p)
              umma_bf16_w(tmem + 256 * part + 32 * p, al + (uint32_t)(p * trows * 4 + hk * 16), bl + (uint32_t)(hk * 16),
                          umma_idesc_bf16(TW_M, 32 * (OZ_S - p)), (s == 0 && hk == 0 && p == 0) ? 0u : 1u, lead);
          umma_commit_w(&bfree[v % nb], lead);
          if (part == 1 && !resident) umma_commit_w(&afree[ab], lead);
          if (part == 1 && s == ns - 1) umma_commit_w(&tdone, lead);
          __syncwarp();
          // the buffers of the piece and of the stage before
          if (v > 0 && lb < nv) {
            ok = __all_sync(0xffffffffu, mbar_wait(&bfree[(v - 1) % nb], ((v - 1) / nb) & 1, TW_POLLS));
            if (!ok) break;
            load_b();
          }
          if (part == 0 && t > 0 && la < na && !resident) {
            ok = __all_sync(0xffffffffu, mbar_wait(&afree[(t - 1) % ad], ((t - 1) / ad) & 1, TW_POLLS));
            if (!ok) break;
            load_a();
          }
        }
      }
    if (!ok) s_ok = 0;
    umma_commit_w(&drained, lead);
    __syncwarp();
    mbar_wait(&drained, 0, ok ? TW_POLLS : TW_DRAIN);
    if (!ok) {   // copies in flight land before the CTA ends
      for (int w = max(0, lb - nb); w < lb; ++w) mbar_wait(&bfull[w % nb], (w / nb) & 1, TW_DRAIN);
      for (int w = resident ? 0 : max(0, la - ad); w < la; ++w)
        mbar_wait(&afull[resident ? w : w % ad], resident ? 0 : (w / ad) & 1, TW_DRAIN);
    }
  } else {
    const int nmax = L.nmax, g = L.g;
    const long long nn = (long long)nmax * nmax;
    const int row = 32 * (warp & 3) + lane, cg = 8 * (warp >> 2), i = i0 + row;
    // A_CC(i, j) at rowb(i) + colb(j)
    auto place = [&](int q, long long& rb, long long& cb) {
      const int cm = R.cmap[q], s = cm >> 16, pos = cm & 0xffff;
      const int u = nbr_box(R.box, g, s % 3 - 1, s / 3 - 1);
      rb = (long long)u * 25 * nn + pos - (long long)((s / 3) * 5 + s % 3) * nn;
      cb = (long long)((s / 3) * 5 + s % 3 + 12) * nn + (long long)pos * nmax;
    };
    long long rowb = 0, rowc = 0;
    int er = 0;
    if (i < c) {
      place(i, rowb, rowc);
      er = R.Eexp[i] - 53;
    }
    bool ok = true;
    for (int q = 0; q < nt && ok; ++q) {
      const int j0 = 32 * (t0 + q * csplit);
      const bool live = j0 + cg < c && 32 * (warp & 3) < rows;   // (of the warp)
      long long jr = 0, jc = 0;   // of column j0 + lane
      int je = 0;
      if (j0 + lane < c) {
        place(j0 + lane, jr, jc);
        je = R.Fexp[j0 + lane];
      }
      ok = mbar_wait(&tdone, q & 1, polls);
      ok = __all_sync(0xffffffffu, ok) && s_ok;
      if (!ok) break;
      tc_fence_after();
      const uint32_t tb = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + cg;
      long long w[2][8];
#pragma unroll
      for (int c0 = 0; c0 < 8; c0 += 4)
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          uint32_t gr[OZ_S][4];
          if (live) {
#pragma unroll
            for (int u = 0; u < OZ_S; ++u) tmem_ldn<4>(gr[u], tb + 256 * part + 32 * u + c0);
            tmem_ld_wait();
            if (ns * TW_K <= TW_KN) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                w[part][c0 + e] = oz_join([&](int u) { return __uint_as_float(gr[u][e]); });
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                w[part][c0 + e] = oz_join<true>([&](int u) { return __uint_as_float(gr[u][e]); });
            }
          }
        }
      // all read: the products of the next tile run while A_CC is updated
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tfree);
#pragma unroll
      for (int c0 = 0; c0 < 8; c0 += 4) {
        zd cv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int j = j0 + cg + c0 + e;
          const long long cb = __shfl_sync(0xffffffffu, jc, cg + c0 + e);
          if (live && i < c && j < c && (!sym || j >= i)) cv[e] = L.blk[rowb + cb];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int j = j0 + cg + c0 + e;
          const long long cb = __shfl_sync(0xffffffffu, jc, cg + c0 + e), rb = __shfl_sync(0xffffffffu, jr, cg + c0 + e);
          const int sx = er + __shfl_sync(0xffffffffu, je, cg + c0 + e);
          if (live && i < c && j < c && (!sym || j >= i)) {
            const zd x = cv[e] - zd{oz_ldexp_int(w[0][c0 + e], sx), oz_ldexp_int(w[1][c0 + e], sx)};
            L.blk[rowb + cb] = x;
            if (sym && j > i) L.blk[rb + rowc] = x;
          }
        }
      }
    }
    if (!ok) s_ok = 0;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == EP_W) tmem_free(tmem, 512);
  if (tid == 0 && !s_ok) set_error(err, RSS_ETIMEOUT);
}
