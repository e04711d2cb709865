// The ID (Definition 1, Eq. 6) from the exact Gram matrix of the proxy stack.
//
// Column-pivoted QR sees the real stack Y (m x n) only through G = Y^T Y: the
// remaining column norms, the pivots, R up to row signs, ||R22||_F and
// T = R11^{-1} R12.  A Gram matrix rounded to FP64 would lose half the digits,
// so here it is formed exactly and factored in 96-bit fixed point:
//   k_idg_split: every column of a part of Y (at most GI_K rows) gets a
//     power-of-two scale 2^e from its largest entry, and x 2^(55-e), rounded to
//     an integer (the backward error of a column is 2^-56 of its largest entry,
//     below that of a Householder QR in FP64), is cut into eight signed 7-bit
//     digits, |d| <= 64, exact in bf16.
//   k_idg_gram: the 64 digit products of every pair of columns on the tensor
//     cores; sums of equal weight u = p + q stay in FP32 in tensor memory, where
//     they are exact (8 * 512 * 64^2 = 2^24), and are joined to 128-bit integers.
//   k_idg_chol: the parts are added under the columns' common scales, then a
//     pivoted Cholesky factorization by the same stop test, tie window and pivot
//     rule as the reflector kernels (k_id, k_id_cl), with norms that carry no
//     downdating error.
//   k_idg_tsolve: T by back substitution in FP64.
// An entry of the factorization carries an absolute error of a few k 2^-96 of the
// largest diagonal, which T sees through 1 / sigma_min^2, about 1 / eps^2; the
// QR's 2^-53 enters through 1 / eps.  For eps >= IDG_EPS the former is smaller:
// against T from a quad-precision QR of the same stack the error here was 0.2 to 1.2
// times the reflectors' for eps from 1e-4 to 1e-9.
//
// The reflector kernels do 4 m n k FP64 flops a box (two FMAs per clock and SM) and
// read the stack once per pivot; here the m n^2 part runs on the tensor cores, the
// rest in 32-bit integer arithmetic, and the stack is read once.  ID phase of a
// factorization, reflectors before, this after: Laplace 1024^2 132.0 -> 42.1 ms,
// 256^2 31.3 -> 8.1, 64^2 (eps 1e-8) 15.7 -> 4.0, Helmholtz 256^2 54.6 -> 11.1.

constexpr int GI_K = 512;                    // rows of a part
constexpr int GI_B = 32;                     // rows and columns of a block of digits
constexpr int GI_BLK = GI_B * GI_B * 2;      // bytes of a block of one digit slice
constexpr int GI_ST = 192 * 1024;            // shared memory of the product kernel's stages
constexpr double IDG_EPS = 1e-9;
constexpr int GI_ZERO = -100000;             // exponent of an all-zero column of a part
constexpr int GI_NAN = 1025;                 // exponent of a column that holds a NaN or an infinity
constexpr size_t GI_CHOL_SM = 220 * 1024;

// Workspace of one box: digits | 128-bit parts | R | exponents | scalars.  Digits:
// block (kb, p, jb) of rows 32 kb .., slice p, columns 32 jb .. at
// ((kb * 8 + p) * J + jb) * GI_BLK (J = column blocks of the box), inside a block
// the no-swizzle K-major layout of 8-row x 16-byte core matrices: column j, row i
// at (j / 8) * 512 + (i / 8) * 128 + (j % 8) * 16 + (i % 8) * 2.  Part c: block
// (ib, jb), ib <= jb, entry (i, j) at (((c * J + ib) * J + jb) * 1024 + i * 32 + j).
struct GramWs {
  unsigned char* p;
  size_t slot, o_part, o_R, o_ex, o_m;   // bytes
  int ch, nch, J;                        // rows and number of parts, column blocks: of the class
};

struct GramShape {
  int nM, mh, m;
};

// Neighbours of box B at distance 2 and the rows of its stack (thread 0 fills Mbox, Moff).
template <typename S>
__device__ __forceinline__ void idg_rows(const IdArgs<double, S>& a, int B, int* Mbox, int* Moff, GramShape* s) {
  const LevelDev<S>& L = a.L;
  if (threadIdx.x == 0) {
    int cnt = 0, off = 0;
    for (int dy = -2; dy <= 2; ++dy)
      for (int dx = -2; dx <= 2; ++dx) {
        if (max(abs(dx), abs(dy)) != 2) continue;
        const int mb = nbr_box(B, L.g, dx, dy);
        if (mb < 0) continue;
        Mbox[cnt] = mb;
        Moff[cnt] = off;
        off += L.nact[mb];
        ++cnt;
      }
    Moff[cnt] = off;
    s->nM = cnt;
    s->mh = off;
    s->m = a.half ? off + a.P : 2 * (off + a.P);
  }
  __syncthreads();
}

// One CTA: 8 columns of one part of one box; a thread holds one column's entries
// of up to two groups of 8 rows, so the stack is read once.
template <typename S> __global__ void __launch_bounds__(256) k_idg_split(IdArgs<double, S> a, GramWs w) {
  __shared__ int Mbox[16], Moff[17];
  __shared__ GramShape sh;
  __shared__ long long roff[GI_K];
  __shared__ unsigned long long cmax[8][8];
  const LevelDev<S>& L = a.L;
  const int box = blockIdx.z, B = a.boxes[a.base + box], n = L.n[B], J = (n + GI_B - 1) / GI_B;
  const int j8 = blockIdx.x * 8, r0 = blockIdx.y * w.ch;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (j8 >= J * GI_B) return;
  idg_rows(a, B, Mbox, Moff, &sh);
  const int mh = sh.mh, m = sh.m, rows = min(w.ch, m - r0);
  unsigned char* slot = w.p + (size_t)box * w.slot;
  if (j8 == 0 && r0 == 0 && tid == 0) *reinterpret_cast<int*>(slot + w.o_m) = m;
  if (rows <= 0) return;
  constexpr bool cplx = !std::is_same<double, S>::value;
  constexpr int W = cplx ? 2 : 1;
  const int nmax = L.nmax;
  const long long nn = (long long)nmax * nmax;
  for (int r = tid; r < rows; r += 256) {
    const int i = r0 + r;
    const bool second = cplx && i >= mh + a.P;
    const int ii = second ? i - mh - a.P : i;
    long long o = -1;   // a proxy row
    if (ii < mh) {
      int q = 0;
      while (Moff[q + 1] <= ii) ++q;
      const int mb = Mbox[q];
      o = W * (((long long)mb * 25 + off_index(mb, B, L.g)) * nn + L.act[mb * nmax + (ii - Moff[q])]) + (second ? 1 : 0);
    }
    roff[r] = o;
  }
  __syncthreads();
  const double* blk = reinterpret_cast<const double*>(L.blk);
  const int jl = tid & 7, j = j8 + jl, kg0 = tid >> 3;
  const long long cj = (long long)j * nmax * W;
  const int bx = B % L.g, by = B / L.g;
  const double cx = a.geo.x0 - 0.5 * a.geo.hg + (bx + 0.5) * a.Lbox;
  const double cy = a.geo.y0 - 0.5 * a.geo.hg + (by + 0.5) * a.Lbox;
  double v[2][8];
  unsigned long long mk = 0;
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int r = (kg0 + 32 * t) * 8 + e;
      double x = 0.0;
      if (j < n && r < rows) {
        const long long o = roff[r];
        x = o >= 0 ? blk[o + cj] : id_entry<double, S>(a, B, r0 + r, j, mh, Mbox, Moff, cx, cy);
      }
      v[t][e] = x;
      mk = max(mk, oz_abs_bits(x));
    }
#pragma unroll
  for (int d = 8; d < 32; d <<= 1) mk = max(mk, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mk, d));
  if (lane < 8) cmax[warp][lane] = mk;
  __syncthreads();
  mk = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) mk = max(mk, cmax[q][jl]);
  const int eb = oz_emax_b(mk);
  if (tid < 8)
    reinterpret_cast<int*>(slot + w.o_ex)[(size_t)blockIdx.y * w.J * GI_B + j] = mk ? eb - 1022 : GI_ZERO;
  const int nkg = ((rows + GI_B - 1) / GI_B) * (GI_B / 8);   // groups of 8 rows, the last block padded with zeros
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int kg = kg0 + 32 * t;
    if (kg >= nkg) break;
    uint32_t dg[4][OZ_S];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      oz_digits2(oz_scaled_int(v[t][2 * e], eb + 1), oz_scaled_int(v[t][2 * e + 1], eb + 1), dg[e]);
    const size_t kb = (size_t)(r0 / GI_B) + kg / 4;
    unsigned char* d = slot + (kb * OZ_S * J + j / GI_B) * GI_BLK + ((j % GI_B) / 8) * 512 + (kg % 4) * 128 + (j % 8) * 16;
#pragma unroll
    for (int p = 0; p < OZ_S; ++p)
      *reinterpret_cast<uint4*>(d + (size_t)p * J * GI_BLK) = make_uint4(dg[0][p], dg[1][p], dg[2][p], dg[3][p]);
  }
}

__host__ __device__ inline int idg_items(int J) {   // column blocks c and row tiles of 128 with a row <= the columns
  int s = 0;
  for (int t = 0; 4 * t < J; ++t) s += J - 4 * t;
  return s;
}

// One CTA: columns 32 c .. of G against the row tile T (rows 128 T ..), for one
// part.  The tile's rows up to the diagonal are stacked with their digit slices:
// SM slices of 128 / SM rows (SM = 4, 2, 1 by the tile's row blocks) fill the 128
// rows of a product, the eight slices of the 32 columns its N = 256; product a
// (slices SM a ..) accumulates at TMEM column 32 SM a, which puts A_p B_q^T, p =
// SM a + i, into column block v = SM a + q of lane block i: its weight is v + i.
// Thread 0 of warp 0 feeds the stages by bulk copies, thread 0 of warp 1 issues
// the products; every wait is bounded, and a wait that runs out sets RSS_ETIMEOUT
// once the products and copies already issued have finished.
__global__ void __launch_bounds__(256, 1) k_idg_gram(const int* npts, const int* boxes, GramWs w, int* err,
                                                       int polls) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t full[8], empty[8], done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_ok;
  const int box = blockIdx.z, part = blockIdx.y;
  const int n = npts[boxes[box]], J = (n + GI_B - 1) / GI_B;
  int T = 0, c = blockIdx.x;
  while (4 * T < w.J && c >= w.J - 4 * T) c -= w.J - 4 * T++;
  c += 4 * T;
  if (c >= J) return;
  unsigned char* slot = w.p + (size_t)box * w.slot;
  const int m = *reinterpret_cast<const int*>(slot + w.o_m), rows = min(w.ch, m - part * w.ch);
  if (rows <= 0) return;
  const int nkb = (rows + GI_B - 1) / GI_B;
  const int nj = min(4, c - 4 * T + 1);              // row blocks up to the diagonal
  const int njp = nj == 3 ? 4 : nj, SM = 4 / njp;    // (a tile of three is padded: the last rows are not read)
  const bool diag = nj == 1;                          // the tile's rows are its columns
  const uint32_t stA = diag ? 0 : (uint32_t)(OZ_S * njp * GI_BLK), stB = OZ_S * GI_BLK, st = stA + stB;
  const int nst = min(8, (int)(GI_ST / st));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&done, 1);
    s_ok = 1;
  }
  if (warp == 0) tmem_alloc(&s_tmem, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  int fed = 0;   // stages filled (thread 0)
  if (warp == 0 && lane == 0) {
    const unsigned char* src = slot + (size_t)(part * (w.ch / GI_B)) * OZ_S * J * GI_BLK;
    for (int it = 0; it < nkb; ++it, ++fed) {
      const int s = it % nst;
      if (it >= nst && !mbar_wait(&empty[s], ((it / nst) - 1) & 1, polls)) {
        s_ok = 0;
        break;
      }
      unsigned char* d = sm + (size_t)s * st;
      mbar_expect_tx(&full[s], (diag ? 0u : (uint32_t)(OZ_S * nj * GI_BLK)) + stB);
      const unsigned char* g = src + (size_t)it * OZ_S * J * GI_BLK;
      for (int p = 0; p < OZ_S; ++p) {
        if (!diag) bulk_g2s(d + p * njp * GI_BLK, g + ((size_t)p * J + 4 * T) * GI_BLK, nj * GI_BLK, &full[s]);
        bulk_g2s(d + stA + p * GI_BLK, g + ((size_t)p * J + c) * GI_BLK, GI_BLK, &full[s]);
      }
    }
  } else if (warp == 1 && lane == 0) {
    int ok = 1;
    for (int it = 0; it < nkb; ++it) {
      const int s = it % nst;
      if (!mbar_wait(&full[s], (it / nst) & 1, polls)) {
        ok = 0;
        break;
      }
      tc_fence_after();
      const unsigned char* b = sm + (size_t)s * st + stA;
      const unsigned char* ab = diag ? b : sm + (size_t)s * st;
      const int na = OZ_S / SM;
      for (int h = 0; h < GI_B / 16; ++h) {
        const uint32_t boff = smem_u32(b) + h * 256, aoff = smem_u32(ab) + h * 256;
        const bool first = it == 0 && h == 0;
        // the last product first, then the first one: between them they cover all
        // columns, the first one's overlap with the last one accumulates
        for (int x = 0; x < na; ++x) {
          const int q = x == 0 ? na - 1 : x - 1;
          const uint64_t ad = umma_desc(aoff + q * 4 * GI_BLK, 128, 512);
          const uint32_t col = tmem + GI_B * SM * q;
          if (first && x == 1) {   // q = 0: columns below the last product's are fresh
            const int nf = GI_B * SM * (na - 1);
            umma_bf16(col, ad, umma_desc(boff, 128, 512), umma_idesc_bf16(128, nf), 0u);
            umma_bf16(col + nf, ad, umma_desc(boff + (OZ_S - SM) * GI_BLK, 128, 512), umma_idesc_bf16(128, 256 - nf), 1u);
          } else {
            umma_bf16(col, ad, umma_desc(boff, 128, 512), umma_idesc_bf16(128, 256), first && x == 0 ? 0u : 1u);
          }
        }
      }
      umma_commit(&empty[s]);
    }
    umma_commit(&done);
    if (!mbar_wait(&done, 0, ST_DRAIN_POLLS)) ok = 0;
    if (!ok) s_ok = 0;
  }
  __syncwarp();
  __syncthreads();
  tc_fence_after();
  const int ok = s_ok;
  if (!ok && tid == 0) {
    set_error(err, RSS_ETIMEOUT);   // the copies in flight land before the CTA ends
    for (int q = max(0, fed - nst); q < fed; ++q) mbar_wait(&full[q % nst], (q / nst) & 1, ST_DRAIN_POLLS);
  }
  if (ok) {
    // 128-bit sums of the lane's row: sum over v of D_v 2^(7 (14 - v - i)), eight columns at a time
    const int quarter = warp & 3, half = warp >> 2, V = 16 - SM;
    const int rl = 32 * quarter + lane, sub = rl / (128 / SM);
    const uint32_t base = tmem + ((uint32_t)(32 * quarter) << 16) + 16 * half;
    uint4* stg = reinterpret_cast<uint4*>(sm);   // 128 x 33
    for (int c0 = 0; c0 < 16; c0 += 8) {
      __int128 acc[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = 0;
#pragma unroll
      for (int v0 = 0; v0 < 15; v0 += 5) {
        uint32_t gr[5][8];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          if (v0 + v < V) tmem_ld8(gr[v], base + GI_B * (v0 + v) + c0);
          else
#pragma unroll
            for (int e = 0; e < 8; ++e) gr[v][e] = 0u;
        }
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          long long t = 0;
#pragma unroll
          for (int v = 0; v < 5; ++v) t = t * 128 + (long long)__float2int_rn(__uint_as_float(gr[v][e]));
          acc[e] = acc[e] * ((__int128)1 << 35) + t;
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const __int128 x = acc[e] >> (7 * sub);   // (exact: v + i <= 14)
        const unsigned long long lo = (unsigned long long)x, hi = (unsigned long long)(x >> 64);
        stg[rl * 33 + 16 * half + c0 + e] =
            make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
      }
    }
    __syncthreads();
    const int RT = 128 / SM;
    uint4* out = reinterpret_cast<uint4*>(slot + w.o_part) + (size_t)part * J * J * (GI_B * GI_B);
    for (int e = tid; e < nj * GI_B * GI_B; e += 256) {
      const int r = e / GI_B, jj = e % GI_B;
      unsigned __int128 s = 0;
      for (int i = 0; i < SM; ++i) {
        const uint4 x = stg[(i * RT + r) * 33 + jj];
        s += ((unsigned __int128)(((unsigned long long)x.w << 32) | x.z) << 64) | (((unsigned long long)x.y << 32) | x.x);
      }
      const unsigned long long lo = (unsigned long long)s, hi = (unsigned long long)(s >> 64);
      out[((size_t)(4 * T + r / GI_B) * J + c) * (GI_B * GI_B) + (r % GI_B) * GI_B + jj] =
          make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, 512);
}

// ------------------------------------------------------------------ 96-bit fixed point
// Magnitudes as three 32-bit limbs (x least significant): a fraction of 96 bits,
// except that entries of G are signed with 95 fraction bits, |g| <= 1/2.
struct U96 {
  uint32_t x, y, z;
};
// the upper 96 bits of the 192-bit product, low by at most a few units
__device__ __forceinline__ U96 u96_mulhi(U96 a, U96 b) {
  const unsigned long long c = (unsigned long long)__umulhi(a.z, b.x) + __umulhi(a.y, b.y) + __umulhi(a.x, b.z);
  const unsigned long long p = (unsigned long long)a.z * b.y, q = (unsigned long long)a.y * b.z;
  const unsigned long long t = (unsigned long long)a.z * b.z;
  const unsigned long long s0 = c + (uint32_t)p + (uint32_t)q;
  const unsigned long long s1 = t + (p >> 32) + (q >> 32) + (s0 >> 32);
  return U96{(uint32_t)s0, (uint32_t)s1, (uint32_t)(s1 >> 32)};
}
__device__ __forceinline__ U96 u96_shl(U96 a, int s) {   // s >= 0
  while (s >= 32) {
    a = U96{0u, a.x, a.y};
    s -= 32;
  }
  return U96{a.x << s, __funnelshift_l(a.x, a.y, s), __funnelshift_l(a.y, a.z, s)};
}
__device__ __forceinline__ int u96_clz(U96 a) { return a.z ? __clz(a.z) : a.y ? 32 + __clz(a.y) : 64 + __clz(a.x); }
__device__ __forceinline__ U96 s96_abs(uint32_t x, uint32_t y, uint32_t z, uint32_t* neg) {
  const uint32_t s = (uint32_t)((int)z >> 31);
  x ^= s; y ^= s; z ^= s;
  const uint32_t c0 = s & 1u;
  const uint32_t xx = x + c0, c1 = xx < c0, yy = y + c1, c2 = yy < c1;
  *neg = s;
  return U96{xx, yy, z + c2};
}

// g -= v / 2, or g += v / 2 where neg is all ones (g signed, 95 fraction bits)
__device__ __forceinline__ void s96_sub_half(uint32_t& x, uint32_t& y, uint32_t& z, U96 v, uint32_t neg) {
  const uint32_t s = ~neg;   // all ones: subtract
  const uint32_t a0 = __funnelshift_r(v.x, v.y, 1) ^ s, a1 = __funnelshift_r(v.y, v.z, 1) ^ s, a2 = (v.z >> 1) ^ s;
  asm("{\n.reg .u32 c;\nadd.cc.u32 c, %6, %6;\naddc.cc.u32 %0, %0, %3;\naddc.cc.u32 %1, %1, %4;\naddc.u32 %2, %2, %5;\n}\n"
      : "+r"(x), "+r"(y), "+r"(z)
      : "r"(a0), "r"(a1), "r"(a2), "r"(s & 0x80000000u));
}
// a / 2^96 2^e2 as the bits of a double, truncated (0 when it would not be normal):
// integer instructions only, and non-negative doubles order like their bits
__device__ __forceinline__ unsigned long long u96_dbits(U96 a, int e2) {
  const int lz = u96_clz(a), f = 1022 - lz + e2;
  if (lz >= 96 || f <= 0) return 0ull;
  const U96 b = u96_shl(a, lz);
  return ((unsigned long long)f << 52) + (((((unsigned long long)b.z << 32) | b.y) << 1) >> 12);
}
// 1 / (2 sqrt(v)) in (1/2, 1] as a 96-bit fraction, v a fraction in [1/4, 1): a 22-bit
// seed, one Newton step in 64 bits (about 43 bits), one third-order step in 96;
// relative error below 2^-91.  Integer instructions but for the seed: a chain of FP64
// instructions here costs several times as long, and every pivot waits for it.
__device__ __forceinline__ U96 u96_rsqrt_half(U96 v) {
  const float r0 = rsqrtf((float)v.z * 0x1p-32f);
  const uint32_t R0 = (uint32_t)fminf(r0 * 0x1p31f, 4294967040.0f);
  const unsigned long long vh = ((unsigned long long)v.z << 32) | v.y;
  const long long e0 = (1ll << 62) - (long long)__umul64hi(vh, (unsigned long long)R0 * R0);   // (1 - 4 v r^2) 2^62
  const long long d0 = ((long long)R0 * (e0 >> 12)) >> 19;
  unsigned long long r1 = ((unsigned long long)R0 << 32) + (unsigned long long)d0;
  if (d0 > 0 && r1 < (unsigned long long)d0) r1 = ~0ull;
  const unsigned long long sh = __umul64hi(r1, r1), sl = r1 * r1;
  const U96 t = u96_mulhi(v, U96{(uint32_t)(sl >> 32), (uint32_t)sh, (uint32_t)(sh >> 32)});
  // (1 - 4 v r^2) 2^94: t is near 2^94, their difference fits 64 bits
  const unsigned long long tl = ((unsigned long long)t.y << 32) | t.x;
  const long long e1 = (long long)(0ull - tl);
  const long long q = e1 >> 24;
  const long long x = e1 + (long long)(((unsigned long long)(q * q) * 3ull) >> 48);
  const __int128 d = ((__int128)(unsigned __int128)r1 * x) >> 63;
  __int128 r = ((__int128)(unsigned __int128)r1 << 32) + d;
  if (r >> 96) r = ((__int128)1 << 96) - 1;
  return U96{(uint32_t)r, (uint32_t)(r >> 32), (uint32_t)(r >> 64)};
}

// shared memory of k_idg_chol: G (upper triangle, three limb planes), the new
// row, norms, exponents, the remaining columns (two lists), permutation
__host__ __device__ inline size_t idg_chol_bytes(int nmax) {
  const size_t tri = ((size_t)nmax * (nmax + 1) / 2 + 3) & ~size_t(3);
  return tri * 12 + (size_t)nmax * (sizeof(uint4) + sizeof(double) + 5 * sizeof(int)) + 16;
}

// One CTA per box: pivoted Cholesky of G (k = -1 after an error, *err).  R (row l of column j at R[j * nmax + l],
// in the columns' scaled units), k, the permutation; then k_idg_tsolve.
template <typename S> __global__ void __launch_bounds__(1024, 1) k_idg_chol(IdArgs<double, S> a, GramWs w,
                                                                             const int* err) {
  extern __shared__ __align__(16) unsigned char sm[];
  const LevelDev<S>& L = a.L;
  const int nmax = L.nmax, box = blockIdx.x, bi = a.base + box, B = a.boxes[bi], n = L.n[B];
  if (*err != 0) {   // the products did not end: no rank, which ends the factorization
    if (threadIdx.x == 0) a.k_out[bi] = -1;
    return;
  }
  const int J = (n + GI_B - 1) / GI_B;
  const size_t tri = ((size_t)nmax * (nmax + 1) / 2 + 3) & ~size_t(3);
  uint4* row = reinterpret_cast<uint4*>(sm);   // limbs and sign of the new row of R
  double* norms = reinterpret_cast<double*>(row + nmax);
  uint32_t* g0 = reinterpret_cast<uint32_t*>(norms + nmax);
  uint32_t *g1 = g0 + tri, *g2 = g1 + tri;
  int* ex = reinterpret_cast<int*>(g2 + tri);
  int* rem = ex + nmax;              // remaining columns, ascending; two lists
  int* perm = rem + 2 * nmax;
  int* pos = perm + nmax;
  __shared__ int s_q, s_stop, s_shift, s_emax;
  __shared__ U96 s_rinv;
  unsigned char* slot = w.p + (size_t)box * w.slot;
  const int m = *reinterpret_cast<const int*>(slot + w.o_m), nparts = (m + w.ch - 1) / w.ch;
  const int* pex = reinterpret_cast<const int*>(slot + w.o_ex);
  const int est = w.J * GI_B;
  const uint4* parts = reinterpret_cast<const uint4*>(slot + w.o_part);
  double* R = reinterpret_cast<double*>(slot + w.o_R);
  double* rinv = R + (size_t)nmax * nmax;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  if (tid == 0) s_emax = GI_ZERO;
  __syncthreads();
  for (int j = tid; j < n; j += nt) {
    int e = GI_ZERO;
    for (int p = 0; p < nparts; ++p) e = max(e, pex[(size_t)p * est + j]);
    ex[j] = e;
    rem[j] = j;
    perm[j] = j;
    pos[j] = j;
    atomicMax(&s_emax, e);
  }
  __syncthreads();
  const int emax = s_emax;
  const int shift = 16 + (m > 1 ? 32 - __clz(m - 1) : 0);   // |G| <= m 2^110 -> |g| <= 1/2 with 95 fraction bits
  auto tidx = [n](int i, int j) { return i * n - i * (i - 1) / 2 - i + j; };   // i <= j
  // remaining squared norm of column j in the true scale, relative to the largest column's
  auto norm_of = [&](int j, uint32_t x, uint32_t y, uint32_t z) {
    const int e2 = max(2 * (ex[j] - emax), -2000);
    return (int)z < 0 ? 0.0 : __longlong_as_double((long long)u96_dbits(U96{x, y, z}, e2));
  };
  // G: the parts under the columns' common scales
  for (int i = warp; i < n; i += nw) {
    const int ei = ex[i];
    for (int j = i + lane; j < n; j += 32) {
      const int ej = ex[j];
      __int128 s = 0;
      for (int p = 0; p < nparts; ++p) {
        const int d = (ei - pex[(size_t)p * est + i]) + (ej - pex[(size_t)p * est + j]);
        if (d > 126) continue;
        const uint4 x = parts[(((size_t)p * J + i / GI_B) * J + j / GI_B) * (GI_B * GI_B) + (i % GI_B) * GI_B + j % GI_B];
        const __int128 v = (__int128)(((unsigned __int128)(((unsigned long long)x.w << 32) | x.z) << 64) |
                                      (((unsigned long long)x.y << 32) | x.x));
        s += v >> d;
      }
      s >>= shift;
      const int t = tidx(i, j);
      const uint32_t x = (uint32_t)s, y = (uint32_t)(s >> 32), z = (uint32_t)(s >> 64);
      g0[t] = x;
      g1[t] = y;
      g2[t] = z;
      if (i == j) norms[i] = ei == GI_ZERO ? 0.0 : norm_of(i, x, y, z);
    }
  }
  __syncthreads();
  // warp 0 picks the pivots, warp 1 runs the stop test
  double thresh = 0.0;
  float y2max = 0.0f;
  if (warp < 2) {
    double s = 0.0, mx = 0.0;
    for (int c = lane; c < n; c += 32) {
      s += norms[c];
      mx = fmax(mx, norms[c]);
    }
    thresh = a.eps * a.eps * warp_sum(s);
    y2max = (float)warp_max(mx);
  }
  int k = 0;
  const int kmax = emax >= GI_NAN ? 0 : min(m, n);
  while (k < kmax) {
    const int nr = n - k;
    const int* rm = rem + (k & 1) * nmax;
    int* rn = rem + ((k + 1) & 1) * nmax;
    if (warp == 0) {   // pivot: largest remaining norm, lowest column among ties
      unsigned long long mk = 0;
      for (int b = lane; b < nr; b += 32) mk = max(mk, (unsigned long long)__double_as_longlong(norms[rm[b]]));
      const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(mk >> 32));
      const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(mk >> 32) == hi ? (uint32_t)mk : 0u);
      mk = ((unsigned long long)hi << 32) | lo;
      const double mx = __longlong_as_double((long long)mk);
      const float mf = (float)mx;
      // (the window to 24 bits: it is a small part of mx)
      const double thr = mx - (double)((float)TIE_REL * mf + (float)TIE_ABS * sqrtf(mf * y2max));
      const unsigned long long tk = thr > 0.0 ? (unsigned long long)__double_as_longlong(thr) : 0ull;
      int q = INT_MAX;
      for (int b = lane; b < nr; b += 32) {
        const int c = rm[b];
        if ((unsigned long long)__double_as_longlong(norms[c]) >= tk) {
          q = c;
          break;
        }
      }
      q = (int)__reduce_min_sync(0xffffffffu, (uint32_t)q);
      if (mk == 0) q = -1;
      if (q >= 0) {
        const int t = tidx(q, q);
        const U96 g{g0[t], g1[t], g2[t]};
        const int sft = (u96_clz(g) - 1) & ~1;   // g 2^sft in [1/4, 1), 95 fraction bits
        const U96 ri = u96_rsqrt_half(u96_shl(g, sft + 1));
        if (lane == 0) {
          s_rinv = ri;
          s_shift = sft / 2;
        }
      }
      if (lane == 0) s_q = q;
    } else if (warp == 1) {
      double s = 0.0;
      for (int b = lane; b < nr; b += 32) s += norms[rm[b]];
      s = warp_sum(s);
      if (lane == 0) s_stop = s <= thresh;
    }
    __syncthreads();
    const int q = s_q;
    if (s_stop || q < 0) break;
    const U96 ri = s_rinv;
    const int sft = s_shift;
    // row k of R: g_qc / sqrt(g_qq) for the remaining columns
    for (int b = tid; b < nr; b += nt) {
      const int c = rm[b];
      if (c != q) {
        const int t = tidx(min(q, c), max(q, c));
        uint32_t neg;
        const U96 v = u96_mulhi(u96_shl(s96_abs(g0[t], g1[t], g2[t], &neg), sft + 1), ri);
        const U96 l = u96_shl(v, 1);
        row[c] = make_uint4(l.x, l.y, l.z, neg);
        const double d = __longlong_as_double((long long)u96_dbits(l, 0));
        R[(size_t)c * nmax + k] = neg ? -d : d;
        rn[b - (c > q)] = c;
      } else {
        rinv[k] = __longlong_as_double((long long)u96_dbits(ri, sft + 1));   // 1 / R_kk in the units of R
        const int pq = pos[q], ck = perm[k];
        perm[k] = q;
        perm[pq] = ck;
        pos[ck] = pq;
        pos[q] = k;
      }
    }
    __syncthreads();
    // G -= row row^T over the remaining columns
    for (int x = warp; x < nr - 1; x += nw) {
      const int i = rn[x];
      const uint4 li = row[i];
      const int rs = tidx(i, 0);
      for (int b = x + lane; b < nr - 1; b += 64) {   // two columns in flight
        const bool two = b + 32 < nr - 1;
        const int j = rn[b], t = rs + j, j2 = two ? rn[b + 32] : j, t2 = rs + j2;
        const uint4 lj = row[j], lk = row[j2];
        uint32_t x0 = g0[t], x1 = g1[t], x2 = g2[t], y0 = g0[t2], y1 = g1[t2], y2 = g2[t2];
        s96_sub_half(x0, x1, x2, u96_mulhi(U96{li.x, li.y, li.z}, U96{lj.x, lj.y, lj.z}), li.w ^ lj.w);
        s96_sub_half(y0, y1, y2, u96_mulhi(U96{li.x, li.y, li.z}, U96{lk.x, lk.y, lk.z}), li.w ^ lk.w);
        g0[t] = x0;
        g1[t] = x1;
        g2[t] = x2;
        if (two) {
          g0[t2] = y0;
          g1[t2] = y1;
          g2[t2] = y2;
        }
        if (i == j) norms[i] = norm_of(i, x0, x1, x2);
      }
    }
    __syncthreads();
    ++k;
  }
  __syncthreads();
  for (int c = tid; c < n; c += nt) {
    a.perm_out[(size_t)bi * nmax + c] = perm[c];
    reinterpret_cast<int*>(slot + w.o_ex)[c] = ex[c] == GI_ZERO ? 0 : ex[c];   // for k_idg_tsolve
  }
  if (tid == 0) a.k_out[bi] = k;
}

// T = R11^{-1} R12 for 32 redundant columns of one box, four lanes per column
// (the dot product over the solved entries in four parts), undoing the columns'
// scales.  R11 (packed rows) and the solution sit in shared memory.
__host__ __device__ inline size_t idg_tsolve_bytes(int nmax) {
  return sizeof(double) * ((size_t)nmax * (nmax + 1) / 2 + 40 * (size_t)nmax) + sizeof(int) * (size_t)nmax;
}
template <typename S> __global__ void __launch_bounds__(128) k_idg_tsolve(IdArgs<double, S> a, GramWs w) {
  extern __shared__ __align__(16) unsigned char sm[];
  const LevelDev<S>& L = a.L;
  const int nmax = L.nmax, box = blockIdx.y, bi = a.base + box, B = a.boxes[bi], n = L.n[B];
  const int k = a.k_out[bi], r = n - k, c0 = blockIdx.x * 32;
  if (c0 >= r || k <= 0) return;
  unsigned char* slot = w.p + (size_t)box * w.slot;
  const double* R = reinterpret_cast<const double*>(slot + w.o_R);
  const double* rinv = R + (size_t)nmax * nmax;
  const int* ex = reinterpret_cast<const int*>(slot + w.o_ex);
  const int* perm = a.perm_out + (size_t)bi * nmax;
  double* xs = reinterpret_cast<double*>(sm);           // k x 40
  double* R11 = xs + (size_t)40 * nmax;                 // entry (i, l), i < l, at l (l - 1) / 2 + i
  int* es = reinterpret_cast<int*>(R11 + (size_t)nmax * (nmax + 1) / 2);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int l = warp; l < k; l += 4) {
    const double* col = R + (size_t)perm[l] * nmax;
    for (int i = lane; i < l; i += 32) R11[l * (l - 1) / 2 + i] = col[i];
    if (lane == 0) {
      R11[(size_t)nmax * (nmax - 1) / 2 + l] = rinv[l];
      es[l] = ex[perm[l]];
    }
  }
  __syncthreads();
  const int cl = tid >> 2, sub = tid & 3, c = c0 + cl;
  const bool on = c < r;
  const int oc = perm[k + (on ? c : 0)], ec = ex[oc];
  const double* Rc = R + (size_t)oc * nmax;
  S* Tw = a.T_ws + (size_t)bi * nmax * nmax + (size_t)c * nmax;
  const double* inv = R11 + (size_t)nmax * (nmax - 1) / 2;
  for (int i = k - 1; i >= 0; --i) {
    double s = sub == 0 ? Rc[i] : 0.0;
    for (int l = i + 1 + sub; l < k; l += 4) s = fma(-R11[l * (l - 1) / 2 + i], xs[l * 40 + cl], s);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s *= inv[i];
    if (sub == 0) {
      xs[i * 40 + cl] = s;
      if (on) Tw[i] = id_store<double, S>(ldexp(s, ec - es[i]));
    }
    __syncwarp();
  }
}
