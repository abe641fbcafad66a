// Exact-slice float64 DST: the weight-stacked GEMM (the default for ceil(n/2) <= 1024).
//
// Same arithmetic as the 8-bit format of the tile kernel: 7 balanced base-256 digits per operand,
// the 28 digit products with i + j <= 8, exact sums in FP32 tensor memory combined in int64.  What
// differs is where the products of one K step meet.  The tile kernel runs one (or two) digit
// products at a time over the whole K range of a 128 x 128 tile, so every digit tile crosses into
// the SM several times (44 tiles per K step for 28 products) and the SM's 64 B/clk port from the L2
// bounds it (59 B/clk measured).  Here a stage holds ALL seven digit tiles of both operands for 16
// values of K, each crosses once (21 tile halves for the same 28 products: 47 B/clk at the tensor
// pipe's full rate; measured 31 - 33 B/clk and the pipe active 65 - 68 % of the time, the rest being drains,
// tile tails and the last wave), and every weight w = i + j keeps its own 64-column accumulator:
//   * tile 128 rows x 64 columns (N below: 32 or 16 for small transforms); accumulator of weight w =
//     2..8 at tensor-memory column 64 (w - 2);
//   * the B digits lie behind one another in shared memory (64 rows each), so A_i x [B_j .. B_j+m-1]
//     is ONE tcgen05.mma of N = 64 m whose column blocks are the m consecutive weights i + j ..:
//     ten MMAs of 64..256 columns per K step do the 28 products in 908 clocks (896 at the tensor
//     pipe's peak).  They are issued narrow ones first: the three 256-column ones at the end of a
//     stage keep the pipe busy while the issuer commits the stage and waits for the next one
//     (the other way round the pipe idled 75 - 275 clocks per stage).  The issuing loop is uniform over
//     its warp with one elected lane issuing (256 against 265 us as a one-lane branch: descriptors stay in
//     uniform registers);
//   * weight w sums w - 1 products per K value, each at most 2^14, so it stays exact (up to 2^24)
//     for 1024 / (w - 1) values of K; eight epilogue warps drain it in time (ow_drain) into int64
//     sums held in registers and zero it.  Drains go by group of weights ({2,3,4}, {5,6}, {7,8}), each
//     group with its own pair of barriers: the stage after a drain issues the other groups' MMAs first;
//   * the FP32-rounded tail is weights 7 and 8 (2^-40 and 2^-48 of the leading products); weight 7 is
//     drained once on the way so that its accumulation error (directed, about linear in the number of
//     MMAs and the size of the sum) stays below the tile kernel's.
// Digits are plain integers (not pre-scaled: every accumulator holds one weight), and both operands'
// expansions are rounded to nearest at 2^-55 instead of truncated (row errors against extended
// precision 2.1e-16 - 2.8e-16 on random rows of 40..2048 values, 2.2e-16 - 3.7e-16 with truncation).
// Measured, whole preconditioner applies (two transforms each), tile kernel -> this one: 1024 x 1024 x
// 256 right-hand sides 21.1 -> 14.2 ms, 2048 x 1024 x 1 287 -> 254 us, 63 x 40 65.6 -> 35 us (45 with
// 64-column tiles only).
constexpr int OW_NS = 7;                          // digits per operand
constexpr int OW_K = 16;                          // K values per stage (one MMA K step)
constexpr int OW_N = 64;                          // columns of a packed B tile
constexpr int OW_ASL = TM * OW_K * 2;             // one A digit of a stage: 128 rows of 32 bytes
constexpr int OW_BSL = OW_N * OW_K * 2;           // one digit of a packed B tile: 64 rows of 32 bytes
constexpr int OW_A = OW_NS * OW_ASL;              // 28 KB
constexpr int OW_B = OW_NS * OW_BSL;              // 14 KB
constexpr int OW_FIX = 38;                        // sums in units of 2^-38 of a weight-2 unit
// Tiles of N = 64, 32 or 16 columns (a packed B tile or its halves / quarters).  A tile's time is its
// MMAs plus a tail that grows with N (the last drains, the conversion and the store: 12 k clocks at
// N = 64), so transforms whose tiles leave SMs idle anyway take the narrowest tile that still runs in
// one wave; above one wave N = 64 (N = 32: 496 clocks a K step for half of the 908's work).
template <int N>
struct OwCfg {
  static constexpr int BSL = N * OW_K * 2;
  static constexpr int STAGE = OW_A + OW_NS * BSL;
  static constexpr int NST = N == 64 ? 4 : (N == 32 ? 5 : 6);
  static constexpr int CW = N / 2;                 // columns per epilogue warp (of each weight)
  static constexpr int CH = CW < 16 ? CW : 16;     // columns transposed at a time
  static constexpr int TPITCH = CH + 1;            // doubles per row of a warp's transposition buffer
  static constexpr int TBUF = 32 * TPITCH * 8;
  static constexpr uint32_t TMEM = N == 64 ? 512 : (N == 32 ? 256 : 128);  // allocated columns (7 N used)
  static constexpr int SMEM = NST * STAGE + 8 * TBUF + 1024 + 256;
};

// element (r, k) of a rows x 16 digit tile: 32-byte rows, K-major SWIZZLE_32B (byte offset)
__device__ __forceinline__ uint32_t ow_swz(int r, int kchunk) {
  return (uint32_t)r * 32u + (uint32_t)((kchunk ^ (r >> 2)) & 1) * 16u;
}

// Stages after which a group of weights is drained (bit c: after c stages of a tile of nk <= 64; every
// group at the tile's end).  Exactness allows weight 3 32 stages (2 x 512 x 2^14 = 2^24), 4 20, 5 16,
// 6 12; a drain costs the MMA stream about 1000 clocks (commit, hand-over, hand-back, the pipe refilling),
// so the weights of a group go together and groups share stages where they can (60, 40; 14.18 against
// 14.31 ms for 1024 x 1024 x 256 with 3, 4 at 18, 38, 58 and 7 at 30).
constexpr unsigned long long OW_E0 = (1ull << 20) | (1ull << 40) | (1ull << 60);                            // 3, 4
constexpr unsigned long long OW_E1 = (1ull << 12) | (1ull << 24) | (1ull << 36) | (1ull << 48) | (1ull << 60);  // 5, 6
constexpr unsigned long long OW_E2 = 1ull << 40;                                                            // 7
__device__ __forceinline__ uint32_t ow_bit(unsigned long long m, int c) { return (uint32_t)(m >> c) & 1u; }

// rn(v 2^(55 - e)) for |v| < 2^e, signed (integer arithmetic on the bits); |result| <= 2^55
__device__ __forceinline__ long long ow_fixed(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7ff);
  const unsigned long long M = ((unsigned long long)b & 0xfffffffffffffull) | (E ? (1ull << 52) : 0ull);
  const int s = (E ? E : 1) - 1020 - e;  // |v| 2^(55 - e) = M 2^s
  unsigned long long t;
  if (s >= 0) t = M << s;                // s <= 3 since |v| < 2^e
  else t = (s < -54) ? 0ull : ((M + (1ull << (-s - 1))) >> (-s));
  return b < 0 ? -(long long)t : (long long)t;
}

// the seven digits of 8 values |T| <= 2^55 (8 consecutive K of one row), as bf16, 16 bytes per digit
// at dst + digit * OW_ASL: T plus 128 in each byte position has bytes d_i + 128 (the leading one up to
// 256); 2^23 + byte as a float by one byte permute, minus 2^23 + 128 is the digit, exact in bf16
template <int STRIDE>
__device__ __forceinline__ void ow_store_digits(const long long (&T)[8], uint8_t *dst) {
  uint32_t th[8], tl[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const unsigned long long Tb = (unsigned long long)(T[q] + 0x0080808080808080ll);
    tl[q] = (uint32_t)Tb;
    th[q] = (uint32_t)(Tb >> 32);
  }
#pragma unroll
  for (int i = 1; i <= OW_NS; ++i) {
    uint32_t hw[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float d[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = 2 * q + h;
        uint32_t fb;
        if (i == 1) fb = 0x4B000000u | (th[v] >> 16);
        else if (i <= 3) fb = __byte_perm(th[v], 0x4B00u, 0x5440u | (uint32_t)(3 - i));
        else fb = __byte_perm(tl[v], 0x4B00u, 0x5440u | (uint32_t)(7 - i));
        d[h] = __uint_as_float(fb) - 8388736.0f;
      }
      hw[q] = oz_pack2(d[0], d[1]);
    }
    *reinterpret_cast<uint4 *>(dst + (i - 1) * STRIDE) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
  }
}

// B digits, once per plan: [mat][column tile of 64][K stage][digit][64 x 16]; the matrices as in
// oz_pack_b_kernel.  One thread per 8 consecutive K values of one output column.
__global__ void ow_pack_b_kernel(const double *m0, int k0n, int n0n, int ld0, const double *m1, int k1n, int n1n,
                                 int ld1, int nk, int nnt, int eB, uint8_t *out) {
  const int which = blockIdx.z;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;  // consecutive columns: coalesced reads
  const int ch = blockIdx.y;
  if (n >= nnt * OW_N || ch >= 2 * nk) return;
  const double *m = which ? m1 : m0;
  const int kn = which ? k1n : k0n, nn = which ? n1n : n0n, ld = which ? ld1 : ld0;
  long long T[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = ch * 8 + q;
    T[q] = (n < nn && k < kn) ? ow_fixed(m[(size_t)k * ld + n], eB) : 0;
  }
  uint8_t *base = out + (((size_t)which * nnt + n / OW_N) * nk + (ch >> 1)) * OW_B;
  ow_store_digits<OW_BSL>(T, base + ow_swz(n % OW_N, ch & 1));
}

// The digits of one row staged in shared memory (its n inputs at OZ_PAD(j)), both parities: the row
// exponent from the largest |input| (b0, b1: this thread's largest bit patterns with the sign cleared, b1
// the odd entries' when gathered), the fold u_j = x_j + x_{n-1-j}, v_j = x_j - x_{n-1-j} as exact integer sums,
// or (gather, the DCT-II inverse) u = the even entries and v = the odd ones.  By NT threads of the CTA, whole
// warps, tid of them (every thread of the CTA calls it, for its own row); layout [parity][m tile][K
// stage][digit][128 x 16], erow[parity][row].
template <int NT>
__device__ __forceinline__ void ow_pack_row(int tid, const double *xs, unsigned long long b0, unsigned long long b1,
                                            int row, bool live, int n, int ku, int kv, int nk, int nmt, uint8_t *out, int *erow,
                                            bool gather) {
  __shared__ unsigned long long red[2][OZ_PACK_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) {
    b0 = max(b0, __shfl_xor_sync(0xffffffffu, b0, o));
    b1 = max(b1, __shfl_xor_sync(0xffffffffu, b1, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = b0;
    red[1][threadIdx.x >> 5] = b1;
  }
  __syncthreads();
  const int w0 = (threadIdx.x >> 5) - (tid >> 5);  // first warp of the row's threads
  int e[2];
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    unsigned long long m = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) m = max(m, red[gather ? par : 0][w0 + w]);
    const int E = (int)(m >> 52);
    // |inputs| <= m < 2^(E - 1022) for normal m, < 2^-1022 for subnormal m; 0 for a zero row; the
    // fold's sums and differences of two inputs stay below 2^(that + 1)
    e[par] = (E == 0x7ff) ? OZ_EXP_NAN : (m == 0 ? 0 : (E == 0 ? -1022 : E - 1022) + (gather ? 0 : 1));
  }
  // a non-finite value anywhere in the row makes every output of the row non-finite
  const bool bad = e[0] == OZ_EXP_NAN || e[1] == OZ_EXP_NAN;
  if (tid < 2 && live) erow[tid * (nmt * TM) + row] = bad ? OZ_EXP_NAN : (tid ? e[1] : e[0]);
  const int mt = row / TM, r = row % TM;
  const bool odd_n = (n & 1) != 0;
  for (int ch = tid; ch < 2 * nk; ch += NT) {
    long long U[8], W[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int j = ch * 8 + q;
      long long u = 0, w = 0;
      if (!bad) {
        if (gather) {
          if (j < ku) u = ow_fixed(xs[OZ_PAD(2 * j)], e[0]);
          if (j < kv) w = ow_fixed(xs[OZ_PAD(2 * j + 1)], e[1]);
        } else if (j < kv) {
          const long long a1 = ow_fixed(xs[OZ_PAD(j)], e[0]), a2 = ow_fixed(xs[OZ_PAD(n - 1 - j)], e[0]);
          u = a1 + a2;
          w = a1 - a2;
        } else if (odd_n && j == ku - 1) {
          u = ow_fixed(xs[OZ_PAD(j)], e[0]);  // middle element of an odd-length row
        }
      }
      U[q] = u;
      W[q] = w;
    }
    uint8_t *t0 = out + ((size_t)mt * nk + (ch >> 1)) * OW_A + ow_swz(r, ch & 1);
    ow_store_digits<OW_ASL>(U, t0);
    ow_store_digits<OW_ASL>(W, t0 + (size_t)nmt * nk * OW_A);
  }
}

// A digits per apply, both parities: NT threads per row (64 for rows of up to 1024 values, whose 64 chunks
// would leave half of 128 threads idle), OZ_PACK_THREADS / NT rows per CTA.  HBM-bound: 22 B a point;
// 262144 rows of 1024: 1.28 -> 1.01 ms with two rows per CTA, 5.9 TB/s.
template <int NT>
__global__ void __launch_bounds__(OZ_PACK_THREADS) ow_pack_a_kernel(const double *__restrict__ x, int rows, int n,
                                                                    int ku, int kv, int nk, int nmt,
                                                                    uint8_t *__restrict__ out, int *__restrict__ erow,
                                                                    const KrylovScalars *__restrict__ sc, int rpr,
                                                                    int gather, int stage) {
  pdl_next();
  pdl_wait();
  extern __shared__ double xs_all[];
  const int tid = threadIdx.x % NT, sub = threadIdx.x / NT;
  double *xs = xs_all + sub * stage;  // the row's n inputs at OZ_PAD(j)
  const int row = blockIdx.x * (OZ_PACK_THREADS / NT) + sub;
  // rows of finished right-hand sides keep whatever the buffer held (a row's operand enters that row's outputs
  // only, and nothing reads those any more); a CTA of two rows packs both if either runs
  if (sc != nullptr) {
    bool any = false;
    for (int q = 0; q < OZ_PACK_THREADS / NT; ++q) {
      const int g = blockIdx.x * (OZ_PACK_THREADS / NT) + q;
      any = any || g >= rows || sc[g / rpr].state == ST_RUN;
    }
    if (!any) return;
  }
  const bool live = row < rows;  // the padding rows of the last tile pack as zeros
  const double *xr = x + (size_t)(live ? row : 0) * n;
  unsigned long long b0 = 0, b1 = 0;
  constexpr int PB = 16;  // a batch of loads all issue before any is used
  for (int jb = 0; jb < n; jb += PB * NT) {
    double vb[PB];
#pragma unroll
    for (int u = 0; u < PB; ++u) {
      const int j = jb + u * NT + tid;
      vb[u] = (live && j < n) ? __ldg(xr + j) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < PB; ++u) {
      const int j = jb + u * NT + tid;
      if (j < n) {
        xs[OZ_PAD(j)] = vb[u];
        const unsigned long long m = (unsigned long long)__double_as_longlong(vb[u]) & 0x7fffffffffffffffull;
        if (gather && (j & 1)) b1 = max(b1, m);
        else b0 = max(b0, m);
      }
    }
  }
  ow_pack_row<NT>(tid, xs, b0, b1, row, live, n, ku, kv, nk, nmt, out, erow, gather != 0);
}

// PCG's x += alpha p, r -= alpha q and (r, r) -> convergence state, and the operand of the next
// iteration's forward transform packed from the new r while its row is on chip: MODE 0 the exact-slice
// digits (one launch and one pass over r less per iteration), MODE 1 the split-bf16 tiles of the mixed
// path (scaled by the power of two of the OLD (r, r), the one known here; recorded in jdone for
// the inverse transform).  A CTA takes whole rows of its right-hand side, grid-stride.  Bound by HBM
// / L2: 48 B a point plus the operand (14 or 4 B).  2048 x 1024: update and pack 22 + 16 us as two
// kernels, 33 us as one (mixed 22 + 9, 24 us; 32 right-hand sides 560 + 170, 510 us).
template <int MODE>
__global__ void __launch_bounds__(OZ_PACK_THREADS) pcg_update_pack_kernel(
    double *__restrict__ x, double *__restrict__ r, const double *__restrict__ p, const double *__restrict__ q, int n,
    int rpr, int ku, int kv, int nk, int nmt, uint8_t *__restrict__ out, int *__restrict__ erow, int max_iter,
    KrylovScalars *sc, Reduce red) {
  pdl_next();
  pdl_wait();
  extern __shared__ double xs[];  // MODE 0: the row at OZ_PAD(j); MODE 1: as float, scaled
  float *xf = reinterpret_cast<float *>(xs);
  const int rhs = blockIdx.y;
  if (sc[rhs].state != ST_RUN) return;
  const double a = sc[rhs].alpha;
  const int es = residual_exponent(sc, rhs);
  double acc = 0.0;
  constexpr int PB = 4;
  for (int row = blockIdx.x; row < rpr; row += gridDim.x) {
    const int g = rhs * rpr + row;
    const size_t o = (size_t)g * n;
    unsigned long long b0 = 0;
    for (int jb = 0; jb < n; jb += PB * OZ_PACK_THREADS) {
      double xv[PB], rv[PB], pv[PB], qv[PB];
#pragma unroll
      for (int u = 0; u < PB; ++u) {
        const int j = jb + u * OZ_PACK_THREADS + threadIdx.x;
        const bool in = j < n;
        xv[u] = in ? x[o + j] : 0.0;
        rv[u] = in ? r[o + j] : 0.0;
        pv[u] = in ? p[o + j] : 0.0;
        qv[u] = in ? q[o + j] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < PB; ++u) {
        const int j = jb + u * OZ_PACK_THREADS + threadIdx.x;
        if (j >= n) continue;
        x[o + j] = fma(a, pv[u], xv[u]);
        const double v = fma(-a, qv[u], rv[u]);
        r[o + j] = v;
        acc = fma(v, v, acc);
        if (MODE == 0) {
          xs[OZ_PAD(j)] = v;
          b0 = max(b0, (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull);
        } else {
          xf[OZ_PAD(j)] = narrow_pow2(v, -es);
        }
      }
    }
    if (MODE == 0) {
      ow_pack_row<OZ_PACK_THREADS>(threadIdx.x, xs, b0, 0, g, true, n, ku, kv, nk, nmt, out, erow, false);
    } else {
      __syncthreads();
      tc_pack_row(xf, g, n, ku, kv, nk, nmt, out);
    }
    __syncthreads();  // the row's stage is reused
  }
  double v1[1] = {acc}, tot[1];
  block_sum<1>(v1);
  if (publish_partials<1>(red, rhs, blockIdx.x, gridDim.x, v1, tot)) {
    KrylovScalars &S = sc[rhs];
    S.rr = tot[0];
    S.jdone = es;
    S.iters += 1;
    if (!isfinite(tot[0])) S.state = ST_NAN;
    else if (tot[0] <= S.tol2 * S.bb) S.state = ST_CONV;
    else if (S.iters >= max_iter) S.state = ST_STOP;
  }
}

// shared-memory descriptor constant bits: K-major SWIZZLE_32B, 8-row groups 256 bytes apart
constexpr uint64_t OW_DHI = ((uint64_t)(256 >> 4) << 32) | (1ull << 46) | (6ull << 61) | (1ull << 16);
constexpr uint32_t ow_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}
template <int ACC>
__device__ __forceinline__ void ow_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
               "l"(a), "l"(b), "r"(idesc), "n"(ACC)
               : "memory");
}
// A digit I (0-based) times the LEN B digits that meet it in weights W0 .. (0-based: w - 2); ACC 0 overwrites
template <int N, int I, int W0, int LEN, int ACC = 1>
__device__ __forceinline__ void ow_mmas(uint32_t tmem, uint32_t sa, uint32_t sb) {
  ow_mma<ACC>(tmem + (uint32_t)(W0 * N), OW_DHI | (sa + I * (OW_ASL >> 4)),
              OW_DHI | (sb + (W0 - I) * (OwCfg<N>::BSL >> 4)), ow_idesc(LEN * N));
}
// all 28 products, narrow ones first; every width adds the products of a weight in the same order (A digits 6, 5, 4,
// 2, 1, 0, 3), so the FP32-rounded weights 7 and 8 and with them the results are the same on each
template <int N>
__device__ __forceinline__ void ow_issue_all(uint32_t tmem, uint32_t sa, uint32_t sb) {
  ow_mmas<N, 6, 6, 1>(tmem, sa, sb);
  ow_mmas<N, 5, 5, 2>(tmem, sa, sb);
  ow_mmas<N, 4, 4, 3>(tmem, sa, sb);
  if constexpr (N == 64) {
    ow_mmas<N, 2, 2, 3>(tmem, sa, sb);
    ow_mmas<N, 2, 5, 2>(tmem, sa, sb);
    ow_mmas<N, 1, 5, 2>(tmem, sa, sb);
    ow_mmas<N, 0, 4, 3>(tmem, sa, sb);
    ow_mmas<N, 1, 1, 4>(tmem, sa, sb);
    ow_mmas<N, 0, 0, 4>(tmem, sa, sb);
    ow_mmas<N, 3, 3, 4>(tmem, sa, sb);
  } else {
    ow_mmas<N, 2, 2, 5>(tmem, sa, sb);
    ow_mmas<N, 1, 1, 6>(tmem, sa, sb);
    ow_mmas<N, 0, 0, 7>(tmem, sa, sb);
    ow_mmas<N, 3, 3, 4>(tmem, sa, sb);
  }
}
// the products of one group of weights.  FIRST (a tile's first stage): the leading A digit, which meets
// every weight, goes first and overwrites, which starts the group's sums afresh; else it goes last
// (the widest MMA)
template <int N, int G, bool FIRST>
__device__ __forceinline__ void ow_issue_group(uint32_t tmem, uint32_t sa, uint32_t sb) {
  constexpr int W0 = G == 0 ? 0 : (G == 1 ? 3 : 5), LEN = G == 0 ? 3 : 2;
  if constexpr (FIRST) ow_mmas<N, 0, W0, LEN, 0>(tmem, sa, sb);
  if constexpr (G == 0) {  // weights 2, 3, 4
    ow_mmas<N, 2, 2, 1>(tmem, sa, sb);
    ow_mmas<N, 1, 1, 2>(tmem, sa, sb);
  } else if constexpr (G == 1) {  // 5, 6
    ow_mmas<N, 4, 4, 1>(tmem, sa, sb);
    ow_mmas<N, 3, 3, 2>(tmem, sa, sb);
    ow_mmas<N, 2, 3, 2>(tmem, sa, sb);
    ow_mmas<N, 1, 3, 2>(tmem, sa, sb);
  } else {  // 7, 8
    ow_mmas<N, 6, 6, 1>(tmem, sa, sb);
    ow_mmas<N, 5, 5, 2>(tmem, sa, sb);
    ow_mmas<N, 4, 5, 2>(tmem, sa, sb);
    ow_mmas<N, 3, 5, 2>(tmem, sa, sb);
    ow_mmas<N, 2, 5, 2>(tmem, sa, sb);
    ow_mmas<N, 1, 5, 2>(tmem, sa, sb);
  }
  if constexpr (!FIRST) ow_mmas<N, 0, W0, LEN>(tmem, sa, sb);
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void ow_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// C columns of this warp's 32 lanes: read, or set to zero
template <int C>
__device__ __forceinline__ void ow_tmem_ld(uint32_t taddr, float (&v)[C]) {
  if constexpr (C == 32) {
    tmem_ld32(taddr, v);
  } else if constexpr (C == 16) {
    tmem_ld16(taddr, v);
  } else {
    static_assert(C == 8, "columns per epilogue warp");
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
  }
}
template <int C>
__device__ __forceinline__ void ow_tmem_zero(uint32_t taddr) {
  for (int c = 0; c < C; c += 8)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};\n" ::"r"(taddr + c), "r"(0)
                 : "memory");
}

// acc += the weight's sums (integers G, or FP32-rounded ones for the tail) in units of 2^-OW_FIX
template <int W, int C>
__device__ __forceinline__ void ow_add(const float (&v)[C], long long (&acc)[C]) {
  constexpr int sh = OW_FIX - 8 * (W - 2);
  if constexpr (sh >= 32) {
#pragma unroll
    for (int q = 0; q < C; ++q) acc[q] += (long long)__float2int_rz(v[q]) << sh;
  } else if constexpr (sh >= 0) {
#pragma unroll
    for (int q = 0; q < C; ++q) acc[q] += (long long)__float2int_rz(v[q]) * (1 << sh);
  } else {
    constexpr float s = 1.0f / (float)(1 << -sh);
#pragma unroll
    for (int q = 0; q < C; ++q) acc[q] += (long long)__float2int_rn(v[q] * s);
  }
}

// RN(v) 2^kx of an int64 v (|v| < 2^63, the result a normal float64 or zero) on 32-bit integer
// operations: the bits of __ll2double_rn(v) with kx added to the exponent.  The FP64 pipe converts one
// value per clock and SM at best; a quarter of the values there and the rest here took 3.5 k clocks for
// a 128 x 64 tile's values against 4.6 k (all FP64) and 5.3 k (oz_to_f64's 64-bit form).
__device__ __forceinline__ double ow_to_f64(long long v, int kx) {
  const uint32_t sg = (uint32_t)(v >> 63);
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
  int ef = 1022 + 63 + kx;
  if (hi == 0) {
    hi = lo;
    lo = 0;
    ef -= 32;
  }
  const int lz = __clz((int)hi);
  hi = __funnelshift_l(lo, hi, lz);  // leading one at bit 63 of hi:lo
  lo <<= (lz & 31);
  // to nearest even at bit 11; a carry out of the top leaves a zero fraction one exponent up
  const uint32_t l2 = lo + 0x3ffu + ((lo >> 11) & 1u);
  const uint32_t c = l2 < lo ? 1u : 0u;
  const uint32_t h2 = hi + c;
  const uint32_t top = (c && h2 == 0) ? (1u << 21) : 0u;
  const uint32_t rl = __funnelshift_r(l2, h2, 11);
  const uint32_t rh = (h2 >> 11) + top + ((uint32_t)(ef - lz) << 20);
  return hi == 0 ? 0.0 : __hiloint2double((int)(rh | (sg & 0x80000000u)), (int)rl);
}

// Persistent warp-specialised GEMM over (parity, m tile, N-column tile): warp 0 streams the stages,
// warp 1 issues the MMAs, warps 2-9 drain (warp w: rows 32 (w % 4).., columns N/2 ((w - 2) / 4).. of every
// weight) and store the tile, its rows transposed through shared memory.  nnt: packed 64-column B tiles.
template <int N>
__global__ void __launch_bounds__(320, 1) oz_wgemm_kernel(const uint8_t *__restrict__ apack,
                                                          const uint8_t *__restrict__ bpack,
                                                          const int *__restrict__ erow, int eB, int nk, int nmt, int nnt,
                                                          int rows, double *__restrict__ y, int ld, int ku, int kv,
                                                          const KrylovScalars *__restrict__ sc, int rpr,
                                                          int *__restrict__ err, int inv) {
  using Cfg = OwCfg<N>;
  constexpr int NST = Cfg::NST, STAGE = Cfg::STAGE, CW = Cfg::CW, CH = Cfg::CH, TPITCH = Cfg::TPITCH;
  constexpr int SUB = OW_N / N;  // tiles per packed B tile
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t *gbase = smem_raw + (base - raw);
  constexpr int BAR_OFF = NST * STAGE + 8 * Cfg::TBUF;
  const uint32_t full0 = base + BAR_OFF, empty0 = full0 + 8 * NST, tfull0 = empty0 + 8 * NST, tempty0 = tfull0 + 24;
  volatile uint32_t *holder = reinterpret_cast<volatile uint32_t *>(gbase + BAR_OFF + 16 * NST + 48);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(gbase + BAR_OFF + 16 * NST + 56);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // column tiles with valid columns, by parity
  const int nt0 = (ku + N - 1) / N, nt1 = ((inv ? ku : kv) + N - 1) / N;
  const int ntiles = nmt * (nt0 + nt1);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)holder)),
                 "r"(Cfg::TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int g = 0; g < 3; ++g) {
      mbar_init(tfull0 + 8 * g, 1);
      mbar_init(tempty0 + 8 * g, 8);  // one arrive per epilogue warp
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  pdl_wait();
  const uint32_t tmem = *holder;

  auto decode = [&](int t, int &par, int &mt, int &nt) {
    par = t >= nmt * nt0;
    const int u = par ? t - nmt * nt0 : t, ntp = par ? nt1 : nt0;
    nt = u % ntp;
    mt = u / ntp;
  };
  auto wanted = [&](int mt) -> bool {  // some row of the tile belongs to a running right-hand side
    if (sc == nullptr) return true;
    const int m0 = mt * TM;
    const int r0 = m0 / rpr, r1 = (min(m0 + TM, rows) - 1) / rpr;
    for (int r = r0; r <= r1; ++r)
      if (sc[r].state == ST_RUN) return true;
    return false;
  };

  if (warp == 0) {
    if (lane == 0) {  // producer
      int s = 0, it = 0;
      uint32_t ph = 0;
      for (int t = blockIdx.x; t < ntiles && !*abort_flag; t += gridDim.x) {
        int par, mt, nt;
        decode(t, par, mt, nt);
        if (!wanted(mt)) continue;
        const uint8_t *at = apack + ((size_t)par * nmt + mt) * nk * OW_A;
        const uint8_t *bt = bpack + ((size_t)par * nnt + nt / SUB) * nk * OW_B + (nt % SUB) * Cfg::BSL;
        for (int k = 0; k < nk; ++k) {
          if (it >= NST && !mbar_wait(empty0 + 8 * s, ph ^ 1u)) {
            atomicExch(err, 11);
            *abort_flag = 1;
            break;
          }
          const uint32_t st = base + s * STAGE, fb = full0 + 8 * s;
          mbar_expect_tx(fb, (uint32_t)STAGE);
          bulk_g2s(st, at + (size_t)k * OW_A, OW_A, fb);
          if constexpr (SUB == 1) {
            bulk_g2s(st + OW_A, bt + (size_t)k * OW_B, OW_B, fb);
          } else {
#pragma unroll
            for (int i = 0; i < OW_NS; ++i)
              bulk_g2s(st + OW_A + i * Cfg::BSL, bt + (size_t)k * OW_B + i * OW_BSL, Cfg::BSL, fb);
          }
          ++it;
          if (++s == NST) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      // only now: blocks of the next kernel that fit beside this one would take issue slots from the MMAs
      pdl_next();
      // after an abort nobody has waited for the last copies: no CTA leaves with copies in flight
      if (*abort_flag)
        for (int i = max(0, it - NST); i < it; ++i) mbar_wait(full0 + 8 * (i % NST), (uint32_t)(i / NST) & 1u);
    }
  } else if (warp == 1) {  // MMA issuer: the loop is uniform over the warp, one lane issues
    const bool lead = elect_one();
    int s = 0;
    uint32_t ph = 0, eph = 0;  // eph: next parity of each group's tempty barrier
    uint32_t pend = 0;         // groups handed to the epilogue and not seen back
    for (int t = blockIdx.x; t < ntiles && !*abort_flag; t += gridDim.x) {
      int par, mt, nt;
      decode(t, par, mt, nt);
      if (!wanted(mt)) continue;
      for (int k = 0; k < nk; ++k) {
        bool ok = mbar_wait(full0 + 8 * s, ph);
        if (!ok && lead) atomicExch(err, 12);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sa = (base + s * STAGE) >> 4, sb = sa + (OW_A >> 4);
        auto wait = [&](int g) {
          const bool got = mbar_wait(tempty0 + 8 * g, (eph >> g) & 1u);
          if (!got && lead) atomicExch(err, 14);
          ok = ok && got;
          eph ^= 1u << g;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        };
        if (k > 0) {
          if (pend == 0) {
            if (lead) ow_issue_all<N>(tmem, sa, sb);
          } else if (pend == 2u) {  // the most frequent drain (weights 5, 6): the other groups meanwhile
            if (lead) {
              ow_issue_group<N, 0, false>(tmem, sa, sb);
              ow_issue_group<N, 2, false>(tmem, sa, sb);
            }
            wait(1);
            if (lead) ow_issue_group<N, 1, false>(tmem, sa, sb);
          } else {
            if (pend & 1u) wait(0);
            if (pend & 2u) wait(1);
            if (pend & 4u) wait(2);
            if (lead) ow_issue_all<N>(tmem, sa, sb);
          }
        } else {  // a tile's first stage starts every sum afresh
          if (pend & 1u) wait(0);
          if (lead) ow_issue_group<N, 0, true>(tmem, sa, sb);
          if (pend & 2u) wait(1);
          if (lead) ow_issue_group<N, 1, true>(tmem, sa, sb);
          if (pend & 4u) wait(2);
          if (lead) ow_issue_group<N, 2, true>(tmem, sa, sb);
        }
        if (!ok) {
          *abort_flag = 1;
          break;
        }
        pend = k + 1 == nk ? 7u : (ow_bit(OW_E0, k + 1) | ow_bit(OW_E1, k + 1) << 1 | ow_bit(OW_E2, k + 1) << 2);
        if (lead) {
          ow_commit(empty0 + 8 * s);
          if (pend & 1u) ow_commit(tfull0);
          if (pend & 2u) ow_commit(tfull0 + 8);
          if (pend & 4u) ow_commit(tfull0 + 16);
        }
        if (++s == NST) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else {  // epilogue warps 2..9
    const int lg = warp & 3, h = (warp - 2) >> 2;
    const uint32_t tw = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(h * CW);  // + N (w - 2)
    double *tbuf = reinterpret_cast<double *>(gbase + NST * STAGE + (warp - 2) * Cfg::TBUF);
    auto hand_back = [&](int g) {
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty0 + 8 * g) : "memory");
    };
    uint32_t fph = 0;  // next parity of each group's tfull barrier
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      int par, mt, nt;
      decode(t, par, mt, nt);
      if (!wanted(mt)) continue;
      const int row = mt * TM + lg * 32 + lane;
      const int e = row < rows ? erow[par * (nmt * TM) + row] : 0;
      long long acc[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) acc[q] = 0;
      bool stop = false;
      for (int c = 1; c <= nk; ++c) {
        const bool last = c == nk;
        if (!last && !ow_bit(OW_E0 | OW_E1 | OW_E2, c)) continue;
        // a group's accumulators: at most two weights in registers at a time, handed back before the
        // last ones are added up
        auto wait_group = [&](int g) {
          const bool ok = mbar_wait(tfull0 + 8 * g, (fph >> g) & 1u);
          fph ^= 1u << g;
          __syncwarp();
          if (!ok) {
            if (lane == 0) atomicExch(err, 13);
            *abort_flag = 1;
            stop = true;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          return ok;
        };
        float va[CW], vb[CW];
        auto take = [&](int w, float (&v)[CW]) {
          ow_tmem_ld<CW>(tw + (w - 2) * N, v);
          if (!last) ow_tmem_zero<CW>(tw + (w - 2) * N);
        };
        if ((last || ow_bit(OW_E0, c)) && !stop && wait_group(0)) {
          if (last) {
            take(2, va);
            ow_add<2>(va, acc);
          }
          take(3, va);
          take(4, vb);
          hand_back(0);
          ow_add<3>(va, acc);
          ow_add<4>(vb, acc);
        }
        if ((last || ow_bit(OW_E1, c)) && !stop && wait_group(1)) {
          take(5, va);
          take(6, vb);
          hand_back(1);
          ow_add<5>(va, acc);
          ow_add<6>(vb, acc);
        }
        if ((last || ow_bit(OW_E2, c)) && !stop && wait_group(2)) {
          take(7, va);
          if (last) take(8, vb);
          hand_back(2);
          ow_add<7>(va, acc);
          if (last) ow_add<8>(vb, acc);
        }
        if (stop) break;
      }
      if (stop) break;
      // the one float64 rounding: int64 -> float64, then exact power-of-two scales (added to the
      // exponent field where every result of the row is a normal float64)
      const int kx = e + eB - 2 * 7 - OW_FIX;
      const bool fast = __all_sync(0xffffffffu, oz_fast_row(e, kx));  // a branch of the whole warp
      const int c0 = nt * N + h * CW;
      const int ncols = min(CW, ((par && !inv) ? kv : ku) - c0);
      const int r0 = mt * TM + lg * 32;
      const int nr = min(32, rows - r0);
      const int ys = inv ? 1 : 2;
      double *yt = y + (inv ? ((size_t)par * rows + r0) * ku + c0 : (size_t)r0 * ld + par + 2 * (size_t)c0);
      const size_t ystep = inv ? (size_t)ku : (size_t)ld;
#pragma unroll
      for (int part = 0; part < CW / CH; ++part) {
        if (fast) {
          // a quarter of the values on the FP64 pipe, the rest on the integer pipe (the same bits)
#pragma unroll
          for (int q = 0; q < CH; ++q) {
            const long long a = acc[part * CH + q];
            double d;
            if ((q & 3) == 0) {
              const long long db = __double_as_longlong(__ll2double_rn(a));
              d = __longlong_as_double(db == 0 ? 0ll : db + ((long long)kx << 52));
            } else {
              d = ow_to_f64(a, kx);
            }
            tbuf[lane * TPITCH + q] = d;
          }
        } else {
          const double scale = e == OZ_EXP_NAN ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, e + eB - 2 * 7);
          const double unit = 1.0 / (double)(1LL << OW_FIX);
#pragma unroll
          for (int q = 0; q < CH; ++q) tbuf[lane * TPITCH + q] = scale * (unit * __ll2double_rn(acc[part * CH + q]));
        }
        __syncwarp();
        const int cq = lane % CH, col = part * CH + cq;
#pragma unroll
        for (int rr = 0; rr < 32; rr += 32 / CH) {
          const int r = rr + lane / CH;
          if (r < nr && col < ncols) yt[(size_t)r * ystep + (size_t)ys * col] = tbuf[r * TPITCH + cq];
        }
        __syncwarp();
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::TMEM) : "memory");
}
