// Panel factor of an inner block (GEQRT / TSQRT / TTQRT) from Gram matrices on the tensor cores, included by kernels.cu.
//
// The factorization column by column is bound by the FP64 units (2 FMA / clock / SM: a 256 x 32 block needs 254k FMA and
// its T factor 131k more, 200k cycles) and by a chain of 32 reductions over the rows.  Here the rows are touched only
// by exact digit products (update_digits.cuh); the 32 steps run on 32 x 32 matrices.  With the columns scaled to
// norms below one (E_c, over the pivot's triangle R and the tile's rows X; GE has no R):
//
//   1. M = R^T R + X^T X.  Its Cholesky factor gives the rows of the new triangle up to signs, R'_j = -sgn(alpha_j) r_j:
//      beta_j = -sgn(alpha_j) ||x_j||, as Householder has it.
//   2. U = R - R' for TS / TT, and for GE L U = A_1 - R' (no pivoting, A_1 the top kb rows): since Q^T [R; X] = [R'; 0]
//      with Q = I - V T V^T means V W2 = [R - R'; X], U is W2 and V = X U^{-1}.  alpha_j is the pivot of the
//      elimination; U_jj = alpha_j - beta_j has no cancellation (reconstructing Householder vectors: Ballard, Demmel,
//      Grigori, Jacquelin, Nguyen, Solomonik, IPDPS 2014).
//   3. V = X U^{-1} as digit products, like an update.
//   4. tau_k = 2 / ||v_k||^2 and T from V^T V (as t_from_gram has it), so that Q is orthogonal to working precision for the V that
//      was stored.
//
// The Gram matrix squares the condition number: an error of 2^-57 in M (the rounding of the 56-bit digits) becomes
// 2^-58 / r_jj in R'.  Blocks in which a column's norm falls below 2^-3.5 of its start under the reflectors before it, in
// which a tail is (nearly) zero (sigma^2 < 2^-20; an exact zero must give H = I), whose U^{-1} exceeds 2^5, or in which X
// has no entry of 2^-8 or a row with no entry above 2^-6 of its largest (2^-10 for a triangle: its rows have their large
// entries on the diagonal, in another block; smaller rows would not be held to their own scale, as in
// update_digits.cuh), are refused before anything is written and factored column by column
// (task_panel_factor); so are the square blocks at a GE panel's end, whose last columns are short.  (Backward error against
// a 113-bit product, 256 rows N(0, 1): 4.6e-16, column by column 8.5e-16; ||Q^T Q - I|| 3e-16 against 8e-16.)

#if BD_EXEC_PART == 1
constexpr int kPanR = kDigC;                        // byte offsets: R's digits (32 rows, 2048 bytes a digit),
constexpr int kPanP = kPanR + 8 * 2048;             // partial sums of a Gram matrix,
constexpr int kPanW = kPanP + 4 * kDigPStride;      // digits of U^{-1},
constexpr int kPanG = kPanW + 8 * 2048;             // U, later V^T V, and scratch (FP64),
constexpr int kPanT = kPanG + 2 * 8192;             // U in fixed point, later U^{-1}, T (FP64),
constexpr int kPanB = kPanT + 8192;                 // the top rows, later the columns of L U_jj,
constexpr int kPanRow = kPanB + kDigPStride;        // the rows r_j of the Cholesky factor (split)
static_assert(kPanRow + 8192 <= kDigHead, "panel scratch fits");
static_assert((kPanR & 511) == 0 && (kPanW & 127) == 0, "operand alignment");

// a b 2^-62 for |a|, |b| < 2^62
__device__ __forceinline__ int64_t mul62(int64_t a, int64_t b) { return __mul64hi(a << 1, b << 1); }
// 1 / x for normal x, from the FP32 reciprocal (e = 1 - x y below 2^-21) by the series of (1 - e)^-1 up to e^2
__device__ __forceinline__ double recip_series(double x) {
  const double y = (double)__frcp_rn((float)x), e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float rsqrt_approx(float x) {     // (rsqrtf, for normal x)
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// m^(-1/2) 2^58 for m = x 2^-62 in [2^-7, 1): y0 = Y 2^-20 from the FP32 approximation, then y0 (1 - e)^(-1/2) with
// e = 1 - m y0^2 (below 2^-18) up to e^2.  Integers: a chain of FP64 operations on one warp takes about 2k cycles here.
__device__ __forceinline__ int64_t rsqrt_q58(int64_t x) {
  const float f = (float)(uint32_t)(x >> 31) * 0x1p-31f;
  const uint32_t Y = __float2uint_rn(rsqrt_approx(f) * 0x1p20f);
  const int64_t e = ((int64_t)1 << 56) - (int64_t)__umul64hi((uint64_t)x << 2, ((uint64_t)Y * Y) << 16);
  const int es = (int)(e >> 8);
  const int64_t c = (e >> 1) + ((3 * (((int64_t)es * es) >> 3)) >> 40);
  return ((int64_t)Y << 38) + (((int64_t)Y * c) >> 18);
}
// u^-1 2^57 for |u| = |x| 2^-61 in [2^-4, 2): the same with y0 = R 2^-19 and e = 1 - |u| y0
__device__ __forceinline__ int64_t recip_q57(int64_t x) {
  const uint64_t a = x < 0 ? (uint64_t)0 - (uint64_t)x : (uint64_t)x;
  const uint32_t R = __float2uint_rn(__fdividef(1.0f, (float)(uint32_t)(a >> 30) * 0x1p-31f) * 0x1p19f);
  const int64_t e = ((int64_t)1 << 58) - (int64_t)__umul64hi(a << 2, (uint64_t)R << 40);
  const int es = (int)(e >> 10);
  const int64_t c = e + (((int64_t)es * es) >> 38);
  const int64_t y = ((int64_t)R << 38) + (((int64_t)R * (c >> 2)) >> 18);
  return x < 0 ? -y : y;
}
// Operands of a product of two 64-bit fixed-point numbers split as x = h 2^31 + l: three 32-bit multiplications, the
// fourth (l l, below one unit of the result) is left out unless the result keeps more than the upper half.
__device__ __forceinline__ int2 split31(int64_t x) { return make_int2((int)(x >> 31), (int)x & 0x7fffffff); }
__device__ __forceinline__ int64_t mul_hi62(int2 a, int2 b) {       // a b 2^-62
  return wide(a.x, b.x, wide(a.x, b.y, (int64_t)a.y * b.x) >> 31);
}
__device__ __forceinline__ int64_t mul_hi57(int2 a, int2 b) {       // a b 2^-57
  const int64_t mid = wide(a.x, b.y, wide(a.y, b.x, ((int64_t)a.y * b.y) >> 31));
  return (int64_t)((uint64_t)((int64_t)a.x * b.x) << 5) + (mid >> 26);
}

// Factors inner block b of a panel task as task_panel_factor does, and publishes it in vd if that is given; false:
// refused, nothing written.
__device__ __noinline__ bool task_panel_digits(unsigned char* sm, int kind, double* X, double* A, int tr, double* Tg, int nb,
                                               int ib, int b, unsigned char* vd, Umma& um, const ExecParams& prm) {
  if ((smem_u32(sm) & 511) || (kind == PM_GE && (b + 1) * ib == nb)) return false;
  if ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(A)) & 15) return false;      // 16-byte loads and stores
  int* colE = reinterpret_cast<int*>(sm + kDigHead);                     // E_c
  uint32_t* red = reinterpret_cast<uint32_t*>(sm + kDigHead + 128);      // reduction scratch of column_exponents, then:
  int64_t* dinv = reinterpret_cast<int64_t*>(red);                       //   1 / U_jj (2^57),
  double* diag = reinterpret_cast<double*>(dinv + 32);                   //   1 / U_jj, later tau,
  int* colS = reinterpret_cast<int*>(diag + 32);                         //   exponents of U^{-1}'s columns,
  int* neg = colS + 32;                                                  //   whether alpha_j < 0,
  int* refuse = neg + 32;
  int64_t* P = reinterpret_cast<int64_t*>(sm + kPanP);
  double* G = reinterpret_cast<double*>(sm + kPanG);
  int64_t* Uf = reinterpret_cast<int64_t*>(sm + kPanT);
  int64_t* Bs = reinterpret_cast<int64_t*>(sm + kPanB);
  double* Td = reinterpret_cast<double*>(sm + kPanT);
  int2* Rw = reinterpret_cast<int2*>(sm + kPanRow);
  int2* Ww = reinterpret_cast<int2*>(P);                                 // rows U_j / U_jj (2^57, split)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kb = ib, c0 = b * ib, r = tid & 255, ch = tid >> 8, cb = 16 * ch, hw = r >> 7;
  const int uwarp = (int)uniform(warp);
  const bool ge = kind == PM_GE, tt = kind == PM_TT;
  const int row_lo = ge ? c0 : 0, row_hi = tt ? c0 + kb : nb;
  const bool own = r >= row_lo && r < row_hi;
  const int ti = ge ? r - c0 : r;                    // row of the top block (GE: this row of X; TS / TT: of R)
  const bool is_top = ti >= 0 && ti < kb;

  // ---- load, E_c --------------------------------------------------------------------------------
  uint32_t* rows = reinterpret_cast<uint32_t*>(sm + kPanG);
  uint32_t big = 0;                    // largest |X| of the thread's half row
  int64_t cf[16];
  {
    auto load_row = [&](const double* src, int row, bool on, int64_t* v) {
      if (tr) {
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          double2 d = make_double2(0.0, 0.0);
          if (on && cb + c < kb) d = __ldcg(reinterpret_cast<const double2*>(src + (size_t)row * nb + c0 + cb + c));
          v[c] = __double_as_longlong(d.x);
          v[c + 1] = __double_as_longlong(d.y);
        }
      } else {
#pragma unroll
        for (int c = 0; c < 16; ++c)
          v[c] = __double_as_longlong((on && cb + c < kb) ? ldg(src + row + (size_t)(c0 + cb + c) * nb) : 0.0);
      }
    };
    load_row(X, r, own, cf);
    if (tt) {
#pragma unroll
      for (int c = 0; c < 16; ++c) cf[c] = r > c0 + cb + c ? 0 : cf[c];
    }
    int64_t cq[16];
    load_row(A, c0 + r, !ge && r < kb, cq);
#pragma unroll
    for (int c = 0; c < 16; ++c) cq[c] = r > cb + c ? 0 : cq[c];          // R's upper triangle (r < kb)
    int E;
    bool zero;
    if (!column_exponents(cf, cq, colE, red, &E, &zero, cb + (lane & 15) >= kb)) return false;
    for (int o = tid; o < 32 * 33; o += kThreads) Bs[o] = 0;
    __syncthreads();
    if (tid == 0) *refuse = 0;
    bool nz = false;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int sh = 63 - __shfl_sync(kFull, E, c);
      nz = nz || cf[c] << 1 != 0;
      cf[c] = to_fixed(__longlong_as_double(cf[c]), sh);
      cq[c] = to_fixed(__longlong_as_double(cq[c]), sh);
      big = max(big, abs_hi(cf[c]));
      if (is_top) Bs[ti * 33 + cb + c] = (ge ? cf[c] : cq[c]) >> 2;       // 2^61
    }
    const uint32_t wmax = __reduce_max_sync(kFull, big);
    const unsigned any = __ballot_sync(kFull, nz);
    if (lane == 0) {
      rows[warp] = wmax;
      rows[16 + warp] = any;
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) put_digits(sm + kDigV, r, 2 * ch + g, cf + 8 * g);
    if (!ge && r < 32) {
#pragma unroll
      for (int g = 0; g < 2; ++g) put_digits(sm + kPanR, r, 2 * ch + g, cq + 8 * g, 2048);
    }
  }
  const uint32_t uV = uniform(smem_u32(sm + kDigV)), uR = uV + kPanR, uW = uV + kPanW, utm = uniform(um.tmem);
  const uint32_t tq = um.tmem + ((uint32_t)((warp & 3) * 32) << 16);
  bool ok = true;
  auto fence_sync = [&]() {          // generic shared-memory writes -> MMA reads
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  // Gram matrix of the rows in the V area (and of R's digits)
  auto gram = [&](bool with_r) {
    if (uwarp == kIssueWarp) {
      const uint32_t i0 = umma_idesc_f16(128, 32 * kDigN, true, true), i1 = umma_idesc_f16(128, 128, true, true);
      const int k0 = uniform(row_lo >> 4), k1 = uniform((row_hi + 15) >> 4);
      const uint64_t d = digit_desc(uV + k0 * 1024, kDigSlice), dr = digit_desc(uR, 2048);
#pragma unroll 4
      for (int k = 0; k < k1 - k0; ++k) {
        umma_f16(utm, d + k * 64, d + k * 64, i0, k > 0);
        umma_f16(utm + 256, d + (4 * kDigSlice >> 4) + k * 64, d + k * 64, i1, k > 0);
      }
      if (with_r) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          umma_f16(utm, dr + k * 64, dr + k * 64, i0, 1);
          umma_f16(utm + 256, dr + (4 * 2048 >> 4) + k * 64, dr + k * 64, i1, 1);
        }
      }
      umma_commit(um.mbar);
    }
    ok = mbar_wait(um.mbar, um.phase & 1u, prm.wait_ns) && ok;
    um.phase ^= 1u;
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  // a completion wait ran out: the error word is set, the MMAs in flight are waited for, nothing more is written
  auto fail = [&]() {
    if (tid == 0) atomicCAS(prm.err, 0, DERR_TIMEOUT);
    for (int i = 0; i < 3; ++i) mbar_wait(um.mbar + 8 * i, ((um.phase >> i) & 1u) ^ 1u, prm.wait_ns);
    wait_image();
    __syncthreads();
    return true;
  };
  const int arow = 2 * warp;          // thread (warp, lane): rows arow, arow + 1 of column lane of the 32 x 32 matrices
  auto sum_partials = [&](int row) {
    const int o = row * 33 + lane;
    return P[o] + P[o + 32 * 33] + P[o + 64 * 33] + P[o + 96 * 33];
  };

  // ---- M = R^T R + X^T X (2^62) -------------------------------------------------------------------
  fence_sync();
  {                                    // rows of another scale (every warp finds the same)
    const uint32_t xmax = __reduce_max_sync(kFull, rows[lane & 15]);
    const unsigned strong = __ballot_sync(kFull, big >= xmax >> (tt ? 10 : 6));
    if (lane == 0) rows[32 + warp] = strong;
    __syncthreads();
    const int w = lane & 7;
    const uint32_t weak = (rows[16 + w] | rows[24 + w]) & ~(rows[32 + w] | rows[40 + w]);
    if (xmax < kSmallRow || __any_sync(kFull, weak != 0)) return false;
  }
  gram(!ge);
  gram_partials<true>(P, tq, 24);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (!__syncthreads_and(ok ? 1 : 0)) return fail();
  // ---- Cholesky of M with the elimination of the top block -------------------------------------------
  // Stage s (one barrier each) takes steps j = 2 s and j + 1.  Warp 0 runs the chain: it applies the pair before to rows
  // j, j + 1 and forms r, U and U / U_jj of both.  The other warps apply that pair to the rows below, two a warp, and
  // the owner of the next pair hands its rows over, so the chain (its latencies: about 220 cycles for a reciprocal
  // square root, 190 for a reciprocal) runs beside their work.  Rows 0 .. 7, done with first, are on warp 0's
  // scheduler.  (Every warp forming its own rows of r and U after a barrier a step: 56.7k cycles for a GE block and 28k for TS,
  // against 37k and 23k.)
  const int pr = (warp & 3) == 0 ? warp >> 2 : 3 + 3 * (warp >> 2) + (warp & 3), erow = 2 * pr;
  int64_t m[2], bt[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    m[k] = sum_partials(erow + k);
    bt[k] = Bs[(erow + k) * 33 + lane];
  }
  __syncthreads();
  int64_t* H = reinterpret_cast<int64_t*>(sm + kPanG);       // rows handed over: two buffers of m, m, bt, bt
  auto eliminate = [&](auto is_ge) {
    constexpr bool kGe = decltype(is_ge)::value;
    const int2 zero = make_int2(0, 0);
    if (warp == 0) {
      int2 rs[2] = {zero, zero}, ws[2] = {zero, zero};
#pragma unroll 1
      for (int j = 0; j < kb; j += 2) {
        if (j > 0) {
          const int64_t* h = H + (j & 2) * 64 + lane;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            m[k] = h[32 * k];
            bt[k] = h[64 + 32 * k];
          }
#pragma unroll
          for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
              m[k] -= mul_hi62(make_int2(__shfl_sync(kFull, rs[q].x, j + k), __shfl_sync(kFull, rs[q].y, j + k)), rs[q]);
            if (kGe) {
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                const int64_t bij = __shfl_sync(kFull, bt[k], j - 2 + q);
                if (lane == 0) Bs[(j + k) * 33 + j - 2 + q] = bij;       // l_ij U_jj
                bt[k] -= mul_hi57(split31(bij), ws[q]);
              }
            }
          }
        }
        const int64_t m0 = __shfl_sync(kFull, m[0], j), al0 = __shfl_sync(kFull, bt[0], j);
        const int64_t rc0 = __mul64hi(m[0] << 1, rsqrt_q58(m0) << 1) << 4;               // 2^62
        rs[0] = lane > j ? split31(rc0) : zero;
        m[1] -= mul_hi62(make_int2(__shfl_sync(kFull, rs[0].x, j + 1), __shfl_sync(kFull, rs[0].y, j + 1)), rs[0]);
        const int64_t m1 = __shfl_sync(kFull, m[1], j + 1), y1 = rsqrt_q58(m1);
        const int64_t u0 = bt[0] - (al0 < 0 ? rc0 >> 1 : -(rc0 >> 1));                   // 2^61
        int64_t d0 = 0, b10 = 0;
        if (kGe) {
          d0 = recip_q57(__shfl_sync(kFull, u0, j));                                     // |d| < 2^(57 + 3.5)
          ws[0] = lane > j ? split31(__mul64hi(u0 << 1, d0 << 2)) : zero;
          b10 = __shfl_sync(kFull, bt[1], j);
          bt[1] -= mul_hi57(split31(b10), ws[0]);
        }
        const int64_t rc1 = __mul64hi(m[1] << 1, y1 << 1) << 4;
        const int64_t al1 = __shfl_sync(kFull, bt[1], j + 1);
        const int64_t u1 = bt[1] - (al1 < 0 ? rc1 >> 1 : -(rc1 >> 1));
        rs[1] = lane > j + 1 ? split31(rc1) : zero;
        int64_t d1 = 0;
        if (kGe) {
          d1 = recip_q57(__shfl_sync(kFull, u1, j + 1));
          ws[1] = lane > j + 1 ? split31(__mul64hi(u1 << 1, d1 << 2)) : zero;
          Ww[j * 32 + lane] = ws[0];
          Ww[j * 32 + 32 + lane] = ws[1];
        }
        Rw[j * 32 + lane] = lane == j ? split31(rc0) : rs[0];
        Rw[j * 32 + 32 + lane] = lane == j + 1 ? split31(rc1) : rs[1];
        Uf[j * 32 + lane] = u0;
        Uf[j * 32 + 32 + lane] = u1;
        if (lane == 0) {
          if (kGe) {
            Bs[(j + 1) * 33 + j] = b10;
            dinv[j] = d0;
            dinv[j + 1] = d1;
          }
          neg[j] = al0 < 0;
          neg[j + 1] = al1 < 0;
          if (min(m0, m1) < (int64_t)1 << 55 || min(m0 - mul62(al0 << 1, al0 << 1), m1 - mul62(al1 << 1, al1 << 1)) < (int64_t)1 << 42)
            *refuse = 1;
        }
        __syncthreads();
      }
    } else {
#pragma unroll 1
      for (int j = 0; j < kb; j += 2) {
        if (erow > j && j > 0) {             // steps j - 2 and j - 1
#pragma unroll
          for (int q = j - 2; q < j; ++q) {
            const int2 rb = Rw[q * 32 + lane];
            const int4 ra = *reinterpret_cast<const int4*>(Rw + q * 32 + erow);
            m[0] -= mul_hi62(make_int2(ra.x, ra.y), rb);
            m[1] -= mul_hi62(make_int2(ra.z, ra.w), rb);
            if (kGe) {
              const int2 wb = Ww[q * 32 + lane];
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                const int64_t bij = __shfl_sync(kFull, bt[k], q);
                if (lane == 0) Bs[(erow + k) * 33 + q] = bij;
                bt[k] -= mul_hi57(split31(bij), wb);
              }
            }
          }
        }
        if (erow == j + 2) {
          int64_t* h = H + (erow & 2) * 64 + lane;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            h[32 * k] = m[k];
            h[64 + 32 * k] = bt[k];
          }
        }
        __syncthreads();
      }
    }
  };
  if (ge) eliminate(std::true_type{});
  else eliminate(std::false_type{});
  if (*refuse) return false;           // (uniform: not written again)
  // ---- U^{-1}, its digits ------------------------------------------------------------------------
#pragma unroll
  for (int k = 0; k < 2; ++k)
    G[arow + k + lane * 32] = (lane > arow + k && lane < kb) ? from_fixed(Uf[(arow + k) * 32 + lane], 61) : 0.0;
  if (tid < 32) diag[tid] = tid < kb ? recip_series(from_fixed(Uf[tid * 33], 61)) : 0.0;
  __syncthreads();
  inverse32(G, diag, Td, G + 1024);
  {
    const double s0 = Td[arow + lane * 32], s1 = Td[arow + 1 + lane * 32];
    uint32_t* hmax = reinterpret_cast<uint32_t*>(P);        // [warp][column]
    uint32_t h = max((uint32_t)__double2hiint(s0) & 0x7fffffffu, (uint32_t)__double2hiint(s1) & 0x7fffffffu);
    hmax[warp * 32 + lane] = h;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kWarps; ++q) h = max(h, hmax[q * 32 + lane]);
    const int eS = max((int)((h + (1u << 14)) >> 20) - 1022, 0);      // |s| < 0.992 x 2^eS
    if (__syncthreads_or(eS > 5)) return false;
    if (warp == 0) colS[lane] = eS;
    uint32_t d[8];
    digit_pair<8>(to_fixed(s0, 63 - eS), to_fixed(s1, 63 - eS), d);
    unsigned char* p = sm + kPanW + (lane >> 3) * 512 + (lane & 7) * 16 + (arow >> 3) * 128 + (arow & 7) * 2;
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<uint32_t*>(p + i * 2048) = d[i];
  }
  // the new triangle
  double* Tri = ge ? X : A;
  for (int o = tid; o < 1024; o += kThreads) {
    const int i = tr ? o >> 5 : o & 31, c = tr ? o & 31 : o >> 5;
    if (i <= c && c < kb) {
      const int64_t v = wide(Rw[i * 32 + c].x, 1 << 30, 0) * 2 + Rw[i * 32 + c].y;   // R' 2^(62 - E_c) up to its row's sign
      stg(Tri + toff(c0 + i, c0 + c, nb, tr), from_fixed(neg[i] ? v : -v, 62 - colE[c]));
    }
  }
  fence_sync();
  // ---- V = X U^{-1} ------------------------------------------------------------------------------
  const int h0 = row_lo >> 7, h1 = (row_hi + 127) >> 7;
  if (uwarp == kIssueWarp) {
    const int uh0 = uniform(h0), uh1 = uniform(h1);
    const uint64_t da = digit_desc(uV, 16), db = umma_desc(uW, 128, 512);
    for (int h = uh0; h < uh1; ++h) {
#pragma unroll
      for (int j = 0; j < kDigN; ++j)
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
          umma_f16(utm + 256 * h + 32 * j, da + ((j * kDigSlice + ks * 32) >> 4) + h * 512, db + ks * 16,
                   umma_idesc_f16(128, 32 * (8 - j), false, false), j + ks > 0);
      umma_commit(um.mbar + 8 + 8 * h);
    }
  }
  if (hw >= h0 && hw < h1) {           // warp-uniform
    ok = mbar_wait(um.mbar + 8 + 8 * hw, (um.phase >> (1 + hw)) & 1u, prm.wait_ns);
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int cg = 0; cg < 16; cg += 4) {
      uint32_t d[8][4];
#pragma unroll
      for (int g = 0; g < 8; ++g) tmem_ld4(tq + 256 * hw + 32 * g + cb + cg, d[g]);
      tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < 4; ++c) {    // V 2^62 = sum of D_g 2^(48 - 8 g + eS)
        const int eS = colS[cb + cg + c];
        const int64_t H = wide(int_of(d[0][c]) * 256 + int_of(d[1][c]), 65536, int_of(d[2][c]) * 256 + int_of(d[3][c]));
        const int64_t L = wide(int_of(d[4][c]) * 256 + int_of(d[5][c]), 65536, int_of(d[6][c]) * 256 + int_of(d[7][c]));
        cf[cg + c] = own ? (int64_t)((uint64_t)H << (24 + eS)) + (L >> (8 - eS)) : 0;
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  for (int h = h0; h < h1; ++h) um.phase ^= 2u << h;
  if (ge && is_top) {
    const int64_t one = ((int64_t)1 << 62) - 1;
#pragma unroll
    for (int c = 0; c < 16; ++c)
      // l = (l U_jj) / U_jj, not above 1 in magnitude
      cf[c] = cb + c < ti ? min(max((int64_t)__mul64hi(Bs[ti * 33 + cb + c] << 2, dinv[cb + c] << 2) << 4, -one), one)
                          : (cb + c == ti ? one + 1 : 0);
  }
  bool nz = false, strong = false;     // V has an entry in the thread's half row, one of 2^-8 beside the unit entry
  if (own && ok) {
#pragma unroll
    for (int c = 0; c < 16; c += 2) {
      const int d = r - (c0 + cb + c);                    // below (> 0) the diagonal of the block's columns
      const bool on = cb + c < kb, w0 = on && (ge ? d > 0 : (!tt || d <= 0)), w1 = on && (ge ? d > 1 : (!tt || d <= 1));
      double* p = X + toff(r, c0 + cb + c, nb, tr);
      const double x = from_fixed(cf[c], 62), y = from_fixed(cf[c + 1], 62);
      nz = nz || (abs_hi(x) | abs_hi(y)) != 0;
      strong = strong || (abs_hi(x) >= kStrong && !(ge && d == 0)) || (abs_hi(y) >= kStrong && !(ge && d == 1));
      cf[c] = to_fixed(x, 62);                            // V as it is stored
      cf[c + 1] = to_fixed(y, 62);
      if (tr && w0 && w1) {
        __stcg(reinterpret_cast<double2*>(p), make_double2(x, y));
      } else {
        if (w0) stg(p, x);
        if (w1) stg(p + (tr ? 1 : nb), y);
      }
    }
  }
#pragma unroll
  for (int g = 0; g < 2; ++g) put_digits(sm + kDigV, r, 2 * ch + g, cf + 8 * g);
  // ---- V^T V (2^61), tau, T ------------------------------------------------------------------------
  fence_sync();
  if (vd) store_image(sm, vd, nb);
  gram(false);
  gram_partials<false>(P, tq, 25);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (!__syncthreads_and(ok ? 1 : 0)) return fail();
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double v = from_fixed(sum_partials(arow + k), 61);
    G[arow + k + lane * 32] = v;
  }
  __syncthreads();
  if (tid < 32) diag[tid] = tid < kb ? 2.0 * recip_series(ge ? G[tid * 33] : 1.0 + G[tid * 33]) : 0.0;
  inverse32(G, diag, Td, G + 1024);
  for (int o = tid; o < kb * kb; o += kThreads)
    stg(Tg + (size_t)c0 * ib + o, Td[kb == 32 ? o : o % kb + o / kb * 32]);
  if (vd) {
    const double t[2] = {Td[arow + lane * 32], Td[arow + 1 + lane * 32]};
    publish_t(vd, nb, t, true, nz, strong, reinterpret_cast<uint32_t*>(colS));
    wait_image();
  }
  __syncthreads();
  return true;
}
#endif  // BD_EXEC_PART == 1
