// FP64 block updates on the 5th-generation tensor cores (tcgen05, kind::f16), included by kernels.cu.
//
// GB300 issues 2 FP64 FMA per clock and SM, and its FP64 and INT8 tensor rates are no better, while the
// f16 tensor pipe does 4096 multiply-adds per clock and SM.  The two contractions of a block update,
// W = Ct + V^T C and C -= V W2, therefore run as exact integer products of 8-bit digits, the error-free
// splitting of Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012):
//
//  * an operand is a 64-bit integer x 2^s (fixed point); its bytes, made signed (digit = byte - 128 after
//    adding 0x80 to every byte), are integers in [-128, 127], exact in f16;
//  * a product of two digits is below 2^14 in magnitude, a sum over 256 rows below 2^22, and up to eight
//    such products over 32 reflectors below 2^22 too: the FP32 accumulators in TMEM hold them exactly;
//  * the digit products are put together in 64-bit integers.
//
// Fixed point.  Column c of the strip has the exponent E_c, the smallest with 1.03 ||[Cp; C](:, c)||_2 < 2^E_c
// over all rows the task touches; the column's norm does not change under the reflectors, so every
// intermediate entry fits C 2^(63 - E_c) in an int64 for the whole task.  Its seven upper digits carry
// 2^-56 of the column's norm, and the updates are exact integer subtractions on all 63 bits, so a column is
// rounded once per task when it is stored instead of once per multiply-add.  V is scaled by the block's
// largest exponent eV (|v| < 2^eV <= 2), T by its largest (eT).  With ||v_k||^2 = 2 / tau_k <= 2:
// |W| <= 1.42 N_c and |W2| <= 2 N_c.  Digit pairs (i, j) with i + j >= 8 are left out (below 2^-60 N_c).
//
// Columns that are not finite, or outside [2^-958, 2^977], and blocks whose V or T are out of range are
// refused; the caller runs them on the FP64 units (task_update).
//
// Layout.  Thread t owns row t of the strip (all columns, int64 in registers): TMEM lane = row, so the
// product V W2 arrives where it is subtracted, and the new digits of the row go to shared memory as 16-byte
// core-matrix rows.  V and C digits: element (row r, digit d, column k) at ((4 d + k / 8) 256 + r) 16 + 2 (k % 8)
// bytes.  For V^T C both operands are read M/N-major from it (M = (digit, reflector), N = (digit, column)), for
// V W2 the same V is read K-major (M = row, K = reflector).

// ---- instruction and layout helpers ---------------------------------------------------------------
constexpr int kDigRows = 256;                       // rows (threads) of the layout
constexpr int kDigSlice = 4 * kDigRows * 16;        // bytes of one digit of 256 rows x 32 columns
constexpr int kDigN = 7;                            // digits of V and C
constexpr int kDigV = 0;                            // byte offsets: V digits,
constexpr int kDigC = kDigN * kDigSlice;            // C digits; when phase 1 is done the same area holds
constexpr int kDigRaw = kDigC;                      //   the next block's V as stored (64 KB),
constexpr int kDigP = kDigRaw + 65536;              //   the partial sums of W: 4 x 32 x 33 int64,
constexpr int kDigPStride = 32 * 33 * 8;            //   (slot 0 then holds W, W2's digits follow it)
constexpr int kDigW2 = kDigP + kDigPStride;
constexpr int kDigT = kDigP + 4 * kDigPStride;      //   and op(T), 32 rows of 34 (two int32 each)
constexpr int kDigBytes = 2 * kDigN * kDigSlice;
static_assert(kDigW2 + 8 * 2048 <= kDigP + 4 * kDigPStride, "W2 digits fit beside W");
static_assert(kDigT + 32 * 34 * 8 <= kDigBytes, "T fits");
static_assert((kDigW2 & 127) == 0, "operand alignment");
constexpr int kDigTmem = 512;

__host__ __device__ constexpr uint32_t umma_idesc_f16(int m, int n, bool a_mn, bool b_mn) {
  return (1u << 4) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// Integer value of an exact FP32 integer |x| <= 2^22 (adding 1.5 x 2^23 puts it into the low mantissa bits).
constexpr uint32_t kMagicBits = 0x4B400000u;
__device__ __forceinline__ uint32_t mag(uint32_t f) { return __float_as_uint(__uint_as_float(f) + 12582912.0f); }
__device__ __forceinline__ int int_of(uint32_t f) { return (int)(mag(f) - kMagicBits); }
__device__ __forceinline__ int64_t wide(int a, int b, int64_t c) { return (int64_t)a * b + c; }
// x 2^s for -63 <= s <= 63
__device__ __forceinline__ int64_t shl_signed(int64_t x, int s) { return s >= 0 ? (int64_t)((uint64_t)x << s) : x >> -s; }

// x 2^sh rounded to an integer (x finite; sh = 63 - E with |x| < 2^E, so the result is below 2^63)
__device__ __forceinline__ int64_t to_fixed(double x, int sh) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ff);
  uint64_t m = ((uint64_t)((hi & 0xfffff) | 0x100000) << 32 | lo) << 10;   // |x| = m 2^(e - 1085)
  const int t = 1085 - e - sh;                                           // >= 0: the result is m >> t
  m = (t < 64 && e > 0) ? (m + (((uint64_t)1 << t) >> 1)) >> t : 0;
  return (int32_t)hi < 0 ? -(int64_t)m : (int64_t)m;
}
// v 2^-sh rounded to FP64 (the result is a normal number or zero)
__device__ __forceinline__ double from_fixed(int64_t v, int sh) {
  const uint64_t a = v < 0 ? (uint64_t)0 - (uint64_t)v : (uint64_t)v;
  const int z = __clzll((long long)a);
  const uint64_t n = a << (z & 63);                       // leading bit at 63
  const uint64_t q = (n >> 11) + ((n >> 10) & 1);         // 53 bits, rounded; a carry moves into the exponent
  const uint64_t bits = ((uint64_t)(1023 + 63 - z - sh - 1) << 52) + q;
  const uint64_t s = a == 0 ? 0 : bits | (v < 0 ? (uint64_t)1 << 63 : 0);
  return __longlong_as_double((long long)s);
}

// Digits [J0, J0 + ND) (0 = most significant) of eight fixed-point values, as f16 pairs: 16 bytes per digit.
template <int ND>
__device__ __forceinline__ void digits8(const int64_t* x, uint4* d) {
  uint32_t w[ND][4];
  const uint32_t k64 = 0x64646464u;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint64_t y0 = (uint64_t)x[2 * p] + 0x8080808080808080ull, y1 = (uint64_t)x[2 * p + 1] + 0x8080808080808080ull;
    const uint32_t h0 = (uint32_t)(y0 >> 32), h1 = (uint32_t)(y1 >> 32), l0 = (uint32_t)y0, l1 = (uint32_t)y1;
    const uint32_t hu = __byte_perm(h0, h1, 0x7362), hl = __byte_perm(h0, h1, 0x5140);
    const uint32_t lu = __byte_perm(l0, l1, 0x7362), ll = __byte_perm(l0, l1, 0x5140);
    uint32_t r[8];
    r[0] = __byte_perm(hu, k64, 0x4342);   // 1024 + byte, as f16 bits, of both values
    r[1] = __byte_perm(hu, k64, 0x4140);
    r[2] = __byte_perm(hl, k64, 0x4342);
    r[3] = __byte_perm(hl, k64, 0x4140);
    r[4] = __byte_perm(lu, k64, 0x4342);
    r[5] = __byte_perm(lu, k64, 0x4140);
    r[6] = __byte_perm(ll, k64, 0x4342);
    r[7] = __byte_perm(ll, k64, 0x4140);
#pragma unroll
    for (int j = 0; j < ND; ++j)           // minus 1152: the signed digit
      asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(w[j][p]) : "r"(r[j]), "r"(0x64806480u));
  }
#pragma unroll
  for (int j = 0; j < ND; ++j) d[j] = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
}

// Sum over the 32 lanes of v[k], left in lane k (k < 32).
__device__ __forceinline__ float transpose_sum(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const bool up = lane & s;
#pragma unroll
    for (int k = 0; k < s; ++k) {
      const float mine = up ? v[k + s] : v[k], other = up ? v[k] : v[k + s];
      v[k] = mine + __shfl_xor_sync(kFull, other, s);
    }
  }
  return v[0];
}

// Whether a block update of these sizes takes this path.  Its cost per block hardly depends on the
// block (about 13k cycles for 256 rows), the FP64 units need rows x ib x columns cycles.
__host__ __device__ inline bool digits_fit(int nb, int ib, int ncols) {
  return nb % 8 == 0 && nb <= kDigRows && ib % 8 == 0 && ib <= 32 && ncols % 8 == 0 && ncols <= 32 && nb * ib >= 1024;
}

// task_update on the digit path: returns the number of blocks applied (from the first in the order of
// application; C and Cp are up to date for them), the rest being out of the path's range.  Arguments as
// task_update.
__device__ __noinline__ int task_update_digits(unsigned char* smb, int type, const double* X, double* Cp, double* C, int tr,
                                  bool notrans, const double* Tg, int nb, int ib, int blk0, int blk1, int col0,
                                  int ncols, Umma& um, const ExecParams& prm) {
  unsigned char* sm = smb + kHeaderDoubles * sizeof(double);
  int* colE = reinterpret_cast<int*>(smb);                       // E_c
  uint32_t* red = reinterpret_cast<uint32_t*>(smb + 128);        // 8 x 32 reduction scratch
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kb = ib, r = tid;
  const bool top = type != UNMQR;
  const int row_lo = (type == UNMQR) ? blk0 * ib : 0, row_hi = (type == TTMQR) ? blk1 * ib : nb;
  const bool own = r >= row_lo && r < row_hi;
  const int nbk = blk1 - blk0;
  auto blk_of = [&](int bb) { return notrans ? blk1 - 1 - bb : blk0 + bb; };

  // V block of the next application, as stored, into the staging area: column-major (ld 256) for tr = 0, rows of
  // 256 bytes with their 16-byte pieces permuted by the row for tr = 1
  auto prefetch_v = [&](int c0) {
    const int r0 = type == UNMQR ? c0 : 0, r1 = type == TTMQR ? c0 + kb : nb;
    if (!tr) {
      for (int a = warp; a < kb; a += kWarps)
        for (int q = r0 + 2 * lane; q < r1; q += 64)
          cp_async16(sm + kDigRaw + (a * kDigRows + q) * 8, X + q + (size_t)(c0 + a) * nb);
    } else {
      const int np = kb >> 1, ln = tid & 15;
      if (ln < np)
        for (int q = r0 + (tid >> 4); q < r1; q += kThreads >> 4)
          cp_async16(sm + kDigRaw + q * 256 + ((ln ^ (q & 7)) << 4), X + (size_t)q * nb + c0 + 2 * ln);
    }
    cp_async_commit();
  };
  // T of a block: entries tid + 256 k of the kb x kb block as stored
  double tv[4];
  auto load_t = [&](int c0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int o = tid + k * kThreads;
      tv[k] = o < kb * kb ? ldg(Tg + (size_t)c0 * ib + o) : 0.0;
    }
  };
  // the pivot tile's rows of a block: thread (warp g, lane c) has rows 2g, 2g + 1, 30 - 2g, 31 - 2g of column c
  const int arow[4] = {2 * warp, 2 * warp + 1, 30 - 2 * warp, 31 - 2 * warp};
  double ct[4] = {0.0, 0.0, 0.0, 0.0};
  auto load_ct = [&](int c0) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      ct[k] = (top && lane < ncols && arow[k] < kb) ? ldg(Cp + toff(c0 + arow[k], col0 + lane, nb, tr)) : 0.0;
  };

  prefetch_v(blk_of(0) * ib);

  // ---- load the strip, find E_c -----------------------------------------------------------------
  int64_t cf[32];
  {
    auto load_row = [&](const double* src, bool on, int64_t* v) {
      if (tr) {
#pragma unroll
        for (int c = 0; c < 32; c += 2) {
          double2 d = make_double2(0.0, 0.0);
          if (on && c < ncols) d = __ldcg(reinterpret_cast<const double2*>(src + (size_t)r * nb + col0 + c));
          v[c] = __double_as_longlong(d.x);
          v[c + 1] = __double_as_longlong(d.y);
        }
      } else {
#pragma unroll
        for (int c = 0; c < 32; ++c)
          v[c] = __double_as_longlong((on && c < ncols) ? ldg(src + r + (size_t)(col0 + c) * nb) : 0.0);
      }
    };
    load_row(C, own, cf);
    // two passes over [Cp; C]: the largest exponent of a column, then the sum of squares scaled by it
    const bool ownp = top && r >= blk0 * ib && r < blk1 * ib;
    int64_t cq[32];
    load_row(Cp, ownp, cq);
    uint32_t mymax = 0;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const uint32_t h0 = (uint32_t)(cf[c] >> 32) & 0x7fffffffu, h1 = (uint32_t)(cq[c] >> 32) & 0x7fffffffu;
      const uint32_t nz = ((uint32_t)cf[c] | (uint32_t)cq[c]) != 0u;
      const uint32_t m = __reduce_max_sync(kFull, max(max(h0, h1), nz));
      if (lane == c) mymax = m;
    }
    red[warp * 32 + lane] = mymax;
    __syncthreads();
    uint32_t mx = 0;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) mx = max(mx, red[q * 32 + lane]);
    const int emax = (int)(mx >> 20);
    // all warps see the same columns: a uniform decision
    if (__any_sync(kFull, mx != 0 && (emax < 64 || emax > 2000))) {
      cp_async_wait_all();
      __syncthreads();
      return 0;
    }
    float sq[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const int base = (__shfl_sync(kFull, emax, c) - 120) * (1 << 20);
      const int d0 = max((int)((uint32_t)(cf[c] >> 32) & 0x7fffffffu) - base, 0);
      const int d1 = max((int)((uint32_t)(cq[c] >> 32) & 0x7fffffffu) - base, 0);
      const float f0 = __int_as_float(d0 << 3), f1 = __int_as_float(d1 << 3);   // |x| 2^(1016 - emax), truncated
      sq[c] = f0 * f0 + f1 * f1;
    }
    const float part = transpose_sum(sq);
    __syncthreads();
    red[warp * 32 + lane] = __float_as_uint(part);
    __syncthreads();
    float s2 = 0.0f;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) s2 += __uint_as_float(red[q * 32 + lane]);
    const int k = (int)(__float_as_uint(sqrtf(s2) * 1.03f) >> 23) - 127;
    const int E = mx == 0 ? 0 : k + 1 + emax - 1016;
    if (warp == 0) colE[lane] = E;
#pragma unroll
    for (int c = 0; c < 32; ++c) cf[c] = to_fixed(__longlong_as_double(cf[c]), 63 - __shfl_sync(kFull, E, c));
    __syncthreads();
  }
  const int myE = colE[lane];          // of column c = lane (the pivot rows' column)

  load_t(blk_of(0) * ib);
  load_ct(blk_of(0) * ib);

  const uint32_t smV = smem_u32(sm + kDigV), smC = smem_u32(sm + kDigC), smW = smem_u32(sm + kDigW2);
  const uint32_t tq = um.tmem + ((uint32_t)((warp & 3) * 32) << 16);
  int done = 0;
  bool ok = true;
  for (int bb = 0; bb < nbk && ok; ++bb) {
    const int c0 = blk_of(bb) * ib;
    const int v0 = type == UNMQR ? c0 : 0, v1 = type == TTMQR ? c0 + kb : nb;   // rows of this block's V
    // ---- V: largest exponent, digits ---------------------------------------------------------------
    cp_async_wait_all();
    __syncthreads();
    const bool vrow = r >= v0 && r < v1;
    auto vmask = [&](int a, double x) {
      if (type == UNMQR) x = r > c0 + a ? x : (r == c0 + a ? 1.0 : 0.0);
      if (type == TTMQR) x = r <= c0 + a ? x : 0.0;
      return (vrow && a < kb) ? x : 0.0;
    };
    auto vraw = [&](int a, double* x) {     // entries a, a + 1 of the row
      if (tr) {
        const double2 d = *reinterpret_cast<const double2*>(sm + kDigRaw + r * 256 + (((a >> 1) ^ (r & 7)) << 4));
        x[0] = vmask(a, d.x);
        x[1] = vmask(a + 1, d.y);
      } else {
        const double* p = reinterpret_cast<const double*>(sm + kDigRaw) + a * kDigRows + r;
        x[0] = vmask(a, p[0]);
        x[1] = vmask(a + 1, p[kDigRows]);
      }
    };
    {
      uint32_t hv = 0, ht = 0;
#pragma unroll
      for (int a = 0; a < 32; a += 2) {
        double x[2];
        vraw(a, x);
        hv = max(hv, max((uint32_t)__double2hiint(x[0]) & 0x7fffffffu, (uint32_t)__double2hiint(x[1]) & 0x7fffffffu));
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) ht = max(ht, (uint32_t)__double2hiint(tv[k]) & 0x7fffffffu);
      hv = __reduce_max_sync(kFull, hv);
      ht = __reduce_max_sync(kFull, ht);
      if (lane == 0) {
        red[warp] = hv;
        red[8 + warp] = ht;
      }
    }
    __syncthreads();
    int eV = 0, eT = 0;
    {
      uint32_t hv = 0, ht = 0;
#pragma unroll
      for (int q = 0; q < kWarps; ++q) {
        hv = max(hv, red[q]);
        ht = max(ht, red[8 + q]);
      }
      // (a largest entry above 0.992 x 2^eV counts as 2^eV, so that the top digit stays below 128)
      eV = max((int)((hv + (1u << 14)) >> 20) - 1022, -12);
      eT = max((int)(ht >> 20) - 1022, 1);
    }
    if (eV > 1 || eT > 12) break;      // uniform: the rest goes to the FP64 units
#pragma unroll 1
    for (int ag = 0; ag < 4; ++ag) {
      int64_t vf[8];
#pragma unroll
      for (int a = 0; a < 8; a += 2) {
        double x[2];
        vraw(8 * ag + a, x);
        vf[a] = to_fixed(x[0], 63 - eV);
        vf[a + 1] = to_fixed(x[1], 63 - eV);
      }
      uint4 d[kDigN];
      digits8<kDigN>(vf, d);
#pragma unroll
      for (int j = 0; j < kDigN; ++j)
        *reinterpret_cast<uint4*>(sm + kDigV + j * kDigSlice + (ag * kDigRows + r) * 16) = d[j];
    }
    __syncthreads();                   // the staged V is free: the C digits take its place
#pragma unroll
    for (int cg = 0; cg < 4; ++cg) {
      uint4 d[kDigN];
      digits8<kDigN>(cf + 8 * cg, d);
#pragma unroll
      for (int j = 0; j < kDigN; ++j)
        *reinterpret_cast<uint4*>(sm + kDigC + j * kDigSlice + (cg * kDigRows + r) * 16) = d[j];
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- phase 1: products of the digits of V^T and C, one accumulator per (digit of V, digit of C) --
    if (tid == 0) {
      const uint32_t i0 = umma_idesc_f16(128, 32 * kDigN, true, true), i1 = umma_idesc_f16(128, 128, true, true);
      const int k0 = v0 >> 4, k1 = (v1 + 15) >> 4;
      for (int ks = k0; ks < k1; ++ks) {
        const uint64_t b = umma_desc(smC + ks * 256, 128, kDigRows * 16);
        umma_f16(um.tmem, umma_desc(smV + ks * 256, 128, kDigRows * 16), b, i0, ks > k0);
        umma_f16(um.tmem + 256, umma_desc(smV + 4 * kDigSlice + ks * 256, 128, kDigRows * 16), b, i1, ks > k0);
      }
      umma_commit(um.mbar);
    }
    ok = __syncthreads_and(mbar_wait(um.mbar, um.phase, prm.wait_ns) ? 1 : 0) != 0;
    um.phase ^= 1u;
    if (!ok) break;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // the C digits are free: stage the next block's V there; T goes beside it
    const double ctv[4] = {ct[0], ct[1], ct[2], ct[3]};
    int2* Ts = reinterpret_cast<int2*>(sm + kDigT);       // op(T)(a, t) at t 34 + a: 2^28 x + y = T 2^(56 - eT)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int o = tid + k * kThreads, i = o & 31, j = o >> 5;
      if (kb != 32) break;
      const int64_t f = to_fixed(tv[k], 63 - eT) >> 7;
      const int h = (int)((f + (1 << 27)) >> 28), l = (int)(f - ((int64_t)h << 28));
      Ts[notrans ? j * 34 + i : i * 34 + j] = make_int2(h, l);
    }
    if (kb != 32) {
      for (int o = tid; o < 1024; o += kThreads) Ts[(o >> 5) * 34 + (o & 31)] = make_int2(0, 0);
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int o = tid + k * kThreads, i = o % kb, j = o / kb;
        if (o < kb * kb) {
          const int64_t f = to_fixed(tv[k], 63 - eT) >> 7;
          const int h = (int)((f + (1 << 27)) >> 28), l = (int)(f - ((int64_t)h << 28));
          Ts[notrans ? j * 34 + i : i * 34 + j] = make_int2(h, l);
        }
      }
    }
    if (bb + 1 < nbk) {
      const int cn = blk_of(bb + 1) * ib;
      prefetch_v(cn);
      load_t(cn);
      load_ct(cn);
    }
    // ---- partial sums of W 2^(62 - E_c): lane = (digit j = q of V, reflector), 16 columns per warp -----
    int64_t* P = reinterpret_cast<int64_t*>(sm + kDigP);
    {
      const int q = warp & 3, ch = (warp >> 2) * 16;
      const int sH = 24 + eV - 8 * q, sL = eV - 8 - 8 * q;
#pragma unroll
      for (int cg = 0; cg < 16; cg += 8) {
        uint32_t d[7][8], e[4][8];
#pragma unroll
        for (int i = 0; i < 7; ++i) tmem_ld8(tq + 32 * i + ch + cg, d[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) tmem_ld8(tq + 256 + 32 * i + ch + cg, e[i]);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          // digit pairs with i + j >= 8 are left out: i <= 7 - q of the first block, i <= 3 - q of the second
          const int d5 = q < 3 ? int_of(d[5][c]) : 0, d6 = q < 2 ? int_of(d[6][c]) : 0;
          const int e0 = q < 3 ? int_of(e[0][c]) : 0, e1 = q < 3 ? int_of(e[1][c]) : 0;
          const int e2 = q < 2 ? int_of(e[2][c]) : 0, e3 = q < 1 ? int_of(e[3][c]) : 0;
          const int64_t H = wide(int_of(d[0][c]), 1 << 24, wide(int_of(d[1][c]), 1 << 16, wide(int_of(d[2][c]), 256, int_of(d[3][c]))));
          const int64_t L = wide(int_of(d[4][c]) + e0, 1 << 24, wide(d5 + e1, 1 << 16, wide(d6 + e2, 256, e3)));
          P[(q * 32 + lane) * 33 + ch + cg + c] = shl_signed(H, sH) + shl_signed(L, sL);
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // ---- W = Ct + V^T C, split for the 32-bit multipliers: W 2^(58 - E_c) = 2^29 x + y --------------
    int64_t c63[4];
    int2* W = reinterpret_cast<int2*>(P);
    {
      int64_t s[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int o = arow[k] * 33 + lane;
        c63[k] = to_fixed(ctv[k], 63 - myE);
        s[k] = (c63[k] >> 1) + P[o] + P[o + 32 * 33] + P[o + 64 * 33] + P[o + 96 * 33];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int64_t f = (s[k] + 8) >> 4;
        const int h = (int)((f + (1 << 28)) >> 29), l = (int)(f - ((int64_t)h << 29));
        W[arow[k] * 33 + lane] = make_int2(h, l);
      }
    }
    __syncthreads();
    // ---- phase 2: W2 = op(T) W in integers, Ct -= W2, digits of W2 ----------------------------------
    int64_t w2[4];
#pragma unroll
    for (int hp = 0; hp < 2; ++hp) {
      const int a = arow[2 * hp];
      int64_t A0 = 0, A1 = 0, B0 = 0, B1 = 0, D0 = 0, D1 = 0;
      const int t0 = notrans ? a : 0, t1 = notrans ? kb : min(kb, a + 2);
#pragma unroll 4
      for (int t = t0; t < t1; ++t) {
        const int2 w = W[t * 33 + lane];
        const int4 x = *reinterpret_cast<const int4*>(Ts + t * 34 + a);
        A0 = wide(x.x, w.x, A0);
        B0 = wide(x.x, w.y, B0);
        D0 = wide(x.y, w.x, D0);
        A1 = wide(x.z, w.x, A1);
        B1 = wide(x.z, w.y, B1);
        D1 = wide(x.w, w.x, D1);
      }
      w2[2 * hp] = (int64_t)((uint64_t)A0 << (5 + eT)) + ((B0 + 2 * D0) >> (24 - eT));
      w2[2 * hp + 1] = (int64_t)((uint64_t)A1 << (5 + eT)) + ((B1 + 2 * D1) >> (24 - eT));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (top && lane < ncols && arow[k] < kb)
        stg(Cp + toff(c0 + arow[k], col0 + lane, nb, tr), from_fixed(c63[k] - 2 * w2[k], 63 - myE));
    }
    {
      const int64_t x[8] = {w2[0], w2[1], w2[2], w2[3], 0, 0, 0, 0};
      uint4 d[8];
      digits8<8>(x, d);
#pragma unroll
      for (int i = 0; i < 8; ++i) {   // W2 digit i, column c, reflector a at i 2048 + (c / 8) 512 + (a / 8) 128 + (c % 8) 16 + 2 (a % 8)
        unsigned char* p = sm + kDigW2 + i * 2048 + (lane >> 3) * 512 + (lane & 7) * 16;
        *reinterpret_cast<uint32_t*>(p + (arow[0] >> 3) * 128 + (arow[0] & 7) * 2) = d[i].x;
        *reinterpret_cast<uint32_t*>(p + (arow[2] >> 3) * 128 + (arow[2] & 7) * 2) = d[i].y;
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- phase 3: V W2, digit pairs of equal weight in one accumulator ------------------------------
    const int h0 = v0 >> 7, h1 = (v1 + 127) >> 7;       // halves of 128 rows
    if (tid == 0) {
      for (int h = h0; h < h1; ++h)
        for (int j = 0; j < kDigN; ++j) {
          const uint32_t idesc = umma_idesc_f16(128, 32 * (8 - j), false, false);
          for (int ks = 0; ks < 2; ++ks)
            umma_f16(um.tmem + 256 * h + 32 * j,
                     umma_desc(smV + j * kDigSlice + h * 2048 + ks * 2 * kDigRows * 16, kDigRows * 16, 128),
                     umma_desc(smW + ks * 256, 128, 512), idesc, j + ks > 0);
        }
      umma_commit(um.mbar);
    }
    ok = __syncthreads_and(mbar_wait(um.mbar, um.phase, prm.wait_ns) ? 1 : 0) != 0;
    um.phase ^= 1u;
    if (!ok) break;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- C -= V W2 in integers: C 2^(63 - E_c) loses D_g 2^(50 + eV - 8 g) --------------------------
    const int hw = warp >> 2;
    if (hw >= h0 && hw < h1) {         // warp-uniform
#pragma unroll
      for (int cg = 0; cg < 32; cg += 8) {
        uint32_t d[8][8];
#pragma unroll
        for (int g = 0; g < 8; ++g) tmem_ld8(tq + 256 * hw + 32 * g + cg, d[g]);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          constexpr uint32_t kOff = kMagicBits * 257u;
          const int p01 = (int)(mag(d[0][c]) * 256 + mag(d[1][c]) - kOff), p23 = (int)(mag(d[2][c]) * 256 + mag(d[3][c]) - kOff);
          const int p45 = (int)(mag(d[4][c]) * 256 + mag(d[5][c]) - kOff), p67 = (int)(mag(d[6][c]) * 256 + mag(d[7][c]) - kOff);
          const int64_t H = wide(p01, 65536, p23), L = wide(p45, 65536, p67);
          if (own) cf[cg + c] -= (int64_t)((uint64_t)H << (26 + eV)) + (L >> (6 - eV));
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    ++done;
  }
  if (!ok) {     // a completion wait ran out: nothing more is issued or written back
    if (tid == 0) atomicCAS(prm.err, 0, DERR_TIMEOUT);
    um.failed = 1;
    cp_async_wait_all();
    __syncthreads();
    return nbk;
  }
  cp_async_wait_all();
  // ---- store the strip ----------------------------------------------------------------------------
  if (own && done > 0) {
    if (tr) {
#pragma unroll
      for (int c = 0; c < 32; c += 2)
        if (c < ncols)
          __stcg(reinterpret_cast<double2*>(C + (size_t)r * nb + col0 + c),
                 make_double2(from_fixed(cf[c], 63 - colE[c]), from_fixed(cf[c + 1], 63 - colE[c + 1])));
    } else {
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (c < ncols) stg(C + r + (size_t)(col0 + c) * nb, from_fixed(cf[c], 63 - colE[c]));
    }
  }
  __syncthreads();
  return done;
}
