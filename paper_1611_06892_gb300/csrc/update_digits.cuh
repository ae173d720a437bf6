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
//  * the digit products are put together in 64-bit integers, in V^T C for 34 pairs of digits (7 of V and of C), in V W2
//    for 35 (7 of V, 8 of W2).
//
// Fixed point.  Column c of the strip has the exponent E_c, the smallest with 1.03 ||[Cp; C](:, c)||_2 < 2^E_c
// over all rows the task touches; the column's norm does not change under the reflectors, so every
// intermediate entry fits C 2^(63 - E_c) in an int64 for the whole task.  Its seven upper digits carry
// 2^-56 of the column's norm, and the updates are exact integer subtractions on all 63 bits, so a column is
// rounded once per task when it is stored instead of once per multiply-add.  V is V 2^62 (|v| <= 1), T is scaled
// by its largest exponent (eT).  With ||v_k||^2 = 2 / tau_k <= 2: |W| <= 1.42 N_c and |W2| <= 2 N_c.
//
// What is left out, in 2^E_c, in the worst case and for random digits: pairs (i, j) of digits with i + j >= 8, over
// 256 rows of V^T C 2^-52.7 and 2^-59.4, over 32 reflectors of V W2 2^-54.4 and 2^-59.8; the eighth digits of C and V
// (2^-56 and 2^-55 an entry) in V^T C 2^-51.5 and 2^-56, and 2^-51 and 2^-55.8; that of V in V W2 2^-49 and 2^-55.  FP64
// sums of the same lengths round to 2^-53 of each partial sum: worst cases of 2^-45 and 2^-48, a few 2^-53 at random.
// (Measured cases, error against 64 bits over that of the FP64 units: bands 0.67 - 0.86, vectors 0.69, gradient 1.0.)
//
// Columns that are not finite, or outside [2^-958, 2^977], and blocks whose V or T are out of range are
// refused; the caller runs them on the FP64 units (task_update).
//
// Rows.  FP64 arithmetic keeps a row that is far smaller than the others to its own scale (weighted least squares;
// rows from 1 to 1e-16: R's rows to 1e-13), fixed point by columns does not.  A block is therefore refused too, before
// any of it is applied, if it changes a row r that is small and stays small: |C(r, c)| < 2^-8 2^E_c and
// |V(r, j)| |W2(j, c)| < 2^-10 2^E_c for all j and c; or a pivot row j as small, under a reflector with next to no tail
// (tau_j > 2 - 2^-14).  Rows of N(0, 1) columns have entries near 2^-4 2^E_c, so that full strips of ordinary matrices
// never come to the second test (rows_lost).  In strips of fewer than 8 columns a row can be small by chance: there the
// row of V has to be small too, |V(r, j)| < 2^-8 ||v_j|| for all j (never with an entry of 2^-8, as ||v_j|| <= 1 beside the
// unit entry).  Rows that no reflector touches are
// not written back.
//
// Layout.  512 threads: thread t owns columns 16 (t / 256) .. + 15 of row t % 256 of the strip (int64 in registers;
// with 256 threads of 32 columns the code was bound by its own latencies, two warps a scheduler): TMEM lane = row,
// so the product V W2 arrives where it is subtracted, and the new digits of the row go to shared memory in 16-byte
// pieces.  V and C digits: digit d of row r is 64 bytes (32 columns) at 16384 d + 64 r, its 16-byte pieces permuted
// by the 64-byte swizzle.  For V^T C both operands are read M/N-major from it (M = (digit, reflector),
// N = (digit, column)), for V W2 the same V is read K-major (M = row, K = reflector).

// ---- instruction and layout helpers ---------------------------------------------------------------
static_assert(kDigitRows == 256, "rows of the layout");
constexpr int kDigRows = 256;                       // rows of the layout
constexpr int kDigSlice = kDigRows * 64;            // bytes of one digit of 256 rows x 32 columns
constexpr int kDigN = 7;                            // digits of V and C
constexpr int kDigV = 0;                            // byte offsets: V digits,
constexpr int kDigC = kDigN * kDigSlice;            // C digits; when phase 1 is done the same area holds
constexpr int kDigRaw = kDigC;                      //   the next block's V as stored (rows of 272 bytes at most),
constexpr int kDigP = kDigRaw + kDigRows * 272;     //   the partial sums of W: 4 x 32 x 33 int64,
constexpr int kDigPStride = 32 * 33 * 8;            //   (slot 0 then holds W, W2's digits follow it)
constexpr int kDigW2 = kDigP + kDigPStride;
constexpr int kDigT = kDigP + 4 * kDigPStride;      //   and op(T), 32 rows of 34 (two int32 each)
constexpr int kDigHead = 2 * kDigN * kDigSlice;     // column exponents, reduction scratch
constexpr int kDigBytes = kDigHead + 128 + 1024;
static_assert(kDigW2 + 8 * 2048 <= kDigP + 4 * kDigPStride, "W2 digits fit beside W");
static_assert(kDigT + 32 * 34 * 8 + kDigitHeadBytes <= kDigHead, "T and the header fit");
static_assert((kDigW2 & 127) == 0, "operand alignment");
constexpr int kDigRow = kDigP + 3 * kDigPStride;    // scratch of the tests of rows, between two uses of that slot
constexpr int kDigTmem = 512;
constexpr int kDigTBytes = 32 * 34 * 8;
static_assert(kDigTBytes == kDigitTBytes && kDigN == kDigitCount, "published blocks");

#if BD_EXEC_PART == 1
__host__ __device__ constexpr uint32_t umma_idesc_f16(int m, int n, bool a_mn, bool b_mn) {
  return (1u << 4) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// size bytes (a multiple of 16) from global to shared memory, both 16-byte aligned
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, int size, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"(src), "r"(size), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t mbar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
constexpr int kIssueWarp = 12;       // of the second row half: the first half's warps go on during the MMAs
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
// Integer value of an exact FP32 integer |x| <= 2^22 (adding 1.5 x 2^23 puts it into the low mantissa bits).
constexpr uint32_t kMagicBits = 0x4B400000u;
__device__ __forceinline__ uint32_t mag(uint32_t f) { return __float_as_uint(__uint_as_float(f) + 12582912.0f); }
__device__ __forceinline__ int int_of(uint32_t f) { return (int)(mag(f) - kMagicBits); }
__device__ __forceinline__ int64_t wide(int a, int b, int64_t c) { return (int64_t)a * b + c; }
// x 2^sh cut to an integer (x finite; sh = 63 - E with |x| < 2^E, so the result is below 2^63; numbers of
// exponent 0 come out as 0 for every E in use)
__device__ __forceinline__ int64_t to_fixed(double x, int sh) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint64_t m = ((uint64_t)((hi & 0xfffff) | 0x100000) << 32 | lo) << 10;   // |x| = m 2^(e - 1085)
  uint64_t v;                                                                  // m >> t, 0 for t > 63
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(1085 - sh - (int)((hi >> 20) & 0x7ff)));
  const int64_t s = (int32_t)hi >> 31;
  return ((int64_t)v ^ s) - s;
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

// The ND most significant digits of two fixed-point values, as f16 pairs.
template <int ND>
__device__ __forceinline__ void digit_pair(int64_t x0, int64_t x1, uint32_t* w) {
  const uint64_t y0 = (uint64_t)x0 + 0x8080808080808080ull, y1 = (uint64_t)x1 + 0x8080808080808080ull;
  const uint32_t h0 = (uint32_t)(y0 >> 32), h1 = (uint32_t)(y1 >> 32), l0 = (uint32_t)y0, l1 = (uint32_t)y1;
  const uint32_t hu = __byte_perm(h0, h1, 0x7362), hl = __byte_perm(h0, h1, 0x5140);
  const uint32_t lu = __byte_perm(l0, l1, 0x7362), ll = __byte_perm(l0, l1, 0x5140);
  const uint32_t k64 = 0x64646464u;          // 1024 + byte, as f16 bits, of both values
  const uint32_t r[8] = {__byte_perm(hu, k64, 0x4342), __byte_perm(hu, k64, 0x4140), __byte_perm(hl, k64, 0x4342),
                         __byte_perm(hl, k64, 0x4140), __byte_perm(lu, k64, 0x4342), __byte_perm(lu, k64, 0x4140),
                         __byte_perm(ll, k64, 0x4342), __byte_perm(ll, k64, 0x4140)};
#pragma unroll
  for (int j = 0; j < ND; ++j)               // minus 1152: the signed digit
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(w[j]) : "r"(r[j]), "r"(0x64806480u));
}
// Digits of eight values of row r, columns 8 g .. 8 g + 7, into an operand at sm (slice: bytes of one digit).
__device__ __forceinline__ void put_digits(unsigned char* sm, int r, int g, const int64_t* x, int slice = kDigSlice) {
  uint32_t w[4][kDigN];
#pragma unroll
  for (int p = 0; p < 4; ++p) digit_pair<kDigN>(x[2 * p], x[2 * p + 1], w[p]);
  unsigned char* o = sm + r * 64 + ((g ^ ((r >> 1) & 3)) << 4);
#pragma unroll
  for (int j = 0; j < kDigN; ++j)
    *reinterpret_cast<uint4*>(o + j * slice) = make_uint4(w[0][j], w[1][j], w[2][j], w[3][j]);
}
// Descriptor of an operand in the digit layout (64-byte swizzle): stride of 32-column slices (M/N-major), and of
// groups of 8 rows (512 bytes).
__device__ __forceinline__ uint64_t digit_desc(uint32_t addr, uint32_t lbo) {
  return umma_desc(addr, lbo, 512) | (uint64_t)4 << 61;
}

// Sum over the 32 lanes of v[k], left in lanes k and k + 16 (k < 16).
__device__ __forceinline__ float transpose_sum16(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 8; s > 0; s >>= 1) {
    const bool up = lane & s;
#pragma unroll
    for (int k = 0; k < s; ++k) {
      const float mine = up ? v[k + s] : v[k], other = up ? v[k] : v[k + s];
      v[k] = mine + __shfl_xor_sync(kFull, other, s);
    }
  }
  return v[0] + __shfl_xor_sync(kFull, v[0], 16);
}

// E_c of the columns whose entries the CTA's threads hold as FP64 bit patterns (thread: 16 columns of a row of x and of
// a row of y): into colE, and that of column lane % 16 of the thread's half into *E, and whether it is zero.  Two passes: the largest exponent
// of a column, then the sum of its squares scaled by it.  False (for all) if a column is out of range, or zero and
// zero_ok is false.
__device__ __forceinline__ bool column_exponents(const int64_t* cf, const int64_t* cq, int* colE, uint32_t* red, int* E,
                                                 bool* zero, bool zero_ok = true) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ch = threadIdx.x >> 8;
  uint32_t mymax = 0;
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const uint32_t h0 = (uint32_t)(cf[c] >> 32) & 0x7fffffffu, h1 = (uint32_t)(cq[c] >> 32) & 0x7fffffffu;
    const uint32_t nz = min((uint32_t)cf[c] | (uint32_t)cq[c], 1u);
    const uint32_t m = __reduce_max_sync(kFull, max(max(h0, h1), nz));
    if ((lane & 15) == c) mymax = m;
  }
  if (lane < 16) red[warp * 16 + lane] = mymax;
  __syncthreads();
  uint32_t mx = 0;                  // of column cb + (lane & 15)
#pragma unroll
  for (int q = 0; q < 8; ++q) mx = max(mx, red[(8 * ch + q) * 16 + (lane & 15)]);
  const int emax = (int)(mx >> 20);
  if (__syncthreads_or(mx == 0 ? !zero_ok : (emax < 64 || emax > 2000))) return false;
  float sq[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const int base = (__shfl_sync(kFull, emax, c) - 120) * (1 << 20);
    const int d0 = max((int)((uint32_t)(cf[c] >> 32) & 0x7fffffffu) - base, 0);
    const int d1 = max((int)((uint32_t)(cq[c] >> 32) & 0x7fffffffu) - base, 0);
    const float f0 = __int_as_float(d0 << 3), f1 = __int_as_float(d1 << 3);   // |x| 2^(1016 - emax), truncated
    sq[c] = f0 * f0 + f1 * f1;
  }
  const float part = transpose_sum16(sq);
  if (lane < 16) red[warp * 16 + lane] = __float_as_uint(part);
  __syncthreads();
  float s2 = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; ++q) s2 += __uint_as_float(red[(8 * ch + q) * 16 + (lane & 15)]);
  const int k = (int)(__float_as_uint(sqrtf(s2) * 1.03f) >> 23) - 127;
  *zero = mx == 0;
  *E = mx == 0 ? 0 : k + 1 + emax - 1016;
  if ((warp & 7) == 0 && lane < 16) colE[16 * ch + lane] = *E;
  return true;
}

// Readout of the digit products of phase 1 (lane = (digit j of A, column of A), column = (digit i of B, column of B)):
// P[q][a][c] += over the digits j = q and q + 4 of A, in units where the pair of leading digits weighs 2^(s + 24).
// kWide: sums may exceed 2^22 (more than 256 rows).
template <bool kWide>
__device__ __forceinline__ void gram_partials(int64_t* P, uint32_t tq, int s) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3;
  const int sH = s - 8 * q, sL = 32 - s + 8 * q;
  auto val = [](uint32_t f) { return kWide ? __float2int_rn(__uint_as_float(f)) : int_of(f); };
#pragma unroll 1
  for (int cg = (warp >> 2) * 8, ce = cg + 8; cg < ce; cg += 4) {
    uint32_t d[7][4], e[4][4];
#pragma unroll
    for (int i = 0; i < 7; ++i) tmem_ld4(tq + 32 * i + cg, d[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) tmem_ld4(tq + 256 + 32 * i + cg, e[i]);
    tmem_wait_ld();
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      // digit pairs with i + j >= 8 are left out: i <= 7 - q of the first block, i <= 3 - q of the second
      const int64_t H = wide(val(d[0][c]) * 256 + val(d[1][c]), 65536, val(d[2][c]) * 256 + val(d[3][c]));
      int l4 = val(d[4][c]), l5 = 0, l6 = 0, l7 = 0;
      if (q < 3) {
        l4 += val(e[0][c]);
        l5 = val(d[5][c]) + val(e[1][c]);
      }
      if (q < 2) l6 = val(d[6][c]) + val(e[2][c]);
      if (q < 1) l7 = val(e[3][c]);
      const int64_t L = wide(l4, 1 << 24, wide(l5, 1 << 16, wide(l6, 256, l7)));
      P[(q * 32 + lane) * 33 + cg + c] = (int64_t)((uint64_t)H << sH) + (L >> sL);
    }
  }
}

// Bits of a warp's 32 rows, the CTA's two column halves in words warp and warp ^ 8: those of row r.
__device__ __forceinline__ bool row_bit(const uint32_t* words) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return ((words[warp] | words[warp ^ 8]) >> lane) & 1;
}
__device__ __forceinline__ uint32_t abs_hi(int64_t x) {        // upper word of |x| (of |x| - 1 for x < 0)
  const int h = (int)(x >> 32);
  return (uint32_t)(h ^ (h >> 31));
}
__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }
constexpr uint32_t kSmallRow = 1u << (31 - 8);                 // 2^-8 of a column, in the upper word of C
constexpr uint32_t kStrong = (1023u - 8) << 20;                // 2^-8, upper word in FP64 (compared as integers: FP64
                                                               // comparisons take 16 cycles of the SM each)

// Whether the block would lose a row's own scale (see the head of this file).  Thread: row r of the strip, 16 columns;
// big: its largest |C| (abs_hi), nz: V has an entry in the row, w2: rows 2 warp, 2 warp + 1 of W2 2^(62 - E_c) in column
// lane, pivot: a pivot row is lost, diag: row of reflector 0's unit entry (out of range: in the pivot tile).  V's
// digits and T are in place.  Called for few strips, outside the ordinary path's registers.
__device__ __noinline__ bool rows_lost(unsigned char* sm, int kb, int eT, uint32_t big, bool nz, int64_t w20, int64_t w21,
                                       bool pivot, bool narrow, int diag) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = tid & 255, ch = tid >> 8;
  float* omega = reinterpret_cast<float*>(sm + kDigRow);       // max over c of |W2(j, c)| 2^-E_c
  float* least = omega + 32;                                   // narrow: (2^-8 ||v_j||)^2 without the unit entry
  uint32_t* bigs = reinterpret_cast<uint32_t*>(least + 32);
  uint32_t* strong = bigs + 16;
  const uint32_t h0 = __reduce_max_sync(kFull, abs_hi(w20)), h1 = __reduce_max_sync(kFull, abs_hi(w21));
  const unsigned bm = __ballot_sync(kFull, big >= kSmallRow);
  if (lane < 2) {
    const int j = 2 * warp + lane;
    omega[j] = (float)(lane ? h1 : h0) * 0x1p-30f;
    const float tau = (float)reinterpret_cast<const int2*>(sm + kDigT)[35 * j].x * exp2f((float)(eT - 28));
    least[j] = tau > 0.0f ? 0x1p-16f * fmaxf(2.0f / tau - 1.0f, 0x1p-12f) : 2.0f;      // ||v_j||^2 = 2 / tau_j
  }
  if (lane == 0) bigs[warp] = bm;
  if (!__syncthreads_or((w20 | w21) != 0)) return __syncthreads_or(pivot) != 0;
  const bool small = nz && !row_bit(bigs);
  bool st = false;
  if (__any_sync(kFull, small)) {
    for (int g = 0; g < 2; ++g) {
      // V(r, j) from its two upper digits (2^-14): |W2| is below 2 x 2^E_c
      const unsigned char* o = sm + kDigV + r * 64 + (((2 * ch + g) ^ ((r >> 1) & 3)) << 4);
      const uint4 a4 = *reinterpret_cast<const uint4*>(o), b4 = *reinterpret_cast<const uint4*>(o + kDigSlice);
      const uint32_t a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float hi, lo;
        asm("cvt.f32.f16 %0, %1;" : "=f"(hi) : "h"((unsigned short)(a[q >> 1] >> (16 * (q & 1)))));
        asm("cvt.f32.f16 %0, %1;" : "=f"(lo) : "h"((unsigned short)(b[q >> 1] >> (16 * (q & 1)))));
        const float v = fabsf(fmaf(hi, 256.0f, lo)) * 0x1p-14f;
        const int j = 16 * ch + 8 * g + q;
        st = st || (j < kb && (v * omega[j] >= 0x1p-10f || (narrow && r != diag + j && v * v >= least[j])));
      }
    }
  }
  const unsigned sb = __ballot_sync(kFull, st);
  if (lane == 0) strong[warp] = sb;
  __syncthreads();
  return __syncthreads_or(pivot || (small && !row_bit(strong))) != 0;
}

// Published blocks: what the updates of a reduction read of a panel block instead of V and T, made once by its factor
// sub-task (a strip spent 4.4k of its 24k cycles a block on V's digits).  Digits of V in the operand layout
// (digit_image_rows(nb) rows, zeros outside the block), T 2^(56 - eT) split as the updates read it, then the header: two
// integers, whether |v| <= 1 and eT <= 12 hold, and eT, from its word 4 on a bit for each row of V that is not zero and
// from word 12 on for each with an entry of 2^-8 beside a unit one.
// Starts the copy of the V area (16 KB a digit) into block vd; wait_image before the sub-task ends.
__device__ __forceinline__ void store_image(unsigned char* sm, unsigned char* vd, int nb) {
  if ((int)uniform(threadIdx.x >> 5) == kIssueWarp) {
    const int lane = threadIdx.x & 31, img = digit_image_rows(nb) * 64;
    if (lane < kDigN) {
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(vd + lane * img),
                   "r"(smem_u32(sm + kDigV + lane * kDigSlice)), "r"(img)
                   : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
  }
}
__device__ __forceinline__ void wait_image() {
  if ((int)uniform(threadIdx.x >> 5) == kIssueWarp) {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async;" ::: "memory");
  }
}
// T and the header; t: rows 2 warp, 2 warp + 1 of column lane, good: the block's V is in range (any thread), nz: this
// thread's half of row r of V has an entry, strong: one of 2^-8; red: 48 words.
__device__ __forceinline__ void publish_t(unsigned char* vd, int nb, const double* t, bool good, bool nz, bool strong,
                                          uint32_t* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t h = max((uint32_t)__double2hiint(t[0]) & 0x7fffffffu, (uint32_t)__double2hiint(t[1]) & 0x7fffffffu);
  const uint32_t hm = __reduce_max_sync(kFull, h);
  const unsigned rows = __ballot_sync(kFull, nz), big = __ballot_sync(kFull, strong);
  if (lane == 0) {
    red[warp] = hm;
    red[16 + warp] = rows;
    red[32 + warp] = big;
  }
  const bool v_ok = __syncthreads_and(good ? 1 : 0) != 0;
  const int eT = max((int)(__reduce_max_sync(kFull, red[lane & 15]) >> 20) - 1022, 1);
  int2* Ts = reinterpret_cast<int2*>(vd + kDigN * digit_image_rows(nb) * 64);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int64_t f = to_fixed(t[k], 63 - eT) >> 7;
    const int x = (int)((f + (1 << 27)) >> 28);
    __stcg(Ts + (2 * warp + k) * 34 + lane, make_int2(x, (int)(f - ((int64_t)x << 28))));
  }
  unsigned char* head = vd + digit_block_bytes(nb) - kDigitHeadBytes;
  if (threadIdx.x == 0) __stcg(reinterpret_cast<int2*>(head), make_int2(v_ok && eT <= 12 ? 1 : 0, eT));
  if (threadIdx.x < 16) {
    const int o = 16 + (threadIdx.x & 7) + 2 * (threadIdx.x & 8);
    __stcg(reinterpret_cast<uint32_t*>(head) + 4 + threadIdx.x, red[o] | red[o + 8]);
  }
}
// Publishes a block that task_panel_factor has just written.
__device__ __noinline__ void publish_block(unsigned char* sm, int kind, const double* X, int tr, const double* Tg, int nb,
                                           int ib, int b, unsigned char* vd) {
  const int tid = threadIdx.x, kb = ib, c0 = b * ib, r = tid & 255, cb = 16 * (tid >> 8);
  const int r0 = kind == PM_GE ? c0 : 0, r1 = kind == PM_TT ? c0 + kb : nb;
  bool good = true, nz = false, strong = false;
  __syncthreads();
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    int64_t v[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int c = cb + 8 * g + a, d = r - (c0 + c);
      double x = 0.0;
      if (c < kb && r >= r0 && r < r1) {
        if (kind == PM_TS || (kind == PM_GE ? d > 0 : d <= 0)) x = ldg(X + toff(r, c0 + c, nb, tr));
        if (kind == PM_GE && d == 0) x = 1.0;
      }
      good = good && abs_hi(x) <= 0x3ff00000u;
      if (abs_hi(x) != 0)                // (not the unit entry of H = I)
        nz = nz || kind != PM_GE || d != 0 || abs_hi(ldg(Tg + (size_t)c0 * ib + c * (kb + 1))) != 0;
      strong = strong || (abs_hi(x) >= kStrong && !(kind == PM_GE && d == 0));
      v[a] = to_fixed(x, 62);
    }
    put_digits(sm + kDigV, r, (cb >> 3) + g, v);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  store_image(sm, vd, nb);
  const int arow = 2 * (tid >> 5), lane = tid & 31;
  double t[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) t[k] = (arow + k < kb && lane < kb) ? ldg(Tg + (size_t)c0 * ib + arow + k + lane * kb) : 0.0;
  publish_t(vd, nb, t, good, nz, strong, reinterpret_cast<uint32_t*>(sm + kDigHead + 128));
  wait_image();
  __syncthreads();
}

// task_update on the digit path: returns the number of blocks applied (from the first in the order of
// application; C and Cp are up to date for them), the rest being out of the path's range.  Arguments as
// task_update; kPre: vd holds the panel's published blocks (Q^T only), and X and Tg are not read.
template <bool kPre>
__device__ __noinline__ int task_update_digits(unsigned char* sm, int type, const double* X, double* Cp, double* C,
                                               int tr, bool notrans, const double* Tg, int nb, int ib, int blk0,
                                               int blk1, int col0, int ncols, const unsigned char* vd, Umma& um,
                                               const ExecParams& prm) {
  static_assert(kThreads == 512, "two threads a row");
  if (smem_u32(sm) & 511) return 0;                                      // the swizzle's alignment, and the copies
  if ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Cp) | reinterpret_cast<uintptr_t>(C)) & 15) return 0;
  int* colE = reinterpret_cast<int*>(sm + kDigHead);                     // E_c
  uint32_t* red = reinterpret_cast<uint32_t*>(sm + kDigHead + 128);      // 16 x 16 reduction scratch
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kb = ib, r = tid & 255, ch = tid >> 8, cb = 16 * ch;         // row, column half, first column
  const int hw = r >> 7;                                                 // row half (warp-uniform)
  const bool top = type != UNMQR;
  const int row_lo = (type == UNMQR) ? blk0 * ib : 0, row_hi = (type == TTMQR) ? blk1 * ib : nb;
  const bool own = r >= row_lo && r < row_hi;
  const int nbk = blk1 - blk0;
  auto blk_of = [&](int bb) { return notrans ? blk1 - 1 - bb : blk0 + bb; };

  const int uwarp = (int)uniform(warp);
  // kPre: V digits of the next application into their place (whole halves of 128 rows: rows outside the block are zeros
  // there), by bulk copies of one warp counted by the fourth mbarrier
  const int img = digit_image_rows(nb) * 64;
  auto load_image = [&](int b) {
    const int c = b * ib, r0 = type == UNMQR ? c & 128 : 0, r1 = type == TTMQR ? c + kb : nb;
    const int o = r0 * 64, size = min(((r1 + 127) & ~127) * 64, img) - o;
    const unsigned char* src = vd + (size_t)b * digit_block_bytes(nb);
    asm volatile("fence.proxy.async;" ::: "memory");
    if (lane == 0) mbar_expect(um.mbar + 24, kDigN * size);
    __syncwarp();
    if (lane < kDigN) bulk_copy(sm + kDigV + lane * kDigSlice + o, src + lane * img + o, size, um.mbar + 24);
  };
  auto load_head = [&](int b) {
    return __ldcg(reinterpret_cast<const int2*>(vd + (size_t)(b + 1) * digit_block_bytes(nb) - kDigitHeadBytes));
  };
  int2 head = make_int2(1, 0);       // published block: whether it is in range, exponent of T
  // V block of the next application, as stored, into the staging area: columns (ld 256) for tr = 0, by bulk copies
  // of one warp counted by the fourth mbarrier; rows of 272 bytes (free of bank conflicts) for tr = 1, in 16-byte
  // pieces (256 bulk copies of a row took 10k cycles to issue)
  auto prefetch_v = [&](int c0) {
    const int r0 = type == UNMQR ? c0 : 0, r1 = type == TTMQR ? c0 + kb : nb;
    if (tr) {
      const int np = kb >> 1, ln = tid & 15;
      if (ln < np)
        for (int q = r0 + (tid >> 4); q < r1; q += kThreads >> 4)
          cp_async16(sm + kDigRaw + q * 272 + 16 * ln, X + (size_t)q * nb + c0 + 2 * ln);
      cp_async_commit();
    } else if (uwarp == kIssueWarp) {
      asm volatile("fence.proxy.async;" ::: "memory");
      if (lane == 0) mbar_expect(um.mbar + 24, (r1 - r0) * kb * 8);
      __syncwarp();
      for (int a = lane; a < kb; a += 32)
        bulk_copy(sm + kDigRaw + (a * kDigRows + r0) * 8, X + r0 + (size_t)(c0 + a) * nb, (r1 - r0) * 8, um.mbar + 24);
    }
  };
  // waits until this thread's part of it is there (all of it for tr = 0)
  auto wait_v = [&]() {
    if (tr && !kPre) {
      cp_async_wait_all();
      return true;
    }
    const bool w = mbar_wait(um.mbar + 24, (um.phase >> 3) & 1u, prm.wait_ns);
    um.phase ^= 8u;
    return w;
  };
  // A completion wait ran out (for any thread): the error word is set, nothing more is issued or written back, the copies
  // and MMAs in flight are waited for (with the same limit)
  auto timed_out = [&]() {
    if (tid == 0) atomicCAS(prm.err, 0, DERR_TIMEOUT);
    for (int b = 0; b < 5; ++b) mbar_wait(um.mbar + 8 * b, ((um.phase >> b) & 1u) ^ 1u, prm.wait_ns);
    for (int b = 3; b < 5; ++b) mbar_wait(um.mbar + 8 * b, (um.phase >> b) & 1u, prm.wait_ns);
    cp_async_wait_all();
    __syncthreads();
    return nbk;
  };
  // T of a block: entries tid + 512 k of the kb x kb block as stored
  double tv[2];
  auto load_t = [&](int c0) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = tid + k * kThreads;
      tv[k] = o < kb * kb ? ldg(Tg + (size_t)c0 * ib + o) : 0.0;
    }
  };
  // the pivot tile's rows of a block: thread (warp g, lane c) has rows 2g and 2g + 1 of column c
  const int arow = 2 * warp;
  double ct[2] = {0.0, 0.0};
  auto load_ct = [&](int c0) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
      ct[k] = (top && lane < ncols && arow + k < kb) ? ldg(Cp + toff(c0 + arow + k, col0 + lane, nb, tr)) : 0.0;
  };

  if constexpr (kPre) {
    if (uwarp == kIssueWarp) load_image(blk_of(0));
    head = load_head(blk_of(0));
  } else {
    prefetch_v(blk_of(0) * ib);
    load_t(blk_of(0) * ib);
  }
  load_ct(blk_of(0) * ib);

  // ---- load the strip, find E_c -----------------------------------------------------------------
  int64_t cf[16];
  {
    auto load_row = [&](const double* src, bool on, int64_t* v) {
      if (tr) {
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          double2 d = make_double2(0.0, 0.0);
          if (on && cb + c < ncols) d = __ldcg(reinterpret_cast<const double2*>(src + (size_t)r * nb + col0 + cb + c));
          v[c] = __double_as_longlong(d.x);
          v[c + 1] = __double_as_longlong(d.y);
        }
      } else {
#pragma unroll
        for (int c = 0; c < 16; ++c)
          v[c] = __double_as_longlong((on && cb + c < ncols) ? ldg(src + r + (size_t)(col0 + cb + c) * nb) : 0.0);
      }
    };
    load_row(C, own, cf);
    const bool ownp = top && r >= blk0 * ib && r < blk1 * ib;
    int64_t cq[16];
    load_row(Cp, ownp, cq);
    int E;
    bool zero;
    if (!column_exponents(cf, cq, colE, red, &E, &zero)) {
      // (the caller's next update writes where the copy of V lands)
      return __syncthreads_and(wait_v() ? 1 : 0) ? 0 : timed_out();
    }
    uint32_t big = 0;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      cf[c] = to_fixed(__longlong_as_double(cf[c]), 63 - __shfl_sync(kFull, E, c));
      big = max(big, abs_hi(cf[c]));
    }
    uint32_t* rw = reinterpret_cast<uint32_t*>(sm + kDigRow);
    const unsigned rows = __ballot_sync(kFull, big >= kSmallRow), cols = __ballot_sync(kFull, !zero && lane < 16);
    if (lane == 0) {
      rw[warp] = rows;
      if ((warp & 7) == 0) rw[16 + ch] = __popc(cols);
    }
  }

  const uint32_t uV = uniform(smem_u32(sm + kDigV)), uC = uV + kDigC, uW = uV + kDigW2, utm = uniform(um.tmem);
  const uint32_t tq = um.tmem + ((uint32_t)((warp & 3) * 32) << 16);
  int done = 0, v0 = 0, v1 = 0, c0 = 0;
  __syncthreads();
  const int myE = colE[lane];          // of column c = lane (the pivot rows' column)
  const uint32_t* rw = reinterpret_cast<const uint32_t*>(sm + kDigRow);
  const int ncols_nz = (int)(rw[16] + rw[17]);         // columns that are not zero
  const bool small_row = ncols_nz > 0 && !row_bit(rw), narrow = ncols_nz < 8;
  bool touched = false;                // a reflector applied so far has an entry in row r
  bool ok = true;                      // this thread's completion waits
  for (int bb = 0; bb < nbk; ++bb) {
    // ---- V digits ---------------------------------------------------------------------------------
    c0 = blk_of(bb) * ib;
    v0 = type == UNMQR ? c0 : 0;
    v1 = type == TTMQR ? c0 + kb : nb;
    int eT;
    if constexpr (kPre) {
      if (!__syncthreads_and(ok ? 1 : 0)) {         // (also: the last block's products and scratch are done with)
        ok = false;
        break;
      }
      if (!head.x) {                                // uniform: the rest goes to the FP64 units
        ok = wait_v() && ok;
        break;
      }
      eT = head.y;
    } else {
      ok = wait_v() && ok;
      if (tr) __syncthreads();
      uint32_t hv = 0, hu = 0;           // largest |v| (high word), and beside the unit entries
      {
        const bool vrow = r >= v0 && r < v1;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          double x[8];
          if (tr) {
            const double2* p = reinterpret_cast<const double2*>(sm + kDigRaw + r * 272 + (cb + 8 * g) * 8);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              const double2 d = p[a];
              x[2 * a] = d.x;
              x[2 * a + 1] = d.y;
            }
          } else {
            const double* p = reinterpret_cast<const double*>(sm + kDigRaw) + (cb + 8 * g) * kDigRows + r;
#pragma unroll
            for (int a = 0; a < 8; ++a) x[a] = p[a * kDigRows];
          }
          const bool in = vrow && cb + 8 * g < kb;        // (kb is a multiple of 8)
          const int d = r - (c0 + cb + 8 * g);            // 0 on the diagonal of column a = 0
          if (type == UNMQR) {
#pragma unroll
            for (int a = 0; a < 8; ++a) {
              hu = max(hu, in && d > a ? (uint32_t)__double2hiint(x[a]) & 0x7fffffffu : 0u);
              x[a] = d > a ? x[a] : (d == a ? 1.0 : 0.0);
            }
          } else if (type == TTMQR) {
#pragma unroll
            for (int a = 0; a < 8; ++a) x[a] = d <= a ? x[a] : 0.0;
          }
          int64_t vf[8];
#pragma unroll
          for (int a = 0; a < 8; ++a) {
            x[a] = in ? x[a] : 0.0;
            hv = max(hv, (uint32_t)__double2hiint(x[a]) & 0x7fffffffu);
            vf[a] = to_fixed(x[a], 62);
          }
          put_digits(sm + kDigV, r, 2 * ch + g, vf);
        }
        uint32_t ht = max((uint32_t)__double2hiint(tv[0]) & 0x7fffffffu, (uint32_t)__double2hiint(tv[1]) & 0x7fffffffu);
        ht = __reduce_max_sync(kFull, ht);
        const unsigned rows = __ballot_sync(kFull, hv != 0);
        const unsigned big = __ballot_sync(kFull, (type == UNMQR ? hu : hv) >= kStrong);
        if (lane == 0) {
          red[warp] = ht;
          red[16 + warp] = rows;
          red[32 + warp] = big;
        }
      }
      // the staged V is free from here on: the C digits take its place.  1: a wait ran out, 2: |v| > 1 (not finite)
      if (__syncthreads_or(!ok || hv > 0x3ff00000u)) {
        if (!__syncthreads_and(ok ? 1 : 0)) ok = false;
        break;                           // uniform: the rest goes to the FP64 units
      }
      eT = max((int)(__reduce_max_sync(kFull, red[lane & 15]) >> 20) - 1022, 1);
      if (eT > 12) break;
    }
    // ---- C digits ---------------------------------------------------------------------------------
#pragma unroll
    for (int g = 0; g < 2; ++g) put_digits(sm + kDigC, r, 2 * ch + g, cf + 8 * g);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- phase 1: products of the digits of V^T and C, one accumulator per (digit of V, digit of C) --
    if (uwarp == kIssueWarp) {
      const uint32_t i0 = umma_idesc_f16(128, 32 * kDigN, true, true), i1 = umma_idesc_f16(128, 128, true, true);
      const int k0 = uniform(v0 >> 4), k1 = uniform((v1 + 15) >> 4);
      const uint64_t da = digit_desc(uV + k0 * 1024, kDigSlice), db = digit_desc(uC + k0 * 1024, kDigSlice);
      if constexpr (kPre) ok = wait_v() && ok;
#pragma unroll 4
      for (int k = 0; k < k1 - k0; ++k) {      // 16 rows: 1024 bytes
        umma_f16(utm, da + k * 64, db + k * 64, i0, k > 0);
        umma_f16(utm + 256, da + (4 * kDigSlice >> 4) + k * 64, db + k * 64, i1, k > 0);
      }
      umma_commit(um.mbar);
    }
    if (kPre && uwarp != kIssueWarp) um.phase ^= 8u;      // (that warp alone waits for V)
    ok = mbar_wait(um.mbar, um.phase & 1u, prm.wait_ns) && ok;
    um.phase ^= 1u;
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // the C digits are free: stage the next block's V there; T goes beside it
    const double ctv[2] = {ct[0], ct[1]};
    const int h0 = v0 >> 7, h1 = (v1 + 127) >> 7;       // h0 .. h1 - 1: halves of 128 rows of this block
    int2* Ts = reinterpret_cast<int2*>(sm + kDigT);       // op(T)(a, t) at t 34 + a: 2^28 x + y = T 2^(56 - eT)
    if constexpr (kPre) {
      if (uwarp == kIssueWarp && lane == 0) {
        mbar_expect(um.mbar + 32, kDigTBytes + kDigitHeadBytes);
        bulk_copy(Ts, vd + (size_t)blk_of(bb) * digit_block_bytes(nb) + kDigN * img, kDigTBytes + kDigitHeadBytes,
                  um.mbar + 32);
      }
      if (bb + 1 < nbk) {
        head = load_head(blk_of(bb + 1));
        load_ct(blk_of(bb + 1) * ib);
      }
    } else {
      if (kb != 32) {
        for (int o = tid; o < 1024; o += kThreads) Ts[(o >> 5) * 34 + (o & 31)] = make_int2(0, 0);
        __syncthreads();
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int o = tid + k * kThreads, i = kb == 32 ? o & 31 : o % kb, j = kb == 32 ? o >> 5 : o / kb;
        if (o < kb * kb) {
          const int64_t f = to_fixed(tv[k], 63 - eT) >> 7;
          const int h = (int)((f + (1 << 27)) >> 28), l = (int)(f - ((int64_t)h << 28));
          Ts[notrans ? j * 34 + i : i * 34 + j] = make_int2(h, l);
        }
      }
      if (bb + 1 < nbk) {
        const int cn = blk_of(bb + 1) * ib;
        prefetch_v(cn);
        load_t(cn);
        load_ct(cn);
      }
    }
    // ---- partial sums of W 2^(62 - E_c): lane = (digit j = q of V, reflector), 8 columns per warp -------
    int64_t* P = reinterpret_cast<int64_t*>(sm + kDigP);
    gram_partials<false>(P, tq, 25);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (!__syncthreads_and(ok ? 1 : 0)) {
      ok = false;
      break;
    }
    // ---- W = Ct + V^T C, split for the 32-bit multipliers: W 2^(58 - E_c) = 2^29 x + y --------------
    int64_t c63[2];
    int2* W = reinterpret_cast<int2*>(P);
    {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int o = (arow + k) * 33 + lane;
        c63[k] = to_fixed(ctv[k], 63 - myE);
        const int64_t s = (c63[k] >> 1) + P[o] + P[o + 32 * 33] + P[o + 64 * 33] + P[o + 96 * 33];
        const int64_t f = (s + 8) >> 4;
        const int h = (int)((f + (1 << 28)) >> 29), l = (int)(f - ((int64_t)h << 29));
        W[o] = make_int2(h, l);        // (only this thread reads P[o] of slot 0)
      }
    }
    __syncthreads();
    // ---- phase 2: W2 = op(T) W in integers, Ct -= W2, digits of W2 ----------------------------------
    if constexpr (kPre) {
      ok = mbar_wait(um.mbar + 32, (um.phase >> 4) & 1u, prm.wait_ns) && ok;
      um.phase ^= 16u;
    }
    int64_t w2[2];
    {
      int64_t A0 = 0, A1 = 0, B0 = 0, B1 = 0, D0 = 0, D1 = 0;
      const int t0 = notrans ? arow : 0, t1 = notrans ? kb : min(kb, arow + 2);
#pragma unroll 4
      for (int t = t0; t < t1; ++t) {
        const int2 w = W[t * 33 + lane];
        const int4 x = *reinterpret_cast<const int4*>(Ts + t * 34 + arow);
        A0 = wide(x.x, w.x, A0);
        B0 = wide(x.x, w.y, B0);
        D0 = wide(x.y, w.x, D0);
        A1 = wide(x.z, w.x, A1);
        B1 = wide(x.z, w.y, B1);
        D1 = wide(x.w, w.x, D1);
      }
      w2[0] = (int64_t)((uint64_t)A0 << (5 + eT)) + ((B0 + 2 * D0) >> (24 - eT));
      w2[1] = (int64_t)((uint64_t)A1 << (5 + eT)) + ((B1 + 2 * D1) >> (24 - eT));
      uint32_t d[8];
      digit_pair<8>(w2[0], w2[1], d);
      // W2 digit i, column c, reflector a at i 2048 + (c / 8) 512 + (a / 8) 128 + (c % 8) 16 + 2 (a % 8)
      unsigned char* p = sm + kDigW2 + (lane >> 3) * 512 + (lane & 7) * 16 + (arow >> 3) * 128 + (arow & 7) * 2;
#pragma unroll
      for (int i = 0; i < 8; ++i) *reinterpret_cast<uint32_t*>(p + i * 2048) = d[i];
    }
    // ---- rows that fixed point would lose ------------------------------------------------------------
    bool nz, strong, pivot = false;    // V has an entry in row r, one of 2^-8; a pivot row is lost
    if constexpr (kPre) {
      const uint32_t* hd = reinterpret_cast<const uint32_t*>(sm + kDigT + kDigTBytes) + 4 + (warp & 7);
      nz = (hd[0] >> lane) & 1;
      strong = (hd[8] >> lane) & 1;
    } else {
      strong = row_bit(red + 32);
      nz = row_bit(red + 16);
      if (type == UNMQR && r >= c0 && r < c0 + kb && Ts[35 * (r - c0)].x == 0) {      // (not the unit entry of H = I)
        nz = false;
        for (int a = c0; a < r; ++a) nz = nz || ldg(X + toff(r, a, nb, tr)) != 0.0;
      }
    }
    if (top) {
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (Ts[(arow + k) * 35].x > ((1 << 29) - (1 << 14)) >> eT) {      // tau, warp-uniform
          const bool is_big = __any_sync(kFull, abs_hi(c63[k]) >= kSmallRow || abs_hi(w2[k]) >= 1u << (30 - 10));
          pivot = pivot || (__any_sync(kFull, w2[k] != 0) && !is_big);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(pivot || (small_row && nz && !(narrow && strong)))) {
      uint32_t big = 0;
#pragma unroll
      for (int c = 0; c < 16; ++c) big = max(big, abs_hi(cf[c]));
      // uniform: the rest goes to the FP64 units
      if (rows_lost(sm, kb, eT, big, nz, w2[0], w2[1], pivot, narrow, type == UNMQR ? c0 : -kDigRows)) {
        if (!kPre && bb + 1 < nbk) ok = wait_v() && ok;
        break;
      }
    }
    touched = touched || nz;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- phase 3: V W2, digit pairs of equal weight in one accumulator ------------------------------
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
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (top && lane < ncols && arow + k < kb && w2[k] != 0)
        stg(Cp + toff(c0 + arow + k, col0 + lane, nb, tr), from_fixed(c63[k] - 2 * w2[k], 63 - myE));
    // ---- C -= V W2 in integers: C 2^(63 - E_c) loses D_g 2^(51 - 8 g) -------------------------------
    if (kPre && uwarp == kIssueWarp && bb + 1 < nbk) {
      // V's place is free when the last half's products are (the first half's were issued before them)
      ok = mbar_wait(um.mbar + 8 * h1, (um.phase >> h1) & 1u, prm.wait_ns) && ok;
      __syncwarp();
      load_image(blk_of(bb + 1));
    }
    if (hw >= h0 && hw < h1) {         // warp-uniform
      ok = mbar_wait(um.mbar + 8 + 8 * hw, (um.phase >> (1 + hw)) & 1u, prm.wait_ns) && ok;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      __syncwarp();
#pragma unroll
      for (int cg = 0; cg < 16; cg += 4) {
        uint32_t d[8][4];
#pragma unroll
        for (int g = 0; g < 8; ++g) tmem_ld4(tq + 256 * hw + 32 * g + cb + cg, d[g]);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          constexpr uint32_t kOff = kMagicBits * 257u;
          const int p01 = (int)(mag(d[0][c]) * 256 + mag(d[1][c]) - kOff), p23 = (int)(mag(d[2][c]) * 256 + mag(d[3][c]) - kOff);
          const int p45 = (int)(mag(d[4][c]) * 256 + mag(d[5][c]) - kOff), p67 = (int)(mag(d[6][c]) * 256 + mag(d[7][c]) - kOff);
          const int64_t x = wide(p23, -(1 << 27), wide(p45, -(1 << 11), cf[cg + c])) - (p67 >> 5);
          cf[cg + c] = x - (int64_t)((uint64_t)(uint32_t)p01 << 43);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    for (int h = h0; h < h1; ++h) um.phase ^= 2u << h;
    ++done;
  }
  if (!__syncthreads_and(ok ? 1 : 0)) return timed_out();
  // ---- store the strip ----------------------------------------------------------------------------
  if (own && touched) {
    if (tr) {
#pragma unroll
      for (int c = 0; c < 16; c += 2)
        if (cb + c < ncols)
          __stcg(reinterpret_cast<double2*>(C + (size_t)r * nb + col0 + cb + c),
                 make_double2(from_fixed(cf[c], 63 - colE[cb + c]), from_fixed(cf[c + 1], 63 - colE[cb + c + 1])));
    } else {
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (cb + c < ncols)
          stg(C + r + (size_t)(col0 + cb + c) * nb, from_fixed(cf[c], 63 - colE[cb + c]));
    }
  }
  __syncthreads();
  return done;
}
#endif  // BD_EXEC_PART == 1
