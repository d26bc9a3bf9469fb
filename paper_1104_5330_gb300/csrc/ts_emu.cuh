// Double-precision contractions on the 5th-generation tensor cores.
//
// GB300 issues 2 FP64 multiply-adds per SM and clock, against 4096 f16 products:
// the FP64 pipe bounds every double-precision pass that contracts on it. Here the
// contractions run as exact integer arithmetic on tcgen05.mma kind::f16:
//  * data: a tile's values are turned into 64-bit fixed point relative to the
//    largest magnitude of their line (61 bits below it), on the integer units, and
//    cut into eight bytes u_i. (Where all values of a block lie within a factor of
//    eight to sixteen of each other, its largest stands for that of its lines.) A byte
//    zero-extended to 16 bits is the f16 subnormal u_i 2^-24, so the digits need no
//    conversion. Balanced digits are d_i = u_i - 128 (the fixed-point value has
//    0x8080...80 added);
//  * matrix: every row scaled to 62 bits, in eight balanced base-256 digits e_j as
//    f16 integers (built on the host from the exact products of its factors);
//  * the products d_i e_j of order o = i + j <= 7 are accumulated in f32, one
//    tensor-memory column per output and order: multiples of 2^-24 that stay below
//    2^22 units (checked on the host), so every accumulation is exact. One MMA per
//    digit i covers all e_j (N = outputs x (8 - i), accumulator columns shifted by
//    i x outputs). A first MMA sets every accumulator to 0.75 - 128 sum e_j
//    2^-24: it removes the byte offset, and the accumulator's bit pattern is then
//    0x3F400000 + (the exact integer sum);
//  * the eight sums are recombined in a 64-bit integer (orders >= 8, 2^-59 of the
//    full scale, are dropped) and rounded once to double on the integer units.
// The method is Ozaki's splitting into slices whose products are exact (Ozaki, Ogita, Oishi
// and Rump 2012, Numer. Algorithms 59) with integer slices (Ootomo, Ozaki and Yokota 2024).
// The error of a contraction is a few units of 2^-57 x (largest matrix entry of the row) x
// (largest value of the line) and that one rounding. In units of 2^-53 x row sum x largest
// value of the point's own lines a right-hand side is off by 0.1 to 10, the FP64 multiply-adds
// by 0.4 to 20 on the same fields: smooth ones, beams, isolated bright points, magnitudes that
// vary by 2^60 between directions or positions (tests/test_gpu_line_precision.py); in the
// relative 2-norm by 4e-16 (17 x 6 x 8 x 16^2, smooth), 1e-15 (33 x 4^2 x 16^2) against 4e-15,
// 6e-15.
// A line that holds an infinity or a NaN gives NaN.
//
// What bounds the passes: no unit (profiles/fp64_tensorcore_passes.md: issue slots 38 to 44 %,
// integer pipes 22 to 36, FP64 22 to 40, tensor pipe 10 to 11, HBM 7 to 20 % busy), but the
// order of work: the 16 warps that registers allow on an SM load, cut, wait for the products
// and finish points in the same phases, with four or more CTA barriers a tile and dependent
// integer instructions (200 to 235 a point) between them.
//
// Every wait is bounded: if one runs out the kernel sets the grid's error flag
// (ts_sync_status reports TS_ERR_TIMEOUT), waits again for its own MMAs, frees its
// tensor memory and returns.
#pragma once

#include <stdint.h>

#include <type_traits>

#include "ts_emu.h"
#include "ts_kernels.cuh"

namespace ts {
namespace emu {

constexpr uint32_t kMagic = 0x3F400000u;   // bits of 0.75f

__device__ __forceinline__ uint32_t sm_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool bar_wait(uint32_t addr, uint32_t parity, long long iters) {
  for (long long it = 0; it < iters; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}

// Shared-memory matrix descriptors, no swizzle. K-major operand (8-row x 16-byte
// cores): lbo the distance of cores along K, sbo of 8-row groups. MN-major operand
// (cores of 8 K x 8 rows, rows fastest): lbo the distance of 8-deep K groups, sbo of
// 8-row groups. Low word: address and lbo in 16-byte units; high word: sbo, version.

// One MMA chain step: D[128 x N] += A B. Called by a whole warp with warp-uniform
// arguments, `one` set on the elected lane: operands in uniform registers issue an
// MMA every 62 clocks, against 163 from a divergent branch of one thread. The
// descriptors come in halves: the high words do not change along a chain.
__device__ __forceinline__ uint32_t idesc_f16(int N, bool a_mn) {
  return (1u << 4) | (a_mn ? 1u << 15 : 0u) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(uint32_t one, uint32_t d, uint32_t alo, uint32_t ahi,
                                        uint32_t blo, uint32_t bhi, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n"
      " setp.ne.b32 q, %7, 0;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n"
      :: "r"(d), "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"(one)
      : "memory");
}
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo) {
  return (saddr >> 4) | ((lbo >> 4) << 16);
}
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }

// The chain of one accumulator tile: the bias step, then for every digit i and K
// step the products with the matrix digits j <= 7 - i. a: digit 0 of the rows (MN-
// major, digit stride ad, row-group stride asbo); K steps: OWN pairs of K cores of
// the line, the same of the partner `part` bytes on (PART), then (ODD) one step of
// the line's and the partner's last cores. b: the matrix (bias core, `skip` more
// cores, K cores), `rows` rows a core; n outputs. Unrolled: an MMA then issues every
// 50 clocks, against 153 from run-time loops over digits and K steps.
template <int OWN, bool PART, bool ODD>
__device__ __forceinline__ void chain_steps(uint32_t one, uint32_t tm, uint32_t bias, uint32_t a,
                                            uint32_t ad, uint32_t asbo, uint32_t part, uint32_t b,
                                            int skip, int rows, int n) {
  const uint32_t core = (uint32_t)rows;   // 16-byte units
  const uint32_t bhi = desc_hi(128), ahi = desc_hi(asbo);
  const uint32_t b0 = desc_lo(b, core * 16u), bk = b0 + core * (uint32_t)(1 + skip);
  const uint32_t a0 = desc_lo(a, 128);
  mma_f16(one, tm, desc_lo(bias, 2048), desc_hi(128), b0, bhi, idesc_f16((8 * n + 15) & ~15, false),
          0);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t id = idesc_f16(((8 - i) * n + 15) & ~15, true);
    const uint32_t d = tm + (uint32_t)(i * n), al = a0 + (uint32_t)i * (ad >> 4);
#pragma unroll
    for (int ks = 0; ks < OWN; ++ks)
      mma_f16(one, d, al + 16u * ks, ahi, bk + 2 * core * ks, bhi, id, 1);
    if (PART) {
#pragma unroll
      for (int ks = 0; ks < OWN; ++ks)
        mma_f16(one, d, al + (part >> 4) + 16u * ks, ahi, bk + 2 * core * (OWN + ks), bhi, id, 1);
      if (ODD)
        mma_f16(one, d, (al & 0xFFFFu) + 16u * OWN + ((part >> 4) << 16), ahi, bk + 4 * core * OWN,
                bhi, id, 1);
    }
  }
}
// The same with run-time K steps, and column blocks of 256 for wider accumulators.
__device__ __noinline__ void chain_any(uint32_t one, uint32_t tm, uint32_t bias, uint32_t a,
                                       uint32_t ad, uint32_t asbo, int own, uint32_t part, bool odd,
                                       uint32_t b, int skip, int rows, int n) {
  const uint32_t core = (uint32_t)rows;
  const uint32_t bhi = desc_hi(128), ahi = desc_hi(asbo);
  const uint32_t b0 = desc_lo(b, core * 16u), bk = b0 + core * (uint32_t)(1 + skip);
  const uint32_t a0 = desc_lo(a, 128);
  for (int c0 = 0; c0 < 8 * n; c0 += 256)
    mma_f16(one, tm + c0, desc_lo(bias, 2048), desc_hi(128), b0 + c0, bhi,
            idesc_f16(min((8 * n - c0 + 15) & ~15, 256), false), 0);
  for (int i = 0; i < 8; ++i)
    for (int c0 = 0; c0 < (8 - i) * n; c0 += 256) {
      const uint32_t id = idesc_f16(min(((8 - i) * n - c0 + 15) & ~15, 256), true);
      const uint32_t d = tm + (uint32_t)(i * n + c0), al = a0 + (uint32_t)i * (ad >> 4);
      uint32_t bl = bk + (uint32_t)c0;
      for (int ks = 0; ks < own; ++ks, bl += 2 * core)
        mma_f16(one, d, al + 16u * ks, ahi, bl, bhi, id, 1);
      if (part) {
        for (int ks = 0; ks < own; ++ks, bl += 2 * core)
          mma_f16(one, d, al + (part >> 4) + 16u * ks, ahi, bl, bhi, id, 1);
        if (odd)
          mma_f16(one, d, (al & 0xFFFFu) + 16u * own + ((part >> 4) << 16), ahi, bl, bhi, id, 1);
      }
    }
}

__device__ __forceinline__ uint32_t elect_one() {
  uint32_t one;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(one));
  return one;
}

__device__ __forceinline__ void mma_commit(uint32_t one, uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n"
      :: "r"(bar), "r"(one) : "memory");
}

// Four consecutive tensor-memory columns of this warp's 32 lanes, for each of the
// eight orders (n columns apart): b[o][e].
__device__ __forceinline__ void tm_ld(uint32_t addr, int n, uint32_t (&b)[8][4]) {
#pragma unroll
  for (int o = 0; o < 8; ++o)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(b[o][0]), "=r"(b[o][1]), "=r"(b[o][2]), "=r"(b[o][3])
                 : "r"(addr + (uint32_t)(o * n)));
}
// Waits for the loads of b (its registers are operands: no use moves ahead).
__device__ __forceinline__ void tm_wait(uint32_t (&b)[8][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int o = 0; o < 8; ++o)
    asm volatile("" : "+r"(b[o][0]), "+r"(b[o][1]), "+r"(b[o][2]), "+r"(b[o][3]));
}

// 64-bit fixed point of v relative to 2^(emax - 1022), 61 bits below it, plus the
// digit bias; EM = emax << 20 | 0xFFFFF with emax >= 64 (zeros and subnormals then
// shift out completely).
__device__ __forceinline__ uint64_t to_fixed(double v, uint32_t EM) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t s = (EM - (hi & 0x7FFFFFFFu)) >> 20;
  const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32 | lo) << 8;
  uint64_t x;
  asm("shr.u64 %0, %1, %2;" : "=l"(x) : "l"(m), "r"(s));   // shifts of 64 and more give 0
  // two's complement and digit bias in one addition
  const uint32_t sg = (uint32_t)((int32_t)hi >> 31);
  const uint32_t xl = (uint32_t)x ^ sg, xh = (uint32_t)(x >> 32) ^ sg;
  return (((uint64_t)xh << 32) | xl) + ((0x80808080ull << 32) | (uint64_t)(0x80808080u - sg));
}
// far: set if v is not zero and more than kNear places below.
constexpr uint32_t kNear = 3;
__device__ __forceinline__ bool far_below(uint32_t mag, uint32_t EM) {   // one range test
  return EM - mag - ((kNear + 1) << 20) < EM - ((kNear + 2) << 20) + 1u;
}
__device__ __forceinline__ uint64_t to_fixed(double v, uint32_t EM, bool& far) {
  far |= far_below((uint32_t)__double2hiint(v) & 0x7FFFFFFFu, EM);
  return to_fixed(v, EM);
}
// Eight values relative to the exponent bases of their lines (16 bits each, 0 for a line of
// zeros). Tiny lines, bases below 64, are brought up first if there are any (lift).
__device__ __forceinline__ void to_fixed_lines(const double (&v)[8], uint4 e, bool lift,
                                               uint64_t (&f)[8]) {
  const uint32_t w[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
  for (int x = 0; x < 8; x += 2) {
    if (!lift) {
      const uint32_t b = __vmaxs2(w[x / 2], 0x00400040u);
      f[x] = to_fixed(v[x], b << 20 | 0xFFFFFu);
      f[x + 1] = to_fixed(v[x + 1], (b & 0xFFFF0000u) << 4 | 0xFFFFFu);
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t b = h ? w[x / 2] >> 16 : w[x / 2] & 0xFFFFu;
        const bool up = b < 64;
        f[x + h] = to_fixed(up ? v[x + h] * __hiloint2double((1023 + 256) << 20, 0) : v[x + h],
                            (up ? b + 256 : b) << 20 | 0xFFFFFu);
      }
    }
  }
}
__device__ __forceinline__ int64_t sra(int64_t v, int n) {   // shifts of 64 and more: the sign
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}

__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// sum_o b_o 256^(7-o) / 256 without the accumulators' offset, as a signed 64-bit
// integer (modulo 2^64; the true value stays below 2^62).
__device__ __forceinline__ int64_t recombine(uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3,
                                             uint32_t b4, uint32_t b5, uint32_t b6, uint32_t b7) {
  constexpr uint64_t M = kMagic;
  constexpr uint64_t C = 0ull - ((M << 48) + (M << 40) + (M << 32) + (M << 24) + (M << 16) +
                                 (M << 8) + M + (M >> 8));
  uint64_t r = mad_wide(b5, 256u, C);
  r = mad_wide(b4, 65536u, r);
  r = mad_wide(b3, 16777216u, r);
  r = mad_wide(b6 + (b7 >> 8), 1u, r);
  const uint32_t h = b0 * 65536u + (b1 * 256u + b2);
  return (int64_t)(r + ((uint64_t)h << 32));
}

// R 2^q as a double, qb = q + 1022: rounded to nearest on the integer units. Rare
// values (|R| < 2^32, exponents near the ends of the range, NaN blocks) take the
// careful path.
__device__ __noinline__ double to_double_slow(int64_t R, int qb) {
  if (qb > 4000) return __longlong_as_double(0x7FF8000000000000ll);   // the block holds Inf or NaN
  if (R == 0) return 0.0;
  return scalbn((double)R, qb - 1022);
}

// The fast path without its checks, e0 = (q + 1022 + 62) << 20; the result is wrong
// where |R| < 2^32 (the high word of |R| is returned in `top`).
__device__ __forceinline__ double to_double_fast(int64_t R, int e0, uint32_t& top) {
  const int32_t sg = (int32_t)(R >> 63);
  const uint32_t hi = (uint32_t)((uint64_t)R >> 32) ^ (uint32_t)sg;
  const uint32_t lo = (uint32_t)R ^ (uint32_t)sg;
  top = hi;
  const int sh = __clz((int)hi) - 1;
  const uint32_t h2 = __funnelshift_l(lo, hi, sh), l2 = lo << (sh & 31);
  const uint64_t w = (((uint64_t)h2 << 32) | l2) + 0x200u;
  const uint32_t wh = (uint32_t)(w >> 32), wl = (uint32_t)w;
  const uint32_t dl = __funnelshift_r(wl, wh, 10);
  const uint32_t dh = (wh >> 10) + (uint32_t)(e0 - (sh << 20));
  return __hiloint2double((int)(dh | ((uint32_t)sg & 0x80000000u)), (int)dl);
}

// The four recombined sums of one thread.
__device__ __forceinline__ void recombine4(const uint32_t (&b)[8][4], int64_t (&R)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e)
    R[e] = recombine(b[0][e], b[1][e], b[2][e], b[3][e], b[4][e], b[5][e], b[6][e], b[7][e]);
}
// y[e] = R[e] 2^q[e], qb[e] = q[e] + 1022; one branch for the rare careful cases of all
// four (lim = 1, or ~0 where the block needs them all).
__device__ __forceinline__ void to_double4(const int64_t (&R)[4], const int (&qb)[4], uint32_t lim,
                                           double (&y)[4]) {
  uint32_t top[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) y[e] = to_double_fast(R[e], (qb[e] + 62) << 20, top[e]);
  if (min(min(top[0], top[1]), min(top[2], top[3])) < lim) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (top[e] < lim) y[e] = to_double_slow(R[e], qb[e]);
  }
}
__device__ __forceinline__ uint32_t slow_limit(int qb);
__device__ __forceinline__ double to_double1(int64_t R, int qb) {
  uint32_t top;
  const double y = to_double_fast(R, (qb + 62) << 20, top);
  return top < slow_limit(qb) ? to_double_slow(R, qb) : y;
}
// 2^n as a double, -1022 < n < 1023
__device__ __forceinline__ double pow2(int n) { return __hiloint2double((1023 + n) << 20, 0); }
__device__ __forceinline__ uint32_t slow_limit(int qb) {
  return (uint32_t)(qb - 1) > 1900u ? 0xFFFFFFFFu : 1u;
}

// A line's key is its largest exponent and a mantissa of ones, 0 for a line of zeros (values
// below 2^-1042 count as such). Nothing is cut relative to less than kLeastKey; lines below
// that, if they are not zero, are scaled up by 2^256 first (tiny_key), and their key says
// so in its last bit.
constexpr uint32_t kLeastKey = 64u << 20 | 0xFFFFFu;
__device__ __forceinline__ uint32_t line_key(uint32_t mx) { return mx ? mx | 0xFFFFFu : 0u; }
__device__ __forceinline__ bool tiny_line(uint32_t mx) { return mx - 1u < (64u << 20) - 1u; }
__device__ __forceinline__ uint32_t tiny_key(uint32_t key) {
  return (max(key >> 20, 1u) + 257u) << 20 | 0xFFFFEu;
}
// The exponent base of a line, 5000 with an infinity or a NaN.
__device__ __forceinline__ int line_exp(uint32_t key) {
  const int e = (int)(key >> 20);
  return key == 0 ? 64 : !(key & 1u) ? e - 256 : e == 2047 ? 5000 : max(e, 64);
}

// The exponent base of a line of its own scale in a two-axis tile: 0 for a line of zeros.
__device__ __forceinline__ int line_base(uint32_t mx) {
  const int e = (int)(mx >> 20);
  return mx == 0 ? 0 : e == 2047 ? 5000 : max(e, 1);
}
// The fixed-point key of a block: its largest exponent, at least 64, and a mantissa of ones.
__device__ __forceinline__ uint32_t fixed_key(uint32_t mx) {
  return ((uint32_t)max((int)(mx >> 20), 64) << 20) | 0xFFFFFu;
}

// The exponent base of a block: emax of the stored maximum (high word of |v|),
// 5000 for a block with an infinity or a NaN.
__device__ __forceinline__ int block_exp(uint32_t mx) {
  const int e = (int)(mx >> 20);
  return e == 2047 ? 5000 : max(e, 64);
}

// Digits of 8 fixed-point values: P[w][h] packs 16-bit pieces of the values, two
// values per word: P[q][0..3] = bytes (2q, 2q+1) of values (0,1), (2,3), (4,5), (6,7).
__device__ __forceinline__ void pack_pairs(const uint64_t (&x)[8], int q, uint32_t (&w)[4]) {
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint32_t a = q < 2 ? (uint32_t)x[2 * p] : (uint32_t)(x[2 * p] >> 32);
    const uint32_t b = q < 2 ? (uint32_t)x[2 * p + 1] : (uint32_t)(x[2 * p + 1] >> 32);
    w[p] = __byte_perm(a, b, (q & 1) ? 0x7632 : 0x5410);
  }
}
__device__ __forceinline__ uint4 digit_of(const uint32_t (&w)[4], bool high) {
  const uint32_t s = high ? 0x4341 : 0x4240;
  return make_uint4(__byte_perm(w[0], 0, s), __byte_perm(w[1], 0, s), __byte_perm(w[2], 0, s),
                    __byte_perm(w[3], 0, s));
}

// Bias operand of the first MMA: every row [0.75, 2^-11, 2^-17, 0...].
__device__ __forceinline__ void fill_bias(unsigned char* ca, int rows) {
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    reinterpret_cast<uint4*>(ca)[r] = make_uint4(0x10003A00u, 0x00000080u, 0u, 0u);
    reinterpret_cast<uint4*>(ca)[rows + r] = make_uint4(0u, 0u, 0u, 0u);
  }
}

__device__ __forceinline__ void copy_in(unsigned char* dst, const void* src, int bytes) {
  const uint4* s = reinterpret_cast<const uint4*>(src);
  for (int x = threadIdx.x; x < bytes / 16; x += blockDim.x) reinterpret_cast<uint4*>(dst)[x] = s[x];
}

// ============================================================================
// Two-axis passes. A tile is Na x Nb x XW points (a, b, x), XW = 8 or 4:
//  * angular: a = Theta, b = Phi, x = XW angular blocks;
//  * plane: a = theta, b = phi, x = XW Phi columns, half of them of each half circle.
// The a axis is a double-Fourier-sphere axis: its operator takes the line and the
// line of the partner (b + Nb/2; in the plane pass also the column of the other
// half circle). The b axis is periodic. Both contractions read the tile's digits
// as MN-major operands, rows (b, x) or (a, x) in groups of eight (8 x of one b or a,
// or 4 x of two):
//   copy 1 [digit][b in 0..Nb-1, 0..Nb/2-1][a][8 rows] -- K along a; the partner's
//           rows start Nb/2 further on, hence the repeated first half;
//   copy 2 [digit][a][b][8 rows]                       -- K along b.
// Where both do not fit, the tile has four x and the copies take turns in one buffer
// (seq): copy 1 is written when the Fourier products are done; the DFS products run
// under the Fourier epilogue.
// The Fourier results (and, in the angular pass, the moments formed from its Phi sums) go
// through shared memory to the threads that finish the points from the DFS results.
// EP_ADJOINT is the transposed angular pass: the same contractions with the transposed
// matrices, lt in place of U, and the adjoint's own epilogue.
enum EmuPass { EP_ANGULAR = 0, EP_PLANE = 1, EP_ADJOINT = 2 };

struct EmuArgs {
  const double* U;
  double* K;
  double sgn;
  int collision, cons;
  // EP_ADJOINT: K holds Ubar (read); gradients, adjoint fields and their weights
  const double* Us;
  double *gk, *ge;
  const double *lam, *lam_in;
  double *lam_out, *Kbar;
  double wl, wu;
  int vec;   // the values may be loaded four (two) at a time
  long long ntiles;
};

struct MatArg {
  const uint16_t* dev;
  int se;          // 3 - s of the whole matrix
};

// A moment's share of this warp: w summed over its rows of the same x (lanes XW apart), added
// to what the warp's earlier rows gave (`add`). One warp owns each share.
template <int XW>
__device__ __forceinline__ void moment(double* s, double w, bool add) {
  if (XW == 4) w += __shfl_xor_sync(0xFFFFFFFFu, w, 4);
  w += __shfl_xor_sync(0xFFFFFFFFu, w, 8);
  w += __shfl_xor_sync(0xFFFFFFFFu, w, 16);
  if ((threadIdx.x & 31) < XW) *s = add ? *s + w : w;
}
// The shift that makes room for the coefficient sinTh cot th.
__device__ __forceinline__ int cot_shift(double cot, int delta) {
  const int e = (int)((uint32_t)__double2hiint(cot) >> 20 & 0x7FFu) - 1023;   // 0: far below
  return max(1, 2 + delta + e);
}

__device__ __forceinline__ void cp8(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" :: "r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Where a tile lies in the field.
template <int PASS>
struct TileAt {
  long long b0 = 0, base = 0;   // angular: first block; plane: (g, i, Theta) offset
  int k = 0, i = 0, m0 = 0;
};
template <int PASS, int XW>
__device__ __forceinline__ TileAt<PASS> tile_at(const Dims& d, long long tile) {
  TileAt<PASS> r;
  if (PASS != EP_PLANE) {
    r.b0 = tile * XW;
  } else {
    constexpr unsigned H = XW / 2;
    const unsigned nch = ((unsigned)(d.NP / 2) + H - 1) / H;
    unsigned q = (unsigned)tile;   // tiles of a field fit 32 bits (checked on the host)
    r.m0 = (int)(q % nch * H);
    q /= nch;
    r.k = (int)(q % (unsigned)d.NT);
    q /= (unsigned)d.NT;
    r.i = (int)(q % (unsigned)d.Nr);
    r.base = (long long)(q / (unsigned)d.Nr) * d.S_g + (long long)r.i * d.S_i +
             (long long)r.k * d.NP;
  }
  return r;
}
__device__ __forceinline__ void ld2(const double* p, double& a, double& b) {
  const double2 y = *reinterpret_cast<const double2*>(p);
  a = y.x;
  b = y.y;
}
// The values of this thread's units (zero outside the tile). A unit is eight rows of
// copy 1 at one a: (b; 8 x), or (b, b + 1; 4 x).
template <int PASS, int U, int XW>
__device__ __forceinline__ void load_units(const Dims& d, const double* F, const TileAt<PASS>& at,
                                           int S, int hP, int Nb, bool vec, const int (&ua)[U],
                                           const int (&ub)[U], double (&v)[U][8]) {
#pragma unroll
  for (int q = 0; q < U; ++q) {
#pragma unroll
    for (int x = 0; x < 8; ++x) v[q][x] = 0.0;
    if (ua[q] < 0) continue;
    if (PASS != EP_PLANE) {
      const double* src = F + at.b0 * S + ua[q] * Nb + ub[q];
      if (XW == 8) {
#pragma unroll
        for (int x = 0; x < 8; ++x)
          if (at.b0 + x < d.nblk) v[q][x] = src[x * S];
      } else {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          if (at.b0 + x >= d.nblk) continue;
          if (vec) {
            ld2(src + x * S, v[q][x], v[q][x + 4]);
          } else {
            v[q][x] = src[x * S];
            v[q][x + 4] = src[x * S + 1];
          }
        }
      }
    } else {
      const double* src = F + at.base + (long long)ua[q] * d.S_j + (long long)ub[q] * d.S_l + at.m0;
      if (XW == 8) {
        if (vec) {   // four columns of a half circle at once: every lane reads its own line
#pragma unroll
          for (int x = 0; x < 8; x += 4)
            asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                         : "=d"(v[q][x]), "=d"(v[q][x + 1]), "=d"(v[q][x + 2]), "=d"(v[q][x + 3])
                         : "l"(src + (x ? hP : 0)));
        } else {
#pragma unroll
          for (int x = 0; x < 8; ++x)
            if (at.m0 + (x & 3) < hP) v[q][x] = src[(x & 3) + (x >= 4 ? hP : 0)];
        }
      } else {
#pragma unroll
        for (int x = 0; x < 8; x += 2) {   // pairs of columns: (b, half)
          const double* z = src + (x >= 4 ? d.S_l : 0) + (x & 2 ? hP : 0);
          if (vec) {
            ld2(z, v[q][x], v[q][x + 1]);
          } else {
            if (at.m0 < hP) v[q][x] = z[0];
            if (at.m0 + 1 < hP) v[q][x + 1] = z[1];
          }
        }
      }
    }
  }
}

// NA_, NB_: the axes' lengths at compile time (0: from the geometry).
template <int PASS, int KF, int T, int NA_, int NB_, int XW>
__global__ void __launch_bounds__(T, T == 256 ? 2 : 1)
k_emu2(Problem p, Tables<double> t, EmuGeo g, MatArg m1, MatArg m2, EmuArgs A) {
  extern __shared__ __align__(128) unsigned char sm[];
  const Dims& d = p.d;
  const uint32_t smb = sm_u32(sm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int uwarp = __shfl_sync(0xFFFFFFFFu, warp, 0);   // warp-uniform
  constexpr int NG = T / 128;                     // threads per tensor-memory lane
  constexpr int U = 1;                            // units of a tile a thread holds (host)
  const int Na = NA_ ? NA_ : g.Na, Nb = NB_ ? NB_ : g.Nb, hb = Nb / 2, exP = Na * XW + 8;
  // small arrays
  unsigned char* ms = sm + g.oMs;
  uint64_t* bar = reinterpret_cast<uint64_t*>(ms);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(ms + 16);
  volatile uint32_t* wmask = reinterpret_cast<volatile uint32_t*>(ms + 20);   // see wide below
  volatile uint32_t* wflag = reinterpret_cast<volatile uint32_t*>(ms + 24);   // [2]
  uint32_t* smax = reinterpret_cast<uint32_t*>(ms + 32);          // [2][8]
  int16_t* ln1 = reinterpret_cast<int16_t*>(sm + g.oLn);   // lines' exponents: a-circles [hb][XW],
  int16_t* ln2 = ln1 + hb * XW;                            // b-lines [Na][XW]
  double* xs = reinterpret_cast<double*>(ms + 96);                // [2][8][8] scalars of a tile's x
  double* xm = xs + 2 * 64;                                       // [10][8] moments
  constexpr int nm = emu_moments(KF), nw = emu_weights(KF);
  double* wt = xm + 80;                                           // angular: weights [nw][Na]
  double* msum = wt + nw * Na;                                    // angular: [4 warps][nm][8]
  int* hs = reinterpret_cast<int*>(xm + 80);                      // plane: shifts [Na]
  double* gp = msum;                      // adjoint: [mt1][warps][8], once the moments are formed
  int64_t* ex = reinterpret_cast<int64_t*>(sm + g.oEx);           // [Nb][a][XW]

  if (Na % 8 || Nb % 16 || g.seq) {   // K paddings hold finite digits (their products vanish)
    for (int x = tid; x < g.oB1 / 16; x += T)
      reinterpret_cast<uint4*>(sm)[x] = make_uint4(0, 0, 0, 0);
  }
  if (tid < 16) smax[tid] = 0;
  if (tid < 2) wflag[tid] = 0;
  copy_in(sm + g.oB1, m1.dev, (1 + g.kc1) * g.r1 * 16);
  copy_in(sm + g.oB2, m2.dev, (1 + g.kc2) * g.r2 * 16);
  fill_bias(sm + g.oCA, 128);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_u32(&bar[0])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_u32(&bar[1])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(sm_u32(tslot)), "r"(g.cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    pass_started();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tslot, 0);

  // this thread's (a, b) units: all eight x of each
  int ua[U], ub[U];
#pragma unroll
  for (int q = 0; q < U; ++q) {
    const int u = tid + q * T;
    if (XW == 8) {
      ua[q] = u < Na * Nb ? u / Nb : -1;
      ub[q] = u - (u / Nb) * Nb;
    } else {   // neighbouring lanes hold a and a + 1: their halves of a row of copy 2
      ua[q] = u / Nb * 2 + (u & 1);
      ub[q] = (u - u / Nb * Nb) / 2 * 2;
      if (ua[q] >= Na) ua[q] = -1;
    }
  }
  const int row = (warp & 3) * 32 + lane, grp = warp >> 2, rx = row & (XW - 1), rg = row / XW;
  constexpr int XH = XW / 2;
  constexpr int RT = 128 / XW;                    // a's or b's of a 128-row tile
  const int jobs = g.mt2 + g.mt1, ahead = g.dual ? 2 : 1;
  const int S = PASS != EP_PLANE ? Na * Nb : d.NT * d.NP, hP = d.NP / 2;
  // The combination W of the two contractions stays in fixed point: a multiply of two
  // 64-bit integers takes 28 issue slots of a warp, an FP64 one 64. Unit of W: 2^h times that
  // of the DFS results; h makes room for the Fourier term's coefficient, delta is the
  // difference of the two matrices' scales.
  const int delta = m2.se - m1.se;
  for (int a = tid; a < Na; a += T) {
    if (PASS == EP_PLANE) {
      hs[a] = max(2, 3 + delta + ilogb(t.inv_sinth[a]));
    } else {   // weights of the moments (Fejer x trapezoid; conservative: of Fhat / sinTh;
               // adjoint: plain sums) times 1, cos and sin of Theta
      const double st = t.sinT[a];
      const double q = PASS == EP_ADJOINT ? 1.0 : A.cons ? t.qdir[a] / st : t.qdir[a];
      wt[a] = q;
      if (KF >= KF_LINEAR) {
        wt[Na + a] = q * t.cosT[a];
        wt[2 * Na + a] = q * st;
      }
    }
  }
  double v[U][8];
  TileAt<PASS> at{};
  // block z of tile `at`: the epilogue's constants, as asynchronous copies (their
  // latency is nobody's): 1/r, kappa, cot th, eta, kappa_s, kappa_s' b, c, sin th
  auto scalars_load = [&](int z, int bf) {
    const long long blk = at.b0 + z < d.nblk ? at.b0 + z : 0;
    const unsigned q = (unsigned)blk / (unsigned)d.Np;
    const unsigned jj = q % (unsigned)d.Nt, ii = q / (unsigned)d.Nt % (unsigned)d.Nr;
    const uint32_t x = sm_u32(xs + bf * 64 + z);
    cp8(x, t.inv_r + ii);
    cp8(x + 64, p.kap + blk);
    cp8(x + 128, t.cot_th + jj);
    cp8(x + 192, p.eta + blk);
    cp8(x + 256, p.kaps + blk);
    if (KF >= KF_LINEAR && p.scb) cp8(x + 320, p.scb + blk);
    if (KF >= KF_QUADRATIC) cp8(x + 384, p.scc + blk);
    cp8(x + 448, t.sin_th + jj);
  };
  pass_wait();
  if ((long long)blockIdx.x < A.ntiles) {
    at = tile_at<PASS, XW>(d, blockIdx.x);
    load_units<PASS, U, XW>(d, A.U, at, S, hP, Nb, A.vec, ua, ub, v);
    if (PASS != EP_PLANE && warp == 1 && lane < XW) scalars_load(lane, 0);
  }
  int coef_n = -1;   // the Fourier coefficient this thread holds, and for what
  double coef_key = 0.0;
  int64_t coef = 0;
  int cth_b = -1;    // plane: cosPh of its DFS rows, and of which
  int64_t cth = 0;
  uint32_t phase = 0;   // one bit per barrier
  bool alive = true, late = false;   // late: a wait of this thread ran out
  bool guess = false;                // the tile before was wide
  int buf = 0;
  for (long long tile = blockIdx.x; tile < A.ntiles && alive; tile += gridDim.x, buf ^= 1) {
    // ---- largest magnitude of each block (angular) or of the tile (plane)
    {
      uint32_t mx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
      for (int q = 0; q < U; ++q)
#pragma unroll
        for (int x = 0; x < 8; ++x)
          mx[x] = max(mx[x], (uint32_t)__double2hiint(v[q][x]) & 0x7FFFFFFFu);
      if (PASS == EP_PLANE) {
#pragma unroll
        for (int x = 1; x < 8; ++x) mx[0] = max(mx[0], mx[x]);
        const uint32_t r = __reduce_max_sync(0xFFFFFFFFu, mx[0]);
        if (lane == 0) atomicMax(&smax[buf * 8], r);
      } else {
        uint32_t mine = 0;
        if (XW == 4) {
#pragma unroll
          for (int x = 0; x < 4; ++x) mx[x] = max(mx[x], mx[x + 4]);
        }
#pragma unroll
        for (int x = 0; x < XW; ++x) {
          const uint32_t r = __reduce_max_sync(0xFFFFFFFFu, mx[x]);
          if (lane == x) mine = r;
        }
        if (lane < XW) atomicMax(&smax[buf * 8 + lane], mine);
      }
    }
    if (PASS != EP_PLANE && warp == 1) cp8_wait();   // this tile's scalars
    __syncthreads();   // the maxima and scalars; the previous tile is finished
    if (tid < 8) {
      smax[(buf ^ 1) * 8 + tid] = 0;
      // tiny blocks and blocks with an infinity or a NaN: line by line
      const uint32_t mx = smax[buf * 8 + tid];
      if (tiny_line(mx) || mx >= 0x7FF00000u) wflag[buf] = 1;
    }
    if (tid == 8) wflag[buf ^ 1] = 0;
    // ---- digits
    auto fence_digits = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    uint64_t f4[XW == 4 ? U : 1][8];   // kept for the second copy
    // the copies of a unit's digits
    auto put = [&](const uint64_t (&f)[8], int q, bool one, bool two) {
      constexpr int H = XW / 2;
      unsigned char* c1 = sm + g.oC1 + ub[q] * XW / 8 * g.sb1 + ua[q] * 16;
      unsigned char* c2 = XW == 8 ? sm + g.oC2 + ua[q] * g.sb2 + ub[q] * 16
                                  : sm + g.oC2 + (ua[q] >> 1) * g.sb2 + ub[q] * 16 + (ua[q] & 1) * 8;
      const bool ring = ub[q] < hb, rot = PASS == EP_PLANE && !ring;
#pragma unroll
      for (int w = 3; w >= 0; --w) {
        uint32_t pk[4];
        pack_pairs(f, w, pk);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int dig = 7 - (2 * w + h);
          const uint4 x4 = digit_of(pk, h);
          if (two) {
            if (XW == 8) {
              *reinterpret_cast<uint4*>(c2 + dig * g.d2) = x4;
            } else {
              *reinterpret_cast<uint2*>(c2 + dig * g.d2) = make_uint2(x4.x, x4.y);
              *reinterpret_cast<uint2*>(c2 + dig * g.d2 + 16) = make_uint2(x4.z, x4.w);
            }
          }
          if (one) {   // the other half circle's columns trade places past Nb / 2
            const uint4 y4 = !rot     ? x4
                             : H == 4 ? make_uint4(x4.z, x4.w, x4.x, x4.y)
                                      : make_uint4(x4.y, x4.x, x4.w, x4.z);
            *reinterpret_cast<uint4*>(c1 + dig * g.d1) = y4;
            if (ring) *reinterpret_cast<uint4*>(c1 + dig * g.d1 + Nb * XW / 8 * g.sb1) = y4;
          }
        }
      }
    };
    // One scale for a block (plane: for the tile) while its values lie within kNear places;
    // the lines of a point then differ by no more. Else (wide) every line has its own: copy 1
    // is cut relative to the largest value of each a-circle (a line and its partner's), copy 2
    // to that of each b-line. Blocks that need it not keep their one scale also beside one
    // that does, and whether the tile before was wide only decides which way is tried first
    // (guess): what a block gives depends on its own values alone. With one scale always, a
    // step of 33 x 16^4 x 4 takes 1467 us (now 1510), its conservative form, whose sin Theta
    // makes most tiles wide, 1589 (1865), the shell run of 129 x 16^2 x 24 x 16 2935 (3189)
    if (!guess) {
      uint32_t em[XW];
#pragma unroll
      for (int x = 0; x < XW; ++x)
        em[x] = fixed_key(smax[buf * 8 + (PASS == EP_PLANE ? 0 : x)]);
      bool far = false;
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (ua[q] < 0) continue;
        if constexpr (XW == 8) {
          uint64_t f[8];
#pragma unroll
          for (int x = 0; x < 8; ++x) f[x] = to_fixed(v[q][x], em[x], far);
          put(f, q, true, true);
        } else {
#pragma unroll
          for (int x = 0; x < 8; ++x) f4[q][x] = to_fixed(v[q][x], em[x & 3], far);
          put(f4[q], q, !g.seq, true);
        }
      }
      if (far) wflag[buf] = 1;
      fence_digits();
    }
    const bool wide = guess || wflag[buf] != 0;
    if (wide) {
      // the values again: kept, they would take registers from the common way
      if (!guess) load_units<PASS, U, XW>(d, A.U, at, S, hP, Nb, A.vec, ua, ub, v);
      int* mx1 = reinterpret_cast<int*>(sm + g.oEx);   // maxima [x][hb], [a][x], in the exchange
      int* mx2 = mx1 + hb * XW;
      for (int z = tid; z < (hb + Na) * XW; z += T) mx1[z] = 0;
      if (tid == 0) *wmask = 0;   // the blocks that are wide
      __syncthreads();
      uint32_t mine = 0;
#pragma unroll
      for (int q = 0; q < U; ++q) {
        uint32_t mag[8];
#pragma unroll
        for (int x = 0; x < 8; ++x)
          mag[x] = ua[q] < 0 ? 0u : (uint32_t)__double2hiint(v[q][x]) & 0x7FFFFFFFu;
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          const uint32_t mx = smax[buf * 8 + (PASS == EP_PLANE ? 0 : x & (XW - 1))];
          if (far_below(mag[x], fixed_key(mx)) || tiny_line(mx) || mx >= 0x7FF00000u)
            mine |= PASS == EP_PLANE ? 0xFFu : 1u << (x & (XW - 1));
          const int xx = x & (XW - 1), b = ub[q] + x / XW, c = b < hb ? b : b - hb;
          if (ua[q] >= 0)
            atomicMax(&mx1[(PASS == EP_PLANE && b >= hb ? xx ^ (XW / 2) : xx) * hb + c], (int)mag[x]);
        }
        if (XW == 8 && Nb % 8 == 0) {   // eight lanes hold one b-line: one value each
          const int l = lane & 7;
#pragma unroll
          for (int h = 4; h > 0; h /= 2) {
#pragma unroll
            for (int x = 0; x < h; ++x) {
              const bool hi = l & h;
              const uint32_t send = hi ? mag[x] : mag[x + h], keep = hi ? mag[x + h] : mag[x];
              mag[x] = max(keep, __shfl_xor_sync(0xFFFFFFFFu, send, h));
            }
          }
          if (ua[q] >= 0) atomicMax(&mx2[ua[q] * XW + l], (int)mag[0]);
        } else if (ua[q] >= 0) {
#pragma unroll
          for (int x = 0; x < 8; ++x) atomicMax(&mx2[ua[q] * XW + (x & (XW - 1))], (int)mag[x]);
        }
      }
      mine = __reduce_or_sync(0xFFFFFFFFu, mine);
      if (lane == 0 && mine) atomicOr(const_cast<uint32_t*>(wmask), mine);
      __syncthreads();
      const uint32_t mask = *wmask & 0xFFu;
      bool low = false;
      for (int z = tid; z < (hb + Na) * XW; z += T) {
        const int y = z - hb * XW, x = y < 0 ? z / hb : y & (XW - 1), c = z - x * hb;
        const bool own = mask >> x & 1u;
        const uint32_t mx = own ? (uint32_t)mx1[z] : smax[buf * 8 + (PASS == EP_PLANE ? 0 : x)];
        low |= own && tiny_line(mx);
        ln1[y < 0 ? c * XW + x : z] = (int16_t)(own ? line_base(mx) : block_exp(mx));
      }
      const bool lift = __syncthreads_or(low ? 1 : 0);
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (ua[q] < 0) continue;
        auto bases = [&](const int16_t* p) {   // of one unit: XW lines of a row
          return XW == 8 ? *reinterpret_cast<const uint4*>(p)
                         : make_uint4(reinterpret_cast<const uint2*>(p)->x,
                                      reinterpret_cast<const uint2*>(p)->y, 0u, 0u);
        };
        uint4 e = bases(ln2 + ua[q] * XW);
        if (XW == 4) e.z = e.x, e.w = e.y;
        uint64_t f[8];
        to_fixed_lines(v[q], e, lift, f);
        put(f, q, false, true);
        const bool part = ub[q] >= hb;
        const int16_t* p1 = ln1 + (part ? ub[q] - hb : ub[q]) * XW;
        e = bases(p1);
        if (XW == 4) {
          const uint4 e2 = bases(p1 + XW);
          e.z = e2.x, e.w = e2.y;
        }
        if (PASS == EP_PLANE && part)   // the other half circle's columns trade places
          e = XW == 8 ? make_uint4(e.z, e.w, e.x, e.y) : make_uint4(e.y, e.x, e.w, e.z);
        if constexpr (XW == 8) {
          to_fixed_lines(v[q], e, lift, f);
          put(f, q, true, false);
        } else {
          to_fixed_lines(v[q], e, lift, f4[q]);
          if (!g.seq) put(f4[q], q, true, false);
        }
      }
      fence_digits();
      guess = mask != 0;
    }
    // issues job n (one call site: the unrolled chains are inlined there, their
    // operands in uniform registers)
    auto issue = [&](int n) {
      const uint32_t r = g.dual ? (uint32_t)(n & 1) : 0u;
      const uint32_t one = elect_one(), tm = tmem + r * (uint32_t)g.half, ca = smb + g.oCA;
      if (n < g.mt2) {
        const uint32_t a = smb + g.oC2 + (uint32_t)(16 * n * g.sb2), b = smb + g.oB2;
        if ((NB_ ? NB_ <= 16 : g.kc2 == 2) && g.n2 <= 32)
          chain_steps<1, false, false>(one, tm, ca, a, g.d2, g.sb2, 0, b, 0, g.r2, g.n2);
        else if (!NB_ && g.kc2 == 4 && g.n2 <= 32)
          chain_steps<2, false, false>(one, tm, ca, a, g.d2, g.sb2, 0, b, 0, g.r2, g.n2);
        else
          chain_any(one, tm, ca, a, g.d2, g.sb2, g.kc2 / 2, 0, false, b, 0, g.r2, g.n2);
      } else {
        const uint32_t a = smb + g.oC1 + (uint32_t)(16 * (n - g.mt2) * g.sb1), b = smb + g.oB1;
        const uint32_t part = (uint32_t)(hb * XW / 8 * g.sb1);
        const int ka = NA_ ? (NA_ + 7) / 8 : g.n1 <= 32 ? g.ka : 0;
        if (ka == 1)
          chain_steps<0, true, true>(one, tm, ca, a, g.d1, g.sb1, part, b, 0, g.r1, g.n1);
        else if (ka == 2)
          chain_steps<1, true, false>(one, tm, ca, a, g.d1, g.sb1, part, b, 0, g.r1, g.n1);
        else if (ka == 3)
          chain_steps<1, true, true>(one, tm, ca, a, g.d1, g.sb1, part, b, 0, g.r1, g.n1);
        else if (ka == 4)
          chain_steps<2, true, false>(one, tm, ca, a, g.d1, g.sb1, part, b, 0, g.r1, g.n1);
        else
          chain_any(one, tm, ca, a, g.d1, g.sb1, g.ka / 2, part, g.ka & 1, b, 0, g.r1, g.n1);
      }
      mma_commit(one, sm_u32(&bar[r]));
      __syncwarp();
    };
    const TileAt<PASS> cur = at;
    int issued = 0;
    const int early = XW == 4 && g.seq ? g.mt2 : 0;   // jobs waited for ahead of their epilogue
    // waits for job n, every warp for itself; where a wait runs out the warp goes on (its
    // results are void) and all leave together: the job's barrier takes the vote (a flag in
    // shared memory could be set by the next job's waits before the last thread reads it)
    auto wait_job = [&](int n) {
      const uint32_t r = g.dual ? (uint32_t)(n & 1) : 0u;
      late |= !bar_wait(sm_u32(&bar[r]), (phase >> r) & 1u, p.wait_operand);
      phase ^= 1u << r;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto end_job = [&](int n) {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      const bool over = __syncthreads_or(late ? 1 : 0);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (over) {
        if (tid == 0 && p.err) atomicExch(p.err, 1);
        // our own MMAs end before the CTA exits (full bound)
        for (int x = n; x < issued; ++x) {
          const uint32_t rr = g.dual ? (uint32_t)(x & 1) : 0u;
          const bool passed = x == n || x < early;   // this thread has gone past that phase
          bar_wait(sm_u32(&bar[rr]), ((phase >> rr) & 1u) ^ (passed ? 1u : 0u), kDefaultWaitIters);
        }
        return false;
      }
      return true;
    };
    auto lanes = [&](int n) {   // this warp's tensor-memory address in job n's region
      const uint32_t r = g.dual ? (uint32_t)(n & 1) : 0u;
      return tmem + r * (uint32_t)g.half + ((uint32_t)((warp & 3) * 32) << 16);
    };
    const int eb = block_exp(smax[buf * 8 + (PASS == EP_PLANE ? 0 : rx)]);
    const double* xc = xs + buf * 64;   // the scalars of this tile
    for (int n = 0; n < jobs; ++n) {
      double gks = 0.0;   // adjoint: this thread's share of sum lt Us
      if constexpr (XW == 8) {
        for (const int upto = min(n + ahead, jobs); issued < upto; ++issued)
          if (uwarp == T / 32 - 1) issue(issued);
      } else {
#pragma unroll 1
        for (int part = n < early ? n : 1; part < 2; ++part) {
          for (const int upto = part ? min(n + ahead, jobs) : early; issued < upto; ++issued)
            if (uwarp == T / 32 - 1) issue(issued);
          if (part == 0) {   // copy 1 takes copy 2's place when the Fourier products are done
            for (int z = 0; z < early; ++z) wait_job(z);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();
#pragma unroll
            for (int q = 0; q < U; ++q)
              if (ua[q] >= 0) put(f4[q], q, true, false);
            fence_digits();
          }
        }
      }
      if (n == 0) {
        // the next tile's values travel while this one is finished
        if (tile + gridDim.x < A.ntiles) {
          at = tile_at<PASS, XW>(d, tile + gridDim.x);
          load_units<PASS, U, XW>(d, A.U, at, S, hP, Nb, A.vec, ua, ub, v);
          if (PASS != EP_PLANE && warp == 1 && lane < XW) scalars_load(lane, buf ^ 1);
        }
      }
      if (n < g.mt2) {
      // ---- Fourier results: rows (a, x), times the coefficient of their term
      const int a = RT * n + rg;
      const bool val = a < Na;
      // the row's coefficient: sinTh cot th (angular), sinPh / sin th (plane). The
      // CTA's next tile mostly has the same th or Phi columns: kept while it does
      const double key = PASS != EP_PLANE ? xc[16 + rx] : (double)cur.m0;
      if (n != coef_n || key != coef_key) {
        coef_n = n;
        coef_key = key;
        coef = 0;
        if (val) {
          if (PASS != EP_PLANE) {
            coef = __double2ll_rn(t.sinT[a] * key * pow2(64 + delta - cot_shift(key, delta)));
          } else {
            const bool ok = cur.m0 + (rx & (XH - 1)) < hP;
            const double sp = ok ? t.sinP[cur.m0 + (rx & (XH - 1)) + (rx >= XH ? hP : 0)] : 0.0;
            coef = __double2ll_rn(sp * t.inv_sinth[a] * pow2(64 + delta - hs[a]));
          }
        }
      }
      if (n >= early) wait_job(n);
      const uint32_t tl = lanes(n);
      const int nreal = Nb + (PASS != EP_PLANE && A.collision ? g.nf - g.nz : 0);
      int64_t* exr = ex + a * XW + rx;
      for (int q = grp; 4 * q < nreal; q += NG) {
        uint32_t bb[8][4];
        tm_ld(tl + (uint32_t)(4 * q), g.n2, bb);
        tm_wait(bb);
        int64_t R[4];
        recombine4(bb, R);
        // functionals: outputs 0 and Nb/2 (whose derivative rows vanish, nz of them) and
        // those from Nb on
        const bool special = PASS != EP_PLANE &&
                             ((g.nz > 0 && q == 0) || (g.nz > 1 && q == hb / 4) || 4 * q + 4 > Nb);
        if (!special) {
          if (val) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (4 * q + e < Nb) exr[(4 * q + e) * exP] = __mul64hi(R[e], coef);
          }
          continue;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int o = 4 * q + e;
          if (o >= nreal) break;
          const bool zero = g.nz > 0 && (o == 0 || (g.nz > 1 && o == hb));
          if (o < Nb && val) exr[o * exP] = zero ? 0 : __mul64hi(R[e], coef);
          const int f = o >= Nb ? o - Nb + g.nz : !zero ? -1 : o == 0 ? 0 : 1;
          if (f < 0 || !A.collision) continue;
          // Phi sums of F times {1, cos, sin, cos^2, cos sin}: their weighted Theta sums are
          // the scattering moments. In double: as fixed point a block's small moment beside
          // a large value (a beam) lost bits that the sum of doubles keeps
          const int e2 = wide && val ? ln2[a * XW + rx] : eb;
          const double y = val ? to_double1(R[e], e2 + m2.se) : 0.0;
          const int av = val ? a : 0;
          const double* wa = wt + av;
          double* s0 = msum + (warp & 3) * nm * 8 + rx;
          if (f == 0) {
            moment<XW>(s0, y * wa[0], n > 0);
            if (KF >= KF_LINEAR) moment<XW>(s0 + 8, y * wa[Na], n > 0);
            if (KF >= KF_QUADRATIC) moment<XW>(s0 + 32, y * wa[Na] * t.cosT[av], n > 0);
          } else {
            const double ys = y * wa[2 * Na];
            if (f < 3) {
              moment<XW>(s0 + 8 * (1 + f), ys, n > 0);
              if (KF >= KF_QUADRATIC) moment<XW>(s0 + 8 * (6 + f), ys * t.cosT[av], n > 0);
            } else {
              moment<XW>(s0 + 8 * (2 + f), ys * t.sinT[av], n > 0);
            }
          }
        }
      }
      } else {
      // ---- DFS results: rows (b, x); every point is finished here
      const int b = RT * (n - g.mt2) + rg;
      const int w = PASS == EP_PLANE && b >= hb ? rx ^ XH : rx;
      bool val = b < Nb;
      long long po = 0;   // adjoint: this column's offset in the fields
      double* Kp;
      const double* Ip;   // what the epilogue reads per point: U (angular) or K (plane)
      unsigned st;        // stride of a (a plane spans less than 2^32 elements)
      if (PASS != EP_PLANE) {
        val = val && cur.b0 + rx < d.nblk;
        const long long o = (cur.b0 + rx) * S + b;
        Kp = A.K + o;
        Ip = A.U + o;
        st = Nb;
        po = o;
      } else {
        val = val && cur.m0 + (w & (XH - 1)) < hP;
        Kp = A.K + cur.base + (long long)b * d.S_l + cur.m0 + (w & (XH - 1)) + (w >= XH ? hP : 0);
        Ip = Kp;
        st = (unsigned)d.S_j;
      }
      const bool rd = val && (PASS == EP_PLANE || A.collision);
      double in[2][4];
      auto load_in = [&](int q) {   // quads q and q + NG
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int a = 4 * (q + h * NG) + e;
            in[h][e] = rd && a < Na ? Ip[(unsigned)a * st] : 0.0;
          }
      };
      load_in(grp);
      wait_job(n);
      const uint32_t tl = lanes(n);
      double c0, kks = 0.0, src = 0.0, hr = 0.0, hc = 0.0, mrr = 0.0, qmc = 0.0, rmc = 0.0;
      int hx = 0;
      if (PASS == EP_PLANE) {
        c0 = A.sgn * t.sinT[cur.k] * t.inv_r[cur.i];
        if (cth_b != b * 64 + cur.m0) {   // cosPh as a fixed-point coefficient of the DFS term
          cth_b = b * 64 + cur.m0;
          cth = val ? __double2ll_rn(t.cosP[cur.m0 + (w & (XH - 1)) + (w >= XH ? hP : 0)] * pow2(62)) : 0;
        }
      } else {
        c0 = -A.sgn * xc[w];
        hx = cot_shift(xc[16 + w], delta);
        if (A.collision) {
          const double ks = xc[32 + w], J = xm[w];
          kks = xc[8 + w] + ks;
          src = PASS == EP_ADJOINT ? ks * J : fma(ks, J, A.cons ? xm[72 + w] : xc[24 + w]);
          if (KF >= KF_LINEAR) {
            const double cp = t.cosP[val ? b : 0], sp = t.sinP[val ? b : 0];
            const double kb = p.scb ? ks * xc[40 + w] : 0.0;
            hr = kb * xm[8 + w];
            hc = kb * (cp * xm[16 + w] + sp * xm[24 + w]);
            if (KF >= KF_QUADRATIC) {
              // M_phph = J - M_rr - M_thth (the trace of omega omega is 1)
              const double kc = ks * xc[48 + w], j3 = J * (1.0 / 3.0);
              const double rr = xm[32 + w], tt = xm[40 + w];
              mrr = kc * (rr - j3);
              qmc = kc * (cp * cp * (tt - j3) + sp * sp * (J - rr - tt - j3) +
                          2.0 * cp * sp * xm[48 + w]);
              rmc = 2.0 * kc * (cp * xm[56 + w] + sp * xm[64 + w]);
            }
          }
        }
      }
      const int qv = eb + m1.se;
      const int e1 = wide ? ln1[(!val ? 0 : b < hb ? b : b - hb) * XW + rx] : 0;
      uint32_t lim = slow_limit(qv);
      const int64_t* exr = ex + (val ? b : 0) * exP + w;
      // own: wide, in a loop of its own (a branch inside slows the common one by 2 %; the
      // adjoint's loop is too long to have twice)
      auto finish = [&](auto lines) {
      const bool own = PASS == EP_ADJOINT ? wide : decltype(lines)::value;
      for (int q0 = grp; 4 * q0 < Na; q0 += 2 * NG) {
        if (q0 != grp) load_in(q0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = q0 + h * NG;
          if (4 * q >= Na) break;
          uint32_t bb[8][4];
          tm_ld(tl + (uint32_t)(4 * q), g.n1, bb);
          tm_wait(bb);
          int64_t W[4];
          int qb[4];
          recombine4(bb, W);
          if (!own) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int a = min(4 * q + e, Na - 1);
              const int ha = PASS != EP_PLANE ? hx : hs[a];
              if (PASS != EP_PLANE) W[e] >>= hx;
              else W[e] = __mul64hi(W[e], cth) >> (ha - 2);
              W[e] += exr[a * XW];
              qb[e] = qv + ha;
            }
          } else {   // the unit of the larger term, 2^top, with a place (plane: two) to spare
            lim = 1u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int a = min(4 * q + e, Na - 1);
              const int ha = PASS != EP_PLANE ? hx : hs[a], sp = PASS != EP_PLANE ? 1 : 2;
              const int e2 = ln2[a * XW + w] + ha, top = max(e1 + sp, e2);
              if (PASS != EP_PLANE) W[e] = sra(W[e], top - e1);
              else W[e] = sra(__mul64hi(W[e], cth), top - e1 - 2);
              W[e] += sra(exr[a * XW], top - e2);
              qb[e] = top + m1.se;
              lim = max(lim, slow_limit(qb[e]));
            }
          }
          double y4[4];
          to_double4(W, qb, lim, y4);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int a = 4 * q + e;
            if (a >= Na) break;
            double r2;
            if (PASS == EP_PLANE) {
              r2 = fma(c0, y4[e], in[h][e]);
            } else {
              double col = 0.0;
              if (A.collision) {
                double gain = src;
                if (KF >= KF_LINEAR) {
                  const double ct = t.cosT[a], sT = t.sinT[a];
                  double u1 = hr, u2 = hc;
                  if (KF >= KF_QUADRATIC) {
                    u1 = fma(ct, mrr, fma(sT, rmc, hr));
                    u2 = fma(sT, qmc, hc);
                  }
                  gain = fma(ct, u1, fma(sT, u2, gain));
                }
                if (A.cons) gain *= t.sinT[a];
                if (PASS == EP_ADJOINT) {
                  if (val) {
                    const long long gi = po + (unsigned)a * st;
                    gks = fma(in[h][e], A.Us[gi], gks);
                    const double ub = fma(c0, y4[e], fma(t.qdir[a], gain,
                                                         fma(-kks, in[h][e], A.K[gi])));
                    const double l0 = A.lam_in[gi];
                    if (A.Kbar) A.Kbar[gi] = fma(A.wl, A.lam[gi], A.wu * ub);
                    A.lam_out[gi] = l0 + ub;
                  }
                  continue;
                }
                col = fma(-kks, in[h][e], gain);
              }
              r2 = fma(c0, y4[e], col);
            }
            if (val) Kp[(unsigned)a * st] = r2;
          }
        }
      }
      };
      if (PASS != EP_ADJOINT && wide) finish(std::true_type{});
      else finish(std::false_type{});
      }
      if (PASS == EP_ADJOINT && n >= g.mt2) {
        if (XW == 4) gks += __shfl_xor_sync(0xFFFFFFFFu, gks, 4);
        gks += __shfl_xor_sync(0xFFFFFFFFu, gks, 8);
        gks += __shfl_xor_sync(0xFFFFFFFFu, gks, 16);
        if (lane < XW) gp[((n - g.mt2) * (T / 32) + warp) * 8 + lane] = gks;
      }
      alive = end_job(n);
      if (!alive) break;
      if (PASS == EP_ADJOINT && n == jobs - 1 && tid < XW && cur.b0 + tid < d.nblk) {
        double gt = 0.0;   // the warps' shares in a fixed order
        for (int z = 0; z < g.mt1 * (T / 32); ++z) gt += gp[z * 8 + tid];
        A.gk[cur.b0 + tid] -= gt;
        A.ge[cur.b0 + tid] += xm[tid];
      }
      if (PASS != EP_PLANE && n == g.mt2 - 1 && A.collision) {
        if (tid < 80) {
      // moment z of block x from the four warps' shares (visible after the next barrier)
      const int z = tid >> 3, x = tid & 7;
      if (x >= XW) {
      } else if (z < nm) {
        const double* m = msum + tid;
        xm[tid] = (m[0] + m[nm * 8]) + (m[2 * nm * 8] + m[3 * nm * 8]);
      } else if (z == 9 && A.cons) {   // eta r^2 sin th
        xm[tid] = xc[24 + x] * xc[56 + x] / (xc[x] * xc[x]);
      }
    }
        __syncthreads();
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 :: "r"(tmem), "r"(g.cols) : "memory");
  }
}

// ============================================================================
// Radial pass: 128 (Theta, Phi) columns of one (g, theta, phi) per tile, all N_r
// nodes. Digits [digit][column / 8][node][8 columns], MN-major; the matrix rows
// are ordered 0, N, 1, 2, ..., N-1 so that the two Tau rows come first. Every line is cut
// relative to its own largest magnitude (a column is a row of the product, so the scale
// joins in the epilogue): lines of one tile do not meet in this pass, and a faint direction
// beside a beam keeps its digits. One scale for the tile was no faster (33 x 16^4 x 4: 1471
// us a step with it, 1472 without).
struct RadArgs {
  const double *U, *Kin;
  double sgn;
  int tau, mode;
  double *F, *Acc, *Uout, *out;
  double dt;   // adjoint: the scale of X
  long long ntiles;
};
constexpr int RAD_ADJOINT = 100;   // MODE of the transposed pass: U = X, Acc = lt, out = Ubar

struct RadMats {
  const uint16_t* dev[8];
  const int* se[8];
};

__device__ __forceinline__ void prefetch_line(const double* p) {
  asm volatile("prefetch.global.L2 [%0];" :: "l"(p));
}

__device__ __forceinline__ int rad_row(int o, int N) { return o == 0 ? 0 : o == 1 ? N : o - 1; }

template <int T, int MODE>
__global__ void __launch_bounds__(T, T == 256 ? 2 : 1)
k_emu_radial(Problem p, Tables<double> t, EmuRadGeo g, RadMats M, RadArgs A) {
  extern __shared__ __align__(128) unsigned char sm[];
  const Dims& d = p.d;
  const uint32_t smb = sm_u32(sm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int uwarp = __shfl_sync(0xFFFFFFFFu, warp, 0);   // warp-uniform
  constexpr int NG = T / 128;
  const int Nr = g.Nr, N = Nr - 1, NP = d.NP, S = d.NT * d.NP;
  unsigned char* ms = sm + g.oMs;
  uint64_t* bar = reinterpret_cast<uint64_t*>(ms);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(ms + 16);
  volatile uint32_t* tiny = reinterpret_cast<volatile uint32_t*>(ms + 24);   // [2] a line is
  uint64_t* barB = reinterpret_cast<uint64_t*>(ms + 32);   // [2]: a streamed matrix has arrived
  volatile unsigned* cnt = reinterpret_cast<volatile unsigned*>(ms + 48);  // [3], issuing warp's
  int* se = reinterpret_cast<int*>(ms + 64);               // [ng * n]
  double* tot = reinterpret_cast<double*>(ms + 64 + (g.ng * g.n * 4 + 15) / 16 * 16);   // [128]
  uint32_t* ckey = reinterpret_cast<uint32_t*>(tot + 128);   // [2][128] keys of the lines
  double* ts = reinterpret_cast<double*>(sm + g.oA);       // adjoint: [warps][128], before the digits
  if (!g.left || Nr != 8 * g.kc + 1) {   // K paddings read as zero
    for (int x = tid; x < g.oB / 16; x += T)
      reinterpret_cast<uint4*>(sm)[x] = make_uint4(0, 0, 0, 0);
  }
  if (tid < 256) ckey[tid] = 0;
  if (tid < 2) tiny[tid] = 0;
  if (tid < 3) cnt[tid] = 0;
  for (int q = 0; q < g.ng; ++q) {
    if (q < g.nb && g.nb == g.ng) copy_in(sm + g.oB + q * g.bB, M.dev[q], g.bB);
    for (int x = tid; x < g.n; x += T) se[q * g.n + x] = M.se[q][x];
  }
  fill_bias(sm + g.oCA, 128);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_u32(&bar[0])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_u32(&bar[1])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_u32(&barB[0])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_u32(&barB[1])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(sm_u32(tslot)), "r"(g.cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    pass_started();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tslot, 0);
  const int nch = (S + 127) / 128;
  const int row = (warp & 3) * 32 + lane, grp = warp >> 2;
  const int ahead = g.dual ? 2 : 1;
  // MODE: the update; RAD_STAGE1 stands for stages 1 and 2 (A.mode tells them apart)
  constexpr bool rA = MODE == RAD_STAGE1 || MODE == RAD_STAGE3 || MODE == RAD_AB2;
  uint32_t phase = 0;
  bool alive = true, late = false;   // late: a wait of this thread ran out
  int buf = 0;
  constexpr int U = kEmuRadUnits;   // (node, 8 columns) units held per thread: all of them
  auto coords = [&](long long tile, int& c0, long long& base) {
    unsigned q0 = (unsigned)tile;   // tiles of a field fit 32 bits (checked on the host)
    c0 = (int)(q0 % (unsigned)nch) * 128;
    q0 /= (unsigned)nch;
    const int l = (int)(q0 % (unsigned)d.Np);
    q0 /= (unsigned)d.Np;
    const int j = (int)(q0 % (unsigned)d.Nt);
    base = (long long)(q0 / (unsigned)d.Nt) * d.S_g + (long long)j * d.S_j +
           (long long)l * d.S_l + c0;
  };
  // Where the matrices do not fit beside the digits they stream through two buffers, in
  // the order of the groups (T = 512): matrix number z of this CTA goes to buffer z & 1 when the
  // products of number z - 2 are done. cnt: matrices requested and waited for, the next
  // one's group (in shared memory: the epilogue needs every register)
  const bool stream = T == 512 && g.nb != g.ng;
  auto load_next = [&]() {
    const unsigned z = cnt[0], q = cnt[2];
    // the groups of all tiles of this CTA (below 2^31, host)
    if (z < (unsigned)((A.ntiles - 1 - (long long)blockIdx.x) / gridDim.x + 1) * g.ng) {
      __syncwarp();
      if (elect_one()) {
        const uint32_t br = sm_u32(&barB[z & 1]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     :: "r"(br), "r"(g.bB) : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
            :: "r"(smb + g.oB + (z & 1) * g.bB), "l"(M.dev[q]), "r"(g.bB), "r"(br)
            : "memory");
        cnt[0] = z + 1;
        cnt[2] = q + 1 == (unsigned)g.ng ? 0 : q + 1;
      }
      __syncwarp();
    }
  };
  if (stream && uwarp == T / 32 - 1) {
    load_next();
    load_next();
  }
  pass_wait();
  for (long long tile = blockIdx.x; tile < A.ntiles && alive; tile += gridDim.x, buf ^= 1) {
    int c0;
    long long base;
    coords(tile, c0, base);
    const int Wc = min(128, S - c0);
    // the lines the epilogue reads are requested into L2 meanwhile (one 128-byte line
    // per request)
    for (int u = tid; u < Nr * 8; u += T) {
      const int w = (u & 7) * 16;
      if (w < Wc) {
        const long long gi = base + (long long)(u >> 3) * d.S_i + w;
        if (MODE != RAD_ADJOINT) prefetch_line(A.Kin + gi);
        if (MODE != RAD_RHS && MODE != RAD_ADJOINT) prefetch_line(A.F + gi);
        if (rA) prefetch_line(A.Acc + gi);
      }
    }
    // the tile's values, and the largest magnitude of every line: all units of a thread hold
    // the same eight lines
    double v[U][8];
    uint32_t mx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    auto load_unit = [&](int u, double (&z)[8]) {
      const int w = (u & 15) * 8;
#pragma unroll
      for (int x = 0; x < 8; ++x) z[x] = 0.0;
      if (u < Nr * 16) {
        const double* src = A.U + base + (long long)(u >> 4) * d.S_i + w;
        if (w + 8 <= Wc) {
#pragma unroll
          for (int x = 0; x < 8; x += 2) {
            const double2 y = *reinterpret_cast<const double2*>(src + x);
            z[x] = y.x;
            z[x + 1] = y.y;
          }
        } else {
#pragma unroll
          for (int x = 0; x < 8; ++x)
            if (w + x < Wc) z[x] = src[x];
        }
      }
    };
#pragma unroll
    for (int q = 0; q < U; ++q) load_unit(tid + q * T, v[q]);
    if (MODE == RAD_ADJOINT) {
      // lt = Tau^T (scale X): every row but the inflow one as it is, that one less
      // T_N(x_b) sum_i T_N(x_i) X_i: a thread's share of its eight columns' sums, then the
      // half warps', then the CTA's, in fixed order
#pragma unroll
      for (int q = 0; q < U; ++q)
#pragma unroll
        for (int x = 0; x < 8; ++x) v[q][x] *= A.dt;
      if (A.tau) {
        double sum[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          sum[x] = 0.0;
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const int i = (tid + q * T) >> 4;
            if (i < Nr) sum[x] += (N - i) & 1 ? -v[q][x] : v[q][x];
          }
          sum[x] += __shfl_xor_sync(0xFFFFFFFFu, sum[x], 16);
          if (lane < 16) ts[(warp * 16 + lane) * 8 + x] = sum[x];
        }
        __syncthreads();
        if (tid < 128) {
          double z = 0.0;
          for (int w = 0; w < T / 32; ++w) z += ts[w * 128 + tid];
          tot[tid] = z;
        }
        __syncthreads();
        if (!g.left || Nr != 8 * g.kc + 1) {   // the K paddings under the sums are zero again
          for (int x = tid; x < T * 2; x += T)
            reinterpret_cast<uint4*>(ts)[x] = make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
          const int i = (tid + q * T) >> 4, w = (tid & 15) * 8;
          if (i != 0 && i != N) continue;
#pragma unroll
          for (int x = 0; x < 8; ++x)
            if (w + x < Wc && i == (t.cosT[(c0 + w + x) / NP] > 0.0 ? 0 : N))
              v[q][x] -= (N - i) & 1 ? -tot[w + x] : tot[w + x];
        }
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const int u = tid + q * T, w = (u & 15) * 8;
        if (u >= Nr * 16) continue;
        double* dst = A.Acc + base + (long long)(u >> 4) * d.S_i + w;
        if (w + 8 <= Wc) {
#pragma unroll
          for (int x = 0; x < 8; x += 2)
            *reinterpret_cast<double2*>(dst + x) = make_double2(v[q][x], v[q][x + 1]);
        } else {
#pragma unroll
          for (int x = 0; x < 8; ++x)
            if (w + x < Wc) dst[x] = v[q][x];
        }
      }
    }
#pragma unroll
    for (int q = 0; q < U; ++q)
#pragma unroll
      for (int x = 0; x < 8; ++x)
        mx[x] = max(mx[x], (uint32_t)__double2hiint(v[q][x]) & 0x7FFFFFFFu);
    bool low = false;
#pragma unroll
    for (int x = 0; x < 4; ++x) {   // the half warps hold the same lines: four each
      const uint32_t send = lane & 16 ? mx[x] : mx[x + 4], keep = lane & 16 ? mx[x + 4] : mx[x];
      const uint32_t r = max(keep, __shfl_xor_sync(0xFFFFFFFFu, send, 16));
      low |= tiny_line(r);
      atomicMax(&ckey[buf * 128 + (lane & 15) * 8 + x + (lane & 16) / 4], line_key(r));
    }
    if (low) tiny[buf] = 1;   // (another node of the line may be larger)
    __syncthreads();
    if (tid < 128) ckey[(buf ^ 1) * 128 + tid] = 0;
    if (tid == 128) tiny[buf ^ 1] = 0;
    const uint32_t* keys = ckey + buf * 128 + (tid & 15) * 8;   // of this thread's lines
    const bool up = tiny[buf] != 0;
    auto lift = [&](double (&z)[8]) {   // brings the values of tiny lines up
#pragma unroll
      for (int x = 0; x < 8; ++x)
        if (!(keys[x] & 1u)) z[x] *= pow2(256);
    };
    if (up) {
      __syncthreads();
      if (tid < 128) {
        const uint32_t key = ckey[buf * 128 + tid];
        if (key != 0 && key < kLeastKey) ckey[buf * 128 + tid] = tiny_key(key);
      }
      __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int u = tid + q * T;
      if (u >= Nr * 16) continue;
      const int ii = u >> 4, wg = u & 15;
      if (up) lift(v[q]);
      uint64_t f[8];
#pragma unroll
      for (int x = 0; x < 8; x += 4) {
        const uint4 k = *reinterpret_cast<const uint4*>(keys + x);
        f[x] = to_fixed(v[q][x], max(k.x, kLeastKey));
        f[x + 1] = to_fixed(v[q][x + 1], max(k.y, kLeastKey));
        f[x + 2] = to_fixed(v[q][x + 2], max(k.z, kLeastKey));
        f[x + 3] = to_fixed(v[q][x + 3], max(k.w, kLeastKey));
      }
      if (g.left && ii == N) {
        // the leftover node: its eight digits beside the bias, one 16-byte row per column
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          const uint32_t lo = (uint32_t)f[x], hi = (uint32_t)(f[x] >> 32);
          *reinterpret_cast<uint4*>(sm + g.oCA + 2048 + (wg * 8 + x) * 16) =
              make_uint4(__byte_perm(hi, 0, 0x4243), __byte_perm(hi, 0, 0x4041),
                         __byte_perm(lo, 0, 0x4243), __byte_perm(lo, 0, 0x4041));
        }
        continue;
      }
      unsigned char* c = sm + g.oA + wg * g.sb + ii * 16;
#pragma unroll
      for (int w = 3; w >= 0; --w) {
        uint32_t pk[4];
        pack_pairs(f, w, pk);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<uint4*>(c + (7 - (2 * w + h)) * g.d) = digit_of(pk, h);
      }
    }
    // every thread of a column reads the inflow node's rate before the barrier: the
    // right-hand side writes over its own Kin, and one of them stores that node first
    const bool val = row < Wc;
    const int kT = val ? (c0 + row) / NP : 0;
    const double cT = t.cosT[kT], ck = A.sgn * cT;
    const int bn = cT > 0.0 ? 0 : N;   // inflow node
    const double* Kc = A.Kin + base + row;
    const unsigned Si = (unsigned)d.S_i;   // a group spans less than 2^32 elements (host)
    double kb = MODE != RAD_ADJOINT && val && A.tau ? Kc[(unsigned)bn * Si] : 0.0;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    auto issue = [&](int n) {
      const uint32_t r = g.dual ? (uint32_t)(n & 1) : 0u;
      const uint32_t one = elect_one(), tm = tmem + r * (uint32_t)g.half;
      const uint32_t ca = smb + g.oCA, a = smb + g.oA;
      uint32_t bq = (uint32_t)n;
      if (stream) {
        const unsigned z = __shfl_sync(0xFFFFFFFFu, cnt[1], 0);
        late |= !bar_wait(sm_u32(&barB[z & 1]), (z >> 1) & 1u, p.wait_operand);
        __syncwarp();
        if (one) cnt[1] = z + 1;
        bq = z & 1;
      }
      const uint32_t b = smb + g.oB + bq * (uint32_t)g.bB;
      if (g.kc == 4)
        chain_steps<2, false, false>(one, tm, ca, a, g.d, g.sb, 0, b, g.left, g.rows, g.n);
      else if (g.kc == 2)
        chain_steps<1, false, false>(one, tm, ca, a, g.d, g.sb, 0, b, g.left, g.rows, g.n);
      else if (g.kc == 6)
        chain_steps<3, false, false>(one, tm, ca, a, g.d, g.sb, 0, b, g.left, g.rows, g.n);
      else if (g.kc == 8)
        chain_steps<4, false, false>(one, tm, ca, a, g.d, g.sb, 0, b, g.left, g.rows, g.n);
      else
        chain_any(one, tm, ca, a, g.d, g.sb, g.kc / 2, 0, false, b, g.left, g.rows, g.n);
      mma_commit(one, sm_u32(&bar[r]));
      __syncwarp();
    };
    int issued = 0;
    const int eb = line_exp(ckey[buf * 128 + row]);
    const double* Fc = A.F + base + row;
    const double* Ac = A.Acc + base + row;
    double* dst = (MODE == RAD_RHS || MODE == RAD_ADJOINT ? A.out
                   : MODE == RAD_STAGE3 || MODE == RAD_AB2 || MODE == RAD_AB2_START ? A.F
                                                                                    : A.Uout) +
                  base + row;
    double* Aw = A.Acc + base + row;
    const double cu = MODE == RAD_STAGE3 ? A.dt / 6.0
                      : MODE == RAD_STAGE0 || (MODE == RAD_STAGE1 && A.mode == RAD_STAGE1)
                          ? 0.5 * A.dt
                          : A.dt;
    double nk[4], nf[4], na[4];
    unsigned noff[4];
    auto load_rows = [&](int n, int q, int no) {   // quad q of group n
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int o = 4 * q + e;
        noff[e] = (unsigned)(o < no ? rad_row(n * g.go + o, N) : 0) * Si;
        nk[e] = nf[e] = na[e] = 0.0;
        if (val && o < no) {
          if (MODE != RAD_ADJOINT) nk[e] = Kc[noff[e]];
          if (MODE != RAD_RHS && MODE != RAD_ADJOINT) nf[e] = Fc[noff[e]];
          if (rA) na[e] = Ac[noff[e]];
        }
      }
    };
    if (tile + gridDim.x < A.ntiles) {   // the next tile's lines, into L2
      int c1;
      long long b1;
      coords(tile + gridDim.x, c1, b1);
      for (int u = tid; u < Nr * 8; u += T)
        if (c1 + (u & 7) * 16 < S)
          prefetch_line(A.U + b1 + (long long)(u >> 3) * d.S_i + (u & 7) * 16);
    }
    for (int n = 0; n < g.ng; ++n) {
      for (const int upto = min(n + ahead, g.ng); issued < upto; ++issued)
        if (uwarp == T / 32 - 1) issue(issued);
      const uint32_t r = g.dual ? (uint32_t)(n & 1) : 0u;
      const int no = min(g.go, Nr - n * g.go);
      if (4 * grp < no) load_rows(n, grp, no);
      // where a wait runs out the warp goes on (its results are void) and all leave
      // together: the group's barrier takes the vote
      late |= !bar_wait(sm_u32(&bar[r]), (phase >> r) & 1u, p.wait_operand);
      phase ^= 1u << r;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (stream && uwarp == T / 32 - 1 && !__any_sync(0xFFFFFFFFu, late))
        load_next();   // this group's matrix is free
      const uint32_t tl = tmem + r * (uint32_t)g.half + ((uint32_t)((warp & 3) * 32) << 16);
      if (MODE != RAD_ADJOINT && n == 0 && A.tau) {   // the finished rate at the inflow node (both rows lead this group)
        uint32_t b[8][4];
        tm_ld(tl, g.n, b);
        tm_wait(b);
        const int qb[4] = {eb + se[0], eb + se[1], 0, 0};
        int64_t R[4];
        recombine4(b, R);
        double y4[4];
        to_double4(R, qb, max(slow_limit(qb[0]), slow_limit(qb[1])), y4);
        kb = fma(ck, bn == 0 ? y4[0] : y4[1], kb);
        if ((N - bn) & 1) kb = -kb;   // times T_N at the inflow node
      }
      for (int q = grp; 4 * q < no; q += NG) {
        uint32_t b[8][4];
        tm_ld(tl + (uint32_t)(4 * q), g.n, b);
        tm_wait(b);
        int qb[4];
        uint32_t lim = 1u;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          qb[e] = eb + se[n * g.n + 4 * q + e];
          lim = max(lim, slow_limit(qb[e]));
        }
        int64_t R[4];
        recombine4(b, R);
        // the next rows' values travel while these are finished
        double kv[4], f[4], ac[4];
        unsigned off[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          kv[e] = nk[e];
          f[e] = nf[e];
          ac[e] = na[e];
          off[e] = noff[e];
        }
        if (4 * (q + NG) < no) load_rows(n, q + NG, no);
        double y4[4];
        to_double4(R, qb, lim, y4);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int o = 4 * q + e;
          if (o >= no) break;
          const double y = y4[e];
          if (MODE == RAD_ADJOINT) {   // Ubar = -cosTh D_r^T lt
            if (val) dst[off[e]] = -cT * y;
            continue;
          }
          double v = fma(ck, y, kv[e]);
          if (A.tau) {   // K_i -= K_b T_N(x_b) T_N(x_i)
            const int flip = ((N - rad_row(n * g.go + o, N)) & 1) << 31;
            v -= __hiloint2double(__double2hiint(kb) ^ flip, __double2loint(kb));
          }
          if (!val) continue;
          if (MODE == RAD_RHS) {
            dst[off[e]] = v;
          } else if (MODE == RAD_STAGE3) {
            dst[off[e]] = fma(cu, ac[e] + v, f[e]);
          } else if (MODE == RAD_AB2) {
            dst[off[e]] = fma(cu, fma(1.5, v, -0.5 * ac[e]), f[e]);
            Aw[off[e]] = v;
          } else {
            dst[off[e]] = fma(cu, v, f[e]);
            Aw[off[e]] = MODE == RAD_STAGE1 ? fma(2.0, v, ac[e]) : v;
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      const bool over = __syncthreads_or(late ? 1 : 0);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (over) {
        if (tid == 0 && p.err) atomicExch(p.err, 1);
        for (int x = n; x < issued; ++x) {   // our own MMAs end first (full bound)
          const uint32_t rr = g.dual ? (uint32_t)(x & 1) : 0u;
          bar_wait(sm_u32(&bar[rr]), ((phase >> rr) & 1u) ^ (x == n ? 1u : 0u), kDefaultWaitIters);
        }
        // and the matrices in flight (the issuing warp's count; full bound)
        if (stream && uwarp == T / 32 - 1)
          for (unsigned z = cnt[0] < 2 ? 0 : cnt[0] - 2; z < cnt[0]; ++z)
            bar_wait(sm_u32(&barB[z & 1]), (uint32_t)(z >> 1) & 1u, kDefaultWaitIters);
        alive = false;
        break;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 :: "r"(tmem), "r"(g.cols) : "memory");
  }
}

}  // namespace emu
}  // namespace ts
