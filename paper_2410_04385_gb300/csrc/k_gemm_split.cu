// FP64 products on the FP16 tensor cores: exact splitting of both operands
// (in the manner of Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 2012),
// fused into one kernel.
//
// On GB300 a DFMA-based product runs at two multiply-adds per SM and clock;
// the tensor cores do ~3600 FP16 ones. An FP64 operand entry, scaled to its
// row, is a 64-bit integer of eight balanced base-256 digits, each exact in
// FP16; products of digits summed over 128 terms of K stay below 2^24, exact
// in an FP32 accumulator. Per chunk of 32 terms of K
//   1. both operand tiles (128 rows x 32, NT columns x 32) are copied to shared
//      memory as FP64, coalesced along whichever index is contiguous; the next
//      chunk's entries are loaded to registers before this chunk's digits are
//      formed and stored under its products (copied asynchronously under the
//      products, whose operand reads fill the shared memory's bandwidth, they
//      took 5000 clocks per chunk);
//   2. each k is scaled by 2^{-t_k} in the row operand and 2^{t_k} in the
//      column operand, t_k half the difference of the two operands' largest
//      exponents at that k. The product is unchanged, and the result does not
//      depend on a diagonal scaling between the factors (the gauge of a TT
//      bond), as an FP64 product does not;
//   3. row i (column j) is scaled by the power of two of its largest entry (the
//      next one up if chunks follow): V = a 2^(1084 - e_i), cut to an integer
//      |V| < 2^62, eight or nine bits more than a double's significand;
//   4. V = sum_p d_p 256^(7-p), d_p in [-128, 127], written as FP16 digits in
//      the K-major core-matrix layout;
//   5. one thread issues the 36 digit products with p + q <= 7: digit p of
//      the rows against digits 0..7-p of the columns, which lie next to each
//      other in shared memory, so one tcgen05.mma of up to 256 columns adds
//      several of them to levels p.. (level p + q in TMEM columns NT (p + q)).
// The chunks of a group of up to four share the scales e_i, f_j of the first
// (a later entry above its row's scale ends the group early), and add to the
// same level sums. At the end of a group
//   6. the 8 level sums of an output are exact integers; they are combined in
//      integer arithmetic to T = sum_l L_l 256^(7-l), rounded once to a double,
//      scaled by 2^(e_i + f_j) and added to the output tile in shared memory.
// Dropped digit products and truncation leave at most 2^-58.8 of S = 2^(e_i + f_j)
// per term (2^-62 rms). Against the rounding of an FP64 chain, 2^-53 sum |a||b|, that
// is small unless the sum is far below S: where a row's large entries meet zeros or
// small entries of the column (block-structured factors of a sum of tensors,
// alternately graded rows). So
//   7. an output keeps its digit sum only if sum |a||b| >= 2^-7.7 S is certain:
//      because the sum itself is that large, or one term has both its entries at
//      4.5 / 64 of their scales or more (one bit per entry, an AND of two 128-bit
//      masks per output). Any other output's group is summed again from the
//      operands in FP64 (fallback). Then a term's error is at most 3.5 2^-53 of
//      sum |a||b|, 0.4 2^-53 rms, and terms' errors are independent: no element is
//      worse than a chain's bound, whatever the operands' grading.
//      Outputs summed twice: none of Gaussian factors, 0.1% where entries are
//      products of two or three Gaussians.
// Rows and columns with a non-finite entry go the same way, so infinities and NaN
// come out where FP64 arithmetic puts them.
//
// Bound: ALU instructions of the conversion (about 45 per operand entry) and of the
// level combination (about 65 per output and group), behind barriers: one digit
// buffer, so conversion and tensor work take turns. ncu at 5760 x 90 x 1600 (NT = 48,
// 450 blocks, 202 us): ALU pipe 54% of active cycles, issue slots 49%, tensor pipe
// 14%, DRAM 5% (79 MB, each operand once); warps wait for barriers, shared memory and
// dependent instructions in equal parts. FP64 instructions appear only in the sums
// over groups, in alpha and in step 7. Step 7's test costs 3 to 5% (12 cores of modes
// 64, ranks 40 x 40, sketch 90: 24.2 -> 25.1 ms); operands that need the FP64 sums
// cost more: at 5760 x 90 x 1600 210 us for Gaussian ones, 520 for blocks 2^60 apart,
// 3450 where every entry has a size of its own (DFMA tiles: 1480 for all).
// 512 threads, one CTA per SM: with NT = 64 an entry of the row operand is converted
// once per 64 columns, which two CTAs of 32 columns each would do twice. Outputs
// are combined in a loop over four columns (1700 to 2400 clocks each: 64-bit
// integer multiply-adds, leading-zero counts and one FP64 add run at a quarter
// of the issue rate and less); unrolled over 16 the code is 100 KB and no faster.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <array>
#include <mutex>
#include <unordered_map>
#include "hatt_internal.cuh"

namespace hatt {

__device__ int g_split_error = 0;

namespace {

constexpr int kRows = 128;               // rows of a tile (tensor-core M, TMEM lanes)
constexpr int kKc = 32;                  // terms of K per chunk
constexpr int kGroup = 4;                // chunks that share scales and level sums
constexpr int kDig = 8;                  // digits per operand entry = levels kept
constexpr int kThreadsS = 512;           // converting threads; one more warp issues the products
constexpr int kThreadsAll = kThreadsS + 32;
constexpr int kLdRaw = kRows + 2;        // raw tiles are [k][row]; 4 k apart = 16 banks apart
constexpr int kABytes = kDig * kRows * kKc * 2;
constexpr int kNonfinite = 1 << 20;      // row / column exponent of a non-finite entry
constexpr int kEmpty = -(1 << 20);       // exponent of an all-zero row / column
constexpr int kSure = 5200;              // 2^20 2^-7.66: a sum this large is no cancelled one

// Shared memory of the NT-column form: digits of both operands, raw tiles,
// output tile (FP64). More than half an SM's, so one CTA per SM, whose
// tensor-memory allocation never waits for another of these kernels.
template <int NT>
struct SplitSmem {
  static constexpr int kBBytes = kDig * NT * kKc * 2;
  static constexpr int kLdC = NT + 2;              // columns of the raw tile
  static constexpr int kLdT = NT + 1;              // columns of the output tile
  static constexpr int kTmem = kDig * NT <= 256 ? 256 : 512;    // a power of two of columns
  static constexpr int kRaw = kABytes + kBBytes;
  static constexpr int kTile = kRaw + (kLdRaw + kLdC) * kKc * 8;
  static constexpr int kBytes = kTile + kRows * kLdT * 8;
};

// Barrier 1: the converting threads. Barrier 2: the digits of a chunk are
// ready (converting threads arrive, the issuing warp waits).
__device__ __forceinline__ void conv_sync() {
  asm volatile("bar.sync 1, %0;" :: "n"(kThreadsS) : "memory");
}
__device__ __forceinline__ bool conv_any(bool p) {
  uint32_t r;
  asm volatile("{\n.reg .pred a, b;\nsetp.ne.u32 a, %1, 0;\nbar.red.or.pred b, 1, %2, a;\n"
               "selp.u32 %0, 1, 0, b;\n}\n"
               : "=r"(r) : "r"((uint32_t)p), "n"(kThreadsS) : "memory");
  return r != 0;
}
__device__ __forceinline__ void digits_ready() {
  asm volatile("bar.arrive 2, %0;" :: "n"(kThreadsAll) : "memory");
}
__device__ __forceinline__ void wait_digits() {
  asm volatile("bar.sync 2, %0;" :: "n"(kThreadsAll) : "memory");
}

// One operand: entry (r, k) of batch (b1, b2) at
// p[b1 sb1 + b2 sb2 + (r / div) s_hi + (r % div) s_lo + k s_k], r < n.
struct SplitOperand {
  const double *p;
  long long sb1, sb2, s_hi, s_lo, s_k;
  int n, div;
};

struct SplitArgs {
  SplitOperand R, C;                     // the 128-row side and the NT-column side
  double *out;                           // batch strides, then the row's and the column's two levels
  long long ob1, ob2, or_hi, or_lo, oc_hi, oc_lo;
  int K, bdiv, tiles_r, tiles_c, ksplit, kchunk;
  double alpha;
  const double *alpha_dev;
  const int *skip_dev;
  double *partial;
  int *health;                           // where a wait that ran out is noted: the caller's word or null
  long long waits;                       // polls of one wait
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// K-major, no swizzle, core matrices of 8 rows x 16 bytes: LBO 128 bytes
// between core matrices along K, SBO between groups of 8 rows.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  constexpr uint32_t lbo = 128, sbo = (kKc / 8) * 128;
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) |
         ((uint64_t)(sbo >> 4) << 32) | ((uint64_t)1 << 46);
}

// The entries of an FP64 tile (rows [0, NR) and terms [k0, k0 + kKc) of an
// operand; rows past nr and terms past kend are zero) that this thread brings
// from global to shared memory: loaded early, stored [k][row] when the tile's
// last use is over. Lanes run along k if it is contiguous, else along rows.
// off[row]: element offset of the row.
template <int NR, int LD>
struct RawLoad {
  static constexpr int n = NR * kKc / kThreadsS;
  double x[n];

  __device__ __forceinline__ void load(const double *base, const long long *off, int nr, long long s_k,
                                       int k0, int kend) {
    if (s_k == 1) {
      const int k = threadIdx.x % kKc;
      const bool in_k = k0 + k < kend;
      const double *p = base + k0 + k;
#pragma unroll
      for (int j = 0; j < n; ++j) {
        const int row = threadIdx.x / kKc + kThreadsS / kKc * j;
        x[j] = (row < nr && in_k) ? p[off[row]] : 0.0;
      }
    } else {
#pragma unroll
      for (int j = 0; j < n; ++j) {
        const int e = threadIdx.x + kThreadsS * j;
        const int row = e % NR, k = e / NR;
        x[j] = (row < nr && k0 + k < kend) ? base[off[row] + (k0 + k) * s_k] : 0.0;
      }
    }
  }
  __device__ __forceinline__ void store(double *dst, long long s_k) const {
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const int e = threadIdx.x + kThreadsS * j;
      const int row = s_k == 1 ? threadIdx.x / kKc + kThreadsS / kKc * j : e % NR;
      const int k = s_k == 1 ? threadIdx.x % kKc : e / NR;
      dst[k * LD + row] = x[j];
    }
  }
};

// Largest high word of x[j] 2^(-sh[j]) without its sign, the shifts given in
// units of the exponent field (sh 2^20): INT_MIN if no entry has an exponent
// field. sub collects the words of those that have none (zeros, subnormals).
__device__ __forceinline__ int max_high(const double (&x)[4], const int (&sh)[4], int sgn, uint32_t &sub) {
  int e = INT_MIN;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t hi = (uint32_t)__double2hiint(x[j]) & 0x7FFFFFFFu;
    if (hi < 0x00100000u) sub |= hi | (uint32_t)__double2loint(x[j]);
    else e = max(e, (int)hi - sgn * sh[j]);
  }
  return e;
}

// The same as an exponent, for the chunks that hold a subnormal, an infinity or
// a NaN: kEmpty if all entries are zero, kNonfinite if one is not finite.
__device__ __noinline__ int max_expo(double x0, double x1, double x2, double x3, const int *sh, int sgn) {
  const double x[4] = {x0, x1, x2, x3};
  int e = kEmpty;
  for (int j = 0; j < 4; ++j) {
    const int f = (__double2hiint(x[j]) >> 20) & 0x7ff;
    if (f == 0x7ff) return kNonfinite;
    if (x[j] != 0.0) e = max(e, max(f, 1) - sgn * (sh[j] >> 20));
  }
  return e;
}

// |x| as 8 biased digits d_p + 128, digit p in byte 7 - p; base = the row's
// exponent plus the scaling of this k, minus 1. The significand is placed 9 bits
// up (an entry at the row's scale fills 62 bits) and moved down by the entry's
// distance from the row's scale (truncated; a distance of 64 or more, or below
// zero as in a non-finite row, gives zero). A subnormal has no hidden bit and the
// exponent 1.
__device__ __forceinline__ unsigned long long digits(double x, int base) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t h = hi & 0x7FF00000u, hb = min(h, 0x00100000u);
  const uint32_t mh = (hi & 0x000FFFFFu) | hb;
  const uint32_t d = (uint32_t)base - ((h - hb) >> 20);
  unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 9) << 32) | (lo << 9);
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(d));         // amounts above 63 give zero
  return m + 0x8080808080808080ull;
}

// One bit per entry of u (four consecutive k, bits 0 to 3): its leading digit is
// 5 or more, i.e. the entry is at least 4.5 / 64 of the row's scale. The biased
// leading bytes are 128 to 192.
__device__ __forceinline__ uint32_t large_bits(const unsigned long long (&u)[4]) {
  const uint32_t a = __byte_perm((uint32_t)(u[0] >> 32), (uint32_t)(u[1] >> 32), 0x0073);
  const uint32_t b = __byte_perm((uint32_t)(u[2] >> 32), (uint32_t)(u[3] >> 32), 0x0073);
  const uint32_t w = __byte_perm(a, b, 0x5410) & 0x7F7F7F7Fu;
  return ((((w + 0x7B7B7B7Bu) >> 7) & 0x01010101u) * 0x10204080u) >> 28;
}

// Adds a group's terms of the outputs marked in todo (bit t: column c4 + t % 4 +
// t / 4 * 16 of this lane's row) to them in FP64: r the row's first term in the
// group, cols + coff[column] the column's. Few outputs of a column: the lanes share
// the terms of one after the other; many: each lane its own.
constexpr int kLaneFallback = 8;
__device__ __noinline__ void fallback(uint32_t todo, const double *r, long long sr, const double *cols,
                                      const long long *coff, long long sc, int n, double *out, int c4) {
  const int lane = threadIdx.x & 31;
  const uint32_t any = __reduce_or_sync(0xffffffffu, todo);
#pragma unroll 1
  for (uint32_t rest = any; rest != 0; rest &= rest - 1) {
    const int t = __ffs(rest) - 1, col = c4 + t % 4 + t / 4 * (kThreadsS / 32);
    const bool mine = todo >> t & 1u;
    uint32_t lanes = __ballot_sync(0xffffffffu, mine);
    const double *c = cols + coff[col];
    if (__popc(lanes) >= kLaneFallback) {
      double v = 0.0;
#pragma unroll 8
      for (int k = 0; k < n; ++k) v = fma(r[k * sr], c[k * sc], v);
      if (mine) out[col] += v;
      continue;
    }
    for (; lanes != 0; lanes &= lanes - 1) {
      const int l = __ffs(lanes) - 1;
      const double *rl = reinterpret_cast<const double *>(
          __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(r), l));
      double v = 0.0;
      for (int k = lane; k < n; k += 32) v = fma(rl[k * sr], c[k * sc], v);
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == l) out[col] += v;
    }
  }
}

// Digits of four consecutive k of one row as FP16 (exact integers): 8 bytes per
// digit slice at dst + p * slice. The bytes of two k are interleaved; a byte
// b = d + 128 under 0x64 is the FP16 number 1024 + b, and one packed
// multiply-add with +-1 and -+1152 gives the signed digit.
__device__ __forceinline__ void store_digits(const unsigned long long (&u)[4], const double (&x)[4],
                                             unsigned char *dst, int slice) {
  uint32_t sg[2], off[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint32_t s = __byte_perm((uint32_t)__double2hiint(x[2 * j]), (uint32_t)__double2hiint(x[2 * j + 1]),
                                   0x7632) & 0x80008000u;
    sg[j] = s | 0x3C003C00u;             // +-1
    off[j] = s ^ 0xE480E480u;            // -+1152
  }
#pragma unroll
  for (int h = 1; h >= 0; --h) {         // digits 0..3, then 4..7
    uint32_t w[4][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t x0 = (uint32_t)(u[2 * j] >> (32 * h)), x1 = (uint32_t)(u[2 * j + 1] >> (32 * h));
      const uint32_t t[2] = {__byte_perm(x0, x1, 0x5140), __byte_perm(x0, x1, 0x7362)};
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint32_t v = __byte_perm(t[b >> 1], 0x64646464u, (b & 1) ? 0x4342 : 0x4140);
        asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(w[3 - b][j]) : "r"(v), "r"(sg[j]), "r"(off[j]));
      }
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
      *reinterpret_cast<uint2 *>(dst + (size_t)(p + 4 * (1 - h)) * slice) = make_uint2(w[p][0], w[p][1]);
  }
}

// A double out of range of the fast packing in combine: q 2^s with |q| <= 2^53.
__device__ __noinline__ double scaled(long long q, int s) {
  return ldexp((double)q, max(-5000, min(5000, s)));
}

// T = sum_l L_l 256^(7-l) times 2^(ex - 2112) as a double: the level sums are
// exact integers in FP32 (|L_l| <= l 2^21, |L_0| <= 2^19 over 128 terms), T is
// formed and rounded (once) in integer arithmetic, mostly additions and shifts:
// a 32 x 32 -> 64 multiply-add runs at 24 lanes per clock, an addition at 128.
// ex = e_i + f_j of the row and column exponents; t3: the sum in units of 2^-20 S.
__device__ __forceinline__ double combine(const uint32_t (&L)[kDig], int ex, int32_t &t3) {
  // levels 0..2 stay within 2^22: 1.5 2^23 + L holds L in its low bits; the
  // others take a conversion (a pipe of its own)
  int32_t v[kDig];
#pragma unroll
  for (int l = 0; l < kDig; ++l)
    v[l] = l < 3 ? __float_as_int(__uint_as_float(L[l]) + 12582912.0f) - 0x4B400000
                 : __float2int_rn(__uint_as_float(L[l]));
  // carries to base 256 from the low end, to base 65536 for the upper levels:
  // T = t3 2^48 + (t2 modulo 2^16) 2^32 + the low bytes of x4, x5, x6, v7
  const int32_t x6 = v[6] + (v[7] >> 8);
  const int32_t x5 = v[5] + (x6 >> 8);
  const int32_t x4 = v[4] + (x5 >> 8);
  const int32_t t2 = v[2] * 256 + v[3] + (x4 >> 8);
  t3 = v[0] * 256 + v[1] + (t2 >> 16);
  const uint32_t s = (uint32_t)(t3 >> 31);           // sign: 0 or ~0
  // |T| = a 2^64 + b 2^32 + c
  uint32_t c = __byte_perm(__byte_perm((uint32_t)v[7], (uint32_t)x6, 0x0040),
                           __byte_perm((uint32_t)x5, (uint32_t)x4, 0x0040), 0x5410) ^ s;
  uint32_t b = __byte_perm((uint32_t)t2, (uint32_t)t3, 0x5410) ^ s;
  uint32_t a = (uint32_t)(t3 >> 16) ^ s;
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, %2, 0;"
      : "+r"(c), "+r"(b), "+r"(a) : "r"(s & 1u));
  int z = 0;                                         // move the first nonzero word to the front
  if (a == 0) { a = b; b = c; c = 0; z = 32; }
  if (a == 0) { a = b; b = c; z += 32; }
  const int n = __clz(a);                            // 32 when T = 0
  z += n;
  a = __funnelshift_l(b, a, n);                      // top 64 bits of |T|, normalized
  b = __funnelshift_l(c, b, n);
  const int E = ex - z - 994;                        // biased exponent: |T| = q 2^(43 - z), q in [2^52, 2^53]
  const uint32_t r = (b >> 10) & 1u;
  if (n == 32) return 0.0;
  if ((unsigned)(E - 1) >= 2045u) {
    const long long q = (long long)((((unsigned long long)a << 32) | b) >> 11) + r;
    return scaled(s ? -q : q, E - 1075);
  }
  uint32_t lo = __funnelshift_r(b, a, 11), hi = (a >> 11) + ((uint32_t)(E - 1) << 20);
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(r));
  return __hiloint2double((int)(hi | (s & 0x80000000u)), (int)lo);
}

template <int NT>
__global__ void __launch_bounds__(kThreadsAll, 1)
gemm_split_kernel(const SplitArgs g) {
  pdl_enter();
  if (g.skip_dev && *g.skip_dev) return;
  using Sm = SplitSmem<NT>;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ long long s_roff[kRows], s_coff[NT], s_rout[kRows], s_cout[NT];
  __shared__ int s_mr[2][kRows], s_mc[2][NT];          // largest exponents of a chunk, by its parity
  __shared__ int s_er[kRows], s_ec[NT];                // scales of the group
  __shared__ __align__(16) int s_sh[kKc];              // exponent moved from rows to columns at each k
  // large entries of the group, a bit per k (large_bits), a word per chunk
  __shared__ __align__(16) uint32_t s_lr[kRows][kGroup], s_lc[NT][kGroup];
  __shared__ uint32_t s_taddr;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_odd, s_go;                  // s_go: 0 / 1 first / later chunk of a group, 2 stop
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned blk = blockIdx.x;
  const int tc = (int)(blk % (unsigned)g.tiles_c); blk /= (unsigned)g.tiles_c;
  const int tr = (int)(blk % (unsigned)g.tiles_r); blk /= (unsigned)g.tiles_r;
  const int ks = (int)(blk % (unsigned)g.ksplit);
  const int b = (int)(blk / (unsigned)g.ksplit);
  const int b1 = b / g.bdiv, b2 = b % g.bdiv;
  const double *Rp = g.R.p + b1 * g.R.sb1 + b2 * g.R.sb2;
  const double *Cp = g.C.p + b1 * g.C.sb1 + b2 * g.C.sb2;
  const int r0 = tr * kRows, c0 = tc * NT;
  const int nr = min(kRows, g.R.n - r0), nc = min(NT, g.C.n - c0);
  const int kbeg = ks * g.kchunk, kend = min(g.K, kbeg + g.kchunk);

  if (warp == kThreadsS / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&s_taddr)), "r"(Sm::kTmem) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
      s_odd = 0;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&s_bar)) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  } else if (tid < kRows) {
    const int r = min(r0 + tid, g.R.n - 1);
    const int h = g.R.div < g.R.n ? r / g.R.div : 0, l = r - h * g.R.div;
    s_roff[tid] = h * g.R.s_hi + l * g.R.s_lo;
    s_rout[tid] = h * g.or_hi + l * g.or_lo;
    s_mr[0][tid] = kEmpty;
  } else if (tid < kRows + NT) {
    const int t = tid - kRows, r = min(c0 + t, g.C.n - 1);
    const int h = g.C.div < g.C.n ? r / g.C.div : 0, l = r - h * g.C.div;
    s_coff[t] = h * g.C.s_hi + l * g.C.s_lo;
    s_cout[t] = h * g.oc_hi + l * g.oc_lo;
    s_mc[0][t] = kEmpty;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  double *raw_r = reinterpret_cast<double *>(sm + Sm::kRaw);
  double *raw_c = raw_r + kLdRaw * kKc;
  double *tile = reinterpret_cast<double *>(sm + Sm::kTile);
  // rows and columns of this thread where it moves whole tiles
  const int row = tid & (kRows - 1);
  const int kb = tid < kThreadsS ? tid >> 7 : NT;   // the issuing warp takes no share of loops from kb
  const int col = tid % NT, kq = tid / NT;
  bool fail = false;
  if (warp == kThreadsS / 32) {          // the issuing warp
    const uint32_t a0 = smem_u32(sm), bs = a0 + kABytes, td = s_taddr;
    for (int k0 = kbeg; k0 < kend; k0 += kKc) {
      wait_digits();
      const int go = *(volatile int *)&s_go;
      if (go == 2) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (lane == 0) {
#pragma unroll
        for (int kk = 0; kk < kKc / 16; ++kk)
#pragma unroll
          for (int p = 0; p < kDig; ++p)
#pragma unroll
            for (int q = 0; q + p < kDig; q += 256 / NT) {   // digits q .. of the columns, N <= 256
              const int n = NT * (kDig - p - q < 256 / NT ? kDig - p - q : 256 / NT);
              const uint64_t ad = smem_desc(a0 + p * (kRows * kKc * 2) + kk * 256);
              const uint64_t bd = smem_desc(bs + q * (NT * kKc * 2) + kk * 256);
              // kind::f16, FP16 x FP16 -> FP32, K-major, M = 128, N = n
              const uint32_t idesc = (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
              // the first products of a group overwrite the level sums
              const uint32_t en = (kk == 0 && p == 0) ? (uint32_t)go : 1u;
              asm volatile("{\n.reg .pred pr;\nsetp.ne.b32 pr, %4, 0;\n"
                           "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pr;\n}\n"
                           :: "r"(td + (uint32_t)((p + q) * NT)), "l"(ad), "l"(bd), "r"(idesc), "r"(en)
                           : "memory");
            }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     :: "r"(smem_u32(&s_bar)) : "memory");
      }
      __syncwarp();
    }
  }
  if (warp < kThreadsS / 32) {
  RawLoad<kRows, kLdRaw> lr;
  RawLoad<NT, Sm::kLdC> lc;
  lr.load(Rp, s_roff, nr, g.R.s_k, kbeg, kend);
  lc.load(Cp, s_coff, nc, g.C.s_k, kbeg, kend);
  // this thread's entries, in units of four k. A warp takes 16 rows x 8 k at a
  // time, lane bits 0-2 and 4 choosing the row and bit 3 the half of the k, so
  // that the 8-byte digit stores of half a warp fill 128 contiguous bytes: row
  // urow, k = 4 ukq + {0..3} and 16 further; in the first NT / 4 warps also
  // column ucol, k = 4 uckq + {0..3}
  const int ur = (lane & 7) + 8 * (lane >> 4), uh = (lane >> 3) & 1;
  const int urow = 16 * (warp & 7) + ur, ukq = 2 * (warp >> 3) + uh;
  const int ucol = 16 * (warp % (NT / 16)) + ur, uckq = 2 * (warp / (NT / 16)) + uh;
  const int units = warp < NT / 4 ? 3 : 2;
  // unit u: its k, its column (u = 2) or row, its entries and shifts
  auto fetch = [&](int u, double (&x)[4], int (&sh)[4]) {
    const int k = 4 * (u == 2 ? uckq : ukq + 4 * u);
    const double *p = u == 2 ? raw_c + k * Sm::kLdC + ucol : raw_r + k * kLdRaw + urow;
    const int ld = u == 2 ? Sm::kLdC : kLdRaw;
    const int4 s = *reinterpret_cast<const int4 *>(s_sh + k);
    sh[0] = s.x; sh[1] = s.y; sh[2] = s.z; sh[3] = s.w;
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = p[j * ld];
    return k;
  };
  uint32_t phase = 0;
  bool first = true;
  // room above the first chunk's largest entries for those of the group's
  // other chunks; none where there are no others
  const int margin = kend - kbeg > kKc ? 1 : 0;
  int par = 0, grp = 0, kgrp = kbeg;     // kgrp: the group's first term
#pragma unroll 1
  for (int k0 = kbeg;; k0 += kKc, par ^= 1) {
    const bool live = k0 < kend;         // false once: only the last group's sums are left
    if (live) {
      if (k0 > kbeg) conv_sync();        // every thread has taken its entries of the chunk before
      lr.store(raw_r, g.R.s_k);
      lc.store(raw_c, g.C.s_k);
      conv_sync();
      // scaling of each k by the largest exponents (an infinity or NaN does not
      // take part): a warp per k
      const uint32_t *hr = reinterpret_cast<const uint32_t *>(raw_r) + 1;
      const uint32_t *hc = reinterpret_cast<const uint32_t *>(raw_c) + 1;
#pragma unroll
      for (int i = 0; i < kKc / (kThreadsS / 32); ++i) {
        const int k = warp + kThreadsS / 32 * i;
        uint32_t h[(NT + 31) / 32 + kRows / 32], c = 0, a = 0;
#pragma unroll
        for (int q = 0; q < (NT + 31) / 32; ++q) {
          h[q] = lane + 32 * q < NT ? hc[2 * (k * Sm::kLdC + lane + 32 * q)] & 0x7FF00000u : 0u;
          c = max(c, h[q]);
        }
#pragma unroll
        for (int q = 0; q < kRows / 32; ++q) {
          h[(NT + 31) / 32 + q] = hr[2 * (k * kLdRaw + lane + 32 * q)] & 0x7FF00000u;
          a = max(a, h[(NT + 31) / 32 + q]);
        }
        if (max(a, c) == 0x7FF00000u) {
          s_odd = 1;
          a = c = 0;
#pragma unroll
          for (int q = 0; q < (NT + 31) / 32 + kRows / 32; ++q) {
            const uint32_t f = h[q] == 0x7FF00000u ? 0u : h[q];
            if (q < (NT + 31) / 32) c = max(c, f); else a = max(a, f);
          }
        }
        a = __reduce_max_sync(0xffffffffu, a);
        c = __reduce_max_sync(0xffffffffu, c);
        if (lane == 0) s_sh[k] = (a != 0 && c != 0) ? ((((int)(a >> 20) - (int)(c >> 20)) >> 1) << 20) : 0;
      }
      conv_sync();
      // exponents of the rows and columns after that scaling
      const bool odd = *(volatile int *)&s_odd != 0;
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        if (u == units) break;
        double x[4];
        int sh[4];
        const int k = fetch(u, x, sh);
        uint32_t sub = 0;
        const int sgn = u == 2 ? -1 : 1;
        int e = max_high(x, sh, sgn, sub);
        e = e == INT_MIN ? kEmpty : e >> 20;
        if (odd || sub != 0) e = max_expo(x[0], x[1], x[2], x[3], s_sh + k, sgn);
        atomicMax(u == 2 ? &s_mc[par][ucol] : &s_mr[par][urow], e);
      }
      conv_sync();
    }
    if (grp > 0) {
      // the digit products issued last (bounded wait)
      uint32_t done = 0;
      for (long long w = 0; w < g.waits && !done; ++w)
        asm volatile("{\n.reg .pred pr;\nmbarrier.try_wait.parity.shared::cta.b64 pr, [%1], %2;\n"
                     "selp.u32 %0, 1, 0, pr;\n}\n"
                     : "=r"(done) : "r"(smem_u32(&s_bar)), "r"(phase) : "memory");
      // after giving up: the products still read shared and write tensor memory, so
      // they get another (bounded) wait before either goes
      for (long long w = 0, late = done; w < kMmaWaits && !late; ++w) {
        uint32_t p;
        asm volatile("{\n.reg .pred pr;\nmbarrier.try_wait.parity.shared::cta.b64 pr, [%1], %2;\n"
                     "selp.u32 %0, 1, 0, pr;\n}\n"
                     : "=r"(p) : "r"(smem_u32(&s_bar)), "r"(phase) : "memory");
        late = p;
      }
      phase ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // a group ends when it is full, or an entry exceeds its row's or
      // column's scale, or no chunk follows
      bool over = grp == kGroup || !live || !done;
      if (live && tid < kRows) over |= s_mr[par][tid] > s_er[tid];
      else if (live && tid < kRows + NT) over |= s_mc[par][tid - kRows] > s_ec[tid - kRows];
      if (conv_any(over)) {
        if (conv_any(!done)) {
          fail = true;
          if (live) {                    // the issuing warp waits for this chunk
            if (tid == 0) *(volatile int *)&s_go = 2;
            digits_ready();
          }
          break;
        }
        // add the level sums to the output tile
        const int orow = 32 * (warp & 3) + lane;
        const int eri = s_er[orow];
        uint4 lrow = *reinterpret_cast<const uint4 *>(s_lr[orow]);
        if (grp < 4) lrow.w = 0;         // chunks the group does not have
        if (grp < 3) lrow.z = 0;
        if (grp < 2) lrow.y = 0;
        uint32_t todo = 0;               // this thread's outputs that need the FP64 sum
        const uint32_t td = s_taddr + ((uint32_t)(32 * (warp & 3)) << 16);
#pragma unroll 1
        for (int c4 = 4 * (warp >> 2); c4 < nc; c4 += kThreadsS / 32) {
          uint32_t L[4][kDig];
#pragma unroll
          for (int l = 0; l < kDig; ++l)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(L[0][l]), "=r"(L[1][l]), "=r"(L[2][l]), "=r"(L[3][l])
                         : "r"(td + (uint32_t)(l * NT + c4)) : "memory");
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          double *o = tile + orow * Sm::kLdT + c4;
          double v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int ecj = s_ec[c4 + j];
            int32_t t3;
            v[j] = combine(L[j], eri + ecj, t3);
            // a row or column of zeros against finite entries: an exact zero. One with a
            // non-finite entry has no digits and so no large bits
            const bool inf = max(eri, ecj) > kNonfinite / 2;
            const bool empty = min(eri, ecj) < kEmpty / 2 && !inf;
            if (empty) v[j] = 0.0;
            const uint4 lcol = *reinterpret_cast<const uint4 *>(s_lc[c4 + j]);
            const uint32_t both = (lrow.x & lcol.x) | (lrow.y & lcol.y) | (lrow.z & lcol.z) | (lrow.w & lcol.w);
            if (both == 0 && (abs(t3) < kSure || inf) && !empty && orow < nr && c4 + j < nc) {
              v[j] = 0.0;
              todo |= 1u << (j + (c4 >> 4) * 4);
            }
          }
          // sums of earlier groups, behind a real branch: a predicated-off FP64
          // addition holds the FP64 unit like a full one
          asm volatile("{\n.reg .pred p;\n.reg .f64 a, b, c, d;\nsetp.ne.u32 p, %5, 0;\n@p bra.uni DONE;\n"
                       "ld.shared.f64 a, [%4];\nld.shared.f64 b, [%4+8];\nld.shared.f64 c, [%4+16];\n"
                       "ld.shared.f64 d, [%4+24];\nadd.rn.f64 %0, %0, a;\nadd.rn.f64 %1, %1, b;\n"
                       "add.rn.f64 %2, %2, c;\nadd.rn.f64 %3, %3, d;\nDONE:\n}\n"
                       : "+d"(v[0]), "+d"(v[1]), "+d"(v[2]), "+d"(v[3])
                       : "r"(smem_u32(o)), "r"((uint32_t)first) : "memory");
#pragma unroll
          for (int j = 0; j < 4; ++j) o[j] = v[j];
        }
        if (__any_sync(0xffffffffu, todo != 0))
          fallback(todo, Rp + s_roff[orow] + kgrp * g.R.s_k, g.R.s_k, Cp + kgrp * g.C.s_k, s_coff, g.C.s_k,
                   min(k0, kend) - kgrp, tile + orow * Sm::kLdT, 4 * (warp >> 2));
        first = false;
        grp = 0;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        conv_sync();                     // s_er, s_ec read before they change
      }
    }
    if (!live) break;
    if (k0 + kKc < kend) {               // in flight under the digits
      lr.load(Rp, s_roff, nr, g.R.s_k, k0 + kKc, kend);
      lc.load(Cp, s_coff, nc, g.C.s_k, k0 + kKc, kend);
    }
    if (grp == 0) {
      if (tid < kRows) s_er[tid] = s_mr[par][tid] + margin;
      else if (tid < kRows + NT) s_ec[tid - kRows] = s_mc[par][tid - kRows] + margin;
      kgrp = k0;
      conv_sync();
    }
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      if (u == units) break;
      double x[4];
      int sh[4];
      const int k = fetch(u, x, sh);
      const int base = (u == 2 ? s_ec[ucol] : s_er[urow]) - 1;
      unsigned long long d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) d[j] = digits(x[j], u == 2 ? base - (sh[j] >> 20) : base + (sh[j] >> 20));
      const int i = u == 2 ? ucol : urow;
      // the other half of these eight k is with lane ^ 8
      uint32_t big = large_bits(d) << (k & 4);
      big |= __shfl_xor_sync(0xffffffffu, big, 8);
      if (uh == 0)
        reinterpret_cast<unsigned char *>(u == 2 ? s_lc[ucol] : s_lr[urow])[4 * grp + (k >> 3)] = (unsigned char)big;
      store_digits(d, x, sm + (u == 2 ? kABytes : 0) + ((i >> 3) * (kKc / 8) + (k >> 3)) * 128 + (i & 7) * 16 +
                             2 * (k & 4), (u == 2 ? NT : kRows) * kKc * 2);
    }
    // the next chunk's exponents start empty
    if (tid < kRows) s_mr[par ^ 1][tid] = kEmpty;
    else if (tid < kRows + NT) s_mc[par ^ 1][tid - kRows] = kEmpty;
    if (tid == 0) *(volatile int *)&s_go = grp > 0;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    digits_ready();
    ++grp;
  }
  }
  fail = __syncthreads_or(fail) != 0;
  if (warp == kThreadsS / 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(s_taddr), "r"(Sm::kTmem)
                 : "memory");
  if (fail) {
    if (tid == 0) atomicOr(g.health != nullptr ? g.health : &g_split_error, kHealthTimeout);
    for (int e = tid; e < kRows * NT; e += kThreadsS)
      tile[(e / NT) * Sm::kLdT + e % NT] = __longlong_as_double(0x7FF8000000000000LL);
    __syncthreads();
  }

  // a K slice of a split product goes to partial (dense, the result's contiguous
  // index fastest), unscaled: split_sum_kernel adds the slices
  double alpha = 1.0;
  double *out;
  if (g.ksplit == 1) {
    alpha = g.alpha * (g.alpha_dev ? *g.alpha_dev : 1.0);
    out = g.out + b1 * g.ob1 + b2 * g.ob2;
  } else {
    out = g.partial + ((long long)b * g.ksplit + ks) * g.R.n * g.C.n;
    const bool rows_fast = g.or_lo == 1;
    __syncthreads();
    if (tid < kRows) s_rout[tid] = (long long)(r0 + tid) * (rows_fast ? 1 : g.C.n);
    else if (tid < kRows + NT) s_cout[tid - kRows] = (long long)(c0 + tid - kRows) * (rows_fast ? g.R.n : 1);
    __syncthreads();
  }
  const bool scale = alpha != 1.0;
  // lanes along the result's contiguous index; four values in flight
  if (g.or_lo == 1) {
    double *o = out + s_rout[row];
    const double *src = tile + row * Sm::kLdT;
#pragma unroll 1
    for (int c4 = kb; c4 < nc; c4 += 4 * (kThreadsS / kRows)) {
      double v[4];
      long long off[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = min(c4 + j * (kThreadsS / kRows), NT - 1);
        v[j] = src[c];
        off[j] = s_cout[c];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c4 + j * (kThreadsS / kRows) < nc && row < nr) o[off[j]] = scale ? v[j] * alpha : v[j];
    }
  } else if (kq < kThreadsS / NT) {
    constexpr int step = kThreadsS / NT;
    double *o = out + s_cout[col];
#pragma unroll 1
    for (int r4 = kq; r4 < nr; r4 += 4 * step) {
      double v[4];
      long long off[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = min(r4 + j * step, kRows - 1);
        v[j] = tile[r * Sm::kLdT + col];
        off[j] = s_rout[r];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (r4 + j * step < nr && col < nc) o[off[j]] = scale ? v[j] * alpha : v[j];
    }
  }
}

// Adds the K slices of a split product in slice order (the result does not
// depend on which block finished when), a thread per output.
__global__ void __launch_bounds__(256)
split_sum_kernel(const SplitArgs g) {
  pdl_enter();
  if (g.skip_dev && *g.skip_dev) return;
  const long long slab = (long long)g.R.n * g.C.n;
  const long long e = blockIdx.x * 256LL + threadIdx.x;
  if (e >= slab) return;
  const int b = blockIdx.y;
  const double *P = g.partial + (long long)b * g.ksplit * slab + e;
  double sum = 0.0;
#pragma unroll 1
  for (int k = 0; k < g.ksplit; k += 8) {              // eight loads in flight
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = k + j < g.ksplit ? P[(k + j) * slab] : 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (k + j < g.ksplit) sum += x[j];
  }
  const bool rows_fast = g.or_lo == 1;
  const unsigned n = rows_fast ? g.R.n : g.C.n, hi = (unsigned)e / n, lo = (unsigned)e - hi * n;
  const int r = (int)(rows_fast ? lo : hi), c = (int)(rows_fast ? hi : lo);
  const int rh = r / g.R.div, ch = c / g.C.div;
  const int b1 = b / g.bdiv, b2 = b % g.bdiv;
  g.out[b1 * g.ob1 + b2 * g.ob2 + rh * g.or_hi + (r - rh * g.R.div) * g.or_lo + ch * g.oc_hi +
        (c - ch * g.C.div) * g.oc_lo] = sum * (g.alpha * (g.alpha_dev ? *g.alpha_dev : 1.0));
}

long long cdiv(long long a, long long b) { return (a + b - 1) / b; }

constexpr int kSms = 152;

struct SplitPlan {
  SplitArgs g;
  int nt = 64, batch = 1;
  long long blocks = 0;
  double cost = 0.0;                     // predicted clocks
};

// What a shape's launches share: the form and the K split, and whether the
// tensor-core product is expected to beat the DFMA one.
struct Choice {
  bool use = false, swap = false;
  int nt = 64, kchunk = 0, ksplit = 1;
};

// The launch of a product (swap: N on the 128-row side, else M) with NT
// columns per tile. Batch indices that one operand does not depend on are
// folded into the other operand's index (a batch of 20 x 20 products with one
// shared factor becomes one tall product): index = (batch index, row) in two
// levels.
SplitPlan orient(const Gemm &q, bool swap, int nt) {
  SplitPlan L;
  SplitArgs &g = L.g;
  const int nb1 = q.batch / q.bdiv, nb2 = q.bdiv;
  SplitOperand A{q.A, q.sA1, q.sA2, 0, q.sAm, q.sAk, q.M, q.M};
  SplitOperand B{q.B, q.sB1, q.sB2, 0, q.sBn, q.sBk, q.N, q.N};
  long long am_hi = 0, bn_hi = 0;        // result strides of the folded levels
  long long ob1 = q.sC1, ob2 = q.sC2;
  int batch = q.batch, bdiv = q.bdiv;
  auto fold = [&](SplitOperand &x, int count, long long sx, long long so, long long &o_hi) {
    if (x.n != x.div) return false;      // one fold per operand
    if ((long long)x.n * count >= (1LL << 31)) return false;
    x.s_hi = sx;
    x.n *= count;
    o_hi = so;
    return true;
  };
  bool f2 = nb2 == 1, f1 = nb1 == 1;
  if (!f2 && q.sA2 == 0) f2 = fold(B, nb2, q.sB2, q.sC2, bn_hi);
  else if (!f2 && q.sB2 == 0) f2 = fold(A, nb2, q.sA2, q.sC2, am_hi);
  if (!f1 && q.sA1 == 0) f1 = fold(B, nb1, q.sB1, q.sC1, bn_hi);
  else if (!f1 && q.sB1 == 0) f1 = fold(A, nb1, q.sA1, q.sC1, am_hi);
  if (f1 && f2) { batch = 1; bdiv = 1; }
  else if (f2) { batch = nb1; bdiv = 1; }                 // b1 left: index b1 = b
  else if (f1) { batch = nb2; bdiv = nb2; }               // b2 left: b1 = 0, b2 = b
  if (f1) { A.sb1 = B.sb1 = 0; ob1 = 0; }
  if (f2) { A.sb2 = B.sb2 = 0; ob2 = 0; }
  g.R = swap ? B : A;
  g.C = swap ? A : B;
  g.out = q.C;
  g.ob1 = ob1;
  g.ob2 = ob2;
  g.or_hi = swap ? bn_hi : am_hi;
  g.or_lo = swap ? q.sCn : q.sCm;
  g.oc_hi = swap ? am_hi : bn_hi;
  g.oc_lo = swap ? q.sCm : q.sCn;
  g.K = q.K;
  g.bdiv = bdiv;
  L.nt = nt;
  g.tiles_r = (int)cdiv(g.R.n, kRows);
  g.tiles_c = (int)cdiv(g.C.n, nt);
  g.alpha = q.alpha;
  g.alpha_dev = q.alpha_dev;
  g.skip_dev = q.skip_dev;
  g.partial = nullptr;
  g.health = nullptr;
  g.waits = kMmaWaits;
  L.batch = batch;
  return L;
}

// The best K split of an oriented product, with its cost.
void plan_split(SplitPlan &L) {
  SplitArgs &g = L.g;
  const long long tiles = (long long)g.tiles_r * g.tiles_c * L.batch;
  // K splits: up to eight blocks per SM. Cost in clocks of the busiest SM,
  // measured with clock marks: ~6500 to start, load the first chunk and store,
  // ~7500 per chunk (exponents, digits, products), ~140 per column and group to
  // combine; a split adds a launch (~5000) and its partial sums' traffic.
  const long long chunks = cdiv(g.K, kKc);
  const int cols = std::min(L.nt, g.C.n);
  const double outputs = (double)g.R.n * g.C.n * L.batch;
  L.cost = 1e300;
  for (long long split = 1; split <= std::min<long long>(chunks, std::max<long long>(1, 8 * kSms / tiles)); ++split) {
    const long long per = cdiv(chunks, split), ns = cdiv(chunks, per);
    if (split > 1 && (ns != split || L.batch > 65535 || (double)g.R.n * g.C.n > 2e9)) continue;
    const double block = 6500.0 + 7500.0 * (double)per + 140.0 * cols * (double)cdiv(per, kGroup);
    const double cost = block * (double)cdiv(tiles * ns, kSms) +
                        (ns > 1 ? 5000.0 + 16.0 * (double)ns * outputs / (64.0 * kSms) : 0.0) +
                        2.0 * (double)(tiles * ns * per);
    if (cost < L.cost) {
      L.cost = cost;
      g.kchunk = (int)(per * kKc);
      g.ksplit = (int)ns;
      L.blocks = tiles * ns;
    }
  }
}

// Choices are cached per shape (callers issue hundreds of small products per
// millisecond). Products under 1e6 multiply-adds are not looked at: every DFMA
// form of them takes under 10 us, and one chunk of digits alone takes 8. Above,
// the DFMA product is predicted at 230 multiply-adds per clock (75% of the FP64
// units, what its mid-sized products reach) plus 12000 clocks. Measured on both
// sides of the line (us, digits against DFMA): 1 x 50 x 50 x 1600 20 and 24,
// 400 x 100 x 100 14 and 20, 50 x 1600 x 50 15 and 13, 300 x 100 x 100 14 and 10.
Choice choose(const Gemm &q) {
  using Key = std::array<int, 6>;
  struct Hash {
    size_t operator()(const Key &k) const {
      size_t h = 1469598103934665603ull;
      for (int v : k) h = (h ^ (size_t)(unsigned)v) * 1099511628211ull;
      return h;
    }
  };
  static std::mutex mu;
  static std::unordered_map<Key, Choice, Hash> cache;
  const Key key{q.M, q.N, q.K, q.batch, q.bdiv,
                (q.sA1 == 0) | (q.sA2 == 0) << 1 | (q.sB1 == 0) << 2 | (q.sB2 == 0) << 3};
  {
    std::lock_guard<std::mutex> lock(mu);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
  }
  Choice c;
  double best = 1e300;
  for (int nt : {64, 48, 32})
    for (bool swap : {false, true}) {
      SplitPlan L = orient(q, swap, nt);
      plan_split(L);
      if (L.cost < best) {
        best = L.cost;
        c = Choice{true, swap, nt, L.g.kchunk, L.g.ksplit};
      }
    }
  c.use = best < (double)q.M * q.N * (double)q.K * q.batch / 230.0 + 12000.0;
  std::lock_guard<std::mutex> lock(mu);
  if (cache.size() < (1u << 16)) cache.emplace(key, c);
  return c;
}

SplitPlan split_plan(const Gemm &q) {
  const Choice c = choose(q);
  SplitPlan L = orient(q, c.swap, c.nt);
  L.g.kchunk = c.kchunk;
  L.g.ksplit = c.ksplit;
  L.blocks = (long long)L.g.tiles_r * L.g.tiles_c * L.batch * c.ksplit;
  return L;
}

template <int NT>
cudaError_t launch_split(const SplitPlan &L, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(gemm_split_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       SplitSmem<NT>::kBytes);
  if (e != cudaSuccess) return e;
  e = launch_k(gemm_split_kernel<NT>, (unsigned)L.blocks, kThreadsAll, SplitSmem<NT>::kBytes, st, L.g);
  note_launch();
  return e;
}

thread_local bool t_split = true;

}  // namespace

void set_split_products(bool on) { t_split = on; }

bool gemm_split_applicable(const Gemm &g) {
  if (!t_split || g.prec != kPrecFP64 || g.dyn_dev != nullptr || g.beta != 0.0) return false;
  if (g.batch % g.bdiv != 0) return false;
  // HATT_GEMM_FORM=dfma (read once): a test hook that keeps every product on
  // the DFMA kernel
  static const bool off = [] {
    const char *v = getenv("HATT_GEMM_FORM");
    return v != nullptr && strcmp(v, "dfma") == 0;
  }();
  if (off) return false;
  if ((double)g.M * g.N * (double)g.K * g.batch < 1e6) return false;
  return choose(g).use;
}

size_t gemm_split_scratch_doubles(const Gemm &g) {
  const SplitPlan L = split_plan(g);
  return L.g.ksplit > 1 ? (size_t)L.g.ksplit * g.batch * (size_t)g.M * g.N : 0;
}

cudaError_t gemm_split(const Gemm &q, double *scratch, cudaStream_t st) {
  SplitPlan L = split_plan(q);
  if (L.g.ksplit > 1 && scratch == nullptr) return cudaErrorInvalidValue;
  if (L.blocks >= (1LL << 31)) return cudaErrorInvalidConfiguration;
  L.g.partial = scratch;
  L.g.health = health_target();
  L.g.waits = mma_waits();
  const cudaError_t e = L.nt == 64 ? launch_split<64>(L, st) : L.nt == 48 ? launch_split<48>(L, st)
                                                                          : launch_split<32>(L, st);
  if (e != cudaSuccess || L.g.ksplit == 1) return e;
  const dim3 grid((unsigned)cdiv((long long)L.g.R.n * L.g.C.n, 256), (unsigned)L.batch);
  launch_k(split_sum_kernel, grid, 256, 0, st, L.g);
  note_launch();
  return cudaGetLastError();
}

cudaError_t split_error_word(int *value, bool clear) {
  cudaError_t e = cudaMemcpyFromSymbol(value, g_split_error, sizeof(int));
  if (e == cudaSuccess && clear && *value != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_split_error, &zero, sizeof(int));
  }
  return e;
}

}  // namespace hatt
