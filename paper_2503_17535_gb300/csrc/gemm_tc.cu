// FP64 and complex128 GEMMs on the tcgen05 tensor cores by exact digit
// slicing (an Ozaki-type splitting of each operand into fp16 digit matrices).
//
// Why: the FP64 FMA pipe of this GPU does 4 flop/clk/SM, while the 16-bit
// tensor cores do ~7000.  A real product C = A B is computed as
//
//   A(i, k) ~ 2^{e_i} sum_p a_p(i, k) 2^{2-8p},   B(k, j) ~ 2^{f_j} sum_q b_q(k, j) 2^{2-8q},
//
// p, q = 1..8, where 2^{e_i} (2^{f_j}) is the power of two above the
// largest |A(i, :)| (|B(:, j)|) and the digits are the balanced base-256
// digits of the scaled value rounded to 62 fraction bits: the leading digit
// in [-64, 64], the others in [-128, 127].  Integers of that size are exact in
// fp16, their products are exact in the fp32 accumulators of tcgen05.mma, and
// so are sums below 2^24 of the products that share one anti-diagonal
// D = p + q (weight 2^{4-8D}).  The product keeps the 36 pairs with p + q <= 9
// and accumulates each diagonal exactly in its own TMEM accumulator over K
// chunks of up to 128.  The epilogue reduces the eight diagonal sums to one
// 64-bit fixed-point integer (as many fraction bits as the sum of K products
// leaves: 63 - ceil(log2 K), at most 62; what lies below rounded once) and
// scales it by 2^{e_i + f_j} into FP64.  Errors: operand
// rounding 2^{-63} 2^{e_i} per entry (unbiased), dropped pairs at most
// 2^{-59} K 2^{e_i + f_j}, half a unit of the fixed point per chunk, and the
// final rounding to FP64: at or below FP64's own rounding error for a dot
// product of length K when rows and columns are not far from their largest
// entries.
//
// Why 8-bit digits: ten 6-bit digits (the earlier form) take 55 tensor-core
// products and ten accumulators per output, allow chunks of 256, and write 20
// digit bytes per entry; eight 8-bit digits take 36 products, eight
// accumulators and 16 bytes.  Wider digits would need chunks below 36.
//
// Layout: the slicing kernel writes each operand's digits, K-major, in the
// tensor core's canonical no-swizzle layout (8-row x 16-byte core matrices;
// a 16-deep k step of a 128-row A tile is one 4 KB block per digit, of a
// TN-column B tile one block of 32 TN bytes), so that one k step of all
// digits is one contiguous bulk copy (cp.async.bulk) per operand.  The GEMM
// kernel computes 128 x TN output tiles (TN = 64 or 32), one CTA per SM
// walking the launch's tiles: a producer warp streams the digit blocks through
// a shared-memory ring, one thread issues the products (digits of B stacked
// along N, up to 256 rows per MMA, land in adjacent diagonal accumulators),
// the eight TMEM accumulators take 512 columns (TN = 64) or 256 (TN = 32, two
// sets, so that the next chunk's products overlap the read-back), and sixteen
// epilogue warps (four per TMEM lane quarter, one per quarter of the columns)
// read them back while the next tile's copies and products proceed.  A product
// with few rows may run transposed (C^T = B^T A^T, C's rows on the TN side).
//
// Complex products are two launches, one per component of C, each
// accumulating two real products in the same TMEM accumulators
// (Re = Ar Br - Ai Bi with the second product negated by the MMA's negate-B
// bit, Im = Ar Bi + Ai Br): the real and imaginary parts of a row of A (a
// column of B) are scaled by one power of two, above the largest |re| or |im|
// of the row, so that their digit products carry the same weights; the
// error bound above then holds with 2K terms and those joint row scales.
#include "devmem.h"
#include "linalg.h"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace hps {
namespace tc {

constexpr int DIG = 8;              // digits per operand
constexpr int BITS = 8;             // bits per digit
constexpr int FRAC = 62;            // fraction bits of the scaled operands (leading digit in [-64, 64])
constexpr int DSUM = 9;             // keep digit pairs with p + q <= DSUM (1-based)
constexpr int NDIAG = DSUM - 1;     // accumulators: D = 2 .. DSUM
constexpr int TM = 128, TK = 16;
constexpr int KC1 = 64;             // summed products a single-chunk tile may hold (KC = 64)
constexpr int KC2 = 128;            // k per exact fp32 accumulation chunk (KC = 128)
constexpr int ABLK = TM * TK * 2;   // bytes of one digit of an A tile k step
constexpr int ASTG = DIG * ABLK;
constexpr int bblk(int tn) { return tn * TK * 2; }   // of a B tile
constexpr int bstg(int tn) { return DIG * bblk(tn); }
constexpr int EPI_WARPS = 16;       // four per TMEM lane quarter, each a quarter of the tile's columns
constexpr int THREADS = 32 * EPI_WARPS + 64;   // + producer warp + MMA-issue warp
constexpr long SPIN = 1L << 22;     // polls before a wait gives up
constexpr int LSB1 = 57, LSB2 = 56; // fixed-point fraction bits of a full KC = 64 tile, of a full KC = 128 chunk
constexpr int LSB_MAX = 62;

// Shared memory: the copy ring; transposed tiles' staging (one block of
// 32 x TN / 4 results per epilogue warp, odd stride); at TN = 32 two tiles of
// old C values, copied a tile ahead.
constexpr int stages(int tn, bool trans) { return trans ? 3 : 4; }
constexpr int stage_bytes(int tn) { return ASTG + bstg(tn); }
constexpr int trans_bytes(int tn, bool trans) { return trans ? EPI_WARPS * 32 * (tn / 4 + 1) * 8 : 0; }
constexpr int old_bytes(int tn) { return tn == 32 ? 2 * TM * 32 * 8 : 0; }
constexpr int smem_bytes(int tn, bool trans) { return stages(tn, trans) * stage_bytes(tn) + trans_bytes(tn, trans) + old_bytes(tn); }
constexpr int accum_sets(int tn) { return 512 / (NDIAG * tn); }

// largest |sum of the digit products on diagonal D| per summed product: two
// pairs with a leading digit (64 * 128 each) and D - 3 others (128 * 128)
constexpr long diag_max(int D, long kc) { return (D == 2 ? 64L * 64 : (D - 2) * 128L * 128) * kc; }
static_assert(diag_max(9, KC2) < (1L << 24), "diagonal sums must stay exact in fp32");
// a float integer of magnitude up to 2^22 plus 1.5 * 2^23 holds it in its low mantissa bits
static_assert(diag_max(6, KC1) <= (1L << 22) && diag_max(7, KC1) / 2 < (1L << 22), "KC = 64 conversion");
static_assert(diag_max(4, KC2) <= (1L << 22) && diag_max(5, KC2) / 2 < (1L << 22) &&
              (diag_max(6, KC2) + 256) / 4 < (1L << 22) && (diag_max(7, KC2) + 512) / 4 < (1L << 22), "KC = 128 conversion");
// the lowest diagonals enter in the unit of the result, 2^(LSB1 - lsb) / 8 or
// 2^(LSB2 - lsb) / 16 of D = 8's, with n 2^(lsb - LSB1) <= 64 (n 2^(lsb - LSB2) <= 128) of
// n summed products, and D = 7's remainder 256 times: that too is a float integer below 2^22
static_assert((diag_max(8, KC1) + diag_max(9, KC1) / 256 + (256L << (LSB_MAX - LSB1))) / 8 < (1L << 22) &&
              (diag_max(8, KC2) + diag_max(9, KC2) / 256 + (512L << (LSB_MAX - LSB2))) / 16 < (1L << 22), "lowest diagonals");
static_assert(smem_bytes(64, true) <= 226 * 1024 && smem_bytes(64, false) <= 226 * 1024 &&
              smem_bytes(32, true) <= 226 * 1024 && smem_bytes(32, false) <= 226 * 1024, "shared memory too large");

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, no swizzle: start address, leading byte
// offset (between core matrices adjacent in K) and stride byte offset
// (between core matrices adjacent in M / N), version bits 46-48 = 0b001.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}

// Bounded wait on an mbarrier phase; gives up when another role has aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort, long limit = SPIN) {
  for (long it = 0; it < limit; ++it) {
    if (mbar_try(bar, parity)) return true;
    if (*abort) return false;
    if (it > 32) __nanosleep(64);
  }
  return false;
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ inline double part_of(double v, int) { return v; }
__device__ inline double part_of(const cplx& v, int part) { return part ? v.im : v.re; }

// One real operand as rows x K: element (r, k) = part(X[rmap(r) * rs + kmap(k) * ks]).
template <typename T>
struct Src {
  BOp<T> X;
  IMap rmap, kmap;
  int64_t rs = 1, ks = 1;
};

// exponent e of a row (max |x| < 2^e) from its biased maximum exponent
__device__ __forceinline__ int row_exp(int evm) { return evm ? evm - 1022 : 0; }

// The operands of one product call (A and B) as rows x K, cut into digit
// blocks.  A complex operand yields the digits of
// its real part in out and of its imaginary part in out2, both scaled by one
// power of two per row (above the row's largest |re| or |im|), so that the
// products of both parts can share accumulators.
constexpr int MAXOPS = 4;
template <typename T>
struct SplitSet {
  Src<T> s[MAXOPS];
  int R[MAXOPS], ltr[MAXOPS], RT[MAXOPS];   // rows, log2 of the tile rows, row tiles
  uint8_t* out[MAXOPS];
  uint8_t* out2[MAXOPS];  // imaginary part's digits (complex operands)
  int* ex[MAXOPS];    // biased exponent of each row's largest |entry| (0: zero row)
  int items[MAXOPS];  // batch items to cut: 1 for an operand shared by every item
};

// upper word of the magnitude (the larger part's of a complex entry)
__device__ __forceinline__ uint32_t mag_hi(double v) { return (uint32_t)__double2hiint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ uint32_t mag_hi(const cplx& v) { return max(mag_hi(v.re), mag_hi(v.im)); }

// Digits of v 2^{FRAC - e} rounded to an integer x (|x| < 2^62), as fp16
// values, for the 8 consecutive k of one 16-byte row segment of a block: blk
// points at digit 0's segment; digit p lies BLK bytes further.  With 128 added
// at every byte position, x's balanced base-256 digits are the bytes of the
// sum minus 128 each; a byte b becomes the fp16 value b - 128 as the difference
// of 1024 + b (bits 0x6400 | b) and 1152, two digits per instruction.
__device__ __forceinline__ void put_digits(const double (&v)[8], int evm, uint8_t* blk, int BLK) {
  uint32_t x[8][2];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t uh = (uint32_t)__double2hiint(v[c]), ul = (uint32_t)__double2loint(v[c]);
    const int ev = (int)((uh >> 20) & 0x7FF);
    // |v| 2^{FRAC - e + 1} is the mantissa << 10 shifted right by the
    // distance of v's exponent to the row's largest
    const unsigned long long full = ((unsigned long long)((uh & 0xFFFFFu) | 0x100000u) << 32 | ul) << 10;
    const int d = min(evm - ev, 63);
    unsigned long long m = full >> d;
    // ties to even (entries 2^-10 of the row's largest and below lose bits, few
    // at first, so that ties are common): up when the bits below the half bit
    // (the lowest d - 10 of the mantissa: of its lower word, and from d = 43 on all of
    // that and the lowest d - 42 of the upper) are not all zero or the integer is odd
    uint32_t below, above;
    asm("shl.b32 %0, %1, %2;" : "=r"(below) : "r"(ul), "r"(max(42 - d, 0)));   // 0 for shifts above 31
    asm("shl.b32 %0, %1, %2;" : "=r"(above) : "r"(uh), "r"(74 - d));
    below |= above;
    m = ev == 0 ? 0ull : (m + ((uint32_t)(m >> 1) & 1u | (below != 0u ? 1u : 0u))) >> 1;
    const unsigned long long t = (int)uh < 0 ? 0x8080808080808080ull - m : 0x8080808080808080ull + m;
    x[c][1] = (uint32_t)t;
    x[c][0] = (uint32_t)(t >> 32);
  }
#pragma unroll
  for (int p = 0; p < DIG; ++p) {
    const uint32_t byte = 3 - (p & 3);
    uint32_t w[4];
#pragma unroll
    for (int c = 0; c < 8; c += 2) {
      const uint32_t b2 =
          (__byte_perm(x[c][p >> 2], x[c + 1][p >> 2], byte | (byte + 4) << 8) & 0x00FF00FFu) | 0x64006400u;
      asm("add.rn.f16x2 %0, %1, %2;" : "=r"(w[c >> 1]) : "r"(b2), "r"(0xE480E480u));
    }
    *reinterpret_cast<uint4*>(blk + (int64_t)p * BLK) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// One launch for all operands.  A warp takes units of 32 rows x UK k (16 for
// real data: a whole k step; 8 for complex); of a CTA's NW warps (4, or 8 when
// so many share rows), KW share 32 rows and split the units of their inner
// dimension, and NW / KW such row groups share the CTA, so that short inner
// dimensions keep every warp busy.
// Long ones spread over the CS CTAs of a cluster as well (few rows and many k
// would leave most SMs idle).  Pass 1 finds each row's largest magnitude (by
// its upper word: only the exponent counts; over both parts of a complex
// row), pass 2 writes the digits, last unit first, which is still in
// registers; when no warp has more than one unit, each entry is read once.
// An operand whose k runs along
// its columns (ks = 1: B, or B^T in the A slot) is read in segments of UK
// entries per row and turned around in shared memory: one row per lane would
// touch 32 cache lines per load.  Rows beyond R are not written: their
// products land in outputs that nobody stores.
//
// Bound by instruction issue (100 per entry; 24 warps an SM) and the latency of
// a CTA's load-write cycle, not by memory (2.5 - 4 TB/s).  Loads by pointer
// steps instead of an index map looked up for each entry, row groups that wait for
// their own warps only and smaller CTAs for short K, us for both operands of
// 4096 items (before -> now): 164 x 164 x 32 339 -> 228, 128 x 128 x 68 538 ->
// 309, 114 x 32 x 64 246 -> 207; one pass over the Helmholtz build's products
// 15.1 -> 11.5 ms, the 3D elliptic's 11.0 -> 7.7.
template <typename T, int NW>
__global__ void __launch_bounds__(32 * NW, 24 / NW) k_split(SplitSet<T> ss, int K, int KT, int b0, int KW, int CS) {
  constexpr int UK = std::is_same<T, cplx>::value ? 8 : 16;   // k per unit
  constexpr int RL = 32 / UK;                                 // rows per load of a turned unit
  const int op = blockIdx.y, bl = blockIdx.z, b = b0 + bl;
  const int R = ss.R[op], lt = ss.ltr[op], Rpad = ss.RT[op] << lt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cr = (int)blockIdx.x % CS;                        // CTA of the cluster (clusters run along x)
  const int rg = (int)blockIdx.x / CS;
  if (rg * (NW / KW) * 32 >= R || bl >= ss.items[op]) return;  // uniform over the cluster
  if (CS > 1) cluster_arrive();   // before the maxima go to the other CTAs, every CTA has started
  const Src<T>& s = ss.s[op];
  const int kw = warp & (KW - 1);
  const int rbase = (rg * (NW / KW) + warp / KW) * 32;
  if (rbase >= R && CS == 1) return;   // a row group without rows: its warps share no barrier with others
  const int r = rbase + lane;
  const T* X = s.X.item(b);
  const bool live = r < R;
  const int64_t roff = live ? (int64_t)s.rmap.at(b, r) * s.rs : 0;
  const int* kidx = s.kmap.idx ? s.kmap.idx + (b % s.kmap.period) * s.kmap.len : nullptr;
  const int64_t rs = s.rs, ks = s.ks;
  const bool turn = ks == 1 && !s.rmap.idx;
  const int nu = KT * (TK / UK), step = KW * CS, u0 = cr * KW + kw;
  __shared__ uint32_t smax[NW][32];
  __shared__ uint32_t cmax[NW == 8 ? 8 : 1][NW][32];   // [CTA of the cluster][row group][row]
  __shared__ T tile[NW][32 * (UK + 1)];
  T xv[UK];
  auto load = [&](int u) {
    if (turn) {
      const int k = u * UK + (lane & (UK - 1));
      const int64_t ko = k < K ? (kidx ? (int64_t)kidx[k] : (int64_t)k) : -1;
      const T* p = X + (int64_t)(rbase + lane / UK) * rs + ko;
#pragma unroll
      for (int q = 0; q < UK; ++q) {
        const int row = rbase + q * RL + lane / UK;
        xv[q] = (ko >= 0 && row < R) ? p[(int64_t)(q * RL) * rs] : T(0.0);
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < UK; ++q) tile[warp][(q * RL + lane / UK) * (UK + 1) + (lane & (UK - 1))] = xv[q];
      __syncwarp();
#pragma unroll
      for (int c = 0; c < UK; ++c) xv[c] = tile[warp][lane * (UK + 1) + c];
    } else if (kidx) {
#pragma unroll
      for (int c = 0; c < UK; ++c) {
        const int k = u * UK + c;
        xv[c] = (live && k < K) ? X[roff + (int64_t)kidx[k] * ks] : T(0.0);
      }
    } else {
      const T* p = X + roff + (int64_t)(u * UK) * ks;
#pragma unroll
      for (int c = 0; c < UK; ++c) xv[c] = (live && u * UK + c < K) ? p[c * ks] : T(0.0);
    }
  };
  uint32_t mx = 0;
  int last = -1;   // the unit in xv
  for (int u = u0; u < nu; u += step) {
    load(last = u);
#pragma unroll
    for (int c = 0; c < UK; ++c) mx = max(mx, mag_hi(xv[c]));
  }
  smax[warp][lane] = mx;
  asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / KW), "r"(32 * KW) : "memory");   // the warps of this row group
  for (int w = 0; w < KW; ++w) mx = max(mx, smax[warp - kw + w][lane]);
  if (CS > 1) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cluster_wait();
    if (kw == 0)
      for (int d = 0; d < CS; ++d) cl.map_shared_rank(&cmax[0][0][0], d)[(cr * NW + warp) * 32 + lane] = mx;
    cl.sync();
    for (int d = 0; d < CS; ++d) mx = max(mx, cmax[d][warp - kw][lane]);
  }
  const int evm = (int)(mx >> 20);
  if (kw == 0 && cr == 0 && live) ss.ex[op][(int64_t)bl * Rpad + r] = evm;
  const int BLK = TK * 2 << lt;
  const int tl = r >> lt, rr = r & ((1 << lt) - 1);
  const int64_t rowoff = ((int64_t)bl * ss.RT[op] + tl) * KT * (int64_t)(DIG * BLK) + (rr >> 3) * 256 + (rr & 7) * 16;
  for (int u = last; u >= 0; u -= step) {
    if (u != last) load(u);
    if (!live) continue;
#pragma unroll
    for (int half = 0; half < UK / 8; ++half) {
      const int k8 = u * (UK / 8) + half;   // 8-deep k group
      const int64_t boff = rowoff + (int64_t)(k8 >> 1) * (DIG * BLK) + (k8 & 1) * 128;
      double v[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = part_of(xv[half * 8 + c], 0);
      put_digits(v, evm, ss.out[op] + boff, BLK);
      if constexpr (std::is_same<T, cplx>::value) {
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = part_of(xv[half * 8 + c], 1);
        put_digits(v, evm, ss.out2[op] + boff, BLK);
      }
    }
  }
}

__device__ __noinline__ double scale_slow(long long R, int es) { return ldexp((double)R, es); }

// R 2^es as the nearest double (ties to even), from the integer's bits;
// falls back to ldexp outside the normal range.
__device__ __forceinline__ double fixed_to_double(long long R, int es) {
  if (R == 0) return 0.0;
  const unsigned long long sgn = R < 0 ? (1ull << 63) : 0ull;
  unsigned long long a = R < 0 ? (unsigned long long)(-R) : (unsigned long long)R;
  const int lz = __clzll((long long)a);
  a <<= lz;                                    // leading one at bit 63
  unsigned long long m = a >> 11;              // 53 significant bits
  const unsigned long long rem = a & 0x7FFull;
  m += (rem > 0x400ull || (rem == 0x400ull && (m & 1ull))) ? 1ull : 0ull;
  const int e2 = es + 63 - lz;                 // value in [2^e2, 2^(e2+1))
  if (e2 + 1023 < 1 || e2 + 1023 > 2046) return scale_slow(R, es);
  // m carries the hidden bit: adding it to (exponent - 1) sets the exponent
  // (and carries once more when rounding reached 2^53)
  return __longlong_as_double((long long)(sgn | (((unsigned long long)(e2 + 1022) << 52) + m)));
}

__device__ __noinline__ double fixed_slow(long long R, int es) { return fixed_to_double(R, es); }

// R 2^(E - 1086) as a double when |R| >= 2^32 and the result is normal (the
// caller has checked both), ties to even: as fixed_to_double with one count of
// leading zeros and no range checks.  (Few bits are dropped, so ties are
// common: rounding them away from zero grew the error of the 3D builds by 30 %.)
__device__ __forceinline__ double fixed_fast(long long R, int E, uint32_t flip) {
  const uint32_t hi = (uint32_t)((unsigned long long)R >> 32);
  const uint32_t s = (uint32_t)((int)hi >> 31);
  const unsigned long long a0 = ((unsigned long long)R ^ ((unsigned long long)s << 32 | s)) + (s & 1u);
  const uint32_t ah = (uint32_t)(a0 >> 32), al = (uint32_t)a0;
  const int sh = __clz((int)ah) - 1;           // 0 .. 30; the leading one goes to bit 62
  const uint32_t sl = al << sh;
  const unsigned long long a = ((unsigned long long)__funnelshift_l(al, ah, sh) << 32 | sl) + (511u + ((sl >> 10) & 1u));
  const uint32_t nh = (uint32_t)(a >> 32), nl = (uint32_t)a;
  // 53 bits; the hidden bit adds one to the exponent field
  const uint32_t oh = (nh >> 10) + ((uint32_t)(E - 2 - sh) << 20);
  return __hiloint2double((int)(oh | ((hi ^ flip) & 0x80000000u)), (int)__funnelshift_r(nl, nh, 10));
}

// The eight diagonal sums x_D (exact floats) of one output as a fixed-point
// integer, rounded once: units of 2^{-57 + sh} (KC = 64, sh = -5 .. 0) or
// 2^{-56 + sh} (KC = 128, sh = -6 .. 6; unit = 2^-sh / 8 or / 16).  A sum below 2^22 becomes an integer with one addition (its
// bits after adding 1.5 * 2^23); a larger one is halved or quartered with
// rounding and its small remainder handed to the next diagonal, where it is
// 256 times as much and the sum stays below 2^24.  The two lowest diagonals
// and the last remainder are rounded to the unit, unbiased.
template <int KC>
__device__ __forceinline__ long long diag_fixed(const float (&x)[NDIAG], int sh, float unit) {
  constexpr float MG = 12582912.0f;            // 1.5 * 2^23
  constexpr uint32_t MB = 0x4B400000u;         // its bits
  if constexpr (KC == KC1) {
    const uint32_t a2 = __float_as_uint(x[0] + MG), a3 = __float_as_uint(x[1] + MG);
    const uint32_t a4 = __float_as_uint(x[2] + MG), a5 = __float_as_uint(x[3] + MG);
    const uint32_t a6 = __float_as_uint(x[4] + MG);
    const float h7 = fmaf(x[5], 0.5f, MG), r7 = fmaf(h7 - MG, -2.0f, x[5]);
    const float z = fmaf(r7, 256.0f, fmaf(x[7], 1.0f / 256.0f, x[6]));
    const uint32_t c = __float_as_uint(fmaf(z, unit, MG));                      // z / 8, units of 2^-57, at sh = 0
    // x6 2^13 + (x7 / 2) 2^6 + c; the offset of c's bits goes into the sum's
    const int P = (int)(a6 * 128u + __float_as_uint(h7) - (129u * MB + (MB >> (6 - sh))));
    const int Q = (int)(a4 * 256u + a5 - 257u * MB);                            // units 2^-36: 2^21
    const int S = (int)(a2 * 256u + a3 - 257u * MB);                            // units 2^-20: 2^37
    long long w = (long long)P * (1 << (6 - sh)) + (long long)(unsigned long long)c;
    w += (long long)Q * (1 << (21 - sh));
    return w + ((long long)S << (37 - sh));
  } else {
    const uint32_t a2 = __float_as_uint(x[0] + MG), a3 = __float_as_uint(x[1] + MG);
    const uint32_t a4 = __float_as_uint(x[2] + MG);
    const float h5 = fmaf(x[3], 0.5f, MG), r5 = fmaf(h5 - MG, -2.0f, x[3]);
    const float y6 = fmaf(r5, 256.0f, x[4]);
    const float h6 = fmaf(y6, 0.25f, MG), r6 = fmaf(h6 - MG, -4.0f, y6);
    const float y7 = fmaf(r6, 256.0f, x[5]);
    const float h7 = fmaf(y7, 0.25f, MG), r7 = fmaf(h7 - MG, -4.0f, y7);
    const float z = fmaf(r7, 256.0f, fmaf(x[7], 1.0f / 256.0f, x[6]));
    const uint32_t c = __float_as_uint(fmaf(z, unit, MG));                      // z / 16, units of 2^-56, at sh = 0
    // in units of 2^-56: (x6 / 4) 2^14 + (x7 / 4) 2^6 + c
    const int P = (int)(__float_as_uint(h6) * 256u + __float_as_uint(h7) - (257u * MB + (MB >> (6 - sh))));
    const int Q = (int)(a4 * 128u + __float_as_uint(h5) - 129u * MB);           // x4 2^28 + (x5 / 2) 2^21
    const int S = (int)(a2 * 256u + a3 - 257u * MB);                            // 2^36
    long long w = (long long)P * (1 << (6 - sh)) + (long long)(unsigned long long)c;
    w += (long long)Q * (1 << (21 - sh));
    return w + ((long long)S << (36 - sh));
  }
}

struct GemmP {
  const uint8_t* As;
  const uint8_t* Bs;
  // two products into the same accumulators (the two terms of one component
  // of a complex product): after the KT k steps of As Bs, KT more of
  // As2 Bs2, negated when neg2 (the operands of both share their row scales)
  const uint8_t* As2;
  const uint8_t* Bs2;
  int pair, neg2;
  const int* ea;
  const int* eb;
  int MT, NT, KT, M, N;
  int lsb;             // fraction bits of the fixed-point result
  double alpha, beta;
  long long asign;     // alpha = +-1: sign bit to flip
  // C as doubles: strides and offsets in doubles, W doubles per entry (2 for
  // complex C, whose component is part of the offset)
  BOp<double> C;
  int W;
  IMap crow;
  int b0;              // first batch item of this launch
  int a_bl, b_bl;      // 1, or 0 for an operand whose digits serve every item
  int nitems;          // batch items of this launch (tiles: MT NT nitems)
  unsigned* err;
};

// Epilogue forms: C <- +-P, C <- C +- P, or alpha P + beta C.  Kept apart:
// FP64 instructions of a form not taken still cost the FP64 pipe its cycles
// when the compiler predicates them.
enum { TC_SET = 0, TC_ADD = 1, TC_GENERAL = 2 };

// What bounds it: at long K the tensor pipe (36 products of 128 x TN x 16 per
// k step), at short K the epilogue: one FP64 addition per output (2 per
// clock and SM) and ~60 other instructions.  Sixteen epilogue warps of at
// most 112 registers keep four warps on each scheduler (eight warps of 167
// registers issued in 27 % of the cycles).
template <int EPI, bool TRANS, int TN, int KC>
__global__ void __launch_bounds__(THREADS, 1) k_gemm_tc(GemmP g) {
  // Persistent: CTA c takes the tiles c, c + gridDim.x, ... of the launch
  // (tile t = item t / (MT NT), then row tile, then column tile), so that the
  // next tile's copies and products overlap this tile's epilogue and the
  // TMEM allocation and barrier set-up happen once per CTA.  The stage ring,
  // the accumulator hand-over (acc_full / acc_empty) and their phases run on
  // across tiles.
  constexpr int NST = stages(TN, TRANS), STAGE = stage_bytes(TN), BBLK = bblk(TN), BSTG = bstg(TN);
  constexpr int NSET = accum_sets(TN);      // accumulator sets taken in turn
  constexpr int QGRP = 256 / TN;            // B digits stacked into one MMA (N <= 256)
  constexpr int ECOLS = TN / 4;             // columns per epilogue warp
  constexpr int KCT = KC2 / TK;             // k steps per chunk (a KC = 64 tile has one chunk)
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[NST], empty[NST], acc_full[NSET], acc_empty[NSET];
  __shared__ uint32_t tslot;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_item = g.MT * g.NT;
  const int ntiles = tiles_item * g.nitems;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tslot)), "n"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 32) {
    for (int i = 0; i < NST; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&empty[i])));
    }
    for (int i = 0; i < NSET; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&acc_full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&acc_empty[i])), "n"(EPI_WARPS));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    abort_flag = 0;
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  volatile int* abrt = &abort_flag;
  const int KTV = g.pair ? 2 * g.KT : g.KT;   // k steps of a tile (both products of a pair)
  const int nchunk = KC == KC1 ? 1 : (KTV + KCT - 1) / KCT;
  const uint32_t sbase = su32(smem);

  if (warp == EPI_WARPS) {
    // producer: one bulk copy per operand per k step, the ring running on
    // across tiles
    if (lane == 0) {
      long it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int bl = t / tiles_item, rem = t % tiles_item;
        const int mt = rem % g.MT, nt = rem / g.MT;
        const int64_t a_off = ((int64_t)(bl * g.a_bl) * g.MT + mt) * g.KT * (int64_t)ASTG;
        const int64_t b_off = ((int64_t)(bl * g.b_bl) * g.NT + nt) * g.KT * (int64_t)BSTG;
        for (int vk = 0; vk < KTV; ++vk, ++it) {
          const bool second = vk >= g.KT;
          const int k = second ? vk - g.KT : vk;
          const uint8_t* a_src = (second ? g.As2 : g.As) + a_off;
          const uint8_t* b_src = (second ? g.Bs2 : g.Bs) + b_off;
          const int s = (int)(it % NST);
          if (it >= NST && !mbar_wait(su32(&empty[s]), (int)((it / NST) & 1) ^ 1, abrt)) {
            ok = false;
            break;
          }
          const uint32_t fb = su32(&full[s]), dst = sbase + s * STAGE;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(STAGE) : "memory");
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                       ::"r"(dst), "l"(a_src + (int64_t)k * ASTG), "r"(ASTG), "r"(fb) : "memory");
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                       ::"r"(dst + ASTG), "l"(b_src + (int64_t)k * BSTG), "r"(BSTG), "r"(fb) : "memory");
        }
      }
      if (!ok) {
        *abrt = 1;
        atomicOr(g.err, DEV_ERR_TIMEOUT);
      }
    }
  } else if (warp == EPI_WARPS + 1) {
    // MMA issue: 36 digit-pair products per k step into the 8 diagonal accumulators
    if (lane == 0) {
      // B's digit blocks lie one after another with the same row-group stride,
      // so digits q0 .. q0+n-1 form one operand of n * TN rows, and A_p times
      // it lands in the accumulators of diagonals p+q0 .. p+q0+n-1, which are
      // adjacent in TMEM: one MMA (N <= 256) per (p, group of <= QGRP digits).
      // Instruction descriptor: fp32 accumulator, A and B fp16, K-major.
      const uint32_t idesc0 = (1u << 4) | ((uint32_t)(TM >> 4) << 24);
      long it = 0, cc = 0;   // k steps and accumulator chunks issued so far
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int kk = 0;
        for (int c = 0; c < nchunk && ok; ++c, ++cc) {
          const int set = (int)(cc % NSET);
          const uint32_t tset = tmem + (uint32_t)(set * NDIAG * TN);
          // the epilogue has read this set's previous chunk
          if (cc >= NSET && !mbar_wait(su32(&acc_empty[set]), (int)((cc / NSET) & 1) ^ 1, abrt)) { ok = false; break; }
          fence_after();
          const int kend = KC == KC1 ? KTV : min(KTV, (c + 1) * KCT);
          const int kbeg = kk;
          for (; kk < kend; ++kk, ++it) {
            const int s = (int)(it % NST);
            if (!mbar_wait(su32(&full[s]), (int)((it / NST) & 1), abrt)) { ok = false; break; }
            fence_after();
            const uint32_t a0 = sbase + s * STAGE, b0 = a0 + ASTG;
            // the second product of a pair enters negated: negate-B bit of the
            // instruction descriptor
            const uint32_t ineg = (g.neg2 && kk >= g.KT) ? (1u << 14) : 0u;
#pragma unroll
            for (int p = 0; p < DIG; ++p) {
              const uint64_t ad = sdesc(a0 + p * ABLK, 128, 256);
              const int nq_all = DSUM - 1 - p;   // q = 0 .. nq_all-1
#pragma unroll
              for (int q0 = 0; q0 < nq_all; q0 += QGRP) {
                const int nq = (nq_all - q0) < QGRP ? (nq_all - q0) : QGRP;
                // the first k step of a chunk overwrites: p = 0 covers every diagonal once
                const uint32_t acc = (kk != kbeg || p != 0) ? 1u : 0u;
                const uint64_t bd = sdesc(b0 + q0 * BBLK, 128, 256);
                const uint32_t idesc = idesc0 | ineg | ((uint32_t)((nq * TN) >> 3) << 17);
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tset + (uint32_t)((p + q0) * TN)),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
              }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             su32(&empty[s]))
                         : "memory");
          }
          if (!ok) break;
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           su32(&acc_full[set]))
                       : "memory");
        }
      }
      if (!ok) {
        *abrt = 1;
        atomicOr(g.err, DEV_ERR_TIMEOUT);
      }
    }
  } else {
    // epilogue: warp w reads TMEM lane quarter w % 4 (its rows) and columns
    // (w / 4) ECOLS ..; thread = row.  A normal tile's rows are C's rows, so
    // its accesses are coalesced as they are; a transposed tile's rows are C's
    // columns: the warp's results pass through its own block of shared memory
    // and leave with the tile column (C's row) fastest.  No barrier between
    // the epilogue warps; a warp none of whose rows or columns exist only
    // waits and arrives.  After a wait gives up (agreed over the warp) it
    // skips the remaining waits and stores.
    const int quarter = warp & 3, c0 = (warp >> 2) * ECOLS;
    double* s_c = reinterpret_cast<double*>(smem + NST * STAGE) + warp * 32 * (ECOLS + 1);
    // TN = 32: the old C values of the next tile are copied into this thread's
    // slots of shared memory while this tile is converted
    double* s_old = reinterpret_cast<double*>(smem + NST * STAGE + trans_bytes(TN, TRANS)) + (warp * 32 + lane) * 1;
    constexpr bool STAGED = TN == 32 && EPI != TC_SET;
    constexpr int OSET = EPI_WARPS * 32 * ECOLS;   // doubles per staged tile
    constexpr int RSTEP = 32 / ECOLS;         // transposed: C columns per store
    const uint32_t flip = (uint32_t)((unsigned long long)g.asign >> 32);
    constexpr int LSBC = KC == KC1 ? LSB1 : LSB2;
    const int sh = min(LSBC - g.lsb, 6), sh2 = LSBC - g.lsb - sh;   // unit of a chunk, rest beyond 6 bits
    const float unit = __int_as_float((127 - (KC == KC1 ? 3 : 4) - sh) << 23);   // 2^-sh / 8, / 16
    struct Tile {
      double* Cp;          // this thread's first C entry (normal: its tile row; transposed: its tile column's row)
      int ebase, eb;       // exponent of its row (with the fixed point's), of column `lane`
      int nrow, ncol;      // rows and columns of this warp that exist (<= 0: none)
      bool safe;           // every exponent is far from the ends of the range
    };
    const int64_t cstep = (int64_t)g.C.ld * g.W * (TRANS ? RSTEP : 1);
    // entry jj of this thread exists
    auto live = [&](const Tile& q, int jj) {
      return TRANS ? (lane % ECOLS < q.ncol && jj * RSTEP + lane / ECOLS < q.nrow) : (lane < q.nrow && jj < q.ncol);
    };
    auto setup = [&](int t, int buf) {
      Tile q;
      const int bl = t / tiles_item, rem = t % tiles_item;
      const int mt = rem % g.MT, nt = rem / g.MT;
      const int i0 = mt * TM + quarter * 32, j0 = nt * TN + c0;
      q.nrow = min(32, g.M - i0);
      q.ncol = min(ECOLS, g.N - j0);
      q.Cp = nullptr;
      q.ebase = q.eb = 0;
      q.safe = true;
      if (q.nrow > 0 && q.ncol > 0) {
        const int b = g.b0 + bl;
        const int crw = TRANS ? j0 + lane % ECOLS : i0 + lane;
        const int ccl = TRANS ? i0 + lane / ECOLS : j0;
        const bool in = crw < (TRANS ? g.N : g.M);
        int er = 0;
        if (lane < q.nrow) er = row_exp(g.ea[(int64_t)(bl * g.a_bl) * g.MT * TM + i0 + lane]);
        if (lane < q.ncol) q.eb = row_exp(g.eb[(int64_t)(bl * g.b_bl) * g.NT * TN + j0 + lane]);
        q.Cp = g.C.item(b) + ((int64_t)(in ? g.crow.at(b, crw) : 0) + (int64_t)ccl * g.C.ld) * g.W;
        if constexpr (STAGED) {
#pragma unroll
          for (int jj = 0; jj < ECOLS; ++jj)
            if (live(q, jj))
              asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(su32(s_old + buf * OSET + jj * (EPI_WARPS * 32))),
                           "l"(q.Cp + cstep * jj) : "memory");
        } else if constexpr (EPI != TC_SET && KC != KC1) {
#pragma unroll
          for (int jj = 0; jj < ECOLS; ++jj)
            if (live(q, jj)) asm volatile("prefetch.global.L2 [%0];" ::"l"(q.Cp + cstep * jj));
        }
        q.safe = __all_sync(0xffffffffu, abs(er) <= 400 && abs(q.eb) <= 400);
        q.ebase = er - g.lsb + 1086;
      }
      if constexpr (STAGED) asm volatile("cp.async.commit_group;" ::: "memory");
      return q;
    };
    bool ok = true;
    long cc = 0;   // accumulator chunks consumed so far
    int buf = 0;
    constexpr bool AHEAD = TN == 32;   // the next tile's addresses, exponents and copies a tile ahead
    Tile nx;
    if (AHEAD && (int)blockIdx.x < ntiles) nx = setup(blockIdx.x, 0);
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, buf ^= 1) {
      const Tile q = AHEAD ? nx : setup(t, 0);
      const bool any = q.nrow > 0 && q.ncol > 0;   // this warp has outputs
      const bool more = t + (int)gridDim.x < ntiles;
      if (AHEAD && more) nx = setup(t + gridDim.x, buf ^ 1);
      double cold[STAGED || EPI == TC_SET ? 1 : ECOLS];
      auto load_old = [&]() {
        if constexpr (!STAGED && EPI != TC_SET) {
#pragma unroll
          for (int jj = 0; jj < ECOLS; ++jj) cold[jj] = live(q, jj) ? q.Cp[cstep * jj] : 0.0;
        }
      };
      auto old_c = [&](int jj) { return STAGED ? s_old[buf * OSET + jj * (EPI_WARPS * 32)] : cold[STAGED ? 0 : jj]; };
      auto finish = [&](double val, int jj) {
        if constexpr (EPI == TC_SET) return val;
        else if constexpr (EPI == TC_ADD) return old_c(jj) + val;
        else return fma(g.alpha, val, g.beta == 0.0 ? 0.0 : g.beta * old_c(jj));
      };
      // four adjacent results.  |R| below 2^32 (zeros among them) and extreme
      // exponents take the general form, all lanes together
      auto convert4 = [&](const long long (&R)[4], int jb) {
        bool fast = q.safe;
#pragma unroll
        for (int j = 0; j < 4; ++j) fast = fast && (uint32_t)((unsigned long long)R[j] >> 32) + 1u > 1u;
        fast = __all_sync(0xffffffffu, fast || lane >= q.nrow);
        double val[4];
        if (fast) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            val[j] = fixed_fast(R[j], q.ebase + __shfl_sync(0xffffffffu, q.eb, jb + j), EPI == TC_GENERAL ? 0u : flip);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            val[j] = fixed_slow(R[j], q.ebase - 1086 + __shfl_sync(0xffffffffu, q.eb, jb + j));
            if (EPI != TC_GENERAL) val[j] = __longlong_as_double(__double_as_longlong(val[j]) ^ g.asign);
          }
        }
        if constexpr (TRANS) {
#pragma unroll
          for (int j = 0; j < 4; ++j) s_c[lane * (ECOLS + 1) + jb + j] = val[j];
        } else if (lane < q.nrow) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (jb + j < q.ncol) q.Cp[cstep * (jb + j)] = finish(val[j], jb + j);
        }
      };
      auto old_ready = [&]() {
        if constexpr (STAGED) {   // this tile's copies: all but the group of the next tile
          if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
          else asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
      };
      if (KC == KC1 && any && ok) load_old();   // arrive while the products finish
      long long R[ECOLS / 4][4];
      for (int c = 0; c < nchunk; ++c, ++cc) {
        if (!ok) continue;
        const int set = (int)(cc % NSET);
        ok = __all_sync(0xffffffffu, mbar_wait(su32(&acc_full[set]), (int)((cc / NSET) & 1), abrt));
        if (!ok) continue;
        fence_after();
        if (any) {
          if (KC == KC1 && !TRANS) old_ready();
          const uint32_t ta0 = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(set * NDIAG * TN + c0);
#pragma unroll
          for (int cg = 0; cg < ECOLS / 4; ++cg) {
            uint32_t v[NDIAG][4];
#pragma unroll
            for (int di = 0; di < NDIAG; ++di)
              asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(v[di][0]), "=r"(v[di][1]), "=r"(v[di][2]), "=r"(v[di][3])
                           : "r"(ta0 + (uint32_t)(di * TN + cg * 4)));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (cg == ECOLS / 4 - 1) {
              fence_before();
              __syncwarp();
              if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&acc_empty[set])) : "memory");
            }
            long long w4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              float x[NDIAG];
#pragma unroll
              for (int di = 0; di < NDIAG; ++di) x[di] = __uint_as_float(v[di][j]);
              w4[j] = diag_fixed<KC>(x, sh, unit);
            }
            if constexpr (KC == KC1) {
              convert4(w4, cg * 4);
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                long long w = w4[j];
                if (sh2 > 0) w = (w + (1ll << (sh2 - 1)) - ((~w >> sh2) & 1)) >> sh2;   // ties to even
                R[cg][j] = c == 0 ? w : R[cg][j] + w;
              }
            }
          }
        } else {
          fence_before();
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&acc_empty[set])) : "memory");
        }
      }
      if (!any || !ok) continue;
      if constexpr (KC != KC1) {
        load_old();
        if (!TRANS) old_ready();
#pragma unroll
        for (int cg = 0; cg < ECOLS / 4; ++cg) convert4(R[cg], cg * 4);
      }
      if constexpr (TRANS) {
        old_ready();
        __syncwarp();
#pragma unroll
        for (int jj = 0; jj < ECOLS; ++jj)
          if (live(q, jj)) q.Cp[cstep * jj] = finish(s_c[(jj * RSTEP + lane / ECOLS) * (ECOLS + 1) + lane % ECOLS], jj);
        __syncwarp();   // read before the next tile's results overwrite it
      }
    }
    if constexpr (STAGED) asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok && lane == 0) {
      *abrt = 1;
      atomicOr(g.err, DEV_ERR_TIMEOUT);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
}

// digit pairs (p, q), 1 <= p, q <= DIG, with p + q <= DSUM
constexpr int npairs() {
  int n = 0;
  for (int p = 1; p <= DIG; ++p)
    for (int q = 1; q <= DIG; ++q) n += (p + q <= DSUM) ? 1 : 0;
  return n;
}
static_assert(npairs() == 36, "digit pair count");
static_assert(DIG == 8 && BITS == 8 && FRAC == 62, "the slicing takes the bytes of a 64-bit integer");

int ceil_log2(int64_t x) {
  int c = 0;
  while ((int64_t(1) << c) < x) ++c;
  return c;
}

template <int EPI, bool TRANS, int TN, int KC>
cudaError_t launch(const GemmP& p, int grid, cudaStream_t st) {
  constexpr int SM = smem_bytes(TN, TRANS);
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_gemm_tc<EPI, TRANS, TN, KC>, cudaFuncAttributeMaxDynamicSharedMemorySize, SM);
  if (attr != cudaSuccess) return attr;
  k_gemm_tc<EPI, TRANS, TN, KC><<<grid, THREADS, SM, st>>>(p);
  return cudaGetLastError();
}

template <int EPI, bool TRANS, int TN>
cudaError_t launch_kc(const GemmP& p, int kc, int grid, cudaStream_t st) {
  return kc == KC1 ? launch<EPI, TRANS, TN, KC1>(p, grid, st) : launch<EPI, TRANS, TN, KC2>(p, grid, st);
}

template <int EPI, bool TRANS>
cudaError_t launch_tn(const GemmP& p, int tn, int kc, int grid, cudaStream_t st) {
  // the general alpha / beta form is not on the build's path: one tile shape
  // and chunk serve it
  if constexpr (EPI == TC_GENERAL) return launch<EPI, TRANS, 64, KC2>(p, grid, st);
  else return tn == 64 ? launch_kc<EPI, TRANS, 64>(p, kc, grid, st) : launch_kc<EPI, TRANS, 32>(p, kc, grid, st);
}

struct Sizes {
  int MT, NT, KT;
  size_t a_item, b_item, ea_item, eb_item;
};

Sizes sizes(int M, int N, int K, int tn) {
  Sizes z;
  z.MT = (M + TM - 1) / TM;
  z.NT = (N + tn - 1) / tn;
  z.KT = (K + TK - 1) / TK;
  z.a_item = (size_t)z.MT * z.KT * ASTG;
  z.b_item = (size_t)z.NT * z.KT * bstg(tn);
  z.ea_item = (size_t)z.MT * TM * sizeof(int);
  z.eb_item = (size_t)z.NT * tn * sizeof(int);
  return z;
}

constexpr size_t WS_CAP = size_t(1) << 30;  // workspace bytes a launch group may use

}  // namespace tc

TcWorkspace*& tc_workspace() {
  static thread_local TcWorkspace* w = nullptr;
  return w;
}

size_t tc_workspace_cap() { return tc::WS_CAP; }

void tc_release(TcWorkspace* w) {
  if (w && w->p) dev_free(w->p, w->st);
  if (w) { w->p = nullptr; w->bytes = 0; }
}

// Fraction of the output tiles that holds the product, in the better of the
// two orientations and tile widths.
static double tile_fill(int M, int N) {
  using namespace tc;
  auto padded = [](int n, int t) { return (double)((n + t - 1) / t) * t; };
  return (double)M * N / std::min(padded(M, TM) * padded(N, 32), padded(N, TM) * padded(M, 32));
}

// At most 8 rows against many columns and a long inner dimension.
static bool few_rows_long_k(int M, int N, int K) { return M <= 8 && N >= 32 && K >= 32; }

template <typename T>
bool tc_applicable(const GemmArgs<T>& g) {
  const TcWorkspace* w = tc_workspace();
  if (!w || !w->enabled || !w->err_slot || !*w->err_slot || g.ta || g.K > (1 << 20)) return false;
  if (w->force) return true;
  // one side of at least 32 and the other of at least 16: the short side
  // goes to the narrow tile dimension (transposed tiling when M is short)
  if (std::min(g.M, g.N) < 1 || std::max(g.M, g.N) < 32 || g.K < 16) return false;
  if (std::min(g.M, g.N) < 16 && !few_rows_long_k(g.M, g.N, g.K)) return false;
  // a side below 32 leaves even the 32-wide tile side part empty: such
  // products go to the tensor cores only while the tiles stay over ~28 % full
  // (measured: 28 x 113 gains there, 28 x 57 loses) -- except products of
  // at most 8 rows, N >= 32 and K >= 32, which half-empty FP64-pipe tiles run
  // at under half their rate (4 x 114 x 64 complex, 4096 items: 1.4 ms of 0.6);
  // few columns stay on the FP64 pipe's skinny kernels
  if (std::min(g.M, g.N) < 32 && tile_fill(g.M, g.N) < 0.28 && !few_rows_long_k(g.M, g.N, g.K)) return false;
  // short inner dimensions: eight accumulators per output are read back for
  // little work, so small items stay on the FP64 pipe
  if (g.K < lu_tune(TUNE_TC_MIN_K) && (g.M < 512 || g.N < 512)) return false;
  if ((double)g.M * g.N * g.K * g.batch < 1.0e5 * lu_tune(TUNE_TC_MIN_WORK_REAL)) return false;
  return true;
}

template <>
bool tc_applicable<cplx>(const GemmArgs<cplx>& g) {
  const TcWorkspace* w = tc_workspace();
  if (!w || !w->enabled || !w->err_slot || !*w->err_slot || g.ta || g.K > (1 << 20)) return false;
  if (g.alpha.im != 0.0 || g.beta.im != 0.0) return false;
  if (w->force) return true;
  if (std::min(g.M, g.N) < 1 || std::max(g.M, g.N) < 32 || g.K < 16) return false;
  if (std::min(g.M, g.N) < 16 && !few_rows_long_k(g.M, g.N, g.K)) return false;
  if (std::min(g.M, g.N) < 32 && tile_fill(g.M, g.N) < 0.28 && !few_rows_long_k(g.M, g.N, g.K)) return false;
  if (g.K < lu_tune(TUNE_TC_MIN_K) && (g.M < 512 || g.N < 512)) return false;
  if ((double)g.M * g.N * g.K * g.batch < 1.0e5 * lu_tune(TUNE_TC_MIN_WORK_CPLX)) return false;
  return true;
}

namespace {

// Orientation and width of the output tiles: C = A B in 128 x TN tiles of C
// (TN columns), or C^T = B^T A^T in 128 x TN tiles of C^T (TN of C's rows).
struct Tiling {
  bool trans;
  int tn;
};

// The choice with the least estimated time: waves of tiles over the SMs (one
// CTA each) times a tile's cycles, the largest of its digit products (measured
// 1840 per k step at TN = 64 and 1300 at 32, where L2 delivers about 30 bytes
// per clock to each SM; with one accumulator set, TN = 64, a third of the
// epilogue per chunk comes on top), its epilogue (by its average number of
// outputs) and its traffic (digits, and C at about 12 bytes per clock and SM
// when all SMs stream: 164 x 164 x 32, 4096 items, 773 us at TN = 64 and
// 1135 us at 32), so that few-row products (the 32-row updates of the
// recursive LU and triangular solves) fill their tiles and small grids spread
// over more SMs.
Tiling choose_tiling(int M, int N, int K, int batch, bool pair) {
  using namespace tc;
  const int64_t sms = device_sms();
  const double kt = (double)((K + TK - 1) / TK) * (pair ? 2 : 1);
  Tiling best{false, 64};
  double bt = -1.0;
  for (int trans = 0; trans < 2; ++trans)
    for (int tn = 64; tn >= 32; tn -= 32) {
      const int64_t r = trans ? N : M, c = trans ? M : N;
      const int64_t rt = (r + TM - 1) / TM, ct = (c + tn - 1) / tn;
      const double waves = (double)((rt * ct * batch + sms - 1) / sms);
      const double outs = (double)r * c / ((double)rt * ct);
      const double epi = (600.0 + 0.55 * outs) * (trans ? 1.15 : 1.0);
      const double chunks = kt * TK <= KC1 ? 1.0 : std::ceil(kt * TK / KC2);
      const double prod = tn == 64 ? 1840.0 * kt + 0.33 * epi * chunks : 1300.0 * kt;
      const double traffic = kt * (ASTG + bstg(tn)) / 30.0 + 16.0 * outs / 12.0;
      const double tile = std::max(std::max(prod, epi), traffic);
      const double t = waves * tile + prod + epi;
      if (bt < 0.0 || t < 0.98 * bt) {
        bt = t;
        best = Tiling{trans != 0, tn};
      }
    }
  return best;
}

cudaError_t ensure_ws(TcWorkspace* w, size_t bytes, cudaStream_t st) {
  if (w->bytes >= bytes) {
    if (w->st != st && w->p) {
      // the buffer moves to another stream: order it after its last use
      cudaError_t e = cudaStreamSynchronize(w->st);
      if (e != cudaSuccess) return e;
      w->st = st;
    }
    return cudaSuccess;
  }
  if (w->p) {
    cudaError_t e = cudaStreamSynchronize(w->st);
    if (e != cudaSuccess) return e;
    dev_free(w->p, st);
    w->p = nullptr;
    w->bytes = 0;
  }
  const size_t nb = std::max(bytes, (size_t)64 << 20);
  cudaError_t e = dev_malloc(&w->p, nb, st);
  if (e != cudaSuccess) { w->p = nullptr; return e; }
  w->bytes = nb;
  w->st = st;
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_split(const tc::SplitSet<T>& ss, int nops, int K, int KT, int b0, int nb, cudaStream_t st, Prof* pf) {
  int rmax = 0;
  for (int o = 0; o < nops; ++o) rmax = std::max(rmax, ss.R[o]);
  if (pf) {
    pf->begin(st);
    pf->note(rmax, nops, K, nb);
  }
  // warps along k: a power of two, at most 8 and no more than units of k;
  // CTAs of a cluster along k while the warps have several units each and
  // the grid leaves SMs idle
  const int nu = KT * (std::is_same<T, cplx>::value ? 2 : 1);
  int kw = 1;
  while (kw < 8 && kw < nu) kw *= 2;
  const int nw = kw <= 4 ? 4 : 8;
  const int rows = 32 * (nw / kw);
  const int64_t ctas = (int64_t)((rmax + rows - 1) / rows) * nops * nb;
  int cs = 1;
  while (nw == 8 && cs < 8 && nu > kw * cs && ctas * cs < 4 * device_sms()) cs *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((rmax + rows - 1) / rows * cs, nops, nb);
  cfg.blockDim = dim3(32 * nw);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cs > 1 ? 1 : 0;
  const cudaError_t e = nw == 8 ? cudaLaunchKernelEx(&cfg, tc::k_split<T, 8>, ss, K, KT, b0, kw, cs)
                                : cudaLaunchKernelEx(&cfg, tc::k_split<T, 4>, ss, K, KT, b0, kw, cs);
  if (pf) pf->end(K_SPLIT, 0.0, st);
  return e;
}

cudaError_t launch_mma(const tc::GemmP& p, const Tiling& tl, int kc, int nb, int M, int N, int K, int sms,
                       cudaStream_t st, Prof* pf) {
  using namespace tc;
  if (pf) {
    pf->begin(st);
    pf->note(M, N, K, nb);
  }
  // persistent (from the tuned inner dimension on): at most one CTA per SM,
  // which the shared-memory ring and the TMEM accumulators allow anyway; else
  // one CTA per tile
  const int64_t ntiles = (int64_t)p.MT * p.NT * nb;
  const bool persist = K >= lu_tune(TUNE_TC_PERSIST_MIN_K);
  const int grid = (int)(persist ? std::min<int64_t>(ntiles, sms) : ntiles);
  const bool unit = p.alpha == 1.0 || p.alpha == -1.0;
  const int epi = unit && p.beta == 0.0 ? TC_SET : unit && p.beta == 1.0 ? TC_ADD : TC_GENERAL;
  cudaError_t e;
  if (epi == TC_SET) e = tl.trans ? launch_tn<TC_SET, true>(p, tl.tn, kc, grid, st) : launch_tn<TC_SET, false>(p, tl.tn, kc, grid, st);
  else if (epi == TC_ADD) e = tl.trans ? launch_tn<TC_ADD, true>(p, tl.tn, kc, grid, st) : launch_tn<TC_ADD, false>(p, tl.tn, kc, grid, st);
  else e = tl.trans ? launch_tn<TC_GENERAL, true>(p, 64, KC2, grid, st) : launch_tn<TC_GENERAL, false>(p, 64, KC2, grid, st);
  // executed: fp16 tensor-core flops of the digit products over the padded
  // tiles; algorithmic: 2 M N K per real product (a pair holds two)
  const double nprod = p.pair ? 2.0 : 1.0;
  const double exec = 2.0 * npairs() * nprod * (double)p.MT * TM * (double)p.NT * tl.tn * (double)p.KT * TK * nb;
  if (pf) pf->end(K_GEMM_TC, 2.0 * nprod * M * (double)N * K * nb, st, exec);
  return e;
}

}  // namespace

// An operand is the same matrix for every batch item when its items share
// one base and its index maps do not depend on the item (the leaf stage's
// Q and QH, for instance): its digits are then cut once and serve all items.
template <typename T>
bool shared_operand(const BOp<T>& X, const IMap& r, const IMap& k) {
  return !X.ptrs && X.stride == 0 && (X.div == 1 || X.sub == 0) && (!r.idx || r.period == 1) &&
         (!k.idx || k.period == 1);
}

template <typename T>
cudaError_t gemm_tc(const GemmArgs<T>& g, cudaStream_t st, Prof* pf) {
  using namespace tc;
  constexpr int NP = std::is_same<T, cplx>::value ? 2 : 1;
  TcWorkspace* w = tc_workspace();
  double alpha, beta;
  if constexpr (NP == 2) { alpha = g.alpha.re; beta = g.beta.re; }
  else { alpha = g.alpha; beta = g.beta; }
  Tiling tl = choose_tiling(g.M, g.N, g.K, g.batch, NP == 2);
  const bool general = (alpha != 1.0 && alpha != -1.0) || (beta != 0.0 && beta != 1.0);
  if (general) tl.tn = 64;   // the general form's tiles
  const bool tr = tl.trans;
  // rows of the A slot (the 128-row tiles) and of the B slot (TN-row tiles)
  const int Ma = tr ? g.N : g.M, Nb = tr ? g.M : g.N;
  const Sizes z = sizes(Ma, Nb, g.K, tl.tn);
  const bool shA = g.batch > 1 && shared_operand(g.A, g.arow, g.acol);
  const bool shB = g.batch > 1 && shared_operand(g.B, g.brow, IMap());
  const bool shSa = tr ? shB : shA, shSb = tr ? shA : shB;   // per slot
  // per item and slot: NP digit arrays and one exponent array (the parts of
  // a complex row share their scale)
  const size_t a_sz = NP * z.a_item + z.ea_item, b_sz = NP * z.b_item + z.eb_item;
  const size_t fixed = (shSa ? a_sz : 0) + (shSb ? b_sz : 0);
  const size_t per_item = std::max<size_t>((shSa ? 0 : a_sz) + (shSb ? 0 : b_sz), 1);
  // batch items per launch group: their digit slices stay within the cap
  // (small enough and they are still in L2 when the products read them)
  const size_t cap = std::min<size_t>(WS_CAP, (size_t)std::max(lu_tune(TUNE_TC_CHUNK_MB), 1) << 20);
  const size_t room = cap > fixed ? cap - fixed : 0;
  const int nb_max = (int)std::max<size_t>(1, std::min<size_t>(std::min(g.batch, 65535 / 2), room / per_item));
  const size_t na = shSa ? 1 : (size_t)nb_max, nbb = shSb ? 1 : (size_t)nb_max;
  cudaError_t e = ensure_ws(w, a_sz * na + b_sz * nbb, st);
  if (e != cudaSuccess) return e;
  uint8_t* base = static_cast<uint8_t*>(w->p);
  uint8_t* As[2] = {nullptr, nullptr};   // digits of the A slot, per real part
  uint8_t* Bs[2] = {nullptr, nullptr};
  int* ea;
  int* eb;
  {
    uint8_t* q = base;
    for (int pt = 0; pt < NP; ++pt) {
      As[pt] = q; q += z.a_item * na;
      Bs[pt] = q; q += z.b_item * nbb;
    }
    ea = reinterpret_cast<int*>(q); q += z.ea_item * na;
    eb = reinterpret_cast<int*>(q); q += z.eb_item * nbb;
  }
  // chunk and fixed-point fraction bits, by the products summed per output (a
  // complex component sums 2K; the padding of K adds zeros): scaled entries stay
  // below 1 - 2^-54, so the sum below 2^63 units with room for the chunks'
  // roundings up to 2^17 terms.  A fixed 57 or 56 bits up to 64 or 128 terms, as
  // once here, lost up to five bits of short sums that cancel.
  const int ksum = NP * z.KT * TK;
  const int kc = ksum <= KC1 && !general ? KC1 : KC2;
  const int lsb = std::min(LSB_MAX, (ksum <= 1 << 17 ? 63 : 62) - ceil_log2((int64_t)NP * g.K));
  for (int b0 = 0; b0 < g.batch; b0 += nb_max) {
    const int nb = std::min(nb_max, g.batch - b0);
    SplitSet<T> ss;
    // A (M x K) and B^T (N x K) as row sources
    Src<T> sa;
    sa.X = g.A; sa.rmap = g.arow; sa.kmap = g.acol; sa.rs = 1; sa.ks = g.A.ld;
    Src<T> sb;
    sb.X = g.B; sb.kmap = g.brow; sb.rs = g.B.ld; sb.ks = 1;
    ss.s[0] = tr ? sb : sa; ss.R[0] = Ma; ss.ltr[0] = 7; ss.RT[0] = z.MT;
    ss.out[0] = As[0]; ss.out2[0] = As[1]; ss.ex[0] = ea;
    ss.items[0] = (shSa && b0 > 0) ? 0 : (shSa ? 1 : nb);  // a shared operand is cut once per call
    ss.s[1] = tr ? sa : sb; ss.R[1] = Nb; ss.ltr[1] = tl.tn == 64 ? 6 : 5; ss.RT[1] = z.NT;
    ss.out[1] = Bs[0]; ss.out2[1] = Bs[1]; ss.ex[1] = eb;
    ss.items[1] = (shSb && b0 > 0) ? 0 : (shSb ? 1 : nb);
    if ((e = launch_split<T>(ss, 2, g.K, z.KT, b0, nb, st, pf)) != cudaSuccess) return e;
    GemmP p;
    p.MT = z.MT; p.NT = z.NT; p.KT = z.KT; p.M = Ma; p.N = Nb; p.lsb = lsb;
    p.crow = g.crow; p.b0 = b0; p.err = *w->err_slot;
    p.W = NP;
    p.C.ptrs = reinterpret_cast<double* const*>(g.C.ptrs);
    p.C.base = reinterpret_cast<double*>(g.C.base);
    p.C.stride = NP * g.C.stride; p.C.sub = NP * g.C.sub; p.C.off = NP * g.C.off;
    p.C.ld = g.C.ld; p.C.div = g.C.div;
    p.a_bl = shSa ? 0 : 1;
    p.b_bl = shSb ? 0 : 1;
    p.nitems = nb;
    p.ea = ea; p.eb = eb;
    p.alpha = alpha;
    p.beta = beta;
    p.asign = alpha == -1.0 ? (long long)(1ull << 63) : 0ll;
    if constexpr (NP == 1) {
      p.As = As[0]; p.Bs = Bs[0];
      p.As2 = nullptr; p.Bs2 = nullptr; p.pair = 0; p.neg2 = 0;
      if ((e = launch_mma(p, tl, kc, nb, g.M, g.N, g.K, device_sms() - g.spare_sms, st, pf)) != cudaSuccess) return e;
    } else {
      // complex (real alpha, beta), each component one launch of two
      // products into the same accumulators:
      //   C.re = alpha (Ar Br - Ai Bi) + beta C.re,  C.im = alpha (Ar Bi + Ai Br) + beta C.im
      // (transposed, the A slot holds B's parts and the B slot A's)
      uint8_t* const* Ap = tr ? Bs : As;   // digits of A's parts
      uint8_t* const* Bp = tr ? As : Bs;   // digits of B's parts
      auto slots = [&](int a_part, int b_part, const uint8_t*& sa_d, const uint8_t*& sb_d) {
        sa_d = tr ? Bp[b_part] : Ap[a_part];
        sb_d = tr ? Ap[a_part] : Bp[b_part];
      };
      p.pair = 1;
      slots(0, 0, p.As, p.Bs);
      slots(1, 1, p.As2, p.Bs2);
      p.neg2 = 1;
      if ((e = launch_mma(p, tl, kc, nb, g.M, g.N, g.K, device_sms() - g.spare_sms, st, pf)) != cudaSuccess) return e;
      slots(0, 1, p.As, p.Bs);
      slots(1, 0, p.As2, p.Bs2);
      p.neg2 = 0;
      p.C.off += 1;   // the imaginary component
      if ((e = launch_mma(p, tl, kc, nb, g.M, g.N, g.K, device_sms() - g.spare_sms, st, pf)) != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

// Bounded-wait check (hps_debug_wait_timeout, which 2): one CTA waits with
// the pipeline's mbarrier wait on phase 0 of a barrier that expects one
// arrival; nothing arrives unless `satisfied`.  A wait that gives up sets
// DEV_ERR_TIMEOUT in *err.
__global__ void k_debug_mbar_wait(int satisfied, long limit, unsigned* err) {
  using namespace tc;
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (satisfied) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&bar)) : "memory");
    if (!mbar_wait(su32(&bar), 0, &abort_flag, limit)) atomicOr(err, DEV_ERR_TIMEOUT);
  }
}

cudaError_t debug_mbar_wait(int satisfied, long limit, unsigned* err, cudaStream_t st) {
  k_debug_mbar_wait<<<1, 32, 0, st>>>(satisfied, limit, err);
  return cudaGetLastError();
}

template bool tc_applicable<double>(const GemmArgs<double>&);
template cudaError_t gemm_tc<double>(const GemmArgs<double>&, cudaStream_t, Prof*);
template cudaError_t gemm_tc<cplx>(const GemmArgs<cplx>&, cudaStream_t, Prof*);

}  // namespace hps
