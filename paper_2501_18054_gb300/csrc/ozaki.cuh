// Complex FP64 products on the 5th-generation tensor cores of sm_103a, by
// error-free splitting of the operands (Ozaki, Ogita, Oishi, Rump 2012; on
// low-precision tensor cores Mukunoki et al. 2020):
//
//   C[i][j] +-= sum_{k<K} A[i][k] B[j][k],   K <= 64, everything complex128
//
// Every row of A and of B is scaled by a power of two (its own largest real or
// imaginary part lies below 2^e) and written in fixed point, X = rint(a 2^(55-e)):
// 7 signed base-256 digits, each a whole number in [-128, 127]
// that bf16 holds exactly.  A product of two digits is at most 2^14 and the
// sums of one accumulator (all digit pairs s + t = g of a K of 64, two
// products per complex part) stay below 2^24, so that the FP32 accumulation of
// tcgen05.mma is exact whole-number arithmetic: the order of the additions
// does not matter and the result is the same for every tile shape and grid.
// The pairs with s + t <= 7 are kept (34 of 49); the rest are 2^-60 of the product
// of the scales.
//
// Accuracy, against a chain of FP64 multiply-adds: what is lost is the rounding of
// the operands to 56 bits of their row's largest entry, 2^-56 of the product
// 2^(ea + eb) of the two rows' scales, where a chain loses some 2^-52 of the sum's
// size.  Where a row of A and a row of B are large at the same k the digits win.
// Where they are large at different k
// (two parts of a region that hardly couple, metal between two pixels) every
// term is small against the scales and the digits would keep fewer bits.  So
//   m2 = sum_k |A_ik|^2 |B_jk|^2   (relative to the scales)
// is formed first, by one more bf16 product of squared magnitudes, and the
// entries where the digits' error exceeds a chain's (oz_lossy) are listed and
// summed in FP64 from the operands themselves (oz_redo), by every warp of the grid.
//
// Why: the FP64 pipe of this part issues 1.7 multiply-adds per clock and SM
// (1.25 TFLOP/s in all).  136 bf16 products replace the four FP64 products of
// a complex multiply-add, on a pipe about 1500 times as fast.
//
// Layout: operands are digitised once into global images laid out as the
// shared-memory tiles (K-major, no swizzle: 8-row x 16-byte core matrices),
// per K-chunk of 16: A in blocks of 128 rows (56 KB a chunk: re and im, 7
// digits each), B in blocks of 64 rows (28 KB).  A tile is 128 x 64, its real
// part first, then its imaginary part: the 8 digit groups of one part, 64
// columns each, fill the 512 columns of tensor memory.  An MMA of M = 128,
// K = 16 takes 45 cycles at N = 32, 48 at N = 64, 64 at N = 128 and 128 at
// N = 256 (measured): 64 columns per part cost half of 32 columns of both.
//
// Measured: a tile of K = 64 takes 27,000 cycles of products (544 at 48 cycles:
// the shared-memory reads of M = 128, N = 64) and 49,000 in all, bound by the
// issue of the read-back (about 120 integer instructions and one FP64 addition per
// real result; 96 registers a thread, some of them spilled).  2048 x 4096 x 64 on
// 152 SMs: 217 us, 20 TFLOP/s of FP64 products against 1.25 on the FP64 pipe.
// (With no sums in FP64 and C in 256-bit accesses 174 us; see there.)  Entries
// summed in FP64, 64 flips at N_d = 1024 of lossy metal: a fifth of the triangle,
// 0.07 ms on 64 CTAs; in a dielectric guide 10^-4 of the substitutions' diagonal
// blocks and none elsewhere.
#pragma once

#include "flush_tc.cuh"
#include "fp64_fast.cuh"

namespace pngf {
namespace {

constexpr int OZ_S = 7;                       // digits per real number
constexpr int OZ_G = 8;                       // digit groups s + t = 0..7
constexpr int OZ_M = 128, OZ_N = 64;          // tile
constexpr int OZ_KC = 16;                     // K per chunk (one bf16 MMA step)
constexpr int OZ_KMAX = 64;                   // K of one exact accumulation
constexpr int OZ_ASUB = OZ_M * OZ_KC * 2;     // one digit image of an A chunk: 4 KB
constexpr int OZ_BSUB = OZ_N * OZ_KC * 2;     // 2 KB
constexpr int OZ_ACHUNK = 2 * OZ_S * OZ_ASUB; // 56 KB
constexpr int OZ_BCHUNK = 2 * OZ_S * OZ_BSUB; // 28 KB
constexpr int OZ_BUF = OZ_ACHUNK + OZ_BCHUNK; // 84 KB
constexpr int OZ_NBUF = 2;
constexpr int OZ_SMEM = OZ_NBUF * OZ_BUF;     // 168 KB: one CTA per SM
constexpr int OZ_TMEM = OZ_G * OZ_N;          // all 512 columns
constexpr int OZ_EW = 16;                     // epilogue warps (the last ones of the CTA)
constexpr int OZ_THREADS = 32 * (2 + OZ_EW);
constexpr int kOzNaN = 0x20000000;            // row exponent of a row with an infinity or NaN

static_assert(OZ_TMEM == 512, "tensor memory");

// byte offset of element (row, k) in a digit image
__device__ __forceinline__ int oz_off(int row, int k) {
  return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

__host__ __device__ __forceinline__ size_t oz_a_bytes(int rows, int K) {
  return (size_t)((rows + OZ_M - 1) / OZ_M) * ((K + OZ_KC - 1) / OZ_KC) * OZ_ACHUNK;
}
__host__ __device__ __forceinline__ size_t oz_b_bytes(int rows, int K) {
  return (size_t)((rows + OZ_N - 1) / OZ_N) * ((K + OZ_KC - 1) / OZ_KC) * OZ_BCHUNK;
}

// ---------------------------------------------------------------- digits
// Biased exponent of the scale of a row whose largest entry has the upper word
// hmax (without its sign): one more than the entry's where X with the digits'
// offsets would not fit 56 bits (from 127.498 / 128 of a power of two on: the
// mantissa's upper bits 0xFDFE0; 0xFDF00 is taken).
__device__ __forceinline__ int oz_scale_exp(int hmax) { return (hmax + 0x2100) >> 20; }
// X = rint(x 2^(55 - e)), e = emax - 1022 (emax: oz_scale_exp of the row), plus the
// offset that turns its base-256 digits into bytes:
// byte 6 - s of the result is digit s + 128.  Integer arithmetic only.
__device__ __forceinline__ unsigned long long oz_fixed(double x, int emax) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int E = (int)(u >> 52) & 0x7ff;
  unsigned long long m = E ? ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 2 : 0ull;
  const int d = emax - E;
  if (d > 0) m = d < 60 ? (m + (1ull << (d - 1))) >> d : 0ull;
  const unsigned long long X = (long long)u < 0 ? 0ull - m : m;
  return X + 0x0080808080808080ull;
}

// digit byte `sel` (0..3) of a 32-bit word as a float in [-128, 127]
template <int sel>
__device__ __forceinline__ unsigned oz_digit(unsigned w) {
  const float f = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540 | sel)) - 8388736.0f;  // 2^23 + byte - (2^23 + 128)
  return __float_as_uint(f);
}
// digits of two consecutive k as a bf16 pair (their float images end in 16 zero bits)
template <int s>
__device__ __forceinline__ unsigned oz_pair(unsigned long long a, unsigned long long b) {
  constexpr int byte = OZ_S - 1 - s;
  const unsigned wa = byte >= 4 ? (unsigned)(a >> 32) : (unsigned)a, wb = byte >= 4 ? (unsigned)(b >> 32) : (unsigned)b;
  return __byte_perm(oz_digit<byte & 3>(wa), oz_digit<byte & 3>(wb), 0x7632);
}

// eight consecutive k of one row: the 14 16-byte pieces of its digit images
template <int s>
__device__ __forceinline__ void oz_store8(unsigned char* base, int sub, const unsigned long long y[8]) {
  uint4 v;
  v.x = oz_pair<s>(y[0], y[1]);
  v.y = oz_pair<s>(y[2], y[3]);
  v.z = oz_pair<s>(y[4], y[5]);
  v.w = oz_pair<s>(y[6], y[7]);
  *reinterpret_cast<uint4*>(base + s * sub) = v;
}
__device__ __forceinline__ void oz_store_digits(unsigned char* base, int sub, const double v[8], int emax) {
  unsigned long long y[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) y[u] = oz_fixed(v[u], emax);
  oz_store8<0>(base, sub, y);
  oz_store8<1>(base, sub, y);
  oz_store8<2>(base, sub, y);
  oz_store8<3>(base, sub, y);
  oz_store8<4>(base, sub, y);
  oz_store8<5>(base, sub, y);
  oz_store8<6>(base, sub, y);
}

// x 2^-e as a float (20 bits), e = emax - 1022; integer arithmetic only
__device__ __forceinline__ float oz_scaled(double x, int emax) {
  const int hi = __double2hiint(x), d = ((hi >> 20) & 0x7ff) - emax;
  return d < -100 ? 0.0f : __int_as_float(((126 + d) << 23) | ((hi & 0xfffff) << 3));
}

// One warp digitises four rows of an operand with nk chunks (K <= 64): lane =
// (row << 3) | group of 8 k.  `load(row, k)` returns the entry (zero past the
// operand's edges).  BLK = rows per image block (128: A, 64: B).  sq: the squared
// magnitudes in bf16; entries below 2^-30 of the row's largest count as 2^-60, so
// that a sum of them is zero only where every product is.  norms: their sum over the
// row; infinity for a row that holds an infinity or NaN.  full: the entries
// themselves.
template <int BLK, class Load>
__device__ __forceinline__ void oz_digitise_rows(int row0, int K, int nk, unsigned char* img, unsigned char* sq, int* exps,
                                                 float* norms, c128* full, Load load) {
  constexpr int SUB = BLK * OZ_KC * 2;
  const int lane = threadIdx.x & 31, row = row0 + (lane >> 3), kg = lane & 7;
  double re[8], im[8];
  int hmax = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int k = kg * 8 + u;
    const c128 z = k < K ? load(row, k) : mk(0.0, 0.0);
    re[u] = z.x;
    im[u] = z.y;
    hmax = max(hmax, max(__double2hiint(z.x) & 0x7fffffff, __double2hiint(z.y) & 0x7fffffff));
  }
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) hmax = max(hmax, __shfl_xor_sync(0xffffffffu, hmax, off));
  const int emax = oz_scale_exp(hmax);
  float q[8], norm = 0.0f;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const float x = oz_scaled(re[u], emax), y = oz_scaled(im[u], emax);
    q[u] = (oz_exp(re[u]) | oz_exp(im[u])) && emax < 0x7ff ? fmaxf(fmaf(x, x, y * y), 0x1p-60f) : 0.0f;
    norm += q[u];
  }
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) norm += __shfl_xor_sync(0xffffffffu, norm, off);
  if (kg == 0) {
    exps[row] = emax >= 0x7ff ? kOzNaN : emax - 1022;
    norms[row] = emax >= 0x7ff ? INFINITY : norm;
  }
  if (kg < 2 * nk) {
    const size_t chunk = (size_t)(row / BLK) * nk + (kg >> 1);
    const int at = oz_off(row % BLK, (kg & 1) * 8);
    unsigned char* base = img + chunk * (2 * OZ_S * SUB) + at;
    oz_store_digits(base, SUB, re, emax);
    oz_store_digits(base + OZ_S * SUB, SUB, im, emax);
    uint4 v;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(v.x) : "f"(q[1]), "f"(q[0]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(v.y) : "f"(q[3]), "f"(q[2]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(v.z) : "f"(q[5]), "f"(q[4]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(v.w) : "f"(q[7]), "f"(q[6]));
    *reinterpret_cast<uint4*>(sq + chunk * SUB + at) = v;
#pragma unroll
    for (int u = 0; u < 8; ++u) full[(size_t)row * OZ_KMAX + kg * 8 + u] = mk(re[u], im[u]);
  }
}

// Whether an entry is less accurate by its digits than as an FP64 chain, in rms
// errors of a real part, in units of 2^(ea + eb - 53):
//   digits: operands rounded to 2^-56 of their scales, and the sum to 2^-55 of
//           their product, (na + nb + 1) / 192;
//   chain:  a rounding of 2^-53 0.41 of the partial sum per step, sums growing to
//           (m2 / 2)^(1/2) like a random walk: 0.168 K m2 / 2.
// na, nb: norms of the two rows.
__device__ __forceinline__ bool oz_lossy(float na, float nb, float m2, float K) {
  const float s = na + nb + 1.0f;
  return s > 16.1f * K * m2 && (m2 > 0.0f || s == INFINITY);
}
// Whether the rounding of C itself (`roundings` of them in the chain: one where a
// sum is added at the end, K where every term is added to C) exceeds that error all
// the same: 0.168 roundings |C|^2; emax: biased exponent of C's larger part
__device__ __forceinline__ bool oz_below_c(float na, float nb, float roundings, int emax, int e_ab) {
  return na + nb + 1.0f < 32.2f * roundings * exp2f(2.0f * (float)(emax - 1023 - e_ab));
}

// ---------------------------------------------------------------- tile products
__device__ __forceinline__ unsigned oz_idesc(bool negate_a) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((negate_a ? 1u : 0u) << 13) | ((unsigned)(OZ_N >> 3) << 17) |
         ((unsigned)(OZ_M >> 4) << 24);
}
__device__ __forceinline__ void oz_mma(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                       unsigned acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n elect.sync _|q, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// descriptor of a digit image: K-major, no swizzle, core matrices 128 B apart
// along K, 256 B along the rows
__device__ __forceinline__ unsigned long long oz_desc(unsigned smem_addr) {
  return (unsigned long long)((smem_addr & 0x3FFFF) >> 4) | ((unsigned long long)(128 >> 4) << 16) |
         ((unsigned long long)(256 >> 4) << 32) | (1ull << 46);
}

// Pipeline state of a thread, kept across tiles and calls.  Barriers: operand
// copies landed (LOAD) and products done (FREE) per buffer, the accumulators
// of a part complete (FULL) and read back (EMPTY), everything issued done
// (DRAIN, after a failure only).  ph: parity of the thread's next wait on each
// barrier (one thread waits on each); pend: operations it has not waited for.
constexpr int OZ_B_LOAD = 0, OZ_B_FREE = OZ_NBUF, OZ_B_FULL = 2 * OZ_NBUF, OZ_B_EMPTY = 2 * OZ_NBUF + 1;
constexpr int OZ_B_DRAIN = 2 * OZ_NBUF + 2, OZ_NBAR = 2 * OZ_NBUF + 3;
struct OzState {
  unsigned tmem;
  unsigned mb0;   // address of barrier 0
  unsigned ph;    // one parity bit per barrier
  unsigned pend;  // one bit per barrier
  unsigned loads; // copies issued by this thread so far
};
constexpr int OZ_MMA_WARP = 0, OZ_LOAD_WARP = 1;

__device__ __forceinline__ void oz_setup(OzState& st, unsigned long long* bars, unsigned* tmem_slot) {
  if (threadIdx.x == 0) {
    for (int q = 0; q < OZ_NBAR; ++q) {
      const unsigned m = (unsigned)__cvta_generic_to_shared(bars + q);
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(m), "r"(q == OZ_B_EMPTY ? (unsigned)OZ_EW : 1u));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (threadIdx.x < 32) {
    const unsigned sl = (unsigned)__cvta_generic_to_shared(tmem_slot);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sl), "r"(OZ_TMEM));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  st.tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  st.mb0 = (unsigned)__cvta_generic_to_shared(bars);
  st.ph = st.pend = st.loads = 0;
}

__device__ __forceinline__ bool oz_wait_phase(OzState& st, int q) {
  if (!mbar_wait(st.mb0 + 8 * q, (st.ph >> q) & 1)) return false;
  st.ph ^= 1u << q;
  return true;
}
__device__ __forceinline__ bool oz_wait(OzState& st, int q) {
  if (!((st.pend >> q) & 1)) return true;
  if (!oz_wait_phase(st, q)) return false;
  st.pend &= ~(1u << q);
  return true;
}

__device__ __forceinline__ void oz_commit(const OzState& st, int q) {
  asm volatile(
      "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(st.mb0 + 8 * q)
      : "memory");
}

// all threads; after a failure the issuing threads first give the copies and
// products in flight a bounded time to land
__device__ __forceinline__ void oz_teardown(OzState& st, bool failed) {
  if (failed && threadIdx.x == 32 * OZ_LOAD_WARP)
    for (unsigned l = st.loads > OZ_NBUF ? st.loads - OZ_NBUF : 0; l < st.loads; ++l)
      mbar_wait(st.mb0 + 8 * (OZ_B_LOAD + l % OZ_NBUF), (l / OZ_NBUF) & 1);
  if (failed && threadIdx.x / 32 == OZ_MMA_WARP) {
    oz_commit(st, OZ_B_DRAIN);
    oz_wait_phase(st, OZ_B_DRAIN);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(st.tmem), "r"(OZ_TMEM));
}

// one copy's barrier, and its pieces
__device__ __forceinline__ void oz_expect(const OzState& st, int bf, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(st.mb0 + 8 * (OZ_B_LOAD + bf)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void oz_copy(const OzState& st, int bf, unsigned dst, const unsigned char* src, unsigned bytes) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(st.mb0 + 8 * (OZ_B_LOAD + bf))
               : "memory");
}

// The squared magnitudes of OZ_SQ tiles at a time, OZ_SQ / 2 in a buffer: one
// accumulator each.  (One tile at a time, the products of the next tile's real
// part wait until the read-back warps are through with the tile before.)
constexpr int OZ_SQ = 6;
constexpr int OZ_SQ_A = OZ_KMAX / OZ_KC * OZ_ASUB, OZ_SQ_TILE = OZ_SQ_A + OZ_KMAX / OZ_KC * OZ_BSUB;
static_assert(OZ_SQ / OZ_NBUF * OZ_SQ_TILE <= OZ_BUF && OZ_SQ * OZ_N <= OZ_TMEM, "squares of a group of tiles");
__device__ __forceinline__ void oz_issue_squares(const OzState& st, unsigned tile_buf, int acc, int nk) {
  asm volatile("tcgen05.fence::after_thread_sync;");
  for (int c = 0; c < nk; ++c)
    oz_mma(st.tmem + (unsigned)acc * OZ_N, oz_desc(tile_buf + c * OZ_ASUB), oz_desc(tile_buf + OZ_SQ_A + c * OZ_BSUB),
           oz_idesc(false), c > 0 ? 1u : 0u);
}

// the 68 products of one chunk for one part of the tile (0: re, 1: im):
// accumulator g at column g OZ_N.  The whole warp runs this, one lane elected
// per product: the operands of a converged warp stay in uniform registers,
// and the products issue at the rate of their shared-memory reads (48 cycles
// at N = 64; 70 when a single lane runs the loop)
__device__ __forceinline__ void oz_issue_mma(const OzState& st, unsigned sbuf, int part, bool first) {
  asm volatile("tcgen05.fence::after_thread_sync;");
  const unsigned id0 = oz_idesc(false), id1 = oz_idesc(part == 0);
  const unsigned long long d0 = oz_desc(sbuf);
  // re: Ar Br - Ai Bi; im: Ar Bi + Ai Br
  const unsigned long long b0 = d0 + ((OZ_ACHUNK + part * OZ_S * OZ_BSUB) >> 4);
  const unsigned long long b1 = d0 + ((OZ_ACHUNK + (1 - part) * OZ_S * OZ_BSUB) >> 4);
#pragma unroll
  for (int g = 0; g < OZ_G; ++g) {
    const unsigned d = st.tmem + (unsigned)g * OZ_N;
    const int s0 = g < OZ_S ? 0 : g - OZ_S + 1, s1 = g < OZ_S ? g : OZ_S - 1;
#pragma unroll
    for (int s = s0; s <= s1; ++s) {
      const int t = g - s;
      oz_mma(d, d0 + ((s * OZ_ASUB) >> 4), b0 + ((t * OZ_BSUB) >> 4), id0, (first && s == s0) ? 0u : 1u);
      oz_mma(d, d0 + (((OZ_S + s) * OZ_ASUB) >> 4), b1 + ((t * OZ_BSUB) >> 4), id1, 1);
    }
  }
}

// The digit groups' whole-number sums D_0 .. D_7 -> sum_g D_g 256^(7 - g) 2^-15
// (the product X Y in units of 2^55), rounded; below 2^62 in magnitude.  The
// sums D_0 and D_1 are at most 2^22 and turn into integers by an addition of
// 1.5 2^23; D_6 and D_7 matter to a part of their range only and are joined in
// FP32 (their rounding there is below 2^-7 units).
__device__ __forceinline__ long long oz_mad(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ long long oz_fixed_sum(const float* d, int stride) {
  constexpr float kMagic = 12582912.0f;  // 1.5 2^23
  constexpr int kBits = 0x4B400000;
  const int D0 = __float_as_int(d[0] + kMagic) - kBits, D1 = __float_as_int(d[stride] + kMagic) - kBits;
  const int D2 = __float2int_rn(d[2 * stride]);
  const int D3 = __float2int_rn(d[3 * stride]), D4 = __float2int_rn(d[4 * stride]), D5 = __float2int_rn(d[5 * stride]);
  const float low = fmaf(d[7 * stride], 0.00390625f, d[6 * stride]);  // D_6 + D_7 / 256
  const int t = __float_as_int(fmaf(low, 0.0078125f, kMagic)) - kBits;  // / 128, rounded
  const long long H = oz_mad(D0, 1 << 24, oz_mad(D1, 1 << 16, oz_mad(D2, 256, (long long)D3)));
  return (H << 17) + oz_mad(D4, 512, oz_mad(D5, 2, (long long)t));
}

// V 2^sh rounded to FP64 (NaN past its range).  Integer arithmetic only: an FP64 instruction
// occupies its pipe for 64 cycles.
__device__ __forceinline__ double oz_to_double(long long V, int sh) {
  const unsigned long long mag = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
  const int lz = __clzll((long long)mag) & 63;
  const unsigned long long sg = (mag << lz) + 0x400ull;  // 53 leading bits, rounded; a carry leaves bit 63 clear
  const int E = 63 - lz + sh + 1023 + ((sg >> 63) == 0 ? 1 : 0);
  unsigned hi = ((unsigned)(sg >> 43) & 0xfffffu) | ((unsigned)E << 20), lo = (unsigned)(sg >> 11);
  if (E >= 0x7ff) hi = 0x7ff80000u;  // an overflow, or a row with an infinity or NaN (even where V is zero)
  else if (mag == 0 || E <= 0) hi = lo = 0;
  hi |= (unsigned)(V >> 32) & 0x80000000u;
  return __hiloint2double((int)hi, (int)lo);
}

// 4 consecutive columns of the eight digit groups' accumulators (OZ_N columns
// apart) for this thread's lane: d[g * 4 + column]
__device__ __forceinline__ void oz_ld_groups(unsigned addr, float d[4 * OZ_G]) {
  unsigned u[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%33];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%34];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%35];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%36];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%37];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%38];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28,%29,%30,%31}, [%39];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
        "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]),
        "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]),
        "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
      : "r"(addr + 0u * OZ_N), "r"(addr + 1u * OZ_N), "r"(addr + 2u * OZ_N), "r"(addr + 3u * OZ_N), "r"(addr + 4u * OZ_N), "r"(addr + 5u * OZ_N), "r"(addr + 6u * OZ_N), "r"(addr + 7u * OZ_N));
#pragma unroll
  for (int q = 0; q < 32; ++q) d[q] = __uint_as_float(u[q]);
}

// 16 consecutive columns of one accumulator for this thread's lane
__device__ __forceinline__ void oz_ld_squares(unsigned addr, float d[16]) {
  unsigned u[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
        "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
      : "r"(addr));
#pragma unroll
  for (int q = 0; q < 16; ++q) d[q] = __uint_as_float(u[q]);
}

// The list of the entries to sum again: (row of A << 16) | row of B.  oz_listed: how
// many, after a barrier that follows the product; oz_list_clear: by one thread
// before the barrier ahead of it.
__device__ __forceinline__ unsigned oz_listed(const OzOperands& im) { return *reinterpret_cast<volatile unsigned*>(im.list); }
__device__ __forceinline__ void oz_list_clear(const OzOperands& im) { *im.list = 0; }

// marks: bit u = column j0 + u of this lane's row r
__device__ __forceinline__ void oz_list_add(const OzOperands& im, unsigned marks, int r, int j0) {
  const int lane = threadIdx.x & 31, cnt = __popc(marks);
  int incl = cnt;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  unsigned at = 0;
  if (lane == 31) at = atomicAdd(im.list, (unsigned)incl);
  at = __shfl_sync(0xffffffffu, at, 31) + (unsigned)(incl - cnt);
  for (; marks; marks &= marks - 1) im.list[1 + at++] = (unsigned)r << 16 | (unsigned)(j0 + __ffs(marks) - 1);
}

// Sums the m listed entries in FP64: four lanes an entry, lane q of them the terms k
// = q, q + 4, ..., their sums added pairwise.  Warps gw of nw.  Bound by the FP64 pipe
// (four instructions of 64 cycles for eight terms).
template <int OP, class Row>
__device__ __forceinline__ void oz_redo(const OzOperands& im, unsigned m, int K, int gw, int nw, Row row_of) {
  const int lane = threadIdx.x & 31, part = lane & 3;
  for (unsigned e0 = 8u * gw; e0 < m; e0 += 8u * nw) {
    const unsigned e = e0 + (lane >> 2);
    const unsigned at = e < m ? im.list[1 + e] : 0u;
    const int r = (int)(at >> 16), j = (int)(at & 0xffffu);
    const c128* fa = im.fa + (size_t)r * OZ_KMAX;
    const c128* fb = im.fb + (size_t)j * OZ_KMAX;
    c128 s = mk(0.0, 0.0);
    if (e < m) {
#pragma unroll 8
      for (int k = part; k < K; k += 4) s = cfma(fa[k], fb[k], s);
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    if (e < m && part == 0) {
      int cols;
      c128* p = row_of(r, j / OZ_N, cols) + j % OZ_N;
      *p = OP == 0 ? s : OP > 0 ? cadd(*p, s) : csub(*p, s);
    }
  }
}

// The tiles [t_begin, T) with step t_step, in a pipeline of three roles:
//   lane 0 of warp 1 streams the operands through two buffers: before every
//   OZ_SQ-th tile the squared magnitudes of the next OZ_SQ, then for each tile the
//   digit chunks 0 .. nk-1 for the real part and again for the imaginary part,
//   which starts with the two chunks still in the buffers;
//   warp 0 issues the products, part by part, once the accumulators have been
//   read back;
//   the last OZ_EW warps read them back (four warps per lane quadrant, 16
//   columns each): which entries to sum again, the real part into registers, then
//   the imaginary part, and with it C += A B^T (OP = +1), C -= A B^T (-1) or C =
//   A B^T (0).
//   tile_of(t, I, J)      tile t: A row block I, B row block J
//   row_of(r, J, cols)    C at the first column of tile column J for row r of
//                         A (nullptr: no such row), and how
//                         many of the tile's columns exist
//   roundings             of C, see oz_below_c
// The entries that need it are listed, and C left as it was there: oz_redo.
// smem: OZ_SMEM bytes, 128-byte aligned; the CTA has at least OZ_THREADS
// threads.  Returns false after a timeout (the caller then calls
// oz_teardown with failed = true).
template <int OP, class Tile, class Row>
__device__ __forceinline__ bool oz_tiles(OzState& st, unsigned char* smem, const OzOperands& im, int K, float roundings,
                                         long long T, long long t_begin, long long t_step, Tile tile_of, Row row_of) {
  const int tid = threadIdx.x, lane = tid & 31, nwarp = blockDim.x >> 5;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const unsigned s0 = (unsigned)__cvta_generic_to_shared(smem);
  __shared__ int s_fail;
  if (tid == 0) s_fail = 0;
  // earlier generic-proxy use of this shared memory before the bulk copies write it
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  const int nk = (K + OZ_KC - 1) / OZ_KC;
  const long long mine = t_begin < T ? (T - 1 - t_begin) / t_step + 1 : 0;
  const int nl = nk + max(0, nk - 2);  // copies per tile
  // tiles k0 .. of a group, and those in its buffer q
  auto group = [&](long long k0) { return (int)min((long long)OZ_SQ, mine - k0); };
  auto in_buffer = [&](int n, int q) { return min(OZ_SQ / OZ_NBUF, n - q * (OZ_SQ / OZ_NBUF)); };
  if (warp == OZ_LOAD_WARP) {
    if (lane == 0) {
      bool ok = true;
      int bf = 0;
      auto next = [&]() {  // the next buffer, free
        bf = (int)(st.loads % OZ_NBUF);
        ok = oz_wait(st, OZ_B_FREE + bf);
        if (!ok) return false;
        ++st.loads;
        st.pend |= 1u << (OZ_B_FREE + bf);
        return true;
      };
      for (long long k = 0; k < mine && ok; ++k) {
        int I, J;
        if (k % OZ_SQ == 0) {
          const int n = group(k);
          for (int q = 0; q < OZ_NBUF && in_buffer(n, q) > 0 && next(); ++q) {
            oz_expect(st, bf, in_buffer(n, q) * nk * (OZ_ASUB + OZ_BSUB));
            for (int t = 0; t < in_buffer(n, q); ++t) {
              tile_of(t_begin + (k + q * (OZ_SQ / OZ_NBUF) + t) * t_step, I, J);
              const unsigned dst = s0 + bf * OZ_BUF + t * OZ_SQ_TILE;
              oz_copy(st, bf, dst, im.sqA + (size_t)I * nk * OZ_ASUB, nk * OZ_ASUB);
              oz_copy(st, bf, dst + OZ_SQ_A, im.sqB + (size_t)J * nk * OZ_BSUB, nk * OZ_BSUB);
            }
          }
        }
        tile_of(t_begin + k * t_step, I, J);
        for (int l = 0; l < nl && ok && next(); ++l) {
          const int c = l < nk ? l : l - nk;
          oz_expect(st, bf, OZ_BUF);
          oz_copy(st, bf, s0 + bf * OZ_BUF, im.A + ((size_t)I * nk + c) * OZ_ACHUNK, OZ_ACHUNK);
          oz_copy(st, bf, s0 + bf * OZ_BUF + OZ_ACHUNK, im.B + ((size_t)J * nk + c) * OZ_BCHUNK, OZ_BCHUNK);
        }
      }
      for (int q = OZ_B_FREE; q < OZ_B_FULL && ok; ++q) ok = oz_wait(st, q);  // the next call starts in step
      if (!ok) s_fail = 1;
    }
  } else if (warp == OZ_MMA_WARP) {
    bool ok = true;
    auto full = [&]() {
      oz_commit(st, OZ_B_FULL);
      st.pend |= 1u << OZ_B_EMPTY;
    };
    for (long long k = 0; k < mine && ok; ++k) {
      if (k % OZ_SQ == 0) {
        const int n = group(k);
        ok = __all_sync(0xffffffffu, oz_wait(st, OZ_B_EMPTY));
        for (int q = 0; q < OZ_NBUF && in_buffer(n, q) > 0 && ok; ++q, ++st.loads) {
          const int bf = (int)(st.loads % OZ_NBUF);
          ok = __all_sync(0xffffffffu, oz_wait_phase(st, OZ_B_LOAD + bf));
          if (!ok) break;
          for (int t = 0; t < in_buffer(n, q); ++t)
            oz_issue_squares(st, s0 + bf * OZ_BUF + t * OZ_SQ_TILE, q * (OZ_SQ / OZ_NBUF) + t, nk);
          oz_commit(st, OZ_B_FREE + bf);
        }
        if (ok) full();
      }
      for (int part = 0; part < 2 && ok; ++part) {
        ok = __all_sync(0xffffffffu, oz_wait(st, OZ_B_EMPTY));
        for (int j = 0; j < nk && ok; ++j) {
          // the copy that step j of this part reads, counted from the tile's first
          const int l = part == 0 ? j : nk == 1 ? 0 : j < 2 ? nk - 2 + j : nk + j - 2;
          const int bf = (int)((st.loads + l) % OZ_NBUF);
          const bool again = part == 1 && l < nk;  // landed in the first part already
          if (!again) ok = __all_sync(0xffffffffu, oz_wait_phase(st, OZ_B_LOAD + bf));
          if (!ok) break;
          oz_issue_mma(st, s0 + bf * OZ_BUF, part, j == 0);
          if (part == 1 || l < nk - 2) oz_commit(st, OZ_B_FREE + bf);  // its last use
        }
        if (ok) full();
      }
      st.loads += nl;
    }
    if (ok) ok = __all_sync(0xffffffffu, oz_wait(st, OZ_B_EMPTY));
    if (!ok) s_fail = 1;
  } else if (warp >= nwarp - OZ_EW) {
    constexpr int CW = OZ_N / (OZ_EW / 4);  // columns per warp
    static_assert(CW == 16, "oz_ld_squares");
    const int ew = warp - (nwarp - OZ_EW), quad = warp & 3, c0 = CW * (ew >> 2);
    const unsigned acc0 = st.tmem + ((unsigned)(32 * quad) << 16) + (unsigned)c0;
    auto freed = [&]() {  // the accumulators are in registers
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(st.mb0 + 8 * OZ_B_EMPTY) : "memory");
    };
    unsigned long long lossy[2] = {0, 0};  // 16 bits per tile of the group
    static_assert(OZ_SQ <= 8, "lossy");
    bool ok = true;
    for (long long k = 0; k < mine && ok; ++k) {
      int I, J, cols = 0;
      tile_of(t_begin + k * t_step, I, J);
      const int r = I * OZ_M + 32 * quad + lane;
      c128* crow = row_of(r, J, cols);
      cols = crow != nullptr ? max(0, min(CW, cols - c0)) : 0;
      const int e_a = im.ea[r];
      const float n_a = im.na[r];
      const int4* ebp = reinterpret_cast<const int4*>(im.eb + J * OZ_N + c0);
      const float4* nbp = reinterpret_cast<const float4*>(im.nb + J * OZ_N + c0);
      // ---- the entries to sum again, of the next OZ_SQ tiles
      if (k % OZ_SQ == 0) {
        if (!__all_sync(0xffffffffu, oz_wait_phase(st, OZ_B_FULL))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        lossy[0] = lossy[1] = 0;
        const int n = group(k);
#pragma unroll 1
        for (int t = 0; t < n; ++t) {
          int It, Jt;
          tile_of(t_begin + (k + t) * t_step, It, Jt);
          const float nat = im.na[It * OZ_M + 32 * quad + lane];
          const float4* nbt = reinterpret_cast<const float4*>(im.nb + Jt * OZ_N + c0);
          float m2[CW];
          oz_ld_squares(acc0 + (unsigned)(t * OZ_N), m2);
          unsigned m = 0;
#pragma unroll
          for (int q = 0; q < CW / 4; ++q) {
            const float4 n4 = nbt[q];
            const float n_b[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (oz_lossy(nat, n_b[u], m2[4 * q + u], (float)K)) m |= 1u << (4 * q + u);
          }
          if (t < 4) lossy[0] |= (unsigned long long)m << (16 * t);
          else lossy[1] |= (unsigned long long)m << (16 * (t - 4));
        }
        freed();
      }
      const int kg = (int)(k % OZ_SQ);
      unsigned marks = (unsigned)((kg < 4 ? lossy[0] : lossy[1]) >> (16 * (kg & 3))) & ((1u << cols) - 1u);
      double re[CW];
#pragma unroll 1
      for (int part = 0; part < 2; ++part) {
        // every warp waits for itself (no barrier among them: they drift apart,
        // and the FP64, integer and memory work of one fills the others' waits)
        if (!__all_sync(0xffffffffu, oz_wait_phase(st, OZ_B_FULL))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // the accumulators are freed once their sums are in registers; all
        // that follows runs beside the products of the next part
        long long V[CW];
#pragma unroll
        for (int q = 0; q < CW / 4; ++q) {
          float d[4 * OZ_G];
          oz_ld_groups(acc0 + (unsigned)(4 * q), d);
#pragma unroll
          for (int u = 0; u < 4; ++u) V[4 * q + u] = oz_fixed_sum(d + u, 4);
        }
        freed();
        if (part == 0) {
#pragma unroll
          for (int q = 0; q < CW / 4; ++q) {
            const int4 e4 = ebp[q];
            const int e_b[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) re[4 * q + u] = oz_to_double(V[4 * q + u], e_a + e_b[u] - 55);
          }
          continue;
        }
        // C, two columns at a time: an even and an odd lane read and write 32
        // consecutive bytes of the even lane's row, then of the odd lane's, and
        // hand each other what belongs to the other's row
        const bool odd = lane & 1;
        c128* const other = reinterpret_cast<c128*>(__shfl_xor_sync(0xffffffffu, reinterpret_cast<unsigned long long>(crow), 1));
        const int ocols = __shfl_xor_sync(0xffffffffu, cols, 1);
        c128* const pe = (odd ? other : crow) + c0 + (odd ? 1 : 0);  // this lane's column of a pair, in the even row
        c128* const po = (odd ? crow : other) + c0 + (odd ? 1 : 0);  // and in the odd row
        const int ce = (odd ? ocols - 1 : cols), co = (odd ? cols - 1 : ocols);  // it exists for columns below
        auto swap2 = [&](c128 z) {
          return mk(__shfl_xor_sync(0xffffffffu, z.x, 1), __shfl_xor_sync(0xffffffffu, z.y, 1));
        };
#pragma unroll
        for (int q = 0; q < CW / 4; ++q) {
          c128 x[4] = {};
          if (OP != 0) {
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
              const int c = 4 * q + u;
              c128 ze = mk(0.0, 0.0), zo = ze;
              if (c < ce) ze = pe[c];
              if (c < co) zo = po[c];
              const c128 got = swap2(odd ? ze : zo);
              x[u] = odd ? got : ze;
              x[u + 1] = odd ? zo : got;
            }
          }
          const int4 e4 = ebp[q];
          const int e_b[4] = {e4.x, e4.y, e4.z, e4.w};
          if (OP != 0 && (marks >> (4 * q) & 15u)) {
            const float4 n4 = nbp[q];
            const float n_b[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (oz_below_c(n_a, n_b[u], roundings, max(oz_exp(x[u].x), oz_exp(x[u].y)), e_a + e_b[u]))
                marks &= ~(1u << (4 * q + u));
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const double v = oz_to_double(V[4 * q + u], e_a + e_b[u] - 55);
            if (marks >> (4 * q + u) & 1u) continue;  // as it was
            if (OP == 0) x[u] = mk(re[4 * q + u], v);
            else if (OP > 0) x[u] = mk(x[u].x + re[4 * q + u], x[u].y + v);
            else x[u] = mk(x[u].x - re[4 * q + u], x[u].y - v);
          }
#pragma unroll
          for (int u = 0; u < 4; u += 2) {
            const int c = 4 * q + u;
            const c128 got = swap2(odd ? x[u] : x[u + 1]);
            if (c < ce) pe[c] = odd ? got : x[u];
            if (c < co) po[c] = odd ? x[u + 1] : got;
          }
        }
      }
      if (!ok) break;
      if (__any_sync(0xffffffffu, marks != 0)) oz_list_add(im, marks, r, J * OZ_N + c0);
    }
    if (!ok) s_fail = 1;
  }
  __syncthreads();
  return s_fail == 0;
}

}  // namespace
}  // namespace pngf
