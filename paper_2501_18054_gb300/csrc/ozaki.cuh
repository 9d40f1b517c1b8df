// Complex FP64 products on the 5th-generation tensor cores of sm_103a, by
// error-free splitting of the operands (Ozaki, Ogita, Oishi, Rump 2012; on
// low-precision tensor cores Mukunoki et al. 2020):
//
//   C[i][j] +-= sum_{k<K} A[i][k] B[j][k],   K <= 64, everything complex128
//
// Every row of A and of B is scaled by a power of two (its own largest real or
// imaginary part lies below 2^e) and written in fixed point, X = rint(a 2^(54-e)),
// |X| <= 2^54: 7 signed base-256 digits, each a whole number in [-128, 127]
// that bf16 holds exactly.  A product of two digits is below 2^14 and the
// sums of one accumulator (all digit pairs s + t = g of a K of 64, two
// products per complex part) stay below 2^24, so that the FP32 accumulation of
// tcgen05.mma is exact whole-number arithmetic: the order of the additions
// does not matter and the result is the same for every tile shape and grid.
// The pairs with s + t <= 7 are kept (34 of 49); the rest are below
// 2^-58 of the largest product.  The dominant error is the rounding of the
// operands to 55 bits of their row's largest entry, below the 53-bit rounding
// of an FP64 multiply-add chain of the same length.
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
// the shared-memory reads of M = 128, N = 64) and 40,000 in all, the rest the
// read-back (about 120 integer instructions and one FP64 addition per real
// result).  2048 x 4096 x 64 on 152 SMs: 174 us, 25 TFLOP/s of FP64 products
// against 1.25 on the FP64 pipe (180 us with a barrier among the read-back
// warps; accumulators freed in two halves: 184, more spills).
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
constexpr int OZ_THREADS = 32 * (2 + OZ_EW);  // 112 registers a thread
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
// X = rint(x 2^(54 - e)), e = emax - 1022 (biased exponent emax of the row's
// largest entry), plus the offset that turns its base-256 digits into bytes:
// byte 6 - s of the result is digit s + 128.  Integer arithmetic only.
__device__ __forceinline__ unsigned long long oz_fixed(double x, int emax) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int E = (int)(u >> 52) & 0x7ff;
  unsigned long long m = E ? ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 1 : 0ull;
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

// One warp digitises four rows of an operand with nk chunks (K <= 64): lane =
// (row << 3) | group of 8 k.  `load(row, k)` returns the entry (zero past the
// operand's edges).  BLK = rows per image block (128: A, 64: B).
template <int BLK, class Load>
__device__ __forceinline__ void oz_digitise_rows(int row0, int K, int nk, unsigned char* img, int* exps, Load load) {
  constexpr int SUB = BLK * OZ_KC * 2;
  const int lane = threadIdx.x & 31, row = row0 + (lane >> 3), kg = lane & 7;
  double re[8], im[8];
  int emax = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int k = kg * 8 + u;
    const c128 z = k < K ? load(row, k) : mk(0.0, 0.0);
    re[u] = z.x;
    im[u] = z.y;
    emax = max(emax, max(oz_exp(z.x), oz_exp(z.y)));
  }
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, off));
  if (kg == 0) exps[row] = emax == 0x7ff ? kOzNaN : emax - 1022;
  if (kg < 2 * nk) {
    unsigned char* base = img + ((size_t)(row / BLK) * nk + (kg >> 1)) * (2 * OZ_S * SUB) +
                          oz_off(row % BLK, (kg & 1) * 8);
    oz_store_digits(base, SUB, re, emax);
    oz_store_digits(base + OZ_S * SUB, SUB, im, emax);
  }
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

__device__ __forceinline__ void oz_issue_copy(const OzState& st, int bf, unsigned sbuf, const unsigned char* a,
                                              const unsigned char* b) {
  const unsigned mb = st.mb0 + 8 * (OZ_B_LOAD + bf);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(OZ_BUF) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sbuf),
               "l"(a), "r"(OZ_ACHUNK), "r"(mb)
               : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   sbuf + OZ_ACHUNK),
               "l"(b), "r"(OZ_BCHUNK), "r"(mb)
               : "memory");
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

// The digit groups' whole-number sums D_0 .. D_7 -> sum_g D_g 256^(7 - g) 2^-13
// (the product X Y in units of 2^53), rounded; below 2^62 in magnitude.  The
// sums up to D_2 are below 2^22 and turn into integers by an addition of
// 1.5 2^23; D_6 and D_7 matter to a part of their range only and are joined in
// FP32 (their rounding there is below 2^-5 units).
__device__ __forceinline__ long long oz_mad(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ long long oz_fixed_sum(const float* d, int stride) {
  constexpr float kMagic = 12582912.0f;  // 1.5 2^23
  constexpr int kBits = 0x4B400000;
  const int D0 = __float_as_int(d[0] + kMagic) - kBits, D1 = __float_as_int(d[stride] + kMagic) - kBits;
  const int D2 = __float_as_int(d[2 * stride] + kMagic) - kBits;
  const int D3 = __float2int_rn(d[3 * stride]), D4 = __float2int_rn(d[4 * stride]), D5 = __float2int_rn(d[5 * stride]);
  const float low = fmaf(d[7 * stride], 0.00390625f, d[6 * stride]);        // D_6 + D_7 / 256
  const int t = __float_as_int(fmaf(low, 0.03125f, kMagic)) - kBits;        // / 32, rounded
  const long long H = oz_mad(D0, 1 << 24, oz_mad(D1, 1 << 16, oz_mad(D2, 256, (long long)D3)));
  return (H << 19) + oz_mad(D4, 2048, oz_mad(D5, 8, (long long)t));
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

// The tiles [t_begin, T) with step t_step, in a pipeline of three roles:
//   lane 0 of warp 1 streams the operand chunks through two buffers.  The
//   chunks 0 .. nk-1 are needed for the real part and again for the imaginary
//   part, which starts with the two chunks still in the buffers;
//   warp 0 issues the products, part by part, once the accumulators have been
//   read back;
//   the last OZ_EW warps read them back (four warps per lane quadrant, 16
//   columns each): the real part into registers, then the imaginary part, and
//   with it C += A B^T (OP = +1), C -= A B^T (-1) or C = A B^T (0).
//   tile_of(t, I, J)      tile t: A row block I, B row block J
//   row_of(r, J, cols)    C at the first column of tile column J for row r of
//                         A (nullptr: no such row), and how
//                         many of the tile's columns exist
// smem: OZ_SMEM bytes, 128-byte aligned; the CTA has at least OZ_THREADS
// threads.  Returns false after a timeout (the caller then calls
// oz_teardown with failed = true).
template <int OP, class Tile, class Row>
__device__ __forceinline__ bool oz_tiles(OzState& st, unsigned char* smem, const unsigned char* imgA,
                                         const unsigned char* imgB, const int* ea, const int* eb, int nk, long long T,
                                         long long t_begin, long long t_step, Tile tile_of, Row row_of) {
  const int tid = threadIdx.x, lane = tid & 31, nwarp = blockDim.x >> 5;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const unsigned s0 = (unsigned)__cvta_generic_to_shared(smem);
  __shared__ int s_fail;
  if (tid == 0) s_fail = 0;
  // earlier generic-proxy use of this shared memory before the bulk copies write it
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  const long long mine = t_begin < T ? (T - 1 - t_begin) / t_step + 1 : 0;
  const int nl = nk + max(0, nk - 2);  // copies per tile
  if (warp == OZ_LOAD_WARP) {
    if (lane == 0) {
      bool ok = true;
      for (long long k = 0; k < mine && ok; ++k) {
        int I, J;
        tile_of(t_begin + k * t_step, I, J);
        for (int l = 0; l < nl && ok; ++l) {
          const int c = l < nk ? l : l - nk, bf = (int)(st.loads % OZ_NBUF);
          ok = oz_wait(st, OZ_B_FREE + bf);
          if (!ok) break;
          oz_issue_copy(st, bf, s0 + bf * OZ_BUF, imgA + ((size_t)I * nk + c) * OZ_ACHUNK,
                        imgB + ((size_t)J * nk + c) * OZ_BCHUNK);
          ++st.loads;
          st.pend |= 1u << (OZ_B_FREE + bf);
        }
      }
      for (int q = OZ_B_FREE; q < OZ_B_FULL && ok; ++q) ok = oz_wait(st, q);  // the next call starts in step
      if (!ok) s_fail = 1;
    }
  } else if (warp == OZ_MMA_WARP) {
    bool ok = true;
    for (long long k = 0; k < mine && ok; ++k) {
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
        if (ok) {
          oz_commit(st, OZ_B_FULL);
          st.pend |= 1u << OZ_B_EMPTY;
        }
      }
      st.loads += nl;
    }
    if (ok) ok = __all_sync(0xffffffffu, oz_wait(st, OZ_B_EMPTY));
    if (!ok) s_fail = 1;
  } else if (warp >= nwarp - OZ_EW) {
    constexpr int CW = OZ_N / (OZ_EW / 4);  // columns per warp
    const int ew = warp - (nwarp - OZ_EW), quad = warp & 3, c0 = CW * (ew >> 2);
    const unsigned acc0 = st.tmem + ((unsigned)(32 * quad) << 16) + (unsigned)c0;
    bool ok = true;
    for (long long k = 0; k < mine && ok; ++k) {
      int I, J, cols = 0;
      tile_of(t_begin + k * t_step, I, J);
      const int r = I * OZ_M + 32 * quad + lane;
      c128* crow = row_of(r, J, cols);
      cols = crow != nullptr ? cols - c0 : 0;
      const int e_a = cols > 0 ? ea[r] : 0;
      const int4* ebp = reinterpret_cast<const int4*>(eb + J * OZ_N + c0);
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
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(st.mb0 + 8 * OZ_B_EMPTY) : "memory");
        if (cols <= 0) continue;
        c128* p = crow + c0;
#pragma unroll
        for (int q = 0; q < CW / 4; ++q, p += 4) {  // four columns; C is read first
          const int left = cols - 4 * q;
          if (left <= 0) continue;
          c128 x[4];
          if (OP != 0 && part == 1) {
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = u < left ? p[u] : mk(0.0, 0.0);
          }
          const int4 e4 = ebp[q];
          const int e_b[4] = {e4.x, e4.y, e4.z, e4.w};
          double v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = oz_to_double(V[4 * q + u], e_a + e_b[u] - 55);
          if (part == 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) re[4 * q + u] = v[u];
            continue;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (OP == 0) x[u] = mk(re[4 * q + u], v[u]);
            else if (OP > 0) x[u] = mk(x[u].x + re[4 * q + u], x[u].y + v[u]);
            else x[u] = mk(x[u].x - re[4 * q + u], x[u].y - v[u]);
          }
          // 16 bytes per access: with a 256-bit store in its place (st.global.v4.f64)
          // nvcc 13.0.88 left the store out, in code that two kernels of a file call
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (u < left) p[u] = x[u];
        }
      }
    }
    if (!ok) s_fail = 1;
  }
  __syncthreads();
  return s_fail == 0;
}

}  // namespace
}  // namespace pngf
