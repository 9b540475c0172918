// FP64-accurate block products C = op(A) B on the BF16 tensor cores, the
// operands sliced on their way into shared memory (error-free fixed-point
// slicing, the Ozaki scheme).  One kernel serves the products A X and A^T Y
// with a dense FP64 operator, the Ritz lifts [S1 S2] Y and the Gram products
// X^T Y of blocks of any storage type.
//
// Slicing: every row of op(A) and every column of B is scaled by a power of
// two 2^e so that its entries lie in (-1, 1), rounded to a fixed-point integer
// of 7 T bits and split into T balanced base-128 digits:
//   x = 2^e (sum_{p=1..T} s_p 2^(-7 p) + r), |s_1| <= 128, |s_p| <= 64,
//   |r| <= 2^(-7 T - 1),
// each an integer that BF16 holds exactly.  Digit pairs with p + q <= T + 1 are
// multiplied.  All pairs of one sum d = p + q - 2 carry the same weight
// 2^(-14 - 7 d) and share one FP32 accumulator: over 32 KG columns of K its
// partial sums stay below 2^24 (T = 7: 36864 * 448, T = 9: 45056 * 352), so
// the tensor core adds exactly.  After KG stages the T accumulators of an
// element are combined with integer arithmetic (one 64-bit sum per element),
// and one integer-to-double conversion per element ends the tile.
//   T = 7 keeps more than the 8 slices of 6 bits used before it (remainder
// 2^-50 against 2^-49, dropped pairs 6 2^-51 against 7 2^-50 of the row and
// column scales) with 28 pair products instead of 36.  A term errs by less than
// 5.1 2^-50 of the two scales, each up to twice its largest entry: 2^-45 of the
// largest entries.  T = 9 serves callers that ask for 9 or 10 slices of 6 bits
// (1.6 2^-62 of the scales, 2^-59 of the largest entries).
//
// Why slicing belongs in this kernel: sliced operands are 14 bytes an entry,
// written once and read back per tile, which bounded every use (a 1M x 160
// Gram moved 10 GB for 1.7 GB of input).  Here an entry is read in its own
// type and its digits go from registers to shared memory.  Against slices in
// memory, 36 pair products and FP64 atomics per pair: Gram 1048576 x (160, 160)
// 11.7 -> 5.3 ms, product 16384 x 4096 x 128 1.74 -> 0.70 ms, lift
// 360001 x (96 + 96) x 96 9.3 -> 1.10 ms; the error against 64 bits halves.
//
// One CTA an SM, persistent over tiles of 128 rows x up to 64 columns (T
// accumulators of 64 columns are 448 of the 512 TMEM columns) and K ranges:
//   warps 0-15  slice: load 128 x 32 entries of A (and of B in the Gram form)
//               a stage, the next stage's loads in flight, write the T digit
//               planes as 64-byte-swizzled K-major tiles, and read the
//               accumulators out every KG stages;
//   warp 16     one lane issues the tcgen05.mma: digit p of A against up to
//               256 / width digits q of B side by side (N up to 256: the MMA
//               rate falls below N = 128), which lands in neighbouring
//               accumulators d = p + q.
// Two stages of T (128 + width) x 64 bytes.  B of the operator products and of
// the lifts is small and read by every row tile: it is sliced once into
// ready-to-copy stage images (k_emu_bslice) that one bulk copy brings in.
// Bounds: 28 products of 128 x 64 x 32 take 1843 cycles a stage (3980 of 4096
// multiply-adds a cycle), the digits of 128 x 32 entries about 1400 (logic and
// shifts at 64 lanes a cycle).
// Every wait is bounded (2 s); on expiry the kernel records an error, drains
// its copies and MMAs, frees its TMEM and returns.
#include <algorithm>
#include <type_traits>

#include "rr_common.cuh"
#include "solver_kernels.cuh"
#include "tc_ptx.cuh"

namespace rr {

__device__ int g_emu_error = 0;

namespace {

constexpr int kKB = 32;            // K entries of a stage (64-byte swizzled rows)
constexpr int kRows = 128;         // rows of a tile
constexpr int kSlicers = 16;       // slicing warps
constexpr int kRing = 2;           // stages
constexpr int kThreads = 32 * (kSlicers + 1);
constexpr int kExpNone = -1100;    // exponent of an all-zero row or column
constexpr int kExpInf = 1025;      // exponent of a row or column with an infinity or NaN

template <int T>
struct EmuConst {
  static constexpr int kg = T == 7 ? 14 : 11;      // stages of one exact FP32 accumulation
  static constexpr int base_shift = 7 * (T - 7) + 3;  // bits dropped from a group's exact integer sum
  // tile columns: T max_w <= 512, and the shared memory: 213 KB for 32 columns of
  // T = 9 (16384 x 4096 x 128 with 16: 2.40 ms, every column tile slices A again)
  static constexpr int max_w = T == 7 ? 64 : 32;
};

// stages of an accumulation group: nst stages in groups of about one size
template <int T>
__device__ __forceinline__ int group_stages(int nst) {
  const int g = (nst + EmuConst<T>::kg - 1) / EmuConst<T>::kg;
  return (nst + g - 1) / g;
}

__device__ __forceinline__ bool emu_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_on(bar, parity, &g_emu_error, kWaitLimitNs);
}

// the same for a whole warp: every lane gets one answer, so no lane leaves alone
__device__ __forceinline__ bool emu_wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, emu_wait(bar, parity)) != 0;
}

// bounded wait that ignores the error word (draining after an error)
__device__ __forceinline__ void emu_drain(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity) && global_timer_ns() - t0 < kWaitLimitNs) {
  }
}

// exponent e with |x| < 2^e; zero and subnormals: kExpNone
__device__ __forceinline__ int exp_of(double x) {
  const int E = (__double2hiint(x) >> 20) & 0x7FF;
  return E == 0 ? kExpNone : E - 1022;
}

// FP64 value of a stored entry through integer operations (the conversion
// instruction runs on the few FP64 units): exact for normal numbers; zero and
// subnormals get an exponent of 2^-127 or less, which slice_pair takes for zero
// in every row whose largest entry is above kTiny32
__device__ __forceinline__ double f32_exact(float f) {
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(u << 29));
}
// Zeros and subnormals count as 2^-1023 (FP64) or 2^-127 (f32_exact) in
// slice_pair and vanish next to a row exponent of at least kTiny64 or kTiny32.
// Rows whose largest entry is smaller than that go up by 200 or 100 binades,
// the row exponent and every nonzero entry (exactly; FP64 subnormals are taken
// for zero).
constexpr int kTiny64 = -950, kTiny32 = -60;
template <bool kWide>
__device__ __forceinline__ int up_exp(int e) {
  constexpr int lim = kWide ? kTiny64 : kTiny32, up = kWide ? 200 : 100;
  return e >= lim ? e : e == kExpNone ? 0 : e + up;
}
__device__ __forceinline__ double up_entry(double x, int e) {
  const int hi = __double2hiint(x);
  if ((hi & 0x7FF00000) == 0) return 0.0;
  return e >= kTiny64 ? x : __hiloint2double(hi + (200 << 20), __double2loint(x));
}
__device__ __forceinline__ float up_scale(int e) { return e >= kTiny32 ? 1.f : 1.2676506e30f; }  // 2^100

// raw bits of stored entries, and of two neighbours (aligned to the pair)
template <typename TS> struct Raw;
template <> struct Raw<double> {
  typedef unsigned long long R;
  static __device__ __forceinline__ R ld(const double* p) { return (R)__double_as_longlong(__ldg(p)); }
  static __device__ __forceinline__ void ld2(const double* p, R& a, R& b) {
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
    a = v.x;
    b = v.y;
  }
};
template <> struct Raw<float> {
  typedef uint32_t R;
  static __device__ __forceinline__ R ld(const float* p) { return __float_as_uint(__ldg(p)); }
  static __device__ __forceinline__ void ld2(const float* p, R& a, R& b) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    a = v.x;
    b = v.y;
  }
};
template <> struct Raw<__nv_bfloat16> {
  typedef uint32_t R;
  static __device__ __forceinline__ R ld(const __nv_bfloat16* p) {
    return __ldg(reinterpret_cast<const unsigned short*>(p));
  }
  static __device__ __forceinline__ void ld2(const __nv_bfloat16* p, R& a, R& b) {
    const unsigned v = __ldg(reinterpret_cast<const unsigned*>(p));
    a = v & 0xFFFFu;
    b = v >> 16;
  }
};
template <> struct Raw<e4m3b_t> {
  typedef uint32_t R;
  static __device__ __forceinline__ R ld(const e4m3b_t* p) { return __ldg(reinterpret_cast<const unsigned char*>(p)); }
  static __device__ __forceinline__ void ld2(const e4m3b_t* p, R& a, R& b) {
    const unsigned short v = __ldg(reinterpret_cast<const unsigned short*>(p));
    a = v & 0xFFu;
    b = v >> 8;
  }
};

// exponent e with |x| < 2^e of a stored entry (infinities and NaN: kExpInf)
template <typename TS>
__device__ __forceinline__ int exp_raw(typename Raw<TS>::R r) {
  if constexpr (sizeof(TS) == 8) {
    return exp_of(__longlong_as_double((long long)r));
  } else {
    const float f = sizeof(TS) == 4   ? __uint_as_float((unsigned)r)
                    : sizeof(TS) == 2 ? __uint_as_float((unsigned)r << 16)
                                      : e4m3b_value((unsigned char)r);
    const unsigned m = __float_as_uint(f) & 0x7FFFFFFFu;
    if (m >= 0x7F800000u) return kExpInf;
    if (m < 0x800000u) return m ? 32 - __clz(m) - 149 : kExpNone;  // subnormals
    return (int)(m >> 23) - 126;
  }
}

// The digits of two entries as BF16 pairs (a in the low half), most
// significant first.  Entries far below 2^e, zeros among them, shift out.
//
// T = 7: |x| 2^(60 - e), rounded at bit 11 and with 64 added to each of the six
// lower digits, holds digits + 64 in bits 11-17, 18-24, 25-31 and 32-38, 39-45,
// 46-52, the leading digit above.  A shift brings a digit to a byte boundary, a
// byte permute pairs it with the other entry's, and under exponent bits 0x4300
// a 7-bit u is the BF16 number 128 + u: one packed FMA makes it +-(u - 64).
// Logic and shifts run at half the FMA rate here, and they bound the whole
// kernel: 17 an entry in this form, 53 with a rounded two's complement value
// split by shifts and masks (16384 x 4096 x 128 product: 0.70 ms).
template <int T>
__device__ __forceinline__ void slice_pair(double xa, double xb, int ea, int eb, uint32_t (&out)[T]) {
  const uint32_t ha = (uint32_t)__double2hiint(xa), hb = (uint32_t)__double2hiint(xb);
  const int Ea = (int)((ha << 1) >> 21), Eb = (int)((hb << 1) >> 21);
  // |x| = (M 2^-63) 2^(E - 1022), M with its leading bit at 63; E - 1022 <= e
  const unsigned long long Ma =
      ((unsigned long long)(__funnelshift_l((uint32_t)__double2loint(xa), ha, 11) | 0x80000000u) << 32) |
      ((uint32_t)__double2loint(xa) << 11);
  const unsigned long long Mb =
      ((unsigned long long)(__funnelshift_l((uint32_t)__double2loint(xb), hb, 11) | 0x80000000u) << 32) |
      ((uint32_t)__double2loint(xb) << 11);
  const uint32_t sa = (uint32_t)(ea + 1022 - Ea), sb = (uint32_t)(eb + 1022 - Eb);  // M >> sh: |x| 2^(64 - e)
  const uint32_t sgn = __byte_perm(ha, hb, 0x7632) & 0x80008000u;
  const uint32_t one = sgn | 0x3F803F80u;  // +-1
  auto fma2 = [](uint32_t a, uint32_t b, uint32_t c) -> uint32_t {
    uint32_t d;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
  };
  // shifts of 64 or more give 0 (a clamped shift, as PTX defines it)
  unsigned long long wa, wb;
  if constexpr (T == 7) {
    constexpr unsigned long long C = ((64ull * (((1ull << 42) - 1) / 127)) << 11) + (1ull << 10);
    asm("shr.u64 %0, %1, %2;" : "=l"(wa) : "l"(Ma), "r"(sa + 4));
    asm("shr.u64 %0, %1, %2;" : "=l"(wb) : "l"(Mb), "r"(sb + 4));
    wa += C;
    wb += C;
    const uint32_t la = (uint32_t)wa, lb = (uint32_t)wb, ua = (uint32_t)(wa >> 32), ub = (uint32_t)(wb >> 32);
    const uint32_t off = sgn ^ 0xC340C340u;  // -+192
    constexpr uint32_t m7 = 0x007F007Fu, ex = 0x43004300u;
    out[6] = fma2((__byte_perm(la << 5, lb << 5, 0x0602) & m7) | ex, one, off);
    out[5] = fma2((__byte_perm(la << 6, lb << 6, 0x0703) & m7) | ex, one, off);
    out[4] = fma2((__byte_perm(la >> 1, lb >> 1, 0x0703) & m7) | ex, one, off);
    out[3] = fma2((__byte_perm(ua, ub, 0x0400) & m7) | ex, one, off);
    out[2] = fma2((__byte_perm(ua << 1, ub << 1, 0x0501) & m7) | ex, one, off);
    out[1] = fma2((__byte_perm(ua << 2, ub << 2, 0x0602) & m7) | ex, one, off);
    // the leading digit is at most 128: 0x4300 + 128 is the BF16 number 256
    out[0] = fma2((__byte_perm(ua << 3, ub << 3, 0x0703) & 0x00FF00FFu) | ex, one, sgn ^ 0xC300C300u);
  } else {  // T = 9: |x| 2^(63 - e)
    constexpr unsigned long long bias = 64ull * (((1ull << (7 * (T - 1))) - 1) / 127);
    asm("shr.u64 %0, %1, %2;" : "=l"(wa) : "l"(Ma), "r"(sa));
    asm("shr.u64 %0, %1, %2;" : "=l"(wb) : "l"(Mb), "r"(sb));
    wa = (wa >> 1) + (wa & 1) + bias;
    wb = (wb >> 1) + (wb & 1) + bias;
#pragma unroll
    for (int i = 0; i < T; ++i) {  // digit i from the least significant end
      const uint32_t m = i == T - 1 ? 0xFFu : 0x7Fu;
      const uint32_t pk = ((uint32_t)(wa >> (7 * i)) & m) | (((uint32_t)(wb >> (7 * i)) & m) << 16) | 0x43004300u;
      out[T - 1 - i] = fma2(pk, one, sgn ^ (i == T - 1 ? 0xC300C300u : 0xC340C340u));
    }
  }
}

// t 2^sc rounded to nearest even, on the bit pattern (the conversion
// instruction runs on the few FP64 units)
__device__ __forceinline__ double scaled_double(long long t, int sc) {
  if (t == 0) return 0.0;
  const unsigned long long u = (unsigned long long)(t < 0 ? -t : t);
  const int lz = __clzll((long long)u);
  const int E = 1086 - lz + sc;  // biased exponent of the leading bit
  if (E < 1 || E > 2045) return ldexp(__ll2double_rn(t), sc);
  const unsigned long long nrm = u << lz;
  unsigned long long m = nrm >> 11;
  const uint32_t rem = (uint32_t)nrm & 0x7FFu;
  m += (rem > 0x400u || (rem == 0x400u && (m & 1ull))) ? 1ull : 0ull;
  // m has its leading bit at 52 (53 after a carry): adding it moves the exponent along
  const unsigned long long bits = ((unsigned long long)(E - 1) << 52) + m;
  return __longlong_as_double((long long)(bits | ((unsigned long long)t & 0x8000000000000000ull)));
}

template <int T>
__device__ __forceinline__ void tmem_wait_regs(uint32_t (&r)[T][4]) {
  // the registers pass through the wait, so no use of them can move above it
#pragma unroll
  for (int d = 0; d < T; ++d)
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[d][0]), "+r"(r[d][1]), "+r"(r[d][2]), "+r"(r[d][3])::"memory");
}

}  // namespace

// One side of a product: element (row, k) of type `type` at p[k + row ld]
// (k contiguous) or p[row + k ld] (rows contiguous); exp: exponent per row.
struct EmuSide {
  const void* p;
  int64_t ld;
  const int* exp;
  int32_t type;
  int32_t vec;  // two neighbouring k as one aligned load
};

struct EmuMm {
  int64_t M, N;          // C is M x N
  EmuSide a[2];          // A: one block, or the two blocks of a lift
  int64_t K[2];          // their K extents
  int nseg;
  EmuSide b;             // B read directly (Gram form)
  const uint8_t* blob[2];  // B as sliced stage images, per block
  const int* bexp[2];
  int ntn, nch;          // column tiles, 16-column chunks of N
  int64_t main_rows;     // rows covered by the main tiles
  int main_tiles, tiles;
  int left_w;            // the remaining M - main_rows rows as a tile width (Gram form), 0: none
  int ranges, per;       // K ranges and their stages
  int items;
  int max_w;             // widest tile
  int mode;              // 0 store, 1 atomic add, 2 partial tiles
  double* C;
  int64_t ldc;
  double* part;          // [item][64 columns][128 rows]
};

namespace {

// column tile jt of a.ntn over a.nch chunks of 16 columns: sizes differ by one chunk at most
__device__ __forceinline__ void col_tile(int ntn, int nch, int jt, int& n0, int& w) {
  const int q = nch / ntn, r = nch % ntn;
  n0 = 16 * (jt * q + min(jt, r));
  w = 16 * (q + (jt < r ? 1 : 0));
}

// Entries on their way to the slicer, by storage class: wide (FP64, 64 raw
// bits) or narrow (FP32, BF16, E4M3: 32 raw bits, the type known at run time).
template <bool kWide> using RawT = std::conditional_t<kWide, unsigned long long, uint32_t>;

// f(TS{}) for the storage types of a class
template <bool kWide, typename F>
__device__ __forceinline__ void with_type(int type, F f) {
  if constexpr (kWide) {
    f(double{});
  } else {
    switch (type) {
      case RR_F32: f(float{}); break;
      case RR_BF16: f(__nv_bfloat16{}); break;
      default: f(e4m3b_t{}); break;
    }
  }
}
__device__ __forceinline__ float narrow_val(int type, uint32_t r) {
  if (type == RR_E4M3) return e4m3b_value((unsigned char)r);
  return __uint_as_float(type == RR_BF16 ? r << 16 : r);
}
// an entry as slice_pair takes it; scale: up_scale of its row
template <bool kWide>
__device__ __forceinline__ double raw_val(int type, RawT<kWide> r, float scale) {
  if constexpr (kWide) return __longlong_as_double((long long)r);
  else return f32_exact(narrow_val(type, r) * scale);
}

// A finished accumulation group: its sums, combined and scaled, to the output
// (store, add, or atomic add).  This warp's 32 TMEM lanes and quarter of the
// columns; accempty is released as soon as they are read.  Out of line: it
// runs once per group and must not cost the slicing loop its registers.
struct ReadOut {
  uint32_t taddr;        // TMEM address of the first column of digit sum 0
  int w, quarter;        // columns of the tile (distance of the sums), columns of this warp
  int ncols;             // of which exist
  int er;                // exponent of this thread's row
  const int* ec;         // exponents of this warp's columns
  double* out;
  int64_t ldo;
  int mode;              // 0 store, 1 atomic add, 2 add
};
struct Pending {  // a group to be read out, as its warp noted it
  double* out;    // row 0 of the tile, first column of the warp
  int64_t ldo;
  int w, rows, cols, mode, buf;
};
template <int T>
__device__ __noinline__ void read_group(const ReadOut q, uint64_t* accempty) {
#pragma unroll 1
  for (int c4 = 0; c4 < q.quarter; c4 += 4) {
    uint32_t r[T][4];
#pragma unroll
    for (int d = 0; d < T; ++d) tmem_ld_32x32b_x4(q.taddr + (uint32_t)(d * q.w + c4), r[d]);
    double old[4];  // of an add, in flight while the sums are combined
#pragma unroll
    for (int j = 0; j < 4; ++j) old[j] = q.mode == 2 && c4 + j < q.ncols ? q.out[(c4 + j) * q.ldo] : 0.0;
    tmem_wait_regs<T>(r);
    if (c4 + 4 >= q.quarter) {  // the accumulators are read: the next group may start
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if ((threadIdx.x & 31) == 0) mbar_arrive(accempty);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int S[T];
#pragma unroll
      for (int d = 0; d < T; ++d) S[d] = __float2int_rn(__uint_as_float(r[d][j]));
      // pairs of neighbouring sums fit 32 bits (bounds at the head of this file)
      const long long hi = (long long)(S[0] * 128 + S[1]) * 16384 + (S[2] * 128 + S[3]);
      long long lo;
      if (T == 7) lo = (long long)(S[4] * 128 + S[5]) * 128 + S[6];
      else lo = ((long long)(S[4] * 128 + S[5]) * 16384 + (S[6] * 128 + S[T == 7 ? 6 : 7])) * 128 + S[T - 1];
      // the lowest bits of the exact sum (2^-53 of the scales for T = 7) round away
      constexpr int sh = EmuConst<T>::base_shift;
      const long long t = (hi << (7 * (T - 4) - sh)) + ((lo + (1ll << (sh - 1))) >> sh);
      const int e = q.ec[c4 + j];
      double v = scaled_double(t, q.er + e - 7 * (T + 1) + sh);
      if (q.er == kExpInf || e == kExpInf) v = __longlong_as_double(0x7FF8000000000000ll);
      if (c4 + j < q.ncols) {
        double* o = q.out + (c4 + j) * q.ldo;
        if (q.mode == 1) atomicAdd(o, v);
        else *o = q.mode == 2 ? old[j] + v : v;
      }
    }
  }
}

// kMC: rows of A contiguous (else k); kPre: B as stage images (else read and
// sliced like A, k contiguous); kW1, kW2: storage classes of A and B, or with
// rows contiguous of the first and second block (template parameters, so that
// one kernel's registers serve one slicing loop, or two where they differ).
template <int T, bool kMC, bool kPre, bool kW1, bool kW2>
__global__ void __launch_bounds__(kThreads, 1) k_emu_mm(const __grid_constant__ EmuMm a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t a_bytes = T * kRows * 64;
  const uint32_t stage_bytes = a_bytes + T * a.max_w * 64;
  __shared__ __align__(8) uint64_t full[kRing], bfull[kRing], empty[kRing], accfull, accempty, segbar, fin;
  __shared__ uint32_t s_tmem;
  __shared__ int sea[3][kRows], seb[3][64];  // exponents of three segments: see below
  __shared__ Pending spend[kSlicers];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t tcols = 32;
  while (tcols < (uint32_t)(T * a.max_w)) tcols <<= 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRing; ++s) {
      mbar_init(&full[s], kSlicers);
      mbar_init(&bfull[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accfull, 1);
    mbar_init(&accempty, kSlicers);
    mbar_init(&segbar, kSlicers);
    mbar_init(&fin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kSlicers) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;

  // stages, accumulation groups and segments so far (every role counts alike)
  int it = 0, grp = 0, seq = 0;
  bool ok = true;

  if (warp == kSlicers) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      for (int item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
        const int range = item / a.tiles, tile = item % a.tiles;
        int n0, w = a.left_w;
        if (tile < a.main_tiles) col_tile(a.ntn, a.nch, tile % a.ntn, n0, w);
        const int nqmax = 256 / w;
        const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kRows >> 4) << 24);
        const uint32_t nstep = (uint32_t)(w >> 3) << 17;  // N field of one digit's columns
        for (int seg = 0; seg < a.nseg && ok; ++seg) {
          const int stages = (int)((a.K[seg] + kKB - 1) / kKB);
          const int st0 = range * a.per, nst = min(stages, st0 + a.per) - st0;
          const int kg = group_stages<T>(nst);
          for (int st = 0; st < nst; ++st) {
            const bool first = st % kg == 0;
            if (first && grp > 0 && !(ok = emu_wait(&accempty, (grp - 1) & 1))) break;
            const int s = it & 1;
            const uint32_t par = (it >> 1) & 1;
            if (!(ok = emu_wait(&full[s], par))) break;
            if (kPre && !(ok = emu_wait(&bfull[s], par))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sa = smem_u32(base + (size_t)s * stage_bytes);
            const uint64_t ad0 = sdesc_sw64(sa), bd0 = sdesc_sw64(sa + a_bytes);
#pragma unroll
            for (int kk = 0; kk < kKB / 16; ++kk) {
#pragma unroll
              for (int p = 0; p < T; ++p) {
                const uint64_t ad = ad0 + (uint64_t)(p * (kRows * 64 / 16) + 2 * kk);
                const uint32_t accum = (first && kk == 0 && p == 0) ? 0u : 1u;
                const int n1 = min(nqmax, T - p), n2 = T - p - n1;  // at most two runs of digits (T w <= 2 * 256)
                umma_bf16(tmem + (uint32_t)(p * w), ad, bd0 + (uint64_t)(2 * kk), idesc0 + (uint32_t)n1 * nstep, accum);
                if (n2 > 0)
                  umma_bf16(tmem + (uint32_t)((p + n1) * w), ad, bd0 + (uint64_t)(n1 * w * 4 + 2 * kk),
                            idesc0 + (uint32_t)n2 * nstep, accum);
              }
            }
            umma_commit(&empty[s]);
            if (st % kg == kg - 1 || st == nst - 1) {
              umma_commit(&accfull);
              ++grp;
            }
            ++it;
          }
        }
      }
      // arrives once every MMA issued above is complete, also after an error,
      // so TMEM is never freed under a running MMA
      umma_commit(&fin);
      emu_drain(&fin, 0);
    }
    __syncwarp();
  } else {
    // ---------------- slicing and epilogue ----------------
    const int tid = threadIdx.x;
    const int rg = warp & 3, qc = warp >> 2;  // 32 rows (also TMEM lanes), quarter of the K entries / of the columns
    const int trow = rg * 32 + lane;
    // k contiguous: two k of rows r0 + 32 i of A (i < 4) and columns r0 + 32 i of B (i < 2)
    const int r0 = 2 * warp + (lane >> 4), k2 = 2 * (lane & 15);
    constexpr int NA = 8, NB = (!kMC && !kPre) ? 4 : 0;  // entries of A and B a thread slices per stage
    // FP64 entries of the next stage wait in this thread's slots (asynchronous
    // copies), narrow ones in registers
    unsigned char* const raw = base + (size_t)kRing * stage_bytes;
    // A finished group, not yet read out (pend): the warps first slice the next
    // two stages (all the ring holds) and then read it, so that the tensor core
    // finds work as soon as its accumulators are free.  Its exponents stay in
    // their table meanwhile: three tables, as a warp can be up to two segments
    // past the group that another one still reads out.
    bool pend = false;
    int psince = 0;
    auto read_out = [&]() -> bool {
      if (!emu_wait_warp(&accfull, grp & 1)) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const Pending& p = spend[warp];
      ReadOut q;
      q.w = p.w;
      q.quarter = p.w >> 2;
      q.taddr = tmem + ((uint32_t)(rg * 32) << 16) + (uint32_t)(qc * q.quarter);
      q.er = sea[p.buf][trow];
      q.ec = &seb[p.buf][qc * q.quarter];
      q.out = p.out + trow;
      q.ldo = p.ldo;
      q.ncols = trow < p.rows ? p.cols : 0;
      q.mode = p.mode;
      read_group<T>(q, &accempty);
      ++grp;
      pend = false;
      return true;
    };

    for (int item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
      const int range = item / a.tiles, tile = item % a.tiles;
      const bool swp = tile >= a.main_tiles;  // a tile of the remaining rows: the sides trade places
      int m0, n0, w;
      if (!swp) {
        m0 = tile / a.ntn * kRows;
        col_tile(a.ntn, a.nch, tile % a.ntn, n0, w);
      } else {
        m0 = (tile - a.main_tiles) * kRows;
        n0 = (int)a.main_rows;
        w = a.left_w;
      }
      const int rows_lim = (int)(swp ? a.N : a.main_rows), cols_lim = (int)(swp ? a.M : a.N);

      // one segment with the storage classes of its sides fixed
      auto run_seg = [&](auto wa_, auto wb_, int seg) -> bool {
        constexpr bool WA = decltype(wa_)::value, WB = decltype(wb_)::value;
        const EmuSide A = swp ? a.b : a.a[seg];
        const EmuSide B = swp ? a.a[0] : a.b;
        const int K = (int)a.K[seg];
        const int stages = (K + kKB - 1) / kKB;
        const int st0 = range * a.per, nst = min(stages, st0 + a.per) - st0;
        const int kg = group_stages<T>(nst);
        const int buf = seq % 3;
        // exponents of the tile's rows and columns.  Rows and columns past the
        // end repeat the last one: their results are never read.
        if (tid < kRows) {
          sea[buf][tid] = max(__ldg(A.exp + min(m0 + tid, rows_lim - 1)), kExpNone);
        } else if (tid < kRows + w) {
          const int j = tid - kRows;
          const int* be = kPre ? a.bexp[seg] : B.exp;
          seb[buf][j] = max(__ldg(be + min(n0 + j, cols_lim - 1)), kExpNone);
        }
        // (an mbarrier and not a named barrier: its wait is bounded)
        __syncwarp();
        if (lane == 0) mbar_arrive(&segbar);
        if (!emu_wait_warp(&segbar, seq & 1)) return false;
        ++seq;
        // FP64 rows or columns near the type's lowest exponent among them
        bool look_a = false, look_b = false;
        if (kMC) {
          look_a = sea[buf][trow] < kTiny64;
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) look_a |= sea[buf][r0 + 32 * i] < kTiny64;
          if (!kPre)
#pragma unroll
            for (int i = 0; i < 2; ++i)
              if (2 * warp + 32 * i < w) look_b |= seb[buf][r0 + 32 * i] < kTiny64;
        }
        look_a = WA && __any_sync(0xffffffffu, look_a);
        look_b = WB && __any_sync(0xffffffffu, look_b);

        [[maybe_unused]] uint32_t na[WA ? 1 : NA], nb[(WB || NB == 0) ? 1 : NB];  // narrow entries of the next stage
        auto narrow_load = [&](auto ts, const EmuSide& S, int i, int r, int k0, uint32_t& x, uint32_t& y) {
          using TS = decltype(ts);
          const TS* q = (const TS*)S.p + k0 + k2 + r * S.ld;
          if (k0 + kKB <= K && S.vec) {
            Raw<TS>::ld2(q, x, y);
          } else {
            x = k0 + k2 < K ? Raw<TS>::ld(q) : 0u;
            y = k0 + k2 + 1 < K ? Raw<TS>::ld(q + 1) : 0u;
          }
        };
        auto fetch_pair = [&](const EmuSide& S, int r, int k0, unsigned char* dst) {
          const double* q = (const double*)S.p + k0 + k2 + r * S.ld;
          if (k0 + kKB <= K && S.vec) {
            cp_async<16>(dst, q, 16);
          } else {  // entries past the end are zeros (and their addresses not used)
            const int left = K - (k0 + k2);
            cp_async<8>(dst, left >= 1 ? q : (const double*)S.p, left >= 1 ? 8 : 0);
            cp_async<8>(dst + 8, left >= 2 ? q + 1 : (const double*)S.p, left >= 2 ? 8 : 0);
          }
        };
        // starts the reads of stage st
        auto fetch = [&](int st) {
          const int k0 = (st0 + st) * kKB;
          if constexpr (kMC) {
            const int64_t at = min(m0 + trow, rows_lim - 1) + (int64_t)(k0 + qc * 8) * A.ld;
            const int left = K - (k0 + qc * 8);
            if constexpr (WA) {
              const double* q = (const double*)A.p + at;
              if (left >= 8) {
#pragma unroll
                for (int c = 0; c < 8; ++c) cp_async<8>(raw + (c * 512 + tid) * 8, q + c * A.ld, 8);
              } else {
#pragma unroll
                for (int c = 0; c < 8; ++c)
                  cp_async<8>(raw + (c * 512 + tid) * 8, c < left ? q + c * A.ld : (const double*)A.p, c < left ? 8 : 0);
              }
            } else {
              with_type<false>(A.type, [&](auto ts) {
                using TS = decltype(ts);
                const TS* q = (const TS*)A.p + at;
#pragma unroll
                for (int c = 0; c < 8; ++c) na[c] = c < left ? Raw<TS>::ld(q + c * A.ld) : 0u;
              });
            }
          } else {
            if constexpr (WA) {
#pragma unroll
              for (int i = 0; i < 4; ++i)
                fetch_pair(A, min(m0 + r0 + 32 * i, rows_lim - 1), k0, raw + (i * 512 + tid) * 16);
            } else {
              with_type<false>(A.type, [&](auto ts) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  narrow_load(ts, A, i, min(m0 + r0 + 32 * i, rows_lim - 1), k0, na[2 * i], na[2 * i + 1]);
              });
            }
            if constexpr (!kPre) {
              if constexpr (WB) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                  if (2 * warp + 32 * i < w)
                    fetch_pair(B, min(n0 + r0 + 32 * i, cols_lim - 1), k0, raw + 32768 + (i * 512 + tid) * 16);
              } else {
                with_type<false>(B.type, [&](auto ts) {
#pragma unroll
                  for (int i = 0; i < 2; ++i)
                    if (2 * warp + 32 * i < w)
                      narrow_load(ts, B, i, min(n0 + r0 + 32 * i, cols_lim - 1), k0, nb[2 * i], nb[2 * i + 1]);
                });
              }
            }
          }
        };
        fetch(0);
        for (int st = 0; st < nst; ++st) {
          // this stage's entries to registers, the next one's reads under way
          RawT<WA> xa[NA];
          RawT<WB> xb[NB + 1];
          asm volatile("cp.async.wait_all;" ::: "memory");
          if constexpr (WA) {
            if constexpr (kMC) {
#pragma unroll
              for (int c = 0; c < 8; ++c) xa[c] = *reinterpret_cast<const unsigned long long*>(raw + (c * 512 + tid) * 8);
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(raw + (i * 512 + tid) * 16);
                xa[2 * i] = v.x;
                xa[2 * i + 1] = v.y;
              }
            }
          } else {
#pragma unroll
            for (int i = 0; i < NA; ++i) xa[i] = na[i];
          }
          if constexpr (NB > 0) {
            if constexpr (WB) {
#pragma unroll
              for (int i = 0; i < 2; ++i)
                if (2 * warp + 32 * i < w) {
                  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(raw + 32768 + (i * 512 + tid) * 16);
                  xb[2 * i] = v.x;
                  xb[2 * i + 1] = v.y;
                }
            } else {
#pragma unroll
              for (int i = 0; i < NB; ++i) xb[i] = nb[i];
            }
          }
          if (st + 1 < nst) fetch(st + 1);
          const int s = it & 1;
          if (!emu_wait_warp(&empty[s], ((uint32_t)(it >> 1) & 1) ^ 1)) return false;
          unsigned char* sa = base + (size_t)s * stage_bytes;
          if (kPre && tid == 0) {
            const int64_t img = (int64_t)T * w * 64;  // bytes of one stage image of B
            mbar_expect_tx(&bfull[s], (uint32_t)img);
            bulk_load(sa + a_bytes, a.blob[seg] + (int64_t)stages * T * 64 * n0 + (st0 + st) * img, (uint32_t)img,
                      &bfull[s]);
          }
          if constexpr (WA)
            if (look_a) {
#pragma unroll
              for (int i = 0; i < NA; ++i)
                xa[i] = (unsigned long long)__double_as_longlong(
                    up_entry(__longlong_as_double((long long)xa[i]), sea[buf][kMC ? trow : r0 + 32 * (i >> 1)]));
            }
          if constexpr (kMC) {
            const int er = sea[buf][trow], e = up_exp<WA>(er);
            const float f = up_scale(er);
            uint32_t dg[4][T];
#pragma unroll
            for (int c = 0; c < 4; ++c)
              slice_pair<T>(raw_val<WA>(A.type, xa[2 * c], f), raw_val<WA>(A.type, xa[2 * c + 1], f), e, e, dg[c]);
            // 64-byte rows, 16-byte chunk index XOR (row / 2) % 4
            unsigned char* dst = sa + trow * 64 + ((qc ^ ((trow >> 1) & 3)) << 4);
#pragma unroll
            for (int p = 0; p < T; ++p)
              *reinterpret_cast<uint4*>(dst + p * (kRows * 64)) = make_uint4(dg[0][p], dg[1][p], dg[2][p], dg[3][p]);
          } else {
            // (32 i rows further on the swizzle is the same)
            unsigned char* dst = sa + r0 * 64 + ((((lane & 15) >> 2) ^ ((r0 >> 1) & 3)) << 4) + (lane & 3) * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int er = sea[buf][r0 + 32 * i], e = up_exp<WA>(er);
              const float f = up_scale(er);
              uint32_t dg[T];
              slice_pair<T>(raw_val<WA>(A.type, xa[2 * i], f), raw_val<WA>(A.type, xa[2 * i + 1], f), e, e, dg);
#pragma unroll
              for (int p = 0; p < T; ++p) *reinterpret_cast<uint32_t*>(dst + p * (kRows * 64) + i * 2048) = dg[p];
            }
            if constexpr (NB > 0) {
              dst += a_bytes;
#pragma unroll
              for (int i = 0; i < 2; ++i)
                if (2 * warp + 32 * i < w) {
                  const int ec = seb[buf][r0 + 32 * i], e = up_exp<WB>(ec);
                  const float f = up_scale(ec);
                  if constexpr (WB)
                    if (look_b) {
#pragma unroll
                      for (int h = 0; h < 2; ++h)
                        xb[2 * i + h] = (unsigned long long)__double_as_longlong(
                            up_entry(__longlong_as_double((long long)xb[2 * i + h]), ec));
                    }
                  uint32_t dg[T];
                  slice_pair<T>(raw_val<WB>(B.type, xb[2 * i], f), raw_val<WB>(B.type, xb[2 * i + 1], f), e, e, dg);
#pragma unroll
                  for (int p = 0; p < T; ++p) *reinterpret_cast<uint32_t*>(dst + p * (w * 64) + i * 2048) = dg[p];
                }
            }
          }
          // generic-proxy writes -> the tensor core's (async proxy) reads
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[s]);
          ++it;
          const bool last = st % kg == kg - 1 || st == nst - 1;
          if (pend && (++psince == kRing || last) && !read_out()) return false;
          if (last) {
            pend = true;
            psince = 0;
            if (lane == 0) {
              Pending p;
              const int c0 = qc * (w >> 2);
              p.buf = buf;
              p.w = w;
              p.rows = a.mode == 2 ? kRows : rows_lim - m0;
              p.cols = a.mode == 2 ? w >> 2 : (int)a.N - n0 - c0;
              p.mode = a.mode == 1 ? 1 : seg > 0 || st >= kg ? 2 : 0;
              p.out = a.mode == 2 ? a.part + (size_t)item * (64 * kRows) + c0 * kRows : a.C + m0 + (n0 + c0) * a.ldc;
              p.ldo = a.mode == 2 ? kRows : a.ldc;
              spend[warp] = p;
            }
            __syncwarp();
          }
        }
        return true;
      };
      constexpr std::bool_constant<kW1> w1{};
      constexpr std::bool_constant<kW2> w2{};
      for (int seg = 0; seg < a.nseg && ok; ++seg) {
        if constexpr (kW1 == kW2) ok = run_seg(w1, w1, seg);
        else if (kMC ? seg > 0 : swp) ok = run_seg(w2, w1, seg);
        else ok = run_seg(w1, w2, seg);
      }
    }
    if (ok && pend) ok = read_out();
    if (!ok && kPre && threadIdx.x == 0)
      // after an error: the copies of the last stages may still be in flight
      for (int i = it > kRing ? it - kRing : 0; i <= it; ++i) emu_drain(&bfull[i & 1], (i >> 1) & 1);
    __syncwarp();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kSlicers) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
  }
}

// B (K x N FP64, column-major) as stage images: for every column tile and
// every 32 rows of K the T digit planes, 64-byte-swizzled as the MMA reads
// them.  One block per column (pad columns write zeros): the column's exponent,
// then its digits, 8 rows of K a thread.
template <int T>
__global__ void __launch_bounds__(256) k_emu_bslice(int64_t K, int64_t N, const double* __restrict__ B, int64_t ldb,
                                                    int ntn, int nch, int stages, uint8_t* __restrict__ blob,
                                                    int* __restrict__ bexp) {
  __shared__ int sm[8];
  const int64_t j = blockIdx.x;
  const bool jv = j < N;
  int e = kExpNone;
  if (jv)
    for (int64_t k = threadIdx.x; k < K; k += 256) e = max(e, exp_of(__ldg(B + k + j * ldb)));
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = e;
  __syncthreads();
  e = sm[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) e = max(e, sm[i]);
  if (threadIdx.x == 0 && jv) bexp[j] = e;
  // the tile of column j
  const int chunk = (int)(j >> 4), q = nch / ntn, r = nch % ntn;
  const int jt = chunk < r * (q + 1) ? chunk / (q + 1) : r + (chunk - r * (q + 1)) / q;
  int n0, w;
  col_tile(ntn, nch, jt, n0, w);
  const int jl = (int)j - n0;
  uint8_t* tile = blob + (int64_t)stages * T * 64 * n0;
  for (int64_t g = threadIdx.x; g < (int64_t)stages * 4; g += 256) {
    const int64_t k0 = g * 8;
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = jv && k0 + u < K ? __ldg(B + k0 + u + j * ldb) : 0.0;
    uint32_t dg[4][T];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      slice_pair<T>(up_entry(x[2 * u], e), up_entry(x[2 * u + 1], e), up_exp<true>(e), up_exp<true>(e), dg[u]);
    uint8_t* dst = tile + (g >> 2) * ((int64_t)T * w * 64) + jl * 64 + (((int)(g & 3) ^ ((jl >> 1) & 3)) << 4);
#pragma unroll
    for (int p = 0; p < T; ++p)
      *reinterpret_cast<uint4*>(dst + p * (w * 64)) = make_uint4(dg[0][p], dg[1][p], dg[2][p], dg[3][p]);
  }
}

// Exponents of the largest entry of every column (atomic maxima over row
// chunks, so that a tall block's few columns fill the GPU; e then starts very
// negative; a plain store with one chunk).  8 loads in flight a thread; bound by HBM.
template <typename TS>
__global__ void __launch_bounds__(256) k_emu_col_exp(int64_t n, const TS* __restrict__ X, int64_t ldx, int64_t rpc,
                                                     int* __restrict__ e) {
  const int64_t j = blockIdx.y, r0 = (int64_t)blockIdx.x * rpc, r1 = min(n, r0 + rpc);
  const TS* x = X + j * ldx;
  int mx = kExpNone;
  for (int64_t i = r0 + threadIdx.x; i < r1; i += 8 * 256) {
    typename Raw<TS>::R v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = i + u * 256 < r1 ? Raw<TS>::ld(x + i + u * 256) : 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) mx = max(mx, exp_raw<TS>(v[u]));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (gridDim.x > 1) {
    if ((threadIdx.x & 31) == 0) atomicMax(e + j, mx);
    return;
  }
  __shared__ int sm[8];
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) mx = max(mx, sm[w]);
    e[j] = mx;
  }
}

// Exponents of the largest entry of every row of a column-major block (lane =
// row, 16 columns a thread, atomic maxima; e starts very negative).  kMore: the
// grid strides over more columns than it has blocks for.
template <typename TS, bool kMore>
__global__ void __launch_bounds__(256) k_emu_row_exp(int64_t m, int64_t n, const TS* __restrict__ A, int64_t lda,
                                                     int* __restrict__ e) {
  const int64_t i = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  int64_t j0 = ((int64_t)blockIdx.y * 8 + (threadIdx.x >> 5)) * 16;
  if (i >= m || j0 >= n) return;
  do {
    typename Raw<TS>::R v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = j0 + u < n ? Raw<TS>::ld(A + i + (j0 + u) * lda) : 0;
    int mx = kExpNone;
#pragma unroll
    for (int u = 0; u < 16; ++u) mx = max(mx, exp_raw<TS>(v[u]));
    atomicMax(e + i, mx);
    j0 += (int64_t)gridDim.y * 128;
  } while (kMore && j0 < n);
}

// G (p x q) = the sum of the K ranges' partial tiles in a fixed order (+ G).
__global__ void __launch_bounds__(256) k_emu_gram_reduce(int64_t p, int64_t q, int ntn, int nch, int64_t main_rows,
                                                         int main_tiles, int tiles, int ranges,
                                                         const double* __restrict__ part, double* __restrict__ G,
                                                         int64_t ldg, int accum) {
  __shared__ double sm[8][32];
  const int il = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + il, j = blockIdx.y;
  double s = 0.0;
  if (i < p) {
    int t, r, c;
    if (i < main_rows) {
      const int chunk = (int)(j >> 4), qq = nch / ntn, rr_ = nch % ntn;
      const int jt = chunk < rr_ * (qq + 1) ? chunk / (qq + 1) : rr_ + (chunk - rr_ * (qq + 1)) / qq;
      int n0, w;
      col_tile(ntn, nch, jt, n0, w);
      t = (int)(i / kRows) * ntn + jt;
      r = (int)(i % kRows);
      c = (int)j - n0;
    } else {  // the sides traded places
      t = main_tiles + (int)(j / kRows);
      r = (int)(j % kRows);
      c = (int)(i - main_rows);
    }
    const double* src = part + (size_t)t * (64 * kRows) + (size_t)c * kRows + r;
    const size_t step = (size_t)tiles * (64 * kRows);
    int x = g;
    for (; x + 24 < ranges; x += 32) {  // four loads in flight
      const double v0 = src[x * step], v1 = src[(x + 8) * step], v2 = src[(x + 16) * step], v3 = src[(x + 24) * step];
      s += v0;
      s += v1;
      s += v2;
      s += v3;
    }
    for (; x < ranges; x += 8) s += src[x * step];
  }
  sm[g][il] = s;
  __syncthreads();
  if (g == 0 && i < p) {
#pragma unroll
    for (int x = 1; x < 8; ++x) s += sm[x][il];
    double* out = G + i + j * ldg;
    *out = accum ? *out + s : s;
  }
}

__global__ void k_zero_f64(int64_t M, int64_t N, double* __restrict__ C, int64_t ldc) {
  const int64_t j = blockIdx.y;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
    C[i + j * ldc] = 0.0;
}

// the ring, and the slots of the next stage's FP64 entries (A, and B in the Gram form)
template <int T, bool kPre>
size_t emu_smem(int max_w) {
  return 1024 + (size_t)kRing * T * 64 * (kRows + max_w) + (kPre ? 32768 : 49152);
}

template <int T, bool kMC, bool kPre, bool kW1 = true, bool kW2 = true>
rr_status launch_mm(cudaStream_t s, const EmuMm& a) {
  const size_t smem = emu_smem<T, kPre>(a.max_w);
  RR_TRY(tc_prepare_attributes());
  const int grid = std::min(a.items, num_sms());
  k_emu_mm<T, kMC, kPre, kW1, kW2><<<grid, kThreads, smem, s>>>(a);
  return check_launch("emu_mm");
}

// the launch for the storage types of two sides (or blocks)
template <int T, bool kMC, bool kPre>
rr_status launch_mm_types(cudaStream_t s, const EmuMm& a, int32_t t1, int32_t t2) {
  const bool w1 = t1 == RR_F64, w2 = t2 == RR_F64;
  if (w1) return w2 ? launch_mm<T, kMC, kPre, true, true>(s, a) : launch_mm<T, kMC, kPre, true, false>(s, a);
  return w2 ? launch_mm<T, kMC, kPre, false, true>(s, a) : launch_mm<T, kMC, kPre, false, false>(s, a);
}

template <int T, bool kMC, bool kPre, bool kW1 = true, bool kW2 = true>
rr_status set_attr() {
  RR_CUDA(cudaFuncSetAttribute(k_emu_mm<T, kMC, kPre, kW1, kW2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)emu_smem<T, kPre>(EmuConst<T>::max_w)));
  return RR_OK;
}

// column tiles of N columns, at most max_w wide
void col_tiles(int64_t N, int max_w, EmuMm& a) {
  a.nch = (int)((N + 15) / 16);
  a.ntn = (a.nch * 16 + max_w - 1) / max_w;
  a.max_w = 16 * ((a.nch + a.ntn - 1) / a.ntn);
}

// K ranges: `tiles` tiles of `stages` stages over the SMs.  An item costs its
// stages, about 2 stages for each read-out of its accumulators (one per kg
// stages) and 2 to start.
void k_ranges(int tiles, int64_t stages, int kg, int cap, EmuMm& a) {
  const int64_t sms = num_sms();
  int64_t best = 0, best_cost = INT64_MAX;
  int64_t rmax = std::min<int64_t>(stages, (8 * sms + tiles - 1) / tiles);
  if (cap > 0) rmax = std::min<int64_t>(rmax, cap);
  for (int64_t r = 1; r <= rmax; ++r) {
    const int64_t per = (stages + r - 1) / r, used = (stages + per - 1) / per;
    const int64_t waves = (tiles * used + sms - 1) / sms;
    const int64_t cost = waves * (per + 2 * ((per + kg - 1) / kg) + 2);
    if (cost < best_cost) {
      best_cost = cost;
      best = used;
    }
  }
  a.per = (int)((stages + best - 1) / best);
  a.ranges = (int)((stages + a.per - 1) / a.per);
  a.items = tiles * a.ranges;
}

bool aligned_pairs(const void* p, int64_t ld, int32_t type) {
  const size_t e = dtype_size(type);
  return (uintptr_t)p % (2 * e) == 0 && ld % 2 == 0;
}

size_t blob_bytes(int64_t K, int64_t N, int T) {
  return align_up((size_t)((K + kKB - 1) / kKB) * T * 64 * ((N + 15) / 16 * 16)) + align_up((size_t)N * 4);
}

// digits a caller of `slices` 6-bit slices needs (see the bounds above)
int digits_for(int slices) { return slices <= 8 ? 7 : 9; }

template <int T>
rr_status slice_b(cudaStream_t s, int64_t K, int64_t N, const double* B, int64_t ldb, const EmuMm& a, void* mem,
                  const uint8_t** blob, const int** bexp) {
  const int stages = (int)((K + kKB - 1) / kKB);
  uint8_t* b = (uint8_t*)mem;
  int* e = (int*)((char*)mem + align_up((size_t)stages * T * 64 * a.nch * 16));
  k_emu_bslice<T><<<(unsigned)(a.nch * 16), 256, 0, s>>>(K, N, B, ldb, a.ntn, a.nch, stages, b, e);
  *blob = b;
  *bexp = e;
  return check_launch("emu B slices");
}

// Row chunks of the column exponents: about 8 blocks an SM over the columns, at
// least 2048 rows each; one up to 4096 rows, where e then needs no start value
// (a small Gram is bound by its launches: the memset is one of five).
int64_t col_exp_chunks(int64_t n, int64_t c) {
  if (n <= 4096) return 1;
  return std::max<int64_t>(1, std::min<int64_t>((n + 2047) / 2048, (8 * (int64_t)num_sms() + c - 1) / c));
}
constexpr int64_t kMaxGridY = 65535;
rr_status col_exps(cudaStream_t s, int32_t type, int64_t n, int64_t c, const void* X, int64_t ldx, int* e) {
  int64_t chunks = col_exp_chunks(n, c);
  const int64_t rpc = (n + chunks - 1) / chunks;
  chunks = (n + rpc - 1) / rpc;
  // columns on y, in as many launches as that takes (an operator may have millions)
  for (int64_t j0 = 0; j0 < c; j0 += kMaxGridY) {
    const dim3 g((unsigned)chunks, (unsigned)std::min<int64_t>(c - j0, kMaxGridY));
    auto go = [&](auto ts) {
      using TS = decltype(ts);
      k_emu_col_exp<TS><<<g, 256, 0, s>>>(n, (const TS*)X + j0 * ldx, ldx, rpc, e + j0);
    };
    switch (type) {
      case RR_F64: go(double{}); break;
      case RR_F32: go(float{}); break;
      case RR_BF16: go(__nv_bfloat16{}); break;
      case RR_E4M3: go(e4m3b_t{}); break;
      default: return RR_ERR_ARG;
    }
    RR_TRY(check_launch("emu column exponents"));
  }
  return RR_OK;
}

rr_status row_exps(cudaStream_t s, int32_t type, int64_t n, int64_t c, const void* X, int64_t ldx, int* e) {
  const dim3 g((unsigned)((n + 31) / 32), (unsigned)std::min<int64_t>((c + 127) / 128, kMaxGridY));
  auto go = [&](auto ts) {
    using TS = decltype(ts);
    if (c > kMaxGridY * 128) k_emu_row_exp<TS, true><<<g, 256, 0, s>>>(n, c, (const TS*)X, ldx, e);
    else k_emu_row_exp<TS, false><<<g, 256, 0, s>>>(n, c, (const TS*)X, ldx, e);
  };
  switch (type) {
    case RR_F64: go(double{}); break;
    case RR_F32: go(float{}); break;
    case RR_BF16: go(__nv_bfloat16{}); break;
    case RR_E4M3: go(e4m3b_t{}); break;
    default: return RR_ERR_ARG;
  }
  return check_launch("emu row exponents");
}

// pair products of T digits, and the work of a launch for the profile
double pair_flops(int T, double M, double N, double K) { return 2.0 * M * N * K * (T * (T + 1) / 2); }

}  // namespace

rr_status emu_prepare_attributes() {
  RR_TRY((set_attr<7, true, true, true, true>()));
  RR_TRY((set_attr<7, true, true, true, false>()));
  RR_TRY((set_attr<7, true, true, false, true>()));
  RR_TRY((set_attr<7, true, true, false, false>()));
  RR_TRY((set_attr<7, false, true>()));
  RR_TRY((set_attr<7, false, false, true, true>()));
  RR_TRY((set_attr<7, false, false, true, false>()));
  RR_TRY((set_attr<7, false, false, false, true>()));
  RR_TRY((set_attr<7, false, false, false, false>()));
  RR_TRY((set_attr<9, true, true>()));
  return set_attr<9, false, true>();
}

// the kernel's error word (0 = ok); the caller synchronises s before it reads *host
rr_status emu_error_fetch(cudaStream_t s, int* host) {
  RR_CUDA(cudaMemcpyFromSymbolAsync(host, g_emu_error, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
  return RR_OK;
}
rr_status emu_error_clear(cudaStream_t s) {
  static const int zero = 0;
  RR_CUDA(cudaMemcpyToSymbolAsync(g_emu_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s));
  return RR_OK;
}

// ---------------------------------------------------------------------------
// products with a dense FP64 operator
// ---------------------------------------------------------------------------
size_t emu_operator_bytes(int64_t m, int64_t n, bool rows, bool cols) {
  return (rows ? align_up((size_t)m * 4) : 0) + (cols ? align_up((size_t)n * 4) : 0);
}

size_t emu_block_bytes(int64_t K, int64_t N, int slices) { return blob_bytes(K, N, digits_for(slices)); }

// The row and / or column exponents of A (m x n, column-major) into mem.
rr_status emu_prepare(cudaStream_t s, const double* A, int64_t m, int64_t n, int64_t lda, EmuOperator& op, void* mem,
                      bool rows, bool cols) {
  Arena ar(mem, emu_operator_bytes(m, n, rows, cols));
  op = EmuOperator{};
  op.m = m;
  op.n = n;
  op.A = A;
  op.lda = lda;
  RR_CUDA(cudaMemsetAsync(mem, 0x80, emu_operator_bytes(m, n, rows, cols), s));  // below every exponent
  if (rows) {
    op.rexp = ar.take<int>(m);
    RR_TRY(row_exps(s, RR_F64, m, n, A, lda, op.rexp));
  }
  if (cols) {
    op.cexp = ar.take<int>(n);
    RR_TRY(col_exps(s, RR_F64, m, n, A, lda, op.cexp));
  }
  return RR_OK;
}

// C (M x N FP64) = A X (trans = 0, M = m, K = n) or A^T X (trans = 1, M = n,
// K = m), X FP64 K x N column-major; mem: emu_block_bytes(K, N, slices).
rr_status emu_gemm(cudaStream_t s, const EmuOperator& op, int trans, int64_t N, const double* X, int64_t ldx,
                   double* C, int64_t ldc, int slices, void* mem) {
  const int64_t M = trans ? op.n : op.m, K = trans ? op.m : op.n;
  const int* aexp = trans ? op.cexp : op.rexp;
  if (!aexp || N <= 0 || N > 256 || ((uintptr_t)mem & 15) || M > 0x7fffffff || K > 0x7fffffff) return RR_ERR_ARG;
  const int T = digits_for(slices);
  EmuMm a{};
  a.M = M;
  a.N = N;
  a.K[0] = K;
  a.nseg = 1;
  a.a[0] = EmuSide{op.A, op.lda, aexp, RR_F64, aligned_pairs(op.A, op.lda, RR_F64) ? 1 : 0};
  a.b = a.a[0];
  col_tiles(N, T == 7 ? EmuConst<7>::max_w : EmuConst<9>::max_w, a);
  a.main_rows = M;
  a.main_tiles = a.tiles = (int)((M + kRows - 1) / kRows) * a.ntn;
  k_ranges(a.tiles, (K + kKB - 1) / kKB, T == 7 ? EmuConst<7>::kg : EmuConst<9>::kg, gemm_split_cap(), a);
  if (T == 7) RR_TRY(slice_b<7>(s, K, N, X, ldx, a, mem, &a.blob[0], &a.bexp[0]));
  else RR_TRY(slice_b<9>(s, K, N, X, ldx, a, mem, &a.blob[0], &a.bexp[0]));
  a.C = C;
  a.ldc = ldc;
  a.mode = a.ranges > 1 ? 1 : 0;
  if (a.mode == 1) {
    const dim3 gz((unsigned)std::min<int64_t>((M + 255) / 256, 1024), (unsigned)N);
    k_zero_f64<<<gz, 256, 0, s>>>(M, N, C, ldc);
    note_launches(1);
  }
  TcProfScope prof(s, 8.0 * M * K + 2.0 * T * K * N + 8.0 * M * N, pair_flops(T, (double)M, (double)N, (double)K), 1);
  if (T == 7) return trans ? launch_mm<7, false, true>(s, a) : launch_mm<7, true, true>(s, a);
  return trans ? launch_mm<9, false, true>(s, a) : launch_mm<9, true, true>(s, a);
}

// ---------------------------------------------------------------------------
// Ritz lift X (n x b) = S1 Y(0:p1, :) + S2 Y(p1:p1+p2, :) (Alg. 3 / Alg. 5
// "U~ = U Y").  Each block has its own row exponents (the refinement's
// correction columns have unit inf-norm while X's unit 2-norm columns have
// entries of 1 / sqrt(n): one exponent per row across both would leave X's
// entries only the bits below the correction block's) and its own sliced rows
// of Y.
// ---------------------------------------------------------------------------
size_t lift_emu_bytes(int64_t n, int64_t b, int64_t K) {
  // (two blocks round their K up separately)
  return 2 * align_up((size_t)n * 4) + blob_bytes(K, b, 7) + blob_bytes(kKB, b, 7) + 256;
}

// *done = false (nothing launched) when the shape is outside this path.  K that
// is no multiple of 8 is left to FP64 arithmetic, whose error is relative to the
// terms summed and not to the largest entries of rows and columns.
rr_status lift_emu(cudaStream_t s, int64_t n, int64_t b, int32_t t1, const void* S1, int64_t ld1, int64_t p1,
                   int32_t t2, const void* S2, int64_t ld2, int64_t p2, const double* Y, int64_t ldy, double* X,
                   int64_t ldx, void* mem, size_t mem_bytes, bool* done) {
  *done = false;
  if (!S2) p2 = 0;
  const int64_t K = p1 + p2;
  if (!mem || n <= 0 || n > 0x7fffff00ll || b <= 0 || b > 256 || K % 8 || K > 512 || p1 <= 0 ||
      ((uintptr_t)mem & 15))
    return RR_OK;
  if (mem_bytes < lift_emu_bytes(n, b, K)) return RR_OK;
  EmuMm a{};
  a.M = n;
  a.N = b;
  a.nseg = p2 > 0 ? 2 : 1;
  a.K[0] = p1;
  a.K[1] = p2;
  char* m = (char*)mem;
  int *e1 = (int*)m, *e2 = (int*)(m + align_up((size_t)n * 4));
  m += 2 * align_up((size_t)n * 4);
  RR_CUDA(cudaMemsetAsync(mem, 0x80, (p2 > 0 ? 2 : 1) * align_up((size_t)n * 4), s));  // below every exponent
  RR_TRY(row_exps(s, t1, n, p1, S1, ld1, e1));
  if (p2 > 0) RR_TRY(row_exps(s, t2, n, p2, S2, ld2, e2));
  a.a[0] = EmuSide{S1, ld1, e1, t1, 0};
  a.a[1] = EmuSide{S2, ld2, e2, t2, 0};
  a.b = a.a[0];
  col_tiles(b, 64, a);
  a.main_rows = n;
  a.main_tiles = a.tiles = a.items = (int)((n + kRows - 1) / kRows) * a.ntn;
  a.ranges = 1;
  a.per = 1 << 20;
  RR_TRY(slice_b<7>(s, p1, b, Y, ldy, a, m, &a.blob[0], &a.bexp[0]));
  if (p2 > 0) RR_TRY(slice_b<7>(s, p2, b, Y + p1, ldy, a, m + blob_bytes(p1, b, 7), &a.blob[1], &a.bexp[1]));
  a.C = X;
  a.ldc = ldx;
  TcProfScope prof(s, (double)n * (p1 * dtype_size(t1) + p2 * dtype_size(p2 > 0 ? t2 : t1)) + 14.0 * K * b + 8.0 * n * b,
                   pair_flops(7, (double)n, (double)b, (double)K), 1);
  RR_TRY((launch_mm_types<7, true, true>(s, a, t1, p2 > 0 ? t2 : t1)));
  *done = true;
  return RR_OK;
}

// ---------------------------------------------------------------------------
// Gram products G = X^T Y (X n x p, Y n x q, any storage type).
// ---------------------------------------------------------------------------
// (Row counts that are no multiple of 8 stay in FP64 arithmetic, as in the lift.)
bool emu_gram_supported(int64_t n, int64_t p, int64_t q) {
  return n >= 64 && n % 8 == 0 && p >= 1 && q >= 1 && p <= 4096 && q <= 4096 && n <= ((int64_t)1 << 30);
}

// Tiles: rows in blocks of 128 of X's columns; a remainder of at most 64 rows
// takes the other role (128 of Y's columns against the remainder as a column
// tile), which wastes less of the 128-row MMA than a nearly empty row tile.
static void gram_tiles(int64_t n, int64_t p, int64_t q, EmuMm& a) {
  const int64_t rem = p % kRows;
  a.M = p;
  a.N = q;
  a.K[0] = n;
  a.nseg = 1;
  col_tiles(q, 64, a);
  const bool left = p > kRows && rem > 0 && rem <= 64;
  a.main_rows = left ? p - rem : p;
  a.left_w = left ? (int)((rem + 15) / 16 * 16) : 0;
  a.main_tiles = (int)((a.main_rows + kRows - 1) / kRows) * a.ntn;
  a.tiles = a.main_tiles + (left ? (int)((q + kRows - 1) / kRows) : 0);
  if (a.left_w > a.max_w) a.max_w = a.left_w;
  k_ranges(a.tiles, (n + kKB - 1) / kKB, EmuConst<7>::kg, 0, a);
}

// Workspace, monotone in n, p and q (one size serves every smaller call):
// exponents and the partial tiles.
size_t emu_gram_bytes(int64_t n, int64_t p, int64_t q) {
  const int64_t tiles = ((p + kRows - 1) / kRows) * ((q + 63) / 64 + 1) + (q + kRows - 1) / kRows;
  const int64_t stages = (n + kKB - 1) / kKB;
  const int64_t items = std::min<int64_t>(tiles * stages, 8 * (int64_t)num_sms() + tiles);
  return align_up((size_t)(p + q) * 4) + align_up((size_t)items * 64 * kRows * 8) + 256;
}

rr_status emu_gram(cudaStream_t s, int64_t n, int64_t p, int64_t q, int32_t xt, const void* X, int64_t ldx,
                   int32_t yt, const void* Y, int64_t ldy, double* G, int64_t ldg, int accum, void* mem,
                   size_t bytes) {
  if (!emu_gram_supported(n, p, q)) return RR_ERR_ARG;
  if (bytes < emu_gram_bytes(n, p, q) || !mem) return RR_ERR_WORKSPACE;
  if ((uintptr_t)mem & 15) return RR_ERR_ARG;
  EmuMm a{};
  gram_tiles(n, p, q, a);
  Arena ar(mem, bytes);
  int* ex = ar.take<int>(p + q);
  int* ey = ex + p;
  a.part = ar.take<double>((size_t)a.items * 64 * kRows);
  if (ar.overflow) return RR_ERR_WORKSPACE;
  const bool same = X == Y && xt == yt && ldx == ldy && p == q;
  if (col_exp_chunks(n, p) > 1 || (!same && col_exp_chunks(n, q) > 1))
    RR_CUDA(cudaMemsetAsync(ex, 0x80, (size_t)(p + q) * 4, s));  // below every exponent
  RR_TRY(col_exps(s, xt, n, p, X, ldx, ex));
  if (same) ey = ex;
  else RR_TRY(col_exps(s, yt, n, q, Y, ldy, ey));
  a.a[0] = EmuSide{X, ldx, ex, xt, aligned_pairs(X, ldx, xt) ? 1 : 0};
  a.b = EmuSide{Y, ldy, ey, yt, aligned_pairs(Y, ldy, yt) ? 1 : 0};
  a.mode = 2;
  {
    TcProfScope prof(s, (double)n * (p * dtype_size(xt) + (same ? 0 : q * dtype_size(yt))) + 8.0 * p * q,
                     pair_flops(7, (double)p, (double)q, (double)n), 1);
    RR_TRY((launch_mm_types<7, false, false>(s, a, xt, yt)));
  }
  const dim3 g((unsigned)((p + 31) / 32), (unsigned)q);
  k_emu_gram_reduce<<<g, 256, 0, s>>>(p, q, a.ntn, a.nch, a.main_rows, a.main_tiles, a.tiles, a.ranges, a.part, G, ldg,
                                      accum);
  return check_launch("emu_gram reduce");
}

}  // namespace rr
