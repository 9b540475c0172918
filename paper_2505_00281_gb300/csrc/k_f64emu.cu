// Preparation of a dense FP64 operator (BF16 hi / lo copies and the row and
// column exponents of its FP64-accurate products) and the C entries of the
// FP64-accurate products on the tensor cores (k_emu_mm.cu).
#include <algorithm>

#include "rr_common.cuh"
#include "solver_kernels.cuh"

namespace rr {

constexpr int kMaxSlices = 10;

// BF16 bits (sign excluded) of v = k 2^s (0 < k < 2^62) rounded the way an
// FP64 value is cast to BF16 here: to FP32 (nearest even), then the FP32
// pattern to BF16 (nearest even; a carry may reach the exponent).  Integer
// operations only (this GPU has few FP64 units).  False when the FP32
// rounding is not a normal number (the caller then uses the conversion
// instructions).
__device__ __forceinline__ bool bf16_of_scaled(unsigned long long k, int s, unsigned& out) {
  int msb = 63 - __clzll((long long)k);
  unsigned long long k24;
  if (msb > 23) {
    const int sh = msb - 23;
    k24 = k >> sh;
    const unsigned long long rem = k & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (k24 & 1ull))) ++k24;
    if (k24 == (1ull << 24)) {
      k24 >>= 1;
      ++msb;
    }
  } else {
    k24 = k << (23 - msb);
  }
  const int e32 = msb + s + 127;  // v rounded = (k24 / 2^23) 2^(msb + s)
  if (e32 < 1 || e32 > 254) return false;
  const unsigned f = ((unsigned)e32 << 23) | (unsigned)(k24 & 0x7FFFFFull);
  out = (f + 0x7FFFu + ((f >> 16) & 1u)) >> 16;
  return true;
}

// hi = bf16(a) and lo = bf16(a - hi) with the cast above (a - hi is exact
// in FP64), as BF16 bit patterns.
__device__ __forceinline__ void bf16_split_bits(double a, unsigned& hi, unsigned& lo) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  const unsigned sgn = (unsigned)(u >> 63);
  const int E = (int)((u >> 52) & 0x7FF);
  const unsigned long long M = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);  // a = M 2^(E - 1075)
  unsigned hb, lb;
  if (E == 0 || E == 0x7FF || !bf16_of_scaled(M, E - 1075, hb)) {
    const __nv_bfloat16 h = __float2bfloat16_rn((float)a);
    hi = __bfloat16_as_ushort(h);
    lo = __bfloat16_as_ushort(__float2bfloat16_rn((float)(a - (double)__bfloat162float(h))));
    return;
  }
  hi = (sgn << 15) | hb;
  // hi in units of a's last place: (128 + m7) 2^(e8 - 134 - (E - 1075))
  const int e8 = (int)(hb >> 7), sh = e8 + 941 - E;  // 45, or 46 after a carry
  const long long d = (long long)M - (long long)((128ull + (hb & 127u)) << sh);
  if (d == 0) {
    lo = 0;
    return;
  }
  if (!bf16_of_scaled((unsigned long long)(d < 0 ? -d : d), E - 1075, lb)) {
    const double hv = (double)__bfloat162float(__ushort_as_bfloat16((unsigned short)hi));
    lo = __bfloat16_as_ushort(__float2bfloat16_rn((float)(a - hv)));
    return;
  }
  lo = ((sgn ^ (d < 0 ? 1u : 0u)) << 15) | lb;
}

// hi only (the same cast)
__device__ __forceinline__ unsigned bf16_bits_of(double a) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  const int E = (int)((u >> 52) & 0x7FF);
  unsigned hb;
  if (E == 0 || E == 0x7FF || !bf16_of_scaled((u & 0xFFFFFFFFFFFFFull) | (1ull << 52), E - 1075, hb))
    return __bfloat16_as_ushort(__float2bfloat16_rn((float)a));
  return ((unsigned)(u >> 63) << 15) | hb;
}

constexpr int kExpNone = -1100;  // exponent of zero (below every finite one)

__global__ void k_exp_init(int64_t count, int* __restrict__ e) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    e[i] = kExpNone;
}

// First pass over a dense FP64 operator (m x n, column-major): the BF16 hi /
// lo split in column-major and row-major copies, and the exponents of the
// largest entry of every row and column (atomic max into rexp / cexp, which
// start at kExpNone).  Every output may be null.  A block takes a 32-row x
// 256-column tile, a warp 32 x 32 (lane = row) in two halves of 16 columns
// (62 registers instead of 120: four blocks per SM, twice the resident
// warps; the pass is bound by the loads in flight): column
// loads are coalesced, a lane writes its row's 16 entries of a half to the
// row-major copies as two 16-byte stores.
__global__ void __launch_bounds__(256, 4) k_op_pass1(int64_t m, int64_t n, const double* __restrict__ A, int64_t lda,
                                                  __nv_bfloat16* __restrict__ hi_col, __nv_bfloat16* __restrict__ hi_row,
                                                  __nv_bfloat16* __restrict__ lo_col, __nv_bfloat16* __restrict__ lo_row,
                                                  int* __restrict__ rexp, int* __restrict__ cexp) {
  __shared__ int rmax[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane;
  const bool rv = i < m;
  const bool need_lo = lo_col || lo_row;
  int emx = kExpNone;
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    const int64_t jw = (int64_t)blockIdx.y * 256 + warp * 32 + 16 * half;
    unsigned hp[8], lp[8];
    double av[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int64_t j = jw + c;
      av[c] = (rv && j < n) ? A[i + j * lda] : 0.0;
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int64_t j = jw + c;
      const double a = av[c];
      const unsigned long long u = (unsigned long long)__double_as_longlong(a);
      const int E = (int)((u >> 52) & 0x7FF);
      const int e = E == 0 ? kExpNone : E - 1022;
      emx = max(emx, e);
      if (cexp) {
        int ce = e;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ce = max(ce, __shfl_xor_sync(0xffffffffu, ce, o));
        if (lane == 0 && j < n) atomicMax(cexp + j, ce);
      }
      unsigned h = 0, l = 0;
      if (need_lo) {
        bf16_split_bits(a, h, l);
      } else {
        h = bf16_bits_of(a);
      }
      if (c & 1) {
        hp[c >> 1] |= h << 16;
        lp[c >> 1] |= l << 16;
      } else {
        hp[c >> 1] = h;
        lp[c >> 1] = l;
      }
      if (rv && j < n) {
        if (hi_col) hi_col[i + j * m] = __ushort_as_bfloat16((unsigned short)h);
        if (lo_col) lo_col[i + j * m] = __ushort_as_bfloat16((unsigned short)l);
      }
    }
    if (rv) {
      const bool vec = (jw + 16 <= n) && (n % 8 == 0);
      if (hi_row) {
        if (vec) {
          uint4* dst = reinterpret_cast<uint4*>(hi_row + i * n + jw);
#pragma unroll
          for (int k = 0; k < 2; ++k) dst[k] = make_uint4(hp[4 * k], hp[4 * k + 1], hp[4 * k + 2], hp[4 * k + 3]);
        } else {
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (jw + c < n) hi_row[i * n + jw + c] = __ushort_as_bfloat16((unsigned short)(hp[c >> 1] >> (16 * (c & 1))));
        }
      }
      if (lo_row) {
        if (vec) {
          uint4* dst = reinterpret_cast<uint4*>(lo_row + i * n + jw);
#pragma unroll
          for (int k = 0; k < 2; ++k) dst[k] = make_uint4(lp[4 * k], lp[4 * k + 1], lp[4 * k + 2], lp[4 * k + 3]);
        } else {
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (jw + c < n) lo_row[i * n + jw + c] = __ushort_as_bfloat16((unsigned short)(lp[c >> 1] >> (16 * (c & 1))));
        }
      }
    }
  }
  if (rexp) {
    rmax[warp][lane] = emx;
    __syncthreads();
    if (warp == 0 && rv) {
      int r = rmax[0][lane];
#pragma unroll
      for (int w = 1; w < 8; ++w) r = max(r, rmax[w][lane]);
      atomicMax(rexp + i, r);
    }
  }
}

// BF16 hi / lo copies of a dense FP64 operator (any of the four may be null)
// and, when emu is given, its row and / or column exponents for FP64-accurate
// products (emu_mem: emu_operator_bytes), in one pass over A.
rr_status op_prepare(cudaStream_t s, const double* A, int64_t m, int64_t n, int64_t lda,
                     __nv_bfloat16* hi_col, __nv_bfloat16* hi_row, __nv_bfloat16* lo_col, __nv_bfloat16* lo_row,
                     EmuOperator* emu, void* emu_mem, bool rows, bool cols) {
  if (m <= 0 || n <= 0) return RR_OK;
  int *rexp = nullptr, *cexp = nullptr;
  if (emu) {
    Arena ar(emu_mem, emu_operator_bytes(m, n, rows, cols));
    *emu = EmuOperator{};
    emu->m = m;
    emu->n = n;
    emu->A = A;
    emu->lda = lda;
    if (rows) {
      emu->rexp = rexp = ar.take<int>(m);
      k_exp_init<<<(unsigned)std::min<int64_t>((m + 255) / 256, 1024), 256, 0, s>>>(m, rexp);
      note_launches(1);
    }
    if (cols) {
      emu->cexp = cexp = ar.take<int>(n);
      k_exp_init<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, s>>>(n, cexp);
      note_launches(1);
    }
  }
  const dim3 g((unsigned)((m + 31) / 32), (unsigned)((n + 255) / 256));
  if (hi_col || hi_row || lo_col || lo_row || rexp || cexp) {
    k_op_pass1<<<g, 256, 0, s>>>(m, n, A, lda, hi_col, hi_row, lo_col, lo_row, rexp, cexp);
    RR_TRY(check_launch("op_prepare"));
  }
  return RR_OK;
}

}  // namespace rr

using namespace rr;

extern "C" rr_status rr_split_operator(int64_t m, int64_t n, const double* A, int64_t lda, void* hi_col,
                                       void* hi_row, void* lo_col, void* lo_row, void* stream) {
  if (m < 0 || n < 0 || lda < m || !A) return RR_ERR_ARG;
  return op_prepare(as_stream(stream), A, m, n, lda, (__nv_bfloat16*)hi_col, (__nv_bfloat16*)hi_row,
                    (__nv_bfloat16*)lo_col, (__nv_bfloat16*)lo_row, nullptr, nullptr, false, false);
}

extern "C" size_t rr_lift_workspace_size(int64_t n, int64_t b, int64_t K) {
  if (n < 0 || b < 0 || K < 0) return 0;
  return lift_emu_bytes(n, b, K);
}

extern "C" rr_status rr_lift(int64_t n, int64_t b, int32_t t1, const void* S1, int64_t ld1, int64_t p1,
                             int32_t t2, const void* S2, int64_t ld2, int64_t p2, const double* Y, int64_t ldy,
                             double* X, int64_t ldx, void* ws, size_t ws_bytes, void* stream) {
  auto ok_type = [](int32_t t) { return t == RR_F64 || t == RR_F32 || t == RR_BF16; };
  if (n < 0 || b < 1 || p1 < 1 || !S1 || !Y || !X || !ok_type(t1) || ld1 < n || ldx < n) return RR_ERR_ARG;
  if (S2 && (p2 < 0 || !ok_type(t2) || ld2 < n)) return RR_ERR_ARG;
  const int64_t p2e = S2 ? p2 : 0;
  if (ldy < p1 + p2e) return RR_ERR_ARG;
  if (n == 0) return RR_OK;
  cudaStream_t s = as_stream(stream);
  bool done = false;
  RR_TRY(lift_emu(s, n, b, t1, S1, ld1, p1, t2, S2, ld2, p2e, Y, ldy, X, ldx, ws, ws_bytes, &done));
  if (done) return RR_OK;
  RR_TRY(lift(s, t1, n, b, p1, S1, ld1, Y, ldy, X, ldx, 0));
  if (S2 && p2e > 0) RR_TRY(lift(s, t2, n, b, p2e, S2, ld2, Y + p1, ldy, X, ldx, 1));
  return RR_OK;
}

extern "C" size_t rr_gemm_f64_emulated_workspace_size(int32_t trans, int64_t M, int64_t N, int64_t K,
                                                      int32_t slices) {
  const int64_t m = trans ? K : M, n = trans ? M : K;
  return emu_operator_bytes(m, n, !trans, trans != 0) + emu_block_bytes(K, N, slices) + 512;
}

extern "C" rr_status rr_gemm_f64_emulated(int32_t trans, int64_t M, int64_t N, int64_t K, const double* A,
                                          int64_t lda, const double* B, int64_t ldb, double* C,
                                          int64_t ldc, int32_t slices, void* ws, size_t ws_bytes,
                                          void* stream) {
  if (M <= 0 || N <= 0 || N > 256 || K <= 0 || !A || !B || !C || ldb < K || ldc < M) return RR_ERR_ARG;
  if (slices < 1 || slices > kMaxSlices) return RR_ERR_ARG;
  if (trans ? lda < K : lda < M) return RR_ERR_ARG;
  const int64_t m = trans ? K : M, n = trans ? M : K;
  if (!ws || ws_bytes < rr_gemm_f64_emulated_workspace_size(trans, M, N, K, slices)) return RR_ERR_WORKSPACE;
  if (n % 8 || m % 8 || ((uintptr_t)ws & 15)) return RR_ERR_ARG;
  cudaStream_t s = as_stream(stream);
  EmuOperator op;
  const size_t ob = align_up(emu_operator_bytes(m, n, !trans, trans != 0));
  RR_TRY(emu_prepare(s, A, m, n, lda, op, ws, !trans, trans != 0));
  return emu_gemm(s, op, trans, N, B, ldb, C, ldc, slices, (char*)ws + ob);
}
