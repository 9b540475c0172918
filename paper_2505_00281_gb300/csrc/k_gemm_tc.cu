// tcgen05 tensor-core block product for the low-precision filter (Sec. 2's
// X_iter = A X with the BF16 basis of the precision map in Sec. 4.2):
//   C (M x N, FP32, column-major) = A_k^T B  [+ coef_j R(:, j)]
// A_k: K x M BF16, K contiguous (the K-major "A" operand: rows of A for
// A V, columns of A for A^T W); B: K x N BF16, K contiguous.
//
// One CTA per 128-row tile of C and K-split, 4 warps:
//   warp 0 (one lane): TMA producer, 128B-swizzled 64-wide K slabs of A and
//                      B into an S-stage shared-memory ring (mbarrier
//                      complete_tx per stage);
//   warp 1 (one lane): issues tcgen05.mma (kind::f16, BF16 x BF16 -> FP32,
//                      M = 128, N = padded N, K = 16 per instruction) into a
//                      TMEM accumulator, tcgen05.commit frees each stage;
//   warps 0-3:        epilogue, tcgen05.ld 32x32b from TMEM (warp w owns
//                      lanes 32w..32w+31 = rows), coalesced column stores.
// K splits (small M) add their partial tiles with FP32 atomics into a C
// pre-initialised to the added term.
// FP8 variant (kF8): E4M3 x E4M3 -> FP32 (tcgen05 kind::f8f6f4, K = 32 per
// instruction), the same 128-byte swizzle rows (128 elements per K step); the
// epilogue multiplies by a per-row scale of A and a per-column scale of B.
// Every mbarrier wait is bounded (2 s); on expiry the kernel records an error
// (read by the host), stops issuing, waits (bounded) for its in-flight copies,
// frees its TMEM and returns.
#include <cuda.h>

#include "rr_common.cuh"
#include "solver_kernels.cuh"
#include "tc_ptx.cuh"

namespace rr {

__device__ int g_tc_error = 0;

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;  // bf16 elements per 128-byte swizzle row

// the kernels' wait: the library-wide error word, 2 s limit
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_on(bar, parity, &g_tc_error, kWaitLimitNs);
}

}  // namespace

struct TcArgs {
  int64_t M, N, K;
  int npad;        // N rounded up to 16 (UMMA N)
  int tmem_cols;   // power of two >= max(32, npad)
  int stages;
  int ksteps_per_split;
  int nk;          // K steps (K / 64 rounded up)
  int nk1;         // same (kept for the launch record)
  int segs;        // 1, or 3 for the split product: per K step A_hi B_hi + A_lo B_hi + A_hi B_lo
  float* C;
  int64_t ldc;
  const double* R;
  int64_t ldr;
  const double* coef;
  int atomic;      // 1: K-split, add into C
  const float* rscale;  // FP8: C(i, j) = rscale[i] cscale[j] acc(i, j)
  const float* cscale;
};

template <bool kF8>
__global__ void __launch_bounds__(128, 1) k_gemm_bf16_tc(const __grid_constant__ CUtensorMap tmA,
                                                          const __grid_constant__ CUtensorMap tmB,
                                                          const __grid_constant__ CUtensorMap tmA2,
                                                          const __grid_constant__ CUtensorMap tmB2,
                                                          TcArgs a) {
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment for the swizzled tiles
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t a_bytes = kBM * kBK * 2;            // 16 KB
  const uint32_t b_bytes = (uint32_t)a.npad * kBK * 2;
  // split product: a stage holds A_hi, B_hi, A_lo, B_lo of one K step
  const bool spl = a.segs > 1;
  const uint32_t stage_bytes = (a_bytes + b_bytes) * (spl ? 2 : 1);  // multiple of 1024
  uint64_t* full = (uint64_t*)(base + (size_t)a.stages * stage_bytes);
  uint64_t* empty = full + a.stages;
  uint64_t* accum = empty + a.stages;
  __shared__ uint32_t s_tmem;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m0 = (int64_t)blockIdx.x * kBM;
  const int split = blockIdx.y;
  const int ks0 = split * a.ksteps_per_split;
  int ks1 = ks0 + a.ksteps_per_split;
  if (ks1 > a.nk) ks1 = a.nk;
  const int nks = ks1 > ks0 ? ks1 - ks0 : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;

  if (nks > 0) {
    if (warp == 0 && lane == 0) {
      // ---------------- TMA producer ----------------
      int issued = 0;
      for (int i = 0; i < nks; ++i) {
        const int s = i % a.stages;
        if (i >= a.stages && !mbar_wait(&empty[s], ((i / a.stages) - 1) & 1)) break;
        unsigned char* sa = base + (size_t)s * stage_bytes;
        unsigned char* sb = sa + a_bytes;
        mbar_expect_tx(&full[s], stage_bytes);
        const int kx = (ks0 + i) * (kF8 ? 2 * kBK : kBK);  // elements per 128-byte row
        tma_load_2d(sa, &tmA, &full[s], kx, (int)m0);
        tma_load_2d(sb, &tmB, &full[s], kx, 0);
        if (spl) {
          tma_load_2d(sb + b_bytes, &tmA2, &full[s], kx, (int)m0);
          tma_load_2d(sb + b_bytes + a_bytes, &tmB2, &full[s], kx, 0);
        }
        ++issued;
      }
      if (issued < nks) {
        // error: drain the copies still in flight (bounded) before leaving
        for (int i = (issued > a.stages ? issued - a.stages : 0); i < issued; ++i) {
          const int s = i % a.stages;
          const uint64_t t0 = global_timer_ns();
          while (!mbar_try_wait(&full[s], (i / a.stages) & 1) && global_timer_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    } else if (warp == 1 && lane == 0) {
      // ---------------- MMA issuer ----------------
      const uint32_t idesc = (1u << 4)                                  // D: FP32
                             | (kF8 ? 0u : (1u << 7) | (1u << 10))       // A, B: BF16 (kind::f16) or E4M3 (0)
                             | ((uint32_t)(a.npad >> 3) << 17)          // N / 8
                             | ((uint32_t)(kBM >> 4) << 24);            // M / 16
      for (int i = 0; i < nks; ++i) {
        const int s = i % a.stages;
        if (!mbar_wait(&full[s], (i / a.stages) & 1)) {
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sa = smem_u32(base + (size_t)s * stage_bytes);
        const uint32_t sb = sa + a_bytes;
        const uint64_t ad = sdesc_sw128(sa), bd = sdesc_sw128(sb);
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk)  // 32 bytes of K per instruction (16 BF16 / 32 E4M3)
          umma<kF8>(tmem, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc, (i > 0 || kk > 0) ? 1u : 0u);
        if (spl) {
          // A_lo B_hi and A_hi B_lo from the same stage (each operand read once)
          const uint64_t ad2 = sdesc_sw128(sb + b_bytes), bd2 = sdesc_sw128(sb + b_bytes + a_bytes);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            umma_bf16(tmem, ad2 + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc, 1u);
            umma_bf16(tmem, ad + (uint64_t)(kk * 2), bd2 + (uint64_t)(kk * 2), idesc, 1u);
          }
        }
        umma_commit(&empty[s]);
      }
      // the final commit arrives once every MMA issued above has completed,
      // also after an error, so TMEM is never freed under a running MMA
      umma_commit(accum);
    }
    // ---------------- epilogue (all 4 warps) ----------------
    __syncwarp();
    bool ready = mbar_wait(accum, 0);
    __syncwarp();
    ready = __all_sync(0xffffffffu, ready) && *(volatile int*)&g_tc_error == 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ready) {
      const int64_t row = m0 + warp * 32 + lane;
      const float rs = (kF8 && row < a.M) ? __ldg(a.rscale + row) : 1.f;
      for (int c0 = 0; c0 < a.npad; c0 += 32) {
        uint32_t r[32];
        tmem_ld_32x32b_x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
        if (row < a.M) {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const int64_t col = c0 + j;
            if (col < a.N) {
              float v = __uint_as_float(r[j]);
              if constexpr (kF8) v = v * rs * __ldg(a.cscale + col);
              float* dst = a.C + row + col * a.ldc;
              if (a.atomic) {
                atomicAdd(dst, v);
              } else {
                if (a.R) v += (float)(a.coef[col] * a.R[row + col * a.ldr]);
                *dst = v;
              }
            }
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols)
                 : "memory");
  }
}

// C = coef_j R(:, j) (or 0): the starting value for K-split accumulation
__global__ void k_tc_init_c(int64_t M, int64_t N, float* __restrict__ C, int64_t ldc,
                            const double* __restrict__ R, int64_t ldr, const double* __restrict__ coef) {
  const int64_t j = blockIdx.y;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
    C[i + j * ldc] = R ? (float)(coef[j] * R[i + j * ldr]) : 0.f;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int& gemm_force_simt() {
  static int v = 0;
  return v;
}

static thread_local TcProf* t_tc_prof = nullptr;
void tc_prof_attach(TcProf* p) { t_tc_prof = p; }

TcProfScope::TcProfScope(cudaStream_t s_, double bytes, double flops, int role) : p(t_tc_prof), s(s_) {
  if (!p) return;
  cudaEvent_t e;
  cudaEventCreate(&e);
  cudaEventRecord(e, s);
  p->ev.push_back(e);
  p->role.push_back(role);
  p->bytes += bytes;
  p->role_bytes[role] += bytes;
  p->role_flops[role] += flops;
  p->launches += 1;
}
TcProfScope::~TcProfScope() {
  if (!p) return;
  cudaEvent_t e;
  cudaEventCreate(&e);
  cudaEventRecord(e, s);
  p->ev.push_back(e);
}

int& gemm_split_cap() {
  static thread_local int v = 0;
  return v;
}

// Raise the kernel's dynamic shared-memory limit once (outside any stream
// capture: rr_batch_svd calls this before it starts capturing).
rr_status tc_prepare_attributes() {
  static bool done = false;
  if (!done) {
    RR_CUDA(cudaFuncSetAttribute(k_gemm_bf16_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    RR_CUDA(cudaFuncSetAttribute(k_gemm_bf16_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    RR_TRY(emu_prepare_attributes());
    done = true;
  }
  return RR_OK;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

bool gemm_bf16_tc_supported(int64_t M, int64_t N, int64_t K, int64_t lda, int64_t ldb, const void* A,
                            const void* B) {
  if (M <= 0 || N <= 0 || N > 256 || K <= 0) return false;
  if (lda % 8 || ldb % 8) return false;                          // 16-byte strides
  if (((uintptr_t)A & 15) || ((uintptr_t)B & 15)) return false;  // 16-byte aligned bases
  if (M > 0x7fffffff || K > 0x7fffffff) return false;
  return encode_fn() != nullptr;
}

static bool make_map(CUtensorMap* m, const void* base, int64_t inner, int64_t outer, int64_t ld_elems,
                     uint32_t box_inner, uint32_t box_outer, bool f8 = false) {
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
  cuuint64_t strides[1] = {(cuuint64_t)ld_elems * (f8 ? 1 : 2)};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t es[2] = {1, 1};
  CUresult r = encode_fn()(m, f8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                           const_cast<void*>(base), dims, strides,
                           box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

static int64_t tc_nk(int64_t K) { return (K + kBK - 1) / kBK; }

static rr_status gemm_bf16_tc_impl(int64_t M, int64_t N, int64_t K, const __nv_bfloat16* A, int64_t lda,
                                   const __nv_bfloat16* B, int64_t ldb, float* C, int64_t ldc,
                                   const double* R, int64_t ldr, const double* coef, cudaStream_t s, const __nv_bfloat16* A2 = nullptr,
                                   const __nv_bfloat16* B2 = nullptr);

rr_status gemm_bf16_tc(int64_t M, int64_t N, int64_t K, const __nv_bfloat16* A, int64_t lda,
                       const __nv_bfloat16* B, int64_t ldb, float* C, int64_t ldc, const double* R,
                       int64_t ldr, const double* coef, cudaStream_t s) {
  return gemm_bf16_tc_impl(M, N, K, A, lda, B, ldb, C, ldc, R, ldr, coef, s);
}

// Split-BF16 product: C (M x N, FP32) = (A_hi + A_lo)^T (B_hi + B_lo) without
// the lo.lo term (+ coef_j R(:, j)), FP32 accumulation; each operand pair is
// the BF16 rounding of a wider value and its BF16 residual.
rr_status gemm_bf16_tc_split(int64_t M, int64_t N, int64_t K, const __nv_bfloat16* A_hi,
                             const __nv_bfloat16* A_lo, int64_t lda, const __nv_bfloat16* B_hi,
                             const __nv_bfloat16* B_lo, int64_t ldb, float* C, int64_t ldc,
                             const double* R, int64_t ldr, const double* coef, cudaStream_t s) {
  if (!A_lo || !B_lo) return RR_ERR_ARG;
  return gemm_bf16_tc_impl(M, N, K, A_hi, lda, B_hi, ldb, C, ldc, R, ldr, coef, s, A_lo, B_lo);
}

// Split product (A2, B2 non-null): C = A^T B + A2^T B + A^T B2 (+ coef R);
// every pipeline stage carries the four tiles of one K step and three MMAs
// consume them, so each operand is read once.
static rr_status gemm_bf16_tc_impl(int64_t M, int64_t N, int64_t K, const __nv_bfloat16* A, int64_t lda,
                                   const __nv_bfloat16* B, int64_t ldb, float* C, int64_t ldc,
                                   const double* R, int64_t ldr, const double* coef, cudaStream_t s, const __nv_bfloat16* A2, const __nv_bfloat16* B2) {
  const bool split = A2 && B2;
  if ((A2 || B2) && !split) return RR_ERR_ARG;
  const int npad = (int)((N + 15) / 16 * 16);
  int tcols = 32;
  while (tcols < npad) tcols <<= 1;
  CUtensorMap ta, tb, ta2, tb2;
  if (!make_map(&ta, A, K, M, lda, kBK, kBM)) return RR_ERR_ARG;
  if (!make_map(&tb, B, K, N, ldb, kBK, (uint32_t)npad)) return RR_ERR_ARG;
  if (split) {
    if (!make_map(&ta2, A2, K, M, lda, kBK, kBM)) return RR_ERR_ARG;
    if (!make_map(&tb2, B2, K, N, ldb, kBK, (uint32_t)npad)) return RR_ERR_ARG;
  } else {
    ta2 = ta;
    tb2 = tb;
  }
  const int64_t tiles = (M + kBM - 1) / kBM;
  const int nk1 = (int)tc_nk(K);
  const int segs = split ? 3 : 1;
  const int nk = nk1;
  const int sms = num_sms();
  int splits = 1;
  if (tiles < sms) {
    splits = (int)(sms / tiles);
    if (splits > nk) splits = nk;
    if (gemm_split_cap() > 0 && splits > gemm_split_cap()) splits = gemm_split_cap();
    if (splits < 1) splits = 1;
  }
  const int per = (nk + splits - 1) / splits;
  splits = (nk + per - 1) / per;
  const uint32_t stage_bytes = (kBM * kBK * 2 + (uint32_t)npad * kBK * 2) * (split ? 2 : 1);
  int stages = (int)((200 * 1024) / stage_bytes);
  if (stages > 8) stages = 8;
  if (stages < 2) return RR_ERR_ARG;
  const size_t smem = 1024 + (size_t)stages * stage_bytes + (2 * stages + 1) * sizeof(uint64_t);
  RR_TRY(tc_prepare_attributes());
  TcArgs a{};
  a.M = M;
  a.N = N;
  a.K = K;
  a.npad = npad;
  a.tmem_cols = tcols;
  a.stages = stages;
  a.ksteps_per_split = per;
  a.nk = nk;
  a.nk1 = nk1;
  a.segs = segs;
  a.C = C;
  a.ldc = ldc;
  a.R = R;
  a.ldr = ldr;
  a.coef = coef;
  a.atomic = splits > 1;
  if (splits > 1) {
    dim3 gi((unsigned)std::min<int64_t>((M + 255) / 256, 256), (unsigned)N);
    k_tc_init_c<<<gi, 256, 0, s>>>(M, N, C, ldc, R, ldr, coef);
    note_launches(1);
  }
  const dim3 grid((unsigned)tiles, (unsigned)splits, 1u);
  a.rscale = a.cscale = nullptr;
  // algorithmic bytes of this launch: every operand read once, the output
  // written once; algorithmic flops: 2 M N K per product it forms
  const double abytes = (split ? 2.0 : 1.0) * 2.0 * K * ((double)M + (double)N) + 4.0 * M * N;
  const double aflops = (split ? 3.0 : 1.0) * 2.0 * (double)M * (double)N * (double)K;
  TcProfScope prof_scope(s, abytes, aflops, 0);
  k_gemm_bf16_tc<false><<<grid, 128, smem, s>>>(ta, tb, ta2, tb2, a);
  return check_launch("gemm_bf16_tc");
}

// E4M3 product: C (M x N, FP32) = diag(rscale) A_k^T B diag(cscale), A_k
// K x M and B K x N E4M3 with K contiguous (ld in elements, multiples of 16),
// FP32 accumulation.
rr_status gemm_e4m3_tc(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const float* rscale,
                       const void* B, int64_t ldb, const float* cscale, float* C, int64_t ldc, cudaStream_t s) {
  if (M <= 0 || N <= 0 || N > 256 || K <= 0 || !rscale || !cscale || !C) return RR_ERR_ARG;
  if (lda % 16 || ldb % 16 || ((uintptr_t)A & 15) || ((uintptr_t)B & 15)) return RR_ERR_ARG;
  if (M > 0x7fffffff || K > 0x7fffffff || !encode_fn()) return RR_ERR_ARG;
  constexpr int kBK8 = 2 * kBK;  // E4M3 elements per 128-byte row
  const int npad = (int)((N + 15) / 16 * 16);
  int tcols = 32;
  while (tcols < npad) tcols <<= 1;
  CUtensorMap ta, tb;
  if (!make_map(&ta, A, K, M, lda, kBK8, kBM, true)) return RR_ERR_ARG;
  if (!make_map(&tb, B, K, N, ldb, kBK8, (uint32_t)npad, true)) return RR_ERR_ARG;
  const int64_t tiles = (M + kBM - 1) / kBM;
  const int nk = (int)((K + kBK8 - 1) / kBK8);
  const int sms = num_sms();
  int splits = 1;
  if (tiles < sms) {
    splits = (int)(sms / tiles);
    if (splits > nk) splits = nk;
    if (splits < 1) splits = 1;
  }
  const int per = (nk + splits - 1) / splits;
  splits = (nk + per - 1) / per;
  const uint32_t stage_bytes = kBM * kBK8 + (uint32_t)npad * kBK8;
  int stages = (int)((200 * 1024) / stage_bytes);
  if (stages > 8) stages = 8;
  if (stages < 2) return RR_ERR_ARG;
  const size_t smem = 1024 + (size_t)stages * stage_bytes + (2 * stages + 1) * sizeof(uint64_t);
  RR_TRY(tc_prepare_attributes());
  TcArgs a{};
  a.M = M;
  a.N = N;
  a.K = K;
  a.npad = npad;
  a.tmem_cols = tcols;
  a.stages = stages;
  a.ksteps_per_split = per;
  a.nk = nk;
  a.nk1 = nk;
  a.segs = 1;
  a.C = C;
  a.ldc = ldc;
  a.atomic = splits > 1;
  a.rscale = rscale;
  a.cscale = cscale;
  if (splits > 1) {
    dim3 gi((unsigned)std::min<int64_t>((M + 255) / 256, 256), (unsigned)N);
    k_tc_init_c<<<gi, 256, 0, s>>>(M, N, C, ldc, nullptr, 0, nullptr);
    note_launches(1);
  }
  dim3 grid((unsigned)tiles, (unsigned)splits, 1u);
  TcProfScope prof_scope(s, (double)K * ((double)M + (double)N) + 4.0 * M * N, 2.0 * (double)M * N * K, 0);
  k_gemm_bf16_tc<true><<<grid, 128, smem, s>>>(ta, tb, ta, tb, a);
  return check_launch("gemm_e4m3_tc");
}

// error words of the tensor-core kernels (0 = ok); cleared on read
rr_status tc_take_error(cudaStream_t s) {
  int e = 0, e2 = 0;
  RR_CUDA(cudaMemcpyFromSymbolAsync(&e, g_tc_error, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
  RR_TRY(emu_error_fetch(s, &e2));
  RR_CUDA(cudaStreamSynchronize(s));
  if (e || e2) {
    int z = 0;
    RR_CUDA(cudaMemcpyToSymbolAsync(g_tc_error, &z, sizeof(int), 0, cudaMemcpyHostToDevice, s));
    RR_TRY(emu_error_clear(s));
    return (rr_status)(e ? e : e2);
  }
  return RR_OK;
}

}  // namespace rr

// ---------------------------------------------------------------------------
// Failure-detection self-test: each bounded wait of the library, made to run
// out on purpose.  mode 0: one CTA enters the grid barrier of the cooperative
// kernels for a grid of two CTAs that has only itself; mode 1: one thread
// waits on an mbarrier that nothing arrives on (the wait of the tensor-core
// kernels).  Both give up after limit_ns, record RR_ERR_TIMEOUT in err and
// return; the kernel ends normally.
// ---------------------------------------------------------------------------
namespace rr {
namespace {
__global__ void k_wait_selftest(int mode, uint64_t limit_ns, GridBarrier* gb, int* err) {
  if (mode == 0) {
    grid_barrier(gb, 2u, err, limit_ns);   // the second CTA never arrives
    return;
  }
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_wait_on(&bar, 0, err, limit_ns);  // phase 0 never completes
  }
}
}  // namespace
}  // namespace rr

extern "C" rr_status rr_wait_selftest(int32_t mode, int64_t limit_ns, void* scratch, void* stream) {
  using namespace rr;
  if ((mode != 0 && mode != 1) || limit_ns <= 0 || limit_ns > 10000000000ll || !scratch ||
      ((uintptr_t)scratch & 15))
    return RR_ERR_ARG;
  cudaStream_t s = as_stream(stream);
  GridBarrier* gb = (GridBarrier*)scratch;
  int* err = (int*)((char*)scratch + sizeof(GridBarrier));
  RR_CUDA(cudaMemsetAsync(scratch, 0, 16, s));
  k_wait_selftest<<<1, 32, 0, s>>>(mode, (uint64_t)limit_ns, gb, err);
  RR_TRY(check_launch("rr_wait_selftest"));
  int h = 0;
  RR_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  RR_CUDA(cudaStreamSynchronize(s));
  return (rr_status)h;
}
