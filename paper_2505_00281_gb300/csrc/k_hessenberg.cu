// Algorithm 8: the right-looking Hessenberg process for a block (Sec. 4.2.2),
// the paper's inner-product-free basis step.  Its output equals P^T L of
// row-pivoted LU.
//
// GB300 design: one cooperative launch; each CTA owns a contiguous slab of
// rows (kept in shared memory when it fits).  Per column j:
//   (a) every CTA finds the largest |W(r, j)| in its slab (first index on
//       ties) and publishes (value, row) plus that row's trailing entries,
//       then releases its flag (step j + 1);
//   (b) every CTA acquires all flags (bounded wait) — an all-gather, not a
//       barrier followed by reads;
//   (c) every CTA reduces the published candidates itself and gets the
//       pivot r, W(r, j) and the weights W(r, j+1:k);
//   (d) every CTA scales its part of column j by 1/W(r, j) and applies the
//       rank-1 update to its rows of the trailing columns.
// The candidate buffers are double-buffered by column parity so no CTA can
// overwrite a buffer another CTA still reads.  Arithmetic: IEEE divide,
// multiply and subtract, each rounded separately (no FMA contraction), so the
// result is bit-reproducible and equals a plain FP32/FP64 loop.
#include <climits>
#include <type_traits>

#include <cooperative_groups.h>

#include "rr_common.cuh"

namespace rr {

template <typename T>
struct HessWs {
  int* err;
  GridBarrier* bar;
  T* pval;      // [2][G] signed candidate pivot value
  int* pidx;    // [2][G] candidate row
  T* prow;      // [2][G][k] candidate row's entries
  T* pcolmax;   // [G][k] per-slab column inf-norms
  int* flags;   // [G] column steps published by each CTA (j + 1 after column j)
  unsigned long long* cand;  // [2][G] packed candidates (FP32 path)
  int64_t rpc;               // rows per CTA (FP32 path; 0: ceil(n / G))
  const T* colmax_ext;       // [k] column inf-norms on entry to the whole process
                             // (the blocked process's panels), or null: computed here
};

// Publish/await the per-column candidates: CTA g releases flags[g] = step once
// its candidate is written; readers acquire every flag before reading.
__device__ __forceinline__ void flag_release(int* f, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(f), "r"(v) : "memory");
}
__device__ __forceinline__ void word_release(unsigned long long* f, unsigned long long v) {
  asm volatile("st.release.gpu.global.b64 [%0], %1;" ::"l"(f), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long word_acquire(const unsigned long long* f) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(f) : "memory");
  return v;
}
__device__ __forceinline__ int flag_acquire(const int* f) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
  return v;
}

template <typename T> __device__ __forceinline__ T ld_cg(const T* p);
template <> __device__ __forceinline__ float ld_cg<float>(const float* p) { return __ldcg(p); }
template <> __device__ __forceinline__ double ld_cg<double>(const double* p) { return __ldcg(p); }
__device__ __forceinline__ int ld_cg_i(const int* p) { return __ldcg(p); }

template <typename T> __device__ __forceinline__ T rn_div(T a, T b);
template <> __device__ __forceinline__ float rn_div<float>(float a, float b) { return __fdiv_rn(a, b); }
template <> __device__ __forceinline__ double rn_div<double>(double a, double b) { return __ddiv_rn(a, b); }
template <typename T> __device__ __forceinline__ T rn_mul(T a, T b);
template <> __device__ __forceinline__ float rn_mul<float>(float a, float b) { return __fmul_rn(a, b); }
template <> __device__ __forceinline__ double rn_mul<double>(double a, double b) { return __dmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T rn_sub(T a, T b);
template <> __device__ __forceinline__ float rn_sub<float>(float a, float b) { return __fsub_rn(a, b); }
template <> __device__ __forceinline__ double rn_sub<double>(double a, double b) { return __dsub_rn(a, b); }

// (|v|, idx) with "larger |v| wins, then smaller idx"
template <typename T>
__device__ __forceinline__ void argmax_merge(T& av, int& ai, T bv, int bi) {
  if (bv > av || (bv == av && bi < ai)) {
    av = bv;
    ai = bi;
  }
}

constexpr int kHessThreads = 512;

// The kernel works on "Wv": the CTA's slab of W, either in shared memory
// (slab mode: rows r0..r1 of all k columns, column-major with ld = rows per
// CTA; loaded once, written back at the end) or W itself in global memory.
//
// Look-ahead: after the pivot of column j is known, a CTA scales column j,
// updates column j+1 only, picks and publishes its candidate for column j+1
// (the candidate row's trailing entries get the same rank-1 update, computed
// with the same operations), and only then applies the rank-1 update to
// columns j+2.. — so that update overlaps the other CTAs' progress instead of
// sitting on the per-column critical path.  Loop indices are 32-bit: lanes run
// over rows (consecutive addresses), warps over columns.
template <typename T, typename TO>
__global__ void __launch_bounds__(kHessThreads) k_hessenberg(
    int64_t n, int k, T* __restrict__ W, int64_t ldw, TO* __restrict__ Q, int64_t ldq,
    int* __restrict__ piv, T tol, HessWs<T> ws, int slab) {
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = kHessThreads / 32;
  const int64_t rpc = (n + G - 1) / G;
  const int64_t r0 = (int64_t)g * rpc;
  const int64_t r1 = r0 + rpc < n ? r0 + rpc : n;
  const int nr = r1 > r0 ? (int)(r1 - r0) : 0;

  extern __shared__ unsigned char smem_raw[];
  T* thr = reinterpret_cast<T*>(smem_raw);   // [k]
  T* wgt = thr + k;                          // [k]
  T* slabp = wgt + k;                        // [k][rpc] in slab mode
  // column c of this CTA's rows: col(c)[i], i = 0..nr-1 (row r0 + i)
  T* const base = slab ? slabp : W + r0;
  const int64_t ldv = slab ? rpc : ldw;
  auto col = [&](int c) -> T* { return base + (int64_t)c * ldv; };
  if (slab) {
    for (int c = warp; c < k; c += nwarps) {
      const T* src = W + r0 + (int64_t)c * ldw;
      T* dst = col(c);
      for (int i = lane; i < nr; i += 32) dst[i] = src[i];
    }
    __syncthreads();
  }
  __shared__ T red_v[32];
  __shared__ int red_i[32];
  __shared__ T s_qr;
  __shared__ int s_r, s_win, s_keep;

  // ---- column inf-norms on entry (relative skip threshold) ----
  for (int c = warp; c < k; c += nwarps) {
    T m = T(0);
    const T* cc = col(c);
    for (int i = lane; i < nr; i += 32) m = fmax(m, fabs(cc[i]));
    m = warp_max(m);
    if (lane == 0) ws.pcolmax[(size_t)g * k + c] = m;
  }
  if (!grid_barrier(ws.bar, G, ws.err)) return;
  for (int c = tid; c < k; c += kHessThreads) {
    T m = T(0);
    for (int h = 0; h < G; ++h) m = fmax(m, ld_cg(ws.pcolmax + (size_t)h * k + c));
    thr[c] = rn_mul(tol, m);
  }
  __syncthreads();

  // local argmax of |column jc| over this CTA's rows, then publish the
  // candidate (value, global row, row entries jc+1..k-1).  When upd is set,
  // the row entries are published as they will be after the pending rank-1
  // update by column jc-1 (weights wgt, multiplier column jc-1).
  auto publish = [&](int jc, bool upd) {
    const int par = jc & 1;
    const T* cj = col(jc);
    T bv = T(-1);
    int bi = INT_MAX;
    for (int i = tid; i < nr; i += kHessThreads) {
      T v = fabs(cj[i]);
      if (v > bv) {  // strictly greater: first index wins within a thread
        bv = v;
        bi = i;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      T ov = __shfl_xor_sync(0xffffffffu, bv, o);
      int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      argmax_merge(bv, bi, ov, oi);
    }
    if (lane == 0) {
      red_v[warp] = bv;
      red_i[warp] = bi;
    }
    __syncthreads();
    if (warp == 0) {
      bv = lane < nwarps ? red_v[lane] : T(-1);
      bi = lane < nwarps ? red_i[lane] : INT_MAX;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        T ov = __shfl_xor_sync(0xffffffffu, bv, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        argmax_merge(bv, bi, ov, oi);
      }
      if (lane == 0) {
        s_r = bi;
        ws.pidx[par * G + g] = (bi != INT_MAX) ? (int)(r0 + bi) : INT_MAX;
        ws.pval[par * G + g] = (bi != INT_MAX) ? cj[bi] : T(0);
      }
    }
    __syncthreads();
    const int rl = s_r;
    T* prow = ws.prow + ((size_t)par * G + g) * k;
    if (rl != INT_MAX) {
      const T m = upd ? col(jc - 1)[rl] : T(0);
      for (int c = jc + 1 + tid; c < k; c += kHessThreads) {
        T v = col(c)[rl];
        if (upd) v = rn_sub(v, rn_mul(wgt[c], m));
        prow[c] = v;
      }
    } else {
      for (int c = jc + 1 + tid; c < k; c += kHessThreads) prow[c] = T(0);
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      flag_release(ws.flags + g, jc + 1);
    }
  };

  publish(0, false);
  for (int j = 0; j < k; ++j) {
    const int par = j & 1;
    // (b) wait for every CTA's candidate for column j (bounded)
    if (warp == 0) {
      const uint64_t t0 = global_timer_ns();
      bool ok = true;
      for (int h = lane; h < G && ok; h += 32) {
        while (flag_acquire(ws.flags + h) < j + 1) {
          if (*(volatile int*)ws.err != 0 || global_timer_ns() - t0 > kWaitLimitNs) {
            atomicCAS(ws.err, 0, (int)RR_ERR_TIMEOUT);
            ok = false;
            break;
          }
        }
      }
      __syncwarp();
    }
    __syncthreads();
    if (*(volatile int*)ws.err != 0) return;
    // (c) global winner, computed redundantly by every CTA
    if (warp == 0) {
      T av = T(-1);
      int ai = INT_MAX, ag = -1;
      for (int h = lane; h < G; h += 32) {
        int hi = ld_cg_i(ws.pidx + par * G + h);
        T hv = fabs(ld_cg(ws.pval + par * G + h));
        if (hi == INT_MAX) continue;
        if (hv > av || (hv == av && hi < ai)) {
          av = hv;
          ai = hi;
          ag = h;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        T ov = __shfl_xor_sync(0xffffffffu, av, o);
        int oi = __shfl_xor_sync(0xffffffffu, ai, o);
        int og = __shfl_xor_sync(0xffffffffu, ag, o);
        if (ov > av || (ov == av && oi < ai)) {
          av = ov;
          ai = oi;
          ag = og;
        }
      }
      if (lane == 0) {
        T qr = (ag >= 0) ? ld_cg(ws.pval + par * G + ag) : T(0);
        s_qr = qr;
        s_r = ai;
        s_win = ag;
        s_keep = (ag >= 0 && qr != T(0) && fabs(qr) >= thr[j]) ? 1 : 0;
        if (g == 0) piv[j] = s_keep ? ai : -1;
      }
    }
    __syncthreads();
    const bool keep = s_keep != 0;
    T* cj = col(j);
    // (d) scale column j, update column j+1, publish column j+1's candidate,
    // then update columns j+2..k-1
    if (keep) {
      const T qr = s_qr;
      const T* prow = ws.prow + ((size_t)par * G + s_win) * k;
      for (int c = j + 1 + tid; c < k; c += kHessThreads) wgt[c] = ld_cg(prow + c);
      for (int i = tid; i < nr; i += kHessThreads) cj[i] = rn_div(cj[i], qr);
      __syncthreads();
      if (j + 1 < k) {
        T* cn = col(j + 1);
        const T wn = wgt[j + 1];
        for (int i = tid; i < nr; i += kHessThreads) cn[i] = rn_sub(cn[i], rn_mul(wn, cj[i]));
      }
    } else {
      for (int i = tid; i < nr; i += kHessThreads) cj[i] = T(0);
    }
    __syncthreads();
    if (j + 1 < k) publish(j + 1, keep);
    if (keep) {
      for (int c = j + 2 + warp; c < k; c += nwarps) {
        T* cc = col(c);
        const T wc = wgt[c];
        for (int i = lane; i < nr; i += 32) cc[i] = rn_sub(cc[i], rn_mul(wc, cj[i]));
      }
    }
    __syncthreads();
  }
  // write the result in the requested storage type (and W itself in slab mode)
  for (int c = warp; c < k; c += nwarps) {
    const T* src = col(c);
    T* dw = W + r0 + (int64_t)c * ldw;
    TO* dq = Q + r0 + (int64_t)c * ldq;
    for (int i = lane; i < nr; i += 32) {
      const T v = src[i];
      if (slab) dw[i] = v;
      if ((void*)Q != (void*)W) dq[i] = from_f64<TO>((double)v);
    }
  }
}

// FP32-arithmetic variant, same per-element arithmetic and results as
// k_hessenberg<float, TO>: a block on one CTA (the batched solver's concurrent
// problems), in shared memory where it fits, and the panels of blocks too tall
// for one resident column, in memory on the whole grid; other FP32 blocks take
// the resident kernels below.  Two changes to the per-column exchange:
//   - a CTA's candidate is one 64-bit word (value bits, global row, column
//     tag), written with a single release store and double-buffered by column
//     parity, so the wait for the candidates also delivers them;
//   - warp 0 reduces and publishes the next candidate (its row's trailing
//     entries, updated, go both to the published copy and back to the slab)
//     while the other warps apply the rank-1 update to every other row.
// Needs n < 2^24 - 1 (row field of the word).
constexpr unsigned kNoRow = 0xFFFFFFu;

__device__ __forceinline__ unsigned long long pack_cand(float v, unsigned row, int col) {
  return ((unsigned long long)__float_as_uint(v) << 32) | ((unsigned long long)(row & 0xFFFFFFu) << 8) |
         (unsigned long long)((col + 1) & 0xFF);
}

// Block argmax of (|value|, local row) with ties to the lower row as one
// 64-bit key: |value| bits above the complemented row (0: no candidate;
// value < 0 marks "none", NaN never wins).  A warp reduces with redux.sync,
// lane 0 folds the warp's key into a shared atomicMax.
__device__ __forceinline__ unsigned long long am_key(float av, int row) {
  return av >= 0.f ? ((unsigned long long)__float_as_uint(av) << 32) | (unsigned)(~row) : 0ull;
}
__device__ __forceinline__ unsigned long long warp_key_max(unsigned long long key) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
  const unsigned mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
  return ((unsigned long long)mhi << 32) | mlo;
}

template <typename TO>
__global__ void __launch_bounds__(kHessThreads) k_hessenberg_f32(
    int64_t n, int k, float* __restrict__ W, int64_t ldw, TO* __restrict__ Q, int64_t ldq,
    int* __restrict__ piv, float tol, HessWs<float> ws, int slab) {
  using T = float;
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = kHessThreads / 32;
  const int64_t rpc = ws.rpc > 0 ? ws.rpc : (n + G - 1) / G;
  const int64_t r0 = (int64_t)g * rpc;
  const int64_t r1 = r0 + rpc < n ? r0 + rpc : n;
  const int nr = r1 > r0 ? (int)(r1 - r0) : 0;

  extern __shared__ unsigned char smem_raw[];
  T* thr = reinterpret_cast<T*>(smem_raw);   // [k]
  T* wgt = thr + k;                          // [2][k] weights, by column parity
  // [k][ldv] in slab mode, 16-byte aligned; with rpc a multiple of 128 the
  // stride is rpc + 4 (column starts 4 banks apart: the candidate row's
  // entries, read across columns, meet 4-way instead of 32-way conflicts)
  // and the rank-1 update moves float4 chunks
  T* slabp = reinterpret_cast<T*>((reinterpret_cast<uintptr_t>(wgt + 2 * k) + 15) & ~(uintptr_t)15);
  T* const base = slab ? slabp : W + r0;
  const bool vec = slab && rpc % 128 == 0 && rpc <= 512;
  const int64_t ldv = slab ? (vec ? rpc + 4 : rpc) : ldw;
  auto col = [&](int c) -> T* { return base + (int64_t)c * ldv; };
  if (slab) {
    for (int c = warp; c < k; c += nwarps) {
      const T* src = W + r0 + (int64_t)c * ldw;
      T* dst = col(c);
      for (int i = lane; i < (int)ldv; i += 32) dst[i] = i < nr ? src[i] : T(0);  // zero padding rows
    }
    __syncthreads();
  }
  __shared__ T red_v[32];
  __shared__ int red_i[32];
  __shared__ T s_qr;
  __shared__ int s_r, s_keep;
  __shared__ unsigned long long s_key[2];  // block argmax keys, by column parity
  if (tid < 2) s_key[tid] = 0ull;

  for (int c = warp; c < k; c += nwarps) {
    T m = T(0);
    const T* cc = col(c);
    for (int i = lane; i < nr; i += 32) m = fmax(m, fabs(cc[i]));
    m = warp_max(m);
    if (lane == 0) ws.pcolmax[(size_t)g * k + c] = m;
  }
  if (!grid_barrier(ws.bar, G, ws.err)) return;
  for (int c = tid; c < k; c += kHessThreads) {
    T m = T(0);
    for (int h = 0; h < G; ++h) m = fmax(m, ld_cg(ws.pcolmax + (size_t)h * k + c));
    thr[c] = rn_mul(tol, ws.colmax_ext ? ws.colmax_ext[c] : m);
  }
  __syncthreads();

  // local argmax of |column jc| (first index on ties) -> s_r (local row or
  // INT_MAX); two CTA barriers
  auto local_argmax = [&](int jc) {
    const T* cj = col(jc);
    T bv = T(-1);
    int bi = INT_MAX;
    for (int i = tid; i < nr; i += kHessThreads) {
      T v = fabs(cj[i]);
      if (v > bv) {
        bv = v;
        bi = i;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      T ov = __shfl_xor_sync(0xffffffffu, bv, o);
      int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      argmax_merge(bv, bi, ov, oi);
    }
    if (lane == 0) {
      red_v[warp] = bv;
      red_i[warp] = bi;
    }
    __syncthreads();
    if (warp == 0) {
      bv = lane < nwarps ? red_v[lane] : T(-1);
      bi = lane < nwarps ? red_i[lane] : INT_MAX;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        T ov = __shfl_xor_sync(0xffffffffu, bv, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        argmax_merge(bv, bi, ov, oi);
      }
      if (lane == 0) s_r = bi;
    }
    __syncthreads();
  };
  // warp 0: publish the candidate of column jc (row rl): its entries jc+1..
  // after the pending update by column jc-1 (upd) go to the published row and
  // back to the slab; then the packed word
  auto publish_w0 = [&](int jc, bool upd, int rl) {
    const int par = jc & 1;
    T* prow = ws.prow + ((size_t)par * G + g) * k;
    if (rl != INT_MAX) {
      const T m = upd ? col(jc - 1)[rl] : T(0);
      for (int c = jc + 1 + lane; c < k; c += 32) {
        T v = col(c)[rl];
        if (upd) {
          v = rn_sub(v, rn_mul(wgt[c], m));
          col(c)[rl] = v;
        }
        prow[c] = v;
      }
    }
    __syncwarp();
    if (lane == 0) {
      const T v = rl != INT_MAX ? col(jc)[rl] : T(0);
      const unsigned row = rl != INT_MAX ? (unsigned)(r0 + rl) : kNoRow;
      __threadfence();
      word_release(ws.cand + (size_t)par * G + g, pack_cand(v, row, jc));
    }
  };

  // warp 0: wait (bounded) for every CTA's word for column jc, reduce to the
  // pivot, and load the pivot row's entries jc+1.. into the weight buffer of
  // column jc's parity; returns false on error
  auto await_pivot = [&](int jc) -> bool {
    const int par = jc & 1;
    const unsigned tag = (unsigned)((jc + 1) & 0xFF);
    const uint64_t t0 = global_timer_ns();
    T av = T(-1), sv = T(0);
    int ai = INT_MAX, ag = -1;
    bool ok = true;
    for (int h = lane; h < G; h += 32) {
      unsigned long long wv;
      while (((wv = word_acquire(ws.cand + (size_t)par * G + h)) & 0xFFull) != tag) {
        if (*(volatile int*)ws.err != 0 || global_timer_ns() - t0 > kWaitLimitNs) {
          atomicCAS(ws.err, 0, (int)RR_ERR_TIMEOUT);
          ok = false;
          break;
        }
      }
      if (!ok) break;
      const unsigned row = (unsigned)((wv >> 8) & 0xFFFFFFull);
      if (row == kNoRow) continue;
      const T hv = __uint_as_float((unsigned)(wv >> 32));
      const T ah = fabs(hv);
      if (ah > av || (ah == av && (int)row < ai)) {
        av = ah;
        ai = (int)row;
        ag = h;
        sv = hv;
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) return false;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      T ov = __shfl_xor_sync(0xffffffffu, av, o);
      int oi = __shfl_xor_sync(0xffffffffu, ai, o);
      int og = __shfl_xor_sync(0xffffffffu, ag, o);
      T osv = __shfl_xor_sync(0xffffffffu, sv, o);
      if (ov > av || (ov == av && oi < ai)) {
        av = ov;
        ai = oi;
        ag = og;
        sv = osv;
      }
    }
    const bool kp = ag >= 0 && sv != T(0) && fabs(sv) >= thr[jc];
    if (kp) {
      T* wb = wgt + (size_t)par * k;
      const T* prow = ws.prow + ((size_t)par * G + ag) * k;
      for (int c = jc + 1 + lane; c < k; c += 32) wb[c] = ld_cg(prow + c);
    }
    if (lane == 0) {
      s_qr = sv;
      s_keep = kp ? 1 : 0;
      if (g == 0) piv[jc] = kp ? ai : -1;
    }
    return true;
  };

  __shared__ int s_ok;
  local_argmax(0);
  if (warp == 0) {
    publish_w0(0, false, s_r);
    const bool ok = await_pivot(0);
    if (lane == 0) s_ok = ok ? 1 : 0;
  }
  __syncthreads();
  bool failed = !s_ok;
  for (int j = 0; j < k && !failed; ++j) {
    const bool keep = s_keep != 0;
    const T qr = s_qr;
    const T* wj = wgt + (size_t)(j & 1) * k;  // weights of column j
    T* cj = col(j);
    // (d) scale column j and update column j+1 row by row, tracking the local
    // argmax of the new column j+1 (first index on ties)
    {
      T* cn = j + 1 < k ? col(j + 1) : nullptr;
      const T wn = (keep && cn) ? wj[j + 1] : T(0);
      T bv = T(-1);
      int bi = INT_MAX;
      for (int i = tid; i < nr; i += kHessThreads) {
        T v = T(0);
        if (keep) v = rn_div(cj[i], qr);
        cj[i] = v;
        if (cn) {
          T u = cn[i];
          if (keep) u = rn_sub(u, rn_mul(wn, v));
          cn[i] = u;
          const T au = fabs(u);
          if (au > bv) {
            bv = au;
            bi = i;
          }
        }
      }
      const unsigned long long wk = warp_key_max(am_key(bv, bi));
      if (lane == 0 && wk) atomicMax(&s_key[j & 1], wk);
    }
    __syncthreads();
    const unsigned long long bkey = s_key[j & 1];
    const int bcand = bkey ? (int)(~(unsigned)bkey) : INT_MAX;  // the CTA's candidate row
    if (tid == 0) s_key[(j + 1) & 1] = 0ull;                    // read last in step j - 1
    if (j + 1 < k) {
      if (warp == 0) {
        // publish the candidate (its row takes column j's pending update,
        // written back to the slab), then wait for the pivot of column j+1
        // while the other warps apply column j's update
        const int rl = bcand;
        const int par = (j + 1) & 1;
        T* prow = ws.prow + ((size_t)par * G + g) * k;
        if (rl != INT_MAX) {
          const T m = cj[rl];
          for (int c = j + 2 + lane; c < k; c += 32) {
            T v = col(c)[rl];
            if (keep) {
              v = rn_sub(v, rn_mul(wj[c], m));
              col(c)[rl] = v;
            }
            prow[c] = v;
          }
        }
        __syncwarp();
        if (lane == 0) {
          const T v = rl != INT_MAX ? col(j + 1)[rl] : T(0);
          const unsigned row = rl != INT_MAX ? (unsigned)(r0 + rl) : kNoRow;
          __threadfence();
          word_release(ws.cand + (size_t)par * G + g, pack_cand(v, row, j + 1));
        }
        // the published candidate is what the other CTAs wait for: the bulk
        // update starts only now, so its shared-memory traffic does not delay it
        asm volatile("bar.arrive 1, %0;" ::"r"(kHessThreads) : "memory");
        const bool ok = await_pivot(j + 1);
        if (lane == 0) s_ok = ok ? 1 : 0;
      } else {
        asm volatile("bar.sync 1, %0;" ::"r"(kHessThreads) : "memory");
      }
      if (warp != 0 && keep) {
        // rank-1 update of columns j+2.. (all rows but the candidate's, which
        // warp 0 updates): the multiplier column in registers, independent
        // loads per target column
        const T* cj_c = cj;
        const int rl = bcand;
        constexpr int kR = 16;  // rows per lane held in registers (nr <= 512)
        // float4 chunks: lane rows 4 lane + 128 t (t < NC = rpc / 128); the
        // padding rows beyond nr are zero and stay finite
        auto upd4 = [&](auto nc) {
          constexpr int NC = decltype(nc)::value;
          float4 xr[NC];
#pragma unroll
          for (int t = 0; t < NC; ++t) xr[t] = reinterpret_cast<const float4*>(cj_c)[lane + 32 * t];
          for (int c = j + 2 + (warp - 1); c < k; c += nwarps - 1) {
            float4* cc = reinterpret_cast<float4*>(col(c));
            const T wc = wj[c];
            float4 yv[NC];
#pragma unroll
            for (int t = 0; t < NC; ++t) yv[t] = cc[lane + 32 * t];
#pragma unroll
            for (int t = 0; t < NC; ++t) {
              const int i0 = 4 * lane + 128 * t;
              float4 o = yv[t];
              o.x = i0 == rl ? yv[t].x : rn_sub(yv[t].x, rn_mul(wc, xr[t].x));
              o.y = i0 + 1 == rl ? yv[t].y : rn_sub(yv[t].y, rn_mul(wc, xr[t].y));
              o.z = i0 + 2 == rl ? yv[t].z : rn_sub(yv[t].z, rn_mul(wc, xr[t].z));
              o.w = i0 + 3 == rl ? yv[t].w : rn_sub(yv[t].w, rn_mul(wc, xr[t].w));
              if ((rl >> 2) == lane + 32 * t) {
                // the candidate's chunk: warp 0 writes row rl concurrently,
                // so only the other three rows are stored
                float* cs = reinterpret_cast<float*>(cc + lane + 32 * t);
                if (i0 != rl) cs[0] = o.x;
                if (i0 + 1 != rl) cs[1] = o.y;
                if (i0 + 2 != rl) cs[2] = o.z;
                if (i0 + 3 != rl) cs[3] = o.w;
              } else {
                cc[lane + 32 * t] = o;
              }
            }
          }
        };
        if (vec) {
          switch (rpc / 128) {
            case 1: upd4(std::integral_constant<int, 1>{}); break;
            case 2: upd4(std::integral_constant<int, 2>{}); break;
            case 3: upd4(std::integral_constant<int, 3>{}); break;
            default: upd4(std::integral_constant<int, 4>{}); break;
          }
        } else if (nr <= 32 * kR) {
          T xr[kR];
#pragma unroll
          for (int t = 0; t < kR; ++t) {
            const int i = lane + 32 * t;
            xr[t] = i < nr ? cj_c[i] : T(0);
          }
          for (int c = j + 2 + (warp - 1); c < k; c += nwarps - 1) {
            T* cc = col(c);
            const T wc = wj[c];
            T yv[kR];
#pragma unroll
            for (int t = 0; t < kR; ++t) {
              const int i = lane + 32 * t;
              yv[t] = i < nr ? cc[i] : T(0);
            }
#pragma unroll
            for (int t = 0; t < kR; ++t) {
              const int i = lane + 32 * t;
              if (i < nr && i != rl) cc[i] = rn_sub(yv[t], rn_mul(wc, xr[t]));
            }
          }
        } else {
          for (int c = j + 2 + (warp - 1); c < k; c += nwarps - 1) {
            T* cc = col(c);
            const T wc = wj[c];
            for (int i = lane; i < nr; i += 32)
              if (i != rl) cc[i] = rn_sub(cc[i], rn_mul(wc, cj_c[i]));
          }
        }
      }
      __syncthreads();
      if (!s_ok) failed = true;
    }
  }
  if (failed) return;
  for (int c = warp; c < k; c += nwarps) {
    const T* src = col(c);
    T* dw = W + r0 + (int64_t)c * ldw;
    TO* dq = Q + r0 + (int64_t)c * ldq;
    for (int i = lane; i < nr; i += 32) {
      const T v = src[i];
      if (slab) dw[i] = v;
      if ((void*)Q != (void*)W) dq[i] = from_f32<TO>(v);
    }
  }
}

template <typename T>
static size_t hess_ws_bytes(int64_t k, int G) {
  size_t b = 0;
  b += align_up(sizeof(int));
  b += align_up(sizeof(GridBarrier));
  b += align_up(2 * (size_t)G * sizeof(T));
  b += align_up(2 * (size_t)G * sizeof(int));
  b += align_up(2 * (size_t)G * k * sizeof(T));
  b += align_up((size_t)G * k * sizeof(T));
  b += align_up((size_t)G * sizeof(int));
  b += align_up(2 * (size_t)G * sizeof(unsigned long long));
  return b;
}

template <typename T, typename TO>
static rr_status hess_launch(int64_t n, int64_t k, T* W, int64_t ldw, TO* Q, int64_t ldq, int* piv,
                             double tol, void* ws, size_t ws_bytes, cudaStream_t s, int max_grid,
                             const T* colmax_ext = nullptr, bool reset_err = true) {
  // FP32 arithmetic: the packed-candidate kernel (rows must fit its 24-bit field)
  const bool packed = sizeof(T) == 4 && n < (int64_t)kNoRow;
  const void* fn = packed ? (const void*)k_hessenberg_f32<TO> : (const void*)k_hessenberg<T, TO>;
  // Grid: about 256 rows per CTA (fewer CTAs make the per-column barrier and
  // candidate reduction cheaper), more CTAs if a slab would not fit in shared
  // memory; slab mode when the CTA's rows of all k columns fit in 200 KB.
  const size_t kSlabLimit = 200 * 1024;
  int G;
  int slab = 0;
  if (max_grid == 1) {
    G = 1;
  } else {
    int64_t g = (n + 255) / 256;
    const int64_t fit = (int64_t)(kSlabLimit / ((size_t)k * sizeof(T)));  // rows per CTA that fit
    if (fit > 0 && (n + g - 1) / g > fit) g = (n + fit - 1) / fit;
    if (g > num_sms()) g = num_sms();
    if (g < 1) g = 1;
    G = (int)g;
  }
  int64_t rpc = (n + G - 1) / G;
  if (packed) {
    // rows per CTA a multiple of 128 where the slab still fits: the FP32
    // kernel's float4 update and padded stride (fewer CTAs when it rounds up)
    const int64_t r128 = (rpc + 127) / 128 * 128;
    if (r128 <= 512 && (size_t)(r128 + 4) * k * sizeof(T) <= kSlabLimit) {
      rpc = r128;
      G = (int)((n + rpc - 1) / rpc);
    }
  }
  const int64_t ldv = (packed && rpc % 128 == 0 && rpc <= 512) ? rpc + 4 : rpc;
  const size_t fixed = (packed ? 3 : 2) * (size_t)k * sizeof(T) + 16;  // thresholds, weights, alignment
  if ((size_t)ldv * k * sizeof(T) <= kSlabLimit && (size_t)ldv * k * sizeof(T) + fixed <= 220 * 1024) slab = 1;
  size_t smem = fixed + (slab ? (size_t)ldv * k * sizeof(T) : 0);
  RR_TRY(allow_dynamic_smem(fn, smem));
  if (ws_bytes < hess_ws_bytes<T>(k, G) || !ws) return RR_ERR_WORKSPACE;
  Arena ar(ws, ws_bytes);
  HessWs<T> h;
  h.err = ar.take<int>(1);
  h.bar = ar.take<GridBarrier>(1);
  h.pval = ar.take<T>(2 * (size_t)G);
  h.pidx = ar.take<int>(2 * (size_t)G);
  h.prow = ar.take<T>(2 * (size_t)G * k);
  h.pcolmax = ar.take<T>((size_t)G * k);
  h.flags = ar.take<int>(G);
  h.cand = ar.take<unsigned long long>(2 * (size_t)G);
  h.rpc = packed ? rpc : 0;
  h.colmax_ext = packed ? colmax_ext : nullptr;
  if (reset_err) RR_CUDA(cudaMemsetAsync(ws, 0, 512, s));  // err + barrier
  RR_CUDA(cudaMemsetAsync(h.flags, 0, (size_t)G * sizeof(int), s));
  RR_CUDA(cudaMemsetAsync(h.cand, 0, 2 * (size_t)G * sizeof(unsigned long long), s));
  T t = tol > 0 ? (T)tol : (T)(4.0 * (double)k * (sizeof(T) == 4 ? 0x1p-23 : 0x1p-52));
  int kk = (int)k;
  void* args[] = {&n, &kk, &W, &ldw, &Q, &ldq, &piv, &t, &h, &slab};
  if (G == 1) {
    // a single CTA never waits on another one: plain launch (graph-capturable,
    // safe to run concurrently with other work)
    RR_CUDA(cudaLaunchKernel(fn, dim3(1), dim3(kHessThreads), args, smem, s));
    return check_launch("rr_hessenberg");
  }
  RR_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kHessThreads), args, smem, s));
  note_launches(1);
  return RR_OK;
}

// ---------------------------------------------------------------------------
// FP32 process on a block held in the CTAs' shared memory (rows spread over
// the CTAs), in panels of 8 columns with the same operations in the same order
// as Algorithm 8, so with its results bit for bit (see the blocked process
// below for why panels do not change them).
//
// What bounds it is the chain of k pivot exchanges.  Per column:
//   - the row threads scale column j, update column j + 1 and find its largest
//     entry; the thread that owns that row updates the row's remaining panel
//     entries and publishes value, row and entries as three 16-byte words, each
//     with the column's tag and each stored and read as one 128-bit access, so
//     that neither a fence nor a second trip for the pivot row is needed;
//   - meanwhile the other rows take column j's update in the panel's remaining
//     columns, and one warp per 32 CTAs polls the words of column j + 1.
// A pivot row's entries beyond the panel go to memory while the panel runs on;
// after the panel every CTA forms the trailing weights by forward substitution
// and updates its rows of the trailing columns from shared memory.
// 16384 x 128: 0.47 ms (0.57 to 0.76 ms with a fenced word and the winner's row
// read behind it, a column at a time), 4096 x 128 in one cluster 0.26 ms (0.42).
// Panels of a block too tall to be resident (1048576 rows: 8 columns fit) run
// as blocks of their own, 85 us each: 1048576 x 160 takes 3.9 ms (14.9 ms with
// 16-column panels in global memory).
// ---------------------------------------------------------------------------
constexpr int kPanelMax = 32;       // columns of a blocked panel
constexpr int kPw = 8;              // columns of a resident panel
constexpr int kRowThreads = 512;
constexpr int kHessMaxCluster = 16;
constexpr int kMaxPoll = 5;         // polling warps: up to 160 CTAs

struct HessRes {
  int* err;
  GridBarrier* bar;
  unsigned* colmax;         // [k] bits of the column inf-norms, zero on entry
  const float* colmax_ext;  // [k] the norms, where the caller has them (else null)
  uint4* msg;               // [2][3][G] candidate words, by column parity: the
                            // CTAs' words side by side, so that a polling warp's
                            // loads fall in few lines
  float* rowbuf;            // [2][kPw][k + kPw] pivot rows, by panel parity
  int* flags;               // [2][kPw] their tags
  int tag0;                 // tag of column j: tag0 + j + 1
  int rpc;                  // rows per CTA
};

__device__ __forceinline__ void st_b128(uint4* p, uint4 v) {
  asm volatile(
      "{\n\t.reg .b128 t;\n\t.reg .b64 lo, hi;\n\t"
      "mov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\tmov.b128 t, {lo, hi};\n\t"
      "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
      : "memory");
}
__device__ __forceinline__ uint4 ld_b128(const uint4* p) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .b128 t;\n\t.reg .b64 lo, hi;\n\t"
      "ld.relaxed.gpu.global.b128 t, [%4];\n\tmov.b128 {lo, hi}, t;\n\t"
      "mov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p)
      : "memory");
  return v;
}

// 32 bits and a tag as one 64-bit word, to a CTA of the cluster and from this one
__device__ __forceinline__ void mail_put(unsigned long long* p, unsigned v, unsigned tag) {
  asm volatile("st.relaxed.cluster.b64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)tag << 32) | v) : "memory");
}
__device__ __forceinline__ unsigned long long mail_get(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.cluster.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

struct HessSlot {  // the best candidate a polling warp saw
  unsigned long long key;  // |value| bits above the complemented row, 0: none
  float val;
  int row;
  float f[kPw - 1];        // its entries in the panel columns after the pivot's
};

// any number of rows per CTA (rows in shared memory only)
template <typename TO>
__global__ void __launch_bounds__(kRowThreads + 32 * kMaxPoll, 1) k_hess_res(
    int64_t n, int k, float* __restrict__ W, int64_t ldw, TO* __restrict__ Q, int64_t ldq, int* __restrict__ piv,
    float tol, HessRes ws) {
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = blockDim.x >> 5, npoll = nwarps - kRowThreads / 32;
  const int rpc = ws.rpc, ldv = rpc | 1;  // odd stride: a row's entries lie in different banks
  const int64_t r0 = (int64_t)g * rpc;
  const int nr = (int)(n - r0 < rpc ? (n > r0 ? n - r0 : 0) : rpc);
  extern __shared__ __align__(16) float sm_f[];
  float* const slab = sm_f;                              // [k][ldv]
  float* const thr = slab + (size_t)k * ldv;             // [k]
  float* const wts = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(thr + k) + 15) & ~(uintptr_t)15);  // [nt][kPw]
  __shared__ HessSlot slot[2][kMaxPoll];
  __shared__ unsigned long long s_key[2][kRowThreads / 32];           // the row warps' best keys, by column parity
  __shared__ float s_l[kPw][kPw];
  __shared__ int s_kept[kPw];
  // a wait that ran out, by column parity (a warp already polling for the next
  // column must not turn the others back) and for the trailing part
  __shared__ int s_bad[3];
  auto col = [&](int c) -> float* { return slab + (size_t)c * ldv; };

  for (int c = warp; c < k; c += nwarps) {
    const float* src = W + r0 + (int64_t)c * ldw;
    float* dst = col(c);
    float m = 0.f;
#pragma unroll 8
    for (int i = lane; i < nr; i += 32) {
      const float v = src[i];
      dst[i] = v;
      m = fmaxf(m, fabsf(v));
    }
    if (!ws.colmax_ext) {
      m = warp_max(m);
      if (lane == 0) atomicMax(ws.colmax + c, __float_as_uint(m));
    }
  }
  if (tid < 3) s_bad[tid] = 0;
  if (!ws.colmax_ext && !grid_barrier(ws.bar, G, ws.err)) return;
  for (int c = tid; c < k; c += blockDim.x)
    thr[c] = __fmul_rn(tol, ws.colmax_ext ? ws.colmax_ext[c] : __uint_as_float(__ldcg(ws.colmax + c)));
  __syncthreads();


  // this CTA's candidate for column j (row < 0: none)
  auto publish = [&](int j, float value, int rl, const float (&f)[kPw - 1]) {
      const unsigned tag = (unsigned)(ws.tag0 + j + 1), row = rl < 0 ? kNoRow : (unsigned)(r0 + rl);
      uint4* m = ws.msg + (size_t)(j & 1) * 3 * G + g;
      st_b128(m, make_uint4(__float_as_uint(value), row, tag, __float_as_uint(f[0])));
      st_b128(m + G, make_uint4(__float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]), tag));
      st_b128(m + 2 * G, make_uint4(__float_as_uint(f[4]), __float_as_uint(f[5]), __float_as_uint(f[6]), tag));
  };
  // polling warps: every CTA's words for column j (bounded), the best to the slot
  auto poll = [&](int j) {
    const unsigned tag = (unsigned)(ws.tag0 + j + 1);
    const int pwi = warp - kRowThreads / 32, h = pwi * 32 + lane;
    // not before this CTA has published: the others are no earlier, and the
    // polling loads would stand in the way of its shared-memory accesses
    asm volatile("bar.sync 2, %0;" ::"r"(blockDim.x) : "memory");
    unsigned long long key = 0ull;
    unsigned val = 0u, row = kNoRow;
    uint4 a, b, c;
    bool ok = true;
    if (h < G) {
      uint64_t t0 = 0;
      for (int spin = 1;; ++spin) {
        {
          const uint4* m = ws.msg + (size_t)(j & 1) * 3 * G + h;
          a = ld_b128(m);
          b = ld_b128(m + G);
          c = ld_b128(m + 2 * G);
          if (a.z == tag && b.w == tag && c.w == tag) {
            val = a.x;
            row = a.y;
            break;
          }
        }
        if ((spin & 63) == 0) {
          const uint64_t t = global_timer_ns();
          if (t0 == 0) t0 = t;
          if (*(volatile int*)ws.err != 0 || t - t0 > kWaitLimitNs) {
            atomicCAS(ws.err, 0, (int)RR_ERR_TIMEOUT);
            ok = false;
            break;
          }
        }
      }
      if (ok && row != kNoRow) key = ((unsigned long long)(val & 0x7FFFFFFFu) << 32) | (unsigned)(~row);
    }
    if (!ok) s_bad[j & 1] = 1;
    const unsigned long long best = warp_key_max(key);
    HessSlot& s = slot[j & 1][pwi];
    if (best == 0ull) {
      if (lane == 0) s.key = 0ull;
    } else if (key == best) {
      s.key = key;
      s.val = __uint_as_float(val);
      s.row = (int)row;
      s.f[0] = __uint_as_float(a.w);
      s.f[1] = __uint_as_float(b.x);
      s.f[2] = __uint_as_float(b.y);
      s.f[3] = __uint_as_float(b.z);
      s.f[4] = __uint_as_float(c.x);
      s.f[5] = __uint_as_float(c.y);
      s.f[6] = __uint_as_float(c.z);
    }
  };
  // row threads: the CTA's candidate row of column j from every thread's
  // largest |entry| (-1: none).  (A 64-bit atomic maximum in shared memory is a
  // compare-and-swap loop: about 800 cycles for 16 warps.)
  auto candidate = [&](int j, float bv, int bi) -> int {
    const unsigned long long wk = warp_key_max(am_key(bv, bi));
    if (lane == 0) s_key[j & 1][warp] = wk;
    asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
    const unsigned long long key = warp_key_max(s_key[j & 1][lane & (kRowThreads / 32 - 1)]);
    return key ? (int)(~(unsigned)key) : -1;
  };

  bool failed = false;  // (the same in every thread)
  for (int b = 0, panel = 0; b < k && !failed; b += kPw, ++panel) {
    const int pe = min(b + kPw, k), nt = k - pe, par = panel & 1;
    float* const rows = ws.rowbuf + (size_t)par * kPw * (k + kPw);
    // the first column's candidate (its row has no pending update)
    if (warp < kRowThreads / 32) {
      float bv = -1.f;
      int bi = INT_MAX;
      const float* cb = col(b);
      for (int i = tid; i < nr; i += kRowThreads) {
        const float v = fabsf(cb[i]);
        if (v > bv) {
          bv = v;
          bi = i;
        }
      }
      const int rl = candidate(b, bv, bi);
      if (rl >= 0 ? tid == rl % kRowThreads : tid == 0) {
        float f[kPw - 1];
#pragma unroll
        for (int c = 0; c < kPw - 1; ++c) f[c] = rl >= 0 && b + 1 + c < pe ? col(b + 1 + c)[rl] : 0.f;
        publish(b, rl >= 0 ? cb[rl] : 0.f, rl, f);
      }
      asm volatile("bar.arrive 2, %0;" ::"r"(blockDim.x) : "memory");
    } else {
      poll(b);
    }
    for (int j = b; j < pe; ++j) {
      __syncthreads();
      if (s_bad[j & 1]) {
        failed = true;
        break;
      }
      // the pivot of column j
      const HessSlot* best = &slot[j & 1][0];
      for (int q = 1; q < npoll; ++q)
        if (slot[j & 1][q].key > best->key) best = &slot[j & 1][q];
      const float qr = best->val;
      const bool keep = best->key != 0ull && qr != 0.f && fabsf(qr) >= thr[j];
      if (tid == 0) {
        if (g == 0) piv[j] = keep ? best->row : -1;
        s_kept[j - b] = keep;
      }
      if (warp >= kRowThreads / 32) {
        // the pivot row beyond the panel, and its multipliers in the panel
        if (warp == kRowThreads / 32 && nt > 0 && keep && best->row >= r0 && best->row < r0 + nr) {
          const int rl = (int)(best->row - r0);
          float* dst = rows + (size_t)(j - b) * (k + kPw);
          if (lane < kPw) dst[lane] = b + lane < j ? col(b + lane)[rl] : 0.f;
          for (int c = lane; c < nt; c += 32) dst[kPw + c] = col(pe + c)[rl];
          __syncwarp();
          if (lane == 0) {
            __threadfence();
            flag_release(ws.flags + par * kPw + (j - b), ws.tag0 + j + 1);
          }
          __syncwarp();
        }
        if (j + 1 < pe) poll(j + 1);
        continue;
      }
      float* cj = col(j);
      if (j + 1 == pe) {
        for (int i = tid; i < nr; i += kRowThreads) cj[i] = keep ? __fdiv_rn(cj[i], qr) : 0.f;
        continue;
      }
      float wt[kPw - 1];  // weights of the panel columns j + 1 ..
#pragma unroll
      for (int c = 0; c < kPw - 1; ++c) wt[c] = best->f[c];
      float* cn = cj + ldv;
      float bv = -1.f;
      int bi = INT_MAX;
      if (keep) {
#pragma unroll 4
        for (int i = tid; i < nr; i += kRowThreads) {
          const float v = __fdiv_rn(cj[i], qr);
          const float u = __fsub_rn(cn[i], __fmul_rn(wt[0], v));
          cj[i] = v;
          cn[i] = u;
          if (fabsf(u) > bv) {
            bv = fabsf(u);
            bi = i;
          }
        }
      } else {
        for (int i = tid; i < nr; i += kRowThreads) {
          cj[i] = 0.f;
          if (fabsf(cn[i]) > bv) {
            bv = fabsf(cn[i]);
            bi = i;
          }
        }
      }
      const int rl = candidate(j + 1, bv, bi);
      const int nc = pe - (j + 2);  // panel columns left to update
      if (rl >= 0 ? tid == rl % kRowThreads : tid == 0) {
        float f[kPw - 1];
        const float v = rl >= 0 ? cj[rl] : 0.f;
#pragma unroll
        for (int c = 0; c < kPw - 1; ++c) {
          f[c] = 0.f;
          if (c < nc && rl >= 0) {
            float* cc = col(j + 2 + c) + rl;
            f[c] = keep && c + 1 < kPw - 1 ? __fsub_rn(*cc, __fmul_rn(wt[c + 1 < kPw - 1 ? c + 1 : 0], v)) : *cc;
            *cc = f[c];
          }
        }
        publish(j + 1, rl >= 0 ? cn[rl] : 0.f, rl, f);
      }
      asm volatile("bar.arrive 2, %0;" ::"r"(blockDim.x) : "memory");
      if (keep && nc > 0) {
#pragma unroll 2
        for (int i = tid; i < nr; i += kRowThreads) {
          if (i == rl) continue;  // its owner, this thread, has done it
          const float v = cj[i];
          float* cc = col(j + 2) + i;
#pragma unroll
          for (int c = 0; c < kPw - 2; ++c)
            if (c < nc) cc[(size_t)c * ldv] = __fsub_rn(cc[(size_t)c * ldv], __fmul_rn(wt[c + 1], v));
        }
      }
    }
    if (failed) break;
    __syncthreads();
    if (nt == 0) break;
    // ---- trailing columns ----
    if (tid < kPw && b + tid < pe && s_kept[tid]) {
      const uint64_t t0 = global_timer_ns();
      while (flag_acquire(ws.flags + par * kPw + tid) != ws.tag0 + b + tid + 1) {
        if (*(volatile int*)ws.err != 0 || global_timer_ns() - t0 > kWaitLimitNs) {
          atomicCAS(ws.err, 0, (int)RR_ERR_TIMEOUT);
          s_bad[2] = 1;
          break;
        }
      }
    }
    __syncthreads();
    if (s_bad[2]) {
      failed = true;
      break;
    }
    if (tid < kPw * kPw) s_l[tid / kPw][tid % kPw] = __ldcg(rows + (size_t)(tid / kPw) * (k + kPw) + tid % kPw);
    __syncthreads();
    for (int c = tid; c < nt; c += blockDim.x) {
      float w[kPw];
#pragma unroll
      for (int q = 0; q < kPw; ++q) w[q] = s_kept[q] ? __ldcg(rows + (size_t)q * (k + kPw) + kPw + c) : 0.f;
#pragma unroll
      for (int q = 1; q < kPw; ++q)
        if (s_kept[q]) {
#pragma unroll
          for (int i = 0; i < q; ++i)
            if (s_kept[i]) w[q] = __fsub_rn(w[q], __fmul_rn(w[i], s_l[q][i]));
        }
#pragma unroll
      for (int q = 0; q < kPw; ++q) wts[c * kPw + q] = w[q];
    }
    __syncthreads();
    // (a skipped column has zero multipliers and zero weights: its step
    // subtracts zero and changes nothing)
    for (int i0 = 0; i0 < nr; i0 += 128) {
      float l[4][kPw];
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int q = 0; q < kPw; ++q) l[t][q] = i0 + lane + 32 * t < nr ? col(b + q)[i0 + lane + 32 * t] : 0.f;
      for (int c = warp; c < nt; c += nwarps) {
        float* cc = col(pe + c) + i0 + lane;
        const float4 wa = reinterpret_cast<const float4*>(wts + c * kPw)[0];
        const float4 wb = reinterpret_cast<const float4*>(wts + c * kPw)[1];
        const float w[kPw] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
        float x[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) x[t] = i0 + lane + 32 * t < nr ? cc[32 * t] : 0.f;
#pragma unroll
        for (int q = 0; q < kPw; ++q)
#pragma unroll
          for (int t = 0; t < 4; ++t) x[t] = __fsub_rn(x[t], __fmul_rn(w[q], l[t][q]));
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (i0 + lane + 32 * t < nr) cc[32 * t] = x[t];
      }
    }
    __syncthreads();
  }
  if (failed) return;
  for (int c = warp; c < k; c += nwarps) {
    const float* src = col(c);
    float* dw = W + r0 + (int64_t)c * ldw;
    TO* dq = Q + r0 + (int64_t)c * ldq;
#pragma unroll 4
    for (int i = lane; i < nr; i += 32) {
      const float v = src[i];
      dw[i] = v;
      if ((void*)Q != (void*)W) dq[i] = from_f32<TO>(v);
    }
  }
}

struct alignas(16) HessBest {  // the best candidate a polling warp saw
  float f[kPw];                // its entries in the panel columns after the pivot's
  float val;
  int row;
  unsigned hi;                 // |value| bits + 1, 0: none
  unsigned pad;
};

// The same process where a CTA has at most 512 rows: a thread per row, its
// panel entries in registers.  With one row a thread a column step is some
// hundred instructions per warp and their latency is what counts next to the
// exchange, so all of a row's panel entries take the update at once and no row
// needs a path of its own.
//
// CL: the CTAs form one thread-block cluster (G <= kHessMaxCluster): the
// candidate's warp writes it into every CTA's shared memory as 64-bit words of
// 32 bits and the column's tag, and each CTA polls its own copy (polling the
// other CTAs' memory took 2900 cycles a column and reading the winner's
// entries behind the word another 1500).
template <typename TO, bool CL>
__global__ void __launch_bounds__(kRowThreads + 32 * kMaxPoll, 1) k_hess_row(
    int64_t n, int k, float* __restrict__ W, int64_t ldw, TO* __restrict__ Q, int64_t ldq, int* __restrict__ piv,
    float tol, HessRes ws, int rt) {
  // rt: row threads, a multiple of 32; the other warps poll
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = blockDim.x >> 5, nrow = rt >> 5, npoll = nwarps - nrow;
  const int rpc = ws.rpc, ldv = rpc | 1;  // odd stride: a row's entries lie in different banks
  const int64_t r0 = (int64_t)g * rpc;
  const int nr = (int)(n - r0 < rpc ? (n > r0 ? n - r0 : 0) : rpc);
  extern __shared__ __align__(16) float sm_f[];
  float* const slab = sm_f;                              // [k][ldv]
  float* const thr = slab + (size_t)k * ldv;             // [k]
  float* const wts = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(thr + k) + 15) & ~(uintptr_t)15);  // [nt][kPw]
  __shared__ HessBest best[2][kMaxPoll];
  __shared__ unsigned long long s_mail[2][kHessMaxCluster][kPw + 2];  // CL: words by column parity and sender
  __shared__ unsigned long long s_key[2][kRowThreads / 32];
  __shared__ float s_l[kPw][kPw];
  __shared__ int s_kept[kPw], s_bad[3];
  if constexpr (CL)
    if (cooperative_groups::this_cluster().num_blocks() != gridDim.x) {
      if (tid == 0) atomicCAS(ws.err, 0, (int)RR_ERR_CUDA);
      return;  // every CTA alike
    }

  for (int c = warp; c < k; c += nwarps) {
    const float* src = W + r0 + (int64_t)c * ldw;
    float* dst = slab + (size_t)c * ldv;
    float m = 0.f;
#pragma unroll 8
    for (int i = lane; i < nr; i += 32) {
      const float v = src[i];
      dst[i] = v;
      m = fmaxf(m, fabsf(v));
    }
    if (!ws.colmax_ext) {
      m = warp_max(m);
      if (lane == 0) atomicMax(ws.colmax + c, __float_as_uint(m));
    }
  }
  if (tid < 3) s_bad[tid] = 0;
  if (CL)  // no column's tag
    for (int e = tid; e < 2 * kHessMaxCluster * (kPw + 2); e += blockDim.x) (&s_mail[0][0][0])[e] = 0ull;
  if (!ws.colmax_ext && !grid_barrier(ws.bar, G, ws.err)) return;
  for (int c = tid; c < k; c += blockDim.x)
    thr[c] = __fmul_rn(tol, ws.colmax_ext ? ws.colmax_ext[c] : __uint_as_float(__ldcg(ws.colmax + c)));
  __syncthreads();
  if constexpr (CL) cooperative_groups::this_cluster().sync();  // the words are zero before anyone reads them

  // row threads: the CTA's candidate for column j is the row with the largest
  // |x[0]| (first row on ties); its thread publishes value, row and x[1 ..]
  auto offer = [&](int j, const float (&x)[kPw], int first) {
    float u = 0.f;
    float f[kPw - 1];
#pragma unroll
    for (int c = 0; c < kPw - 1; ++c) f[c] = 0.f;
#pragma unroll
    for (int c = 0; c < kPw; ++c) {
      if (c == first) u = x[c];
    }
#pragma unroll
    for (int s = 0; s < kPw; ++s)
      if (s == first) {
#pragma unroll
        for (int c = s + 1; c < kPw; ++c) f[c - s - 1] = x[c];
      }
    const unsigned ab = __float_as_uint(u) & 0x7FFFFFFFu;
    const unsigned hi = tid < nr && ab <= 0x7F800000u ? ab + 1u : 0u;  // NaN and rows past the end never win
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const bool mine = mh != 0u && lane == __ffs(__ballot_sync(0xffffffffu, hi == mh)) - 1;
    if (mine) s_key[j & 1][warp] = ((unsigned long long)mh << 32) | (unsigned)tid;
    else if (mh == 0u && lane == 0) s_key[j & 1][warp] = 0ull;
    asm volatile("bar.sync 1, %0;" ::"r"(rt) : "memory");
    const unsigned kh = lane < nrow ? (unsigned)(s_key[j & 1][lane] >> 32) : 0u;
    const unsigned bh = __reduce_max_sync(0xffffffffu, kh);
    const int bw = __ffs(__ballot_sync(0xffffffffu, kh == bh)) - 1;  // lower warps have lower rows
    const unsigned tag = (unsigned)(ws.tag0 + j + 1);
    if constexpr (CL) {
      if (warp == (bh ? bw : 0)) {
        const int src = bh ? __ffs(__ballot_sync(0xffffffffu, mine)) - 1 : 0;
        const float v = __shfl_sync(0xffffffffu, u, src);
        const unsigned row = bh ? (unsigned)(r0 + warp * 32 + src) : kNoRow;
#pragma unroll
        for (int c = 0; c < kPw - 1; ++c) f[c] = __shfl_sync(0xffffffffu, f[c], src);
        if (lane < G) {
          unsigned long long* m = cooperative_groups::this_cluster().map_shared_rank(&s_mail[j & 1][g][0], lane);
          mail_put(m, __float_as_uint(v), tag);
          mail_put(m + 1, row, tag);
#pragma unroll
          for (int c = 0; c < kPw - 1; ++c) mail_put(m + 2 + c, __float_as_uint(f[c]), tag);
        }
      }
    } else if (bh != 0u ? mine && warp == bw : tid == 0) {
      const unsigned row = bh ? (unsigned)(r0 + tid) : kNoRow;
      uint4* m = ws.msg + (size_t)(j & 1) * 3 * G + g;
      st_b128(m, make_uint4(__float_as_uint(u), row, tag, __float_as_uint(f[0])));
      st_b128(m + G, make_uint4(__float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]), tag));
      st_b128(m + 2 * G, make_uint4(__float_as_uint(f[4]), __float_as_uint(f[5]), __float_as_uint(f[6]), tag));
    }
    asm volatile("bar.arrive 2, %0;" ::"r"(blockDim.x) : "memory");
  };
  // polling warps: every CTA's word for column j (bounded), the best to best[j & 1]
  auto poll = [&](int j) {
    const int pwi = warp - nrow, h = pwi * 32 + lane;
    // not before this CTA has published: the others are no earlier
    asm volatile("bar.sync 2, %0;" ::"r"(blockDim.x) : "memory");
    unsigned hi = 0u, val = 0u, row = kNoRow;
    uint4 a, b, c;
    [[maybe_unused]] unsigned mw[kPw + 1];
    bool ok = true;
    if (h < G) {
      uint64_t t0 = 0;
      const unsigned tag = (unsigned)(ws.tag0 + j + 1);
      for (int spin = 1;; ++spin) {
        if constexpr (CL) {
          bool all = true;
          const unsigned long long* m = &s_mail[j & 1][h][0];
#pragma unroll
          for (int q = 0; q < kPw + 1; ++q) {
            const unsigned long long w = mail_get(m + q);
            mw[q] = (unsigned)w;
            all &= (unsigned)(w >> 32) == tag;
          }
          if (all) {
            val = mw[0];
            row = mw[1];
            break;
          }
        } else {
          const uint4* m = ws.msg + (size_t)(j & 1) * 3 * G + h;
          a = ld_b128(m);
          b = ld_b128(m + G);
          c = ld_b128(m + 2 * G);
          if (a.z == tag && b.w == tag && c.w == tag) {
            val = a.x;
            row = a.y;
            break;
          }
        }
        if ((spin & 63) == 0) {
          const uint64_t t = global_timer_ns();
          if (t0 == 0) t0 = t;
          if (*(volatile int*)ws.err != 0 || t - t0 > kWaitLimitNs) {
            atomicCAS(ws.err, 0, (int)RR_ERR_TIMEOUT);
            ok = false;
            break;
          }
        }
      }
      if (ok && row != kNoRow) hi = (val & 0x7FFFFFFFu) + 1u;
    }
    if (!ok) s_bad[j & 1] = 1;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    HessBest& s = best[j & 1][pwi];
    if (mh == 0u) {
      if (lane == 0) s.hi = 0u;
    } else if (lane == __ffs(__ballot_sync(0xffffffffu, hi == mh)) - 1) {  // lower CTAs have lower rows
      s.hi = mh;
      s.val = __uint_as_float(val);
      s.row = (int)row;
      if constexpr (CL) {
#pragma unroll
        for (int q = 0; q < kPw - 1; ++q) s.f[q] = __uint_as_float(mw[2 + q]);
      } else {
        s.f[0] = __uint_as_float(a.w);
        s.f[1] = __uint_as_float(b.x);
        s.f[2] = __uint_as_float(b.y);
        s.f[3] = __uint_as_float(b.z);
        s.f[4] = __uint_as_float(c.x);
        s.f[5] = __uint_as_float(c.y);
        s.f[6] = __uint_as_float(c.z);
      }
    }
  };

  bool failed = false;  // (the same in every thread)
  for (int b = 0, panel = 0; b < k && !failed; b += kPw, ++panel) {
    const int pe = min(b + kPw, k), nt = k - pe, par = panel & 1;
    float* const rows = ws.rowbuf + (size_t)par * kPw * (k + kPw);
    float x[kPw];  // this row's panel entries
    const bool rowt = warp < nrow, live = rowt && tid < nr;
#pragma unroll
    for (int c = 0; c < kPw; ++c) x[c] = live && b + c < pe ? slab[(size_t)(b + c) * ldv + tid] : 0.f;
    if (rowt) offer(b, x, 0);
    else poll(b);
#pragma unroll
    for (int jj = 0; jj < kPw; ++jj) {
      const int j = b + jj;
      if (j >= pe || failed) break;
      __syncthreads();
      if (s_bad[j & 1]) {
        failed = true;
        break;
      }
      // the pivot of column j
      int bi = 0;
      unsigned bh = best[j & 1][0].hi;
      for (int q = 1; q < npoll; ++q) {
        const unsigned h = best[j & 1][q].hi;
        if (h > bh) {
          bh = h;
          bi = q;
        }
      }
      const HessBest* bp = &best[j & 1][bi];
      const float qr = bp->val;
      const bool keep = bh != 0u && qr != 0.f && fabsf(qr) >= thr[j];
      if (rowt) {
        float w[kPw];
        const float4 fa = reinterpret_cast<const float4*>(bp->f)[0], fb = reinterpret_cast<const float4*>(bp->f)[1];
        w[0] = fa.x, w[1] = fa.y, w[2] = fa.z, w[3] = fa.w, w[4] = fb.x, w[5] = fb.y, w[6] = fb.z, w[7] = 0.f;
        if (keep) {
          x[jj] = __fdiv_rn(x[jj], qr);
#pragma unroll
          for (int c = jj + 1; c < kPw; ++c) x[c] = __fsub_rn(x[c], __fmul_rn(w[c - jj - 1], x[jj]));
        } else {
          x[jj] = 0.f;
        }
        if (live) slab[(size_t)j * ldv + tid] = x[jj];
        if (tid == 0) {
          if (g == 0) piv[j] = keep ? bp->row : -1;
          s_kept[jj] = keep;
        }
        if (jj + 1 < kPw && j + 1 < pe) offer(j + 1, x, jj + 1);
      } else {
        // the pivot row beyond the panel, and its multipliers in the panel
        if (warp == nrow && nt > 0 && keep && bp->row >= r0 && bp->row < r0 + nr) {
          const int rl = (int)(bp->row - r0);
          float* dst = rows + (size_t)jj * (k + kPw);
          if (lane < kPw) dst[lane] = lane < jj ? slab[(size_t)(b + lane) * ldv + rl] : 0.f;
          for (int c = lane; c < nt; c += 32) dst[kPw + c] = slab[(size_t)(pe + c) * ldv + rl];
          __syncwarp();
          if (lane == 0) {
            __threadfence();
            flag_release(ws.flags + par * kPw + jj, ws.tag0 + j + 1);
          }
          __syncwarp();
        }
        if (j + 1 < pe) poll(j + 1);
      }
    }
    if (failed || nt == 0) break;
    __syncthreads();
    // ---- trailing columns ----
    if (tid < kPw && b + tid < pe && s_kept[tid]) {
      const uint64_t t0 = global_timer_ns();
      while (flag_acquire(ws.flags + par * kPw + tid) != ws.tag0 + b + tid + 1) {
        if (*(volatile int*)ws.err != 0 || global_timer_ns() - t0 > kWaitLimitNs) {
          atomicCAS(ws.err, 0, (int)RR_ERR_TIMEOUT);
          s_bad[2] = 1;
          break;
        }
      }
    }
    __syncthreads();
    if (s_bad[2]) {
      failed = true;
      break;
    }
    if (tid < kPw * kPw) s_l[tid / kPw][tid % kPw] = __ldcg(rows + (size_t)(tid / kPw) * (k + kPw) + tid % kPw);
    __syncthreads();
    for (int c = tid; c < nt; c += blockDim.x) {
      float w[kPw];
#pragma unroll
      for (int q = 0; q < kPw; ++q) w[q] = s_kept[q] ? __ldcg(rows + (size_t)q * (k + kPw) + kPw + c) : 0.f;
#pragma unroll
      for (int q = 1; q < kPw; ++q)
        if (s_kept[q]) {
#pragma unroll
          for (int i = 0; i < q; ++i)
            if (s_kept[i]) w[q] = __fsub_rn(w[q], __fmul_rn(w[i], s_l[q][i]));
        }
#pragma unroll
      for (int q = 0; q < kPw; ++q) wts[c * kPw + q] = w[q];
    }
    __syncthreads();
    // (a skipped column has zero multipliers and zero weights: its step
    // subtracts zero and changes nothing)
    if (live) {
      float* t = slab + (size_t)pe * ldv + tid;
      int c = 0;
      for (; c + 4 <= nt; c += 4) {
        float y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = t[(size_t)(c + u) * ldv];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 w = reinterpret_cast<const float4*>(wts + (c + u) * kPw)[h];
            y[u] = __fsub_rn(y[u], __fmul_rn(w.x, x[4 * h]));
            y[u] = __fsub_rn(y[u], __fmul_rn(w.y, x[4 * h + 1]));
            y[u] = __fsub_rn(y[u], __fmul_rn(w.z, x[4 * h + 2]));
            y[u] = __fsub_rn(y[u], __fmul_rn(w.w, x[4 * h + 3]));
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) t[(size_t)(c + u) * ldv] = y[u];
      }
      for (; c < nt; ++c) {
        float y = t[(size_t)c * ldv];
#pragma unroll
        for (int q = 0; q < kPw; ++q) y = __fsub_rn(y, __fmul_rn(wts[c * kPw + q], x[q]));
        t[(size_t)c * ldv] = y;
      }
    }
    // (a row's entries are read next by its own thread, and by the polling
    // warps only after the barrier of the next column)
  }
  if constexpr (CL) cooperative_groups::this_cluster().sync();  // no CTA leaves while its words may be read
  if (failed) return;
  __syncthreads();
  for (int c = warp; c < k; c += nwarps) {
    const float* src = slab + (size_t)c * ldv;
    float* dw = W + r0 + (int64_t)c * ldw;
    TO* dq = Q + r0 + (int64_t)c * ldq;
#pragma unroll 4
    for (int i = lane; i < nr; i += 32) {
      const float v = src[i];
      dw[i] = v;
      if ((void*)Q != (void*)W) dq[i] = from_f32<TO>(v);
    }
  }
}

// Dynamic shared memory a plan may ask for: the 227 KB a CTA can have less 2 KB
// for the static arrays of the cooperative kernels (1040 bytes, -Xptxas -v).  The
// cluster form holds 2560 bytes more of them: 228848 bytes.
constexpr int64_t kHessSmem = 225 * 1024;
constexpr int64_t kHessClusterSmem = kHessSmem + 1008 - 2560;

// ... of k resident columns: slab, thresholds, trailing weights
static size_t hess_res_smem(int64_t rpc, int64_t k) {
  return (size_t)(rpc | 1) * 4 * k + 4 * (size_t)k + 32 + (k > kPw ? (size_t)(k - kPw) * kPw * 4 : 0);
}

// rows per CTA, CTAs and the columns that fit in shared memory
struct HessPlan {
  int G, rpc, kr;
};
static HessPlan hess_plan(int64_t n, int64_t k) {
  HessPlan p;
  // about 256 rows per CTA (fewer CTAs poll fewer words: 16384 x 128 takes
  // 0.65 ms with 128 rows, 0.50 ms with 256, 0.55 ms with 400), more CTAs where all k columns then fit
  int64_t G = (n + 255) / 256;
  const int64_t fit = (int64_t)((kHessSmem - 32 - 36 * k) / (4 * k)) - 1;
  if (fit >= 1 && (n + G - 1) / G > fit) G = (n + fit - 1) / fit;
  // one CTA more where the block then fits one cluster (the exchange through
  // distributed shared memory: 1024 x 216 takes 0.59 ms on 4 CTAs of the
  // cooperative grid, 1024 x 200 0.46 in one cluster)
  int64_t gc = G;
  while (gc <= kHessMaxCluster && hess_res_smem((n + gc - 1) / gc, k) > (size_t)kHessClusterSmem) ++gc;
  if (gc <= kHessMaxCluster) G = gc;
  if (G > num_sms()) G = num_sms();
  if (G > 32 * kMaxPoll) G = 32 * kMaxPoll;
  if (G < 1) G = 1;
  p.rpc = (int)((n + G - 1) / G);
  p.G = (int)((n + p.rpc - 1) / p.rpc);
  // a column: its rows, its threshold, its trailing weights
  const size_t per = (size_t)(p.rpc | 1) * 4 + 4 + kPw * 4;
  p.kr = (int)std::min<int64_t>(k, (int64_t)((kHessSmem - 32) / per));
  // the weights are needed only beyond one panel
  if (p.kr < kPw && p.kr < k) p.kr = (int)std::min<int64_t>(std::min<int64_t>(k, kPw), (int64_t)((kHessSmem - 32) / ((size_t)(p.rpc | 1) * 4 + 4)));
  return p;
}
static size_t hess_res_bytes(int64_t k) {
  return align_up(2 * (size_t)num_sms() * 64) + align_up(2 * kPw * sizeof(int)) + align_up((size_t)k * 4) +
         align_up(2 * (size_t)kPw * (k + kPw) * 4);
}

// One launch of the resident kernel on k columns.  mem: hess_res_bytes, its
// words, flags and maxima zeroed by hess_res_reset once per process (tag0
// tells the launches of one process apart).
static rr_status hess_res_reset(void* mem, int64_t k, cudaStream_t s) {
  RR_CUDA(cudaMemsetAsync(mem, 0, align_up(2 * (size_t)num_sms() * 64) + align_up(2 * kPw * sizeof(int)) + align_up((size_t)k * 4), s));
  return RR_OK;
}
template <typename TO>
static rr_status hess_res_launch(int64_t n, int64_t k, float* W, int64_t ldw, TO* Q, int64_t ldq, int* piv, float tol,
                                 const HessPlan& p, void* ws, void* mem, int64_t kmem, int tag0,
                                 const float* colmax_ext, cudaStream_t s) {
  const size_t smem = hess_res_smem(p.rpc, k);
  const bool byrow = p.rpc <= kRowThreads;
  int rt = byrow ? (p.rpc + 31) / 32 * 32 : kRowThreads;
  const unsigned threads = rt + 32 * ((p.G + 31) / 32);
  // one cluster where the CTAs fit one (checked against the GPU's cluster
  // occupancy): the words go through distributed shared memory, and the
  // cluster's own co-scheduling stands in for a cooperative launch (the two
  // attributes together are not kept by every tool that replays a launch, and
  // without its cluster the kernel would address memory that is not there: it
  // checks).  A slab that leaves no room for the cluster form's larger static
  // arrays (216 and more columns that fill their CTAs) runs on the cooperative
  // grid.
  const void* fn = (const void*)k_hess_row<TO, true>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.G);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = p.G;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at + 1;
  cfg.numAttrs = 1;
  bool cl = false;
  if (byrow && p.G <= kHessMaxCluster) {
    bool fits = false;
    RR_TRY(allow_dynamic_smem(fn, smem, &fits));
    if (fits) {
      int nc = 0;
      cl = (p.G <= 8 || cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
           cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) == cudaSuccess && nc >= 1;
      if (!cl) (void)cudaGetLastError();
    }
  }
  if (!cl) {
    fn = byrow ? (const void*)k_hess_row<TO, false> : (const void*)k_hess_res<TO>;
    cfg.attrs = at;
    RR_TRY(allow_dynamic_smem(fn, smem));
  }
  Arena ar(mem, hess_res_bytes(kmem));
  HessRes h;
  h.err = (int*)ws;
  h.bar = (GridBarrier*)((char*)ws + align_up(sizeof(int)));
  h.msg = (uint4*)ar.take_bytes(2 * (size_t)num_sms() * 64);
  h.flags = (int*)ar.take_bytes(2 * kPw * sizeof(int));
  h.colmax = (unsigned*)ar.take_bytes((size_t)kmem * 4);
  h.rowbuf = (float*)ar.take_bytes(2 * (size_t)kPw * (kmem + kPw) * 4);
  h.colmax_ext = colmax_ext;
  h.tag0 = tag0;
  h.rpc = p.rpc;
  int kk = (int)k;
  void* args[] = {&n, &kk, &W, &ldw, &Q, &ldq, &piv, &tol, &h, &rt};  // (the last for k_hess_row)
  RR_CUDA(cudaLaunchKernelExC(&cfg, fn, args));
  note_launches(1);
  return RR_OK;
}

// ---------------------------------------------------------------------------
// Blocked (level-3) Hessenberg process for blocks too tall for the slab
// kernel's shared memory (the panel form of Algorithm 8 that Table 1's "Block"
// row and the closing future-work passage point to).  Columns go in panels of
// r: the panel is factored by the right-looking kernel above on its r columns
// only (thresholds from the column norms on entry to the whole process), then
// the trailing columns T take the whole panel at once:
//   weights  w_j(c) = T(pi_j, c) - sum_{i < j} L(pi_j, i) w_i(c)   (forward
//            substitution with the panel's unit lower triangle at its pivot rows)
//   update   T(:, c) <- T(:, c) - sum_j L(:, j) w_j(c)
// Every entry sees the same operations in the same order as in the
// right-looking process (the weights are exactly the pivot-row entries it
// would read; each step a separately rounded multiply and subtract, j
// ascending), so the blocked result equals it bit for bit, while the trailing
// columns are streamed once per panel instead of once per column.
// ---------------------------------------------------------------------------
// colmax[c] = max_i |W(i, c)| (non-negative floats order like their bits):
// CTA (c, chunk) reduces 64K rows and merges with an atomic max
__global__ void k_hess_colmax(int64_t n, int k, const float* __restrict__ W, int64_t ldw,
                              unsigned* __restrict__ colmax_bits) {
  const int c = blockIdx.x;
  const int64_t i0 = (int64_t)blockIdx.y * 65536, i1 = i0 + 65536 < n ? i0 + 65536 : n;
  float m = 0.f;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) m = fmaxf(m, fabsf(W[i + c * ldw]));
  m = warp_max(m);
  __shared__ float red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
    atomicMax(colmax_bits + c, __float_as_uint(m));
  }
}

// weights of the panel (r columns at L, pivots piv[0..r)) for the nt trailing
// columns T: w[j * nt + c]; a skipped panel column (pivot -1) has weight 0
// and takes no part in the substitution.  One thread per trailing column; the
// panel's triangle at its pivot rows is staged in shared memory first.
__global__ void __launch_bounds__(128) k_hess_weights(int r, int nt, const float* __restrict__ L,
                                                      const float* __restrict__ T, int64_t ldw,
                                                      const int* __restrict__ piv, float* __restrict__ w) {
  __shared__ float ls[kPanelMax][kPanelMax + 1];
  __shared__ int sp[kPanelMax];
  if (threadIdx.x < kPanelMax) sp[threadIdx.x] = (int)threadIdx.x < r ? piv[threadIdx.x] : -1;
  __syncthreads();
  for (int e = threadIdx.x; e < r * r; e += 128) {
    const int j = e / r, i = e % r;
    ls[j][i] = sp[j] >= 0 && i < j ? L[sp[j] + (int64_t)i * ldw] : 0.f;
  }
  __syncthreads();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nt) return;
  float wr[kPanelMax];
#pragma unroll
  for (int j = 0; j < kPanelMax; ++j) wr[j] = sp[j] >= 0 ? T[sp[j] + (int64_t)c * ldw] : 0.f;
#pragma unroll
  for (int j = 0; j < kPanelMax; ++j) {
    if (sp[j] >= 0) {
#pragma unroll
      for (int i = 0; i < j; ++i)
        if (sp[i] >= 0) wr[j] = __fsub_rn(wr[j], __fmul_rn(wr[i], ls[j][i]));
    }
    if (j < r) w[(size_t)j * nt + c] = wr[j];
  }
}

// T(i, c) <- T(i, c) - sum_j L(i, j) w_j(c), j ascending, every row i.  A
// thread takes two rows (packed FP32 pairs: each component is a separately
// rounded multiply and add of the negated product, the same bits as multiply
// and subtract) with their R panel entries in registers and 4 columns' loads in
// flight; the negated weights come from shared memory four at a time (a
// broadcast 16-byte load takes as long as 8 packed operations).  A skipped
// panel column has zero entries and zero weights.  1048576 rows: R = 8 at the
// HBM rate (24 columns 36 us); R = 32 is bound by the FP32 pipe
// (128 columns: 0.45 ms against 0.58 ms with the weights stored in pairs).
// (the products as FMAs with a minus zero that the compiler cannot see: a
// packed multiply next to a packed add would be fused into one rounding)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
      "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
template <int R, bool kVec>
__global__ void __launch_bounds__(256) k_hess_trail(int64_t n, int r, int nt, const float* __restrict__ L,
                                                    float* __restrict__ T, int64_t ldw, const float* __restrict__ w,
                                                    int wld, float minus_zero) {
  const float2 mz = make_float2(minus_zero, minus_zero);
  extern __shared__ __align__(16) float sw[];  // [nt][R] -w
  for (int e = threadIdx.x; e < R * nt; e += blockDim.x) {
    const int c = e / R, j = e % R;
    sw[e] = -(j < r ? w[j * (size_t)wld + c] : 0.f);  // (padding: -0 times its zero entries, x + -0 = x)
  }
  __syncthreads();
  auto ld = [&](const float* p, bool two) -> float2 {
    if (kVec && two) return *reinterpret_cast<const float2*>(p);
    return make_float2(p[0], two ? p[1] : 0.f);
  };
  auto st = [&](float* p, bool two, float2 v) {
    if (kVec && two) {
      *reinterpret_cast<float2*>(p) = v;
    } else {
      p[0] = v.x;
      if (two) p[1] = v.y;
    }
  };
  for (int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); i < n;
       i += 2 * (int64_t)gridDim.x * blockDim.x) {
    const bool two = i + 1 < n;
    float2 l[R];
#pragma unroll
    for (int j = 0; j < R; ++j) l[j] = j < r ? ld(L + i + (int64_t)j * ldw, two) : make_float2(0.f, 0.f);
    int c = 0;
    for (; c + 4 <= nt; c += 4) {
      float2 t[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u] = ld(T + i + (int64_t)(c + u) * ldw, two);
#pragma unroll
      for (int j = 0; j < R; j += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 wv = *reinterpret_cast<const float4*>(sw + (c + u) * R + j);
          t[u] = add2(t[u], fma2(make_float2(wv.x, wv.x), l[j], mz));
          t[u] = add2(t[u], fma2(make_float2(wv.y, wv.y), l[j + 1], mz));
          t[u] = add2(t[u], fma2(make_float2(wv.z, wv.z), l[j + 2], mz));
          t[u] = add2(t[u], fma2(make_float2(wv.w, wv.w), l[j + 3], mz));
        }
#pragma unroll
      for (int u = 0; u < 4; ++u) st(T + i + (int64_t)(c + u) * ldw, two, t[u]);
    }
    for (; c < nt; ++c) {
      float2 t = ld(T + i + (int64_t)c * ldw, two);
#pragma unroll
      for (int j = 0; j < R; ++j) t = add2(t, fma2(make_float2(sw[c * R + j], sw[c * R + j]), l[j], mz));
      st(T + i + (int64_t)c * ldw, two, t);
    }
  }
}

// the trailing update of nt columns T by the panel of r <= kPanelMax columns at L
static rr_status hess_trail(int64_t n, int r, int nt, const float* L, float* T, int64_t ldw, const int* piv,
                            float* wts, cudaStream_t s) {
  if (nt <= 0) return RR_OK;
  k_hess_weights<<<(unsigned)((nt + 127) / 128), 128, 0, s>>>(r, nt, L, T, ldw, piv, wts);
  RR_TRY(check_launch("hessenberg panel weights"));
  const bool vec = ldw % 2 == 0 && (uintptr_t)L % 8 == 0 && (uintptr_t)T % 8 == 0;
  const int R = r <= 8 ? 8 : r <= 16 ? 16 : 32;
  // trailing columns in chunks whose weights fit 96 KB of shared memory
  const int ncmax = (int)((96 * 1024) / ((size_t)R * sizeof(float)));
  const unsigned g = (unsigned)std::min<int64_t>((n + 511) / 512, 8 * (int64_t)num_sms());
  for (int c0 = 0; c0 < nt; c0 += ncmax) {
    const int nc = std::min(nt - c0, ncmax);
    const size_t sm = (size_t)R * nc * sizeof(float);
    auto go = [&](auto fn) -> rr_status {
      RR_TRY(allow_dynamic_smem((const void*)fn, sm));
      fn<<<g, 256, sm, s>>>(n, r, nc, L, T + (int64_t)c0 * ldw, ldw, wts + c0, nt, -0.0f);
      return check_launch("hessenberg trailing update");
    };
    if (R == 8) RR_TRY(vec ? go(k_hess_trail<8, true>) : go(k_hess_trail<8, false>));
    else if (R == 16) RR_TRY(vec ? go(k_hess_trail<16, true>) : go(k_hess_trail<16, false>));
    else RR_TRY(vec ? go(k_hess_trail<32, true>) : go(k_hess_trail<32, false>));
  }
  return RR_OK;
}

// The extra workspace of the blocked process, after the kernel's own part:
// column maxima (k) and panel weights (kPanelMax x k).
static size_t hess_blocked_extra(int64_t k) {
  return align_up((size_t)k * sizeof(float)) + align_up((size_t)kPanelMax * k * sizeof(float)) + hess_res_bytes(k);
}

template <typename TO>
static rr_status hess_blocked(int64_t n, int64_t k, float* W, int64_t ldw, TO* Q, int64_t ldq, int* piv,
                              double tol, int r, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (r < 1 || r > kPanelMax) return RR_ERR_ARG;
  const size_t base = hess_ws_bytes<float>(k, num_sms());
  if (!ws || ws_bytes < base + hess_blocked_extra(k)) return RR_ERR_WORKSPACE;
  float* colmax = (float*)((char*)ws + base);
  float* wts = (float*)((char*)ws + base + align_up((size_t)k * sizeof(float)));
  RR_CUDA(cudaMemsetAsync(colmax, 0, (size_t)k * sizeof(float), s));
  k_hess_colmax<<<dim3((unsigned)k, (unsigned)((n + 65535) / 65536)), 256, 0, s>>>(n, (int)k, W, ldw,
                                                                                 (unsigned*)colmax);
  RR_TRY(check_launch("hessenberg colmax"));
  // the default tolerance scales with the whole block's width, as the
  // unblocked process's does
  const double t = tol > 0 ? tol : 4.0 * (double)k * 0x1p-23;
  // panels that fit the CTAs' shared memory: the resident kernel, several to a
  // panel where need be; else the right-looking kernel on W in memory
  void* mem = (char*)wts + align_up((size_t)kPanelMax * k * sizeof(float));
  const HessPlan p = hess_plan(n, r);
  const int inner = p.kr >= r ? r : p.kr;
  if (inner > 0) {
    RR_CUDA(cudaMemsetAsync(ws, 0, 512, s));  // err + barrier
    RR_TRY(hess_res_reset(mem, k, s));
  }
  for (int64_t c0 = 0; c0 < k; c0 += r) {
    const int64_t c1 = c0 + r < k ? c0 + r : k;
    const int pr = (int)(c1 - c0);
    if (inner > 0) {
      for (int64_t i0 = c0; i0 < c1; i0 += inner) {
        const int64_t i1 = i0 + inner < c1 ? i0 + inner : c1;
        RR_TRY(hess_res_launch<TO>(n, i1 - i0, W + i0 * ldw, ldw, Q + i0 * ldq, ldq, piv + i0, (float)t, p, ws, mem, k,
                                   (int)i0, colmax + i0, s));
        RR_TRY(hess_trail(n, (int)(i1 - i0), (int)(c1 - i1), W + i0 * ldw, W + i1 * ldw, ldw, piv + i0, wts, s));
      }
    } else {
      const rr_status st = hess_launch<float, TO>(n, pr, W + c0 * ldw, ldw, Q + c0 * ldq, ldq, piv + c0, t, ws, base,
                                                  s, 0, colmax + c0, c0 == 0);
      if (st != RR_OK) return st;
    }
    RR_TRY(hess_trail(n, pr, (int)(k - c1), W + c0 * ldw, W + c1 * ldw, ldw, piv + c0, wts, s));
  }
  return RR_OK;
}

// The FP32 process of a whole block: resident where it fits the CTAs' shared
// memory, blocked where it does not (panels of 32 with as many resident columns
// as fit; panels of 16 on W in memory past 8.7 million rows, where not even one
// column is resident: 10M x 96 took 380 ms as one right-looking panel), and the
// right-looking kernel for a single CTA (the batched solver's concurrent
// problems), for rows beyond its candidate word and for one such panel.
template <typename TO>
static rr_status hess_f32(int64_t n, int64_t k, float* W, int64_t ldw, TO* Q, int64_t ldq, int* piv, double tol,
                          void* ws, size_t ws_bytes, cudaStream_t s, int max_grid) {
  const HessPlan p = hess_plan(n, k);
  if (max_grid == 1 || n >= (int64_t)kNoRow || (p.kr < 1 && k <= 16))
    return hess_launch<float, TO>(n, k, W, ldw, Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
  if (p.kr < k) return hess_blocked<TO>(n, k, W, ldw, Q, ldq, piv, tol, p.kr < 1 ? 16 : kPanelMax, ws, ws_bytes, s);
  const size_t base = hess_ws_bytes<float>(k, num_sms());
  if (!ws || ws_bytes < base + hess_blocked_extra(k)) return RR_ERR_WORKSPACE;
  RR_CUDA(cudaMemsetAsync(ws, 0, 512, s));  // err + barrier
  void* mem = (char*)ws + base;
  RR_TRY(hess_res_reset(mem, k, s));
  const float t = (float)(tol > 0 ? tol : 4.0 * (double)k * 0x1p-23);
  return hess_res_launch<TO>(n, k, W, ldw, Q, ldq, piv, t, p, ws, mem, k, 0, nullptr, s);
}

}  // namespace rr

using namespace rr;

extern "C" size_t rr_hessenberg_workspace_size(int64_t n, int64_t k, int32_t arith) {
  int G = num_sms();
  return arith == RR_F64 ? hess_ws_bytes<double>(k, G) : hess_ws_bytes<float>(k, G) + hess_blocked_extra(k);
}

namespace rr {
rr_status hessenberg_ex(int32_t arith, int64_t n, int64_t k, void* W, int64_t ldw, int32_t qtype,
                        void* Q, int64_t ldq, int32_t* piv, double tol, void* ws, size_t ws_bytes,
                        cudaStream_t s, int max_grid);

// A block without rows: every column is skipped (and no plan is made: it would
// divide by the rows of a CTA).
static rr_status hess_no_rows(int64_t k, int32_t* piv, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!ws || ws_bytes < sizeof(int)) return RR_ERR_WORKSPACE;
  RR_CUDA(cudaMemsetAsync(ws, 0, sizeof(int), s));  // the error word
  RR_CUDA(cudaMemsetAsync(piv, 0xff, (size_t)k * sizeof(int32_t), s));
  return RR_OK;
}
}
extern "C" rr_status rr_hessenberg(int32_t arith, int64_t n, int64_t k, void* W, int64_t ldw,
                                   int32_t qtype, void* Q, int64_t ldq, int32_t* piv, double tol,
                                   void* ws, size_t ws_bytes, void* stream) {
  return hessenberg_ex(arith, n, k, W, ldw, qtype, Q, ldq, piv, tol, ws, ws_bytes,
                       as_stream(stream), 0);
}

rr_status rr::hessenberg_ex(int32_t arith, int64_t n, int64_t k, void* W, int64_t ldw,
                            int32_t qtype, void* Q, int64_t ldq, int32_t* piv, double tol,
                            void* ws, size_t ws_bytes, cudaStream_t s, int max_grid) {
  if (n < 0 || k < 0 || k > 4096 || ldw < n || ldq < n || !W || !Q || !piv) return RR_ERR_ARG;
  if (n > INT_MAX) return RR_ERR_ARG;
  if (k == 0) return RR_OK;
  auto known = [](int32_t t, bool f8) { return t == RR_F64 || t == RR_F32 || t == RR_BF16 || (f8 && t == RR_E4M3); };
  if (n == 0 && (arith == RR_F32 || arith == RR_F64) && known(qtype, arith == RR_F32))
    return hess_no_rows(k, piv, ws, ws_bytes, s);
  if (arith == RR_F32) {
    float* w = (float*)W;
    switch (qtype) {
      case RR_F32: return hess_f32<float>(n, k, w, ldw, (float*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
      case RR_BF16: return hess_f32<__nv_bfloat16>(n, k, w, ldw, (__nv_bfloat16*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
      case RR_E4M3: return hess_f32<e4m3b_t>(n, k, w, ldw, (e4m3b_t*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
      case RR_F64: return hess_f32<double>(n, k, w, ldw, (double*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
    }
  } else if (arith == RR_F64) {
    double* w = (double*)W;
    switch (qtype) {
      case RR_F64: return hess_launch<double, double>(n, k, w, ldw, (double*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
      case RR_F32: return hess_launch<double, float>(n, k, w, ldw, (float*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
      case RR_BF16: return hess_launch<double, __nv_bfloat16>(n, k, w, ldw, (__nv_bfloat16*)Q, ldq, piv, tol, ws, ws_bytes, s, max_grid);
    }
  }
  return RR_ERR_ARG;
}

extern "C" rr_status rr_hessenberg_blocked(int64_t n, int64_t k, float* W, int64_t ldw, int32_t qtype, void* Q,
                                           int64_t ldq, int32_t* piv, double tol, int32_t panel, void* ws,
                                           size_t ws_bytes, void* stream) {
  if (n < 0 || k < 0 || k > 4096 || ldw < n || ldq < n || !W || !Q || !piv) return RR_ERR_ARG;
  if (n >= (int64_t)kNoRow || panel < 1 || panel > kPanelMax) return RR_ERR_ARG;
  if (k == 0) return RR_OK;
  cudaStream_t s = as_stream(stream);
  if (n == 0 && (qtype == RR_F32 || qtype == RR_BF16 || qtype == RR_F64)) return hess_no_rows(k, piv, ws, ws_bytes, s);
  switch (qtype) {
    case RR_F32: return hess_blocked<float>(n, k, W, ldw, (float*)Q, ldq, piv, tol, panel, ws, ws_bytes, s);
    case RR_BF16: return hess_blocked<__nv_bfloat16>(n, k, W, ldw, (__nv_bfloat16*)Q, ldq, piv, tol, panel, ws, ws_bytes, s);
    case RR_F64: return hess_blocked<double>(n, k, W, ldw, (double*)Q, ldq, piv, tol, panel, ws, ws_bytes, s);
  }
  return RR_ERR_ARG;
}
