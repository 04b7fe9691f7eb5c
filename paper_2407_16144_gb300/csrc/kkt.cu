// Standalone evaluation of the relative KKT error of a point (x, y) of an LP held in device
// memory: the termination measure of the solver (Section 7, "Termination criteria"; the l2 form
// described in include/rhpdhg.h), available to callers who want to check any point.
//
//   rel_p   = || (b - A x, (h - G x)^+) ||_2 / (1 + ||q||_2)
//   rel_d   = || c - K^T y - lambda ||_2 / (1 + ||c||_2),  lambda = proj_Lambda(c - K^T y)
//   rel_gap = |p - d| / (1 + |p| + |d|),  p = c^T x + off,  d = q^T y + sum(l lambda^+ - u lambda^-) + off
//
// K^T y is formed by scattering each row's contribution (atomic FP64 adds) into an n-vector of
// scratch, so only the CSR of K is needed; the sums are then reduced per block into scratch
// partials and finished by one block.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "../../include/rhpdhg.h"
#include "bufcache.h"
#include "internal.h"

namespace rh {

namespace {

constexpr int kKktThreads = 256;
constexpr int kKktSlots = kKktSlotCount;   // stride of a block's partials
constexpr int kKktUsed = 7;                // 0 rp2, 1 qy, 2 qq, 3 rd2, 4 cx, 5 bnd, 6 cc
constexpr int kKktRowSlots = 3;            // the first three come from the row kernel
constexpr int kKktFlag = 5;                // dout[5]: 1 if the CSR held an index out of range
constexpr int kKktStage = 704;             // entries a warp stages at a time (22 per row of 32): a
                                           // multiple of 4
constexpr int kKktRowCtas = 4;             // resident CTAs per SM of the row kernel: 45 KB each, and 64
                                           // registers a thread, under which it spills (76 bytes of
                                           // stores, 52 of loads); fewer CTAs were not measured

__device__ __forceinline__ double block_sum(double v, double *sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kKktThreads / 32; ++w) r += sh[w];
  return r;   // valid in thread 0
}

// One warp takes 32 consecutive rows: their entries are read as one contiguous segment, kKktStage at
// a time, a lane on four consecutive entries (one thread per row read 12 bytes here and 12 bytes
// 200 bytes further on).  The lane finds its first entry's row among the 32 row ends by a search in
// shuffles and follows the ends through the bits of row_ends; it scatters val * y_row and adds
// val * x_j up within its four entries and the row, as stage_segment does, so that a row's sum is
// left with a quarter of its additions.  Bound by the FP64 pipe (a multiplication and a fused
// multiply-add per entry) and the scattered FP64 additions in L2.  The evaluation of a 30M-entry
// LP took 950 us with a thread per row, a cudaMalloc and cudaFree per call and floating-point
// comparisons in the column kernel, 464 us with runs of entries balanced over the lanes, and takes
// 407 us.
//
// Rows whose offsets fall outside [0, nnz] or decrease, and entries whose column lies outside
// [0, n), are skipped and reported through flag (the caller's CSR is not validated beforehand);
// 32 rows with such an offset among them are walked one thread per row.
__global__ void __launch_bounds__(kKktThreads, kKktRowCtas)
k_kkt_rows(int m, int m_eq, int n, long long nnz, const long long *__restrict__ rp,
           const int *__restrict__ col, const double *__restrict__ val,
           const double *__restrict__ x, const double *__restrict__ y,
           const double *__restrict__ q, double *kty, double *part, double *flag) {
  __shared__ double sh[kKktThreads / 32];
  __shared__ double staged[kKktThreads / 32][kKktStage];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double *st = staged[threadIdx.x >> 5];
  double s_rp2 = 0.0, s_qy = 0.0, s_qq = 0.0;
  const long long nwarps = (long long)gridDim.x * (kKktThreads / 32);
  for (long long t = blockIdx.x * (kKktThreads / 32) + (threadIdx.x >> 5); t * 32 < m;
       t += nwarps) {
    const long long i = t * 32 + lane;
    const bool in = i < m;
    const long long p0 = rp[in ? i : m], p1 = rp[in ? i + 1 : m];
    const double yi = in ? y[i] : 0.0, qi = in ? q[i] : 0.0;
    double kx = 0.0;
    const bool bad = p0 < 0 || p1 < p0 || p1 > nnz;
    if (__any_sync(full, bad)) {
      if (bad && in) *flag = 1.0;
      for (long long p = p0; in && !bad && p < p1; ++p) {
        const int j = col[p];
        if (j < 0 || j >= n) {
          *flag = 1.0;
          continue;
        }
        kx += val[p] * x[j];
        atomicAdd(kty + j, val[p] * yi);
      }
    } else {
      const long long seg_e = __shfl_sync(full, p1, 31);
      for (long long base = __shfl_sync(full, p0, 0); base < seg_e; base += kKktStage) {
        const int len = (int)min((long long)kKktStage, seg_e - base);
        const int lo = (int)min(max(p0 - base, 0ll), (long long)len);
        const int hi = (int)min(max(p1 - base, 0ll), (long long)len);
        unsigned *ends = row_ends_clear();
        row_end(ends, 0, lo, hi);
        const unsigned some = __ballot_sync(full, hi > lo);
        __syncwarp();
        for (int o = 4 * lane; o - 4 * lane < len; o += 32 * 4) {
          int j[4];
          double v[4], xj[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            j[u] = o + u < len ? col[base + o + u] : 0;
            v[u] = o + u < len ? val[base + o + u] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const bool ok = j[u] >= 0 && j[u] < n;
            if (!ok) *flag = 1.0;
            xj[u] = ok && o + u < len ? x[j[u]] : 0.0;
            if (!ok) v[u] = 0.0;
          }
          int r = 0;                         // rows that end at or before entry o
#pragma unroll
          for (int h = 16; h > 0; h >>= 1)
            if (__shfl_sync(full, hi, r + h - 1) <= o) r += h;
          const unsigned end = o < len ? ends[o >> 5] >> (o & 31) : 0u;
          double acc = 0.0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const double yr = __shfl_sync(full, yi, r);
            if (o + u < len && j[u] >= 0 && j[u] < n) atomicAdd(kty + j[u], v[u] * yr);
            acc = fma(v[u], xj[u], acc);
            if ((end >> u) & 1u) {
              st[o + u] = acc;
              acc = 0.0;
              const unsigned rest = some & ~((2u << r) - 1u);    // the next row that is not empty
              r = rest ? __ffs((int)rest) - 1 : r;
            } else if (u == 3 && o < len) {
              st[o + 3] = acc;
            }
            __syncwarp();
          }
        }
        __syncwarp();
        if (lo < hi) {
          int q = lo | 3;                    // the last entry of the row's first four
          kx += st[min(q, hi - 1)];
          while (q < hi - 1) {
            q += 4;
            kx += st[min(q, hi - 1)];
          }
        }
        __syncwarp();
      }
    }
    if (in) {
      double r = qi - kx;
      if (i >= m_eq) r = fmax(r, 0.0);
      s_rp2 += r * r;
      s_qy += qi * yi;
      s_qq += qi * qi;
    }
  }
  const double a = block_sum(s_rp2, sh), b = block_sum(s_qy, sh), c = block_sum(s_qq, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x * kKktSlots + 0] = a;
    part[blockIdx.x * kKktSlots + 1] = b;
    part[blockIdx.x * kKktSlots + 2] = c;
  }
}

__global__ void __launch_bounds__(kKktThreads)
k_kkt_cols(int n, const double *c, const double *l, const double *u, const double *x,
           const double *kty, double *part) {
  __shared__ double sh[kKktThreads / 32];
  double s_rd2 = 0.0, s_cx = 0.0, s_bnd = 0.0, s_cc = 0.0;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    const double cj = c[j], lj = l[j], uj = u[j];
    const double g = cj - kty[j];
    // The FP64 pipe bounds this kernel: six FP64 instructions per column are left, with the
    // comparisons on the integer pipe (10M columns: 291 us with floating-point comparisons, 80% of
    // the pipe, about 130 us without).
    const bool lf = dbl_finite(lj), uf = dbl_finite(uj);
    double lam = 0.0;
    if (lf && uf) lam = g;
    else if (lf) lam = dbl_pos(g) ? g : 0.0;
    else if (uf) lam = dbl_neg(g) ? g : 0.0;
    const double rd = g - lam;
    s_rd2 += rd * rd;
    s_cx += cj * x[j];
    const bool pos = dbl_pos(lam), neg = dbl_neg(lam);
    s_bnd += (pos ? lj : neg ? uj : 0.0) * (pos || neg ? lam : 0.0);
    s_cc += cj * cj;
  }
  const double a = block_sum(s_rd2, sh), b = block_sum(s_cx, sh), d = block_sum(s_bnd, sh),
               e = block_sum(s_cc, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x * kKktSlots + 3] = a;
    part[blockIdx.x * kKktSlots + 4] = b;
    part[blockIdx.x * kKktSlots + 5] = d;
    part[blockIdx.x * kKktSlots + 6] = e;
  }
}

// One warp per used slot: lane l adds blocks l, l + 32, ... in order, then a fixed shuffle tree (one
// thread per slot spent about 1000 dependent FP64 additions on a full grid).
__global__ void __launch_bounds__(32 * kKktUsed)
k_kkt_final(int nb_rows, int nb_cols, const double *part, double off, double *out) {
  __shared__ double tot[kKktUsed];
  const int slot = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nb = slot < kKktRowSlots ? nb_rows : nb_cols;
  double s = 0.0;
#pragma unroll 8
  for (int b = lane; b < nb; b += 32) s += part[b * kKktSlots + slot];
  s = warp_sum(s);
  if (lane == 0) tot[slot] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    const double rel_p = sqrt(tot[0]) / (1.0 + sqrt(tot[2]));
    const double rel_d = sqrt(tot[3]) / (1.0 + sqrt(tot[6]));
    const double p = tot[4] + off, d = tot[1] + tot[5] + off;
    out[0] = rel_p;
    out[1] = rel_d;
    out[2] = fabs(p - d) / (1.0 + fabs(p) + fabs(d));
    out[3] = p;
    out[4] = d;
  }
}

__global__ void k_kkt_zero(int n, double *v, double *flag) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    v[i] = 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) *flag = 0.0;
}


}  // namespace

int kkt_blocks(int rows) {
  const int need = (rows + kKktThreads - 1) / kKktThreads;
  return need < 1 ? 1 : (need > kKktMaxBlocks ? kKktMaxBlocks : need);
}

// Runs the evaluation with caller-provided scratch: kty (n doubles), part (kKktMaxBlocks *
// kKktSlots doubles) and dout (8 doubles), all device memory; copies the 5 results to out (host).
// *bad_index is set when the CSR held a row offset or column index out of range.
cudaError_t kkt_eval_with_scratch(const rhpdhg_problem *lp, const double *x, const double *y,
                                  cudaStream_t st, double *kty, double *part, double *dout,
                                  double *out, bool *bad_index) {
  const int m = lp->m_eq + lp->m_ineq, n = lp->n;
  const int nbc = kkt_blocks(n);
  // the row kernel's grid is at most the CTAs resident at once: its tiles go round robin, and a
  // second, partly filled wave would leave SMs idle
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int nbr = std::min(kkt_blocks(m), std::max(1, sms * kKktRowCtas));
  double *flag = dout + kKktFlag;
  e = launch_kernel(k_kkt_zero, nbc, kKktThreads, 0, st, n, kty, flag);
  if (e == cudaSuccess)
    e = launch_kernel(k_kkt_rows, nbr, kKktThreads, 0, st, m, lp->m_eq, n, (long long)lp->nnz,
               (const long long *)lp->row_ptr, lp->col_idx, lp->val, x, y, lp->rhs, kty, part,
               flag);
  if (e == cudaSuccess)
    e = launch_kernel(k_kkt_cols, nbc, kKktThreads, 0, st, n, lp->c, lp->l, lp->u, x, (const double *)kty,
               part);
  if (e == cudaSuccess)
    e = launch_kernel(k_kkt_final, 1, 32 * kKktUsed, 0, st, nbr, nbc, (const double *)part, lp->obj_offset, dout);
  if (e != cudaSuccess) return e;
  count_launches(4);
  double h[6] = {0};
  e = cudaMemcpyAsync(h, dout, 6 * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  for (int i = 0; i < 5; ++i) out[i] = h[i];
  *bad_index = h[kKktFlag] != 0.0;
  return cudaSuccess;
}

// Host checks shared by both entry points; returns an empty string when the arguments are usable.
std::string kkt_arg_error(const rhpdhg_problem *lp, const double *x, const double *y,
                          const double *out) {
  if (!lp || !x || !out) return "lp, x or out is NULL";
  if (lp->memory != RHPDHG_MEM_DEVICE) return "the problem's arrays must be in device memory";
  if (lp->n < 1 || lp->m_eq < 0 || lp->m_ineq < 0 || lp->nnz < 0)
    return "negative size or n < 1";
  if ((long long)lp->m_eq + lp->m_ineq > 2147483646LL) return "m exceeds the 32-bit range";
  const bool rows = lp->m_eq + lp->m_ineq > 0;
  if (!lp->row_ptr || !lp->c || !lp->l || !lp->u || (rows && (!y || !lp->rhs)) ||
      (lp->nnz > 0 && (!lp->col_idx || !lp->val)))
    return "missing problem array or point";
  return "";
}

// Result of a finished evaluation as a return code, with the message for rhpdhg_last_error.
int kkt_finish(const char *who, cudaError_t e, bool bad_index) {
  if (e != cudaSuccess) {
    set_global_error(std::string(who) + ": " + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? RHPDHG_ERR_OOM : RHPDHG_ERR_CUDA;
  }
  if (bad_index) {
    set_global_error(std::string(who) +
                     ": a row offset or column index of the CSR is out of range (entries skipped)");
    return RHPDHG_ERR_INVALID_ARG;
  }
  return RHPDHG_OK;
}

}  // namespace rh

extern "C" int rhpdhg_kkt_eval(const rhpdhg_problem *lp, const double *x, const double *y,
                               void *stream, double *out) {
  using namespace rh;
  const std::string bad = kkt_arg_error(lp, x, y, out);
  if (!bad.empty()) {
    set_global_error("rhpdhg_kkt_eval: " + bad);
    return RHPDHG_ERR_INVALID_ARG;
  }
  const int n = lp->n;
  cudaStream_t st = (cudaStream_t)stream;
  double *kty = nullptr, *part = nullptr, *dout = nullptr;
  bool bad_index = false;
  // scratch from the buffer cache (a cudaMalloc and cudaFree of n doubles per call synchronised the
  // device and took longer than the evaluation of a mid-size LP)
  cudaError_t e = buf_alloc((void **)&kty, (size_t)n * sizeof(double));
  if (e == cudaSuccess)
    e = buf_alloc((void **)&part, (size_t)kKktMaxBlocks * kKktSlotCount * sizeof(double));
  if (e == cudaSuccess) e = buf_alloc((void **)&dout, 8 * sizeof(double));
  if (e == cudaSuccess) e = kkt_eval_with_scratch(lp, x, y, st, kty, part, dout, out, &bad_index);
  if (e != cudaSuccess) cudaStreamSynchronize(st);   // nothing in flight uses the scratch
  buf_release(kty);
  buf_release(part);
  buf_release(dout);
  return kkt_finish("rhpdhg_kkt_eval", e, bad_index);
}

// ---------------------------------------------------------------------------------------------
// Allocation-free variant.  Some callers may not call cudaMalloc: code that lives inside a
// framework which owns all device memory through its own pool and forbids raw allocations, code
// in latency-critical loops that must not take the allocator's device-wide synchronisation, and
// services that must keep a fixed device-memory footprint.  For them the same evaluation runs on
// a scratch array fixed at file scope: every GPU that loads this library holds it until the
// process exits.  Its host-side name is only a stand-in for the device symbol, so the device
// address is looked up once per device with cudaGetSymbolAddress and kept.

namespace {

constexpr long long kNoAllocMaxN = 1LL << 20;   // largest n accepted (8 MiB of K^T y scratch)
constexpr long long kNoAllocDoubles =
    kNoAllocMaxN + (long long)rh::kKktMaxBlocks * rh::kKktSlotCount + 8;
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) double g_kkt_noalloc_scratch[kNoAllocDoubles];

std::mutex g_noalloc_mu;
double *g_noalloc_addr[kNoAllocMaxDevices] = {nullptr};

}  // namespace

extern "C" int rhpdhg_kkt_eval_noalloc(const rhpdhg_problem *lp, const double *x,
                                       const double *y, void *stream, double *out) {
  using namespace rh;
  const std::string bad = kkt_arg_error(lp, x, y, out);
  if (!bad.empty()) {
    set_global_error("rhpdhg_kkt_eval_noalloc: " + bad);
    return RHPDHG_ERR_INVALID_ARG;
  }
  if ((long long)lp->n > kNoAllocMaxN) {
    set_global_error("rhpdhg_kkt_eval_noalloc: n = " + std::to_string(lp->n) +
                     " exceeds the fixed scratch of this entry point (n <= " +
                     std::to_string(kNoAllocMaxN) + "); use rhpdhg_kkt_eval");
    return RHPDHG_ERR_INVALID_ARG;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return kkt_finish("rhpdhg_kkt_eval_noalloc: cudaGetDevice", e, false);
  if (dev < 0 || dev >= kNoAllocMaxDevices) {
    set_global_error("rhpdhg_kkt_eval_noalloc: device ordinal out of range");
    return RHPDHG_ERR_INVALID_ARG;
  }
  double *base = nullptr;
  {
    // one-time set-up per device, with that device current
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void *p = nullptr;
      e = cudaGetSymbolAddress(&p, g_kkt_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        set_global_error(std::string("rhpdhg_kkt_eval_noalloc: cudaGetSymbolAddress: ") +
                         cudaGetErrorString(e));
        return RHPDHG_ERR_CUDA;
      }
      g_noalloc_addr[dev] = static_cast<double *>(p);
    }
    base = g_noalloc_addr[dev];
  }
  // kty and the index flag in dout are cleared by the first kernel; the used slots of every
  // launched block's partials are written before the final sum reads them
  double *kty = base;
  double *part = base + kNoAllocMaxN;
  double *dout = part + (long long)kKktMaxBlocks * kKktSlotCount;
  bool bad_index = false;
  e = kkt_eval_with_scratch(lp, x, y, (cudaStream_t)stream, kty, part, dout, out, &bad_index);
  return kkt_finish("rhpdhg_kkt_eval_noalloc", e, bad_index);
}
