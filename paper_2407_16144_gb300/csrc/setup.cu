// Create-time kernels: validation, transpose, diagonal scaling (Ruiz + Pock-Chambolle, the
// "preprocessing" the paper's solver inherits, Section 7), split-CSR layout construction,
// plain products and small vector utilities used by the power iteration.
#include <cub/cub.cuh>

#include <algorithm>
#include <atomic>
#include <climits>
#include <type_traits>
#include <utility>
#include <vector>

#include "bufcache.h"
#include "plan.h"
#include "internal.h"

namespace rh {

namespace {

inline int nblocks(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > (1LL << 30)) b = (1LL << 30);
  return (int)b;
}

// bit 1: row_ptr malformed; 2: column index out of range / not increasing; 4: non-finite value;
// 8: non-finite c or rhs; 16: l > u or NaN bound; 32: l = +inf or u = -inf
__global__ void k_validate_rows(int m, int n, long long nnz, const long long *rp, const int *col,
                                const double *val, const double *q, unsigned int *flags) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && (rp[0] != 0 || rp[m] != nnz)) atomicOr(flags, 1u);
  if (i >= m) return;
  long long b = rp[i], e = rp[i + 1];
  if (!(0 <= b && b <= e && e <= nnz)) { atomicOr(flags, 1u); return; }
  int prev = -1;
  unsigned int f = 0;
  for (long long p = b; p < e; ++p) {
    int j = col[p];
    if (j < 0 || j >= n || j <= prev) f |= 2u;
    prev = j;
    if (!isfinite(val[p])) f |= 4u;
  }
  if (!isfinite(q[i])) f |= 8u;
  if (f) atomicOr(flags, f);
}

__global__ void k_validate_cols(int n, const double *c, const double *l, const double *u,
                                unsigned int *flags) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  unsigned int f = 0;
  if (!isfinite(c[j])) f |= 8u;
  double lj = l[j], uj = u[j];
  if (isnan(lj) || isnan(uj) || lj > uj) f |= 16u;
  if (lj == INFINITY || uj == -INFINITY) f |= 32u;
  if (isfinite(uj)) f |= kHasFiniteUpper;
  if (f) atomicOr(flags, f);
}

__global__ void k_rp_convert(int m, const long long *rp64, int *rp32) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i <= m) rp32[i] = (int)rp64[i];
}

__global__ void k_expand_rows(int m, const int *rp, int *rows_of) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  for (int p = rp[i]; p < rp[i + 1]; ++p) rows_of[p] = i;
}

__global__ void k_iota(int n, int *x) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = i;
}

__global__ void k_count_cols(int nnz, const int *col, int *cnt) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < nnz) atomicAdd(cnt + col[p], 1);
}

__global__ void k_gather_csc(int nnz, const int *perm, const int *rows_of, const double *val,
                             int *ridx, double *cval) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nnz) return;
  int p = perm[s];
  ridx[s] = rows_of[p];
  cval[s] = val[p];
}

// One scaling pass of a CSR side: out_r = rs_r / sqrt(stat_r) (rs_r where the row has no nonzero),
// with stat_r over the row's entries of |v_p| rs_r cs_{idx_p}: OP 0 their maximum, OP 1 their sum, OP
// 2 the sum of their powers alpha.  G consecutive lanes share a row (strided over its entries, then a
// fixed shuffle tree); the rows of a CTA with more than kStatLong entries per lane are then taken by
// the whole CTA, one after the other (a power-law column of 5000 entries kept 16 lanes busy
// for 125 us).
//
// Bound by the FP64 pipe, where an instruction costs the same with one active lane or 32: two
// multiplications per entry are left, the order of non-negative doubles being that of their bits; few
// lanes share a row, so that few are past its end; and the square root and division (about 20
// instructions) run on packed rows, not in the one lane of a group that has the statistic (61 to 77
// ms for the create below).  Not a reciprocal square root: on matrices of +-1 the factors lie on
// the ties of the rounding to powers of two, where the last bit decides.  Create, 64 iterations and
// free, with few lanes a row in k_copy_rows as well: 30M entries 61.1 to 47.4 ms, 2.5M entries 11.4
// to 10.0 ms.
constexpr int kStatLong = 32;

template <int OP>
struct StatAcc {
  double s = 0.0;                    // not negative
  __device__ __forceinline__ void join(double t) {
    if (OP == 0) s = __double_as_longlong(t) > __double_as_longlong(s) ? t : s;
    else s += t;
  }
  __device__ __forceinline__ void add(double v, double sr, double c, double alpha) {
    const double a = v * sr * c;
    join(OP == 2 ? pow(a, alpha) : a);
  }
};

template <int OP, int G>
__global__ void __launch_bounds__(256)
k_side_scale(int nrows, const int *__restrict__ ptr, const int *__restrict__ idx,
             const double *__restrict__ val, const double *__restrict__ rs,
             const double *__restrict__ cs, double alpha, double *__restrict__ out) {
  constexpr int kRows = 256 / G;               // rows of a CTA
  __shared__ int longs[kRows], nlong;
  __shared__ double part[8], stat[kRows];
  if (threadIdx.x == 0) nlong = 0;
  __syncthreads();
  const long long r0 = (long long)blockIdx.x * kRows;
  const int mine = threadIdx.x / G, sub = threadIdx.x % G;
  const bool in = r0 + mine < nrows;
  const int r = in ? (int)(r0 + mine) : 0;
  const int pb = in ? ptr[r] : 0, pe = in ? ptr[r + 1] : 0;
  const double sr = in ? rs[r] : 0.0;
  // (a sum keeps one order, that of its G lanes: its last bits reach mixed-precision results)
  const bool lg = OP == 0 && pe - pb > kStatLong * G;
  StatAcc<OP> acc;
  if (!lg)
    for_strided(pb, pe, sub, G, [&](int p) { acc.add(fabs(val[p]), sr, cs[idx[p]], alpha); });
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) acc.join(__shfl_xor_sync(0xffffffffu, acc.s, o, G));
  if (sub == 0) {
    if (lg) longs[atomicAdd(&nlong, 1)] = mine;
    else stat[mine] = acc.s;
  }
  __syncthreads();
  for (int k = 0; k < nlong; ++k) {            // the same order of additions whatever the list's
    const int q = (int)r0 + longs[k];
    const double sq = rs[q];
    const int qe = ptr[q + 1];
    StatAcc<OP> a;
    for_strided(ptr[q], qe, threadIdx.x, 256,
                [&](int p) { a.add(fabs(val[p]), sq, cs[idx[p]], alpha); });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a.join(__shfl_xor_sync(0xffffffffu, a.s, o));
    if (threadIdx.x % 32 == 0) part[threadIdx.x / 32] = a.s;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) a.join(part[w]);
      stat[longs[k]] = a.s;
    }
    __syncthreads();
  }
  const int t = threadIdx.x;
  if (t < kRows && r0 + t < nrows) {
    const double s = stat[t], f = rs[r0 + t];
    out[r0 + t] = s > 0.0 ? f / sqrt(s) : f;
  }
}

// One scaled entry to its place in the short or long arrays, with an FP32 (LOWP 1) or BF16 (LOWP 2)
// copy of the value.
template <int LOWP>
struct EntryOut {
  int *idx;
  double *val;
  float *val32;
  __nv_bfloat16 *val16;
  __device__ __forceinline__ void put(int o, int j, double v) const {
    idx[o] = j;
    val[o] = v;
    if (LOWP == 1) val32[o] = (float)v;
    if (LOWP == 2) val16[o] = __float2bfloat16_rn((float)v);
  }
};

// The short rows' entries, G lanes per row (a warp per row left most lanes idle on rows of a few
// entries).
template <int LOWP, int G>
__global__ void __launch_bounds__(256)
k_copy_rows(int nrows, const int *__restrict__ ptr, const int *__restrict__ idx,
            const double *__restrict__ val, const double *__restrict__ rs,
            const double *__restrict__ cs, const int *__restrict__ ptr_s,
            const uint32_t *__restrict__ long_mask, EntryOut<LOWP> out) {
  const long long w = (blockIdx.x * 256LL + threadIdx.x) / G;
  if (w >= nrows) return;
  const int r = (int)w;
  if ((long_mask[r >> 5] >> (r & 31)) & 1u) return;
  const int b = ptr[r], len = ptr[r + 1] - b, o = ptr_s[r];
  const double sr = rs[r];
#pragma unroll 4
  for (int t = threadIdx.x % G; t < len; t += G) {
    const int j = idx[b + t];
    out.put(o + t, j, sr * val[b + t] * cs[j]);
  }
}

// The long rows' entries, a warp per chunk with its eight entries a lane in flight.  (With the lanes
// of a short row, chosen from the mean length, one row's dependent loads were the whole pass: in mixed
// precision a row of 1M entries took 75.8 ms, with one warp 23.8, now 0.05; the power-law columns of
// 2.5M entries 427 us, 182, now 63 with their short columns.)
template <int LOWP>
__global__ void __launch_bounds__(256)
k_copy_chunks(int nchunks, const int4 *__restrict__ desc, const int *__restrict__ long_rows,
              const int *__restrict__ beg_l, const int *__restrict__ ptr,
              const int *__restrict__ idx, const double *__restrict__ val,
              const double *__restrict__ rs, const double *__restrict__ cs, EntryOut<LOWP> out) {
  const long long w = (blockIdx.x * 256LL + threadIdx.x) / kWarp;
  if (w >= nchunks) return;
  const int4 d = desc[w];                      // long row, entries [d.y, d.z) of the long array
  const int r = long_rows[d.x], len = d.z - d.y;
  const int b = ptr[r] + (d.y - beg_l[d.x]);
  const double sr = rs[r];
#pragma unroll
  for (int u = 0; u < kChunk / kWarp; ++u) {
    const int t = u * kWarp + threadIdx.x % kWarp;
    if (t < len) {
      const int j = idx[b + t];
      out.put(d.y + t, j, sr * val[b + t] * cs[j]);
    }
  }
}

// each factor rounded to the power of two nearest to it on a log scale
__global__ void k_round_pow2(int n, double *v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int e = 0;
  const double f = frexp(v[i], &e);           // v = f 2^e, f in [0.5, 1)
  v[i] = ldexp(1.0, f >= 0.70710678118654752440 ? e : e - 1);
}

// flag = 1 if some value has more than 8 significant bits (not exact in BF16) or lies outside
// the FP32 exponent range
__global__ void k_check_bf16(long long nnz, const double *val, unsigned int *flag) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < nnz;
       p += (long long)gridDim.x * blockDim.x) {
    const double v = val[p];
    const float f = (float)v;
    const float h = __bfloat162float(__float2bfloat16_rn(f));
    if ((double)h != v) atomicOr(flag, 1u);
  }
}

__global__ void k_sumsq_part(int n, const double *x, double *part) {
  // fixed grid of 256 blocks x 256 threads; deterministic
  __shared__ double sh[256];
  double s = 0.0;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += 256LL * gridDim.x) {
    double v = x[i];
    s += v * v;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_sum_final(int nparts, const double *part, double *out) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 256) s += part[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

template <typename T>
__global__ void k_fill(int n, T v, T *x) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = v;
}

__global__ void k_vmul(int n, const double *a, const double *x, double *y, int div) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  // 0 and +-inf divided by a positive factor are themselves (bounds, mostly; a division takes
  // about ten FP64 instructions)
  const long long b = __double_as_longlong(v) & 0x7fffffffffffffffll;
  if (!div) y[i] = a[i] * v;
  else y[i] = b == 0 || b == 0x7ff0000000000000ll ? v : v / a[i];
}

__global__ void k_vclamp(int n, double *x, const double *l, const double *u) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = fmin(fmax(x[i], l[i]), u[i]);
}

__global__ void __launch_bounds__(kBlockThreads)
k_side_spmv(SideLayout lay, SideVals<double> vals, WalkScratch ws,
            const double *__restrict__ src, double *out) {
  extern __shared__ double smem[];
  double *my = smem + (threadIdx.x >> 5) * lay.seg;
  auto epi = [&](int row, double dot, bool) { out[row] = dot; };
  auto gather = [&](int j) { return src[j]; };
  auto gdone = [&](int) {};
  walk_tiles<double, double>(lay, vals, gather, my, ws, epi, gdone);
}

// One product of the power iteration on K^T K^: out = side * (src * in_scale[0]) (in_scale NULL:
// 1), plus ss[0] = ||out||^2 and ss[1] = 1 / ||out|| (0 for a zero vector) from the grid's
// deterministic ticket reduction.  The next product reads ss + 1 as its input scale, so the
// normalisation v = w / ||w|| costs no launch of its own.  PT is the vector, product and row-sum
// type: FP64 with the FP64 values; FP32 with the FP32 or BF16 values of a mixed-precision handle,
// where the input scale is applied to each row's sum (in FP64) instead of to every gathered entry
// and the norm is still an FP64 sum, of the rows before they are rounded to the FP32 vector.  (An
// FP64 vector, rounded as it was gathered, gave the same bits with twice the vector traffic:
// create, 64
// iterations and free of a 30M-entry LP in BF16 76.3 to 69.1 ms, of a 2.5M-entry LP in FP32 13.3 to
// 12.8 ms.)
template <typename VT, typename PT>
__global__ void __launch_bounds__(kBlockThreads)
k_side_spmv_pw(SideLayout lay, SideVals<VT> vals, WalkScratch ws,
               const PT *__restrict__ src, const double *in_scale, PT *out, double *part,
               unsigned int *ticket, double *ss) {
  extern __shared__ double smem[];
  PT *my = reinterpret_cast<PT *>(smem) + (threadIdx.x >> 5) * lay.seg;
  constexpr bool kF64 = sizeof(PT) == sizeof(double);
  const double sc = in_scale ? *in_scale : 1.0;
  const double post = kF64 ? 1.0 : sc;
  Acc<1, 0> a, al;
  a.zero();
  al.zero();
  auto epi = [&](int row, PT dot, bool lg) {
    const double o = (double)dot * post;
    out[row] = (PT)o;
    if (lg) al.s[0] += o * o;
    else a.s[0] += o * o;
  };
  auto gather = [&](int j) { return kF64 ? PT(src[j] * sc) : src[j]; };
  auto gdone = [&](int grp) { store_group(al, 0x1u, ws.group_part, grp); };
  walk_tiles<VT, PT>(lay, vals, gather, my, ws, epi, gdone);
  if (!ss) return;       // a product whose norm nothing reads (every K^ v but the last)
  if (cta_reduce_and_ticket(a, 0x1u, 0u, 0u, part, ticket)) {
    double r[1];
    grid_finish<1, 0>(part, r, 0x1u, 0u, ws.group_part, lay.n_long_tiles);
    if (threadIdx.x == 0) {
      ss[0] = r[0];
      ss[1] = r[0] > 0.0 ? 1.0 / sqrt(r[0]) : 0.0;
      *ticket = 0u;
    }
  }
}

// ---- layout plan on the device ---------------------------------------------------------------
// The plan of plan_side (plan.h) from row pointers in device memory, by one warp per tile of 32
// rows, a lane per row; the host reads back one summary and the arrays are written where they are
// used.  (Planned on one host core, with the row pointers copied down and the arrays copied up, the
// 10M columns and 1.75M rows of a 30M-entry flow LP took 42 of the 119 ms of create, 64 iterations
// and free; planned here, the whole took 76 ms.  250k columns and 100k rows: 14.5 to 13.3 ms.)
// Three passes: k_plan_tiles makes every tile's long-row mask and counts and each block's totals,
// k_plan_scan turns the totals into starts (one block; there is one record per kPlanTiles tiles),
// k_plan_emit writes the arrays.

constexpr int kPlanTiles = 64;       // tiles of a block: 8 warps, 8 tiles each; a multiple of
                                     // kMaxTileMult, so that no tile group spans two blocks
constexpr int kPlanThreads = 256;
static_assert(kPlanTiles % kMaxTileMult == 0 && kPlanTiles % (kPlanThreads / 32) == 0, "");

// What a tile, a block, or all tiles hold: entries of the short array (each tile's segment padded
// to 4) and of the long array (each row padded to 4), long rows and their chunks.
struct PlanCount {
  long long s, l;
  int nl, nc;
};
__device__ __forceinline__ PlanCount operator+(PlanCount a, const PlanCount &b) {
  a.s += b.s;
  a.l += b.l;
  a.nl += b.nl;
  a.nc += b.nc;
  return a;
}
struct PlanTile {
  uint32_t mask;     // long rows
  int seg, nc;       // entries of the short segment; chunks of the long rows
  int pad_;
  long long l;       // padded entries of the long rows
};
struct PlanBlock {
  PlanCount c;                  // totals; after k_plan_scan what precedes the block
  long long plain, best;        // FP64 adds of wide_rows_pay
  int maxseg[3];                // longest group segment of 1, 2 and 4 tiles
};

__device__ __forceinline__ int plan_align4(int v) { return (v + 3) & ~3; }

__global__ void __launch_bounds__(kPlanThreads)
k_plan_tiles(int nrows, int ntiles, const int *__restrict__ ptr, PlanTile *tiles,
             PlanBlock *blocks) {
  __shared__ PlanTile sh[kPlanTiles];
  __shared__ int cost[kPlanTiles][2];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x >> 5; k < kPlanTiles; k += kPlanThreads / 32) {
    const int t = blockIdx.x * kPlanTiles + k;
    const long long r = (long long)t * kTileRows + lane;
    const int len = t < ntiles && r < nrows ? ptr[r + 1] - ptr[r] : 0;
    bool lg = len > kShortMax;
    int sum = (int)__reduce_add_sync(full, lg ? 0u : (unsigned)len);
    while (sum > kSegBudget) {            // the longest short row, the first of equal ones
      const unsigned key = lg ? 0u : (unsigned)(len * 32 + 31 - lane) + 1u;
      const unsigned top = __reduce_max_sync(full, key) - 1u;
      if (lane == 31 - (int)(top & 31u)) lg = true;
      sum -= (int)(top >> 5);
    }
    const uint32_t mask = __ballot_sync(full, lg);
    // FP64 adds of the lane-per-row sums and of the best warp-wide threshold (wide_rows_pay)
    const int sl = lg ? 0 : len;
    const int mx = (int)__reduce_max_sync(full, (unsigned)sl);
    const int plain = plan_align4(mx);
    int best = plain;
    if (mx > 16)
      for (int c = 8; c <= 32 && c < mx; c *= 2)
        best = min(best, c + (int)__reduce_add_sync(
                                 full, sl > c ? (unsigned)(((sl + 31) >> 5) + 5) : 0u));
    int nc = 0;
    long long l = 0;
    if (mask) {                            // warp-uniform
      nc = (int)__reduce_add_sync(full, lg ? (unsigned)((len + kChunk - 1) / kChunk) : 0u);
      l = lg ? ((long long)len + 3) & ~3LL : 0;
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(full, l, o);
    }
    if (lane == 0) {
      sh[k] = PlanTile{mask, sum, nc, 0, l};
      cost[k][0] = plain;
      cost[k][1] = best;
      if (t < ntiles) tiles[t] = sh[k];
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    static_assert(kPlanTiles == 64, "two tiles per lane below");
    PlanCount c{};
    int plain = 0, best = 0;
    const PlanTile a = sh[2 * lane], b = sh[2 * lane + 1];   // tiles past the last hold zeros
    c.s = plan_align4(a.seg) + plan_align4(b.seg);
    c.l = a.l + b.l;
    c.nl = __popc(a.mask) + __popc(b.mask);
    c.nc = a.nc + b.nc;
    plain = cost[2 * lane][0] + cost[2 * lane + 1][0];
    best = cost[2 * lane][1] + cost[2 * lane + 1][1];
    // group segments run to the last tile's unpadded end; a ragged last group has fewer tiles
    const int t0 = blockIdx.x * kPlanTiles + 2 * lane;
    const bool has_b = t0 + 1 < ntiles;
    const int m1 = max(a.seg, b.seg);
    const int m2 = has_b ? plan_align4(a.seg) + b.seg : a.seg;
    const int up = __shfl_down_sync(full, m2, 1);
    const int m4 = t0 + 2 < ntiles ? plan_align4(a.seg) + plan_align4(b.seg) + up : m2;
    const int x1 = (int)__reduce_max_sync(full, (unsigned)m1);
    const int x2 = (int)__reduce_max_sync(full, (unsigned)m2);
    const int x4 = (int)__reduce_max_sync(full, lane % 2 == 0 ? (unsigned)m4 : 0u);
    for (int o = 16; o > 0; o >>= 1) {
      c.s += __shfl_xor_sync(full, c.s, o);
      c.l += __shfl_xor_sync(full, c.l, o);
      c.nl += __shfl_xor_sync(full, c.nl, o);
      c.nc += __shfl_xor_sync(full, c.nc, o);
      plain += __shfl_xor_sync(full, plain, o);
      best += __shfl_xor_sync(full, best, o);
    }
    if (lane == 0) blocks[blockIdx.x] = PlanBlock{c, plain, best, {x1, x2, x4}};
  }
}

// One block: every block's totals become what precedes it; all[0] the totals over all blocks.
__global__ void __launch_bounds__(kPlanThreads)
k_plan_scan(int nblocks, PlanBlock *blocks, PlanBlock *all) {
  __shared__ PlanCount sh[kPlanThreads];
  __shared__ long long cost[kPlanThreads][2];
  __shared__ int mxs[kPlanThreads][3];
  const int tid = threadIdx.x;
  const int per = (nblocks + kPlanThreads - 1) / kPlanThreads;
  const int b0 = min(tid * per, nblocks), b1 = min(b0 + per, nblocks);
  PlanCount c{};
  long long plain = 0, best = 0;
  int mx[3] = {0, 0, 0};
#pragma unroll 4
  for (int b = b0; b < b1; ++b) {
    const PlanBlock r = blocks[b];
    c = c + r.c;
    plain += r.plain;
    best += r.best;
    for (int k = 0; k < 3; ++k) mx[k] = max(mx[k], r.maxseg[k]);
  }
  sh[tid] = c;
  cost[tid][0] = plain;
  cost[tid][1] = best;
  for (int k = 0; k < 3; ++k) mxs[tid][k] = mx[k];
  __syncthreads();
  for (int o = 1; o < kPlanThreads; o *= 2) {       // inclusive scan; totals in the last thread
    PlanCount p{};
    long long q0 = 0, q1 = 0;
    int m[3] = {0, 0, 0};
    if (tid >= o) {
      p = sh[tid - o];
      q0 = cost[tid - o][0];
      q1 = cost[tid - o][1];
      for (int k = 0; k < 3; ++k) m[k] = mxs[tid - o][k];
    }
    __syncthreads();
    sh[tid] = sh[tid] + p;
    cost[tid][0] += q0;
    cost[tid][1] += q1;
    for (int k = 0; k < 3; ++k) mxs[tid][k] = max(mxs[tid][k], m[k]);
    __syncthreads();
  }
  if (tid == kPlanThreads - 1)
    *all = PlanBlock{sh[tid], cost[tid][0], cost[tid][1], {mxs[tid][0], mxs[tid][1], mxs[tid][2]}};
  PlanCount before{};
  if (tid > 0) before = sh[tid - 1];
  for (int b = b0; b < b1; ++b) {
    const PlanCount own = blocks[b].c;
    blocks[b].c = before;
    before = before + own;
  }
}

__global__ void __launch_bounds__(kPlanThreads)
k_plan_emit(int nrows, int ntiles, const int *__restrict__ ptr, const PlanTile *tiles,
            const PlanBlock *blocks, int *ptr_s, int *tile_end, uint32_t *long_mask,
            int *long_rows, int *beg_l, int *end_l, int *chunk_ptr, int *chunk_row) {
  __shared__ PlanCount sh[kPlanTiles];      // what precedes each tile, from the block's start
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, tid = threadIdx.x;
  const int first = blockIdx.x * kPlanTiles;
  if (tid < kPlanTiles) {
    PlanCount c{};
    if (first + tid < ntiles) {
      const PlanTile x = tiles[first + tid];
      c.s = plan_align4(x.seg);
      c.l = x.l;
      c.nl = __popc(x.mask);
      c.nc = x.nc;
    }
    sh[tid] = c;
  }
  __syncthreads();
  for (int o = 1; o < kPlanTiles; o *= 2) {
    PlanCount p{};
    if (tid < kPlanTiles && tid >= o) p = sh[tid - o];
    __syncthreads();
    if (tid < kPlanTiles) sh[tid] = sh[tid] + p;
    __syncthreads();
  }
  const PlanCount base = blocks[blockIdx.x].c;
  if (blockIdx.x == 0 && tid == 0) chunk_ptr[0] = 0;
  for (int k = tid >> 5; k < kPlanTiles; k += kPlanThreads / 32) {
    const int t = first + k;
    if (t >= ntiles) break;
    PlanCount at = base;
    if (k > 0) at = at + sh[k - 1];
    const long long r = (long long)t * kTileRows + lane;
    const int len = r < nrows ? ptr[r + 1] - ptr[r] : 0;
    const uint32_t mask = tiles[t].mask;
    const bool lg = (mask >> lane) & 1u;
    int incl = lg ? 0 : len;                 // short entries up to and with this row
    for (int o = 1; o < 32; o *= 2) {
      const int v = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += v;
    }
    const int start = (int)at.s + incl - (lg ? 0 : len);
    if (mask) {                              // warp-uniform
      const int nc = lg ? (len + kChunk - 1) / kChunk : 0;
      const long long pl = lg ? ((long long)len + 3) & ~3LL : 0;
      int ci = nc;
      long long li = pl;
      for (int o = 1; o < 32; o *= 2) {
        const int v = __shfl_up_sync(full, ci, o);
        const long long w = __shfl_up_sync(full, li, o);
        if (lane >= o) {
          ci += v;
          li += w;
        }
      }
      const int row = at.nl + __popc(mask & ((1u << lane) - 1u));
      if (lg) {
        const int to = (int)(at.l + li - pl);
        long_rows[row] = (int)r;
        beg_l[row] = to;
        end_l[row] = to + len;
        chunk_ptr[row + 1] = at.nc + ci;
      }
      for (uint32_t left = mask; left; left &= left - 1u) {
        const int b = __ffs((int)left) - 1;
        const int n = __shfl_sync(full, nc, b), c1 = at.nc + __shfl_sync(full, ci, b);
        const int id = __shfl_sync(full, row, b);
        for (int c = c1 - n + lane; c < c1; c += 32) chunk_row[c] = id;
      }
    }
    if (r < nrows) ptr_s[r] = start;
    if (lane == 0) {
      tile_end[t] = (int)at.s + tiles[t].seg;
      long_mask[t] = mask;
    }
  }
}

// Per chunk: its long row, entry range, and the chunk count of its group of 32 long rows.
__global__ void k_plan_desc(int nchunks, int nlong, const int *chunk_row, const int *chunk_ptr,
                            const int *beg_l, const int *end_l, int4 *desc) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nchunks) return;
  const int li = chunk_row[c];
  const int cb = beg_l[li] + (c - chunk_ptr[li]) * kChunk;
  const int g0 = (li / kTileRows) * kTileRows, g1 = min(g0 + kTileRows, nlong);
  desc[c] = make_int4(li, cb, min(cb + kChunk, end_l[li]), chunk_ptr[g1] - chunk_ptr[g0]);
}

}  // namespace

static std::atomic<long long> g_launches{0};
void count_launches(long long n) { g_launches += n; }
long long launches_so_far() { return g_launches.load(); }

unsigned int validate_problem(cudaStream_t st, int m, int n, long long nnz,
                              const long long *row_ptr, const int *col, const double *val,
                              const double *c, const double *q, const double *l, const double *u,
                              unsigned int *d_flags) {
  cudaMemsetAsync(d_flags, 0, sizeof(unsigned int), st);
  k_validate_rows<<<nblocks(m + 1, 256), 256, 0, st>>>(m, n, nnz, row_ptr, col, val, q, d_flags);
  k_validate_cols<<<nblocks(n, 256), 256, 0, st>>>(n, c, l, u, d_flags);
  count_launches(2);
  unsigned int h = 0;
  cudaMemcpyAsync(&h, d_flags, sizeof(h), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return h;
}

void convert_row_ptr(cudaStream_t st, int m, const long long *rp64, int *rp32) {
  k_rp_convert<<<nblocks(m + 1, 256), 256, 0, st>>>(m, rp64, rp32);
  count_launches(1);
}

cudaError_t build_transpose(cudaStream_t st, int m, int n, int nnz, const int *rp, const int *col,
                            const double *val, int *cp, int *ridx, double *cval) {
  cudaError_t err;
  int *rows_of = nullptr, *iota = nullptr, *keys_out = nullptr, *perm = nullptr, *cnt = nullptr;
  void *tmp = nullptr;
  size_t tmp_bytes = 0, scan_bytes = 0;
  const size_t nz = (size_t)std::max(nnz, 1);
  if ((err = buf_alloc((void **)&rows_of, nz * sizeof(int)))) goto done;
  if ((err = buf_alloc((void **)&iota, nz * sizeof(int)))) goto done;
  if ((err = buf_alloc((void **)&keys_out, nz * sizeof(int)))) goto done;
  if ((err = buf_alloc((void **)&perm, nz * sizeof(int)))) goto done;
  if ((err = buf_alloc((void **)&cnt, (size_t)(n + 1) * sizeof(int)))) goto done;
  {
    int end_bit = 1;
    while ((1LL << end_bit) < (long long)n) ++end_bit;
    cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, col, keys_out, iota, perm, nnz, 0, end_bit,
                                    st);
    cub::DeviceScan::ExclusiveSum(nullptr, scan_bytes, cnt, cp, n + 1, st);
    tmp_bytes = std::max(tmp_bytes, scan_bytes);
    if ((err = buf_alloc(&tmp, std::max<size_t>(tmp_bytes, 16)))) goto done;
    k_expand_rows<<<nblocks(m, 256), 256, 0, st>>>(m, rp, rows_of);
    k_iota<<<nblocks(nnz, 256), 256, 0, st>>>(nnz, iota);
    if (nnz > 0)
      cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, col, keys_out, iota, perm, nnz, 0, end_bit,
                                      st);
    cudaMemsetAsync(cnt, 0, (size_t)(n + 1) * sizeof(int), st);
    k_count_cols<<<nblocks(nnz, 256), 256, 0, st>>>(nnz, col, cnt);
    cub::DeviceScan::ExclusiveSum(tmp, tmp_bytes, cnt, cp, n + 1, st);
    k_gather_csc<<<nblocks(nnz, 256), 256, 0, st>>>(nnz, perm, rows_of, val, ridx, cval);
    count_launches(4);
    err = cudaStreamSynchronize(st);
    if (err == cudaSuccess) err = cudaGetLastError();
  }
done:
  cudaStreamSynchronize(st);     // nothing in flight uses the scratch when it goes back
  buf_release(rows_of);
  buf_release(iota);
  buf_release(keys_out);
  buf_release(perm);
  buf_release(cnt);
  buf_release(tmp);
  return err;
}

// f(std::integral_constant<int, G>) for a side's lanes per row, which decide only the time: an
// eighth of the mean row length, at least kMin (1 or 4) and at most 32.  More lanes leave more of
// them idle past the rows' ends (17 entries take 5 steps of 4 lanes, 85% busy, or one and a bit of
// 16); fewer than four do not read whole sectors, which only pays where rows have about as few entries.
template <int kMin, class F>
static void with_group(long long nnz, int nrows, F &&f) {
  const double mean = nrows > 0 ? (double)nnz / nrows : 0.0;
  if (kMin == 1 && mean <= 4.0) f(std::integral_constant<int, kMin>{});
  else if (mean <= 32.0) f(std::integral_constant<int, 4>{});
  else if (mean <= 64.0) f(std::integral_constant<int, 8>{});
  else if (mean <= 128.0) f(std::integral_constant<int, 16>{});
  else f(std::integral_constant<int, 32>{});
}
// The same for sums, whose order they decide: the mean row length rounded up to a power of two.
template <class F>
static void with_sum_group(long long nnz, int nrows, F &&f) {
  const double mean = nrows > 0 ? (double)nnz / nrows : 0.0;
  if (mean <= 4.0) f(std::integral_constant<int, 4>{});
  else if (mean <= 8.0) f(std::integral_constant<int, 8>{});
  else if (mean <= 16.0) f(std::integral_constant<int, 16>{});
  else f(std::integral_constant<int, 32>{});
}

template <int OP>
static void side_scale(cudaStream_t st, int nrows, long long nnz, const int *ptr, const int *idx,
                       const double *val, const double *rs, const double *cs, double alpha,
                       double *out) {
  if (nrows <= 0) return;
  auto pass = [&](auto G) {
    k_side_scale<OP, G()><<<nblocks((long long)nrows * G(), 256), 256, 0, st>>>(
        nrows, ptr, idx, val, rs, cs, alpha, out);
  };
  if (OP == 0) with_group<1>(nnz, nrows, pass);
  else with_sum_group(nnz, nrows, pass);
  count_launches(1);
}

void compute_scaling(cudaStream_t st, int m, int n, long long nnz, const int *rp, const int *col,
                     const double *val, const int *cp, const int *ridx, const double *cval,
                     int ruiz_iters, double alpha, double *D, double *E, double *tmp_m,
                     double *tmp_n) {
  // both sides' new factors from the same current ones, so every pass goes from one pair of
  // buffers to the other; the last lands in D, E
  const int passes = ruiz_iters + (alpha >= 0.0 ? 1 : 0);
  if (passes % 2) {
    std::swap(D, tmp_m);
    std::swap(E, tmp_n);
  }
  k_fill<<<nblocks(m, 256), 256, 0, st>>>(m, 1.0, D);
  k_fill<<<nblocks(n, 256), 256, 0, st>>>(n, 1.0, E);
  count_launches(2);
  for (int it = 0; it < passes; ++it) {
    if (it < ruiz_iters) {
      side_scale<0>(st, m, nnz, rp, col, val, D, E, 1.0, tmp_m);
      side_scale<0>(st, n, nnz, cp, ridx, cval, E, D, 1.0, tmp_n);
    } else {
      auto pock_chambolle = [&](auto OP, auto OQ) {
        side_scale<OP()>(st, m, nnz, rp, col, val, D, E, alpha, tmp_m);
        side_scale<OQ()>(st, n, nnz, cp, ridx, cval, E, D, 2.0 - alpha, tmp_n);
      };
      using One = std::integral_constant<int, 1>;
      using Pow = std::integral_constant<int, 2>;
      if (alpha == 1.0) pock_chambolle(One{}, One{});
      else pock_chambolle(Pow{}, Pow{});
    }
    std::swap(D, tmp_m);
    std::swap(E, tmp_n);
  }
}

// A side is skewed (its ordered FP64 tiles take tile_rows_wide) when summing its tiles' longest rows
// by whole warps saves at least 15% of the FP64 adds of lane-per-row sums.
static bool wide_pays(long long plain, long long best) {
  return plain > 0 && (double)best <= 0.85 * (double)plain;
}

// That cost model over all short tiles: FP64 adds per warp of the lane-per-row sums (the longest
// row, rounded up to 4) against the best threshold's (c + the sum over rows longer than c of
// ceil(len / 32) + 5, c in 8, 16, 32).
static bool wide_rows_pay(const int *hp, const std::vector<uint32_t> &mask, int nrows) {
  long long plain = 0, best = 0;
  for (int t = 0; t * kTileRows < nrows; ++t) {
    int len[kTileRows];
    int mx = 0;
    for (int r = 0; r < kTileRows; ++r) {
      const int row = t * kTileRows + r;
      len[r] = (row < nrows && !((mask[t] >> r) & 1u)) ? hp[row + 1] - hp[row] : 0;
      mx = std::max(mx, len[r]);
    }
    const int p = (mx + 3) & ~3;
    int b = p;
    if (mx > 16) {
      for (int c = 8; c <= 32 && c < mx; c *= 2) {
        int cost = c;
        for (int r = 0; r < kTileRows; ++r)
          if (len[r] > c) cost += ((len[r] + 31) >> 5) + 5;
        b = std::min(b, cost);
      }
    }
    plain += p;
    best += b;
  }
  return wide_pays(plain, best);
}

// Tiles per work item: where tiles are short (a few entries per row), M consecutive tiles are
// staged as one segment, so that each warp's chain of dependent loads carries M tiles' bytes.
// M is the largest of kMaxTileMult, ..., 2 whose mean group segment fits one staging round
// (128 * kStageUnroll entries) and whose longest fits the staging budget; else 1.  nnz_s: entries
// of the short array; maxseg_mult: longest group segments (-1: over the budget).
static int rule_mult(int ntiles, long long nnz_s, const long long *maxseg_mult) {
  for (int k = 2, cand = kMaxTileMult; cand >= 2; --k, cand /= 2) {
    if (ntiles < 2 * cand) continue;
    if (nnz_s * cand > (long long)ntiles * kWarp * kStageUnroll * 4) continue;
    if (maxseg_mult[k] >= 0) return cand;
  }
  return 1;
}

bool plan_side(const int *hp, int nrows, SidePlan *p) {
  SidePlan &P = *p;
  const int ntiles = (nrows + kTileRows - 1) / kTileRows;
  P = SidePlan();
  P.nrows = nrows;
  P.ntiles = ntiles;
  P.ptr_s.assign(std::max(nrows, 1), 0);
  P.tile_end.assign(std::max(ntiles, 1), 0);
  P.dst.assign(std::max(nrows, 1), 0);
  P.mask.assign(std::max(ntiles, 1), 0u);
  P.chunk_ptr.assign(1, 0);
  long long cur = 0, cl = 0, maxseg = 0;
  auto align4 = [](long long v) { return (v + 3) & ~3LL; };
  for (int t = 0; t < ntiles; ++t) {
    const int r0 = t * kTileRows, r1 = std::min(nrows, (t + 1) * kTileRows);
    // membership: rows over kShortMax are long; then, while the tile's short segment exceeds
    // kSegBudget, its longest short row (the first of equal ones) becomes long
    long long sum = 0;
    for (int r = r0; r < r1; ++r) {
      const int len = hp[r + 1] - hp[r];
      if (len > kShortMax) P.mask[t] |= 1u << (r - r0);
      else sum += len;
    }
    while (sum > kSegBudget) {
      int best = -1, blen = -1;
      for (int r = r0; r < r1; ++r) {
        const int len = hp[r + 1] - hp[r];
        if (!((P.mask[t] >> (r - r0)) & 1u) && len > blen) { best = r; blen = len; }
      }
      P.mask[t] |= 1u << (best - r0);
      sum -= blen;
    }
    cur = align4(cur);
    const long long seg_b = cur;
    for (int r = r0; r < r1; ++r) {
      const int len = hp[r + 1] - hp[r];
      P.ptr_s[r] = (int)cur;
      if (!((P.mask[t] >> (r - r0)) & 1u)) {
        P.dst[r] = (int)cur;
        cur += len;
      } else {
        cl = align4(cl);
        const int li = (int)P.long_rows.size();
        P.long_rows.push_back(r);
        P.beg_l.push_back((int)cl);
        P.end_l.push_back((int)(cl + len));
        P.dst[r] = (int)cl;
        cl += len;
        const int nc = (len + kChunk - 1) / kChunk;
        for (int c = 0; c < nc; ++c) P.chunk_row.push_back(li);
        P.chunk_ptr.push_back(P.chunk_ptr.back() + nc);
      }
      if (cur > INT_MAX - 8 || cl > INT_MAX - 2 * kChunk) return false;   // casts stay in range
    }
    P.tile_end[t] = (int)cur;
    maxseg = std::max(maxseg, cur - seg_b);
  }
  P.nnz_s = align4(cur) + 4;
  P.nnz_l = align4(cl) + kChunk;
  if (P.nnz_s > INT_MAX || P.nnz_l > INT_MAX) return false;
  P.maxseg_mult[0] = maxseg;
  for (int k = 1, cand = 2; cand <= kMaxTileMult; ++k, cand *= 2) {
    long long mx = 0;
    for (int t0 = 0; t0 < ntiles; t0 += cand) {
      const int t1 = std::min(ntiles, t0 + cand) - 1;
      mx = std::max(mx, (long long)P.tile_end[t1] - P.ptr_s[(size_t)t0 * kTileRows]);
    }
    P.maxseg_mult[k] = (ntiles > 0 && mx <= kSegBudget) ? mx : -1;
  }
  P.mult = rule_mult(ntiles, align4(cur), P.maxseg_mult);
  P.maxseg = P.maxseg_mult[P.mult == 4 ? 2 : P.mult - 1];
  P.wide_rows = wide_rows_pay(hp, P.mask, nrows) ? 1 : 0;
  return true;
}

cudaError_t build_side(cudaStream_t st, int nrows, const int *ptr, const int *idx,
                       const double *val, const double *rscale, const double *cscale,
                       int lowp, SideStore *out) {
  SideStore s;
  cudaError_t err = cudaSuccess;
  const int ntiles = (int)(((long long)nrows + kTileRows - 1) / kTileRows);
  const int nplan = (ntiles + kPlanTiles - 1) / kPlanTiles;
  PlanTile *d_tiles = nullptr;
  PlanBlock *d_blocks = nullptr;
  PlanBlock tot{};
  long long nnz_s = 0, nnz_l = 0;
  int nlong = 0, nch = 0;
  size_t ng = 1;
  auto get = [](auto **d, size_t count) {
    return buf_alloc((void **)d, std::max<size_t>(count, 1) * sizeof(**d));
  };
#define TRY(x)                 \
  do {                         \
    if ((err = (x))) goto fail; \
  } while (0)
  // ---- structure: counts, then arrays of their sizes -----------------------------------------
  TRY(get(&d_tiles, ntiles));
  TRY(get(&d_blocks, (size_t)nplan + 1));
  if (ntiles > 0) {
    k_plan_tiles<<<nplan, kPlanThreads, 0, st>>>(nrows, ntiles, ptr, d_tiles, d_blocks);
    k_plan_scan<<<1, kPlanThreads, 0, st>>>(nplan, d_blocks, d_blocks + nplan);
    count_launches(2);
    TRY(cudaMemcpyAsync(&tot, d_blocks + nplan, sizeof(tot), cudaMemcpyDeviceToHost, st));
    TRY(cudaStreamSynchronize(st));
  }
  if (tot.c.s > INT_MAX - 16 || tot.c.l > INT_MAX - 2 * kChunk - 16) {
    // at the limit of the int32 offsets the host plan says whether they hold (its limits are on
    // unpadded ends)
    std::vector<int> hp((size_t)nrows + 1);
    SidePlan P;
    TRY(cudaMemcpy(hp.data(), ptr, hp.size() * sizeof(int), cudaMemcpyDeviceToHost));
    if (!plan_side(hp.data(), nrows, &P)) {
      err = cudaErrorInvalidValue;
      goto fail;
    }
  }
  nlong = tot.c.nl;
  nch = tot.c.nc;
  nnz_s = tot.c.s + 4;
  nnz_l = tot.c.l + kChunk;
  for (int k = 0; k < 3; ++k)
    s.maxseg_mult[k] =
        k == 0 || (ntiles > 0 && tot.maxseg[k] <= kSegBudget) ? (long long)tot.maxseg[k] : -1;
  s.rule_mult = rule_mult(ntiles, tot.c.s, s.maxseg_mult);
  s.lay.nrows = nrows;
  s.lay.n_short_tiles = ntiles;
  apply_mult(s, s.rule_mult);
  s.lay.n_long = nlong;
  s.lay.n_long_tiles = (nlong + kTileRows - 1) / kTileRows;
  s.lay.n_chunks = nch;
  s.lay.wide_rows = wide_pays(tot.plain, tot.best) ? 1 : 0;
  s.nnz_short = nnz_s;
  s.nnz_long = nnz_l;
  ng = (size_t)std::max(s.lay.n_long_tiles, 1);
  TRY(get(&s.ptr_s, nrows));
  TRY(get(&s.tile_end, ntiles));
  TRY(get(&s.long_rows, nlong));
  TRY(get(&s.beg_l, nlong));
  TRY(get(&s.end_l, nlong));
  TRY(get(&s.chunk_ptr, (size_t)nlong + 1));
  TRY(get(&s.chunk_row, nch));
  TRY(get(&s.chunk_desc, nch));
  TRY(get(&s.long_mask, ntiles));
  if (ntiles > 0) {
    k_plan_emit<<<nplan, kPlanThreads, 0, st>>>(nrows, ntiles, ptr, d_tiles, d_blocks, s.ptr_s,
                                                s.tile_end, s.long_mask, s.long_rows,
                                                s.beg_l, s.end_l, s.chunk_ptr, s.chunk_row);
    count_launches(1);
    if (nch > 0) {
      k_plan_desc<<<nblocks(nch, 256), 256, 0, st>>>(nch, nlong, s.chunk_row, s.chunk_ptr, s.beg_l,
                                                     s.end_l, s.chunk_desc);
      count_launches(1);
    }
  }
  // ---- entries (zero padding), scaled on the device ------------------------------------------
  TRY(buf_alloc((void **)&s.idx_s, nnz_s * sizeof(int)));
  TRY(buf_alloc((void **)&s.val64_s, nnz_s * sizeof(double)));
  TRY(buf_alloc((void **)&s.idx_l, nnz_l * sizeof(int)));
  TRY(buf_alloc((void **)&s.val64_l, nnz_l * sizeof(double)));
  TRY(cudaMemsetAsync(s.idx_s, 0, nnz_s * sizeof(int), st));
  TRY(cudaMemsetAsync(s.val64_s, 0, nnz_s * sizeof(double), st));
  TRY(cudaMemsetAsync(s.idx_l, 0, nnz_l * sizeof(int), st));
  TRY(cudaMemsetAsync(s.val64_l, 0, nnz_l * sizeof(double), st));
  if (lowp == 1) {
    TRY(buf_alloc((void **)&s.val32_s, nnz_s * sizeof(float)));
    TRY(buf_alloc((void **)&s.val32_l, nnz_l * sizeof(float)));
    TRY(cudaMemsetAsync(s.val32_s, 0, nnz_s * sizeof(float), st));
    TRY(cudaMemsetAsync(s.val32_l, 0, nnz_l * sizeof(float), st));
  } else if (lowp == 2) {
    TRY(buf_alloc((void **)&s.val16_s, nnz_s * sizeof(__nv_bfloat16)));
    TRY(buf_alloc((void **)&s.val16_l, nnz_l * sizeof(__nv_bfloat16)));
    TRY(cudaMemsetAsync(s.val16_s, 0, nnz_s * sizeof(__nv_bfloat16), st));
    TRY(cudaMemsetAsync(s.val16_l, 0, nnz_l * sizeof(__nv_bfloat16), st));
  }
  if (nrows > 0) {
    auto copy = [&](auto LP) {
      const EntryOut<LP()> shorts{s.idx_s, s.val64_s, s.val32_s, s.val16_s};
      const EntryOut<LP()> longs{s.idx_l, s.val64_l, s.val32_l, s.val16_l};
      with_group<4>(tot.c.s, nrows, [&](auto G) {
        k_copy_rows<LP(), G()><<<nblocks((long long)nrows * G(), 256), 256, 0, st>>>(
            nrows, ptr, idx, val, rscale, cscale, s.ptr_s, s.long_mask, shorts);
      });
      count_launches(1);
      if (nch == 0) return;
      k_copy_chunks<LP()><<<nblocks((long long)nch * kWarp, 256), 256, 0, st>>>(
          nch, s.chunk_desc, s.long_rows, s.beg_l, ptr, idx, val, rscale, cscale, longs);
      count_launches(1);
    };
    if (lowp == 1) copy(std::integral_constant<int, 1>{});
    else if (lowp == 2) copy(std::integral_constant<int, 2>{});
    else copy(std::integral_constant<int, 0>{});
  }
  // ---- walk scratch ------------------------------------------------------------------------
  TRY(buf_alloc((void **)&s.part_a, (size_t)std::max(nch, 1) * sizeof(double)));
  TRY(buf_alloc((void **)&s.part_b, (size_t)std::max(nch, 1) * sizeof(double)));
  TRY(buf_alloc((void **)&s.done_a, ng * sizeof(unsigned int)));
  TRY(buf_alloc((void **)&s.done_b, ng * sizeof(unsigned int)));
  TRY(buf_alloc((void **)&s.gpart_a, ng * kMaxPartials * sizeof(double)));
  TRY(buf_alloc((void **)&s.gpart_b, ng * kMaxPartials * sizeof(double)));
  TRY(cudaMemsetAsync(s.done_a, 0, ng * sizeof(unsigned int), st));
  TRY(cudaMemsetAsync(s.done_b, 0, ng * sizeof(unsigned int), st));
  TRY(cudaStreamSynchronize(st));
  TRY(cudaGetLastError());
#undef TRY
  buf_release(d_tiles);
  buf_release(d_blocks);
  s.lay.ptr_s = s.ptr_s;
  s.lay.tile_end = s.tile_end;
  s.lay.idx_s = s.idx_s;
  s.lay.long_mask = s.long_mask;
  s.lay.long_rows = s.long_rows;
  s.lay.beg_l = s.beg_l;
  s.lay.end_l = s.end_l;
  s.lay.idx_l = s.idx_l;
  s.lay.chunk_ptr = s.chunk_ptr;
  s.lay.chunk_row = s.chunk_row;
  s.lay.chunk_desc = s.chunk_desc;
  s.v64.s = s.val64_s;
  s.v64.l = s.val64_l;
  s.v32.s = s.val32_s;
  s.v32.l = s.val32_l;
  s.v16.s = s.val16_s;
  s.v16.l = s.val16_l;
  s.wa.chunk_part = s.part_a;
  s.wa.group_done = s.done_a;
  s.wa.group_part = s.gpart_a;
  s.wb.chunk_part = s.part_b;
  s.wb.group_done = s.done_b;
  s.wb.group_part = s.gpart_b;
  *out = s;
  return cudaSuccess;
fail:
  cudaStreamSynchronize(st);
  buf_release(d_tiles);
  buf_release(d_blocks);
  free_side(&s);
  return err;
}

void round_pow2(cudaStream_t st, int n, double *v) {
  if (n <= 0) return;
  k_round_pow2<<<nblocks(n, 256), 256, 0, st>>>(n, v);
  count_launches(1);
}

unsigned int values_exact_in_bf16(cudaStream_t st, long long nnz, const double *val,
                                  unsigned int *d_flag) {
  cudaMemsetAsync(d_flag, 0, sizeof(unsigned int), st);
  if (nnz > 0) {
    k_check_bf16<<<std::min<long long>(nblocks(nnz, 256), 4096), 256, 0, st>>>(nnz, val, d_flag);
    count_launches(1);
  }
  unsigned int h = 0;
  cudaMemcpyAsync(&h, d_flag, sizeof(h), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return h == 0;
}

void free_side(SideStore *s) {
  void *bufs[] = {s->ptr_s, s->tile_end, s->idx_s, s->long_mask, s->long_rows, s->beg_l,
                  s->end_l, s->idx_l,
                  s->chunk_ptr, s->chunk_row, s->chunk_desc, s->val64_s, s->val64_l,
                  s->val32_s, s->val32_l,
                  s->val16_s, s->val16_l,
                  s->part_a, s->part_b, s->done_a, s->done_b, s->gpart_a, s->gpart_b};
  for (void *b : bufs) buf_release(b);
  *s = SideStore();
}

int tile_grid(const SideLayout &lay, int sm_count, int blocks_per_sm) {
  const int w = lay.cta_warps > 0 ? lay.cta_warps : kBlockWarps;
  long long need = ((long long)lay.total_items() + w - 1) / w;
  long long cap = (long long)sm_count * std::max(blocks_per_sm, 1);
  long long g = std::min(need, cap);
  return (int)std::max<long long>(g, 1);
}

void allow_large_smem_setup(int bytes) {
  cudaFuncSetAttribute(k_side_spmv, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_side_spmv_pw<double, double>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_side_spmv_pw<float, float>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_side_spmv_pw<__nv_bfloat16, float>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

static int pw_smem(const SideStore &side, int lowp) {
  return kBlockWarps * side.lay.seg * (lowp ? (int)sizeof(float) : (int)sizeof(double));
}

void side_spmv_pw(cudaStream_t st, const SideStore &side, int lowp, const void *src,
                  const double *in_scale, void *out, double *part, unsigned int *ticket,
                  double *ss, int grid) {
  const int smem = pw_smem(side, lowp);
  const float *sf = (const float *)src;
  float *of = (float *)out;
  if (lowp == 2)
    k_side_spmv_pw<__nv_bfloat16, float><<<grid, kBlockThreads, smem, st>>>(
        side.lay, side.v16, side.wa, sf, in_scale, of, part, ticket, ss);
  else if (lowp == 1)
    k_side_spmv_pw<float, float><<<grid, kBlockThreads, smem, st>>>(
        side.lay, side.v32, side.wa, sf, in_scale, of, part, ticket, ss);
  else
    k_side_spmv_pw<double, double><<<grid, kBlockThreads, smem, st>>>(
        side.lay, side.v64, side.wa, (const double *)src, in_scale, (double *)out, part, ticket,
        ss);
  count_launches(1);
}

// grid of the power-iteration product on `side`: whole resident waves, at most the work items
int side_spmv_pw_grid(const SideStore &side, int lowp, int sm_count) {
  const int smem = pw_smem(side, lowp);
  int b = 0;
  if (lowp == 2)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_side_spmv_pw<__nv_bfloat16, float>,
                                                  kBlockThreads, smem);
  else if (lowp == 1)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_side_spmv_pw<float, float>,
                                                  kBlockThreads, smem);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_side_spmv_pw<double, double>,
                                                  kBlockThreads, smem);
  return tile_grid(side.lay, sm_count, b);
}

void side_spmv(cudaStream_t st, const SideStore &side, const double *src, double *out, int grid) {
  int smem = kBlockWarps * side.lay.seg * (int)sizeof(double);
  k_side_spmv<<<grid, kBlockThreads, smem, st>>>(side.lay, side.v64, side.wa, src, out);
  count_launches(1);
}

void sumsq(cudaStream_t st, int n, const double *x, double *out, double *tmp) {
  k_sumsq_part<<<256, 256, 0, st>>>(n, x, tmp);
  k_sum_final<<<1, 256, 0, st>>>(256, tmp, out);
  count_launches(2);
}

void fill(cudaStream_t st, int n, double v, double *x) {
  k_fill<<<nblocks(n, 256), 256, 0, st>>>(n, v, x);
  count_launches(1);
}

void fill_f32(cudaStream_t st, int n, float v, float *x) {
  k_fill<<<nblocks(n, 256), 256, 0, st>>>(n, v, x);
  count_launches(1);
}

void vmul(cudaStream_t st, int n, const double *a, const double *x, double *y, int div) {
  k_vmul<<<nblocks(n, 256), 256, 0, st>>>(n, a, x, y, div);
  count_launches(1);
}

void vclamp(cudaStream_t st, int n, double *x, const double *l, const double *u) {
  k_vclamp<<<nblocks(n, 256), 256, 0, st>>>(n, x, l, u);
  count_launches(1);
}

}  // namespace rh
