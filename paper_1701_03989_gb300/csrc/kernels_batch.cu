// Many independent systems advancing block by block in lockstep (batched
// solves and the solve server). Each system keeps its own operator, basis,
// x and b; a device table of descriptors (SysDesc) points at them. Work is
// cut into row items of one system each (RowItem: up to 256 rows starting on
// a 32-row slice), so one launch serves every system and adding or retiring
// a system only changes the tables. A kernel reads nothing of the other
// systems, so each system's result is the same alone and in any mix.
#include "ascg_common.cuh"

namespace ascg {
namespace {

__device__ __forceinline__ bool item_row(const RowItem* items, int64_t* row, int* sys) {
  const RowItem it = items[blockIdx.x];
  if ((int)threadIdx.x >= it.nrows) return false;
  *row = it.row0 + threadIdx.x;
  *sys = it.sys;
  return true;
}

// Matrix powers step j in the monomial basis (theta = sigma = 0, gamma = 1;
// eq. (polybasiscg)) for every system q with j < sys_steps[q]: column 2j+2 =
// A column 2j and, while j + 1 < sbar_q, column 2j+3 = A column 2j+1, A = D + O.
//
// Two ways of summing a row, chosen per system (items_by_chain). By chain: one
// warp per 32-row slice and chain (P or R), an item of 64 rows per CTA of 128
// threads; the second warp of a slice finds A in L1. A row's sum is one chain of
// dependent FMAs, 64 cycles each on GB300, so a long row costs its length in
// latency however idle the GPU is: the two chains on two warps halve that, and
// small CTAs spread a small system over more SMs. row_chain keeps two groups of A
// and one of gathers in flight. 8 CTAs per SM (64 registers) beat 7 (72) by 4 %
// and 10 (48, spilling) by 18 %. FP64-bound: 1.71M warp FMAs (10 systems, two
// banded of 117 and 129 entries a row) take 111 us, 0.79 of the FP64 pipe at its
// nominal rate. 32 systems of 1e3..1e5 rows, targets 1e-8 and 1e-12: 236.4 -> 195.1
// ms a batch with the exponents folded in below (one thread per row with both
// chains in 256-row CTAs, and a pass over the bases for the exponents before).
// Such an item records the largest biased exponent of the columns written (and,
// at step 0, of the input columns) for the tensor-core Gram, in place of another
// pass over the basis: one atomic without return per warp, into one of the
// system's kEmaxCopies copies.
//
// Both chains in a thread: A and its indices are read once, for short rows in
// batches that fill the GPU, where the doubled loads are what counts. The
// exponents of such systems take a pass of their own (recording them here, even
// once per CTA, was slower: 140^3, 60 iterations, 29.7 ms against 27.8). In a
// batch that has both kinds (MIXED) such an item is 128 rows of the same kernel;
// a batch that has no other takes mpk_items_both_kernel, 256 rows.
template <bool MIXED>
__global__ void __launch_bounds__(128, 8) mpk_items_kernel(const SysDesc* __restrict__ descs,
                                                           const RowItem* __restrict__ items,
                                                           const int* __restrict__ sys_steps, int j,
                                                           int* __restrict__ emax_all) {
  const RowItem it = items[blockIdx.x];
  const SysDesc d = descs[it.sys];
  const bool chain = !MIXED || it.by_chain;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ch = chain ? warp & 1 : 0, first = kSlice * (chain ? warp >> 1 : warp);
  const bool any = first < it.nrows, on = first + lane < it.nrows;
  const int64_t row = (int64_t)it.row0 + first + lane;
  int64_t b = 0;
  int width = 0;
  double dg = 0.0;
  if (any) {
    const int64_t sl = row >> 5;
    b = d.o_ptr[sl];
    width = (int)((d.o_ptr[sl + 1] - b) >> 5);
    if (on) dg = d.diag[row];
  }
  const double* x = d.Y + (int64_t)(2 * j + ch) * d.ldY;
  pdl_wait(x);  // the step before (its column of Y) and the lanes' tables
  pdl_release();
  const int steps = load_after_wait(sys_steps + it.sys);
  if (!any || j + ch >= steps) return;  // uniform over the warp: no step j, or no R chain in the last one
  const double* v = d.o_val + b + lane;
  const int32_t* c = d.o_col + b + lane;
  const double xi = on ? x[row] : 0.0;
  double t = dg * xi;
  if (MIXED && !chain && j + 1 < steps) {
    const double* r = x + d.ldY;
    double tr = dg * (on ? r[row] : 0.0);
    for (int k = 0; k < width; ++k) {
      const double a = __ldg(v + kSlice * k);
      const int cc = __ldg(c + kSlice * k);
      t = fma(a, __ldca(x + cc), t);
      tr = fma(a, __ldca(r + cc), tr);
    }
    if (on) d.Y[(int64_t)(2 * j + 3) * d.ldY + row] = tr;
  } else {
    t = row_chain(v, c, width, x, t);
  }
  if (on) d.Y[(int64_t)(2 * j + 2 + ch) * d.ldY + row] = t;
  if (!emax_all || !chain) return;
  int* em = emax_all + ((int64_t)it.sys * kEmaxCopies + (blockIdx.x & (kEmaxCopies - 1))) * kMaxW + ch;
  const unsigned e = __reduce_max_sync(0xffffffffu, on ? biased_exp(t) : 0u);
  if (lane == 0) atomicMax(em + 2 * j + 2, (int)e);
  if (j == 0) {
    const unsigned e0 = __reduce_max_sync(0xffffffffu, biased_exp(xi));
    if (lane == 0) atomicMax(em, (int)e0);
  }
}

__global__ void __launch_bounds__(kRowItem) mpk_items_both_kernel(const SysDesc* __restrict__ descs,
                                                                  const RowItem* __restrict__ items,
                                                                  const int* __restrict__ sys_steps, int j) {
  pdl_wait();
  pdl_release();
  int64_t row;
  int q;
  if (!item_row(items, &row, &q)) return;
  const int steps = load_after_wait(sys_steps + q);
  if (j >= steps) return;  // uniform over the CTA
  const SysDesc d = descs[q];
  const double* pj = d.Y + (int64_t)(2 * j) * d.ldY;
  const double* rj = d.Y + (int64_t)(2 * j + 1) * d.ldY;
  const int64_t sl = row >> 5;
  const int l = (int)(row & 31);
  const int64_t b = d.o_ptr[sl];
  const int width = (int)((d.o_ptr[sl + 1] - b) >> 5);
  const double* v = d.o_val + b + l;
  const int32_t* c = d.o_col + b + l;
  const double dg = d.diag[row];
  double tp = dg * pj[row];
  if (j + 1 < steps) {
    double tr = dg * rj[row];
    for (int k = 0; k < width; ++k) {
      const double a = __ldg(v + kSlice * k);
      const int cc = __ldg(c + kSlice * k);
      tp = fma(a, __ldca(pj + cc), tp);
      tr = fma(a, __ldca(rj + cc), tr);
    }
    d.Y[(int64_t)(2 * j + 3) * d.ldY + row] = tr;
  } else {
    for (int k = 0; k < width; ++k) tp = fma(__ldg(v + kSlice * k), __ldca(pj + __ldg(c + kSlice * k)), tp);
  }
  d.Y[(int64_t)(2 * j + 2) * d.ldY + row] = tp;
}

// Residual of the systems with sel[q] != 0: into columns 1 (r) and 0 (p) of Y
// (setup), or into column 2 (true residual at the end).
__global__ void __launch_bounds__(kRowItem) residual_items_kernel(const SysDesc* __restrict__ descs,
                                                                  const RowItem* __restrict__ items,
                                                                  const int* __restrict__ sel, int into_col2) {
  int64_t row;
  int q;
  if (!item_row(items, &row, &q)) return;
  if (!sel[q]) return;
  const SysDesc d = descs[q];
  const int64_t sl = row >> 5;
  const int l = (int)(row & 31);
  const int64_t o = d.o_ptr[sl];
  const int width = (int)((d.o_ptr[sl + 1] - o) >> 5);
  double ax = d.diag[row] * d.x[row];
  for (int k = 0; k < width; ++k)
    ax = fma(__ldg(d.o_val + o + kSlice * k + l), d.x[__ldg(d.o_col + o + kSlice * k + l)], ax);
  const double rr = d.b[row] - ax;
  if (into_col2) {
    d.Y[2 * d.ldY + row] = rr;
  } else {
    d.Y[d.ldY + row] = rr;
    d.Y[row] = rr;
  }
}

// out[q] = sum of squares of a vector of each selected system (one CTA per
// selected system; fixed order: strided thread sums, then a fixed tree).
// which: 0 = b, 1 = Y column 1 (r), 2 = Y column 2.
__global__ void __launch_bounds__(1024) seg_sumsq_kernel(const SysDesc* __restrict__ descs,
                                                         const int* __restrict__ list, int which,
                                                         double* __restrict__ out) {
  const int q = list[blockIdx.x];
  const SysDesc d = descs[q];
  const double* v = which == 0 ? d.b : d.Y + (int64_t)which * d.ldY;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < d.n; i += 1024) s = fma(v[i], v[i], s);
  s = warp_sum(s);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = warp_sum(red[threadIdx.x]);
    if (threadIdx.x == 0) out[q] = s;
  }
}

// x += Y x', r = Y r', p = Y p' (eq. (coords)) for every active system
// (w_q = sys_w[q] > 0); its coordinates sit at coords + q * c_stride as x'[w_q],
// r'[w_q], p'[w_q]. A thread reads its whole row of Y before writing r and p
// into columns 1 and 0.
template <int W>
__global__ void __launch_bounds__(kRowItem) recover_items_kernel(const SysDesc* __restrict__ descs,
                                                                 const RowItem* __restrict__ items,
                                                                 const int* __restrict__ sys_w,
                                                                 const double* __restrict__ coords, int64_t c_stride) {
  pdl_wait();
  pdl_release();
  int64_t row;
  int q;
  if (!item_row(items, &row, &q)) return;
  const int w = load_after_wait(sys_w + q);
  if (w == 0) return;  // uniform over the CTA
  const SysDesc d = descs[q];
  const double* cq = coords + (int64_t)q * c_stride;
  double y[W];
#pragma unroll
  for (int c = 0; c < W; ++c) y[c] = c < w ? d.Y[(int64_t)c * d.ldY + row] : 0.0;
  double sx = 0.0, sr = 0.0, sp = 0.0;
#pragma unroll
  for (int c = 0; c < W; ++c) {
    if (c < w) {
      sx = fma(y[c], __ldca(cq + c), sx);
      sr = fma(y[c], __ldca(cq + w + c), sr);
      sp = fma(y[c], __ldca(cq + 2 * w + c), sp);
    }
  }
  d.x[row] += sx;
  d.Y[d.ldY + row] = sr;
  d.Y[row] = sp;
}

// v[i] in [-1, 1) from a 64-bit mix of (seed, i) (the SplitMix64 finaliser of
// Steele, Lea and Flood, "Fast splittable pseudorandom number generators",
// OOPSLA 2014): synthetic data for the autotuner's timings.
__global__ void fill_uniform_kernel(double* __restrict__ v, int64_t count, uint64_t seed) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = seed + (uint64_t)i * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    v[i] = (double)(int64_t)(z >> 11) * 0x1.0p-52 - 1.0;
  }
}

}  // namespace

cudaError_t launch_fill_uniform(double* v, int64_t count, uint64_t seed, cudaStream_t s) {
  if (count < 1) return cudaSuccess;
  fill_uniform_kernel<<<grid_for(count, 256, 152 * 16), 256, 0, s>>>(v, count, seed);
  return cudaGetLastError();
}

cudaError_t launch_mpk_items(const SysDesc* descs, const RowItem* items, int nitems, const int* sys_steps, int j,
                             bool mixed, int* emax_all, cudaStream_t s) {
  if (nitems < 1) return cudaSuccess;
  if (mixed) return launch_pdl(mpk_items_kernel<true>, nitems, 128, s, descs, items, sys_steps, j, emax_all);
  return launch_pdl(mpk_items_kernel<false>, nitems, 128, s, descs, items, sys_steps, j, emax_all);
}

cudaError_t launch_mpk_items_both(const SysDesc* descs, const RowItem* items, int nitems, const int* sys_steps, int j,
                                  cudaStream_t s) {
  if (nitems < 1) return cudaSuccess;
  return launch_pdl(mpk_items_both_kernel, nitems, kRowItem, s, descs, items, sys_steps, j);
}

cudaError_t launch_residual_items(const SysDesc* descs, const RowItem* items, int nitems, const int* sel,
                                  int into_col2, cudaStream_t s) {
  if (nitems < 1) return cudaSuccess;
  residual_items_kernel<<<nitems, kRowItem, 0, s>>>(descs, items, sel, into_col2);
  return cudaGetLastError();
}

cudaError_t launch_seg_sumsq(const SysDesc* descs, const int* list, int nlist, int which, double* out,
                             cudaStream_t s) {
  if (nlist < 1) return cudaSuccess;
  seg_sumsq_kernel<<<nlist, 1024, 0, s>>>(descs, list, which, out);
  return cudaGetLastError();
}

cudaError_t launch_recover_items(int W, const SysDesc* descs, const RowItem* items, int nitems, const int* sys_w,
                                 const double* coords, int64_t c_stride, cudaStream_t s) {
  if (nitems < 1) return cudaSuccess;
  switch (W) {
#define ASCG_RB(WW)                                                                             \
  case WW:                                                                                      \
    return launch_pdl(recover_items_kernel<WW>, nitems, kRowItem, s, descs, items, sys_w, coords, c_stride);
    ASCG_RB(3) ASCG_RB(5) ASCG_RB(7) ASCG_RB(9) ASCG_RB(11) ASCG_RB(13) ASCG_RB(15) ASCG_RB(17) ASCG_RB(19)
    ASCG_RB(21) ASCG_RB(23) ASCG_RB(25) ASCG_RB(27) ASCG_RB(29) ASCG_RB(31) ASCG_RB(33)
#undef ASCG_RB
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace ascg
