// Rules that choose between kernels by sizes: host code only, with the measured
// sides beside each line.
#pragma once

#include <cstdint>

namespace ascg {

// Rows of a batch, and how long they are (entries of O per row, padding included).
struct BatchRows {
  int64_t rows = 0;
  double mean_len = 0.0, max_len = 0.0;  // over the rows, and of the system with the longest
};

// Whether a batched matrix powers step sums the rows of a system (row_len entries
// on average) with a warp per slice and chain, or both chains in a thread. By chain
// halves a row's dependent FMAs and keeps more loads in flight, which counts for
// long rows and while the GPU is not full; it reads A twice (through L1), which
// counts for short rows once it is. 60 iterations, s = 10, ms, all by chain / all
// both in a thread:
//   2D Poisson (4 a row)  362^2 3.66 / 3.95, 512^2 5.02 / 4.82, 1024^2 13.5 / 12.3,
//                         16 x 180^2 7.74 / 7.28, 10 x 300^2 11.3 / 10.0
//   3D Poisson (6)        50^3 3.46 / 3.67, 64^3 5.09 / 4.84, 100^3 13.85 / 12.27
//   banded, 8 a row       131072 4.67 / 5.20, 262144 6.71 / 6.64, 750000 14.9 / 13.4
//   banded, 12 a row      200000 6.54 / 6.91, 400000 9.85 / 10.09, 600000 14.5 / 13.3
//   banded, 20 a row      200000 7.75 / 8.50, 400000 13.07 / 12.88, 600000 17.7 / 16.9
//   banded, 32 a row      400000 16.59 / 16.64, 1000000 34.2 / 34.0
//   banded, 48 a row      400000 21.0 / 21.6, 1000000 44.5 / 45.4
// Each system by its own rows in one launch, where a few long rows stand beside
// many short ones (mean at most 8): 1000^2 and banded 5000 of 40 a row 13.6 against
// 14.4 / 15.0 ms, 90^3 and banded 3000 of 100 a row 11.7 against 12.5 / 16.2. Where
// long rows are a larger part, the FP64 pipe sets the time and hides the doubled
// loads: 600^2, 80^3 and banded 100000 of 60 a row (mean 10.8) 17.9 by chain, 18.3
// each by its own; 16 served requests (mean about 25) 338 and 355. From 2^20 rows
// everything is both in a thread, in system order, which mixes FP64-bound with
// HBM-bound rows (256 systems of 1e3..2e5 rows 2.61 s; each by its own 2.94).
inline bool items_by_chain(const BatchRows& b, double row_len) {
  if (b.rows >= (int64_t)1 << 20) return false;
  if (b.max_len >= 40.0 && b.mean_len > 8.0) return true;
  return row_len >= 40.0 || b.rows < 196608 || (row_len >= 7.0 && b.rows <= 400000);
}

// Whether classical CG's product sums its rows with pipelined loads (row_chain) or
// an entry at a time, with A kept in L2 up to 32 MiB of values and columns and
// streamed past it above. Pipelined hides the gathers' latency but holds four CTAs
// of 256 rows per SM, and keeps A in L2. us for 60 iterations, an entry at a time /
// pipelined, by rows and entries a row:
//   20000   13 1206 / 1166, 81 1859 / 1497     40000   13 1266 / 1268, 81 2759 / 1859
//   70000   13 1351 / 1395, 49 2217 / 1666     90000   21 1484 / 1530, 33 1870 / 1666
//   100000  33 1951 / 1845, 201 7164 / 4924    110000  21 1486 / 1837, 61 2407 / 2619
//   116000  61 2872 / 2583                     130000  21 1660 / 1879, 81 3868 / 3067
//   150000  33 2000 / 2122, 49 2634 / 2468     160000  21 2449 / 1995, 81 4353 / 4093
//   175000  49 3613 / 3189, 61 3794 / 3850     200000  33 3270 / 2756, 49 3451 / 3693
//   230000  33 3242 / 2844, 49 3519 / 3746     262144  21 2665 / 2482, 33 2929 / 3159
// Up to 50000 rows latency is all. To four CTAs per SM (155648 rows) an entry at a
// time is better where A stays in L2, also streamed up to 80 MiB once there are
// more than 102400 rows. Beyond, pipelined is better as long as A, which it reads
// from L2, and what the iteration streams through it fit in its 129 MB.
inline bool cg_rows_pipelined(int64_t n, int64_t nnz) {
  if (nnz < 12 * n || n > 262144) return false;
  const int64_t a = 12 * nnz, mib = (int64_t)1 << 20;
  if (n <= 50000) return true;
  if (n <= 155648) return a > 32 * mib && (n <= 102400 || a >= 80 * mib);
  return a + 128 * n <= 128000000 || (n <= 163840 && a >= 80 * mib);
}

}  // namespace ascg
