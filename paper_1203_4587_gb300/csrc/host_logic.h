// Host-side planning logic with no CUDA types, so that it also builds as
// plain C++ for the CPU checks in tests/host_logic_check.cpp.
//
//   fft_factor, fft_stages  the stage radices of the Stockham FFTs (every
//                   transform of the library: rows, columns and time)
//   lpt_work_lists  the per-CTA column lists of the column-inverse kernel
//   plan_tc_cols    image columns that the tensor-core inversion takes at once;
//   plan_tc_pays, block_tc_pays  the sizes from which it takes less time than the other forms
//   mask_rows       the sampled ky rows of each frame of a Cartesian mask
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

namespace recon {

// Radices of an n-point FFT, at most max_stages of them: 4s first, then 2, 3,
// 5 and 7, then the remaining odd factors in increasing order (each done by
// the generic direct stage).  Returns the stage count; the radices multiply
// to n unless n needs more than max_stages stages.
inline int fft_factor(int n, int* radix, int max_stages) {
  int m = n, ns = 0;
  const int pref[] = {4, 2, 3, 5, 7};
  for (int r : pref) {
    while (m % r == 0 && ns < max_stages) { radix[ns++] = r; m /= r; }
  }
  for (int r = 11; m > 1 && ns < max_stages; r += 2) {
    while (m % r == 0) { radix[ns++] = r; m /= r; }
  }
  return ns;
}

// The stages as the kernels run them (fft.cuh): the factors of fft_factor with
// its 4s and 2 regrouped into 8s (fewer passes over shared memory), primes
// first, where no twiddles are due.
inline int fft_stages(int n, int* radix, int max_stages) {
  int f[32], two = 0, ns = 0;
  const int nf = fft_factor(n, f, 32);
  for (int k = nf - 1; k >= 0; --k) {
    if (f[k] == 4) two += 2;
    else if (f[k] == 2) two += 1;
    else if (ns < max_stages) radix[ns++] = f[k];
  }
  while (two > 0 && ns < max_stages) {
    const int b = two == 4 || two == 2 ? 2 : two == 1 ? 1 : 3;
    radix[ns++] = 1 << b;
    two -= b;
  }
  return ns;
}

// Column work lists: column c of slice q (ncols[q] columns, each streaming
// cost[q] bytes) becomes the item (q << 24) | c.  With one slice the columns
// are interleaved (CTA b takes b, b + grid, ...); otherwise they go out by
// longest-processing-time-first to the least-loaded CTA, and each CTA's list
// is then ordered by (slice, column).  CTA b's items are
// work[off[b] .. off[b+1]); work_max is the longest list.  q < 256 and
// c < 2^24.
inline void lpt_work_lists(const std::vector<long long>& cost, const std::vector<int>& ncols, int grid,
                           std::vector<unsigned>& work, std::vector<int>& off, int& work_max) {
  struct Col { long long cost; int q, c; };
  const int n = (int)ncols.size();
  std::vector<Col> cols;
  for (int q = 0; q < n; ++q)
    for (int c = 0; c < ncols[q]; ++c) cols.push_back({cost[q], q, c});
  std::vector<std::vector<std::pair<int, int>>> per(grid);
  if (n == 1) {
    for (size_t k = 0; k < cols.size(); ++k) per[k % grid].push_back({cols[k].q, cols[k].c});
  } else {
    std::stable_sort(cols.begin(), cols.end(), [](const Col& a, const Col& b) { return a.cost > b.cost; });
    using Load = std::pair<long long, int>;
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> pq;
    for (int b = 0; b < grid; ++b) pq.push({0, b});
    for (const Col& c : cols) {
      Load l = pq.top();
      pq.pop();
      per[l.second].push_back({c.q, c.c});
      pq.push({l.first + c.cost, l.second});
    }
    for (auto& v : per) std::sort(v.begin(), v.end());
  }
  work.clear();
  off.assign(grid + 1, 0);
  work_max = 0;
  for (int b = 0; b < grid; ++b) {
    off[b] = (int)work.size();
    for (const auto& w : per[b]) work.push_back(((unsigned)w.first << 24) | (unsigned)w.second);
    work_max = std::max(work_max, (int)per[b].size());
  }
  off[grid] = (int)work.size();
}

// Image columns (of Nt matrices each) a chunk of the tensor-core inversion: about 4 matrices an SM
// (whole waves of every kernel), more while that is under 256 MB of scratch; but no more scratch
// than 600 MB or a quarter more than the inverses it makes, whichever is more (a slab of 19 columns of
// 256 x 32 frames makes 164 MB and would take 2.2 GB).  Without the quarter a plan of 256 x 256 x 32 takes
// chunks of 18 columns instead of 19, one chunk more, and 50.4 ms instead of 48.3.
inline int plan_tc_cols(int Nx, int Nt, int sms, double matrix_bytes, double inverse_bytes) {
  const double most = std::max(6e8, 1.25 * inverse_bytes) / matrix_bytes;
  const double mats = std::min(most, std::max(4.0 * sms, 2.56e8 / matrix_bytes));
  return std::max(1, std::min(Nx, (int)(mats / Nt)));
}

// Whether the tensor-core inversion pays for a plan of mats = Nx Nt blocks: its dozen launches, scratch
// allocation and second synchronisation cost 100 to 300 us, which small sizes only earn with many
// blocks.  recon_plan_set_mu, double-float sweep and this, us (152 SMs):
//   Ny = 48    64 blocks 387 / 467, 608 647 / 728, 2432 1596 / 1692: never
//   Ny = 56   304 blocks 541 / 584, 608 784 / 723, 2432 2100 / 1695: four blocks an SM
//   Ny = 64    16 blocks 275 / 445, 152 448 / 490, 304 595 / 571, 608 872 / 725: two an SM
//   Ny = 80     4 blocks 376 / 472, 16 536 / 491, 152 588 / 588, 608 1320 / 1040: 16
//   Ny = 96     4 blocks 515 / 474, 152 724 / 584, 2432 6351 / 2603: always
inline bool plan_tc_pays(int Ny, long long mats, int sms) {
  if (Ny >= 96) return true;
  if (Ny >= 80) return mats >= 16;
  return Ny >= 56 && mats >= (Ny >= 64 ? 2ll : 4ll) * sms;
}

// The same for nblk separate blocks that run `chunk` at a time (a chunk of 16 MiB costs 115 us up to
// Ny = 64 and 150 to 96, whatever its blocks' own size), against as many FP64 workspaces as there is
// room for.  FP64 and this, us:
//   Ny = 33    70 blocks 286 / 172, 130 279 / 290, 1024 844 / 1716: one chunk
//   Ny = 40   130 blocks 379 / 288, 256 460 / 513: two
//   Ny = 44   130 blocks 432 / 288, 512 790 / 951: three
//   Ny = 48   130 blocks 484 / 288, 2048 3305 / 3247: any
//   Ny = 65   256 blocks 1809 / 1271, 512 2803 / 2456, 1024 4794 / 4826, 2048 8740 / 9617: 20 chunks
//   Ny = 72  2048 blocks 13362 / 9692: any
inline bool block_tc_pays(int Ny, int nblk, int chunk) {
  if (Ny < 33 || chunk < 1) return false;
  const int chunks = (nblk - 1) / chunk + 1;
  if (Ny < 48) return chunks <= (Ny >= 44 ? 3 : Ny >= 36 ? 2 : 1);
  return Ny < 65 || Ny >= 70 || chunks <= 20;
}

// Sampled ky rows of a Cartesian ky-t mask (Section II-A: every kx of a
// sampled row is sampled).  mask is [Nt][Ny] (full = false) or [Nt][Ny][Nx]
// (full = true, and then each row must be constant along kx).  Frame t's
// rows, in increasing ky, are rows[rowoff[t] .. rowoff[t+1]).  Returns the
// largest per-frame count, or -1 with (*bad_t, *bad_j) the first row that
// differs along kx.
inline int mask_rows(const uint8_t* mask, int Nt, int Ny, int Nx, bool full, std::vector<int>& rows,
                     std::vector<int>& rowoff, int* bad_t, int* bad_j) {
  rows.clear();
  rowoff.assign(Nt + 1, 0);
  int maxm = 0;
  for (int t = 0; t < Nt; ++t) {
    for (int j = 0; j < Ny; ++j) {
      bool on;
      if (full) {
        const uint8_t* rowp = &mask[((size_t)t * Ny + j) * Nx];
        on = rowp[0] != 0;
        for (int i = 1; i < Nx; ++i) {
          if ((rowp[i] != 0) != on) {
            *bad_t = t;
            *bad_j = j;
            return -1;
          }
        }
      } else {
        on = mask[(size_t)t * Ny + j] != 0;
      }
      if (on) rows.push_back(j);
    }
    rowoff[t + 1] = (int)rows.size();
    maxm = std::max(maxm, rowoff[t + 1] - rowoff[t]);
  }
  return maxm;
}

}  // namespace recon
