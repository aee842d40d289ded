// Work lists of the preconditioner's CSR row kernel and block-solve kernel,
// planned on the host from the matrix structure and the V_e block sizes.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

#include "sparse.h"

namespace dg {

// Row tiers of the CSR row kernel for one matrix: rows of more than
// kCsrCtaRow entries take a CTA each, rows of more than long_min entries a
// warp each (both lists longest first, ties in row order), the rest `group`
// lanes each.
struct CsrTierPlan {
  int group = 1;
  int long_min = 0;
  std::vector<int32_t> cta, warp;
};
CsrTierPlan plan_csr_tiers(const Csr& C);

// Work units of the V_e block solves (4 ints per unit), largest blocks first:
// blocks of more than 16 nodes give one unit per 32-row panel,
// {slot of the block's first node, d, first row, 0}, with ubase = the offset
// of the panel's first row in the inverses; blocks of at most W = 4, 8 or 16
// nodes (W the smallest of these that holds d) are packed 32 / W to a unit,
// {index of the first packed block, count, 0, W}, and listed in brec as
// {slot, d, inverse offset low 32 bits, high 32 bits} (ubase = 0).
void plan_block_units(const std::vector<int32_t>& dims, const std::vector<int32_t>& slot,
                      const std::vector<int64_t>& inv_off, std::vector<int32_t>& unit,
                      std::vector<int64_t>& ubase, std::vector<int32_t>& brec);

// A CSR matrix cut into slices for the row kernel.  A row of length len takes
// `lanes` lanes (a power of two up to 32, the smallest with at most `rounds`
// entries per lane) and a slice holds 32 / lanes rows of one width and one
// number of rounds, in row order; entry j of a row is read by lane j mod lanes
// in round j / lanes, so that every round of a slice is 32 consecutive entries.
// rounds is the largest of 16, 8, 4 that still gives half the GPU's threads a
// lane; rows of more than 128 * rounds entries or more than kCsrCtaRow make
// slices of 256 lanes.
struct SlicePlan {
  std::vector<int32_t> hdr;   // 4 per slice, see DevSlices
  std::vector<int32_t> row;
  int n_cta = 0, n_warp = 0;
  int64_t entries = 0;        // padded entries (a multiple of 32)
};
SlicePlan plan_slices(const Csr& C);
// columns and values of the slices' entries (-1 / 0 where there is none), each
// S.entries long, every one of them written.  Large matrices on several threads:
// a batch of 72 instances (37M entries) spent 195 ms of its 1.02 s here on one.
template <typename T>
void fill_slices(const Csr& C, const SlicePlan& S, int32_t* idx, T* val) {
  const int n = S.n_cta + S.n_warp;
  auto fill = [&](int s0, int s1) {
    for (int s = s0; s < s1; ++s) {
      const int32_t* h = &S.hdr[4 * (size_t)s];
      const int lanes = h[2], width = s < S.n_cta ? 256 : 32;
      const int64_t e0 = 32 * (int64_t)h[0], e1 = e0 + (int64_t)h[1] * width;
      std::fill(idx + e0, idx + e1, -1);
      std::fill(val + e0, val + e1, T(0));
      for (int r = 0; r < width / lanes; ++r) {
        const int32_t row = S.row[h[3] + r];
        if (row < 0) continue;
        const int64_t b = C.ptr[row], len = C.ptr[row + 1] - b;
        int64_t e = e0 + r * lanes;
        for (int64_t j = 0; j < len; j += lanes, e += width) {   // a round
          const int64_t m = len - j < lanes ? len - j : lanes;
          for (int64_t u = 0; u < m; ++u) {
            idx[e + u] = C.idx[b + j + u];
            val[e + u] = (T)C.val[b + j + u];
          }
        }
      }
    }
  };
  const int parts = (int)std::min<int64_t>(64, S.entries >> 17);
  if (parts < 2) {
    fill(0, n);
    return;
  }
  // parts of about equal numbers of entries; slices lie one after another
  std::vector<int> cut(parts + 1, n);
  cut[0] = 0;
  for (int k = 1, s = 0; k < parts; ++k) {
    while (s < n && 32 * (int64_t)S.hdr[4 * (size_t)s] < S.entries * k / parts) ++s;
    cut[k] = s;
  }
  on_threads(parts, [&](int k) { fill(cut[k], cut[k + 1]); });
}

}  // namespace dg
