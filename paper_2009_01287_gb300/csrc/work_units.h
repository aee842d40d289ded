// Work lists of the preconditioner's CSR row kernel and block-solve kernel,
// planned on the host from the matrix structure and the V_e block sizes.
#pragma once

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
// columns and values of the slices' entries (-1 / 0 where there is none)
template <typename T>
void fill_slices(const Csr& C, const SlicePlan& S, std::vector<int32_t>& idx, std::vector<T>& val) {
  idx.assign(S.entries, -1);
  val.assign(S.entries, T(0));
  for (int s = 0; s < S.n_cta + S.n_warp; ++s) {
    const int32_t* h = &S.hdr[4 * (size_t)s];
    const int lanes = h[2], width = s < S.n_cta ? 256 : 32;
    for (int r = 0; r < width / lanes; ++r) {
      const int32_t row = S.row[h[3] + r];
      if (row < 0) continue;
      const int64_t b = C.ptr[row], len = C.ptr[row + 1] - b;
      int64_t e = 32 * (int64_t)h[0] + r * lanes;
      for (int64_t j = 0; j < len; j += lanes, e += width) {   // a round
        const int64_t n = len - j < lanes ? len - j : lanes;
        for (int64_t u = 0; u < n; ++u) {
          idx[e + u] = C.idx[b + j + u];
          val[e + u] = (T)C.val[b + j + u];
        }
      }
    }
  }
}

}  // namespace dg
