// Order of the entries of 8 consecutive rows of a hopping table against shared-memory bank conflicts,
// by one thread: in the row kernels the lanes of rows 8m .. 8m+7 gather 16-byte words [source]
// together at every slot, and such a load takes one shared-memory wavefront when the sources' indices
// mod 8 differ.  Per slot, a maximum matching of the rows that still have entries to the eight
// residues (augmenting paths; rows with more remaining entries first, each row trying its most
// frequent residues first) picks one entry per matched row; unmatched rows take their first remaining
// entry.  Every row keeps its entry set, so only the order of the additions changes.
// On the host this was most of the creation of a large cluster: 48.2 ms for 12,870 rows (4x4), 6.3 ms for
// 3,432 (2x7); the creation takes 1.35 and 0.68 ms with it here.
#pragma once

#include "ed_common.cuh"

namespace ed {

constexpr int kOrderWords = kMaxHops / 64;

// put(slot, row in the group, entry) for every entry of rows r0 .. r0 + nr - 1 (nr <= 8).
template <typename Put>
__device__ void bank_order_group(const int32_t* __restrict__ ptr, const uint32_t* __restrict__ ent, int64_t r0, int nr, Put&& put) {
  unsigned long long left[8][kOrderWords];  // bit i: entry ptr[row] + i is still to place
  unsigned long long res[8];                // entries left per residue, a byte each
  int nleft[8];
  for (int i = 0; i < 8; ++i) {
    for (int w = 0; w < kOrderWords; ++w) left[i][w] = 0ull;
    res[i] = 0ull;
    nleft[i] = 0;
    if (i >= nr) continue;
    const int32_t p0 = ptr[r0 + i], n = ptr[r0 + i + 1] - p0;
    for (int k = 0; k < n; ++k) {
      left[i][k >> 6] |= 1ull << (k & 63);
      res[i] += 1ull << (8 * (ent_col(ent[p0 + k]) & 7u));
    }
    nleft[i] = n;
  }
  for (int slot = 0;; ++slot) {
    int order[8], na = 0;
    for (int i = 0; i < nr; ++i) {  // stable insertion by remaining entries, most first
      if (nleft[i] == 0) continue;
      int j = na++;
      while (j > 0 && nleft[order[j - 1]] < nleft[i]) {
        order[j] = order[j - 1];
        --j;
      }
      order[j] = i;
    }
    if (na == 0) break;
    int owner[8];
    for (int b = 0; b < 8; ++b) owner[b] = -1;
    for (int o = 0; o < na; ++o) {
      unsigned seen = 0u;
      int row[9], bank[9], depth = 0;
      row[0] = order[o];
      while (depth >= 0) {
        int r = -1, best = 0;
        for (int b = 0; b < 8; ++b) {
          const int c = (int)(res[row[depth]] >> (8 * b) & 0xffull);
          if (!(seen >> b & 1u) && c > best) {
            best = c;
            r = b;
          }
        }
        if (r < 0) {
          --depth;
          continue;
        }
        seen |= 1u << r;
        bank[depth] = r;
        if (owner[r] < 0) {
          for (int d = depth; d >= 0; --d) owner[bank[d]] = row[d];
          break;
        }
        row[depth + 1] = owner[r];
        ++depth;
      }
    }
    int res_of[8];
    for (int i = 0; i < 8; ++i) res_of[i] = -1;
    for (int b = 0; b < 8; ++b)
      if (owner[b] >= 0) res_of[owner[b]] = b;
    for (int o = 0; o < na; ++o) {
      const int i = order[o];
      const int32_t p0 = ptr[r0 + i];
      int pick = -1, first = -1;
      for (int w = 0; w < kOrderWords && pick < 0; ++w) {
        unsigned long long m = left[i][w];
        while (m) {
          const int k = w * 64 + __ffsll((long long)m) - 1;
          m &= m - 1ull;
          if (first < 0) first = k;
          if (res_of[i] < 0 || (int)(ent_col(ent[p0 + k]) & 7u) == res_of[i]) {
            pick = k;
            break;
          }
        }
      }
      if (pick < 0) pick = first;
      const uint32_t e = ent[p0 + pick];
      left[i][pick >> 6] &= ~(1ull << (pick & 63));
      res[i] -= 1ull << (8 * (ent_col(e) & 7u));
      --nleft[i];
      put(slot, i, e);
    }
  }
}

}  // namespace ed
