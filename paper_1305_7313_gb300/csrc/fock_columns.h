// fock_columns.h — host side of the column sets (ColumnSet): which columns
// (k2, k3) of a spectrum hold something, in the forms the kernels read.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "fock_internal.h"

namespace fockx {
namespace columns {

struct HostColumns {
  std::vector<int> ncol;    // [N] per k3: k2 < (ncol & 0xffff) or k2 >= N - (ncol >> 16)
  std::vector<int> kept;    // (k2 << 16) | k3, rows outer
  std::vector<int> rowpos;  // [2][N] places of the kept rows in a transformed plane, ascending, per tiling
  std::vector<int> lines;   // column map: (k2 << 16) | (self << 15) | k3, or -1, padded to whole CTAs
  int ncta = 1;
  int row_lo = 0, row_hi = 0, col_lo = 1, col_hi = 0;
};

// The smallest set of columns that holds the marked ones (mark[k2 N + k3]) and
// keeps two runs k2 < up, k2 >= N - dn of every column k3.  mirror: the set is
// also closed under (k2, k3) -> (-k2, -k3), and the column map lists one line
// of each mirror pair, per_cta pairs per CTA; otherwise it lists every line.
// row_place(tile, k2): the row of a transformed plane that holds frequency k2.
inline void build(int n, const std::vector<unsigned char>& mark, bool mirror, int per_cta,
                  int (*row_place)(int tile, int k2), HostColumns& out) {
  out.ncol.assign(n, 0);
  const int khi = mirror ? n / 2 + 1 : n;
  for (int k3 = 0; k3 < khi; ++k3) {
    int up = 0, dn = 0;
    for (int k2 = 0; k2 < n; ++k2)
      if (mark[(size_t)k2 * n + k3]) {
        if (2 * k2 <= n) up = std::max(up, k2 + 1);
        else dn = std::max(dn, n - k2);
      }
    if (up == 0 && dn == 0) continue;
    if (mirror) {
      // the mirror column n - k3 keeps the mirror images; columns 0 and N/2 are
      // their own mirror images: up = dn + 1 (k2 = 0 has no partner)
      up = std::max(up, 1);
      if (k3 == 0 || 2 * k3 == n) {
        up = std::max(up, dn + 1);
        dn = up - 1;
      } else {
        out.ncol[n - k3] = (dn + 1) | ((up - 1) << 16);
      }
    }
    out.ncol[k3] = up | (dn << 16);
  }
  const auto keeps = [&](int k2, int k3) {
    return k2 < (out.ncol[k3] & 0xffff) || k2 >= n - (out.ncol[k3] >> 16);
  };
  out.col_lo = 1;
  out.col_hi = 0;
  for (int k3 = 0; k3 < n; ++k3) {
    out.row_lo = std::max(out.row_lo, out.ncol[k3] & 0xffff);
    out.row_hi = std::max(out.row_hi, out.ncol[k3] >> 16);
    if (out.ncol[k3] == 0) continue;
    if (2 * k3 <= n) out.col_lo = std::max(out.col_lo, k3 + 1);
    else out.col_hi = std::max(out.col_hi, n - k3);
  }
  out.row_lo = std::max(out.row_lo, 1);
  if (out.row_lo + out.row_hi >= n) {
    out.row_lo = n;
    out.row_hi = 0;
  }
  if (out.col_lo + out.col_hi >= n) {
    out.col_lo = n;
    out.col_hi = 0;
  }
  for (int t = 0; t < 2; ++t) {
    std::vector<int> rows;
    for (int k2 = 0; k2 < n; ++k2)
      if (k2 < out.row_lo || k2 >= n - out.row_hi) rows.push_back(row_place(t, k2));
    std::sort(rows.begin(), rows.end());
    rows.resize(n, 0);
    out.rowpos.insert(out.rowpos.end(), rows.begin(), rows.end());
  }
  for (int k2 = 0; k2 < n; ++k2)
    for (int k3 = 0; k3 < n; ++k3) {
      if (!keeps(k2, k3)) continue;
      out.kept.push_back((k2 << 16) | k3);
      const int m2 = (n - k2) % n, m3 = (n - k3) % n;
      const bool self = mirror && m2 == k2 && m3 == k3;
      // of a mirror pair the line with 0 < k3 < N/2, or the one with k2 <= N/2
      if (!mirror || k3 < m3 || (k3 == m3 && k2 <= m2)) out.lines.push_back((k2 << 16) | (self ? 1 << 15 : 0) | k3);
    }
  out.ncta = std::max(1, (int)((out.lines.size() + per_cta - 1) / per_cta));
  out.lines.resize((size_t)out.ncta * per_cta, -1);
}

// The coefficient map of a sphere (Miller indices, 3 per coefficient): entry
// (cta N + k1) nl + slot is the position of the coefficient at (k1, k2, k3) of
// the CTA's line in that slot, or -1.  Slots [0, per_cta) hold the column map's
// lines; with mirror images, slots [per_cta, 2 per_cta) hold those of the same
// pairs.
template <class Int>
inline std::vector<int> coefficient_map(int n, const HostColumns& c, int per_cta, bool mirror, const Int* miller,
                                        size_t npw) {
  std::vector<int> at((size_t)n * n * n, -1);
  const auto wrap = [n](int m) { return ((m % n) + n) % n; };
  for (size_t g = 0; g < npw; ++g)
    at[((size_t)wrap(miller[3 * g]) * n + wrap(miller[3 * g + 1])) * n + wrap(miller[3 * g + 2])] = (int)g;
  const int nl = mirror ? 2 * per_cta : per_cta;
  std::vector<int> map((size_t)c.ncta * n * nl, -1);
  for (int cta = 0; cta < c.ncta; ++cta)
    for (int s = 0; s < nl; ++s) {
      const int code = c.lines[(size_t)cta * per_cta + s % per_cta];
      if (code < 0) continue;
      int k2 = code >> 16, k3 = code & 0x7fff;
      if (s >= per_cta) {
        k2 = (n - k2) % n;
        k3 = (n - k3) % n;
      }
      for (int k1 = 0; k1 < n; ++k1)
        map[((size_t)cta * n + k1) * nl + s] = at[((size_t)k1 * n + k2) * n + k3];
    }
  return map;
}

// The set on the device: one buffer (*buf, the caller frees it) for all its lists.
inline cudaError_t upload(const HostColumns& c, const std::vector<int>& coef, int** buf, ColumnSet* set,
                          int64_t* bytes) {
  std::vector<int> all;
  const std::vector<int>* parts[] = {&c.ncol, &c.lines, &c.rowpos, &c.kept, &coef};
  size_t at[5];
  for (int k = 0; k < 5; ++k) {
    at[k] = all.size();
    all.insert(all.end(), parts[k]->begin(), parts[k]->end());
  }
  *bytes += (int64_t)(sizeof(int) * all.size());
  cudaError_t e = cudaMalloc((void**)buf, sizeof(int) * all.size());
  if (e == cudaSuccess) e = cudaMemcpy(*buf, all.data(), sizeof(int) * all.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  set->ncol = *buf + at[0];
  set->lines = *buf + at[1];
  set->rowpos = *buf + at[2];
  set->kept = *buf + at[3];
  set->coef = coef.empty() ? nullptr : *buf + at[4];
  set->ncta = c.ncta;
  set->row_lo = c.row_lo;
  set->row_hi = c.row_hi;
  set->col_lo = c.col_lo;
  set->col_hi = c.col_hi;
  set->nkept = (int)c.kept.size();
  return cudaSuccess;
}

}  // namespace columns
}  // namespace fockx
