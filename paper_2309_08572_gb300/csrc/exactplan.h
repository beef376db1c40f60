// Plan of the exact-slice products (tcgemm.cu): how their stages are dealt out to CTAs and how K
// is cut into pieces whose operands and parts fit a workspace.  Plain C++: the arithmetic runs in
// tests without a GPU.
#pragma once
#include <stddef.h>

#include <algorithm>

namespace mpdo {

constexpr int kExactRows = 128;   // output tile: rows ...
constexpr int kExactCols = 64;    // ... and real columns
constexpr int kExactK = 32;       // K terms of a stage
constexpr int kExactSlices = 6;   // slices per operand
constexpr long kExactPart = (long)kExactRows * kExactCols;   // entries of a CTA's part of a tile
constexpr long kExactPartBytes = kExactPart * 16;            // two 64-bit sums each
constexpr long kExactSms = 152;
constexpr int kExactFusedPackK = 256;   // up to here exponents and packing are one launch

struct ExactPlan {
  int tiles, nst, ctas;
  long per, total;   // stages of a CTA, of all tiles of the batch
  bool parts;        // ranges end within tiles
};
// How many stages a CTA takes: whole tiles, or (may_split) an equal share of the stages (at least
// four) where that is less on the busiest SM, counting 4 stages' time for a CTA's prologue and last
// drain, one for a tile's output and 10 for the parts and the launch that adds them.
inline ExactPlan exact_plan(long m, long n, long kc, int batch, bool gram, bool may_split = true) {
  ExactPlan p;
  const long mt = (m + kExactRows - 1) / kExactRows, nt = (2 * n + kExactCols - 1) / kExactCols;
  long tiles = mt * nt;
  if (gram) {
    tiles = 0;
    for (long i = 0; i < mt; ++i) tiles += nt - i * (kExactRows / (kExactCols / 2));
  }
  p.tiles = (int)tiles;
  p.nst = (int)((2 * kc + kExactK - 1) / kExactK);
  p.total = tiles * batch * p.nst;
  const long whole = (tiles * batch + kExactSms - 1) / kExactSms;
  const long ctas = std::min(kExactSms, std::max(1L, p.total / 4));
  const long share = (p.total + ctas - 1) / ctas;
  p.parts = may_split && share + share / p.nst + 10 < whole * p.nst + whole;
  p.per = std::max(1L, p.parts ? share : whole * p.nst);   // 1: no tiles at all
  p.ctas = (int)((p.total + p.per - 1) / p.per);
  return p;
}

inline size_t exact_align(size_t bytes) { return (bytes + 255) & ~(size_t)255; }
// K terms of a slice's segment in a packed row
inline long exact_ldk(long kc) { return (2 * kc + kExactK - 1) / kExactK * kExactK; }
// Workspace of a piece of kc terms: the packed operands and exponents ...
inline size_t exact_operand_bytes(long m, long n, long kc, int batch, bool gram) {
  const size_t row = (size_t)batch * kExactSlices * exact_ldk(kc) * 2;
  return (gram ? 0 : exact_align(m * row)) + exact_align(2 * n * row) +
         exact_align((size_t)batch * (m + n) * sizeof(int)) + 256;
}
// ... and behind them the parts of its plan.
inline size_t exact_part_bytes(const ExactPlan& p) {
  return p.parts ? (size_t)p.ctas * 2 * kExactPartBytes : 0;
}
// The plan of a piece in a workspace: shares of tiles only where their parts fit.  A shorter piece
// can need more of them than a longer one (the CTAs are total / per rounded up), so every piece is
// planned against the workspace itself.
inline ExactPlan exact_piece_plan(long m, long n, long kc, int batch, bool gram, size_t ws) {
  const ExactPlan p = exact_plan(m, n, kc, batch, gram);
  if (exact_operand_bytes(m, n, kc, batch, gram) + exact_part_bytes(p) <= ws) return p;
  return exact_plan(m, n, kc, batch, gram, false);
}
// K terms of a piece, a multiple of 64 unless it is all of K: the fewest equal pieces that fit with
// the parts they want; pieces of 64 may go without.  0: the workspace is too small.
inline long exact_piece(long m, long n, long k, int batch, bool gram, size_t ws) {
  // fewer cannot hold the operands alone
  const long least = (long)(exact_operand_bytes(m, n, k, batch, gram) / std::max<size_t>(ws, 1));
  for (long pieces = std::max(1L, std::min(least, (k + 63) / 64));; ++pieces) {
    const long kc = pieces == 1 ? k : (k + 64 * pieces - 1) / (64 * pieces) * 64;
    const size_t operands = exact_operand_bytes(m, n, kc, batch, gram);
    if (operands + exact_part_bytes(exact_plan(m, n, kc, batch, gram)) <= ws) return kc;
    if (kc <= 64) return operands <= ws ? kc : 0;
  }
}
// Workspace with which a product runs in pieces of up to 4096 terms, each with the parts it wants.
// gram: as the product will be planned -- a Gram has half of the tiles, which may be too few to go
// round whole and then takes up to 40 MB of parts where the general product of its size takes none
// (768 columns, 1024 rows: four pieces in the general product's workspace, one in its own).
inline size_t exact_ws_bytes(long m, long n, long k, int batch, bool gram) {
  const long pieces = std::max(1L, (k + 4095) / 4096);
  const long kc = pieces == 1 ? k : (k + 64 * pieces - 1) / (64 * pieces) * 64;
  size_t ws = 0;
  for (const long kn : {kc, k - (k - 1) / kc * kc})
    ws = std::max(ws, exact_operand_bytes(m, n, kn, batch, gram) +
                          exact_part_bytes(exact_plan(m, n, kn, batch, gram)));
  return ws;
}

// Time of an exact product against the same product on the FP64 CUDA cores.  The slice kernel
// costs a fixed part (exponents, packing, output) and its stages on the busiest SM, 1.4 us each;
// FP64 runs at 304 FMA per clock over the chip.  Both sides as measured: the Gram 41 x 41 x 1968 takes
// 25 us in FP64 and 36 us plus its packing in slices, the Gram 400 x 400 x 5043 2.6 ms and 74 us.
inline bool exact_faster(long m, long n, long k, int batch, bool gram) {
  const ExactPlan p = exact_plan(m, n, k, batch, gram);
  const double elems = (double)batch * k * ((gram ? 0 : m) + 2.0 * n);   // packed complex entries
  const double tc = (k <= kExactFusedPackK ? 12.0 : 24.0) + (p.parts ? 8.0 : 0.0) +
                    1.4 * (p.per + 4 + p.per / p.nst) + elems * 24.0 / 3.0e6;
  const double fp64 = 8.0 + 1.2 * 4.0 * m * n * (double)k * batch * (gram ? 0.5 : 1.0) / (304.0 * 2.0e3);
  return tc < fp64;
}
// Which products with FP64 results run as slices: those of min_macs complex multiply-adds with both
// sides of at least 16, where that is estimated faster, or (forced: the caller has set the threshold)
// whatever the estimate.
struct ExactRoute {
  double min_macs;
  bool forced;
  bool takes(long m, long n, long k, int batch, bool gram) const {
    return m >= 16 && n >= 16 && k >= 1 && (double)m * n * k * batch >= min_macs &&
           (forced || exact_faster(m, n, k, batch, gram));
  }
};

}  // namespace mpdo
