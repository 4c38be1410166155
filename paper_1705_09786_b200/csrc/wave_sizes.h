// Sizes of the encoder's scratch (wave_encode.cu) for a graph whose positions and payload rows are bounded: plain host code, so that the
// arithmetic can be checked without a device.
#pragma once
#include <algorithm>
#include <vector>

#include "wave.h"

namespace wave {

constexpr unsigned long long MAX_SCRATCH_WORDS = 1ull << 28;      // of one encoding warp

// Fills in what depends on the loaded data: key spaces, scratch of an encoding warp, the most entries and steps of an instance.  False
// where the encoder cannot take the data: positions and iterations travel in sixteen bits, and a warp's scratch is at most 1 GB.  All
// sums are 64 bits wide and checked before they are narrowed: a graph of some thousand nodes with one hub passes 2^32 words.
inline bool encoder_sizes(EncModel& E, const std::vector<amp::DevNode>& nodes, const int max_out_degree) {
  using namespace amp;
  constexpr int MOST = 1 << 24;                  // (keeps every product below 2^64)
  if (E.IT > 65535 || max_out_degree > MOST) return false;
  for (auto& h : nodes) if (h.U_in > 65535 || h.U_out > 65535 || h.rows_in > MOST || h.rows_out > MOST) return false;
  unsigned long long w = 0, rows = 64, front = 64;
  const unsigned long long IT = (unsigned long long)E.IT;
  for (int i = 0; i < E.n_nodes; i++) {
    const DevNode& h = nodes[i];
    EncNode& N = E.nodes[i];
    N.U = h.U_in; N.J = 0;
    bool counted = true;
    switch (h.type) {
      case CONCAT: N.U = h.U_out; N.J = h.fn_arg; break;
      case BCAST: case SPLIT: N.J = h.fn_arg; break;
      case GROUP: N.U = h.U_out; N.J = h.rows_out; break;
      case UNGROUP: N.J = h.rows_in; break;
      case FLATMAP: N.J = max_out_degree; break;
      case NPT_LSTM: N.J = 2; break;
      case PHI: case NPT_SUMROWS: break;
      default: counted = false;
    }
    const unsigned long long keys = IT * N.U;
    N.ref_off = (unsigned)w; w += keys * N.J;
    N.cnt_off = (unsigned)w; if (counted) w += keys;
    rows += IT * std::max((unsigned long long)h.U_in * h.rows_in, (unsigned long long)h.U_out * h.rows_out) * (2 + std::max(h.n_succ, h.n_pred));
    if (h.ppt >= 0) { EncPpt& P = E.ppts[h.ppt]; P.U = h.U_in; P.save_off = (unsigned)w; w += keys * 3; front += 3ull * h.U_in; }
    if (w > MAX_SCRATCH_WORDS || rows > MAX_SCRATCH_WORDS) return false;      // (the offsets above fit where this holds)
  }
  const unsigned long long table = (w + 3) & ~3ull, scratch = (table + 12ull * front + 6ull * rows + 2ull * rows + 31) & ~31ull;
  if (scratch > MAX_SCRATCH_WORDS) return false;
  E.table_words = (unsigned)table;
  bool forks = false;
  for (int i = 0; i < E.n_nodes; i++) forks |= nodes[i].type == UNGROUP || nodes[i].type == GROUP || nodes[i].type == FLATMAP;
  E.stack_cap = forks ? 1024 : 256;
  E.front_cap = (unsigned)front; E.row_cap = (unsigned)rows; E.term_cap = (unsigned)(3 * rows);
  unsigned long long messages = 4;
  for (int c = 0; c < E.n_cells; c++) E.bound[c] = 0;
  for (int p = 0; p < E.n_ppts; p++) {
    const DevNode& h = nodes[E.ppts[p].node];
    const unsigned long long b = IT * h.U_in * h.rows_in;          // (at most `rows`)
    for (int k = 0; k < 6; k++) if (E.ppts[p].cell[k] >= 0) E.bound[E.ppts[p].cell[k]] = (unsigned)b;
    messages += 2 * IT * h.U_in;
  }
  E.steps_cap = (unsigned)std::min<unsigned long long>(messages + 4, 60000);
  E.scratch_words = (unsigned)scratch;
  E.near_scratch = (size_t)E.scratch_words * 4 + E.stack_cap * 16 <= 100 * 1024;
  return true;
}

}  // namespace wave
