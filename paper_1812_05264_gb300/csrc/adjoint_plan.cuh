// Scratch panels of the doubled adjoint: which y_k are stored, and how many ybar panels stand beside them.  Host code
// without CUDA.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstddef>

namespace tbk {

constexpr int SDW = 4;  // steps of an outer-product window

struct AdjointPlan {
  int npan = 0;             // y_1 .. y_npan
  size_t panel = 0;         // bytes
  bool windowed = false;    // outer products of SDW steps together
  bool batch = false;       // a batch also keeps its probe panel
  int defer = 0;            // outer products of so many steps after them (0: inside each step)
  int seg = 1;              // steps of a segment: npan where all y_k are stored
  size_t prefix_tail = 0;   // bytes of a batch's compact panels y_0 .. y_{npan+1}, where it stores those; else 0

  // ybar_j lives in ring slot j mod nb(): the two of the recurrence, and the ones that outer products wait for
  int nb() const { return windowed ? SDW + 2 : (defer > 1 ? defer + 1 : 2); }
  int nx() const { return nb() + (batch ? 1 : 0); }
  int nseg() const { return (npan + seg - 1) / seg; }
  size_t n_ckpt() const { return nseg() <= 1 ? 0 : 2 * (size_t)nseg(); }
  // panels of a segment, checkpoints, y_{t1+1}, ybar (and the probe panel)
  size_t bytes() const {
    if (prefix_tail) return prefix_tail + (size_t)nx() * panel;
    return panel * ((size_t)seg + 1 + n_ckpt() + 1 + nx());
  }
  // Segments of a multiple of SDW steps, so that windows never straddle one; replayed from checkpoints, no outer
  // product waits across them.
  void segment() {
    const int r = std::max(2, (int)std::ceil(std::sqrt(2.0 * npan)));
    seg = (r + SDW - 1) / SDW * SDW;
    defer = 0;
    prefix_tail = 0;
  }
  // The next smaller plan, false where there is none: two ybar panels, then segments.
  bool shrink() {
    if (nseg() > 1) return false;
    if (!windowed && defer > 1) {
      defer = 1;
      return true;
    }
    if (npan <= 2) return false;
    const size_t was = bytes();
    segment();
    return bytes() < was;
  }
};

}  // namespace tbk
