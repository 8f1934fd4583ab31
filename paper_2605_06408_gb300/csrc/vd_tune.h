// vd_tune.h -- which knobs a trial of the autotuner can change for a
// configuration: those that the kernels it runs read. Host code, no CUDA.
#pragma once

#include <stdint.h>

#include <initializer_list>
#include <vector>

#include "vd.h"

namespace vd {

// A configuration with an ablation mode, the event counters or plain FP32:
// the kernels of the default modes have these folded in.
inline bool generic_config(const vd_config& g) {
  return g.cull_mode != 0 || g.traversal != 0 || g.counters != 0 || g.precision != 0;
}

struct TuneValue {
  int32_t vd_config::*field;
  int32_t value;
};

// The knobs in the order in which the tuner settles them. The warm start comes
// before the leaf size: with the KNN start larger leaves win.
constexpr int kTuneKnobs = 6;

// The other values of knob `k` that make a difference to builds with
// configuration `c`. `large`: the last build had cells for the large-cell
// pass. The default kernels have fixed capacities, start from the KNN list and
// walk a tree with leaves of its own; blocks of at most four warps. In those
// builds only the large-cell pass reads the leaf size, and of the warm start
// only whether there is one. The thread form reads none but the leaf size.
inline std::vector<TuneValue> tune_values(const vd_config& c, int k, bool large) {
  const bool thread = c.cell_mode == 1, wide = !thread && !generic_config(c);
  std::vector<TuneValue> out;
  auto add = [&](int32_t vd_config::*f, std::initializer_list<int32_t> values, int32_t now) {
    for (int32_t v : values)
      if (v != now) out.push_back({f, v});
  };
  switch (k) {
    case 0:
      add(&vd_config::cell_mode, {0, 1}, c.cell_mode);
      break;
    case 1:
      if (wide && large) add(&vd_config::warm_start, {0, 1}, c.warm_start ? 1 : 0);
      if (!wide && !thread) add(&vd_config::warm_start, {0, 1, 2}, c.warm_start);
      break;
    case 2:
      if (!wide && !thread) add(&vd_config::verts_per_lane, {2, 4}, c.verts_per_lane);
      break;
    case 3:
      if (!wide && !thread) add(&vd_config::queue_per_lane, {2, 4, 8}, c.queue_per_lane);
      break;
    case 4:
      if (!wide || large) add(&vd_config::leaf_size, {8, 16, 32}, c.leaf_size);
      break;
    case 5:
      if (wide) add(&vd_config::warps_per_block, {2, 4}, c.warps_per_block > 4 ? 4 : c.warps_per_block);
      if (!wide && !thread) add(&vd_config::warps_per_block, {2, 4, 8}, c.warps_per_block);
      break;
  }
  return out;
}

// What of a configuration decides which kernels run, and so which result of
// the tuner holds for it: part of its cache's key.
inline int tune_form(const vd_config& c) {
  return c.cull_mode + 3 * (c.traversal + 2 * (c.precision + 2 * c.counters));
}

}  // namespace vd
