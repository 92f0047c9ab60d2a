// Host entry point of the step of small lattices (lb_small.cu).
#pragma once

#include "lb_internal.h"

namespace lbfe {

constexpr int kSmallMaxThreads = 256;
// FP64 tiles of at most this many rows run on two threads per node.
constexpr int kSmallSplitRows = 3;

// Several steps per launch: a CTA's threads cover its tile and 2 (steps - 1)
// nodes around it, 32 columns in all.
constexpr int kStepsMaxThreads = 768;
constexpr int small_steps_cols(int steps) { return 32 - 4 * (steps - 1); }
constexpr int small_steps_threads(int steps, int rows) { return 32 * (rows + 4 * (steps - 1)); }

// One step on tiles of 32 columns x `rows` rows (1..8; FP32 full storage 3..8),
// without obstacles: of
// the single domain d (items NULL), or of the n_items tiles of a batch's list
// (descs, items in device memory; d any of its domains).
int launch_small_step(int precision, int coll, const DomDesc& d, const DomDesc* descs,
                      const WorkItem* items, int n_items, int parity, int rows, void* stream);

// `steps` (2 ..) steps of the single domain d (FP32, no obstacles, nx and ny at least
// 2 * steps) on tiles of small_steps_cols(steps) columns x `rows`
// rows, small_steps_threads(steps, rows) <= kStepsMaxThreads; flips the buffer
// once.
int launch_small_steps(int coll, const DomDesc& d, int parity, int steps, int rows, void* stream);
// Its shared-memory opt-in (once per device, outside any capture).
int prepare_small_steps();

}  // namespace lbfe
