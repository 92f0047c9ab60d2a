// Host entry point of the step of small lattices (lb_small.cu).
#pragma once

#include "lb_internal.h"

namespace lbfe {

constexpr int kSmallMaxThreads = 256;
// FP64 tiles of at most this many rows run on two threads per node.
constexpr int kSmallSplitRows = 3;

// One step on tiles of 32 columns x `rows` rows (1..8), without obstacles: of
// the single domain d (items NULL), or of the n_items tiles of a batch's list
// (descs, items in device memory; d any of its domains).
int launch_small_step(int precision, int coll, const DomDesc& d, const DomDesc* descs,
                      const WorkItem* items, int n_items, int parity, int rows, void* stream);

}  // namespace lbfe
