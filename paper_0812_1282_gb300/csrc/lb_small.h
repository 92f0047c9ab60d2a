// Host entry point of the step of small lattices (lb_small.cu).
#pragma once

#include "lb_internal.h"

namespace lbfe {

constexpr int kSmallMaxThreads = 256;

// One step of a single domain without obstacles on tiles of 32 columns x
// `rows` rows (1..8).
int launch_small_step(int precision, int coll, const DomDesc& d, int parity, int rows, void* stream);

}  // namespace lbfe
