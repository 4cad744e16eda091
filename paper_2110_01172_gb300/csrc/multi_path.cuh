// multi_path.cuh - what the multi-shape executor sets on its groups' plans.
#pragma once

#include "../../include/gbdct.h"

namespace gbdct {

// The plan's intermediate array shares L2 with those of other plans in flight and
// does not stay there: write it evict-first instead of evict-last.
void plan_stream_work(gbdct_plan_t p);

}  // namespace gbdct
