// Entry points between the library's own translation units.
#pragma once

#include "../../include/grpic.h"

namespace grpic {

// grpic_create with a choice: metric_table = false leaves out the field kernels' metric table of an FP64 context (the
// server's runs, whose admission charges the memory that grpic_request_bytes states).
grpic_status create_context(const grpic_config* cfg, void* stream, bool metric_table, grpic_ctx** out);

// Free one metric table that came from this allocator (null: cudaMalloc) on the current device and is not in use by a
// running batched step.  Returns whether there was one.
bool give_up_metric_table(grpic_alloc_fn alloc, void* user);

}  // namespace grpic
