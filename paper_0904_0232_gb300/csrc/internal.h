// Entry points between the library's own translation units.
#pragma once

#include "../../include/grpic.h"

namespace grpic {

// grpic_create with a choice: metric_table = false leaves out the field kernels' metric table of an FP64 context (the
// server's runs, whose admission charges the memory that grpic_request_bytes states).
grpic_status create_context(const grpic_config* cfg, void* stream, bool metric_table, grpic_ctx** out);

}  // namespace grpic
