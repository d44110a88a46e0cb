// Device memory of a request, and contexts without optional workspace (internal; host only).
#pragma once
#include <stddef.h>

#include "../../include/caspt2.h"

namespace caspt2 {

// caspt2_create, with (sliced) or without the workspace that the plain form can do without:
// class H then runs in its fused kernel.
int create_context(caspt2_ctx** out, const caspt2_dims* dims, const caspt2_options* opt,
                   bool sliced);
// Device bytes that create_context, one solve and (densities) one caspt2_densities hold: the sum
// of their allocations, with the split products' workspace from above.
size_t context_bytes(const caspt2_dims& dims, const caspt2_options& opt, bool densities,
                     bool sliced);

}  // namespace caspt2
