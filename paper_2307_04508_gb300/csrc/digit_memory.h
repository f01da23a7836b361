// What the server needs to know of a context's digit workspace (api.cu).
#pragma once

#include <stddef.h>

#include "../../include/ltgw.h"

namespace ltgw {

constexpr size_t kSliceHold = (size_t)6 << 30;   // default of ltgw_set_digit_memory

// Bytes with which the digits and partial sums of a solve with N auxiliary functions
// after the NAF step (or fewer) run: `limit`, less where all of them take less, more where
// the smallest piece of a product takes more.
size_t solve_digit_bytes(const ltgw_params &p, int n_tgt, int N, size_t limit);

// Free the arenas of a context's products only (no call in flight).
void release_products(ltgw_ctx *ctx);

}  // namespace ltgw
