// Test-only exports of the arithmetic of the matrix-entry pool.
#include "pool.h"

extern "C" {
int pool_is_padded(int steps, int rest) { return spider::pool_padded(steps, rest); }
int32_t pool_takes(int steps, int rest) { return spider::pool_grains(steps, rest); }
int64_t pool_begin(int32_t gb) { return spider::pool_first(gb); }
int64_t pool_size(int64_t N, int64_t P) { return spider::pool_entries(N, P); }
}
