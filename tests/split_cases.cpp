// The tile split of the library (tile_split.h) behind a C interface for ctypes (test infrastructure).
#include "tile_split.h"

extern "C" int64_t split_groups(int64_t rest, int64_t slots, int64_t P, int64_t W, int64_t base)
{
    return rs::split_groups(rest, slots, P, W, base);
}
