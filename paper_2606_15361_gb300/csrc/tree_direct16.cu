// The direct tree kernel with 16-bit table entries (see tree_direct.cu).
#define SND_DIRECT_NARROW
#include "tree_direct.cu"
