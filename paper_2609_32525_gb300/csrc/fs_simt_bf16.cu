// The tiled fp32 passes on bf16 point tensors.
#include "fs_simt_tiles.cuh"

template struct fs::SimtTiles<__nv_bfloat16>;
