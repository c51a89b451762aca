// The tiled fp32 passes on fp32 point tensors.
#include "fs_simt_tiles.cuh"

template struct fs::SimtTiles<float>;
