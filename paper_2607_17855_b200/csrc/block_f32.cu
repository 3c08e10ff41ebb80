// Float32 instantiations of the block kernels.
#include "block.cuh"

const void *bi_block_kernel_f32(int BR, int BC, bool window, int sync, bool hass) {
  return bi_block::pick_kernel<float>(BR, BC, window, sync, hass);
}
