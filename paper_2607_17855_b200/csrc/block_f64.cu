// Float64 instantiations of the block kernels.
#include "block.cuh"

const void *bi_block_kernel_f64(int BR, int BC, bool window, int sync, bool hass) {
  return bi_block::pick_kernel<double>(BR, BC, window, sync, hass);
}
