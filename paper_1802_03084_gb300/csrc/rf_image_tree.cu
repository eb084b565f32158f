// Row pass with derived images (sums of 2 .. 16 images) for image sides 64 .. 8192.
#include "rf_image.cuh"

namespace rf {
RF_INSTANTIATE_TREE(64)
RF_INSTANTIATE_TREE(128)
RF_INSTANTIATE_TREE(256)
RF_INSTANTIATE_TREE(512)
RF_INSTANTIATE_TREE(1024)
RF_INSTANTIATE_TREE(2048)
RF_INSTANTIATE_TREE(4096)
RF_INSTANTIATE_TREE(8192)
}  // namespace rf
