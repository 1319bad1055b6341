// prec_fp32_tile.cu -- the tile kernel on D2Q9, float storage.
#include "table_impl.cuh"

namespace mclb {

void fill_fp32_tile(KernelTable& t) { fill_tile<float>(t); }

}  // namespace mclb
