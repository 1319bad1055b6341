// prec_fp16_tile.cu -- the tile kernel on D2Q9, __half storage.
#include "table_impl.cuh"

namespace mclb {

void fill_fp16_tile(KernelTable& t) { fill_tile<__half>(t); }

}  // namespace mclb
