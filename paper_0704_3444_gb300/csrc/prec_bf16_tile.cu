// prec_bf16_tile.cu -- the tile kernel on D2Q9, __nv_bfloat16 storage.
#include "table_impl.cuh"

namespace mclb {

void fill_bf16_tile(KernelTable& t) { fill_tile<__nv_bfloat16>(t); }

}  // namespace mclb
