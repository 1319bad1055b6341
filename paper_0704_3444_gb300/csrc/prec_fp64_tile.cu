// prec_fp64_tile.cu -- the tile kernel on D2Q9, double storage.
#include "table_impl.cuh"

namespace mclb {

void fill_fp64_tile(KernelTable& t) { fill_tile<double>(t); }

}  // namespace mclb
