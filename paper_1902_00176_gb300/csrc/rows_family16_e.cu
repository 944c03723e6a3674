// rows_family16_e.cu -- register-resident row passes in 16 bits for row lengths
// 1120 1200 1372 1400 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_E(GFC_ROW_SHAPE16)

}  // namespace gfc
