// rows_family_e.cu -- register-resident row passes in FP32 for row lengths
// 1120 1200 1372 1400 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_E(GFC_ROW_SHAPE)

}  // namespace gfc
