// rows_family_b.cu -- register-resident row passes in FP32 for row lengths
// 252 294 320 360 400 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_B(GFC_ROW_SHAPE)

}  // namespace gfc
