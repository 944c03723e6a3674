// rows_family_a.cu -- register-resident row passes in FP32 for row lengths
// 140 160 180 200 224 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_A(GFC_ROW_SHAPE)

}  // namespace gfc
