// rows_family_u.cu -- register-resident row passes in FP32 for row lengths
// 100 112 120 126 128 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_U(GFC_ROW_SHAPE)

}  // namespace gfc
