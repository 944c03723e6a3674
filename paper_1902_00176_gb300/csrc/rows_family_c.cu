// rows_family_c.cu -- register-resident row passes in FP32 for row lengths
// 448 500 560 630 700 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_C(GFC_ROW_SHAPE)

}  // namespace gfc
