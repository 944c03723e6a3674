// rows_family_s.cu -- register-resident row passes in FP32 for row lengths
// 32 36 40 42 48 50 54 56 60 64 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_S(GFC_ROW_SHAPE)

}  // namespace gfc
