// rows_family16_u.cu -- register-resident row passes in 16 bits for row lengths
// 100 112 120 126 128 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_U(GFC_ROW_SHAPE16)

}  // namespace gfc
