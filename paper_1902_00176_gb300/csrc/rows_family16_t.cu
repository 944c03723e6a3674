// rows_family16_t.cu -- register-resident row passes in 16 bits for row lengths
// 70 72 80 84 90 96 98 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_T(GFC_ROW_SHAPE16)

}  // namespace gfc
