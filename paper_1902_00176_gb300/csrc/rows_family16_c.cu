// rows_family16_c.cu -- register-resident row passes in 16 bits for row lengths
// 448 500 560 630 700 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_C(GFC_ROW_SHAPE16)

}  // namespace gfc
