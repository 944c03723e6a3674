// rows_family16_d.cu -- register-resident row passes in 16 bits for row lengths
// 784 882 980 1080 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_D(GFC_ROW_SHAPE16)

}  // namespace gfc
