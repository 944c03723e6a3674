// rows_family_d.cu -- register-resident row passes in FP32 for row lengths
// 784 882 980 1080 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_D(GFC_ROW_SHAPE)

}  // namespace gfc
