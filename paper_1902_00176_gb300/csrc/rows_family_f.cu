// rows_family_f.cu -- register-resident row passes in FP32 for row lengths
// 1536 1750 1960 2058 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_F(GFC_ROW_SHAPE)

}  // namespace gfc
