// rows_family16_f.cu -- register-resident row passes in 16 bits for row lengths
// 1536 1750 1960 2058 (recursive column solve only).
#include "rows_family.cuh"

namespace gfc {

GFC_ROWS_F(GFC_ROW_SHAPE16)

}  // namespace gfc
