// rt_rows_plain.cu -- rows and columns of G: one wall or none, optical_depth (EV of rt_internal.h).
#include "rt_rows_kernels.cuh"

namespace rt {
template struct RowEval<EV_PLAIN>;
}
