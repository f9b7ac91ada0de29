// rt_rows_general.cu -- rows and columns of G: every term and medium (EV of rt_internal.h).
#include "rt_rows_kernels.cuh"

namespace rt {
template struct RowEval<EV_GENERAL>;
}
