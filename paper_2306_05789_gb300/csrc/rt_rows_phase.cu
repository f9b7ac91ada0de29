// rt_rows_phase.cu -- rows and columns of G: phase tables (EV of rt_internal.h).
#include "rt_rows_kernels.cuh"

namespace rt {
template struct RowEval<EV_PHASE>;
}
