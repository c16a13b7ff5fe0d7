// The consumer kernels of wide ensembles (see k_explain.cuh).
#include "k_explain.cuh"

namespace wdf {
WDF_EXPLAIN_WIDE(2, )
WDF_EXPLAIN_WIDE(3, )
WDF_EXPLAIN_WIDE(4, )
WDF_EXPLAIN_WIDE(5, )
WDF_EXPLAIN_WIDE(6, )
WDF_EXPLAIN_WIDE(7, )
WDF_EXPLAIN_WIDE(8, )
}  // namespace wdf
