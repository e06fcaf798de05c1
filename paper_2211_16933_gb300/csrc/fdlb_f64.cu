// FP64 kernels: everything in FP64.
#include "qlbm_internal.h"
namespace qlbm {
// 16-byte aligned: the stage kernels read the table rows as pairs.
static __constant__ __align__(16) double QL_TAB[kTabTotal];
// log_<double>: (1 / c_j, log c_j leading), (log c_j trailing, 0) at 2 j; log 2 in two parts at 257.
// Read per lane at different j, so not in the constant bank.
static __device__ double2 QL_LOGTAB[258];
}
#define QL_LOGTAB QL_LOGTAB
#define QL_REAL double
#define QL_SUFFIX f64
#include "fdlb_impl.cuh"
#include "fdlb_cells.cuh"
#include "fdlb_lq.cuh"
