// k_rows32.cu -- the Cholesky-QR step of the mixed path compiled for blocks of 17 to 32 columns
// (rows_qr.cuh only: blocks this wide fall back to the generic passes of k_krylov.cu when a
// single factor is not accurate enough).
#include <algorithm>

#include "mma.cuh"
#include "rows_api.h"
#include "rows_common.cuh"

namespace expm {
namespace rows32 {
#include "rows_chol.cuh"
#include "rows_qr.cuh"
}  // namespace rows32
}  // namespace expm
