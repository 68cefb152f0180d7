// Batch-kernel instances for FP32 storage.
#include "lbm_launch.h"

namespace lbm {

LBM_DEFINE_BATCH(fp32, kFP32)

}  // namespace lbm
