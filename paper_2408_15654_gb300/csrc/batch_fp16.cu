// Batch-kernel instances for FP16 storage.
#include "lbm_launch.h"

namespace lbm {

LBM_DEFINE_BATCH(fp16, kFP16)

}  // namespace lbm
