// Batch-kernel instances for FP16_FG storage.
#include "lbm_launch.h"

namespace lbm {

LBM_DEFINE_BATCH(fp16fg, kFP16FG)

}  // namespace lbm
