// Batch-kernel instances for BF16_FG storage.
#include "lbm_launch.h"

namespace lbm {

LBM_DEFINE_BATCH(bf16fg, kBF16FG)

}  // namespace lbm
