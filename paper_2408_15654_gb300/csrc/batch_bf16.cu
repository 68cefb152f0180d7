// Batch-kernel instances for BF16 storage.
#include "lbm_launch.h"

namespace lbm {

LBM_DEFINE_BATCH(bf16, kBF16)

}  // namespace lbm
