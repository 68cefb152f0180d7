// Host-side definitions shared by the single-lattice API (lbm_api.cu) and the many-lattice
// runtime (lbm_batch.cu).
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <string>

#include "lbm.h"
#include "lbm_launch.h"

namespace lbm_host {

extern thread_local std::string g_err;  // message of the last failing call of this thread
int fail(int code, const char* fmt, ...);

constexpr size_t kAlign = 256;
inline size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

struct Layout {
    int pitch;
    size_t plane;       // cells per plane
    size_t pops_bytes;  // one population buffer
    size_t off_pops[2], off_hist[2], off_shist[2], shist_bytes, off_status, off_partials, total;
};

// Counters of a run of steps: the tile counter, then the row counters.  They share the reduction's
// partial sums (work of one handle is ordered on its stream).
constexpr int kRowOffset = 32, kRowCounters = 2016;
static_assert((kRowOffset + kRowCounters) * sizeof(unsigned) <= lbm::kMaxPartials * sizeof(double),
              "the counters fit the partial sums");

// Most steps of one launch of a run over so many tiles.  A run's CTAs hold their SMs until its last step, and
// kernels of other streams wait as long, so a run takes some 35 ms at most: 2^22 updates of a tile (8.2 ns each
// with FP32 storage, 5.2 ns with FP16, at 2048 x 1024), and 4096 steps, since the step of a small grid takes 4 us
// however few its tiles.  Lattices of more than 2^20 tiles, which would take fewer than four steps, go
// step by step: from 65536 tiles on a run gains 0.4 % (FP32) to 2 % (FP16) over that.
constexpr int64_t kRunTiles = 1 << 20;
inline int64_t longest_run(int64_t tiles) { return std::min<int64_t>(4096, 4 * kRunTiles / tiles); }

}  // namespace lbm_host

#define LBM_CUDA(call)                                                                                   \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) return lbm_host::fail(LBM_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

struct lbm_handle {
    lbm_params prm;
    lbm_host::Layout L;
    lbm::Phys phys;
    cudaStream_t stream;
    char* ws;
    void* pops[2];
    float2* hist[2];         // u history, alternating with the population buffers
    float2* shist[2];        // mass-flux history (density ratio != 1), else null
    unsigned* status;
    unsigned* tile_ctr;      // two tile counters of the pipelined kernel (status region + 8 bytes)
    int64_t last_pipe_step;  // step index of the last pipelined launch (-2: none since a reset)
    double* partials;
    CUtensorMap tm_fg[2];    // TMA descriptors of the (f, g) pair planes of each buffer
    CUtensorMap tm_h[2];     // TMA descriptors of the h planes of each buffer
    CUtensorMap tm_hist[2];  // TMA descriptors of the u history buffers
    int tiles_x, tiles_y;    // step-kernel grid: one tile per CTA (lbm::tile_dims of the storage mode)
    int kernel;              // LBM_KERNEL_TILE or LBM_KERNEL_PIPELINED
    int pipe_ctas;           // CTAs of the pipelined kernel (0: it does not fit, -1: not prepared)
    int chosen;              // 1: lbm_set_kernel chose it, and every step is a launch of it
    int stall;               // 1: runs wait for tiles that nobody updates (lbm_selftest_stall)
    int sms;                 // SMs of the device
    lbm::RunDims run;        // the kernel of a run of steps (blocks_per_sm 0: it does not fit)
    int cur;          // buffer holding the current state
    int initialized;
    int first;        // 1 until the first step after lbm_init_fields
    int64_t steps;
    int64_t launches;  // step kernels launched for this lattice alone
};

namespace lbm_host {

// Tile rows above and below a tile that its step reads: two rows of cells, which only a last tile row of one
// cell row, next to the first around a periodic edge, makes two tile rows.
int reach_of(const lbm_handle* h);

// Whether (nearly) every tile row reads every other, so that in a run each step waits for the whole step before
// it, and there are more tiles than that leaves room for: one launch per step is then faster (100000 x 8, us per
// step one by one / 64 steps in a run: FP32 34.6 / 35.9, FP16 25.5 / 28.6, rising bubble 30.7 / 35.2; 4000 x 24
// prescribed FP32 4.5 / 6.0; 50000 x 32, four rows: rising bubble FP16 49.3 / 51.3, FP16 drop 41.3 / 39.4; five rows
// with a reach of two, 20000 x 33 and 4000 x 33: FP32 28.9 / 27.8, 7.4 / 7.8; FP16 23.3 / 23.9, 10.5 / 9.2).
bool few_rows(const lbm_handle* h);

// Whether lbm_step does `n` steps in a row as runs (many steps in one launch).
bool takes_run(const lbm_handle* h, int64_t n);

}  // namespace lbm_host
