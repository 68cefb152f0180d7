// The launch and set-up functions of the step kernels, recorded instead of launched.
#include <vector>

#include "lbm_launch.h"

namespace {

struct Record {
    int kind;        // 's' step, 'r' run, 'b' step of a batch, 'R' run of a batch
    int status;      // what it returned
    int nsteps;
    int cooperative; // every CTA has to be resident at once
    int ctas, members;
    long long steps; // steps taken before it (of the first member)
    long long tiles;
};
std::vector<Record> records;
int fail_kind = 0, fail_at = 0, fail_code = 0;  // the fail_at-th launch of fail_kind from now returns fail_code
int prepared[128];                              // set-ups by kind

cudaError_t record(Record r) {
    if (r.kind == fail_kind && fail_at-- == 0) r.status = fail_code;
    records.push_back(r);
    return static_cast<cudaError_t>(r.status);
}

}  // namespace

namespace lbm {

cudaError_t launch_step(int, const StepArgs&, int, const Variant&, dim3 grid, int pipe, cudaStream_t) {
    return record({'s', 0, 1, 0, pipe ? pipe : (int)(grid.x * grid.y), 1, 0, (long long)grid.x * grid.y});
}
cudaError_t launch_run(int, const RunArgs& a, const Variant&, int ctas, cudaStream_t) {
    return record({'r', 0, a.nsteps, a.ctr ? 0 : 1, ctas, 1, a.steps, (long long)a.ntx * a.nty});
}
cudaError_t launch_batch(int, const BatchArgs& b, const Variant&, unsigned tiles, cudaStream_t) {
    return record({'b', 0, 1, 0, b.ws_ctas, b.ndescs, b.s, (long long)tiles});
}
cudaError_t launch_batch_run(int, const RunManyArgs& a, const Variant&, int ctas, cudaStream_t) {
    long long tiles = 0;
    for (int k = 0; k < a.members; ++k) tiles += a.m[k].ntx * a.m[k].nty;
    return record({'R', 0, a.nsteps, 0, ctas, a.members, a.m[0].steps, tiles});
}

cudaError_t prepare_step(int, const Variant&, int* blocks, int* pipe_blocks) {
    prepared['s']++;
    *blocks = 5;
    if (pipe_blocks) *pipe_blocks = 4;
    return cudaSuccess;
}
cudaError_t prepare_run(int, const Variant&, RunDims* d) {
    prepared['r']++;
    *d = RunDims{1, 5};
    return cudaSuccess;
}
cudaError_t prepare_batch(int, int* blocks) {
    prepared['b']++;
    *blocks = 2;
    return cudaSuccess;
}
cudaError_t prepare_batch_run(int, const Variant&, RunDims* d) {
    prepared['R']++;
    *d = RunDims{1, 5};
    return cudaSuccess;
}

}  // namespace lbm

extern "C" {

void fake_reset() {
    records.clear();
    fail_kind = 0;
    for (int& p : prepared) p = 0;
}
void fake_fail(int kind, int at, int code) {
    fail_kind = kind;
    fail_at = at;
    fail_code = code;
}
int fake_prepared(int kind) { return prepared[kind]; }
int fake_count() { return (int)records.size(); }
void fake_get(int k, long long* out) {
    const Record& r = records[k];
    const long long v[] = {r.kind, r.status, r.nsteps, r.cooperative, r.ctas, r.members, r.steps, r.tiles};
    for (int i = 0; i < 8; ++i) out[i] = v[i];
}

}  // extern "C"
