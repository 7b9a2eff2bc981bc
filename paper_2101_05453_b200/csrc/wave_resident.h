// Wavefront kernel with resident weights (wave_resident_sm100.cu), as wave_sm100.cu sees it.
#pragma once
#include "wave_common.cuh"

namespace ql {

struct ResidentStack;

// Plans the calls of 1 .. max_B rows of a stack whose layers' formats and state offsets are in `base`; null where no call of it fits.
ResidentStack *resident_plan(const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, int max_T, int max_B, int max_smem,
                             int y_stride);
void resident_destroy(ResidentStack *s);
// Its memory, taken front to back from `keep` (weight images, counters) and `work` (a call's activations); with `fill` also written.
int resident_place(ResidentStack *s, const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, WaveArena &keep, WaveArena &work, bool fill);
bool resident_supported(const ResidentStack *s, int T, int B);
int launch_resident(const ResidentStack *s, const int8_t *x, int T, int B, int8_t *const (&h)[2], int16_t *const (&c)[2], int8_t *y, int *status,
                    int *status2, unsigned missing, unsigned long long limit_ns, bool refuse, cudaStream_t st);
void resident_debug_plan(const ResidentStack *s, int T, int B, int *out4);

}  // namespace ql
