// Host check of the trust-region step's shared memory (fit.cu): the column that the FP32
// factorisation reads as float4 starts on a 16-byte boundary by its type and holds the last
// read, and the two uses of the memory share one size.
#include "fit.cu"

#include <cstddef>

using cel::TrShared;
static_assert(alignof(TrShared) >= 16, "the dynamic shared array starts on a 16-byte boundary");
static_assert(offsetof(TrShared::Search, cb) % 16 == 0, "so does the column");
static_assert(sizeof(TrShared::Search::cb) >= 16 * ((cel::TRN + 3) / 4), "whole float4s of TRN entries");
static_assert(sizeof(TrShared) >= sizeof(TrShared::Step) && sizeof(TrShared) >= sizeof(TrShared::Search), "both uses fit");

namespace cel {
// the launchers that fit.cu calls are not linked here
#define STUB { return cudaErrorNotSupported; }
cudaError_t launch_prep(const DevProblem&, const double*, int, cudaStream_t, bool, bool) STUB
cudaError_t launch_contrib(const DevProblem&, int, cudaStream_t, bool) STUB
cudaError_t launch_hess_pixels(const DevProblem&, int, const double*, double*, cudaStream_t) STUB
cudaError_t launch_finalize_hess(const DevProblem&, int, double*, double*, double*, cudaStream_t) STUB
void set_last_error(const char*) {}
}  // namespace cel

int main() { return 0; }
