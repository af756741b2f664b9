// Host check of the launch code of the FP32 value / gradient path (item_kernels.cu) on a
// stand-in for the CUDA runtime.  Argument: which check.  Exit status 1 on a failure.
//   flags   An evaluation whose k-th launch fails leaves the tables' ready flags, the queue
//           counter and the status word cleared: tables published by a kernel with no epilogue
//           kernel behind it must not pass for the next evaluation's.
//   devices After problems on two devices were set up, the item kernel has its shared-memory
//           limit raised on both, and its grid is that of the device it is launched on.
#include "fake_runtime.cuh"

#include "item_kernels.cu"

#include <cstring>

static cel::DevProblem problem(std::vector<int32_t>& ready, int32_t* done, cel::ZTask* tasks) {
    cel::DevProblem P{};
    P.n_src = 3;
    P.n_patch = 7;
    P.n_task = 5000;
    P.ztasks = tasks;
    P.model_ne = 6;
    P.model_nd = 8;
    ready.assign(P.n_patch + 2, 0);
    P.zready = ready.data();
    P.zf_done = done;
    return P;
}

static int check_flags() {
    std::vector<int32_t> ready;
    int32_t done[2];
    cel::ZTask task;
    const cel::DevProblem P = problem(ready, done, &task);
    for (int mode : {cel::MODE_LL, cel::MODE_GRAD})
        for (int stage = 0; stage < 3; ++stage) {
            fake::sets.clear();
            fake::last_error = stage == 0 ? cudaErrorMemoryAllocation : cudaSuccess;
            fake::launch_error = stage == 0 ? cudaSuccess : cudaErrorInvalidValue;
            const cudaError_t e = cel::launch_items_stage(P, stage, mode, nullptr, nullptr, nullptr, nullptr, nullptr);
            bool flags = false, words = false;
            for (const fake::Set& s : fake::sets) {
                flags = flags || (s.p == P.zready && s.bytes == sizeof(int32_t) * ready.size());
                words = words || (s.p == P.zf_done && s.bytes == sizeof done);
            }
            if (e == cudaSuccess || !flags || !words) {
                printf("mode %d, stage %d failed: error %d, flags cleared %d, counters cleared %d\n", mode, stage,
                       (int)e, flags, words);
                return 1;
            }
        }
    return 0;
}

static int check_devices() {
    std::vector<int32_t> ready;
    int32_t done[2];
    cel::ZTask task;
    const cel::DevProblem P = problem(ready, done, &task);
    for (int d : {0, 1, 0}) {
        fake::device = d;
        fake::launched_unset = false;
        if (cel::prime_items_kernels() != cudaSuccess) return printf("set-up failed on device %d\n", d), 1;
        for (int mode : {cel::MODE_LL, cel::MODE_GRAD}) {
            const cudaError_t e = cel::launch_items_stage(P, 1, mode, nullptr, nullptr, nullptr, nullptr, nullptr);
            const unsigned want = 4u * fake::sm_of_device[d];   // the stand-in's four CTAs per multiprocessor
            if (e != cudaSuccess || fake::launched_unset || fake::grid != want)
                return printf("device %d, mode %d: error %d, limit missing %d, grid %u (expected %u)\n", d, mode, (int)e,
                              fake::launched_unset, fake::grid, want), 1;
        }
    }
    return 0;
}

int main(int argc, char** argv) {
    fake::no_real_device();
    const char* what = argc > 1 ? argv[1] : "";
    if (!strcmp(what, "flags")) return check_flags();
    if (!strcmp(what, "devices")) return check_devices();
    printf("unknown check %s\n", what);
    return 1;
}
