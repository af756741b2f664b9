// GPU check of what a warp of the item kernel does after one of its waits gave up
// (item_kernels.cu, drain): the bulk copies that its CTA has in flight have landed when it
// returns, and a barrier that no copy is on its way to ends it within the limit.  One CTA of
// one warp: at item i the copies of stage i & 1 and of record (i + 1) & 1 are under way, the
// other two barriers have nothing coming.  The barriers' earlier phases (i / 2 of them) are
// completed by plain arrivals first.
#include "item_kernels.cu"

#include <cstdio>
#include <vector>

using namespace cel;

constexpr int N = 8192;   // ints per copy: 32 KB

__global__ void __launch_bounds__(32) k_check(const int* src, int* out, long long* cycles, int i) {
    extern __shared__ __align__(128) uint8_t smem[];
    int* buf = reinterpret_cast<int*>(smem);   // two copies
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + 2 * N * sizeof(int));
    uint64_t* fetched = full + 2;
    const int lane = threadIdx.x;
    for (int k = lane; k < 2 * N; k += 32) buf[k] = -1;
    if (lane == 0) {
        for (int x = 0; x < 2; ++x) {
            mbar_init(&full[x], 1);
            mbar_init(&fetched[x], 1);
        }
        mbar_init_fence();
        for (int x = i; x < i + 2; ++x)   // the phases before the ones of items i and i + 1
            for (int p = 0; p < (x >> 1); ++p) {
                mbar_arrive_plain(&full[x & 1]);
                mbar_arrive_plain(&fetched[x & 1]);
            }
        fence_proxy_async_smem();
        uint64_t* bar[2] = {&full[i & 1], &fetched[(i + 1) & 1]};
        for (int c = 0; c < 2; ++c) {
            mbar_expect_arrive(bar[c], N * sizeof(int));
            bulk_g2s_tx(buf + c * N, src + c * N, N * sizeof(int), bar[c]);
        }
    }
    __syncwarp();
    const long long t0 = clock64();
    drain(full, fetched, i);
    __syncwarp();
    if (lane == 0) *cycles = clock64() - t0;
    for (int k = lane; k < 2 * N; k += 32) out[k] = buf[k];
}

int main() {
    std::vector<int> h(2 * N), got(2 * N);
    for (int k = 0; k < 2 * N; ++k) h[k] = 3 * k + 1;
    int *src, *out;
    long long *cycles, c = 0;
    const int bytes = 2 * N * sizeof(int) + 64;
    bool ok = cudaMalloc(&src, sizeof(int) * 2 * N) == cudaSuccess && cudaMalloc(&out, sizeof(int) * 2 * N) == cudaSuccess &&
              cudaMalloc(&cycles, sizeof(long long)) == cudaSuccess &&
              cudaFuncSetAttribute(k_check, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess &&
              cudaMemcpy(src, h.data(), sizeof(int) * 2 * N, cudaMemcpyHostToDevice) == cudaSuccess;
    for (int i = 0; ok && i < 6; ++i) {
        k_check<<<1, 32, bytes>>>(src, out, cycles, i);
        ok = cudaMemcpy(got.data(), out, sizeof(int) * 2 * N, cudaMemcpyDeviceToHost) == cudaSuccess &&
             cudaMemcpy(&c, cycles, sizeof c, cudaMemcpyDeviceToHost) == cudaSuccess;
        if (!ok) break;
        if (got != h) return printf("item %d: a copy had not landed\n", i), 1;
        // two barriers that nothing reaches, each up to the limit
        if (c > 3 * (MBAR_MAX_CYCLES / 100)) return printf("item %d: %lld cycles\n", i, c), 1;
    }
    if (!ok) return printf("CUDA: %s\n", cudaGetErrorString(cudaGetLastError())), 1;
    printf("ok\n");
    return 0;
}
