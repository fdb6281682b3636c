// A team whose last CTA arrives at a barrier late, by a bounded delay: what the barrier returns to every CTA.
#include "../paper_1903_01665_gb300/csrc/fg_internal.cuh"

namespace {
__global__ void __launch_bounds__(fg::kBlock) late_arrival(fg::Ctrl *c, unsigned long long timeout_ns,
                                                           unsigned long long late_ns, int *ok,
                                                           unsigned long long *took_ns) {
    const fg::Team t{(int)blockIdx.x, (int)gridDim.x, c->bar};
    fg::team_begin();
    if (blockIdx.x == gridDim.x - 1) {
        const unsigned long long t0 = fg::global_ns();
        for (int i = 0; i < 1000000 && fg::global_ns() - t0 < late_ns; i++) __nanosleep(1000);
    }
    const unsigned long long t1 = fg::global_ns();
    const bool r = fg::team_sync(t, c, timeout_ns, 1);
    if (threadIdx.x == 0) {
        ok[blockIdx.x] = r && fg::team_total() == (int64_t)gridDim.x * fg::kBlock;
        took_ns[blockIdx.x] = fg::global_ns() - t1;
    }
}
}  // namespace

// ok[grid], took_ns[grid]: each CTA's result and time in the barrier; returns the status bits, or -1 on a CUDA error.
extern "C" int run_late_arrival(int grid, double timeout_ms, double late_ms, int *ok, unsigned long long *took_ns) {
    fg::Ctrl *c = nullptr;
    int *d_ok = nullptr, status = -1;
    unsigned long long *d_took = nullptr;
    unsigned long long timeout_ns = (unsigned long long)(timeout_ms * 1e6), late_ns = (unsigned long long)(late_ms * 1e6);
    if (cudaMalloc(&c, sizeof(fg::Ctrl)) == cudaSuccess && cudaMalloc(&d_ok, grid * sizeof(int)) == cudaSuccess &&
        cudaMalloc(&d_took, grid * sizeof(unsigned long long)) == cudaSuccess) {
        cudaMemset(c, 0, sizeof(fg::Ctrl));
        void *args[] = {&c, &timeout_ns, &late_ns, &d_ok, &d_took};
        if (cudaLaunchCooperativeKernel((void *)late_arrival, dim3(grid), dim3(fg::kBlock), args, 0, 0) == cudaSuccess &&
            cudaDeviceSynchronize() == cudaSuccess) {
            cudaMemcpy(ok, d_ok, grid * sizeof(int), cudaMemcpyDeviceToHost);
            cudaMemcpy(took_ns, d_took, grid * sizeof(unsigned long long), cudaMemcpyDeviceToHost);
            if (cudaMemcpy(&status, &c->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) status = -1;
        }
    }
    cudaFree(c);
    cudaFree(d_ok);
    cudaFree(d_took);
    return status;
}
