// What a context remembers of driver calls holds for its own device only.  Host code, with a stand-in for cudaGetDevice.
#include <cuda_runtime.h>

static int current_device = 0;
static cudaError_t fake_get_device(int *d) {
    *d = current_device;
    return current_device < 0 ? cudaErrorNoDevice : cudaSuccess;
}
#define cudaGetDevice fake_get_device
#include "finch_internal.cuh"

int main() {
    finch::Ctx ctx = {};
    ctx.cfg.device = 1;
    ctx.smem_set(finch::kSmemTc);  // another device is current: its kernels' limits were raised, not device 1's
    if (ctx.smem_ready(finch::kSmemTc)) return 1;
    current_device = -1;
    ctx.smem_set(finch::kSmemTc);
    if (ctx.smem_ready(finch::kSmemTc)) return 2;
    current_device = 1;
    ctx.smem_set(finch::kSmemTc);
    return ctx.smem_ready(finch::kSmemTc) && !ctx.smem_ready(finch::kSmemFused) ? 0 : 3;
}
