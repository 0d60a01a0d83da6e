// npx_step_gp.cu -- the step kernels of worlds too large to be on the device at once: flat ground, the
// posed points of the scenes in flight in global memory.  A translation unit of their own, so that
// they compile beside the others.
#define NPX_STEP_DEVICE_CODE
#include "npx_step.cu"

// Flat ground with the points in global memory: a slot is a third of its size (hexapods 2.6 of 8.2
// KB), so registers (16 warps per SM) and not shared memory (7 at 8 lanes) bound the scenes in
// flight, and the few points a step touches are L1 hits.  Taken by chunked stepping where not every
// scene fits on the device at once: evolution of 16,000 hexapods, 400 steps: 3.58 -> 2.53 ms.  The rule
// in npx_world.cpp says which worlds, and which launches of few steps, keep them in the slots.
template <int LPS>
__global__ void __launch_bounds__(512) step_kernel_gp(const __grid_constant__ WorldDev W, int n_steps, int sbytes,
                                                      const __grid_constant__ CUtensorMap tmap) {
    step_body<LPS, true, false, false, true>(W, n_steps, sbytes, &tmap);
}

void *step_gp_kernel(int lps) {
    switch (lps) {
        case 4: return (void *)step_kernel_gp<4>;
        case 8: return (void *)step_kernel_gp<8>;
        case 16: return (void *)step_kernel_gp<16>;
        case 32: return (void *)step_kernel_gp<32>;
        default: return nullptr;
    }
}

}  // namespace npx
