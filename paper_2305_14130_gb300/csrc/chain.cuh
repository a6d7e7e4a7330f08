// Launches of the time loops' kernels that overlap their start with the end of the kernel before.
#pragma once

#include "plan.hpp"

namespace efwi {

// A kernel of a time loop reads what the launch before it wrote, so the stream runs one after the
// other, and at small grids the gap between two launches (about a microsecond) is a good part of a
// step.  Launched through launch_chained, a kernel's CTAs may become resident while the last CTAs of
// the launch before still run; they set up their barriers and wait in chain_begin(), which returns
// when that launch has completed and its writes are visible.  Every CTA of a chained kernel calls
// chain_begin() before it touches anything but the plan's constants (geometry, work items), so each
// launch still starts its work after all earlier ones.  It lets its successor's CTAs in only then:
// one launch at most is waiting on the device.  200 x 100, one shot, 1000 steps: 4.70 -> 4.14 ms, its
// gradient 14.8 -> 12.6 ms; 128 x 128, 4 shots, gradient 11.8 -> 10.8 ms.
//
// Only steps with all tiles resident at once are chained.  A larger step lasts long against the gap,
// and the waiting CTAs take the places of the last tiles' CTAs: 1000 x 300, 32 shots, 300 steps
// 42.3 -> 42.8 ms; 8 shots with the energy sum between the steps 15.5 -> 16.0 ms.
inline bool chain_fwd(const efwi_plan *p) {
    return p->chained && lean_fwd(p) && p->tiles.n <= p->tma_grid;
}
inline bool chain_adj(const efwi_plan *p) {
    return p->chained && p->adj_form == EFWI_ADJ_FORM_SCALED && p->adj_stencil == EFWI_STENCIL_TMA &&
           p->adjs_vec >= 4 && p->adj_tiles.n <= p->tma_adj_grid;
}

__device__ __forceinline__ void chain_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
void launch_chained(bool chained, void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st,
                    A... args) {
    cudaLaunchAttribute at[1] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = at;
    c.numAttrs = chained ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, P(args)...);
}

}  // namespace efwi
