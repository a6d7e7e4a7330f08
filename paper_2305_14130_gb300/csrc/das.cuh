// DAS sampling K_r (eq. 3) of one time step: by a launch of its own (k_misc.cu), or by the next
// forward step (k_tile.cu), which reads the same velocities and leaves them as they are.
#pragma once

#include "plan.hpp"

namespace efwi {

struct DasArgs {
    const int *tr_shot, *tr_off;
    const float *tr_w;
    double *acc;                // running strain
    const float *vx, *vz;       // v^{n+1/2}
    float *d;                   // [ntr][nt] (null: nothing to sample)
    int t0, ntr, nt, n;         // first trace and number of traces
    float dt;
    int strain;
};

inline DasArgs das_args(const efwi_plan *p, const Fields &F, int n, float *d) {
    return DasArgs{p->tr_shot, p->tr_off, p->tr_w, p->tr_acc, F.vx, F.vz, d, 0, p->d.ntr, p->d.nt, n, (float)p->d.dt,
                   p->d.das_mode == EFWI_DAS_STRAIN};
}

// strain rate of trace t = sum of 16 weighted velocity samples (weights carry +-t_k / L); strain =
// running time integral
__device__ __forceinline__ void das_sample(const ShotDev *shots, const DasArgs &a, int t) {
    const long long base = shots[a.tr_shot[t]].off;
    float rate = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float *f = (k >> 2) & 1 ? a.vz : a.vx;
        rate += a.tr_w[t * 16 + k] * f[base + a.tr_off[t * 16 + k]];
    }
    float out = rate;
    if (a.strain) {
        const double s = a.acc[t] + (double)a.dt * rate;
        a.acc[t] = s;
        out = (float)s;
    }
    a.d[(long long)t * a.nt + a.n] = out;
}

}  // namespace efwi
