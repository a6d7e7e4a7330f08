// What the TMA kernels of the scaled-stress adjoint step share (k_adjs_tma.cu, k_adj_tile.cu):
// arguments, the layout of a staged tile, its copies and the view of the forward velocities.
#pragma once

#include <type_traits>

#include "plan.hpp"
#include "tma.cuh"

namespace efwi {

struct TmaAdjsArgs {
    const ShotDev *shots;
    const int4 *tiles;
    const AdjsMaps *maps;
    int ntiles;
    int af;                     // first field of the read adjoint buffer in the adjoint-state maps
    int vf;                     // first field of this step's forward velocities in the segment map
    Fields out;                 // adjoint buffer written
    Pml pml;                    // current adjoint PML memory (V and S blocks, read)
    float *n1, *n3, *n2, *n4;   // next V block
    float *n5, *n8, *n6, *n7;   // next S block
    float *Glam, *Gmu, *Gmuxz, *Gbx, *Gbz;
    float dt, rdx, rdz;
    int *err;
    int *count;                 // tile counter of the lean kernel (TileFeed)
    const float *hmax;          // snapshot maxima of the step (SK != 0): the power-of-two scales
    int ns;
};

// One stage (halo-4 coordinates: column x = cell i - i0 + 4, row y = cell j - j0 + 4):
// R2 arrays hold rows 2 .. TZ+5, F_zz rows 1 .. TZ+7, F_xz rows 0 .. TZ+6 (R3 rows each,
// padded to 128 bytes); tile arrays TX x TZ.  Every array starts 128-byte aligned.
template <int TX, int TZ, int SK>
struct AdjsLayout {
    static constexpr int SX = TX + 8;
    static constexpr int R2 = TZ + 4, R3 = TZ + 7;
    static constexpr int A2 = SX * R2;
    static constexpr int A3 = SX * R3, A3P = (A3 + 31) & ~31;
    static constexpr int NC = TX * TZ;
    // forward velocities: FP32, or 2-byte FP16/BF16 snapshot elements (SK != 0)
    static constexpr int WB = SK ? 2 : 4, AW = A2 * WB / 4;                    // floats of one of them
    static constexpr int OVX = 0, OVZ = A2, OFXX = 2 * A2, OFZZ = 3 * A2, OFXZ = OFZZ + A3P, OBX = OFXZ + A3P,
                         OBZ = OBX + A2, OWX = OBZ + A2, OWZ = OWX + AW, OLAM = (OWZ + AW + 31) & ~31,
                         OG = OLAM + 3 * NC;
    static constexpr int BUF = (OG + 5 * NC + 31) & ~31;                      // floats per stage
    static constexpr unsigned LOADED = (5u * A2 + 2u * A3 + 8u * NC) * 4u + 2u * A2 * WB;   // bytes the copies bring
    // per CTA, edge tiles only: F_xz with its x-strip CPML term (g4), e^2, e^4 (R2 rows)
    // and F of the tile before its update
    static constexpr int EXTRA = 3 * A2 + 3 * NC;
    static constexpr size_t smem() { return (2 * (size_t)BUF + EXTRA) * 4 + 128; }
    static_assert(A2 % 32 == 0 && NC % 32 == 0, "arrays must keep 128-byte alignment");
};

// tl: the tile's work item, already in a register (no global load on the issuing thread's
// path between the tile's barriers)
template <int TX, int TZ, int SK>
__device__ __forceinline__ void issue_adjs(const TmaAdjsArgs &a, const int4 tl, float *buf, uint64_t *bar) {
    using L = AdjsLayout<TX, TZ, SK>;
    const AdjsMaps *m = a.maps + tl.x;
    mbar_expect_tx(bar, L::LOADED);
    // element x = cell i + GX (halo-4 column 0 = cell i0 - 4), row y = cell j + GZ: halo-4 row r
    // of the tile is map row j0 - 4 + r + GZ = tl.z - 2 + r
    tma_load_3d(buf + L::OVX, &m->a2, bar, tl.y - 4 + EFWI_GX, tl.z, a.af);            // v^x, v^z: rows 2..
    tma_load_3d(buf + L::OFXX, &m->a1, bar, tl.y - 4 + EFWI_GX, tl.z, a.af + 2);       // F_xx: rows 2..
    tma_load_3d(buf + L::OFZZ, &m->a3, bar, tl.y - 4 + EFWI_GX, tl.z - 1, a.af + 3);   // F_zz: rows 1..
    tma_load_3d(buf + L::OFXZ, &m->a3, bar, tl.y - 4 + EFWI_GX, tl.z - 2, a.af + 4);   // F_xz: rows 0..
    tma_load_3d(buf + L::OBX, &m->mb, bar, tl.y - 4 + EFWI_GX, tl.z, 3);               // b_x, b_z: rows 2..
    tma_load_3d(buf + L::OWX, &m->sv, bar, tl.y - 4 + EFWI_GX, tl.z, a.vf);            // forward v_x, v_z: rows 2..
    tma_load_3d(buf + L::OLAM, &m->mc, bar, tl.y + EFWI_GX, tl.z + 2, 0);      // lambda, mu, mu_xz: tile
    tma_load_3d(buf + L::OG, &m->gi, bar, tl.y + EFWI_GX, tl.z + 2, 0);        // imaging sums: tile
}

// A 2-byte snapshot element as a float (the conversion of the per-thread-load kernels).
template <int SK>
__device__ __forceinline__ float h2f(unsigned short u) {
    if constexpr (SK == EFWI_STORE_FP16) return __half2float(__ushort_as_half(u));
    else return __bfloat162float(__ushort_as_bfloat16(u));
}

// Read access to a tile's staged forward velocity: FP32 (SK = 0), or 2-byte FP16/BF16
// snapshot elements times the snapshot's power-of-two scale s, the value the per-thread
// kernels compute from the same element.  at(base, o0, s): element o0 of the array that
// starts at base (shared memory).
template <int SK>
struct FvView {
    using T = typename std::conditional<SK == 0, float, unsigned short>::type;
    const T *p;
    float s;
    __device__ __forceinline__ static FvView at(const float *base, int o0, float s) {
        return {reinterpret_cast<const T *>(base) + o0, s};
    }
    __device__ __forceinline__ FvView operator+(int o) const { return {p + o, s}; }
    __device__ __forceinline__ float operator[](int o) const {
        if constexpr (SK == 0) return p[o];
        else return h2f<SK>(p[o]) * s;
    }
    __device__ __forceinline__ float2 pair(int o) const {   // elements o, o + 1; o even
        if constexpr (SK == 0) {
            return ld2(p + o);
        } else {
            const unsigned int w = *reinterpret_cast<const unsigned int *>(p + o);
            return make_float2(h2f<SK>((unsigned short)(w & 0xffffu)) * s, h2f<SK>((unsigned short)(w >> 16)) * s);
        }
    }
};

// C1 (a - b) + C2 (c - d): the 4th-order staggered difference, one rounding per operation
__device__ __forceinline__ float st4(float a, float b, float c, float d) { return C1 * (a - b) + C2 * (c - d); }

// The arguments of an adjoint step of plan p reading the forward velocities si (k_adjs_tma.cu).
TmaAdjsArgs tma_adjs_args(efwi_plan *p, const SnapIn &si);

}  // namespace efwi
