// What the TMA tile kernels of the forward step share (k_tma.cu, k_tile.cu): arguments, the layout
// of a staged tile and its copies.
#pragma once

#include "das.cuh"
#include "plan.hpp"
#include "tma.cuh"

namespace efwi {

struct TmaFwdArgs {
    const ShotDev *shots;
    const int4 *tiles;
    const FwdMaps *maps;
    int ntiles;
    int scur;                   // state buffer read (z offset 5 * scur in the state map)
    Fields out;                 // state buffer written
    Pml pml;                    // V block = current (read), S block = in place
    float *n1, *n3, *n2, *n4;   // next V block
    float *segx, *segz;
    const float *dw;
    const float *wv;            // w_n / (dx dz) of force sources (null without)
    int nt, n;
    float dt, rdx, rdz;
    int *err;
    int *count;                 // tile counter of the lean kernel (TileFeed)
    int ofield;                 // state-map field of the written buffer's vx (output staging)
    int segf;                   // segment-map field of this step's vx, or -1 (output staging)
    SnapW sw;                   // reduced-precision snapshot work (sw.h / sw.amax null: none)
    DasArgs das;                // lean kernel: traces of the previous step to sample (das.d null: none),
    int ncta, das0, das_ctas;   // CTAs with tiles; first CTA that samples and how many do
    float *esum, *ecmp;         // lean kernel: |v|^2 of the step goes to this compensated sum (null: not)
    int pf;                     // 1: L2 prefetch of the tile one beyond the shared-memory pipeline
};

// Shared-memory stage of one tile.  Fields are staged on the tile + 4-cell halo in x
// (SX columns) and, in z, only on the rows their readers use (halo-4 row coordinates,
// rows 0 .. TZ+7): vx, vz, sigma_xx, b_x, b_z on rows 2 .. TZ+5 (R2 rows), sigma_zz on
// rows 1 .. TZ+7 and sigma_xz on rows 0 .. TZ+6 (R3 rows each); lambda, mu, mu_xz on the
// tile.  Every array starts 128-byte aligned; vx|vz and b_x|b_z are 2-field boxes.
template <int TX, int TZ, int NST, int VEC = 1>
struct FwdLayout {
    static constexpr int SX = TX + 8, SZ = TZ + 8;
    static constexpr int R2 = TZ + 4, R3 = TZ + 7;
    static constexpr int A2 = SX * R2;                              // floats of an R2 field
    static constexpr int A3 = SX * R3, A3P = (A3 + 31) & ~31;       // R3 field, padded to 128 B
    static constexpr int NC = TX * TZ;                              // one tile field
    static constexpr int OVX = 0, OVZ = A2, OSXX = 2 * A2, OSZZ = 3 * A2, OSXZ = OSZZ + A3P,
                         OBX = OSXZ + A3P, OBZ = OBX + A2, OLAM = OBZ + A2;
    static constexpr int BUF = (OLAM + 3 * NC + 31) & ~31;          // floats per stage
    static constexpr unsigned LOADED = (5u * A2 + 2u * A3 + 3u * NC) * 4u;   // bytes the copies bring
    static constexpr size_t smem() { return NST * (size_t)BUF * 4 + 128; }
    static_assert(A2 % 32 == 0, "R2 fields must keep 128-byte alignment");
    static_assert(2 * NC <= 2 * A2, "staged velocities must fit over b_x, b_z");
};

// tl: the tile's work item, already in a register (the issuing thread's refill then has no
// dependent global load between the tile's barriers)
template <int TX, int TZ, int NST, int VEC>
__device__ __forceinline__ void issue_fwd(const TmaFwdArgs &a, const int4 tl, float *buf, uint64_t *bar) {
    using L = FwdLayout<TX, TZ, NST, VEC>;
    const FwdMaps *m = a.maps + tl.x;
    mbar_expect_tx(bar, L::LOADED);
    // element x = cell i + GX (halo-4 column 0 = cell i0 - 4), row y = cell j + GZ: halo-4 row r
    // of the tile is map row j0 - 4 + r + GZ = tl.z - 2 + r
    const int f = 5 * a.scur;
    tma_load_3d(buf + L::OVX, &m->s2, bar, tl.y - 4 + EFWI_GX, tl.z, f);          // vx, vz: rows 2..
    tma_load_3d(buf + L::OSXX, &m->s1, bar, tl.y - 4 + EFWI_GX, tl.z, f + 2);     // sigma_xx: rows 2..
    tma_load_3d(buf + L::OSZZ, &m->s3, bar, tl.y - 4 + EFWI_GX, tl.z - 1, f + 3); // sigma_zz: rows 1..
    tma_load_3d(buf + L::OSXZ, &m->s3, bar, tl.y - 4 + EFWI_GX, tl.z - 2, f + 4); // sigma_xz: rows 0..
    tma_load_3d(buf + L::OBX, &m->mb, bar, tl.y - 4 + EFWI_GX, tl.z, 3);          // b_x, b_z: rows 2..
    tma_load_3d(buf + L::OLAM, &m->mc, bar, tl.y + EFWI_GX, tl.z + 2, 0); // lambda, mu, mu_xz: tile
}

// The arguments of a forward step of plan p (k_tma.cu).
TmaFwdArgs tma_fwd_args(efwi_plan *p, int n, const SnapOut &so);   // das empty

}  // namespace efwi
