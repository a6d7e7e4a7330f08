// Adjoint step in scaled-stress form with TMA staging, lean form of k_adjs_tma.cu's cell-pair
// layouts: the same persistent grid, 32 x 16 tiles, stages and copies, and the same arithmetic,
// term by term (all variants of the form agree bit for bit), with fewer instructions per cell:
//   * packed FP32 arithmetic on a thread's cell pair (PairOps);
//   * 384-thread CTAs: the tile's 256 pairs on the first threads, the velocity halo ring as 104
//     pairs on the others;
//   * every position of a thread inside a tile computed once per launch, one 32-bit offset for a
//     pair's elements of every field;
//   * edge tiles: the CPML memory loaded before the wait for the tile's copies, the stress CPML pass
//     on pairs, and F of a tile pair kept in the registers of the thread that updates it.
// 32 shots of 1000 x 300: 266 -> 247 us (108 B a cell: 5.0 TB/s, 74 % of the measured HBM bandwidth);
// FP16 snapshots, 8 shots 75 -> 69 us; 2000 x 600, 4 shots 140 -> 114 us; 200 x 100, one shot
// 10.5 -> 5.8 us.  Two CTAs of two 46 KB stages fill shared memory; the copies in flight bound it.  At the
// 80 registers that two CTAs of 384 threads leave, edge tiles spill (56 bytes a thread at a stride, 76 with
// the counter): the CPML memory of a pair and of two frame pairs is alive across the wait.
#include <algorithm>

#include "adjs_tile.cuh"
#include "chain.cuh"
#include "pair_ops.cuh"

namespace efwi {
namespace {

constexpr int kTX = 32, kTZ = 16, kOwn = kTX / 2 * kTZ, kThreads = 384, kIssue = kThreads - 1;
constexpr int kSX = kTX + 8;
constexpr int kRingRow = kTX / 2 + 2, kRing = 4 * kRingRow + 2 * kTZ;   // pairs of the velocity halo ring
// pairs of the stage's 4-cell frame around the tile: 8 rows, then two pairs on each side
constexpr int kFrameRow = kSX / 2, kFrame = 8 * kFrameRow + 4 * kTZ, kHalo = kThreads - kOwn;
static_assert(kRing <= kHalo && kFrame <= 2 * kHalo, "one ring pair and two frame pairs per halo thread");

template <int SK>
constexpr size_t smem_bytes() {
    return (2 * (size_t)AdjsLayout<kTX, kTZ, SK>::BUF + 3 * AdjsLayout<kTX, kTZ, SK>::A2) * 4 + 128;
}

// halo-4 column and row of frame pair q
__device__ __forceinline__ void frame_pair(int q, int &x, int &y) {
    if (q < 8 * kFrameRow) {
        const int r = q / kFrameRow;
        x = 2 * (q - r * kFrameRow);
        y = r < 4 ? r : kTZ + r;
    } else {
        const int r = q - 8 * kFrameRow, c = r & 3;
        x = c < 2 ? 2 * c : kTX + 2 * c;
        y = 4 + (r >> 2);
    }
}

// DYN: tiles from the counter (TileFeed), else at a stride of the grid
template <int SK, bool DYN>
__global__ void __launch_bounds__(kThreads, 2) k_adj_tile(TmaAdjsArgs a, float mz) {
    using L = AdjsLayout<kTX, kTZ, SK>;
    constexpr int NC = L::NC;
    extern __shared__ float4 smem_raw[];
    float *smb = align128(smem_raw);
    // edge tiles: F_xz with its x-strip CPML term, e^2, e^4
    float *xg4 = smb + 2 * L::BUF - 2 * kSX, *xe2 = xg4 + L::A2, *xe4 = xe2 + L::A2;
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ int ok_s;
    __shared__ int4 next_s;
    const int tid = threadIdx.x;
    const PairOps op{make_float2(mz, mz)};
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    int4 tl = __ldg(a.tiles + blockIdx.x);       // the grid has at most ntiles CTAs
    __syncthreads();
    chain_begin();
    TileFeed feed;
    if (tid == kIssue) {
        issue_adjs<kTX, kTZ, SK>(a, tl, smb, &bar[0]);
        if (DYN) feed.start((int)gridDim.x, a.tiles, a.ntiles, a.count);
    }
    // halo-4 position of the thread's pair of the tile or of the velocity ring
    const bool own = tid < kOwn, ring = !own && tid - kOwn < kRing;
    int x, y;
    if (own) {
        x = 4 + 2 * (tid % (kTX / 2));
        y = 4 + tid / (kTX / 2);
    } else if (tid - kOwn < 4 * kRingRow) {
        const int r = (tid - kOwn) / kRingRow;
        x = 2 + 2 * (tid - kOwn - r * kRingRow);
        y = r < 2 ? 2 + r : kTZ + 2 + r;
    } else {
        const int r = tid - kOwn - 4 * kRingRow;
        x = r & 1 ? kTX + 4 : 2;
        y = 4 + (r >> 1);
    }
    const int o = y * kSX + x;
    const float2 dt2 = PairOps::both(a.dt), rx2 = PairOps::both(a.rdx), rz2 = PairOps::both(a.rdz);
    uint32_t phase = 0;
    int b = 0;
    int t = blockIdx.x + gridDim.x;              // the next tile (at a stride)
    for (;; b ^= 1) {
        float *buf = smb + b * L::BUF;
        const ShotDev *sp = a.shots + tl.x;
        const int pitch = __ldg(&sp->pitch);
        const long long off = __ldg(&sp->off);
        const float dnx = SK ? snap_scale_down(a.hmax, 0, tl.x, a.ns) : 1.f;
        const float dnz = SK ? snap_scale_down(a.hmax, 1, tl.x, a.ns) : 1.f;
        // bytes of the pair's first cell in a field (fields are smaller than 4 GB: tile_ok)
        const unsigned c4 = 4u * ((unsigned)off + (unsigned)((tl.z - 4 + EFWI_GZ + y) * pitch + tl.y - 4 + EFWI_GX + x));

        int4 tl_next = make_int4(-1, 0, 0, 0);
        if (!DYN && t < a.ntiles) tl_next = __ldg(a.tiles + t);
        // false: the wait for the tile's copies gave up
        auto tile = [&](auto edge_c) -> bool {
            constexpr bool edge = decltype(edge_c)::value;   // the 4-cell halo touches a CPML strip or the grid's edge
            PairPos pos, fpos[2];
            PairPsi qv, qs, qf[2];
            int fx[2], fy[2], NX = 0, NZ = 0, PP = 0;
            if (edge) {
                NX = __ldg(&sp->NX); NZ = __ldg(&sp->NZ); PP = __ldg(&sp->P);
                const unsigned psx = (unsigned)__ldg(&sp->psx), psz = (unsigned)__ldg(&sp->psz);
                pos = PairPos(tl.y - 4 + x, tl.z - 4 + y, NX, NZ, PP, psx, psz);
                if (own || ring) qv = pos.load(a.pml.x[0], a.pml.x[1], a.pml.z[0], a.pml.z[1]);
                if (own) {
                    qs = pos.load(a.pml.x[2], a.pml.x[3], a.pml.z[2], a.pml.z[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int q = tid - kOwn + k * kHalo;
                        if (q >= kFrame) continue;
                        frame_pair(q, fx[k], fy[k]);
                        fpos[k] = PairPos(tl.y - 4 + fx[k], tl.z - 4 + fy[k], NX, NZ, PP, psx, psz);
                        qf[k] = fpos[k].load(a.pml.x[2], a.pml.x[3], a.pml.z[2], a.pml.z[3]);
                    }
                }
            }
            if (tid == kIssue) ok_s = mbar_wait_bounded(&bar[b], (phase >> b) & 1u);
            __syncthreads();
            if (!ok_s) return false;
            mbar_wait_bounded(&bar[b], (phase >> b) & 1u);   // completed: acquire for every thread
            phase ^= 1u << b;
            // refill the stage of the previous tile: every thread has released it and passed the
            // barrier above
            if (tid == kIssue) {
                if (DYN) next_s = tl_next = feed.next;   // read by every thread after the next barrier
                if (tl_next.x >= 0) issue_adjs<kTX, kTZ, SK>(a, tl_next, smb + (b ^ 1) * L::BUF, &bar[b ^ 1]);
            }
            const int profx = edge ? __ldg(&sp->profx) : 0;

            // base pointers in halo-4 coordinates
            float *svx = buf + L::OVX - 2 * kSX, *svz = buf + L::OVZ - 2 * kSX;
            float *fxx = buf + L::OFXX - 2 * kSX, *fzz = buf + L::OFZZ - kSX, *fxz = buf + L::OFXZ;
            float *g4 = edge ? xg4 : fxz, *e2w = edge ? xe2 : svx, *e4w = edge ? xe4 : svz;
            const float *sg = buf + L::OG + (y - 4) * kTX + x - 4, *sm = buf + L::OLAM + (y - 4) * kTX + x - 4;
            float2 Fxx, Fzz, Fxz;                            // F of the tile pair before its update

            // 1. edge tiles: the stress-sub-step CPML terms over the staged F, in place (F_xz with its
            //    x-strip term apart), and the tile's adjoint CPML memory
            if constexpr (edge) {
                auto spml = [&](const int xx, const int yy, const PairPos &ps, const PairPsi &q, const bool mine, float2 &Ex,
                                float2 &Ez, float2 &Es) {
                    const int u = yy * kSX + xx, i = tl.y - 4 + xx, j = tl.z - 4 + yy;
                    const bool rxx = mine || (yy >= 2 && yy < kTZ + 6), rzz = mine || yy >= 1, rxz = mine || yy < kTZ + 7;
                    Ex = rxx ? ld2(fxx + u) : make_float2(0.f, 0.f);
                    Ez = rzz ? ld2(fzz + u) : make_float2(0.f, 0.f);
                    Es = rxz ? ld2(fxz + u) : make_float2(0.f, 0.f);
                    float2 g1 = Ex, g2 = Ez, g3 = Es, gg = Es;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (!ps.in[h]) half_of(gg, h) = 0.f;  // the staged F is zero there
                        if (ps.x[h]) {
                            const int pq = profx + i + h;
                            const float s5 = q.x0[h] + half_of(Ex, h), s8 = q.x1[h] + half_of(Es, h);
                            half_of(g1, h) += a.pml.ax_i[pq] * s5;
                            half_of(gg, h) += a.pml.ax_h[pq] * s8;
                            if (mine) {
                                at_byte(a.n5, ps.kx)[h] = a.pml.bx_i[pq] * s5;
                                at_byte(a.n8, ps.kx)[h] = a.pml.bx_h[pq] * s8;
                            }
                        }
                    }
                    if (ps.z) {
                        const float ai = a.pml.az_i[j], ah = a.pml.az_h[j], bi = a.pml.bz_i[j], bh = a.pml.bz_h[j];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (!ps.in[h]) continue;
                            const float s6 = q.z0[h] + half_of(Ez, h), s7 = q.z1[h] + half_of(Es, h);
                            half_of(g2, h) += ai * s6;
                            half_of(g3, h) += ah * s7;
                            if (mine) { at_byte(a.n6, ps.kz)[h] = bi * s6; at_byte(a.n7, ps.kz)[h] = bh * s7; }
                        }
                    }
                    if (rxx) { st2(fxx + u, g1); st2(g4 + u, gg); }
                    if (rzz) st2(fzz + u, g2);
                    if (rxz) st2(fxz + u, g3);
                };
                if (own) {
                    spml(x, y, pos, qs, true, Fxx, Fzz, Fxz);
                } else {
                    float2 d0, d1, d2;
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (tid - kOwn + k * kHalo < kFrame) spml(fx[k], fy[k], fpos[k], qf[k], false, d0, d1, d2);
                }
                __syncthreads();
            }
            const int ncell = !edge || pos.in[1] ? 2 : pos.in[0] ? 1 : 0;   // the pair's cells inside the grid
            auto put = [&](float *base, const float2 v) {
                float *q = at_byte(base, c4);
                if (!edge || ncell == 2) st2g(q, v);
                else if (ncell == 1) *q = v.x;
            };
            const FvView<SK> wvx = FvView<SK>::at(buf + L::OWX, o - 2 * kSX, dnx),
                             wvz = FvView<SK>::at(buf + L::OWZ, o - 2 * kSX, dnz);

            // 2. v^ += D^T f^ on the tile + 2-cell halo; e^ = dt b v^ over the staged v^
            if (own || ring) {
                const float *px = fxx + o, *pz = fzz + o, *ps = fxz + o, *pg = g4 + o;
                const float2 xb = ld2(px), gb = ld2(pg);
                // tx = -(increment of v^_x), tz = -(increment of v^_z)
                const float2 tx = PairOps::add(
                    op.mul(op.diff_p(px[-1], xb, ld2(px + 2)), rx2),
                    op.mul(op.diff(ld2(ps), ld2(ps - kSX), ld2(ps + kSX), ld2(ps - 2 * kSX)), rz2));
                const float2 tz = PairOps::add(
                    op.mul(op.diff(ld2(pz + kSX), ld2(pz), ld2(pz + 2 * kSX), ld2(pz - kSX)), rz2),
                    op.mul(op.diff_m(ld2(pg - 2), gb, pg[2]), rx2));
                const float2 vx = PairOps::sub(ld2(svx + o), tx), vz = PairOps::sub(ld2(svz + o), tz);
                const float2 bx = ld2(buf + L::OBX - 2 * kSX + o), bz = ld2(buf + L::OBZ - 2 * kSX + o);
                float2 h1 = op.mul(op.mul(dt2, bx), vx), h3 = op.mul(op.mul(dt2, bz), vz), h2 = h1, h4 = h3;
                if (edge) {
                    const int i = tl.y - 4 + x, j = tl.z - 4 + y;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (pos.x[h]) {
                            const int pq = profx + i + h;
                            const float s1 = qv.x0[h] + half_of(h1, h), s3 = qv.x1[h] + half_of(h3, h);
                            half_of(h1, h) += a.pml.ax_h[pq] * s1;
                            half_of(h3, h) += a.pml.ax_i[pq] * s3;
                            if (own) {
                                at_byte(a.n1, pos.kx)[h] = a.pml.bx_h[pq] * s1;
                                at_byte(a.n3, pos.kx)[h] = a.pml.bx_i[pq] * s3;
                            }
                        }
                    }
                    if (pos.z) {
                        const float ai = a.pml.az_i[j], ah = a.pml.az_h[j], bi = a.pml.bz_i[j], bh = a.pml.bz_h[j];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (!pos.in[h]) continue;
                            const float s2 = qv.z0[h] + half_of(h2, h), s4 = qv.z1[h] + half_of(h4, h);
                            half_of(h2, h) += ai * s2;
                            half_of(h4, h) += ah * s4;
                            if (own) { at_byte(a.n2, pos.kz)[h] = bi * s2; at_byte(a.n4, pos.kz)[h] = bh * s4; }
                        }
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (!pos.in[h]) half_of(h1, h) = half_of(h2, h) = half_of(h3, h) = half_of(h4, h) = 0.f;
                }
                if (own) {
                    put(a.out.vx, vx);
                    put(a.out.vz, vz);
                    const float2 gx = PairOps::sub(ld2(sg + 3 * NC), op.mul(wvx.pair(0), tx));
                    const float2 gz = PairOps::sub(ld2(sg + 4 * NC), op.mul(wvz.pair(0), tz));
                    if (!edge) {
                        st2g(at_byte(a.Gbx, c4), gx);
                        st2g(at_byte(a.Gbz, c4), gz);
                    } else {
                        const int i = tl.y - 4 + x, j = tl.z - 4 + y;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (i + h >= PP - 1 && i + h <= NX - PP && j >= PP - 1 && j <= NZ - PP) {
                                at_byte(a.Gbx, c4)[h] = half_of(gx, h);
                                at_byte(a.Gbz, c4)[h] = half_of(gz, h);
                            }
                    }
                }
                // each thread reads only its own staged v^ before writing e^ over it
                st2(svx + o, h1);
                st2(svz + o, h3);
                if (edge) { st2(e2w + o, h2); st2(e4w + o, h4); }
            }
            __syncthreads();
            if (DYN) {
                tl_next = next_s;
                if (tid == kIssue) feed.advance((int)gridDim.x, a.tiles, a.ntiles, a.count);
            }

            // 3. F += dt C (-D^T e^) on the tile, with the imaging in F
            if (own && (!edge || ncell > 0)) {
                if (!edge) { Fxx = ld2(fxx + o); Fzz = ld2(fzz + o); Fxz = ld2(fxz + o); }
                {
                    const float2 p0 = wvx.pair(0), q0 = wvz.pair(0);
                    const float2 gx = op.mul(op.diff_m(wvx.pair(-2), p0, wvx[2]), rx2);
                    const float2 gz = op.mul(op.diff(q0, wvz.pair(-kSX), wvz.pair(kSX), wvz.pair(-2 * kSX)), rz2);
                    const float2 gs = PairOps::add(
                        op.mul(op.diff(wvx.pair(kSX), p0, wvx.pair(2 * kSX), wvx.pair(-kSX)), rz2),
                        op.mul(op.diff_p(wvz[-1], q0, wvz.pair(2)), rx2));
                    const float2 nl = PairOps::add(ld2(sg), op.mul(PairOps::add(Fxx, Fzz), PairOps::add(gx, gz)));
                    const float2 nm = PairOps::add(ld2(sg + NC), op.mul(PairOps::sub(Fxx, Fzz), PairOps::sub(gx, gz)));
                    const float2 ns = PairOps::add(ld2(sg + 2 * NC), op.mul(Fxz, gs));
                    if (!edge) {
                        st2g(at_byte(a.Glam, c4), nl);
                        st2g(at_byte(a.Gmu, c4), nm);
                        st2g(at_byte(a.Gmuxz, c4), ns);
                    } else {
                        const int i = tl.y - 4 + x, j = tl.z - 4 + y;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (i + h >= PP && i + h < NX - PP && j >= PP && j < NZ - PP) {
                                at_byte(a.Glam, c4)[h] = half_of(nl, h);
                                at_byte(a.Gmu, c4)[h] = half_of(nm, h);
                            }
                            if (i + h >= PP - 1 && i + h < NX - PP && j >= PP - 1 && j < NZ - PP)
                                at_byte(a.Gmuxz, c4)[h] = half_of(ns, h);
                        }
                    }
                }
                const float *e1 = svx + o, *e3 = svz + o, *e2 = e2w + o, *e4 = e4w + o;
                const float2 E0 = ld2(e1), T0 = ld2(e3);
                // the negated derivatives
                const float2 dxx = op.mul(op.diff_m(ld2(e1 - 2), E0, e1[2]), rx2);
                const float2 dzz = op.mul(op.diff(ld2(e4), ld2(e4 - kSX), ld2(e4 + kSX), ld2(e4 - 2 * kSX)), rz2);
                const float2 dxz = PairOps::add(
                    op.mul(op.diff(ld2(e2 + kSX), ld2(e2), ld2(e2 + 2 * kSX), ld2(e2 - kSX)), rz2),
                    op.mul(op.diff_p(e3[-1], T0, ld2(e3 + 2)), rx2));
                const float2 lam = ld2(sm), l2m = PairOps::add(lam, op.mul(PairOps::both(2.f), ld2(sm + NC)));
                put(a.out.sxx, PairOps::sub(Fxx, op.mul(dt2, PairOps::add(op.mul(l2m, dxx), op.mul(lam, dzz)))));
                put(a.out.szz, PairOps::sub(Fzz, op.mul(dt2, PairOps::add(op.mul(lam, dxx), op.mul(l2m, dzz)))));
                put(a.out.sxz, PairOps::sub(Fxz, op.mul(dt2, op.mul(ld2(sm + 2 * NC), dxz))));
            }
            return true;
        };
        if (!((tl.w & 4) ? tile(std::true_type{}) : tile(std::false_type{}))) {
            if (tid == kIssue) {
                atomicOr(a.err, EFWI_FLAG_TIMEOUT);
                // the copy in flight is this tile's (the next tile's is issued after the wait)
                mbar_drain_bounded(bar, phase, b, 2, 1);
            }
            return;
        }
        stage_release();
        tl = tl_next;
        t += gridDim.x;
        if (tl.x < 0) break;
    }
}

// f(std::integral_constant snapshot kind, std::integral_constant tiles from the counter)
template <class F>
void with_variant(int sk, bool dyn, F f) {
    auto g = [&](auto k) {
        if (dyn) f(k, std::true_type());
        else f(k, std::false_type());
    };
    if (sk == EFWI_STORE_FP16) g(std::integral_constant<int, EFWI_STORE_FP16>());
    else if (sk == EFWI_STORE_BF16) g(std::integral_constant<int, EFWI_STORE_BF16>());
    else g(std::integral_constant<int, 0>());
}

}  // namespace

int adj_tile_blocks_per_sm(int sk, int vec) {
    int nb = 0;
    with_variant(sk, vec == 4, [&](auto k, auto d) {
        constexpr int K = decltype(k)::value;
        constexpr auto kernel = k_adj_tile<K, decltype(d)::value>;
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<K>());
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kThreads, smem_bytes<K>());
    });
    return std::max(1, nb);
}

void launch_adj_tile(efwi_plan *p, const SnapIn &si, cudaStream_t st) {
    const TmaAdjsArgs a = tma_adjs_args(p, si);
    const int grid = std::min(p->grid_adj_override > 0 ? p->grid_adj_override : p->tma_adj_grid, a.ntiles);
    with_variant(p->snap_store, p->adjs_vec == 4, [&](auto k, auto d) {
        constexpr int K = decltype(k)::value;
        launch_chained(chain_adj(p), k_adj_tile<K, decltype(d)::value>, grid, kThreads, smem_bytes<K>(), st, a, -0.f);
    });
}

}  // namespace efwi
