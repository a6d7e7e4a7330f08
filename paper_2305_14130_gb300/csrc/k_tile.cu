// Forward time step with TMA staging, lean form of k_tma.cu's split cell-pair layout: the same
// persistent grid, 32 x 16 tiles, stages and copies, and the same arithmetic, term by term (all
// variants agree bit for bit), with fewer instructions and waits per cell:
//   * packed FP32 arithmetic on a thread's cell pair (PairOps);
//   * the halo ring of the velocity region as 104 cell pairs instead of 208 single cells;
//   * every position of a thread inside a tile computed once per launch: a tile's shared-memory
//     accesses are one base and constants, its global ones one 32-bit offset;
//   * the CPML memory of an edge tile loaded before the wait for the tile's copies, all of it in
//     flight together, instead of in each half step after the barrier.
// The cell-pair kernel was bound by its warps' barriers and load latencies at 260 instructions a cell
// (205 now; barrier 3.2 and long-scoreboard 2.3 of 10 stalls per instruction are what is left).  32 shots
// of 1000 x 300, keeping v: 176 -> 163 us (68 B a cell without CPML memory: 4.8 TB/s, 70 % of the
// measured HBM bandwidth; copies and stores of 60 B alone, without arithmetic, take 115 us); FP16 snapshots, 8 shots 53 -> 47 us;
// 200 x 100, one shot, with the sampling 8.8 -> 4.8 us, where the chain of a tile's copies, two
// barriers and stores is what is left.  Tried and slower: 64 x 16 tiles in 512 threads, three stages
// with the moduli in registers (195 us), a CTA marching down a strip with its rows in registers (165 to 190 us).
#include <algorithm>
#include <string>
#include <type_traits>

#include "chain.cuh"
#include "fwd_tile.cuh"
#include "pair_ops.cuh"

namespace efwi {
namespace {

constexpr int kThreads = 256, kTX = 32, kTZ = 16, kNST = 2;
using L = FwdLayout<kTX, kTZ, kNST, 2>;
constexpr int kSX = L::SX;
constexpr int kIssue = 224;                      // the thread that issues the copies: on a warp without ring cells
constexpr int kRingRow = kTX / 2 + 2, kRing = 4 * kRingRow + 2 * kTZ;   // cell pairs of the velocity halo ring

// DYN: tiles from the counter (TileFeed), else at a stride of the grid
// EN: the pseudo-Hessian's sum of |v|^2 (k_hessian.cu's expressions on the staged v^{n+1/2}).  A pass
// of its own reads v from memory again and costs a launch per step: 8 shots of 1000 x 300, 300 steps
// 15.4 -> 14.4 ms.
template <int SK, bool DYN, bool EN = false>
__global__ void __launch_bounds__(kThreads, 3) k_step_tile(TmaFwdArgs a, float mz) {
    constexpr bool SNAP = SK != 0;
    extern __shared__ float4 smem_raw[];
    float *smb = align128(smem_raw);
    __shared__ __align__(8) uint64_t bar[kNST];
    __shared__ int ok_s;
    __shared__ int4 next_s;
    __shared__ unsigned wmax_s[2 * (kThreads / 32)];
    const int tid = threadIdx.x;
    auto sample = [&]() {                        // this CTA's share of the previous step's traces
        for (int k = ((int)blockIdx.x - a.das0) * kThreads + tid; k < a.das.ntr; k += a.das_ctas * kThreads)
            das_sample(a.shots, a.das, k);
    };
    if ((int)blockIdx.x >= a.ncta) {
        chain_begin();
        sample();
        return;
    }
    const PairOps op{make_float2(mz, mz)};
    if (tid == 0) {
        for (int b = 0; b < kNST; ++b) mbar_init(&bar[b], 1);
        fence_mbar_init();
    }
    int4 tl = __ldg(a.tiles + blockIdx.x);       // the grid has at most ntiles CTAs
    __syncthreads();
    chain_begin();
    TileFeed feed;
    if (tid == kIssue) {
        issue_fwd<kTX, kTZ, kNST, 2>(a, tl, smb, &bar[0]);
        if (DYN) feed.start(a.ncta, a.tiles, a.ntiles, a.count);
    }
    if (a.das.d && (int)blockIdx.x >= a.das0) sample();
    // this thread's pair of the tile (16 pairs a row) and, on the first 104 threads, its pair of the
    // ring around it (rows -2, -1, 16, 17 over 18 pairs, then one pair left and right of each row)
    const int px = 2 * (tid & 15), py = tid >> 4;
    int rx, ry;
    if (tid < 4 * kRingRow) {
        const int r = tid / kRingRow;
        rx = 2 * (tid - r * kRingRow) - 2;
        ry = r < 2 ? r - 2 : kTZ - 2 + r;
    } else {
        const int r = tid - 4 * kRingRow;
        rx = r & 1 ? kTX : -2;
        ry = r >> 1;
    }
    const bool ring = tid < kRing;
    const int so = (py + 4) * kSX + px + 4, sr = (ry + 4) * kSX + rx + 4;   // halo-4 elements
    const float2 dt2 = PairOps::both(a.dt), rx2 = PairOps::both(a.rdx), rz2 = PairOps::both(a.rdz);
    uint32_t phase = 0;
    int b = 0;
    int t = blockIdx.x + a.ncta;              // the next tile (at a stride)
    for (;; b ^= 1) {
        float *buf = smb + b * L::BUF;
        const ShotDev *sp = a.shots + tl.x;
        const int pitch = __ldg(&sp->pitch);
        const long long off = __ldg(&sp->off);
        const float upx = SNAP && a.sw.h ? snap_scale_up(a.sw.hmax, 0, tl.x, a.sw.ns) : 1.f;
        const float upz = SNAP && a.sw.h ? snap_scale_up(a.sw.hmax, 1, tl.x, a.sw.ns) : 1.f;
        // element of the pair's first cell in a field (fields are smaller than 4 GB: tile_ok)
        const unsigned c0 = (unsigned)off + (unsigned)((tl.z + EFWI_GZ + py) * pitch + tl.y + EFWI_GX + px);

        int4 tl_next = make_int4(-1, 0, 0, 0);
        if (!DYN && t < a.ntiles) tl_next = __ldg(a.tiles + t);
        // false: the wait for the tile's copies gave up
        auto tile = [&](auto edge_c) -> bool {
            constexpr bool edge = decltype(edge_c)::value;   // the tile + 2 cells touches a CPML strip or the grid's edge
            PairPos pos, rpos;
            PairPsi qv, qs, qr;
            if (edge) {
                const int NX = __ldg(&sp->NX), NZ = __ldg(&sp->NZ), P = __ldg(&sp->P);
                const unsigned psx = (unsigned)__ldg(&sp->psx), psz = (unsigned)__ldg(&sp->psz);
                pos = PairPos(tl.y + px, tl.z + py, NX, NZ, P, psx, psz);
                rpos = PairPos(tl.y + rx, tl.z + ry, NX, NZ, P, psx, psz);
                qv = pos.load(a.pml.x[0], a.pml.x[1], a.pml.z[0], a.pml.z[1]);
                qs = pos.load(a.pml.x[2], a.pml.x[3], a.pml.z[2], a.pml.z[3]);
                if (ring) qr = rpos.load(a.pml.x[0], a.pml.x[1], a.pml.z[0], a.pml.z[1]);
            }
            // one thread polls (256 polling the same barrier slow each other down), the others follow
            if (tid == kIssue) ok_s = mbar_wait_bounded(&bar[b], (phase >> b) & 1u);
            __syncthreads();
            if (!ok_s) return false;
            mbar_wait_bounded(&bar[b], (phase >> b) & 1u);   // completed: acquire for every thread
            phase ^= 1u << b;
            // refill the stage of the previous tile: every thread has released it and passed the
            // barrier above
            if (tid == kIssue) {
                if (DYN) next_s = tl_next = feed.next;   // read by every thread after the next barrier
                if (tl_next.x >= 0) issue_fwd<kTX, kTZ, kNST, 2>(a, tl_next, smb + (b ^ 1) * L::BUF, &bar[b ^ 1]);
            }
            const int profx = edge ? __ldg(&sp->profx) : 0;

            // v^{n+1/2} of the pair at halo-4 element o, from v^{n-1/2} = (vxo, vzo)
            auto velocity = [&](const int o, const PairPos &ps, const PairPsi &q, const bool own, float2 &vxo, float2 &vzo,
                                float2 &vx, float2 &vz) {
                const float *sxx = buf + L::OSXX - 2 * kSX + o, *szz = buf + L::OSZZ - kSX + o, *sxz = buf + L::OSXZ + o;
                const float2 xb = ld2(sxx), zb = ld2(sxz);
                float2 e1 = op.mul(op.diff_p(sxx[-1], xb, ld2(sxx + 2)), rx2);
                float2 e2 = op.mul(op.diff(zb, ld2(sxz - kSX), ld2(sxz + kSX), ld2(sxz - 2 * kSX)), rz2);
                float2 e3 = op.mul(op.diff_m(ld2(sxz - 2), zb, sxz[2]), rx2);
                float2 e4 = op.mul(op.diff(ld2(szz + kSX), ld2(szz), ld2(szz + 2 * kSX), ld2(szz - kSX)), rz2);
                if (edge) {
                    const int i = tl.y + o % kSX - 4, j = tl.z + o / kSX - 4;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (ps.x[h]) {
                            const int pq = profx + i + h;
                            const float p1 = a.pml.bx_h[pq] * q.x0[h] + a.pml.ax_h[pq] * half_of(e1, h);
                            const float p3 = a.pml.bx_i[pq] * q.x1[h] + a.pml.ax_i[pq] * half_of(e3, h);
                            if (own) { at_byte(a.n1, ps.kx)[h] = p1; at_byte(a.n3, ps.kx)[h] = p3; }
                            half_of(e1, h) += p1; half_of(e3, h) += p3;
                        }
                    }
                    if (ps.z) {
                        const float bi = a.pml.bz_i[j], ai = a.pml.az_i[j], bh = a.pml.bz_h[j], ah = a.pml.az_h[j];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (!ps.in[h]) continue;
                            const float p2 = bi * q.z0[h] + ai * half_of(e2, h);
                            const float p4 = bh * q.z1[h] + ah * half_of(e4, h);
                            if (own) { at_byte(a.n2, ps.kz)[h] = p2; at_byte(a.n4, ps.kz)[h] = p4; }
                            half_of(e2, h) += p2; half_of(e4, h) += p4;
                        }
                    }
                }
                float *svx = buf + L::OVX - 2 * kSX + o, *svz = buf + L::OVZ - 2 * kSX + o;
                const float2 bx = ld2(buf + L::OBX - 2 * kSX + o), bz = ld2(buf + L::OBZ - 2 * kSX + o);
                vxo = ld2(svx);
                vzo = ld2(svz);
                vx = PairOps::add(vxo, op.mul(op.mul(dt2, bx), PairOps::add(e1, e2)));
                vz = PairOps::add(vzo, op.mul(op.mul(dt2, bz), PairOps::add(e3, e4)));
                if (edge) {
                    if (!ps.in[0]) vx.x = vz.x = 0.f;
                    if (!ps.in[1]) vx.y = vz.y = 0.f;
                }
                if (tl.w & 8) {                          // vector force of this shot (k_force's expression)
                    const int x = o % kSX, y = o / kSX;
                    const int lc = (tl.z - 4 + y + EFWI_GZ) * pitch + (tl.y - 4 + x + EFWI_GX);
                    const float wvn = a.wv[(long long)tl.x * a.nt + a.n];
#pragma unroll 1
                    for (int k = 0; k < 4; ++k) {
                        const int qx = sp->inj_vx[k] - lc, qz = sp->inj_vz[k] - lc;
                        const float fx = sp->fx * wvn * sp->inj_vxw[k], fz = sp->fz * wvn * sp->inj_vzw[k];
                        if (qx == 0) vx.x = vx.x + a.dt * bx.x * fx;
                        if (qx == 1) vx.y = vx.y + a.dt * bx.y * fx;
                        if (qz == 0) vz.x = vz.x + a.dt * bz.x * fz;
                        if (qz == 1) vz.y = vz.y + a.dt * bz.y * fz;
                    }
                }
                st2(svx, vx);
                st2(svz, vz);
            };
            if (ring) {
                float2 vxo, vzo, vx, vz;
                velocity(sr, rpos, qr, false, vxo, vzo, vx, vz);
            }
            // the pair's cells inside the grid (0, 1, 2)
            const int ncell = !edge || pos.in[1] ? 2 : pos.in[0] ? 1 : 0;
            auto put = [&](float *base, const float2 v) {
                float *q = at_byte(base, 4u * c0);
                if (!edge || ncell == 2) st2g(q, v);
                else if (ncell == 1) *q = v.x;
            };
            float2 vxo, vzo, vx, vz;
            velocity(so, pos, qv, true, vxo, vzo, vx, vz);
            put(a.out.vx, vx);
            put(a.out.vz, vz);
            if (a.segx) { put(a.segx, vx); put(a.segz, vz); }
            if (SNAP && a.sw.h) {                        // snapshot of v^{n-1/2}
                if (!edge || ncell == 2) {
                    snap_put2<SK>(a.sw.h, c0, vxo.x * upx, vxo.y * upx);
                    snap_put2<SK>(a.sw.h, a.sw.F + c0, vzo.x * upz, vzo.y * upz);
                } else if (ncell == 1) {
                    snap_put1<SK>(a.sw.h, c0, vxo.x * upx);
                    snap_put1<SK>(a.sw.h, a.sw.F + c0, vzo.x * upz);
                }
            }
            if (SNAP && a.sw.amax)                       // scale of v^{n+1/2} (zero past the grid)
                snap_max_warp(fmaxf(fabsf(vx.x), fabsf(vx.y)), fmaxf(fabsf(vz.x), fabsf(vz.y)), wmax_s);
            __syncthreads();
            if (DYN) {
                tl_next = next_s;
                if (tid == kIssue) feed.advance(a.ncta, a.tiles, a.ntiles, a.count);
            }
            if (SNAP && a.sw.amax && tid == 32) snap_max_commit(wmax_s, a.sw.amax, tl.x, a.sw.ns);

            // sigma^{n+1} of the pair and the moment-tensor source
            if (!edge || ncell > 0) {
                const float *svx = buf + L::OVX - 2 * kSX + so, *svz = buf + L::OVZ - 2 * kSX + so;
                const float2 vb = ld2(svx), wb = ld2(svz);
                if constexpr (EN) {
                    bool phys[2] = {true, true};
                    if (edge) {
                        const int P = __ldg(&sp->P), i = tl.y + px, j = tl.z + py;
                        const bool row = j >= P && j < __ldg(&sp->NZ) - P;
                        for (int h = 0; h < 2; ++h) phys[h] = row && i + h >= P && i + h < __ldg(&sp->NX) - P;
                    }
                    float *es = at_byte(a.esum, 4u * c0), *ec = at_byte(a.ecmp, 4u * c0);
                    float2 sum = make_float2(0.f, 0.f), cmp = sum;
                    if (!edge || (phys[0] && phys[1])) {
                        sum = ld2(es);
                        cmp = ld2(ec);
                    } else {
                        if (phys[0]) { sum.x = es[0]; cmp.x = ec[0]; }
                        if (phys[1]) { sum.y = es[1]; cmp.y = ec[1]; }
                    }
                    const float2 wu = ld2(svz - kSX);
                    auto add = [&](float &s, float &c, float v0, float v1, float w0, float w1) {
                        const float vx = 0.5f * (v0 + v1), vz = 0.5f * (w0 + w1);
                        const float y = (vx * vx + vz * vz) - c, t1 = s + y;
                        c = (t1 - s) - y;
                        s = t1;
                    };
                    add(sum.x, cmp.x, svx[-1], vb.x, wu.x, wb.x);
                    add(sum.y, cmp.y, vb.x, vb.y, wu.y, wb.y);
                    if (!edge || (phys[0] && phys[1])) {
                        st2(es, sum);
                        st2(ec, cmp);
                    } else {
                        if (phys[0]) { es[0] = sum.x; ec[0] = cmp.x; }
                        if (phys[1]) { es[1] = sum.y; ec[1] = cmp.y; }
                    }
                }
                float2 f1 = op.mul(op.diff_m(ld2(svx - 2), vb, svx[2]), rx2);
                float2 f2 = op.mul(op.diff(wb, ld2(svz - kSX), ld2(svz + kSX), ld2(svz - 2 * kSX)), rz2);
                float2 f3 = op.mul(op.diff(ld2(svx + kSX), vb, ld2(svx + 2 * kSX), ld2(svx - kSX)), rz2);
                float2 f4 = op.mul(op.diff_p(svz[-1], wb, ld2(svz + 2)), rx2);
                if (edge) {
                    const int i = tl.y + px, j = tl.z + py;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (pos.x[h]) {
                            const int pq = profx + i + h;
                            const float p5 = a.pml.bx_i[pq] * qs.x0[h] + a.pml.ax_i[pq] * half_of(f1, h);
                            const float p8 = a.pml.bx_h[pq] * qs.x1[h] + a.pml.ax_h[pq] * half_of(f4, h);
                            at_byte(a.pml.x[2], pos.kx)[h] = p5; at_byte(a.pml.x[3], pos.kx)[h] = p8;
                            half_of(f1, h) += p5; half_of(f4, h) += p8;
                        }
                    }
                    if (pos.z) {
                        const float bi = a.pml.bz_i[j], ai = a.pml.az_i[j], bh = a.pml.bz_h[j], ah = a.pml.az_h[j];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (!pos.in[h]) continue;
                            const float p6 = bi * qs.z0[h] + ai * half_of(f2, h);
                            const float p7 = bh * qs.z1[h] + ah * half_of(f3, h);
                            at_byte(a.pml.z[2], pos.kz)[h] = p6; at_byte(a.pml.z[3], pos.kz)[h] = p7;
                            half_of(f2, h) += p6; half_of(f3, h) += p7;
                        }
                    }
                }
                const float *m = buf + L::OLAM + py * kTX + px;
                const float2 lam = ld2(m), m2 = op.mul(PairOps::both(2.f), ld2(m + L::NC)), mxz = ld2(m + 2 * L::NC);
                const float2 tr = op.mul(lam, PairOps::add(f1, f2));
                float2 nxx = PairOps::add(ld2(buf + L::OSXX - 2 * kSX + so),
                                          op.mul(dt2, PairOps::add(tr, op.mul(m2, f1))));
                float2 nzz = PairOps::add(ld2(buf + L::OSZZ - kSX + so), op.mul(dt2, PairOps::add(tr, op.mul(m2, f2))));
                float2 nxz = PairOps::add(ld2(buf + L::OSXZ + so), op.mul(op.mul(dt2, mxz), PairOps::add(f3, f4)));
                if (tl.w & 1) {
                    const float dwn = a.dw[(long long)tl.x * a.nt + a.n];
                    const int lc = (tl.z + py + EFWI_GZ) * pitch + (tl.y + px + EFWI_GX);
#pragma unroll 1
                    for (int k = 0; k < 4; ++k) {
                        const int qn = sp->inj_n[k] - lc, qx = sp->inj_x[k] - lc;
                        const float sx = sp->mxx * dwn * sp->inj_nw[k], sz = sp->mzz * dwn * sp->inj_nw[k],
                                    sc = sp->mxz * dwn * sp->inj_xw[k];
                        if (qn == 0) { nxx.x -= sx; nzz.x -= sz; }
                        if (qn == 1) { nxx.y -= sx; nzz.y -= sz; }
                        if (qx == 0) nxz.x -= sc;
                        if (qx == 1) nxz.y -= sc;
                    }
                }
                put(a.out.sxx, nxx);
                put(a.out.szz, nzz);
                put(a.out.sxz, nxz);
            }
            return true;
        };
        if (!((tl.w & 2) ? tile(std::true_type{}) : tile(std::false_type{}))) {
            if (tid == kIssue) {
                atomicOr(a.err, EFWI_FLAG_TIMEOUT);
                // the copy in flight is this tile's (the next tile's is issued after the wait)
                mbar_drain_bounded(bar, phase, b, kNST, 1);
            }
            return;
        }
        stage_release();
        tl = tl_next;
        t += a.ncta;
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

bool tile_ok(const efwi_plan *p) { return p->fsz_total < (1LL << 30) && p->H < (1LL << 30); }

int tile_blocks_per_sm(int sk, int vec) {
    int nb = 0;
    with_variant(sk, vec == 4, [&](auto k, auto d) {
        constexpr auto kernel = k_step_tile<decltype(k)::value, decltype(d)::value>;
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem());
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        constexpr auto energy = k_step_tile<0, decltype(d)::value, true>;
        cudaFuncSetAttribute(energy, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem());
        cudaFuncSetAttribute(energy, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kThreads, L::smem());
    });
    return std::max(1, nb);
}

void launch_step_tile(efwi_plan *p, int n, const SnapOut &so, const StepMore &more, cudaStream_t st) {
    TmaFwdArgs a = tma_fwd_args(p, n, so);
    a.ncta = std::min(p->grid_fwd_override > 0 ? p->grid_fwd_override : p->tma_grid, a.ntiles);
    int grid = a.ncta;
    if (more.d_prev && p->d.ntr > 0) {
        // CTAs of their own for the traces where all fit on the device at once (on a CTA with tiles
        // the sampling's two dependent loads would lengthen the step); else the last CTAs take them
        // before their tiles.  A launch after the step cost 2 us: 1000 x 300, 32 shots, 300 steps
        // 43.3 -> 42.4 ms, 128 x 128, 4 shots, gradient 13.5 -> 11.6 ms
        a.das = das_args(p, state_fields(p, p->scur), n - 1, more.d_prev);
        a.das_ctas = (p->d.ntr + kThreads - 1) / kThreads;
        if (grid + a.das_ctas <= p->tma_grid) {
            a.das0 = a.ncta;
            grid += a.das_ctas;
        } else {
            a.das_ctas = std::min(a.das_ctas, a.ncta);
            a.das0 = a.ncta - a.das_ctas;
        }
    }
    if (more.esum) {
        a.esum = more.esum;
        a.ecmp = more.ecmp;
        with_variant(EFWI_STORE_FP32, p->tma_vec == 4, [&](auto k, auto d) {
            launch_chained(chain_fwd(p), k_step_tile<0, decltype(d)::value, true>, grid, kThreads, L::smem(), st, a, -0.f);
        });
        return;
    }
    with_variant(p->snap_store, p->tma_vec == 4, [&](auto k, auto d) {
        launch_chained(chain_fwd(p), k_step_tile<decltype(k)::value, decltype(d)::value>, grid, kThreads, L::smem(), st, a, -0.f);
    });
}

}  // namespace efwi
