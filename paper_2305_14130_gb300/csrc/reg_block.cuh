// Consistency term of the extended model (eqs. 8, 11, 12) and its collapse (eqs. 9, 15),
// shared by the plan's kernels and the allocation-free one.  Per pixel, over the ns components:
//   B = sum b_i;  c_s = (1 - b_s)/(B - b_s) inside sink_s else 0;  d_s = b_s inside else 1
//   (W m)_s = (d_s - c_s b_s) m_s + c_s sum_i b_i m_i              (eq. 11)
//   omega_s = b'_s / sum b'                                        (eq. 12)
//   r = (I - 1 omega^T) W m;  phi += 1/2 eta^2 |r|^2
//   y = r - omega (1^T r);  g_i += eta^2 [(d_i - c_i b_i) y_i + b_i sum_s c_s y_s]
//   collapse: omega^T W m
//
// The residual is the small difference of nearly equal components, so its sums need more than
// FP32.  GB300 does about 2 FP64 operations per SM and clock, and 11 of them per component
// (conversions included) bounded the former FP64 loop (64 components of 2000 x 600: 1.95 ms, 10 %
// of the HBM bandwidth).  Here the sums run in FP32 with their rounding errors carried along
// (two-sum, two-product; Knuth, Dekker), and the few FP64 operations left are per pixel:
//   * The rows of W and omega sum to 1, so every quantity is shift-invariant: with the pivot
//     c = m_0 the differences e_s = m_s - c are exact in FP32 for components within a factor of
//     two of each other, and sum e, sum e^2, sum b' and sum b' e give mean, 1^T r and |r|^2.  The
//     pivot's own residual is -mean, which bounds the cancellation in |r|^2 by a factor of about 2 ns.
//     W changes a component at its sinkhole, so the pivot is one without a sinkhole at the pixel;
//     where all have one, the FP64 sums are shifted by the mean of all components.
//   * The collapse sums b' m itself: no pivot, whose infinity or size (beside a weight of 0) would
//     spoil the others, and no difference that gradients of either sign would round.
//   * A component whose difference is not exact, whose values leave the range in which the
//     products' errors are representable, or which has its sinkhole here, is added in FP64.
// A block takes 32 pixels x 8 groups of components (128-byte rows; a grid of few pixels
// still fills the chip); a thread keeps the m, b', flag and g of its components in registers, so
// every array is read once: 17 B per component, b only where a sinkhole lies.  64 components of
// 2000 x 600 (1.31 GB): 1.95 -> 0.72 ms, a quarter of the HBM bandwidth; waits for the loads of the
// next pixels (24 warps per SM, issue slots 40 % used) are what is left.  Four blocks per SM (64
// registers, spills) took 2 % longer, 16 groups of 4 kept components 19 %.
#pragma once

#include <cstdint>
#include <type_traits>

namespace efwi {

constexpr int kRegPx = 32, kRegGroups = 8, kRegThreads = kRegPx * kRegGroups;

// Unevaluated sum hi + lo of an FP32 accumulation and the errors of its additions.
struct Df {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float s = hi + x, t = s - hi;
        lo += (hi - (s - t)) + (x - t);
        hi = s;
    }
    __device__ __forceinline__ void add_product(float a, float b) {
        const float p = a * b;
        lo += __fmaf_rn(a, b, -p);
        add(p);
    }
    __device__ __forceinline__ void add(const Df &o) {
        add(o.hi);
        lo += o.lo;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
    // |hi| >= |lo| again
    __device__ __forceinline__ Df normal() const {
        const float s = hi + lo;
        return {s, lo - (s - hi)};
    }
};

// quotient, product and sum of normalised pairs (relative error a few 2^-47)
__device__ __forceinline__ Df df_div(const Df &a, const Df &b) {
    const float q = a.hi / b.hi;
    const float r = __fmaf_rn(-q, b.lo, __fmaf_rn(-q, b.hi, a.hi) + a.lo);
    return Df{q, r / b.hi}.normal();
}
__device__ __forceinline__ Df df_mul(const Df &a, const Df &b) {
    const float p = a.hi * b.hi;
    const float e = __fmaf_rn(a.hi, b.hi, -p);
    return Df{p, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e))}.normal();
}
__device__ __forceinline__ Df df_add(Df a, const Df &b) {
    a.add(b);
    return a.normal();
}

// FP32 sums of one thread's components, and the FP64 sums of those that need FP64
struct RegSums {
    Df s1, s2, sbe, sb;                      // sum w, w^2, b' w, b' with w = (W m)_s - c
    double x1 = 0, x2 = 0, xbe = 0, xb = 0;
};

struct RegShared {
    float f[kRegGroups][8][kRegPx];
    double x[kRegGroups][4][kRegPx];
    double B[kRegPx], BE[kRegPx], h[kRegPx], delta[kRegPx], rwd[kRegPx];
    int first[kRegGroups][kRegPx];
    float rw[kRegPx], dh[kRegPx], dl[kRegPx];
};

// Pixels [p0, p0 + 32) of one block.  CPT: components kept per thread (ns <= 8 CPT), 0: any ns,
// the arrays are read again where needed.  COLLAPSE: out[p] = collapsed field; else g += gradient
// (null: none) and the return value is the thread's part of sum |r|^2 (only group 0 has one).
// Called by every thread of the block with the same arguments.
template <int CPT, bool COLLAPSE>
__device__ double reg_block(const float *__restrict__ m, const float *__restrict__ b, const float *__restrict__ bp,
                            const uint8_t *__restrict__ sink, int ns, long long npix, long long p0, double eta2,
                            float *__restrict__ g, float *__restrict__ out, RegShared &sh) {
    constexpr bool KEEP = CPT > 0;
    constexpr int N = KEEP ? CPT : 1;
    const int px = threadIdx.x % kRegPx, gr = threadIdx.x / kRegPx;
    const long long p = p0 + px;
    const bool live = p < npix;
    float mv[N], bpv[N], gv[N];
    unsigned smask = 0;
    bool any = false;
    float c = !COLLAPSE && live ? m[p] : 0.f;
    if (KEEP) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int s = gr + kRegGroups * k;
            if (live && s < ns) {
                const long long o = s * npix + p;
                mv[k] = m[o];
                bpv[k] = bp[o];
                if (sink[o] != 0) smask |= 1u << k;
                if (!COLLAPSE && g) gv[k] = g[o];
            }
        }
        any = smask != 0;
    } else if (live) {
        for (int s = gr; s < ns; s += kRegGroups) any |= sink[s * npix + p] != 0;
    }
    // body(k, s, offset, m_s, b'_s, sinkhole flag) over the thread's components
    auto each = [&](auto body) {
        if (!live) return;
        if (KEEP) {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const int s = gr + kRegGroups * k;
                if (s < ns) body(k, s, s * npix + p, mv[k], bpv[k], ((smask >> k) & 1u) != 0 && ns > 1);
            }
        } else {
            for (int s = gr; s < ns; s += kRegGroups) {
                const long long o = s * npix + p;
                body(0, s, o, m[o], bp[o], sink[o] != 0 && ns > 1);
            }
        }
    };
    // m_s - c (the collapse: m_s), and whether it and the products formed from it are safe in FP32
    auto diff = [&](float ms, float w, float &e) {
        const float aw = fabsf(w);
        if (COLLAPSE) {
            e = ms;
            const float ap = fabsf(w * ms);
            return ((ap >= 1e-30f && ap <= 1e30f) || ms == 0.f) && aw >= 1e-12f && aw <= 1e12f;
        }
        e = ms - c;
        const float t = e - ms, err = (ms - (e - t)) - (c + t);
        const float ae = fabsf(e);
        return err == 0.f && (ae == 0.f || (ae >= 1e-12f && ae <= 1e15f)) && (aw == 0.f || (aw >= 1e-12f && aw <= 1e12f));
    };
    // f(s, offset, m_s, b'_s, sinkhole flag) over the components set in a mask (with KEEP; all
    // otherwise), read again and not unrolled: the few that are added in FP64
    auto wide_each = [&](unsigned mask, auto f) {
        if (!live) return;
#pragma unroll 1
        for (int k = 0, s = gr; s < ns; ++k, s += kRegGroups) {
            if (KEEP && !((mask >> k) & 1u)) continue;
            const long long o = s * npix + p;
            f(o, m[o], bp[o], sink[o] != 0 && ns > 1);
        }
    };

    // 1. where a sinkhole lies: the pivot, B and sum b_i e_i of its pixel
    const bool block_sink = __syncthreads_or(any && ns > 1) != 0;
    bool pixel_sink = false;
    if (block_sink) {
        int first = ns;                          // of the thread's components, without a sinkhole here
        if (live)
            for (int k = 0, s = gr; s < ns && first == ns; ++k, s += kRegGroups)
                if (KEEP ? !((smask >> k) & 1u) : sink[s * npix + p] == 0) first = s;
        sh.first[gr][px] = any ? -1 - first : first;
        __syncthreads();
        first = ns;
        for (int q = 0; q < kRegGroups; ++q) {
            const int f = sh.first[q][px];
            pixel_sink |= f < 0;
            first = min(first, f < 0 ? -1 - f : f);
        }
        if (!COLLAPSE && pixel_sink) c = m[(first < ns ? first : 0) * npix + p];
        double vb = 0, ve = 0;
        if (pixel_sink)
            wide_each(~0u, [&](long long o, float ms, float, bool) {
                const double bs = b[o];
                vb += bs;
                ve += bs * ((double)ms - (double)c);
            });
        sh.x[gr][0][px] = vb;
        sh.x[gr][1][px] = ve;
        __syncthreads();
        if (gr == 0) {
            double B = 0, BE = 0;
            for (int q = 0; q < kRegGroups; ++q) { B += sh.x[q][0][px]; BE += sh.x[q][1][px]; }
            sh.B[px] = B;
            sh.BE[px] = BE;
            sh.h[px] = !COLLAPSE && pixel_sink && first == ns && B != 0 ? BE / B : 0.0;
        }
        __syncthreads();
    }
    // w = (W m)_s - (c + h) in FP64, c_s and d_s - c_s b_s
    auto wide = [&](long long o, float ms, bool in, double &cs, double &dc) {
        const double e = (double)ms - (double)c;
        cs = 0.0;
        dc = 1.0;
        if (!in) return e;
        const double bs = b[o];
        cs = (1.0 - bs) / (sh.B[px] - bs);
        dc = bs - cs * bs;
        return dc * e + cs * sh.BE[px] - sh.h[px];
    };

    // 2. the sums over the components
    RegSums a;
    unsigned wmask = 0;                          // components added in FP64 (KEEP)
    bool spec = false;
    auto add_wide = [&](long long o, float ms, float w, bool in) {
        double cs, dc;
        const double v = wide(o, ms, in, cs, dc);
        a.x1 += v;
        a.x2 += v * v;
        a.xbe += (double)w * v;
        a.xb += w;
    };
    each([&](int k, int, long long o, float ms, float w, bool in) {
        float e;
        if (diff(ms, w, e) && !in) {
            a.sb.add(w);
            if (!COLLAPSE) {
                a.s1.add(e);
                a.s2.add_product(e, e);
            }
            a.sbe.add_product(w, e);
        } else {
            if (KEEP) wmask |= 1u << k;
            else add_wide(o, ms, w, in);
            spec = true;
        }
    });
    if (KEEP && wmask) wide_each(wmask, add_wide);
    sh.f[gr][0][px] = a.s1.hi; sh.f[gr][1][px] = a.s1.lo;
    sh.f[gr][2][px] = a.s2.hi; sh.f[gr][3][px] = a.s2.lo;
    sh.f[gr][4][px] = a.sbe.hi; sh.f[gr][5][px] = a.sbe.lo;
    sh.f[gr][6][px] = a.sb.hi; sh.f[gr][7][px] = a.sb.lo;
    if (__syncthreads_or(spec)) {                // block-uniform
        sh.x[gr][0][px] = a.x1;
        sh.x[gr][1][px] = a.x2;
        sh.x[gr][2][px] = a.xbe;
        sh.x[gr][3][px] = a.xb;
        spec = true;
        __syncthreads();
    }
    double part = 0.0;
    if (gr == 0) {
        Df s[4];
#pragma unroll
        for (int q = 0; q < kRegGroups; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) s[k].add(Df{sh.f[q][2 * k][px], sh.f[q][2 * k + 1][px]});
        if (spec) {
            double s1 = s[0].value(), s2 = s[1].value(), sbe = s[2].value(), sb = s[3].value();
            for (int q = 0; q < kRegGroups; ++q) {
                s1 += sh.x[q][0][px];
                s2 += sh.x[q][1][px];
                sbe += sh.x[q][2][px];
                sb += sh.x[q][3][px];
            }
            const double delta = sbe / sb;       // mean of W m under omega, minus c
            if (COLLAPSE) {
                if (live) out[p] = (float)delta;
            } else {
                const double R = s1 - ns * delta;                // 1^T r
                if (live) part = s2 - delta * (s1 + R);          // sum (w - delta)^2
                const float dh = (float)delta;
                sh.delta[px] = delta;
                sh.dh[px] = dh;
                sh.dl[px] = (float)(delta - (double)dh);
                sh.rwd[px] = R / sb;
                sh.rw[px] = (float)(R / sb);
            }
        } else {
            // the same in FP32 pairs: an FP64 chain of 30 operations per pixel would cost more than
            // the components' sums
            const Df s1 = s[0].normal(), sb = s[3].normal(), delta = df_div(s[2].normal(), sb);
            if (COLLAPSE) {
                if (live) out[p] = delta.hi;
            } else {
                const Df nd = df_mul(Df{(float)-ns, 0.f}, delta), R = df_add(s1, nd), t = df_mul(delta, df_add(s1, R));
                const Df q = df_add(s[1].normal(), Df{-t.hi, -t.lo});
                if (live) part = q.value();
                sh.dh[px] = delta.hi;
                sh.dl[px] = delta.lo;
                sh.rw[px] = R.hi / sb.hi;
            }
        }
    }
    if (COLLAPSE || !g) {
        __syncthreads();                         // the shared sums are free for the next pixels
        return part;
    }
    __syncthreads();

    // 3. the gradient: omega_s (1^T r) = b'_s rw
    const float dh = sh.dh[px], dl = sh.dl[px], rw = sh.rw[px], e2 = (float)eta2;
    const double delta = spec ? sh.delta[px] : 0.0;
    if (block_sink) {
        double cy = 0;
        if (pixel_sink)
            wide_each(wmask, [&](long long o, float ms, float w, bool in) {
                if (!in) return;
                double cs, dc;
                const double v = wide(o, ms, in, cs, dc);
                cy += cs * ((v - delta) - (double)w * sh.rwd[px]);
            });
        sh.x[gr][0][px] = cy;
        __syncthreads();
    }
    if (pixel_sink) {
        double cy = 0;
        for (int q = 0; q < kRegGroups; ++q) cy += sh.x[q][0][px];
        wide_each(~0u, [&](long long o, float ms, float w, bool in) {
            double cs, dc;
            const double y = (wide(o, ms, in, cs, dc) - delta) - (double)w * sh.rwd[px];
            g[o] = (float)((double)g[o] + eta2 * (dc * y + (double)b[o] * cy));
        });
    } else if (KEEP) {
        each([&](int k, int, long long o, float ms, float w, bool) {
            if (!((wmask >> k) & 1u)) g[o] = gv[k] + e2 * ((((ms - c) - dh) - dl) - w * rw);
        });
        if (wmask)
            wide_each(wmask, [&](long long o, float ms, float w, bool) {
                g[o] = g[o] + e2 * ((float)(((double)ms - (double)c) - delta) - w * rw);
            });
    } else {
        each([&](int, int, long long o, float ms, float w, bool) {
            float e;
            const float r = diff(ms, w, e) ? (e - dh) - dl : (float)(((double)ms - (double)c) - delta);
            g[o] = g[o] + e2 * (r - w * rw);
        });
    }
    __syncthreads();                             // the shared sums are free for the next pixels
    return part;
}

// components kept per thread for ns components (0: too many to keep)
__host__ __device__ constexpr int reg_cpt(int ns) {
    return ns <= 16 ? 2 : ns <= 32 ? 4 : ns <= 64 ? 8 : ns <= 128 ? 16 : ns <= 256 ? 32 : 0;
}

// blocks per SM asked of the compiler: 24 warps hide the loads up to 64 components; above, the kept
// components take the registers
__host__ __device__ constexpr int reg_blocks(int cpt) { return cpt == 32 ? 1 : cpt == 16 ? 2 : 3; }

// calls f(std::integral_constant<int, CPT>) for ns components
template <class F>
void reg_dispatch(int ns, F f) {
    switch (reg_cpt(ns)) {
        case 2: f(std::integral_constant<int, 2>()); break;
        case 4: f(std::integral_constant<int, 4>()); break;
        case 8: f(std::integral_constant<int, 8>()); break;
        case 16: f(std::integral_constant<int, 16>()); break;
        case 32: f(std::integral_constant<int, 32>()); break;
        default: f(std::integral_constant<int, 0>()); break;
    }
}

}  // namespace efwi
