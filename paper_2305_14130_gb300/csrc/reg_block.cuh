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
//   * The rows of W and omega sum to 1, so every quantity is shift-invariant: with the pivot c =
//     m_0 the differences e_s = m_s - c are exact in FP32 for components within a factor of two of
//     each other (else a pair of FP32 each), and sum e, sum e^2, sum b' and sum b' e give mean, 1^T
//     r and |r|^2.  The pivot's own residual is -mean, which bounds the cancellation in |r|^2 by a
//     factor of about 2 ns. W changes a component at its sinkhole, so the pivot is one without a
//     sinkhole at the pixel; where all have one, the FP64 sums are shifted by the mean of all
//     components.
//   * The collapse sums b' m itself: no pivot, whose infinity or size (beside a weight of 0) would
//     spoil the others, and no difference that gradients of either sign would round.
//   * A component whose values leave the range in which the products' errors are representable,
//     or which has its sinkhole here, is added in FP64.
// A block takes 256 / G pixels x G groups of components (128-byte rows; a grid of few pixels still fills the
// chip); a thread keeps the m, b', flag and g of its components in registers, so every array is read
// once: 17 B per component, b only where a sinkhole lies.  64 components of 2000 x 600 (1.31 GB): 1.89 ->
// 0.79 ms, a quarter of the HBM bandwidth (1.07 ms where the differences take pairs); collapse 2.45 ->
// 0.50 ms.  Waits for the loads of the next pixels (24 warps per SM, issue slots 40 % used) are what is
// left.  Four blocks per SM (64 registers, spills) took 2 % longer, 16 groups of 4 kept components 19 %.
// G falls with ns (reg_split).
#pragma once

#include <cstdint>
#include <type_traits>

namespace efwi {

constexpr int kRegThreads = 256;

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

// quotient (rb = 1 / b.hi), product and sum of normalised pairs (relative error a few 2^-47)
__device__ __forceinline__ Df df_div(const Df &a, const Df &b, float rb) {
    const float q = a.hi * rb;
    const float r = __fmaf_rn(-q, b.lo, __fmaf_rn(-q, b.hi, a.hi) + a.lo);
    return Df{q, r * rb}.normal();
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
    Df s1, s2, sbe, sb;                      // sum e, e^2, b' e, b' with e = m_s - c
    double x[4] = {0, 0, 0, 0};
};

struct RegShared {
    float f[8 * kRegThreads];                // [group][sum][pixel]
    double x[4 * kRegThreads];
    double B[kRegThreads], BE[kRegThreads], h[kRegThreads], delta[kRegThreads], rwd[kRegThreads];
    float rw[kRegThreads], mh[kRegThreads], ml[kRegThreads];
};

// Pixels [p0, p0 + 256 / G) of one block, the components of a pixel over G threads.  CPT: components
// kept per thread (ns <= G CPT), 0: any ns, the arrays are read again where needed.  COLLAPSE: out[p] =
// collapsed field; else g += gradient (null: none) and the return value is the thread's part of
// sum |r|^2.  Called by every thread of the block with the same arguments.
template <int G, int CPT, bool COLLAPSE>
__device__ double reg_block(const float *__restrict__ m, const float *__restrict__ b, const float *__restrict__ bp,
                            const uint8_t *__restrict__ sink, int ns, long long npix, long long p0, double eta2,
                            float *__restrict__ g, float *__restrict__ out, RegShared &sh) {
    constexpr bool KEEP = CPT > 0;
    constexpr int N = KEEP ? CPT : 1, PX = kRegThreads / G;
    const int px = threadIdx.x % PX, gr = threadIdx.x / PX;
    const long long p = p0 + px;
    const bool live = p < npix;
    // with one thread per pixel nothing is shared and the threads need not meet
    auto sync = [] { if (G > 1) __syncthreads(); };
    auto any_of = [](bool f) { return G > 1 ? __syncthreads_or(f) != 0 : f; };
    // v summed over the pixel's threads, in the order of the groups, on those of group 0 (with more than
    // one group the FP64 additions of all threads would cost more than a barrier) and, with all, on every
    // thread
    auto total = [&](auto &v, bool all) {
        if constexpr (G > 1) {
            constexpr int K = sizeof(v) / sizeof(double);
#pragma unroll
            for (int k = 0; k < K; ++k) sh.x[(gr * K + k) * PX + px] = v[k];
            __syncthreads();
            if (gr == 0)
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    for (int q = 1; q < G; ++q) v[k] += sh.x[(q * K + k) * PX + px];
                    if (all) sh.x[k * PX + px] = v[k];
                }
            if (!all) return;
            __syncthreads();
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = sh.x[k * PX + px];
        }
    };
    float mv[N], bpv[N], gv[N];
    unsigned smask = 0;
    bool any = false;                            // one of the thread's components has its sinkhole here
    float c = !COLLAPSE && live ? m[p] : 0.f;
    if (KEEP) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int s = gr + G * k;
            if (live && s < ns) {
                const long long o = s * npix + p;
                mv[k] = m[o];
                bpv[k] = bp[o];
                if (sink[o] != 0 && ns > 1) smask |= 1u << k;
                if (!COLLAPSE && g) gv[k] = g[o];
            }
        }
        any = smask != 0;
    } else if (live && ns > 1) {
        for (int s = gr; s < ns; s += G) any |= sink[s * npix + p] != 0;
    }
    // body(k, offset, m_s, b'_s, sinkhole flag) over the thread's components
    auto each = [&](auto body) {
        if (!live) return;
        if (KEEP) {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const int s = gr + G * k;
                if (s < ns) body(k, s * npix + p, mv[k], bpv[k], ((smask >> k) & 1u) != 0);
            }
        } else {
            for (int s = gr; s < ns; s += G) {
                const long long o = s * npix + p;
                body(0, o, m[o], bp[o], sink[o] != 0 && ns > 1);
            }
        }
    };
    // f(offset, m_s, b'_s, sinkhole flag) over the thread's components, read again and not unrolled: the
    // few pixels that are added in FP64
    auto wide_each = [&](auto f) {
        if (!live) return;
#pragma unroll 1
        for (int s = gr; s < ns; s += G) {
            const long long o = s * npix + p;
            f(o, m[o], bp[o], sink[o] != 0 && ns > 1);
        }
    };
    // the same with their numbers, over those set in a mask (with KEEP; all otherwise): each thread goes from
    // one of its own to the next, so that a warp takes as many rounds as its busiest thread has components.
    // 8 components of 2000 x 600, a random quarter of the pixels with a sinkhole: collapse 513 -> 326 us (FP64
    // loop 469), term 1540 -> 1150 us (1832)
    auto mask_each = [&](unsigned mask, auto f) {
        if (!live) return;
#pragma unroll 1
        for (int k = 0, s = gr; KEEP ? mask != 0 : s < ns; ++k, s += G, mask &= mask - 1) {
            if (KEEP) {
                k = __ffs(mask) - 1;
                s = gr + G * k;
            }
            const long long o = s * npix + p;
            f(k, o, m[o], bp[o], sink[o] != 0 && ns > 1);
        }
    };

    // 1. where a sinkhole lies: B and sum b_i e_i of the pixel, the pivot from the first component without
    //    a sinkhole here, or, with none, the weighted mean of all (c + h)
    const bool block_sink = any_of(any);
    bool pixel_sink = any;
    if (block_sink) {
        double B[2] = {0, 0};                    // B, sum b_i e_i
        bool all = false;                        // every component has its sinkhole here
        if (!COLLAPSE || G > 1) {
            int first = ns;
            if (live && !COLLAPSE)
                for (int k = 0, s = gr; s < ns && first == ns; ++k, s += G)
                    if (KEEP ? !((smask >> k) & 1u) : sink[s * npix + p] == 0) first = s;
            if (G > 1) {
                sh.f[threadIdx.x] = any ? 1.f : 0.f;
                sh.f[kRegThreads + threadIdx.x] = __int_as_float(first);
                __syncthreads();
                for (int q = 0; q < G; ++q) {
                    pixel_sink |= sh.f[q * PX + px] != 0.f;
                    first = min(first, __float_as_int(sh.f[kRegThreads + q * PX + px]));
                }
            }
            if (!COLLAPSE && pixel_sink) {
                all = first == ns;
                c = m[(first < ns ? first : 0) * npix + p];
            }
        }
        auto add_b = [&](long long o, float ms) {
            const double bs = b[o];
            B[0] += bs;
            B[1] += bs * ((double)ms - (double)c);
        };
        if (pixel_sink) {
            if (G == 1) each([&](int, long long o, float ms, float, bool) { add_b(o, ms); });
            else wide_each([&](long long o, float ms, float, bool) { add_b(o, ms); });
        }
        total(B, false);
        if (gr == 0) {
            sh.B[px] = B[0];
            sh.BE[px] = B[1];
            sh.h[px] = all && B[0] != 0 ? B[1] / B[0] : 0.0;
        }
        sync();
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
        const double v = dc * e + cs * sh.BE[px];
        return COLLAPSE ? v : v - sh.h[px];
    };

    // 2. the sums over the components
    // e = hi + lo exactly (without a pivot e = m_s); false where a product's error would underflow or
    // a sum overflow
    auto diff = [&](float ms, float w, float &hi, float &lo) {
        const float aw = fabsf(w);
        if (COLLAPSE) {
            hi = ms;
            lo = 0.f;
            const float ap = fabsf(w * ms);
            return ((ap >= 1e-30f && ap <= 1e30f) || ms == 0.f) && aw >= 1e-12f && aw <= 1e12f;
        }
        hi = ms - c;
        const float t = hi - ms, ae = fabsf(hi);
        lo = (ms - (hi - t)) - (c + t);
        return (ae == 0.f || (ae >= 1e-12f && ae <= 1e15f)) && (aw == 0.f || (aw >= 1e-12f && aw <= 1e12f));
    };
    RegSums a;
    unsigned rest = 0, wmask = 0;                // components not of the first kind; added in FP64 (KEEP)
    bool spec = false;
    auto add_wide = [&](int, long long o, float ms, float w, bool in) {
        double cs, dc;
        const double v = wide(o, ms, in, cs, dc);
        a.x[0] += v;
        a.x[1] += v * v;
        a.x[2] += (double)w * v;
        a.x[3] += w;
    };
    auto add_high = [&](float eh, float w) {
        a.sb.add(w);
        a.sbe.add_product(w, eh);
        if (!COLLAPSE) {
            a.s1.add(eh);
            a.s2.add_product(eh, eh);
        }
    };
    auto add_other = [&](int k, long long o, float ms, float w, bool in) {
        float eh, el;
        if (diff(ms, w, eh, el) && !in) {
            add_high(eh, w);
            a.s1.lo += el;
            a.s2.lo += el * (2.f * eh + el);
            a.sbe.lo += w * el;
        } else {
            if (KEEP) wmask |= 1u << k;
            else add_wide(k, o, ms, w, in);
            spec = true;
        }
    };
    each([&](int k, long long o, float ms, float w, bool in) {
        float eh, el;
        if (diff(ms, w, eh, el) && el == 0.f && !in) add_high(eh, w);
        else if (KEEP) rest |= 1u << k;
        else add_other(k, o, ms, w, in);
    });
    if (KEEP && rest) mask_each(rest, add_other);
    if (KEEP && wmask) mask_each(wmask, add_wide);
    Df s[4] = {a.s1, a.s2, a.sbe, a.sb};
    if constexpr (G > 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sh.f[(gr * 8 + 2 * k) * PX + px] = s[k].hi;
            sh.f[(gr * 8 + 2 * k + 1) * PX + px] = s[k].lo;
        }
    }
    spec = any_of(spec);                         // uniform over the block, or the thread's own pixel
    if (spec) total(a.x, false);
    double part = 0.0;
    Df mean;                                     // of m under omega
    float rw = 0.f;                              // 1^T r / sum b'
    if (gr == 0) {
        if constexpr (G > 1) {
#pragma unroll
            for (int q = 1; q < G; ++q)
#pragma unroll
                for (int k = 0; k < 4; ++k) s[k].add(Df{sh.f[(q * 8 + 2 * k) * PX + px], sh.f[(q * 8 + 2 * k + 1) * PX + px]});
        }
        if (spec) {
            const double s1 = s[0].value() + a.x[0], s2 = s[1].value() + a.x[1], sbe = s[2].value() + a.x[2],
                         sb = s[3].value() + a.x[3];
            const double delta = sbe / sb;               // mean of W m under omega, minus (c + h)
            if (COLLAPSE) {
                if (live) out[p] = (float)delta;
            } else {
                const double R = s1 - ns * delta;                // 1^T r
                if (live) part = s2 - delta * (s1 + R);          // sum (w - delta)^2
                mean.hi = (float)(c + delta);
                mean.lo = (float)(delta - ((double)mean.hi - (double)c));
                rw = (float)(R / sb);
                sh.delta[px] = delta;
                sh.rwd[px] = R / sb;
            }
        } else {
            // the same in FP32 pairs: an FP64 chain of 30 operations per pixel would cost more than
            // the components' sums
            const Df s1 = s[0].normal(), sb = s[3].normal();
            const float rb = 1.f / sb.hi;
            const Df dd = df_div(s[2].normal(), sb, rb);
            if (COLLAPSE) {
                if (live) out[p] = dd.hi;
            } else {
                const Df nd = df_mul(Df{(float)-ns, 0.f}, dd), R = df_add(s1, nd), t = df_mul(dd, df_add(s1, R));
                const Df q = df_add(s[1].normal(), Df{-t.hi, -t.lo});
                if (live) part = q.value();
                mean = df_add(Df{c, 0.f}, dd);
                rw = df_div(R, sb, rb).hi;
            }
        }
    }
    if (COLLAPSE || !g) {
        sync();                                  // the shared sums are free for the next pixels
        return part;
    }
    if constexpr (G > 1) {
        if (gr == 0) {
            sh.mh[px] = mean.hi;
            sh.ml[px] = mean.lo;
            sh.rw[px] = rw;
        }
        __syncthreads();
        mean = Df{sh.mh[px], sh.ml[px]};
        rw = sh.rw[px];
    }

    // 3. the gradient: omega_s (1^T r) = b'_s rw
    if (block_sink) {
        double cy[1] = {0};
        if (pixel_sink)
            mask_each(wmask, [&](int, long long o, float ms, float w, bool in) {
                if (!in) return;
                double cs, dc;
                const double v = wide(o, ms, in, cs, dc);
                cy[0] += cs * ((v - sh.delta[px]) - (double)w * sh.rwd[px]);
            });
        total(cy, true);
        if (pixel_sink)
            wide_each([&](long long o, float ms, float w, bool in) {
                double cs, dc;
                const double y = (wide(o, ms, in, cs, dc) - sh.delta[px]) - (double)w * sh.rwd[px];
                g[o] = (float)((double)g[o] + eta2 * (dc * y + (double)b[o] * cy[0]));
            });
    }
    if (!pixel_sink) {
        const float e2 = (float)eta2;
        each([&](int k, long long o, float ms, float w, bool) {
            // m_s - mean, rounded once: the difference from the mean's high part is exact within a factor
            // of two
            const float t = ms - mean.hi;
            float r = t - mean.lo;
            if (rest || !KEEP) {
                const float z = t - ms;
                r = t + (((ms - (t - z)) - (mean.hi + z)) - mean.lo);
            }
            g[o] = (KEEP ? gv[k] : g[o]) + e2 * (r - w * rw);
        });
    }
    sync();                                      // the shared sums are free for the next pixels
    return part;
}

// threads of a pixel and components kept by each for ns components (0 kept: too many).  Eight groups
// everywhere left threads without a component, and one warp of eight with the pixels' chains; 2000 x 600,
// FP64 loop of one thread per pixel / 8 groups / this split: 2 components 121 / 167 / 42 us, 4 160 / 177 /
// 58 us, 8 268 / 193 / 111 us, 16 492 / 260 / 199 us; collapse of 2 components 101 / 102 / 18 us, 4 178 / 107
// / 28 us.  From 17 components on fewer groups would keep more than 8 components a thread.
struct RegSplit {
    int groups, cpt;
};
__host__ __device__ constexpr RegSplit reg_split(int ns) {
    return ns <= 2     ? RegSplit{1, 2}
           : ns <= 4   ? RegSplit{1, 4}
           : ns <= 8   ? RegSplit{2, 4}
           : ns <= 16  ? RegSplit{4, 4}
           : ns <= 32  ? RegSplit{8, 4}
           : ns <= 64  ? RegSplit{8, 8}
           : ns <= 128 ? RegSplit{8, 16}
           : ns <= 256 ? RegSplit{8, 32}
                       : RegSplit{8, 0};
}

// blocks per SM asked of the compiler: 24 warps hide the loads up to 64 components; above, the kept
// components take the registers
__host__ __device__ constexpr int reg_blocks(int cpt) { return cpt == 32 ? 1 : cpt == 16 ? 2 : 3; }

// calls f(std::integral_constant<int, G>, std::integral_constant<int, CPT>) for ns components
template <class F>
void reg_dispatch(int ns, F f) {
    const RegSplit r = reg_split(ns);
    auto call = [&](auto g, auto c) {
        if (r.groups == decltype(g)::value && r.cpt == decltype(c)::value) f(g, c);
    };
    using std::integral_constant;
    call(integral_constant<int, 1>(), integral_constant<int, 2>());
    call(integral_constant<int, 1>(), integral_constant<int, 4>());
    call(integral_constant<int, 2>(), integral_constant<int, 4>());
    call(integral_constant<int, 4>(), integral_constant<int, 4>());
    call(integral_constant<int, 8>(), integral_constant<int, 4>());
    call(integral_constant<int, 8>(), integral_constant<int, 8>());
    call(integral_constant<int, 8>(), integral_constant<int, 16>());
    call(integral_constant<int, 8>(), integral_constant<int, 32>());
    call(integral_constant<int, 8>(), integral_constant<int, 0>());
}

}  // namespace efwi
