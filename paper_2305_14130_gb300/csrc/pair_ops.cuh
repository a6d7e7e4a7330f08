// Packed FP32 arithmetic on two adjacent cells.
#pragma once

namespace efwi {

// GB300 adds and multiplies pairs of FP32 in one instruction, each half rounded as the scalar
// operation, which halves the issue slots of the stencils' arithmetic.  The compiler contracts a
// packed product whose only use is a packed sum into a multiply-add, even with contraction off and
// explicit rounding in the PTX, which would round differently from the scalar kernels; a product is
// therefore written as fma(a, b, -0) with a -0 that the compiler does not know (a kernel argument),
// which rounds as the product.
struct PairOps {
    float2 mz;                                   // (-0, -0)
    __device__ __forceinline__ static float2 fma(float2 a, float2 b, float2 c) {
        float2 r;
        asm("{\n\t.reg .b64 x, y, z, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 w, {%6, %7};\n\t"
            "fma.rn.f32x2 z, x, y, w;\n\tmov.b64 {%0, %1}, z;\n\t}"
            : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
        return r;
    }
    __device__ __forceinline__ static float2 both(float v) { return make_float2(v, v); }
    __device__ __forceinline__ float2 mul(float2 a, float2 b) const { return fma(a, b, mz); }
    __device__ __forceinline__ static float2 add(float2 a, float2 b) {
        float2 r;
        asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
            "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
            : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
        return r;
    }
    __device__ __forceinline__ static float2 sub(float2 a, float2 b) { return fma(b, both(-1.f), a); }   // a - b
    // C1 x + C2 y: the 4th-order staggered difference from x = a - b, y = c - d
    __device__ __forceinline__ float2 comb(float2 x, float2 y) const {
        return add(mul(both(C1), x), mul(both(C2), y));
    }
    // C1 (a - b) + C2 (c - d)
    __device__ __forceinline__ float2 diff(float2 a, float2 b, float2 c, float2 d) const {
        return comb(sub(a, b), sub(c, d));
    }
    // C1 (f[1] - f[0]) + C2 (f[2] - f[-1]) of cells c, from the cell before and the two after
    __device__ __forceinline__ float2 diff_p(float m1, float2 c, float2 p) const {
        return comb(make_float2(c.y - c.x, p.x - c.y), make_float2(p.x - m1, p.y - c.x));
    }
    // C1 (f[0] - f[-1]) + C2 (f[1] - f[-2]) of cells c, from the two before and the one after
    __device__ __forceinline__ float2 diff_m(float2 m, float2 c, float p0) const {
        return comb(make_float2(c.x - m.y, c.y - c.x), make_float2(c.y - m.x, p0 - m.y));
    }
};

__device__ __forceinline__ float &half_of(float2 &q, int h) { return h ? q.y : q.x; }
__device__ __forceinline__ float half_of(const float2 &q, int h) { return h ? q.y : q.x; }

// element of a field smaller than 4 GB at a byte offset
__device__ __forceinline__ float *at_byte(float *base, unsigned bytes) {
    return reinterpret_cast<float *>(reinterpret_cast<char *>(base) + bytes);
}

// Tiles of a persistent grid handed out by a counter in device memory as CTAs become free (the first
// ncta, their number, statically).  With a fixed stride instead, a CTA meets only a few tile columns when the
// grid and the tiles per row share factors, and those that hold the slower CPML tiles finish last
// (adjoint, 32 shots of 1000 x 300 with 1 CPML cell, 32 tiles per row on 304 CTAs: 292 us against
// 194 us with the counter); where they share none the stride balances by itself and needs no work
// item through shared memory (20 CPML cells, 33 tiles per row: 247 us against 261 us).  The lean
// kernels are compiled for both and the autotuner times them.  One thread of the CTA owns the feed;
// the counter is read two tiles ahead and the work item one tile ahead, so neither latency is waited
// for.  Every CTA draws exactly one number past the end; the last of these leaves the counter at zero
// for the next launch.
struct TileFeed {
    int4 next;                   // the CTA's next work item (x < 0: none)
    int q;                       // number drawn for the one after
    __device__ __forceinline__ void draw(int ncta, const int4 *tiles, int ntiles, int *count) {
        const int t = ncta + q;
        if (t < ntiles) {
            next = __ldg(tiles + t);
            q = atomicAdd(count, 1);
        } else {
            if (q == ntiles - 1) *count = 0;
            next.x = -1;
        }
    }
    __device__ __forceinline__ void start(int ncta, const int4 *tiles, int ntiles, int *count) {
        q = atomicAdd(count, 1);
        draw(ncta, tiles, ntiles, count);
    }
    // the work item after `next` becomes `next`
    __device__ __forceinline__ void advance(int ncta, const int4 *tiles, int ntiles, int *count) {
        if (next.x >= 0) draw(ncta, tiles, ntiles, count);
    }
};

// CPML memory of a cell pair: psi of the x strips (two arrays) and of the z strips (two arrays)
struct PairPsi {
    float x0[2], x1[2], z0[2], z1[2];
};

// Position of a cell pair against the grid and the CPML strips.  The strip elements of its two
// cells are adjacent (no pair touches both x strips: they are at least one column apart).
struct PairPos {
    bool in[2], x[2], z;        // inside the grid; in an x strip; the row in a z strip
    unsigned kx, kz;            // bytes of the first cell's element in the x- and z-strip arrays
    __device__ __forceinline__ PairPos() {}
    __device__ __forceinline__ PairPos(int i, int j, int NX, int NZ, int P, unsigned psx, unsigned psz) {
        const bool row = j >= 0 && j < NZ;
        z = row && (j < P || j >= NZ - P);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            in[h] = row && i + h >= 0 && i + h < NX;
            x[h] = in[h] && (i + h < P || i + h >= NX - P);
        }
        kx = 4u * (psx + (unsigned)(j * 2 * P + (i < P ? i : i - NX + 2 * P)));
        kz = 4u * (psz + (unsigned)((j < P ? j : j - NZ + 2 * P) * NX + i));
    }
    __device__ __forceinline__ PairPsi load(float *x0, float *x1, float *z0, float *z1) const {
        PairPsi q;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            q.x0[h] = x[h] ? at_byte(x0, kx)[h] : 0.f;
            q.x1[h] = x[h] ? at_byte(x1, kx)[h] : 0.f;
            q.z0[h] = z && in[h] ? at_byte(z0, kz)[h] : 0.f;
            q.z1[h] = z && in[h] ? at_byte(z1, kz)[h] : 0.f;
        }
        return q;
    }
};

}  // namespace efwi
