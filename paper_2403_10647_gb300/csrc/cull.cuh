// The triangle / cell overlap test of the culling mode, shared by the kernels
// that cull.
#pragma once

#include "device.cuh"

namespace gg {

// A triangle in grid space: vertices q (q[3k + a]), edges e_0 = q_1 - q_0,
// e_1 = q_2 - q_1, e_2 = q_0 - q_2 and the normal n = e_0 x e_1.
struct GridTri {
    float q[9];
    float e[9];
    float n[3];
};

// Grid coordinates q = min((v - lo) * scale, res): the cell mapping's two
// FP32 operations and its clamp to the grid's far face (the FP32 scale can put
// the far face's vertices a rounding error beyond res).
__device__ __forceinline__ void grid_tri(const float *__restrict__ verts, long long nverts,
                                         const int *__restrict__ tris, unsigned o, const float (&lo)[3],
                                         const float (&scale)[3], const float (&resf)[3], GridTri &t, Ctl *ctl)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int vi = __ldg(tris + 3ll * o + k);
        if (vi < 0 || (long long)vi >= nverts) {   // never read outside verts: flag and use vertex 0
            atomicOr(&ctl->err, ERR_BADINDEX);
            vi = 0;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
            t.q[3 * k + a] = fminf(__fmul_rn(__fsub_rn(__ldg(verts + 3ll * vi + a), lo[a]), scale[a]), resf[a]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t.e[a] = __fsub_rn(t.q[3 + a], t.q[a]);
        t.e[3 + a] = __fsub_rn(t.q[6 + a], t.q[3 + a]);
        t.e[6 + a] = __fsub_rn(t.q[a], t.q[6 + a]);
    }
    t.n[0] = __fsub_rn(__fmul_rn(t.e[1], t.e[5]), __fmul_rn(t.e[2], t.e[4]));
    t.n[1] = __fsub_rn(__fmul_rn(t.e[2], t.e[3]), __fmul_rn(t.e[0], t.e[5]));
    t.n[2] = __fsub_rn(__fmul_rn(t.e[0], t.e[4]), __fmul_rn(t.e[1], t.e[3]));
}

// One separating axis a against the cell: projections of the local vertices
// w, box radius S / 2 widened by the slack S t.  Each product and sum is one
// round-to-nearest FP32 operation in a fixed order, so the decision is the
// same on every IEEE machine.
__device__ __forceinline__ bool axis_separates(float a0, float a1, float a2, const float (&w)[9], float t)
{
    float pmin = 0.0f, pmax = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float p = __fadd_rn(__fmul_rn(a0, w[3 * k]), __fmul_rn(a1, w[3 * k + 1]));
        p = __fadd_rn(p, __fmul_rn(a2, w[3 * k + 2]));
        pmin = k == 0 ? p : fminf(pmin, p);
        pmax = k == 0 ? p : fmaxf(pmax, p);
    }
    const float S = __fadd_rn(__fadd_rn(fabsf(a0), fabsf(a1)), fabsf(a2));
    const float R = __fadd_rn(__fmul_rn(0.5f, S), __fmul_rn(S, t));
    return pmin > R || pmax < -R;
}

// The same for an axis with one zero component, a0 and a1 its others and i, j
// their coordinates: the products with zero add nothing to the projections
// and sums above (all operands are finite), so they are left out.
__device__ __forceinline__ bool axis2_separates(float a0, float a1, int i, int j, const float (&w)[9], float t)
{
    float pmin = 0.0f, pmax = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float p = __fadd_rn(__fmul_rn(a0, w[3 * k + i]), __fmul_rn(a1, w[3 * k + j]));
        pmin = k == 0 ? p : fminf(pmin, p);
        pmax = k == 0 ? p : fmaxf(pmax, p);
    }
    const float S = __fadd_rn(fabsf(a0), fabsf(a1));
    const float R = __fadd_rn(__fmul_rn(0.5f, S), __fmul_rn(S, t));
    return pmin > R || pmax < -R;
}

// Axes that can separate a cell of the triangle's cell box: bit 0 the
// normal, bit 1 + 3 j + f the f-th cross product with edge j.  An axis with
// at most one non-zero component is parallel to a coordinate axis; along it
// the triangle's extent meets the cell's (the cell lies in the box), so the
// vertex projections nearest the cell stay within S / 2 of its centre
// (rounding included) while the test needs them beyond S / 2 + S t: such an
// axis never separates and is skipped without changing any decision.
__device__ __forceinline__ unsigned live_axes(const GridTri &t)
{
    auto two = [](float a, float b, float c) {
        return (a != 0.0f ? 1 : 0) + (b != 0.0f ? 1 : 0) + (c != 0.0f ? 1 : 0) >= 2;
    };
    unsigned m = two(t.n[0], t.n[1], t.n[2]) ? 1u : 0u;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float ex = t.e[3 * j], ey = t.e[3 * j + 1], ez = t.e[3 * j + 2];
        if (ez != 0.0f && ey != 0.0f) m |= 2u << (3 * j);
        if (ez != 0.0f && ex != 0.0f) m |= 4u << (3 * j);
        if (ey != 0.0f && ex != 0.0f) m |= 8u << (3 * j);
    }
    return m;
}

// The culling test: is triangle t separated from cell (x, y, z), the closed
// unit cube centred at (x, y, z) + 1/2?  Axes: the normal, then unit x e for
// every edge (those of `live` only); slack t = max|w| 2^-16 + 2^-10 (bounds
// the rounding error of the projections from above by a wide margin: a
// touching cell is never rejected).
__device__ __forceinline__ bool tri_cell_separated(const GridTri &t, unsigned live, unsigned x, unsigned y,
                                                   unsigned z)
{
    const float c[3] = {__fadd_rn(__uint2float_rn(x), 0.5f), __fadd_rn(__uint2float_rn(y), 0.5f),
                        __fadd_rn(__uint2float_rn(z), 0.5f)};
    float w[9];
    float W = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            w[3 * k + a] = __fsub_rn(t.q[3 * k + a], c[a]);
            W = fmaxf(W, fabsf(w[3 * k + a]));
        }
    const float slack = __fadd_rn(__fmul_rn(W, 1.52587890625e-05f), 9.765625e-04f);   // 2^-16, 2^-10
    if ((live & 1u) && axis_separates(t.n[0], t.n[1], t.n[2], w, slack)) return true;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float ex = t.e[3 * j], ey = t.e[3 * j + 1], ez = t.e[3 * j + 2];
        if (((live >> (3 * j)) & 2u) && axis2_separates(-ez, ey, 1, 2, w, slack)) return true;
        if (((live >> (3 * j)) & 4u) && axis2_separates(ez, -ex, 0, 2, w, slack)) return true;
        if (((live >> (3 * j)) & 8u) && axis2_separates(-ey, ex, 0, 1, w, slack)) return true;
    }
    return false;
}

// The cell x | y << 16 | z << 32 of vertex k: the floor of its (clamped) grid
// coordinate, into the object's box [bl, bh] as the cell mapping clamps it; the
// vertex lies in that closed cell, which culling therefore always keeps.
__device__ __forceinline__ unsigned long long vertex_cell(const GridTri &t, int k, const unsigned (&bl)[3],
                                                          const unsigned (&bh)[3])
{
    unsigned long long key = 0ull;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const float f = floorf(t.q[3 * k + ax]);
        const unsigned cc = f <= (float)bl[ax] ? bl[ax] : (f >= (float)bh[ax] ? bh[ax] : (unsigned)f);
        key |= (unsigned long long)cc << (16 * ax);
    }
    return key;
}

}  // namespace gg
