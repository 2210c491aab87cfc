// Device helpers shared by the waveprop kernels.
#pragma once
#include "internal.h"

#define WP_DEV __device__ __forceinline__

WP_DEV long long gidx(const GridDev &g, int x, int y, int z)
{
    return ((long long)x * g.NY + y) * g.PZ + z;
}

// depth (cells, continuous) of coordinate s into the absorbing layer of an
// axis with physical points [nbl, nbl + n - 1]
WP_DEV float layer_depth(float s, int nbl, int n)
{
    float lo = (float)nbl, hi = (float)(nbl + n - 1);
    return s < lo ? lo - s : (s > hi ? s - hi : 0.f);
}

// TTI damping rate at a node: sum over axes of sig0 * (d/L)^2, L = nbl*h
// (per-axis table).
WP_DEV float tti_sigma(const GridDev &g, int x, int y, int z)
{
    return __ldg(g.tab + x) + __ldg(g.tab + g.NX + y) + __ldg(g.tab + g.NX + g.NY + z);
}

// Cerjan taper: product over axes of exp(-(0.015 d)^2) at the position
// (sx, sy, sz), each coordinate a node i or a half point i + 1/2 (table).
WP_DEV float cerjan(const GridDev &g, float sx, float sy, float sz)
{
    const int ix = (int)sx, iy = (int)sy, iz = (int)sz;
    const int hx = (sx - ix) > 0.25f, hy = (sy - iy) > 0.25f, hz = (sz - iz) > 0.25f;
    return __ldg(g.tab + 2 * ix + hx) * __ldg(g.tab + 2 * g.NX + 2 * iy + hy) *
           __ldg(g.tab + 2 * (g.NX + g.NY) + 2 * iz + hz);
}

// load with zero extension outside the computational grid
WP_DEV float ldz(const float *__restrict__ f, const GridDev &g, int x, int y, int z)
{
    return (x >= 0 && x < g.NX && y >= 0 && y < g.NY && z >= 0 && z < g.NZ) ? __ldg(f + gidx(g, x, y, z)) : 0.f;
}

// one receiver: the weighted sum over its corners (the fields without restrict: a
// pass that samples may have been launched while they were written)
WP_DEV float record_point(const long long *__restrict__ idx, const float *__restrict__ w, int i, const float *f0,
                          const float *f1, const float *f2)
{
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < 8; c++) {
        const long long q = idx[8 * (long long)i + c];
        const float wc = w[8 * (long long)i + c];
        if (wc != 0.f) {
            float v = f0[q];
            if (f1) v += f1[q];
            if (f2) v += f2[q];
            s = __fmaf_rn(wc, v, s);
        }
    }
    return s;
}
// source term of a cell: the weighted sum of its traces at time t
WP_DEV float inject_sum(const int *__restrict__ ptr, const int *__restrict__ tr, const float *__restrict__ w,
                        const float *__restrict__ traces, int nt, int t, int j)
{
    float acc = 0.f;
    for (int e = ptr[j]; e < ptr[j + 1]; e++) acc = __fmaf_rn(w[e], traces[(long long)tr[e] * nt + t], acc);
    return acc;
}
// a source term is rounded before it is added to a field (the same bits in every
// kernel that injects)
WP_DEV void inject_add(float &f, float coef, float acc) { f = __fadd_rn(f, __fmul_rn(coef, acc)); }
// scale / A, A = m (1 + sig dt/2): the factor of a TTI or acoustic source term
WP_DEV float inject_coef(const GridDev &g, float scale, float m, int x, int y, int z)
{
    return scale / (m * (1.f + 0.5f * tti_sigma(g, x, y, z) * g.dt));
}

WP_DEV int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }
