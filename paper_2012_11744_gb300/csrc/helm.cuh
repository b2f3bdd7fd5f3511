// FP64 Laplacian of the viscous step's kernels (viscous.cu, helmmg.cu).
#pragma once

#include "kernels.cuh"

namespace paris {

// The column (i, j) of unknowns over planes [k0, k1) of an array x with
// strides st: base points at (i, j, 0).  next(k) returns Lap_h x / ih2 at
// plane k: the neighbours present (or wrapped) summed, minus the diagonal
// count times the value: 2 an axis, one more at a no-slip end (ghost value
// minus the end value), 0 along a periodic axis of one point.
struct HelmColumn {
    const double* base;
    int64_t sz, oxm, oxp, oym, oyp;  // plane stride; offsets of the x and y neighbours
    bool hxm, hxp, hym, hyp;         // which of them exist
    int m2, kz;                      // planes and the kind of the z axis
    double dxy;                      // diagonal count of the x and y axes
    double zm, zc;

    __device__ __forceinline__ HelmColumn(const HelmGeo& g, const double* x, const int64_t (&st)[3], int i, int j,
                                          int k0) {
        base = x + i * st[0] + j * st[1];
        sz = st[2];
        auto axis = [&](int a, int p, bool& hm, bool& hp, int64_t& om, int64_t& op) {
            const int m = g.m[a];
            const bool per = g.kind[a] == HELM_PERIODIC;
            hm = per ? m > 1 : p > 0;
            hp = per ? m > 1 : p < m - 1;
            om = p > 0 ? -st[a] : (int64_t)(m - 1) * st[a];
            op = p < m - 1 ? st[a] : -(int64_t)(m - 1) * st[a];
            return (double)count(g.kind[a], m, p);
        };
        dxy = axis(0, i, hxm, hxp, oxm, oxp) + axis(1, j, hym, hyp, oym, oyp);
        m2 = g.m[2];
        kz = g.kind[2];
        zc = base[k0 * sz];
        zm = below(k0);
    }
    __device__ __forceinline__ static int count(int kind, int m, int p) {
        if (kind == HELM_PERIODIC) return m > 1 ? 2 : 0;
        return 2 + (kind == HELM_NOSLIP ? (p == 0) + (p == m - 1) : 0);
    }
    __device__ __forceinline__ double below(int k) const {
        if (k > 0) return base[(k - 1) * sz];
        return kz == HELM_PERIODIC && m2 > 1 ? base[(m2 - 1) * sz] : 0.0;
    }
    __device__ __forceinline__ double above(int k) const {
        if (k < m2 - 1) return base[(k + 1) * sz];
        return kz == HELM_PERIODIC && m2 > 1 ? base[0] : 0.0;
    }
    __device__ __forceinline__ double next(int k, double& xc) {
        const double* c = base + k * sz;
        const double xm = hxm ? c[oxm] : 0.0, xp = hxp ? c[oxp] : 0.0;
        const double ym = hym ? c[oym] : 0.0, yp = hyp ? c[oyp] : 0.0;
        const double zp = above(k);
        xc = zc;
        const double dg = dxy + (double)count(kz, m2, k);
        const double s = ((xm + xp) + (ym + yp)) + (zm + zp);
        zm = zc;
        zc = zp;
        return fma(-dg, xc, s);
    }
};

}  // namespace paris
