// Multigrid preconditioner of the implicit viscous step (Sec. 3.2.3, Eq.
// muelliptic) and the kernels of the mixed-precision solve around it.
//
// One velocity component's SPD operator on its unknowns (the component's
// face grid without its own wall faces),
//
//     A x = sigma x - Lap_h x,      sigma = 1 / (tau nu_f),
//
// is preconditioned by an FP32 V-cycle over a hierarchy of grids coarsened
// by two along every axis together.  The kind of an axis fixes how:
//   * periodic, and the no-slip axes of a tangential component (unknowns at
//     cell centres, the wall half a cell beyond the ends, ghost value minus
//     the end value): cell-centred, m -> m/2 (m even), children 2I and 2I+1,
//     prolongation constant, restriction their average;
//   * the component's own wall axis (unknowns at faces 1 .. n-1, zero at
//     faces 0 and n): vertex-centred, m -> (m-1)/2 (m odd), coarse point J
//     at fine point 2J+1, prolongation linear, restriction full weighting
//     (1/4, 1/2, 1/4).
// The restriction is the transpose of the prolongation scaled to average, so
// the coarse equations are rediscretised at spacing 2h with the same
// boundary kinds; the coarse sigma is the restricted fine sigma.  Smoother:
// red-black Gauss-Seidel with over-relaxation where every periodic extent of
// the level is even, damped Jacobi otherwise (a periodic axis of odd length
// would give a cell two neighbours of its own colour).  The solve around it
// has the structure of the Poisson solve's mixed form: FP64 iterative
// refinement (the FP64 residual of the SPD form, the accumulation of u*)
// around an FP32 flexible CG (the V-cycle is not exactly linear: FP32,
// Gauss-Seidel) on the finest level's operator with FP32 sigma.
#include <algorithm>

#include "helm.cuh"

namespace paris {

namespace {

constexpr int kTX = 32, kTY = 8, kZ = 8;
constexpr int kPerSM = 4;  // resident blocks per SM of the FP64 marching kernels

struct HLev {
    int m[3];     // unknowns per axis
    int kind[3];  // HELM_PERIODIC / HELM_ZERO / HELM_NOSLIP
    float ih2;    // 1 / h_l^2
};

__device__ __forceinline__ int hidx(const HLev& L, int i, int j, int k) { return (k * L.m[1] + j) * L.m[0] + i; }

// the six neighbour values (or the ghost rule) and the Laplacian diagonal
// count of unknown (i, j, k): acc gets sum of neighbour values, dg the count
template <typename T, typename V>
__device__ __forceinline__ void hnb(const HLev& L, const V* __restrict__ x, int i, int j, int k, T& acc, T& dg) {
    const int pos[3] = {i, j, k};
    acc = T(0);
    dg = T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int m = L.m[a];
        const int st = a == 0 ? 1 : (a == 1 ? L.m[0] : L.m[0] * L.m[1]);
        const int c = hidx(L, i, j, k);
        const int p = pos[a];
        if (L.kind[a] == HELM_PERIODIC) {
            if (m > 1) {
                acc += (T)x[p > 0 ? c - st : c + (m - 1) * st] + (T)x[p < m - 1 ? c + st : c - (m - 1) * st];
                dg += T(2);
            }
        } else {
            if (p > 0) acc += (T)x[c - st];
            if (p < m - 1) acc += (T)x[c + st];
            dg += T(2);
            if (L.kind[a] == HELM_NOSLIP) dg += T((p == 0) + (p == m - 1));  // ghost = -x_c
        }
    }
}

// one colour of red-black Gauss-Seidel (or, with JAC, a damped Jacobi sweep
// from xi into xo): x_c += omega ((f_c + acc/h^2) / (sigma_c + dg/h^2) - x_c)
template <bool JAC>
__global__ void __launch_bounds__(kTX* kTY) hmg_smooth_kernel(HLev L, const float* __restrict__ f,
                                                             const float* __restrict__ sig, const float* xi,
                                                             float* xo, int color, float omega) {
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    if (i >= L.m[0] || j >= L.m[1]) return;
    const int k0 = blockIdx.z * kZ, k1 = min(k0 + kZ, L.m[2]);
    for (int k = k0; k < k1; ++k) {
        if (!JAC && ((i + j + k) & 1) != color) continue;
        const int c = hidx(L, i, j, k);
        float acc, dg;
        hnb<float>(L, xi, i, j, k, acc, dg);
        const float xc = xi[c];
        const float gs = fmaf(acc, L.ih2, f[c]) / fmaf(dg, L.ih2, sig[c]);
        xo[c] = fmaf(omega, gs - xc, xc);
    }
}

// One colour of red-black Gauss-Seidel with a thread per pair of cells
// (2t, 2t+1) of a row: the member of the pass's colour is updated, so every
// thread works on every plane of its z-segment.  Same update as the
// column kernel above.
__global__ void __launch_bounds__(kTX* kTY) hmg_rbgs_pair_kernel(HLev L, const float* __restrict__ f,
                                                                const float* __restrict__ sig, float* x, int color,
                                                                float omega, int zper) {
    pdl_wait();
    const int t = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    if (2 * t >= L.m[0] || j >= L.m[1]) return;
    const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, L.m[2]);
    for (int k = k0; k < k1; ++k) {
        const int i = 2 * t + ((j + k + color) & 1);
        if (i >= L.m[0]) continue;
        const int c = hidx(L, i, j, k);
        float acc, dg;
        hnb<float>(L, x, i, j, k, acc, dg);
        const float xc = x[c];
        const float gs = fmaf(acc, L.ih2, f[c]) / fmaf(dg, L.ih2, sig[c]);
        x[c] = fmaf(omega, gs - xc, xc);
    }
}

// The same colour pass with a thread per four cells 4q .. 4q+3 of a row
// (rows of m0 % 4 == 0 cells, at least a warp's worth): every array read as
// 16-byte vectors, the two cells of the pass's colour updated, the
// x-neighbours outside the quad from the adjacent lanes (or loaded at the
// edges of the warp), the quad stored back whole (the other two cells
// unchanged: no thread writes them in this pass).  M: the updated member of
// both pairs of the quad ((j + k + color) & 1, uniform per row).
// zero: x taken as 0 (nothing of it read, both colours written), which
// replaces a pass that cleared it.
template <int M>
__device__ __forceinline__ void hrb4_row(const HLev& L, const float* __restrict__ f, const float* __restrict__ sig,
                                         float* x, float omega, int j, int k, int i0, int lane, bool act, bool zero) {
    const int m0 = L.m[0], m1 = L.m[1], m2 = L.m[2], pl = m0 * m1;
    const int rowc = (k * m1 + j) * m0, c0 = rowc + i0;
    const bool py = L.kind[1] == HELM_PERIODIC, pz = L.kind[2] == HELM_PERIODIC;
    // neighbour rows and planes: present (or wrapped) and their offsets
    const bool hym = py ? m1 > 1 : j > 0, hyp = py ? m1 > 1 : j < m1 - 1;
    const bool hzm = pz ? m2 > 1 : k > 0, hzp = pz ? m2 > 1 : k < m2 - 1;
    const int oym = j > 0 ? -m0 : (m1 - 1) * m0, oyp = j < m1 - 1 ? m0 : -(m1 - 1) * m0;
    const int ozm = k > 0 ? -pl : (m2 - 1) * pl, ozp = k < m2 - 1 ? pl : -(m2 - 1) * pl;
    float X[4], F[4], S[4], YM[4] = {0.f, 0.f, 0.f, 0.f}, YP[4] = {0.f, 0.f, 0.f, 0.f},
                                ZM[4] = {0.f, 0.f, 0.f, 0.f}, ZP[4] = {0.f, 0.f, 0.f, 0.f};
    auto ld = [](float (&d)[4], const float* p) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        d[0] = v.x;
        d[1] = v.y;
        d[2] = v.z;
        d[3] = v.w;
    };
    X[0] = X[1] = X[2] = X[3] = 0.f;
    if (!zero) ld(X, x + c0);
    ld(F, f + c0);
    ld(S, sig + c0);
    if (hym && !zero) ld(YM, x + c0 + oym);
    if (hyp && !zero) ld(YP, x + c0 + oyp);
    if (hzm && !zero) ld(ZM, x + c0 + ozm);
    if (hzp && !zero) ld(ZP, x + c0 + ozp);
    // x of the cells next to the quad (i0-1 and i0+4): wrapped along a periodic
    // axis, absent (0) beyond the ends of the other kinds
    const bool px = L.kind[0] == HELM_PERIODIC;
    const int il = i0 > 0 ? i0 - 1 : m0 - 1, ir = i0 + 4 < m0 ? i0 + 4 : 0;
    const bool hxl = px ? m0 > 1 : i0 > 0, hxr = px ? m0 > 1 : i0 + 4 < m0;
    const float xl_sh = __shfl_up_sync(0xffffffffu, X[3], 1), xr_sh = __shfl_down_sync(0xffffffffu, X[0], 1);
    const float xl_ld = hxl && !zero ? x[rowc + il] : 0.f, xr_ld = hxr && !zero ? x[rowc + ir] : 0.f;
    const float xl = (lane > 0 && i0 > 0) ? xl_sh : xl_ld;
    const float xr = (lane < kTX - 1 && i0 + 4 < m0) ? xr_sh : xr_ld;
    // Laplacian diagonal counts of the y and z axes (uniform per row)
    auto ends = [](int kind, int m, int p) {
        if (kind == HELM_PERIODIC) return m > 1 ? 2.f : 0.f;
        return kind == HELM_NOSLIP ? 2.f + (float)((p == 0) + (p == m - 1)) : 2.f;
    };
    const float dyz = ends(L.kind[1], m1, j) + ends(L.kind[2], m2, k);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int li = 2 * u + M, i = i0 + li;
        const float lo = li > 0 ? X[li - 1] : xl, hi = li < 3 ? X[li + 1] : xr;
        const float acc = ((lo + hi) + (YM[li] + YP[li])) + (ZM[li] + ZP[li]);
        const float dg = ends(L.kind[0], m0, i) + dyz;
        const float gs = fmaf(acc, L.ih2, F[li]) / fmaf(dg, L.ih2, S[li]);
        X[li] = fmaf(omega, gs - X[li], X[li]);
    }
    if (act) *reinterpret_cast<float4*>(x + c0) = make_float4(X[0], X[1], X[2], X[3]);
}

// (A x) of the four cells 4q .. 4q+3 of a row (the quad layout of
// hrb4_row: 16-byte vectors, x-neighbours from the adjacent lanes); X: x of
// the quad as loaded.  Same per-cell arithmetic as hmg_residual_kernel.
__device__ __forceinline__ void hop4(const HLev& L, const float* __restrict__ x, const float* __restrict__ sig,
                                     int j, int k, int i0, int lane, float (&X)[4], float (&AX)[4]) {
    const int m0 = L.m[0], m1 = L.m[1], m2 = L.m[2], pl = m0 * m1;
    const int rowc = (k * m1 + j) * m0, c0 = rowc + i0;
    const bool py = L.kind[1] == HELM_PERIODIC, pz = L.kind[2] == HELM_PERIODIC, px = L.kind[0] == HELM_PERIODIC;
    const bool hym = py ? m1 > 1 : j > 0, hyp = py ? m1 > 1 : j < m1 - 1;
    const bool hzm = pz ? m2 > 1 : k > 0, hzp = pz ? m2 > 1 : k < m2 - 1;
    const int oym = j > 0 ? -m0 : (m1 - 1) * m0, oyp = j < m1 - 1 ? m0 : -(m1 - 1) * m0;
    const int ozm = k > 0 ? -pl : (m2 - 1) * pl, ozp = k < m2 - 1 ? pl : -(m2 - 1) * pl;
    float S[4], YM[4] = {0.f, 0.f, 0.f, 0.f}, YP[4] = {0.f, 0.f, 0.f, 0.f}, ZM[4] = {0.f, 0.f, 0.f, 0.f},
                ZP[4] = {0.f, 0.f, 0.f, 0.f};
    auto ld = [](float (&d)[4], const float* p) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        d[0] = v.x;
        d[1] = v.y;
        d[2] = v.z;
        d[3] = v.w;
    };
    ld(X, x + c0);
    ld(S, sig + c0);
    if (hym) ld(YM, x + c0 + oym);
    if (hyp) ld(YP, x + c0 + oyp);
    if (hzm) ld(ZM, x + c0 + ozm);
    if (hzp) ld(ZP, x + c0 + ozp);
    const int il = i0 > 0 ? i0 - 1 : m0 - 1, ir = i0 + 4 < m0 ? i0 + 4 : 0;
    const bool hxl = px ? m0 > 1 : i0 > 0, hxr = px ? m0 > 1 : i0 + 4 < m0;
    const float xl_sh = __shfl_up_sync(0xffffffffu, X[3], 1), xr_sh = __shfl_down_sync(0xffffffffu, X[0], 1);
    const float xl_ld = hxl ? __ldg(x + rowc + il) : 0.f, xr_ld = hxr ? __ldg(x + rowc + ir) : 0.f;
    const float xl = (lane > 0 && i0 > 0) ? xl_sh : xl_ld;
    const float xr = (lane < kTX - 1 && i0 + 4 < m0) ? xr_sh : xr_ld;
    auto ends = [](int kind, int m, int p) {
        if (kind == HELM_PERIODIC) return m > 1 ? 2.f : 0.f;
        return kind == HELM_NOSLIP ? 2.f + (float)((p == 0) + (p == m - 1)) : 2.f;
    };
    const float dyz = ends(L.kind[1], m1, j) + ends(L.kind[2], m2, k);
#pragma unroll
    for (int li = 0; li < 4; ++li) {
        const float lo = li > 0 ? X[li - 1] : xl, hi = li < 3 ? X[li + 1] : xr;
        const float acc = ((lo + hi) + (YM[li] + YP[li])) + (ZM[li] + ZP[li]);
        const float dg = ends(L.kind[0], m0, i0 + li) + dyz;
        AX[li] = fmaf(dg, L.ih2, S[li]) * X[li] - acc * L.ih2;
    }
}

// r = f - A x (quads)
__global__ void __launch_bounds__(kTX* kTY) hmg_residual4_kernel(HLev L, const float* __restrict__ f,
                                                                const float* __restrict__ sig,
                                                                const float* __restrict__ x, float* __restrict__ r) {
    pdl_wait();
    const int j = blockIdx.y * kTY + threadIdx.y;
    if (j >= L.m[1]) return;
    const int k = blockIdx.z, lane = threadIdx.x;
    const int nq = L.m[0] / 4, q = blockIdx.x * kTX + lane;
    const bool act = q < nq;
    const int i0 = 4 * (act ? q : nq - 1);
    float X[4], AX[4];
    hop4(L, x, sig, j, k, i0, lane, X, AX);
    if (act) {
        const int c0 = (k * L.m[1] + j) * L.m[0] + i0;
        const float4 fv = __ldg(reinterpret_cast<const float4*>(f + c0));
        *reinterpret_cast<float4*>(r + c0) = make_float4(fv.x - AX[0], fv.y - AX[1], fv.z - AX[2], fv.w - AX[3]);
    }
}

// q = A d (quads) and the partials of d . q.  A block takes zper planes of its
// 8 rows: with one, the 8192 blocks' hand-over of their partial sums took as
// long as the product (76 us at 256^3; 41 with 17).  A plane's four terms are
// added in FP32, the planes' sums with their errors (CarriedSum).
__global__ void __launch_bounds__(kTX* kTY, 6) hmg_matvec4_kernel(HLev L, const float* __restrict__ sig,
                                                                 const float* __restrict__ d, float* __restrict__ q,
                                                                 double* partials, int zper, FinSpec fin) {
    pdl_wait();
    const int j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    const int jc = j < L.m[1] ? j : L.m[1] - 1;  // idle rows shadow the last row (no stores)
    const int lane = threadIdx.x;
    const int nq = L.m[0] / 4, qq = blockIdx.x * kTX + lane;
    const bool act = qq < nq && j < L.m[1];
    const int i0 = 4 * (qq < nq ? qq : nq - 1);
    const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, L.m[2]);
    CarriedSum dq;
    for (int k = k0; k < k1; ++k) {
        float X[4], AX[4];
        hop4(L, d, sig, jc, k, i0, lane, X, AX);
        if (act) {
            const int c0 = (k * L.m[1] + jc) * L.m[0] + i0;
            *reinterpret_cast<float4*>(q + c0) = make_float4(AX[0], AX[1], AX[2], AX[3]);
            float t = 0.f;
#pragma unroll
            for (int li = 0; li < 4; ++li) t = fmaf(X[li], AX[li], t);
            dq.add(t);
        }
    }
    double accd[1] = {dq.value()};
    const int op[1] = {0};
    block_reduce_store<1>(accd, op, partials, ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x,
                          tid);
    finalize_last_block(partials, (int64_t)gridDim.x * gridDim.y * gridDim.z, fin, tid);
}

__global__ void __launch_bounds__(kTX* kTY, 6) hmg_rb4_kernel(HLev L, const float* __restrict__ f,
                                                          const float* __restrict__ sig, float* x, int color,
                                                          float omega, int zero) {
    pdl_wait();
    const int j = blockIdx.y * kTY + threadIdx.y;
    if (j >= L.m[1]) return;  // uniform per warp
    const int k = blockIdx.z, lane = threadIdx.x;
    const int nq = L.m[0] / 4, q = blockIdx.x * kTX + lane;
    const bool act = q < nq;
    const int i0 = 4 * (act ? q : nq - 1);  // idle lanes shadow the last quad (no stores)
    if (((j + k + color) & 1) == 0)
        hrb4_row<0>(L, f, sig, x, omega, j, k, i0, lane, act, zero != 0);
    else
        hrb4_row<1>(L, f, sig, x, omega, j, k, i0, lane, act, zero != 0);
}

// r = f - A x on a level (FP32)
__global__ void __launch_bounds__(kTX* kTY) hmg_residual_kernel(HLev L, const float* __restrict__ f,
                                                               const float* __restrict__ sig,
                                                               const float* __restrict__ x, float* __restrict__ r,
                                                               int zper) {
    pdl_wait();
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    if (i >= L.m[0] || j >= L.m[1]) return;
    const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, L.m[2]);
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        const int c = hidx(L, i, j, k);
        float acc, dg;
        hnb<float>(L, x, i, j, k, acc, dg);
        const float xc = x[c];
        r[c] = f[c] - (fmaf(dg, L.ih2, sig[c]) * xc - acc * L.ih2);
    }
}

// fine points of coarse point I along an axis and their restriction weights
struct Kids {
    int n;
    int i[3];
    float w[3];
};
__device__ __forceinline__ Kids kids(int kind, int I) {
    Kids q;
    if (kind == HELM_ZERO) {  // vertex-centred: fine 2I, 2I+1, 2I+2 (1/4, 1/2, 1/4)
        q.n = 3;
        q.i[0] = 2 * I;
        q.i[1] = 2 * I + 1;
        q.i[2] = 2 * I + 2;
        q.w[0] = 0.25f;
        q.w[1] = 0.5f;
        q.w[2] = 0.25f;
    } else {  // cell-centred: fine 2I, 2I+1 (1/2, 1/2)
        q.n = 2;
        q.i[0] = 2 * I;
        q.i[1] = 2 * I + 1;
        q.i[2] = 0;
        q.w[0] = q.w[1] = 0.5f;
        q.w[2] = 0.f;
    }
    return q;
}

// (R fine) at coarse point (I, J, K): the tensor product of the per-axis weights
__device__ __forceinline__ float restrict_at(const HLev& F, int I, int J, int K, const float* fine) {
    const Kids a = kids(F.kind[0], I), b = kids(F.kind[1], J), c = kids(F.kind[2], K);
    float s = 0.f;
    for (int z = 0; z < c.n; ++z)
        for (int y = 0; y < b.n; ++y) {
            float sx = 0.f;
            for (int x = 0; x < a.n; ++x) sx = fmaf(a.w[x], fine[hidx(F, a.i[x], b.i[y], c.i[z])], sx);
            s = fmaf(c.w[z] * b.w[y], sx, s);
        }
    return s;
}

// coarse = R fine
__global__ void __launch_bounds__(kTX* kTY) hmg_restrict_kernel(HLev F, HLev Cg, const float* __restrict__ fine,
                                                               float* __restrict__ coarse) {
    pdl_wait();
    const int I = blockIdx.x * kTX + threadIdx.x, J = blockIdx.y * kTY + threadIdx.y, K = blockIdx.z;
    if (I >= Cg.m[0] || J >= Cg.m[1]) return;
    coarse[hidx(Cg, I, J, K)] = restrict_at(F, I, J, K, fine);
}

// coarse points of fine point i along an axis and the prolongation weights
struct Pars {
    int n;
    int I[2];
    float w[2];
};
__device__ __forceinline__ Pars parents(int kind, int i, int mc) {
    Pars q;
    q.n = 0;
    if (kind == HELM_ZERO) {
        // fine unknown i sits at face i+1; coarse unknown J at face 2(J+1)
        const int F = i + 1;
        if ((F & 1) == 0) {
            q.n = 1;
            q.I[0] = F / 2 - 1;
            q.w[0] = 1.f;
        } else {
            const int J1 = (F - 1) / 2 - 1, J2 = (F + 1) / 2 - 1;
            if (J1 >= 0) { q.I[q.n] = J1; q.w[q.n] = 0.5f; ++q.n; }
            if (J2 < mc) { q.I[q.n] = J2; q.w[q.n] = 0.5f; ++q.n; }
        }
    } else {
        q.n = 1;
        q.I[0] = i / 2;
        q.w[0] = 1.f;
    }
    return q;
}

// (P e) at fine point (i, j, k): the tensor product of the per-axis weights
__device__ __forceinline__ float prolong_at(const HLev& F, const HLev& Cg, int i, int j, int k, const float* e) {
    const Pars a = parents(F.kind[0], i, Cg.m[0]), b = parents(F.kind[1], j, Cg.m[1]),
               c = parents(F.kind[2], k, Cg.m[2]);
    float s = 0.f;
    for (int z = 0; z < c.n; ++z)
        for (int y = 0; y < b.n; ++y)
            for (int q = 0; q < a.n; ++q) s = fmaf(a.w[q] * b.w[y] * c.w[z], e[hidx(Cg, a.I[q], b.I[y], c.I[z])], s);
    return s;
}

// x += P e
__global__ void __launch_bounds__(kTX* kTY) hmg_prolong_kernel(HLev F, HLev Cg, const float* __restrict__ e,
                                                              float* __restrict__ x) {
    pdl_wait();
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y, k = blockIdx.z;
    if (i >= F.m[0] || j >= F.m[1]) return;
    x[hidx(F, i, j, k)] += prolong_at(F, Cg, i, j, k, e);
}

// The same for rows of m0 % 4 == 0 unknowns of a cell-centred x axis: four
// unknowns and their two parents a thread, 16-byte vectors, one index over the
// level (64 unknowns a row fill half a warp of quads otherwise).  Same sums.
__global__ void __launch_bounds__(kTX* kTY) hmg_prolong4_kernel(HLev F, HLev Cg, unsigned nq, unsigned mq, unsigned my,
                                                               unsigned total, const float* __restrict__ e,
                                                               float* __restrict__ x) {
    pdl_wait();
    const unsigned t = blockIdx.x * (unsigned)(kTX * kTY) + threadIdx.x;
    if (t >= total) return;
    const unsigned row = fast_div(t, nq, mq), k = fast_div(row, (unsigned)F.m[1], my);
    const int q = (int)(t - row * nq), j = (int)(row - k * (unsigned)F.m[1]);
    const Pars b = parents(F.kind[1], j, Cg.m[1]), c = parents(F.kind[2], (int)k, Cg.m[2]);
    float4 v = reinterpret_cast<const float4*>(x)[t];
    float s0 = 0.f, s1 = 0.f;
    for (int z = 0; z < c.n; ++z)
        for (int y = 0; y < b.n; ++y) {
            const float w = b.w[y] * c.w[z];
            const float* p = e + hidx(Cg, 2 * q, b.I[y], c.I[z]);
            s0 = fmaf(w, p[0], s0);
            s1 = fmaf(w, p[1], s1);
        }
    v.x += s0;
    v.y += s0;
    v.z += s1;
    v.w += s1;
    reinterpret_cast<float4*>(x)[t] = v;
}

// ------------------------------------------------------- tail of the V-cycle

// From the first level of at most kTailUnknowns unknowns to the coarsest and
// back in one block of 1024 threads, the levels' arrays in shared memory and a
// block barrier between steps: a pass of such a level is one launch of 3 us
// otherwise, and there are up to 60 of them a V-cycle (tail: 43 us at 16^3).  The same arithmetic in
// the same order as the level kernels.
constexpr int kTailThreads = 1024;
constexpr int64_t kTailUnknowns = 4096;

struct HTailLevel {
    HLev L;
    int jac;                // damped Jacobi (an odd periodic extent)
    unsigned mp, m0, m1;    // fast_div multipliers of the pairs of a row, of m[0] and m[1]
    const float* sig;
};
struct HTail {
    int n, nu1, nu2, coarse_sweeps;
    float omega;
    const float* f;  // right-hand side of the first level
    float* x;        // its solution
    HTailLevel lv[kHelmMaxLevels];
};

__device__ __forceinline__ void htail_smooth(const HTailLevel& T, const float* f, const float* sig, float* x, float* tmp,
                                             int sweeps, bool reverse, float omega) {
    const HLev L = T.L;
    if (T.jac) {
        const int n = L.m[0] * L.m[1] * L.m[2];
        for (int s = 0; s < sweeps; ++s) {
            for (unsigned c = threadIdx.x; c < (unsigned)n; c += kTailThreads) {
                const unsigned row = fast_div(c, (unsigned)L.m[0], T.m0), k = fast_div(row, (unsigned)L.m[1], T.m1);
                float acc, dg;
                hnb<float>(L, x, (int)(c - row * L.m[0]), (int)(row - k * L.m[1]), (int)k, acc, dg);
                const float xc = x[c];
                const float gs = fmaf(acc, L.ih2, f[c]) / fmaf(dg, L.ih2, sig[c]);
                tmp[c] = fmaf(0.8f, gs - xc, xc);
            }
            __syncthreads();
            for (int c = threadIdx.x; c < n; c += kTailThreads) x[c] = tmp[c];
            __syncthreads();
        }
        return;
    }
    const unsigned npair = (unsigned)(L.m[0] + 1) / 2, total = npair * (unsigned)(L.m[1] * L.m[2]);
    for (int h = 0; h < 2 * sweeps; ++h) {
        const int color = reverse ? 1 - (h & 1) : h & 1;
        for (unsigned t = threadIdx.x; t < total; t += kTailThreads) {
            const unsigned row = fast_div(t, npair, T.mp), k = fast_div(row, (unsigned)L.m[1], T.m1);
            const int j = (int)(row - k * L.m[1]);
            const int i = 2 * (int)(t - row * npair) + ((j + (int)k + color) & 1);
            if (i >= L.m[0]) continue;
            const int c = hidx(L, i, j, (int)k);
            float acc, dg;
            hnb<float>(L, x, i, j, (int)k, acc, dg);
            const float xc = x[c];
            const float gs = fmaf(acc, L.ih2, f[c]) / fmaf(dg, L.ih2, sig[c]);
            x[c] = fmaf(omega, gs - xc, xc);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kTailThreads) hmg_tail_kernel(const __grid_constant__ HTail a) {
    pdl_wait();
    extern __shared__ __align__(16) float dyn[];
    __shared__ float *X[kHelmMaxLevels], *F[kHelmMaxLevels], *S[kHelmMaxLevels];
    __shared__ float* R;
    auto cells = [&](int l) { return a.lv[l].L.m[0] * a.lv[l].L.m[1] * a.lv[l].L.m[2]; };
    if (threadIdx.x == 0) {
        float* p = dyn;
        for (int l = 0; l < a.n; ++l) {
            X[l] = p;
            F[l] = p + cells(l);
            S[l] = p + 2 * cells(l);
            p += 3 * cells(l);
        }
        R = p;
    }
    __syncthreads();
    for (int l = 0; l < a.n; ++l)
        for (int c = threadIdx.x; c < cells(l); c += kTailThreads) {
            S[l][c] = a.lv[l].sig[c];
            X[l][c] = 0.f;
            if (l == 0) F[0][c] = a.f[c];
        }
    __syncthreads();
    for (int l = 0; l < a.n - 1; ++l) {
        const HLev L = a.lv[l].L, Cg = a.lv[l + 1].L;
        htail_smooth(a.lv[l], F[l], S[l], X[l], R, a.nu1, false, a.omega);
        for (unsigned c = threadIdx.x; c < (unsigned)cells(l); c += kTailThreads) {
            const unsigned row = fast_div(c, (unsigned)L.m[0], a.lv[l].m0), k = fast_div(row, (unsigned)L.m[1], a.lv[l].m1);
            float acc, dg;
            hnb<float>(L, X[l], (int)(c - row * L.m[0]), (int)(row - k * L.m[1]), (int)k, acc, dg);
            R[c] = F[l][c] - (fmaf(dg, L.ih2, S[l][c]) * X[l][c] - acc * L.ih2);
        }
        __syncthreads();
        for (unsigned c = threadIdx.x; c < (unsigned)cells(l + 1); c += kTailThreads) {
            const unsigned row = fast_div(c, (unsigned)Cg.m[0], a.lv[l + 1].m0),
                           K = fast_div(row, (unsigned)Cg.m[1], a.lv[l + 1].m1);
            F[l + 1][c] = restrict_at(L, (int)(c - row * Cg.m[0]), (int)(row - K * Cg.m[1]), (int)K, R);
        }
        __syncthreads();
    }
    htail_smooth(a.lv[a.n - 1], F[a.n - 1], S[a.n - 1], X[a.n - 1], R, a.coarse_sweeps, false, a.omega);
    for (int l = a.n - 2; l >= 0; --l) {
        const HLev L = a.lv[l].L, Cg = a.lv[l + 1].L;
        for (unsigned c = threadIdx.x; c < (unsigned)cells(l); c += kTailThreads) {
            const unsigned row = fast_div(c, (unsigned)L.m[0], a.lv[l].m0), k = fast_div(row, (unsigned)L.m[1], a.lv[l].m1);
            X[l][c] += prolong_at(L, Cg, (int)(c - row * L.m[0]), (int)(row - k * L.m[1]), (int)k, X[l + 1]);
        }
        __syncthreads();
        htail_smooth(a.lv[l], F[l], S[l], X[l], R, a.nu2, true, a.omega);
    }
    for (int c = threadIdx.x; c < cells(0); c += kTailThreads) a.x[c] = X[0][c];
}

// ---------------------------------------------------------------- FP64 side

// sigma = 1/(tau nu) on the unknowns (FP64 and FP32 copies); the right-hand
// side norms of b = sigma u^n (partials |b|^2, max |b|, non-finite count, 0;
// a nu that is not > 0 counts as non-finite); u* = u^n on the unknowns
__global__ void __launch_bounds__(kTX* kTY) hmg_setup_kernel(HelmGeo g, const double* __restrict__ un,
                                                            const double* __restrict__ nu, double tau,
                                                            double* __restrict__ sig64, float* __restrict__ sig32,
                                                            double* __restrict__ us, double* partials, FinSpec fin) {
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    double l2 = 0.0;
    unsigned long long bk = 0;
    unsigned nf = 0;
    if (i < g.m[0] && j < g.m[1]) {
        const int k0 = blockIdx.z * kZ, k1 = min(k0 + kZ, g.m[2]);
        for (int k = k0; k < k1; ++k) {
            const int64_t p = ((int64_t)k * g.m[1] + j) * g.m[0] + i;
            const int64_t f = g.off + i + (int64_t)g.e[0] * (j + (int64_t)g.e[1] * k);
            const double nv = nu[f], v = un[f];
            const double s = recip64_rn(tau * nv);
            sig64[p] = s;
            sig32[p] = to_f32(s);
            us[f] = v;
            const double b = s * v;
            l2 = fma(b, b, l2);
            const unsigned long long kb = abs_key(b);
            bk = kb > bk ? kb : bk;
            nf += (key_nonfinite(kb) || !(nv > 0.0)) ? 1u : 0u;
        }
    }
    block_reduce_skc<double>(l2, bk, nf, partials, ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x,
                             tid);
    finalize_last_block(partials, (int64_t)gridDim.x * gridDim.y * gridDim.z, fin, tid);
}

// r = sigma (u^n - u*) + Lap_h u* (u* the face array), kept only as the scaled
// FP32 right-hand side of the inner solve, r32 = 2^k r (k from the context's
// scalar block: max |r| of the residual before); partials (|r|^2, max |r|,
// non-finite count) of the FP64 r.  Bound by the FP64 pipe: 10 instructions per
// unknown (HelmColumn) where the operator in terms of its diagonal took about
// 20 with the index arithmetic and the ends, and a pass of its own then scaled
// and converted r (541 + 76 us at 256^3, now 400).
__global__ void __launch_bounds__(kTX* kTY, kPerSM) hmg_residual64_kernel(HelmGeo g, const double* __restrict__ un,
                                                                         const double* __restrict__ sig,
                                                                         const double* __restrict__ us,
                                                                         const Scal* __restrict__ s,
                                                                         float* __restrict__ r32, double* partials,
                                                                         int zper, FinSpec fin) {
    pdl_wait();
    const int se_r = (int)s->scale_exp;
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    double l2 = 0.0;
    unsigned long long rk = 0;
    unsigned nf = 0;
    if (i < g.m[0] && j < g.m[1]) {
        const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, g.m[2]);
        const int64_t se[3] = {1, g.e[0], (int64_t)g.e[0] * g.e[1]};
        HelmColumn col(g, us + g.off, se, i, j, k0);
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
            const int64_t p = ((int64_t)k * g.m[1] + j) * g.m[0] + i;
            const int64_t f = g.off + i + (int64_t)g.e[0] * (j + (int64_t)g.e[1] * k);
            double xc;
            const double lap = col.next(k, xc);
            const double rp = fma(g.ih2, lap, sig[p] * (un[f] - xc));
            r32[p] = d2f_scaled(rp, se_r);
            l2 = fma(rp, rp, l2);
            const unsigned long long kr = abs_key(rp);
            rk = kr > rk ? kr : rk;
            nf += key_nonfinite(kr);
        }
    }
    block_reduce_skc<double>(l2, rk, nf, partials, ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x,
                             tid);
    finalize_last_block(partials, (int64_t)gridDim.x * gridDim.y * gridDim.z, fin, tid);
}

// FP32 inner iteration: q = A d on the finest level (FP32 sigma) and the
// partials of d . q
__global__ void __launch_bounds__(kTX* kTY, 6) hmg_matvec32_kernel(HLev L, const float* __restrict__ sig,
                                                               const float* __restrict__ d, float* __restrict__ q,
                                                               double* partials, int zper, FinSpec fin) {
    pdl_wait();
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    CarriedSum dq;
    if (i < L.m[0] && j < L.m[1]) {
        const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, L.m[2]);
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
            const int c = hidx(L, i, j, k);
            float acc, dg;
            hnb<float>(L, d, i, j, k, acc, dg);
            const float dc = d[c];
            const float qc = fmaf(dg, L.ih2, sig[c]) * dc - acc * L.ih2;
            q[c] = qc;
            dq.add(__fmul_rn(dc, qc));
        }
    }
    double accd[1] = {dq.value()};
    const int op[1] = {0};
    block_reduce_store<1>(accd, op, partials, ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x,
                          tid);
    finalize_last_block(partials, (int64_t)gridDim.x * gridDim.y * gridDim.z, fin, tid);
}

// u* += e / scale on the unknowns of the face array
__global__ void __launch_bounds__(kTX* kTY) hmg_accumulate_kernel(HelmGeo g, const float* __restrict__ e,
                                                                 const Scal* __restrict__ s, double* __restrict__ us) {
    pdl_wait();
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    if (i >= g.m[0] || j >= g.m[1]) return;
    const double inv = s->inv_scale;
    const int k0 = blockIdx.z * kZ, k1 = min(k0 + kZ, g.m[2]);
    for (int k = k0; k < k1; ++k) {
        const int64_t p = ((int64_t)k * g.m[1] + j) * g.m[0] + i;
        const int64_t f = g.off + i + (int64_t)g.e[0] * (j + (int64_t)g.e[1] * k);
        us[f] = fma(to_f64(e[p]), inv, us[f]);
    }
}

// Grid of the level kernels with a thread per column of zper planes: as many
// planes, up to kZ, as still leave six blocks per SM (a small level's planes one
// after the other cost a memory latency each: 9 us a pass on 32^3 with eight,
// 3 with one).
inline dim3 thin_grid(int mx, int my, int mz, int& zper) {
    const int tx = (mx + kTX - 1) / kTX, ty = (my + kTY - 1) / kTY;
    const int64_t planes = (int64_t)tx * ty * mz;
    zper = (int)std::max<int64_t>(1, std::min<int64_t>(kZ, planes / ((int64_t)device_sms() * 6)));
    return dim3(tx, ty, (mz + zper - 1) / zper);
}

inline dim3 hgrid(const int (&m)[3], int zper) {
    return dim3((m[0] + kTX - 1) / kTX, (m[1] + kTY - 1) / kTY, (m[2] + zper - 1) / zper);
}

}  // namespace

// ------------------------------------------------------------------ plan

HelmPlan helm_plan(const HelmGeo& g, int max_levels) {
    HelmPlan P{};
    int m[3] = {g.m[0], g.m[1], g.m[2]};
    double h2 = 1.0 / g.ih2;
    for (int l = 0; l < max_levels && l < kHelmMaxLevels; ++l) {
        for (int a = 0; a < 3; ++a) {
            P.lv[l].m[a] = m[a];
            P.lv[l].kind[a] = g.kind[a];
        }
        P.lv[l].ih2 = 1.0 / h2;
        P.nl = l + 1;
        bool ok = true;
        int mc[3];
        for (int a = 0; a < 3; ++a) {
            if (g.kind[a] == HELM_ZERO) {
                ok = ok && (m[a] % 2 == 1) && m[a] >= 5;
                mc[a] = (m[a] - 1) / 2;
            } else {
                ok = ok && (m[a] % 2 == 0) && m[a] >= 4;
                mc[a] = m[a] / 2;
            }
        }
        if (!ok) break;
        for (int a = 0; a < 3; ++a) m[a] = mc[a];
        h2 *= 4.0;
    }
    return P;
}

// ------------------------------------------------------------- launchers

namespace {
inline HLev hlev(const HelmLevelDesc& d) {
    HLev L;
    for (int a = 0; a < 3; ++a) {
        L.m[a] = d.m[a];
        L.kind[a] = d.kind[a];
    }
    L.ih2 = (float)d.ih2;
    return L;
}
inline int64_t hcount(const HelmLevelDesc& d) { return (int64_t)d.m[0] * d.m[1] * d.m[2]; }
inline bool rb_ok(const HelmLevelDesc& d) {
    for (int a = 0; a < 3; ++a)
        if (d.kind[a] == HELM_PERIODIC && d.m[a] % 2 == 1 && d.m[a] > 1) return false;
    return true;
}
}  // namespace

int64_t launch_hmg_setup(const HelmGeo& g, const double* un, const double* nu, double tau, double* sig64,
                         float* sig32, double* us, double* partials, cudaStream_t st, FinSpec fin) {
    const dim3 gr = hgrid(g.m, kZ);
    hmg_setup_kernel<<<gr, dim3(kTX, kTY), 0, st>>>(g, un, nu, tau, sig64, sig32, us, partials, fin);
    count_launch();
    launch_helm_wall_zero(g, us, st);
    return (int64_t)gr.x * gr.y * gr.z;
}

void launch_hmg_sigma(const HelmPlan& P, float* const* sig, cudaStream_t st) {
    for (int l = 0; l + 1 < P.nl; ++l) {
        const HLev F = hlev(P.lv[l]), Cg = hlev(P.lv[l + 1]);
        dim3 gr((Cg.m[0] + kTX - 1) / kTX, (Cg.m[1] + kTY - 1) / kTY, Cg.m[2]);
        launch_pdl(hmg_restrict_kernel, gr, dim3(kTX, kTY), 0, st, F, Cg, sig[l], sig[l + 1]);
        count_launch();
    }
}

void launch_hmg_residual64(const HelmGeo& g, const double* un, const double* sig, const double* us, const Scal* s,
                           float* r32, double* partials, cudaStream_t st, FinSpec fin) {
    const int tx = (g.m[0] + kTX - 1) / kTX, ty = (g.m[1] + kTY - 1) / kTY;
    const int zper = march_planes((int64_t)tx * ty, g.m[2], kPerSM);
    const dim3 gr(tx, ty, (g.m[2] + zper - 1) / zper);
    launch_pdl(hmg_residual64_kernel, gr, dim3(kTX, kTY), 0, st, g, un, sig, us, s, r32, partials, zper, fin);
    count_launch();
}

// z32 = V f32 on FP32 vectors of the finest level (f32 and z32 are not
// the work arrays of level 0, which the V-cycle uses for its own x and f)
static void hmg_vcycle_core(const HelmPlan& P, const HelmWork& W, const float* f0, float* x0, int nu1, int nu2,
                            int coarse_sweeps, float omega, cudaStream_t st);

void launch_hmg_vcycle32(const HelmPlan& P, const HelmWork& W, const float* r32, float* z32, int nu1, int nu2,
                         int coarse_sweeps, float omega, cudaStream_t st) {
    hmg_vcycle_core(P, W, r32, z32, nu1, nu2, coarse_sweeps, omega, st);
}

// First level of the tail launch (P.nl: none); the finest level stays out.
static int tail_level(const HelmPlan& P) {
    int t = P.nl;
    while (t > 1 && hcount(P.lv[t - 1]) <= kTailUnknowns) --t;
    return t;
}

static void launch_tail(const HelmPlan& P, const HelmWork& W, int l0, const float* f, float* x, int nu1, int nu2,
                        int coarse_sweeps, float omega, cudaStream_t st) {
    HTail a{};
    a.n = P.nl - l0;
    a.nu1 = nu1;
    a.nu2 = nu2;
    a.coarse_sweeps = coarse_sweeps;
    a.omega = omega;
    a.f = f;
    a.x = x;
    int64_t cells = hcount(P.lv[l0]);  // the residual's buffer
    for (int l = l0; l < P.nl; ++l) {
        HTailLevel& T = a.lv[l - l0];
        T.L = hlev(P.lv[l]);
        T.jac = rb_ok(P.lv[l]) ? 0 : 1;
        T.mp = fast_div_mul((T.L.m[0] + 1) / 2);
        T.m0 = fast_div_mul(T.L.m[0]);
        T.m1 = fast_div_mul(T.L.m[1]);
        T.sig = W.sig[l];
        cells += 3 * hcount(P.lv[l]);
    }
    // at most 4096 (1 + 3 (1 + 1/8 + ...)) floats
    static SmemOptIn opted;
    allow_smem(opted, (const void*)hmg_tail_kernel, 4 * 4096 * 5);  // a failure shows at the launch
    launch_pdl(hmg_tail_kernel, 1, kTailThreads, sizeof(float) * (size_t)cells, st, a);
    count_launch();
}

static void hmg_vcycle_core(const HelmPlan& P, const HelmWork& W, const float* f0, float* x0, int nu1, int nu2,
                            int coarse_sweeps, float omega, cudaStream_t st) {
    auto F = [&](int l) { return l == 0 ? f0 : (const float*)W.f[l]; };
    auto X = [&](int l) { return l == 0 ? x0 : W.x[l]; };
    // zero: x starts from 0 (only the quads' first pass takes that without a cleared x)
    auto smooth = [&](int l, int sweeps, bool reverse, bool zero) {
        const HLev L = hlev(P.lv[l]);
        const dim3 gr = hgrid(P.lv[l].m, kZ);
        const bool quads = P.lv[l].m[0] % 4 == 0 && P.lv[l].m[0] >= 4 * kTX &&
                           ((uintptr_t)F(l) | (uintptr_t)W.sig[l] | (uintptr_t)X(l)) % 16 == 0;
        if (zero && !(rb_ok(P.lv[l]) && quads && sweeps > 0))
            cudaMemsetAsync(X(l), 0, sizeof(float) * hcount(P.lv[l]), st);
        if (rb_ok(P.lv[l]) && quads) {
            const dim3 g4((P.lv[l].m[0] / 4 + kTX - 1) / kTX, (P.lv[l].m[1] + kTY - 1) / kTY, P.lv[l].m[2]);
            for (int s = 0; s < sweeps; ++s)
                for (int h = 0; h < 2; ++h) {
                    const int color = reverse ? 1 - h : h;
                    launch_pdl(hmg_rb4_kernel, g4, dim3(kTX, kTY), 0, st, L, F(l), W.sig[l], X(l), color,
                        omega, zero && s == 0 && h == 0 ? 1 : 0);
                    count_launch();
                }
        } else if (rb_ok(P.lv[l])) {
            int zper;
            const dim3 gp = thin_grid((P.lv[l].m[0] + 1) / 2, P.lv[l].m[1], P.lv[l].m[2], zper);
            for (int s = 0; s < sweeps; ++s)
                for (int h = 0; h < 2; ++h) {
                    const int color = reverse ? 1 - h : h;
                    launch_pdl(hmg_rbgs_pair_kernel, gp, dim3(kTX, kTY), 0, st, L, F(l), W.sig[l], X(l), color,
                        omega, zper);
                    count_launch();
                }
        } else {  // damped Jacobi, ping-pong through the level's residual buffer, ending in x
            const int64_t n = hcount(P.lv[l]);
            for (int s = 0; s < sweeps; ++s) {
                hmg_smooth_kernel<true><<<gr, dim3(kTX, kTY), 0, st>>>(L, F(l), W.sig[l], X(l), W.r[l], 0,
                                                                      0.8f);
                cudaMemcpyAsync(X(l), W.r[l], sizeof(float) * n, cudaMemcpyDeviceToDevice, st);
                count_launch();
            }
        }
    };
    const int tail = tail_level(P);
    for (int l = 0; l < P.nl; ++l) {
        if (l == tail) {
            launch_tail(P, W, l, F(l), X(l), nu1, nu2, coarse_sweeps, omega, st);
            break;
        }
        if (l == P.nl - 1) {
            smooth(l, coarse_sweeps, false, true);
            break;
        }
        smooth(l, nu1, false, true);
        const HLev L = hlev(P.lv[l]), Cg = hlev(P.lv[l + 1]);
        const bool q4 = P.lv[l].m[0] % 4 == 0 && P.lv[l].m[0] >= 4 * kTX &&
                        ((uintptr_t)F(l) | (uintptr_t)W.sig[l] | (uintptr_t)X(l) | (uintptr_t)W.r[l]) % 16 == 0;
        if (q4)
            launch_pdl(hmg_residual4_kernel,
                       dim3((P.lv[l].m[0] / 4 + kTX - 1) / kTX, (P.lv[l].m[1] + kTY - 1) / kTY, P.lv[l].m[2]),
                       dim3(kTX, kTY), 0, st, L, F(l), W.sig[l], X(l), W.r[l]);
        else {
            int zper;
            const dim3 gt = thin_grid(P.lv[l].m[0], P.lv[l].m[1], P.lv[l].m[2], zper);
            launch_pdl(hmg_residual_kernel, gt, dim3(kTX, kTY), 0, st, L, F(l), W.sig[l], X(l), W.r[l], zper);
        }
        dim3 gr((Cg.m[0] + kTX - 1) / kTX, (Cg.m[1] + kTY - 1) / kTY, Cg.m[2]);
        launch_pdl(hmg_restrict_kernel, gr, dim3(kTX, kTY), 0, st, L, Cg, W.r[l], W.f[l + 1]);
        count_launch(2);
    }
    for (int l = std::min(tail, P.nl - 1) - 1; l >= 0; --l) {
        const HLev L = hlev(P.lv[l]), Cg = hlev(P.lv[l + 1]);
        if (L.m[0] % 4 == 0 && L.kind[0] != HELM_ZERO && (uintptr_t)X(l) % 16 == 0) {
            const unsigned nq = (unsigned)(L.m[0] / 4), total = nq * (unsigned)(L.m[1] * L.m[2]);
            launch_pdl(hmg_prolong4_kernel, (total + kTX * kTY - 1) / (kTX * kTY), kTX * kTY, 0, st, L, Cg, nq,
                       fast_div_mul((int)nq), fast_div_mul(L.m[1]), total, (const float*)X(l + 1), X(l));
        } else {
            dim3 gr((L.m[0] + kTX - 1) / kTX, (L.m[1] + kTY - 1) / kTY, L.m[2]);
            launch_pdl(hmg_prolong_kernel, gr, dim3(kTX, kTY), 0, st, L, Cg, X(l + 1), X(l));
        }
        count_launch();
        smooth(l, nu2, true, false);
    }
}

}  // namespace paris

namespace paris {

int64_t launch_hmg_matvec32(const HelmPlan& P, const float* sig, const float* d, float* q, double* partials,
                            cudaStream_t st, FinSpec fin) {
    const HLev L = hlev(P.lv[0]);
    // quads where the rows fill a warp
    if (L.m[0] % 4 == 0 && L.m[0] >= 4 * kTX && ((uintptr_t)sig | (uintptr_t)d | (uintptr_t)q) % 16 == 0) {
        const int tx = (L.m[0] / 4 + kTX - 1) / kTX, ty = (L.m[1] + kTY - 1) / kTY;
        const int zper = march_planes((int64_t)tx * ty, L.m[2], 6);
        const dim3 g4(tx, ty, (L.m[2] + zper - 1) / zper);
        launch_pdl(hmg_matvec4_kernel, g4, dim3(kTX, kTY), 0, st, L, sig, d, q, partials, zper, fin);
        count_launch();
        return (int64_t)g4.x * g4.y * g4.z;
    }
    const int tx = (L.m[0] + kTX - 1) / kTX, ty = (L.m[1] + kTY - 1) / kTY;
    const int zper = march_planes((int64_t)tx * ty, L.m[2], 6);
    const dim3 gr(tx, ty, (L.m[2] + zper - 1) / zper);
    launch_pdl(hmg_matvec32_kernel, gr, dim3(kTX, kTY), 0, st, L, sig, d, q, partials, zper, fin);
    count_launch();
    return (int64_t)gr.x * gr.y * gr.z;
}

void launch_hmg_accumulate(const HelmGeo& g, const float* e, const Scal* s, double* us, cudaStream_t st) {
    launch_pdl(hmg_accumulate_kernel, hgrid(g.m, kZ), dim3(kTX, kTY), 0, st, g, e, s, us);
    count_launch();
}

}  // namespace paris
