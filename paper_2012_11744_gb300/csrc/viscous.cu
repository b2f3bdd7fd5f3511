// Implicit viscous step on one velocity component (Sec. 3.2.3, Eq.
// muelliptic): the kernels of the Jacobi-preconditioned conjugate gradients
// that solve its symmetric positive definite form
//
//     (diag(1/(tau nu)) - Lap_h) u* = u^n / (tau nu)
//
// on the component's unknowns, its face grid without the wall faces of its
// own axis (where the component is zero).  Lap_h is the 7-point Laplacian
// with spacing h; beyond the ends of an axis the value is the wrapped one
// (periodic), zero (the component's own wall faces) or minus the end value
// (no-slip for a tangential component: zero velocity on the wall, half a
// cell away, Sec. 2.2).
//
// u^n, nu and u* are full face arrays (the library's face layout); the
// Krylov vectors r, d, q and the per-unknown sigma = 1/(tau nu) and
// w = 1/diag hold only the unknowns, x fastest.
//
// What bounds these kernels is the FP64 pipe (1/64 of the FP32 rate on this
// GPU, 0.58e12 instructions a second), so everything that does not change
// during a solve is formed once: sigma and w by one setup pass, where each
// product and update used to divide by tau nu and by the diagonal (a division
// is about ten FP64 instructions).  A Laplacian is five additions of
// neighbours and one fused step with the integer diagonal count; maxima and
// non-finite tests are integer comparisons; z = w r is formed where it is
// used and never stored.  That leaves 9 FP64 instructions per unknown for the
// product, 5 for the update and 2 for the direction.  At 128^3 (ncu, cold
// caches): product 97 -> 56 us, update 118 -> 41 us a launch, the FP64 pipe 80 %
// busy while the product's blocks run; a step of three components 55.3 ->
// 26.0 ms.  The product's threads own z-columns of a 32 x 8 tile (no index
// divisions), the column's values carried from plane to plane.
#include <algorithm>

#include "helm.cuh"

namespace paris {

namespace {

constexpr int kTX = 32, kTY = 8;  // tile of the marching kernels
constexpr int kPerSM = 4;         // their resident blocks per SM (at most 64 registers)

__device__ __forceinline__ int64_t helm_block() {
    return ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
}
__device__ __forceinline__ int64_t helm_blocks() { return (int64_t)gridDim.x * gridDim.y * gridDim.z; }

// sigma = 1/(tau nu) and w = 1/(sigma + diag(-Lap_h)) on the unknowns;
// u* = u^n there (the initial guess), 0 on the component's wall faces;
// partials of |b|^2, max |b| and the non-finite count (a nu that is not
// positive counts), with b = sigma u^n
__global__ void __launch_bounds__(kTX* kTY, kPerSM) helm_init_kernel(HelmGeo g, const double* __restrict__ un,
                                                            const double* __restrict__ nu, double tau,
                                                            double* __restrict__ sig, double* __restrict__ w,
                                                            double* __restrict__ us, double* partials, int zper, FinSpec fin) {
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    double l2[1] = {0.0};
    unsigned long long bk = 0;
    unsigned nf = 0;
    if (i < g.m[0] && j < g.m[1]) {
        const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, g.m[2]);
        const int dxy = HelmColumn::count(g.kind[0], g.m[0], i) + HelmColumn::count(g.kind[1], g.m[1], j);
        for (int k = k0; k < k1; ++k) {
            const int64_t p = ((int64_t)k * g.m[1] + j) * g.m[0] + i;
            const int64_t f = g.off + i + (int64_t)g.e[0] * (j + (int64_t)g.e[1] * k);
            const double v = un[f], nv = nu[f];
            us[f] = v;
            const double s = recip64_rn(tau * nv);
            sig[p] = s;
            w[p] = recip64_rn(fma((double)(dxy + HelmColumn::count(g.kind[2], g.m[2], k)), g.ih2, s));
            const double b = s * v;
            l2[0] = fma(b, b, l2[0]);
            const unsigned long long kb = abs_key(b);
            bk = kb > bk ? kb : bk;
            nf += (key_nonfinite(kb) || !(nv > 0.0)) ? 1u : 0u;
        }
    }
    block_reduce_sums_kc<1>(l2, bk, nf, partials, helm_block(), tid);
    finalize_last_block(partials, helm_blocks(), fin, tid);
}

// the two wall planes of the component's own axis: u* = 0 there
__global__ void helm_wall_zero_kernel(HelmGeo g, double* __restrict__ us) {
    const int c = g.comp, a1 = c == 0 ? 1 : 0, a2 = c == 2 ? 1 : 2;
    const int64_t plane = (int64_t)g.e[a1] * g.e[a2];
    const int64_t se[3] = {1, g.e[0], (int64_t)g.e[0] * g.e[1]};
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < 2 * plane; w += (int64_t)gridDim.x * blockDim.x) {
        const int side = w >= plane;
        const int64_t rem = w - side * plane;
        const int64_t i2 = rem / g.e[a1], i1 = rem - i2 * g.e[a1];
        us[i1 * se[a1] + i2 * se[a2] + (int64_t)side * (g.e[c] - 1) * se[c]] = 0.0;
    }
}

// r = sigma (u^n - x) + Lap_h x; partials of r . r, max |r|, the non-finite
// count, r . w r
__global__ void __launch_bounds__(kTX* kTY, kPerSM) helm_residual_kernel(HelmGeo g, const double* __restrict__ un,
                                                                const double* __restrict__ sig,
                                                                const double* __restrict__ w,
                                                                const double* __restrict__ x, double* __restrict__ r,
                                                                double* partials, int zper, FinSpec fin) {
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    double sums[2] = {0.0, 0.0};  // r . r and r . z
    unsigned long long rk = 0;
    unsigned nf = 0;
    if (i < g.m[0] && j < g.m[1]) {
        const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, g.m[2]);
        const int64_t se[3] = {1, g.e[0], (int64_t)g.e[0] * g.e[1]};
        HelmColumn col(g, x + g.off, se, i, j, k0);
        for (int k = k0; k < k1; ++k) {
            const int64_t p = ((int64_t)k * g.m[1] + j) * g.m[0] + i;
            const int64_t f = g.off + i + (int64_t)g.e[0] * (j + (int64_t)g.e[1] * k);
            double xc;
            const double lap = col.next(k, xc);
            const double rp = fma(g.ih2, lap, sig[p] * (un[f] - xc));
            r[p] = rp;
            sums[0] = fma(rp, rp, sums[0]);
            sums[1] = fma(rp, rp * w[p], sums[1]);
            const unsigned long long kr = abs_key(rp);
            rk = kr > rk ? kr : rk;
            nf += key_nonfinite(kr);
        }
    }
    block_reduce_sums_kc<2>(sums, rk, nf, partials, helm_block(), tid);
    finalize_last_block(partials, helm_blocks(), fin, tid);
}

// q = sigma d - Lap_h d and the partials of d . q
__global__ void __launch_bounds__(kTX* kTY, kPerSM) helm_matvec_dot_kernel(HelmGeo g, const double* __restrict__ sig,
                                                                  const double* __restrict__ d,
                                                                  double* __restrict__ q, double* partials,
                                                                  int zper, FinSpec fin) {
    pdl_wait();
    const int i = blockIdx.x * kTX + threadIdx.x, j = blockIdx.y * kTY + threadIdx.y;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    double dq = 0.0;
    if (i < g.m[0] && j < g.m[1]) {
        const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, g.m[2]);
        const int64_t su[3] = {1, g.m[0], (int64_t)g.m[0] * g.m[1]};
        HelmColumn col(g, d, su, i, j, k0);
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
            const int64_t p = ((int64_t)k * g.m[1] + j) * g.m[0] + i;
            double dc;
            const double lap = col.next(k, dc);
            const double qp = fma(-g.ih2, lap, sig[p] * dc);
            q[p] = qp;
            dq = fma(dc, qp, dq);
        }
    }
    double acc[1] = {dq};
    const int op[1] = {0};
    block_reduce_store<1>(acc, op, partials, helm_block(), tid);
    finalize_last_block(partials, helm_blocks(), fin, tid);
}

constexpr int kUU = 4;  // unknowns in flight per thread of the update

// x += alpha d, r -= alpha q; partials as the residual kernel's.  A
// grid-stride loop on resident blocks only (no last wave), four unknowns in
// flight per thread.
__global__ void __launch_bounds__(kRedThreads, kPerSM) helm_update_kernel(HelmGeo g, unsigned n, unsigned mul0,
                                                                         unsigned mul1,
                                                                         const double* __restrict__ w,
                                                                         const Scal* __restrict__ s,
                                                                         const double* __restrict__ d,
                                                                         const double* __restrict__ q,
                                                                         double* __restrict__ x,
                                                                         double* __restrict__ r, double* partials,
                                                                         FinSpec fin) {
    pdl_wait();
    const double alpha = s->alpha;
    double sums[2] = {0.0, 0.0};
    unsigned long long rk = 0;
    unsigned nf = 0;
    const unsigned m0 = (unsigned)g.m[0], m1 = (unsigned)g.m[1];
    const bool flat = g.e[0] == g.m[0] && g.e[1] == g.m[1];  // the face array minus its offset is the vector
    auto face = [&](unsigned p) {
        if (flat) return g.off + (int64_t)p;
        const unsigned row = fast_div(p, m0, mul0), k = fast_div(row, m1, mul1);
        return g.off + (int64_t)(p - row * m0) + (int64_t)g.e[0] * ((row - k * m1) + (int64_t)g.e[1] * k);
    };
    const unsigned stride = gridDim.x * blockDim.x;
    auto one = [&](double rp, double wp) {
        sums[0] = fma(rp, rp, sums[0]);
        sums[1] = fma(rp, rp * wp, sums[1]);
        const unsigned long long kr = abs_key(rp);
        rk = kr > rk ? kr : rk;
        nf += key_nonfinite(kr);
    };
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; p + (int64_t)(kUU - 1) * stride < n; p += (int64_t)kUU * stride) {
        double dv[kUU], qv[kUU], xv[kUU], rv[kUU], wv[kUU];
        int64_t f[kUU];
#pragma unroll
        for (int u = 0; u < kUU; ++u) {
            const int64_t c = p + (int64_t)u * stride;
            f[u] = face((unsigned)c);
            dv[u] = d[c];
            qv[u] = q[c];
            rv[u] = r[c];
            wv[u] = w[c];
            xv[u] = x[f[u]];
        }
#pragma unroll
        for (int u = 0; u < kUU; ++u) {
            x[f[u]] = fma(alpha, dv[u], xv[u]);
            rv[u] = fma(-alpha, qv[u], rv[u]);
            r[p + (int64_t)u * stride] = rv[u];
            one(rv[u], wv[u]);
        }
    }
    for (; p < n; p += stride) {
        const int64_t f = face((unsigned)p);
        x[f] = fma(alpha, d[p], x[f]);
        const double rp = fma(-alpha, q[p], r[p]);
        r[p] = rp;
        one(rp, w[p]);
    }
    block_reduce_sums_kc<2>(sums, rk, nf, partials, blockIdx.x, threadIdx.x);
    finalize_last_block(partials, gridDim.x, fin, threadIdx.x);
}

// d = w r + beta d (first: d = w r)
__global__ void helm_direction_kernel(int64_t n, const Scal* __restrict__ s, const double* __restrict__ w,
                                      const double* __restrict__ r, double* __restrict__ d, int first) {
    pdl_wait();
    const double beta = s->beta;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; p + 3 * stride < n; p += 4 * stride) {  // four unknowns in flight
        double z[4], dv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            z[u] = w[p + u * stride] * r[p + u * stride];
            dv[u] = first ? 0.0 : d[p + u * stride];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) d[p + u * stride] = first ? z[u] : fma(beta, dv[u], z[u]);
    }
    for (; p < n; p += stride) {
        const double z = w[p] * r[p];
        d[p] = first ? z : fma(beta, d[p], z);
    }
}

// nu_f = (mu_L + mu_R) / (rho_L + rho_R) on every face of the component,
// mu and rho from Eq. muH in the two cells sharing the face; 0 on its wall
// faces.  Rounded products and sums (no contraction), in the order written.
// Bound by the FP64 pipe: a cell's mu and rho (7 instructions) are formed once
// and reach its other face through the plane before (z), the warp (x) or the
// tile (y), where every face formed both cells' (788 -> 572 us at 256^3).
__global__ void __launch_bounds__(kTX* kTY, kPerSM) helm_face_nu_kernel(HelmGeo g, int nx, int ny, int nz,
                                                                       const double* __restrict__ C, double mu1,
                                                                       double mu2, double rho1, double rho2,
                                                                       double* __restrict__ nu, int zper) {
    __shared__ double2 sh[2][kTY][kTX];  // (mu, rho) of the tile's cells, by plane parity
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int i = blockIdx.x * kTX + tx, j = blockIdx.y * kTY + ty, comp = g.comp;
    const int ic = min(i, nx - 1), jc = min(j, ny - 1);  // idle threads shadow a cell
    const int k0 = blockIdx.z * zper, k1 = min(k0 + zper, nz);
    const bool in = i < nx && j < ny;
    auto cell = [&](int ci, int cj, int ck) {
        const double c = C[((int64_t)ck * ny + cj) * nx + ci], d = __dsub_rn(1.0, c);
        return make_double2(__dadd_rn(__dmul_rn(mu1, c), __dmul_rn(mu2, d)),
                            __dadd_rn(__dmul_rn(rho1, c), __dmul_rn(rho2, d)));
    };
    // the cell below the face along the component's axis: wrapped, or not read on a wall
    const int im = ic > 0 ? ic - 1 : nx - 1, jm = jc > 0 ? jc - 1 : ny - 1;
    const int pos0 = comp == 0 ? i : j;
    double2 below = make_double2(0.0, 0.0);
    if (comp == 2) below = cell(ic, jc, k0 > 0 ? k0 - 1 : nz - 1);
    for (int k = k0; k < k1; ++k) {
        const double2 here = cell(ic, jc, k);
        double2 lo = below;
        if (comp == 0) {
            lo = make_double2(__shfl_up_sync(0xffffffffu, here.x, 1), __shfl_up_sync(0xffffffffu, here.y, 1));
            if (tx == 0) lo = cell(im, jc, k);
        } else if (comp == 1) {
            sh[k & 1][ty][tx] = here;
            __syncthreads();
            lo = ty > 0 ? sh[k & 1][ty - 1][tx] : cell(ic, jm, k);
        }
        below = here;
        const int pos = comp == 2 ? k : pos0;
        if (in) {
            const int64_t f = i + (int64_t)g.e[0] * (j + (int64_t)g.e[1] * k);
            nu[f] = g.wall && pos == 0 ? 0.0 : div_pos(__dadd_rn(lo.x, here.x), __dadd_rn(lo.y, here.y));
        }
    }
    // the far wall face of the component's axis
    if (g.wall && in) {
        const int64_t se[3] = {1, g.e[0], (int64_t)g.e[0] * g.e[1]};
        if (comp == 2) {
            if (k1 == nz) nu[i + se[1] * j + se[2] * nz] = 0.0;
        } else if (pos0 == (comp == 0 ? nx : ny) - 1) {
            for (int k = k0; k < k1; ++k) nu[i + se[1] * j + se[2] * k + se[comp]] = 0.0;
        }
    }
}

}  // namespace

HelmGeo helm_geo(const Geo& g0, int comp, double h) {
    HelmGeo g{};
    const int n[3] = {g0.nx, g0.ny, g0.nz};
    const int wl[3] = {g0.wx, g0.wy, g0.wz};
    g.comp = comp;
    g.wall = wl[comp] ? 1 : 0;
    for (int a = 0; a < 3; ++a) {
        g.e[a] = n[a] + (a == comp && wl[a] ? 1 : 0);
        g.m[a] = n[a] - (a == comp && wl[a] ? 1 : 0);
        g.kind[a] = !wl[a] ? HELM_PERIODIC : (a == comp ? HELM_ZERO : HELM_NOSLIP);
    }
    const int64_t se[3] = {1, g.e[0], (int64_t)g.e[0] * g.e[1]};
    g.off = g.wall ? se[comp] : 0;
    g.ih2 = 1.0 / (h * h);
    return g;
}

int64_t helm_unknowns(const HelmGeo& g) { return (int64_t)g.m[0] * g.m[1] * g.m[2]; }
int64_t helm_faces(const HelmGeo& g) { return (int64_t)g.e[0] * g.e[1] * g.e[2]; }

// grid of the marching kernels; zper: planes per block
static dim3 helm_grid(const HelmGeo& g, int& zper) {
    const int tx = (g.m[0] + kTX - 1) / kTX, ty = (g.m[1] + kTY - 1) / kTY;
    zper = march_planes((int64_t)tx * ty, g.m[2], kPerSM);
    return dim3(tx, ty, (g.m[2] + zper - 1) / zper);
}

void launch_helm_init(const HelmGeo& g, const double* un, const double* nu, double tau, double* sig, double* w,
                      double* us, double* partials, cudaStream_t st, FinSpec fin) {
    int zper;
    const dim3 gr = helm_grid(g, zper);
    helm_init_kernel<<<gr, dim3(kTX, kTY), 0, st>>>(g, un, nu, tau, sig, w, us, partials, zper, fin);
    count_launch();
    launch_helm_wall_zero(g, us, st);
}

void launch_helm_wall_zero(const HelmGeo& g, double* us, cudaStream_t st) {
    if (!g.wall) return;
    const int c = g.comp, a1 = c == 0 ? 1 : 0, a2 = c == 2 ? 1 : 2;
    const int64_t n = 2 * (int64_t)g.e[a1] * g.e[a2];
    helm_wall_zero_kernel<<<elementwise_blocks(n), kRedThreads, 0, st>>>(g, us);
    count_launch();
}

void launch_helm_residual(const HelmGeo& g, const double* un, const double* sig, const double* w, const double* x,
                          double* r, double* partials, cudaStream_t st, FinSpec fin) {
    int zper;
    const dim3 gr = helm_grid(g, zper);
    helm_residual_kernel<<<gr, dim3(kTX, kTY), 0, st>>>(g, un, sig, w, x, r, partials, zper, fin);
    count_launch();
}

void launch_helm_matvec_dot(const HelmGeo& g, const double* sig, const double* d, double* q, double* partials,
                            cudaStream_t st, FinSpec fin) {
    int zper;
    const dim3 gr = helm_grid(g, zper);
    launch_pdl(helm_matvec_dot_kernel, gr, dim3(kTX, kTY), 0, st, g, sig, d, q, partials, zper, fin);
    count_launch();
}

void launch_helm_update(const HelmGeo& g, const double* w, const Scal* s, const double* d, const double* q,
                        double* x, double* r, double* partials, cudaStream_t st, FinSpec fin) {
    const int64_t n = helm_unknowns(g);
    int64_t nb = (n + kRedThreads * kUU - 1) / (kRedThreads * kUU);
    nb = std::max<int64_t>(1, std::min<int64_t>(nb, (int64_t)device_sms() * kPerSM));
    launch_pdl(helm_update_kernel, (unsigned)nb, kRedThreads, 0, st, g, (unsigned)n, fast_div_mul(g.m[0]), fast_div_mul(g.m[1]), w, s, d,
               q, x, r, partials, fin);
    count_launch();
}

void launch_helm_direction(int64_t n, const Scal* s, const double* w, const double* r, double* d, bool first,
                           cudaStream_t st) {
    launch_pdl(helm_direction_kernel, elementwise_blocks(n), kRedThreads, 0, st, n, s, w, r, d, first ? 1 : 0);
    count_launch();
}

void launch_helm_face_nu(const HelmGeo& g, const Geo& g0, const double* C, double mu1, double mu2, double rho1,
                         double rho2, double* nu, cudaStream_t st) {
    const int tx = (g0.nx + kTX - 1) / kTX, ty = (g0.ny + kTY - 1) / kTY;
    const int zper = march_planes((int64_t)tx * ty, g0.nz, kPerSM);
    helm_face_nu_kernel<<<dim3(tx, ty, (g0.nz + zper - 1) / zper), dim3(kTX, kTY), 0, st>>>(
        g, g0.nx, g0.ny, g0.nz, C, mu1, mu2, rho1, rho2, nu, zper);
    count_launch();
}

}  // namespace paris
