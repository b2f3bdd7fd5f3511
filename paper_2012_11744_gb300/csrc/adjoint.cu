// Adjoint (reverse-mode derivative) of the projection step.
//
// The paper has no adjoint; it follows from Eqs. fotm and poisson.  With
// B = diag(beta), D the divergence and G the face gradient (D = -G^T on
// non-wall faces), the projection is u = u* - B G L^{-1} D u* (dt cancels),
// L = D B G.  For a loss with gradient g = dLoss/du, and q the mean-free
// solution of L q = D (B g):
//   dLoss/du*_f   = g_f - (G q)_f
//   dLoss/dbeta_f = dt (G p)_f ((G q)_f - g_f)
//   dLoss/dC_c    = sum over the faces f of c of dLoss/dbeta_f dbeta_f/dC_c,
//                   dbeta_f/dC_c = -beta_f^2 (rho1 - rho2) / 2
// (beta_f = 2/(rho_L + rho_R), rho = rho1 C + rho2 (1 - C)).  Wall faces carry
// neither velocity nor coefficient, so every derivative there is zero.
#include "kernels.cuh"

namespace paris {

namespace {
constexpr int kTX = 32, kTY = 8, kZ = 8;
}

// c = D (B g): the divergence of the face field beta*g (walls carry no flux).
// FP64 instructions bound it (two lanes a clock and SM): a thread marches
// through planes, the flux through the z-face above carried to the next one,
// and nothing is summed that the solve's own prologue sums.  128^3 77 -> 53 us.
__global__ void __launch_bounds__(kTX* kTY)
    weighted_div_kernel(Geo g, const double* __restrict__ bx, const double* __restrict__ by,
                        const double* __restrict__ bz, const double* __restrict__ gx,
                        const double* __restrict__ gy, const double* __restrict__ gz, double inv_h,
                        double* __restrict__ out) {
    const int i = blockIdx.x * kTX + threadIdx.x;
    const int j = blockIdx.y * kTY + threadIdx.y;
    if (i >= g.nx || j >= g.ny) return;
    const int k0 = blockIdx.z * kZ, k1 = min(k0 + kZ, g.nz);
    const AxisNb ax = axis_nb(i, g.nx, g.wx), ay = axis_nb(j, g.ny, g.wy);
    double wm = 0.0;
    if (!(g.wz && k0 == 0)) wm = bz[g.fz(i, j, k0)] * gz[g.fz(i, j, k0)];
    for (int k = k0; k < k1; ++k) {
        const AxisNb az = axis_nb(k, g.nz, g.wz);
        const int64_t fxp = g.fx(ax.fp, j, k), fxm = g.fx(i, j, k);
        const int64_t fyp = g.fy(i, ay.fp, k), fym = g.fy(i, j, k);
        const int64_t fzp = g.fz(i, j, az.fp);
        const double up = ax.wp ? 0.0 : bx[fxp] * gx[fxp];
        const double um = ax.wm ? 0.0 : bx[fxm] * gx[fxm];
        const double vp = ay.wp ? 0.0 : by[fyp] * gy[fyp];
        const double vm = ay.wm ? 0.0 : by[fym] * gy[fym];
        const double wp = az.wp ? 0.0 : bz[fzp] * gz[fzp];
        out[g.cidx(i, j, k)] = (((up - um) + (vp - vm)) + (wp - wm)) * inv_h;
        wm = wp;
    }
}

void launch_weighted_div(const Geo& g, const double* bx, const double* by, const double* bz, const double* gx,
                         const double* gy, const double* gz, double inv_h, double* out, cudaStream_t st) {
    dim3 gr((g.nx + kTX - 1) / kTX, (g.ny + kTY - 1) / kTY, (g.nz + kZ - 1) / kZ);
    weighted_div_kernel<<<gr, dim3(kTX, kTY), 0, st>>>(g, bx, by, bz, gx, gy, gz, inv_h, out);
    count_launch();
}

// Per face: gq = (q_R - q_L)/h, gp = (p_R - p_L)/h;
//   gus = g - gq,  gbeta = dt gp (gq - g) = -(dt gp) gus;  both 0 on wall faces.
// Five FP64 instructions a face, which bound it: 128^3 88 -> 64 us (eight before).
// One thread per cell handles its - faces (and the + wall face of the last
// cell along a wall axis).
__global__ void adjoint_faces_kernel(Geo g, const double* __restrict__ p, const double* __restrict__ q,
                                     double inv_h, double dt_h, const double* __restrict__ gx,
                                     const double* __restrict__ gy, const double* __restrict__ gz,
                                     double* __restrict__ usx, double* __restrict__ usy,
                                     double* __restrict__ usz, double* __restrict__ bbx,
                                     double* __restrict__ bby, double* __restrict__ bbz) {
    const int i = blockIdx.x * kTX + threadIdx.x;
    const int j = blockIdx.y * kTY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.nx || j >= g.ny) return;
    const int64_t c = g.cidx(i, j, k);
    const double pc = p[c], qc = q[c];
    AxisNb ax = axis_nb(i, g.nx, g.wx), ay = axis_nb(j, g.ny, g.wy), az = axis_nb(k, g.nz, g.wz);
    auto face = [&](bool wall, int64_t f, int64_t left, const double* gin, double* us, double* bb) {
        if (wall) {
            us[f] = 0.0;
            bb[f] = 0.0;
            return;
        }
        const double v = fma(q[left] - qc, inv_h, gin[f]);
        us[f] = v;
        bb[f] = (p[left] - pc) * dt_h * v;
    };
    face(ax.wm, g.fx(i, j, k), g.cidx(ax.m, j, k), gx, usx, bbx);
    face(ay.wm, g.fy(i, j, k), g.cidx(i, ay.m, k), gy, usy, bby);
    face(az.wm, g.fz(i, j, k), g.cidx(i, j, az.m), gz, usz, bbz);
    if (g.wx && i == g.nx - 1) { usx[g.fx(g.nx, j, k)] = 0.0; bbx[g.fx(g.nx, j, k)] = 0.0; }
    if (g.wy && j == g.ny - 1) { usy[g.fy(i, g.ny, k)] = 0.0; bby[g.fy(i, g.ny, k)] = 0.0; }
    if (g.wz && k == g.nz - 1) { usz[g.fz(i, j, g.nz)] = 0.0; bbz[g.fz(i, j, g.nz)] = 0.0; }
}

void launch_adjoint_faces(const Geo& g, const double* p, const double* q, double inv_h, double dt,
                          const double* gx, const double* gy, const double* gz, double* usx,
                          double* usy, double* usz, double* bbx, double* bby, double* bbz,
                          cudaStream_t st) {
    dim3 gr((g.nx + kTX - 1) / kTX, (g.ny + kTY - 1) / kTY, g.nz);
    adjoint_faces_kernel<<<gr, dim3(kTX, kTY), 0, st>>>(g, p, q, inv_h, dt * inv_h, gx, gy, gz, usx, usy, usz,
                                                         bbx, bby, bbz);
    count_launch();
}

// dLoss/dC_c = -(rho1 - rho2)/2 * sum over the six non-wall faces of c of
// gbeta_f beta_f^2 (gather: one thread per cell, no atomics).
__global__ void face_coeffs_adjoint_kernel(Geo g, double half_drho, const double* __restrict__ bx,
                                           const double* __restrict__ by,
                                           const double* __restrict__ bz,
                                           const double* __restrict__ gbx,
                                           const double* __restrict__ gby,
                                           const double* __restrict__ gbz, double* __restrict__ gC) {
    const int i = blockIdx.x * kTX + threadIdx.x;
    const int j = blockIdx.y * kTY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.nx || j >= g.ny) return;
    AxisNb ax = axis_nb(i, g.nx, g.wx), ay = axis_nb(j, g.ny, g.wy), az = axis_nb(k, g.nz, g.wz);
    auto term = [](bool wall, const double* b, const double* gb, int64_t f) {
        if (wall) return 0.0;
        const double bf = b[f];
        return gb[f] * bf * bf;
    };
    double s = term(ax.wm, bx, gbx, g.fx(i, j, k)) + term(ax.wp, bx, gbx, g.fx(ax.fp, j, k));
    s += term(ay.wm, by, gby, g.fy(i, j, k)) + term(ay.wp, by, gby, g.fy(i, ay.fp, k));
    s += term(az.wm, bz, gbz, g.fz(i, j, k)) + term(az.wp, bz, gbz, g.fz(i, j, az.fp));
    gC[g.cidx(i, j, k)] = -half_drho * s;
}

void launch_face_coeffs_adjoint(const Geo& g, double rho1, double rho2, const double* bx,
                                const double* by, const double* bz, const double* gbx,
                                const double* gby, const double* gbz, double* gC, cudaStream_t st) {
    dim3 gr((g.nx + kTX - 1) / kTX, (g.ny + kTY - 1) / kTY, g.nz);
    face_coeffs_adjoint_kernel<<<gr, dim3(kTX, kTY), 0, st>>>(g, 0.5 * (rho1 - rho2), bx, by, bz, gbx,
                                                               gby, gbz, gC);
    count_launch();
}

}  // namespace paris
