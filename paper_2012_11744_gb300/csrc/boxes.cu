// A small level's half of the V-cycle in one launch.
//
// Between the levels that fill the GPU and the single-block tail lie levels of
// 16^3 to 32^3 cells, whose colour passes, restriction and prolongation each
// take little more than the latency of a launch and of one dependent memory
// access: ten launches a level and V-cycle.  Here a block takes a box of the
// level and everything that its cells depend on: four colour passes reach four
// cells outwards, so the box with a halo of four holds all inputs, and the
// passes run in shared memory over boxes that shrink by one cell a pass, with
// a block barrier between them.  Down: the pre-smoothing from x = 0 and the
// restriction of the residual; up: the prolongation and the post-smoothing.
// A halo cell is updated by several blocks, each time to the same value; the
// passes are those of rbgs_kernel, the restriction that of
// restrict_residual_kernel, in the same arithmetic and order, so the results
// are the same bit for bit (from rho/2: those of the plane tiles, rho0.cu; where
// nx/2 is odd the z-column kernels stand in for these, whose restriction sums
// all faces and differs by rounding).
//
// What bounds it is latency: of the launch, of one access to memory, and of
// the dependent instructions of four passes on one SM.  So a thread owns one
// pair of cells of a row, loads its coefficients, inverse diagonals and
// right-hand sides straight into registers, all in flight together, and keeps
// them over the passes; shared memory holds x only.  (With all arrays staged in
// shared memory and read from there in each pass, the step on 32^3 cells, whose
// V-cycles have one such level, took 964 us; it takes 798 with this form and took
// 887 with ten launches a level.)  The coefficients are loaded before the wait for
// the preceding launch, which lets this one start early (818 -> 798 us).  Cells
// further than four steps along the axes from the box (in total) are not needed and
// have no thread: of the 864 pairs around 4^3 cells 424 remain, of the 1536 around
// 8 x 8 x 4 952.
#include "kernels.cuh"

#include <type_traits>

namespace paris {

namespace {

constexpr int kHalo = 4;  // two sweeps of two colours

// steps from local index l to the box's t cells along an axis
__host__ __device__ constexpr int axis_steps(int l, int t) { return l < kHalo ? kHalo - l : l >= kHalo + t ? l - (kHalo + t - 1) : 0; }

template <int TX, int TY, int TZ>
struct Box {
    static constexpr int bx = TX + 2 * kHalo, by = TY + 2 * kHalo, bz = TZ + 2 * kHalo;
    static constexpr int cells = bx * by * bz;
    static constexpr bool listed(int p, int m, int n) {
        const int a = axis_steps(2 * p, TX), b = axis_steps(2 * p + 1, TX);
        return (a < b ? a : b) + axis_steps(m, TY) + axis_steps(n, TZ) <= kHalo;
    }
    static constexpr int count() {
        int c = 0;
        for (int n = 0; n < bz; ++n)
            for (int m = 0; m < by; ++m)
                for (int p = 0; p < bx / 2; ++p) c += listed(p, m, n) ? 1 : 0;
        return c;
    }
    static constexpr int pairs = count();
    static constexpr int threads = (pairs + 31) / 32 * 32;
};

// the pairs that have a thread: p + 32 m + 1024 n
template <int TX, int TY, int TZ>
struct BoxTable {
    unsigned short v[Box<TX, TY, TZ>::pairs];
    constexpr BoxTable() : v() {
        using B = Box<TX, TY, TZ>;
        int c = 0;
        for (int n = 0; n < B::bz; ++n)
            for (int m = 0; m < B::by; ++m)
                for (int p = 0; p < B::bx / 2; ++p)
                    if (B::listed(p, m, n)) v[c++] = (unsigned short)(p + 32 * m + 1024 * n);
    }
};
template <int TX, int TY, int TZ>
__device__ constexpr BoxTable<TX, TY, TZ> kBoxTable{};

template <typename T, typename TB>
struct BoxArgs {
    Geo g, cg;
    int fac[3], tc[3];  // coarsening factors; coarse cells of a box along each axis
    const TB* b[3];  // coefficients, or rho/2 in b[0]
    const T* w;    // inverse diagonals (null: from the coefficients)
    const T* sig;  // diagonal excess, or null
    const T* f;
    const T* xin;  // up: x of the pre-smoothing
    T* x;
    T* fc;         // down: the coarse right-hand side
    const T* xc;   // up: the coarse solution
    T hs, rs;      // the right-hand side's factor in a pass; the operator's in the residual
    T omega;
    int sweeps;    // 1 or 2
};

__device__ __forceinline__ float2 ld_pair(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
__device__ __forceinline__ float2 ld_pair(const __half* p) {
    return __half22float2(__ldg(reinterpret_cast<const __half2*>(p)));
}
__device__ __forceinline__ float2 ld_pair(const double*) { return {}; }  // FP64 levels have face arrays

__device__ __forceinline__ float box_rcp(float v) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
}
__device__ __forceinline__ double box_rcp(double v) { return v; }

// index i of an axis of n, wrapped around if it is periodic; -1: beyond a wall
__device__ __forceinline__ int box_wrap(int i, int n, int wall) {
    if (wall) return i >= 0 && i < n ? i : -1;
    i = i < 0 ? i + n : i >= n ? i - n : i;
    if ((unsigned)i >= (unsigned)n) {  // an axis shorter than the halo
        i %= n;
        if (i < 0) i += n;
    }
    return i;
}

// A pair's cells (local index c and c + 1) while it is smoothed; by colour
// (0: (i+j+k) even) where an array has two.
template <typename T>
struct BoxPair {
    T bx[3], by[2][2], bz[2][2], w[2], f[2];  // bx: left of the pair, between, right of it
    int c;
    int d[2];    // steps to the box
    bool black;  // the left cell is black
};

// Colour pass M over the cells at most D steps from the box (RHO: the pass of
// tile_update, which takes a cell's x-face outside its pair first).
template <typename T, typename B, int M, int D, bool RHO>
__device__ __forceinline__ void box_pass(const BoxPair<T>& o, T* x, T hs, bool scaled, T omega) {
    if (o.d[M] <= D) {
        const bool right = o.black == (M == 0);
        const int c = o.c + (right ? 1 : 0);
        T acc = scaled ? o.f[M] * hs : o.f[M];
        if (RHO) {
            acc = fma(right ? o.bx[2] : o.bx[0], x[right ? c + 1 : c - 1], acc);
            acc = fma(o.bx[1], x[right ? c - 1 : c + 1], acc);
        } else {
            acc = fma(right ? o.bx[1] : o.bx[0], x[c - 1], acc);
            acc = fma(right ? o.bx[2] : o.bx[1], x[c + 1], acc);
        }
        acc = fma(o.by[M][0], x[c - B::bx], acc);
        acc = fma(o.by[M][1], x[c + B::bx], acc);
        acc = fma(o.bz[M][0], x[c - B::bx * B::by], acc);
        acc = fma(o.bz[M][1], x[c + B::bx * B::by], acc);
        const T xc = x[c];
        x[c] = fma(omega, fma(o.w[M], acc, -xc), xc);
    }
    __syncthreads();
}

// UP: prolongation and post-smoothing; else pre-smoothing and restriction.
// RHO: the finest level of the mixed step, coefficients 1/(rh_L + rh_R) from
// rho/2 and vectors in the colour-split layout, with the arithmetic of
// tile_update and op_rho_tile_kernel.
template <typename T, typename TB, int TX, int TY, int TZ, bool UP, bool RHO>
__global__ void __launch_bounds__(Box<TX, TY, TZ>::threads, Box<TX, TY, TZ>::threads <= 512 ? 2 : 1)
    box_kernel(const __grid_constant__ BoxArgs<T, TB> a) {
    using B = Box<TX, TY, TZ>;
    constexpr bool kScaled = RHO || sizeof(TB) == 2;
    __shared__ T x[B::cells];
    __shared__ T term[UP ? 1 : TX * TY * TZ];
    const int tid = threadIdx.x;
    const bool own = tid < B::pairs;
    pdl_trigger();
    const unsigned e = own ? kBoxTable<TX, TY, TZ>.v[tid] : 0u;
    const Geo g = a.g, cg = a.cg;
    const int I0 = blockIdx.x * a.tc[0], J0 = blockIdx.y * a.tc[1], K0 = blockIdx.z * a.tc[2];
    const int i0 = I0 * a.fac[0], j0 = J0 * a.fac[1], k0 = K0 * a.fac[2];
    const int l = 2 * (e & 31u), m = (e >> 5) & 31u, n = e >> 10;
    const int syz = axis_steps(m, TY) + axis_steps(n, TZ);
    // the core's extent (its last coarse cell of an odd axis has three children)
    const int I1 = min(I0 + a.tc[0], cg.nx), J1 = min(J0 + a.tc[1], cg.ny), K1 = min(K0 + a.tc[2], cg.nz);
    const int xe = (I1 == cg.nx ? g.nx : I1 * a.fac[0]) - i0, ye = (J1 == cg.ny ? g.ny : J1 * a.fac[1]) - j0;
    const int ze = (K1 == cg.nz ? g.nz : K1 * a.fac[2]) - k0;
    BoxPair<T> o;
    o.c = (n * B::by + m) * B::bx + l;
    o.black = ((m + n) & 1) != 0;  // the box starts on an even cell of each axis
    const int sl = axis_steps(l, TX) + syz, sr = axis_steps(l + 1, TX) + syz;
    o.d[0] = own ? (o.black ? sr : sl) : 99;
    o.d[1] = own ? (o.black ? sl : sr) : 99;
    // global indices (-1: none) of the pair's cells and of the faces around them
    const int i = box_wrap(i0 - kHalo + l, g.nx, g.wx), j = box_wrap(j0 - kHalo + m, g.ny, g.wy);
    const int k = box_wrap(k0 - kHalo + n, g.nz, g.wz);
    const bool inl = own && i >= 0 && j >= 0 && k >= 0, inr = inl && i + 1 < g.nx;
    const int row = k * g.ny + j, c = row * g.nx + i;
    T bl = T(0), bm = T(0), br = T(0);
    T byl[2] = {T(0), T(0)}, byr[2] = {T(0), T(0)}, bzl[2] = {T(0), T(0)}, bzr[2] = {T(0), T(0)};
    T fl = T(0), fr = T(0), wl = T(0), wr = T(0), xl = T(0), xr = T(0);
    if constexpr (RHO) {
        if (inl) {  // even axes: the pair is whole
            const TB* p = a.b[0] + c;
            const int jm = j > 0 ? -g.nx : (g.ny - 1) * g.nx, jp = j + 1 < g.ny ? g.nx : -(g.ny - 1) * g.nx;
            const int pl = g.nx * g.ny;
            const int km = k > 0 ? -pl : (g.nz - 1) * pl, kp = k + 1 < g.nz ? pl : -(g.nz - 1) * pl;
            const float2 r = ld_pair(p), rym = ld_pair(p + jm), ryp = ld_pair(p + jp), rzm = ld_pair(p + km);
            const float2 rzp = ld_pair(p + kp);
            const float rl = (float)ldc(p + (i > 0 ? -1 : g.nx - 1)), rr = (float)ldc(p + (i + 2 < g.nx ? 2 : 2 - g.nx));
            const bool y0 = g.wy && j == 0, y1 = g.wy && j == g.ny - 1, z0 = g.wz && k == 0, z1 = g.wz && k == g.nz - 1;
            bl = g.wx && i == 0 ? T(0) : (T)box_rcp(r.x + rl);
            bm = (T)box_rcp(r.x + r.y);
            br = g.wx && i + 2 == g.nx ? T(0) : (T)box_rcp(r.y + rr);
            byl[0] = y0 ? T(0) : (T)box_rcp(r.x + rym.x);
            byr[0] = y0 ? T(0) : (T)box_rcp(r.y + rym.y);
            byl[1] = y1 ? T(0) : (T)box_rcp(r.x + ryp.x);
            byr[1] = y1 ? T(0) : (T)box_rcp(r.y + ryp.y);
            bzl[0] = z0 ? T(0) : (T)box_rcp(r.x + rzm.x);
            bzr[0] = z0 ? T(0) : (T)box_rcp(r.y + rzm.y);
            bzl[1] = z1 ? T(0) : (T)box_rcp(r.x + rzp.x);
            bzr[1] = z1 ? T(0) : (T)box_rcp(r.y + rzp.y);
            wl = box_rcp(((bl + bm) + (byl[0] + byl[1])) + (bzl[0] + bzl[1]));
            wr = box_rcp(((br + bm) + (byr[0] + byr[1])) + (bzr[0] + bzr[1]));
        }
    } else if (inl) {
        const TB* p = a.b[0] + row * (g.nx + g.wx) + i;
        if (!(g.wx && i == 0)) bl = (T)ldc(p);
        if (inr) bm = (T)ldc(p + 1);
        else if (!g.wx) bm = (T)ldc(p + 1 - g.nx);  // not reached: a periodic axis is even
        if (inr && i + 2 < g.nx) br = (T)ldc(p + 2);
        else if (inr && !g.wx) br = (T)ldc(p + 2 - g.nx);
        const TB* q = a.b[1] + (k * (g.ny + g.wy) + j) * g.nx + i;
        const int qp = j + 1 < g.ny ? g.nx : -(g.ny - 1) * g.nx;
        const bool q0 = !(g.wy && j == 0), q1 = !(g.wy && j == g.ny - 1);
        const TB* r = a.b[2] + c;
        const int rp = k + 1 < g.nz ? g.nx * g.ny : -(g.nz - 1) * g.nx * g.ny;
        const bool r0 = !(g.wz && k == 0), r1 = !(g.wz && k == g.nz - 1);
        if (q0) byl[0] = (T)ldc(q);
        if (q1) byl[1] = (T)ldc(q + qp);
        if (r0) bzl[0] = (T)ldc(r);
        if (r1) bzl[1] = (T)ldc(r + rp);
        if (a.w) wl = a.w[c];
        if (inr) {
            if (q0) byr[0] = (T)ldc(q + 1);
            if (q1) byr[1] = (T)ldc(q + qp + 1);
            if (r0) bzr[0] = (T)ldc(r + 1);
            if (r1) bzr[1] = (T)ldc(r + rp + 1);
            if (a.w) wr = a.w[c + 1];
        }
    }
    // what the preceding launches of the V-cycle wrote
    pdl_wait();
    // the pair's entries in the vectors: side by side, or one in each half of a split row
    const int hx = g.nx / 2, cl = RHO ? row * g.nx + i / 2 + (o.black ? hx : 0) : c;
    const int cr = RHO ? row * g.nx + i / 2 + (o.black ? 0 : hx) : c + 1;
    if (inl) {
        fl = a.f[cl];
        if (UP) xl = a.xin[cl];
        if (inr) {
            fr = a.f[cr];
            if (UP) xr = a.xin[cr];
        }
        if (UP) {
            const int pr = (parent_of(k, cg.nz, a.fac[2]) * cg.ny + parent_of(j, cg.ny, a.fac[1])) * cg.nx;
            xl += a.xc[pr + parent_of(i, cg.nx, a.fac[0])];
            if (inr) xr += a.xc[pr + parent_of(i + 1, cg.nx, a.fac[0])];
        }
    }
    // down: the coarse faces of the core's cells, and the sum that a thread forms
    unsigned ml = 0, mr = 0;
    const bool core = syz == 0 && own && l >= kHalo && l < kHalo + xe && m < kHalo + ye && n < kHalo + ze;
    int tp = 0, tn0 = 0, tn1 = 0, tn2 = 0, tc = -1;
    T inv = T(1);
    if (!UP) {
        if (core) {
            const int J = parent_of(j, cg.ny, a.fac[1]), K = parent_of(k, cg.nz, a.fac[2]);
            const int nj = child_count(J, cg.ny, g.ny, a.fac[1]), nk = child_count(K, cg.nz, g.nz, a.fac[2]);
            const int Il = parent_of(i, cg.nx, a.fac[0]), Ir = parent_of(i + 1, cg.nx, a.fac[0]);
            ml = surface_faces(i - a.fac[0] * Il, j - a.fac[1] * J, k - a.fac[2] * K, child_count(Il, cg.nx, g.nx, a.fac[0]),
                               nj, nk);
            mr = surface_faces(i + 1 - a.fac[0] * Ir, j - a.fac[1] * J, k - a.fac[2] * K,
                               child_count(Ir, cg.nx, g.nx, a.fac[0]), nj, nk);
        }
        const int cw = I1 - I0, ch = J1 - J0;
        if (tid < cw * ch * (K1 - K0)) {
            const int I = I0 + tid % cw, r = tid / cw, J = J0 + r % ch, K = K0 + r / ch;
            tn0 = child_count(I, cg.nx, g.nx, a.fac[0]);
            tn1 = child_count(J, cg.ny, g.ny, a.fac[1]);
            tn2 = child_count(K, cg.nz, g.nz, a.fac[2]);
            tp = ((K * a.fac[2] - k0) * TY + J * a.fac[1] - j0) * TX + I * a.fac[0] - i0;
            tc = (K * cg.ny + J) * cg.nx + I;
            // factors are 1 or 2
            inv = (a.fac[0] == 2 ? T(0.5) : T(1)) * (a.fac[1] == 2 ? T(0.5) : T(1)) * (a.fac[2] == 2 ? T(0.5) : T(1));
        }
    }
    const T hs = a.hs;
    if (!RHO && !a.w) {
        const T s[6] = {bl, bm, byl[0], byl[1], bzl[0], bzl[1]}, t[6] = {bm, br, byr[0], byr[1], bzr[0], bzr[1]};
        wl = inv_sum6(s);
        wr = inv_sum6(t);
    }
    o.bx[0] = bl;
    o.bx[1] = bm;
    o.bx[2] = br;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        o.by[0][h] = o.black ? byr[h] : byl[h];
        o.by[1][h] = o.black ? byl[h] : byr[h];
        o.bz[0][h] = o.black ? bzr[h] : bzl[h];
        o.bz[1][h] = o.black ? bzl[h] : bzr[h];
    }
    o.w[0] = o.black ? wr : wl;
    o.w[1] = o.black ? wl : wr;
    o.f[0] = o.black ? fr : fl;
    o.f[1] = o.black ? fl : fr;
    if (own) {
        if (UP) {
            x[o.c] = xl;
            x[o.c + 1] = xr;
        } else {  // the first pass, from x = 0
            const T v = a.omega * o.w[0] * (kScaled ? o.f[0] * hs : o.f[0]);
            x[o.c] = o.black ? T(0) : v;
            x[o.c + 1] = o.black ? v : T(0);
        }
    }
    __syncthreads();
    box_pass<T, B, 1, 3, RHO>(o, x, hs, kScaled, a.omega);
    if (!UP) {
        if (a.sweeps == 2) {
            box_pass<T, B, 0, 2, RHO>(o, x, hs, kScaled, a.omega);
            box_pass<T, B, 1, 1, RHO>(o, x, hs, kScaled, a.omega);
        }
    } else {
        box_pass<T, B, 0, 2, RHO>(o, x, hs, kScaled, a.omega);
        if (a.sweeps == 2) {
            box_pass<T, B, 1, 1, RHO>(o, x, hs, kScaled, a.omega);
            box_pass<T, B, 0, 0, RHO>(o, x, hs, kScaled, a.omega);
        }
    }
    if (core) {
        a.x[cl] = x[o.c];
        if (inr) a.x[cr] = x[o.c + 1];
        if (!UP) {  // each cell's term of its parent's sum
            auto residual = [&](int M, int cl, T b0, T b1, unsigned mask) {
                const T xc = x[cl];
                T acc = T(0);
                if (mask & 1u) acc = fma(b0, xc - x[cl - 1], acc);
                if (mask & 2u) acc = fma(b1, xc - x[cl + 1], acc);
                if (mask & 4u) acc = fma(M ? o.by[1][0] : o.by[0][0], xc - x[cl - B::bx], acc);
                if (mask & 8u) acc = fma(M ? o.by[1][1] : o.by[0][1], xc - x[cl + B::bx], acc);
                if (mask & 16u) acc = fma(M ? o.bz[1][0] : o.bz[0][0], xc - x[cl - B::bx * B::by], acc);
                if (mask & 32u) acc = fma(M ? o.bz[1][1] : o.bz[0][1], xc - x[cl + B::bx * B::by], acc);
                const T f = M ? o.f[1] : o.f[0];
                if (kScaled) return fma(-a.rs, acc, f);  // never with a diagonal excess
                if (a.sig) acc = fma(a.sig[c + cl - o.c], xc, acc);
                return f - acc;
            };
            const int tt = ((n - kHalo) * TY + m - kHalo) * TX + l - kHalo;
            term[tt] = residual(o.black ? 1 : 0, o.c, o.bx[0], o.bx[1], ml);
            if (inr) term[tt + 1] = residual(o.black ? 0 : 1, o.c + 1, o.bx[1], o.bx[2], mr);
        }
    }
    if (!UP) {
        __syncthreads();
        if (tc >= 0) {
            T sum = T(0);
            if (RHO) {  // rows of both planes, then the two rows
                const T* p = term + tp;
                sum = ((p[0] + p[1]) + (p[TY * TX] + p[TY * TX + 1])) +
                      ((p[TX] + p[TX + 1]) + (p[TY * TX + TX] + p[TY * TX + TX + 1]));
            } else {
                for (int dk = 0; dk < tn2; ++dk)
                    for (int dj = 0; dj < tn1; ++dj)
                        for (int di = 0; di < tn0; ++di) sum += term[tp + (dk * TY + dj) * TX + di];
            }
            a.fc[tc] = sum * inv;
        }
    }
}

template <typename T, typename TB, int TX, int TY, int TZ, bool RHO = false>
void launch_box(BoxArgs<T, TB>& a, bool up, cudaStream_t st) {
    const int n[3] = {a.g.nx, a.g.ny, a.g.nz}, cn[3] = {a.cg.nx, a.cg.ny, a.cg.nz}, tt[3] = {TX, TY, TZ};
    int nb[3];
    for (int q = 0; q < 3; ++q) {
        // the last coarse cell of an odd axis has three children: a box of one coarse cell less holds it
        a.tc[q] = a.fac[q] == 1 ? tt[q] : (n[q] % 2 ? tt[q] / 2 - 1 : tt[q] / 2);
        nb[q] = (cn[q] + a.tc[q] - 1) / a.tc[q];
    }
    using B = Box<TX, TY, TZ>;
    launch_pdl(up ? box_kernel<T, TB, TX, TY, TZ, true, RHO> : box_kernel<T, TB, TX, TY, TZ, false, RHO>,
               dim3(nb[0], nb[1], nb[2]), B::threads, 0, st, a);
    count_launch();
}

// Up to here a level goes by boxes, and up to here by the small ones.  FP32: with
// 64^3 cells by boxes too, a step at 128^3 is 12 % slower (the halo's work no longer
// hides in latency); 32^3 by small boxes 3 % slower, 16^3 by large ones 2 %.
// FP64 runs at two lanes a clock: 32^3 cells by boxes of 4^3 take 2 % more of a
// 128^3 step than by passes.
constexpr int64_t kBoxCells = 32768, kBoxCells64 = 8192, kSmallBoxCells = 8192;

}  // namespace

bool box_level_fits(const Geo& g, int nu1, int nu2, bool fp64) {
    if (nu1 < 1 || nu1 > 2 || nu2 < 1 || nu2 > 2 || g.ncell() > (fp64 ? kBoxCells64 : kBoxCells)) return false;
    const int n[3] = {g.nx, g.ny, g.nz}, wall[3] = {g.wx, g.wy, g.wz};
    for (int q = 0; q < 3; ++q)
        if (!wall[q] && n[q] % 2) return false;
    return true;
}

template <typename T, typename TB>
void launch_box_level(const Geo& g, const TB* const b[3], T scale, const T* w, const T* sig, const T* f, const Geo& cg,
                      const int fac[3], bool up, const T* xin, T* x, T* fc, const T* xc, double omega, int sweeps,
                      cudaStream_t st) {
    BoxArgs<T, TB> a{};
    a.g = g;
    a.cg = cg;
    for (int q = 0; q < 3; ++q) {
        a.fac[q] = fac[q];
        a.b[q] = b[q];
    }
    a.w = w;
    a.sig = sig;
    a.f = f;
    a.xin = xin;
    a.x = x;
    a.fc = fc;
    a.xc = xc;
    a.hs = T(1) / scale;
    a.rs = scale;
    a.omega = (T)omega;
    a.sweeps = sweeps;
    if constexpr (sizeof(T) == 4) {
        if (g.ncell() > kSmallBoxCells) {
            launch_box<T, TB, 8, 8, 4>(a, up, st);
            return;
        }
    }
    launch_box<T, TB, 4, 4, 4>(a, up, st);
}

template <typename RT>
void launch_box_rho(const Geo& g, const RT* rh, double h, const float* f, const Geo& cg, bool up, const float* xin, float* x,
                    float* fc, const float* xc, double omega, int sweeps, cudaStream_t st) {
    BoxArgs<float, RT> a{};
    a.g = g;
    a.cg = cg;
    for (int q = 0; q < 3; ++q) a.fac[q] = 2;
    a.b[0] = rh;
    a.f = f;
    a.xin = xin;
    a.x = x;
    a.fc = fc;
    a.xc = xc;
    a.hs = (float)(h * h);
    a.rs = (float)(1.0 / (h * h));
    a.omega = (float)omega;
    a.sweeps = sweeps;
    // 32^3: 707 us a step by large boxes, 765 by small ones, 798 by passes
    if (g.ncell() > kSmallBoxCells) launch_box<float, RT, 8, 8, 4, true>(a, up, st);
    else launch_box<float, RT, 4, 4, 4, true>(a, up, st);
}
template void launch_box_rho<float>(const Geo&, const float*, double, const float*, const Geo&, bool, const float*, float*,
                                    float*, const float*, double, int, cudaStream_t);
template void launch_box_rho<__half>(const Geo&, const __half*, double, const float*, const Geo&, bool, const float*, float*,
                                     float*, const float*, double, int, cudaStream_t);

template void launch_box_level<float, float>(const Geo&, const float* const[3], float, const float*, const float*,
                                             const float*, const Geo&, const int[3], bool, const float*, float*, float*,
                                             const float*, double, int, cudaStream_t);
template void launch_box_level<float, __half>(const Geo&, const __half* const[3], float, const float*, const float*,
                                              const float*, const Geo&, const int[3], bool, const float*, float*, float*,
                                              const float*, double, int, cudaStream_t);
template void launch_box_level<double, double>(const Geo&, const double* const[3], double, const double*, const double*,
                                               const double*, const Geo&, const int[3], bool, const double*, double*,
                                               double*, const double*, double, int, cudaStream_t);

}  // namespace paris
