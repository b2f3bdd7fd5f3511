// Tail of the V-cycle in one launch.
//
// The coarsest levels are too small to fill even one SM: a colour pass on 8^3
// cells costs the launch and memory latency of one on 32^3.  From the first
// level with at most 512 cells down to the dense coarsest solve and back up, this kernel
// runs every step of the V-cycle (Sec. 3.7.3: pre-smoothing, restriction of
// the residual, the coarsest solve, prolongation, post-smoothing) in one
// block, with a block barrier between steps.  Each cell
// update, restriction sum, prolongation and the dense solve use the same
// arithmetic in the same order as the separate kernels, so the result is the
// same bit for bit.
#include "kernels.cuh"

namespace paris {

namespace {

constexpr int kTailThreads = 512;

// One element from global to shared memory without a register round trip
// (cp.async; completed by cp.async.wait_all).  Both addresses are aligned to
// the element size.
__device__ __forceinline__ void async_copy(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void async_copy(double* dst, const double* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// t / n by the multiplier m of TailLevel (exact for t, n < 2^16)
__device__ __forceinline__ unsigned udiv(unsigned t, unsigned n, unsigned m) { return n == 1 ? t : __umulhi(t, m); }

// (i, j, k) of index t on an n0 x n1 x n2 box, x fastest (m0, m1: the multipliers of n0, n1)
__device__ __forceinline__ void tail_split(unsigned t, unsigned n0, unsigned n1, unsigned m0, unsigned m1, int& i,
                                           int& j, int& k) {
    const unsigned row = udiv(t, n0, m0);
    i = (int)(t - row * n0);
    const unsigned kk = udiv(row, n1, m1);
    j = (int)(row - kk * n1);
    k = (int)kk;
}

// One colour pass of over-relaxed red-black Gauss-Seidel on a tail level (the
// update of rbgs_kernel; zero: x taken as 0, the other colour zeroed).  tmp: a
// value per cell, for the new values until all are formed (odd_seam).
template <typename T>
__device__ void tail_pass(const TailLevel<T>& L, int color, bool zero, T omega, T* tmp) {
    const Geo g = L.g;
    const bool seam = !zero && odd_seam(g);
    const int npair = (g.nx + 1) / 2;
    const int total = npair * g.ny * g.nz;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int tp, j, k;
        tail_split((unsigned)t, (unsigned)npair, (unsigned)g.ny, L.mp, L.my, tp, j, k);
        const int i0 = 2 * tp;
        const int i = i0 + ((i0 + j + k + color) & 1);
        const int io = i0 + 1 - (i - i0);
        if (i < g.nx) {
            Stencil<T> s;
            int c;
            load_stencil_fast<T>(g, L.bx, L.by, L.bz, i, j, k, s, c);
            if (zero) {
                L.x[c] = omega * L.w[c] * L.f[c];
            } else {
                T acc = L.f[c];
#pragma unroll
                for (int q = 0; q < 6; ++q) acc = fma(s.b[q], L.x[s.nb[q]], acc);
                const T xc = L.x[c];
                (seam ? tmp : L.x)[c] = fma(omega, fma(L.w[c], acc, -xc), xc);
            }
        }
        if (zero && io < g.nx) L.x[g.cidx(io, j, k)] = T(0);
    }
    if (!seam) return;
    __syncthreads();
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int tp, j, k;
        tail_split((unsigned)t, (unsigned)npair, (unsigned)g.ny, L.mp, L.my, tp, j, k);
        const int i = 2 * tp + ((j + k + color) & 1);
        if (i < g.nx) L.x[g.cidx(i, j, k)] = tmp[g.cidx(i, j, k)];
    }
}

template <typename T>
__device__ void tail_smooth(const TailLevel<T>& L, int sweeps, bool first_zero, bool reverse, T omega, T* tmp) {
    for (int s = 0; s < sweeps; ++s) {
        tail_pass<T>(L, reverse ? 1 : 0, first_zero && s == 0, omega, tmp);
        __syncthreads();
        tail_pass<T>(L, reverse ? 0 : 1, false, omega, tmp);
        __syncthreads();
    }
}

// coarse f = average over the children of the fine residual f - A x (A x on
// the coarse cell's surface faces, as restrict_residual_kernel): every fine
// cell's term first, by all threads, then the sums in the children's order.
template <typename T>
__device__ void tail_restrict(const TailLevel<T>& F, const TailLevel<T>& C, T* term) {
    const Geo fg = F.g;
    const Geo cg = C.g;
    const int fa0 = C.fac[0], fa1 = C.fac[1], fa2 = C.fac[2];
    const int fine = fg.nx * fg.ny * fg.nz, total = cg.nx * cg.ny * cg.nz;
    for (int t = threadIdx.x; t < fine; t += blockDim.x) {
        int i, j, k, c;
        tail_split((unsigned)t, (unsigned)fg.nx, (unsigned)fg.ny, F.mx, F.my, i, j, k);
        const int I = parent_of(i, cg.nx, fa0), J = parent_of(j, cg.ny, fa1), K = parent_of(k, cg.nz, fa2);
        const unsigned mask =
            surface_faces(i - fa0 * I, j - fa1 * J, k - fa2 * K, child_count(I, cg.nx, fg.nx, fa0),
                          child_count(J, cg.ny, fg.ny, fa1), child_count(K, cg.nz, fg.nz, fa2));
        Stencil<T> s;
        load_stencil_fast<T>(fg, F.bx, F.by, F.bz, i, j, k, s, c);
        T ax = apply_A_faces(s, F.x, F.x[c], F.scale, mask);
        if (F.sig) ax = fma(F.scale * F.sig[c], F.x[c], ax);
        term[t] = F.f[c] - ax;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int I, J, K;
        tail_split((unsigned)t, (unsigned)cg.nx, (unsigned)cg.ny, C.mx, C.my, I, J, K);
        const int n0 = child_count(I, cg.nx, fg.nx, fa0), n1 = child_count(J, cg.ny, fg.ny, fa1);
        const int n2 = child_count(K, cg.nz, fg.nz, fa2);
        T sum = T(0);
        for (int dk = 0; dk < n2; ++dk)
            for (int dj = 0; dj < n1; ++dj)
                for (int di = 0; di < n0; ++di)
                    sum += term[((K * fa2 + dk) * fg.ny + J * fa1 + dj) * fg.nx + I * fa0 + di];
        C.f[t] = sum / T(fa0 * fa1 * fa2);
    }
}

// x_fine += x_coarse[parent]
template <typename T>
__device__ void tail_prolong(const TailLevel<T>& C, const TailLevel<T>& F) {
    const Geo fg = F.g;
    const Geo cg = C.g;
    const int total = fg.nx * fg.ny * fg.nz;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int i, j, k;
        tail_split((unsigned)t, (unsigned)fg.nx, (unsigned)fg.ny, F.mx, F.my, i, j, k);
        F.x[t] += C.x[cg.cidx(parent_of(i, cg.nx, C.fac[0]), parent_of(j, cg.ny, C.fac[1]),
                              parent_of(k, cg.nz, C.fac[2]))];
    }
}

// x = M (f - mean f) on the coarsest level (FP64 arithmetic)
template <typename T>
__device__ void tail_coarse_solve(const TailLevel<T> L, const double* __restrict__ M, double* fs,
                                  double* mean, int keep_mean) {
    const int n = L.g.nx * L.g.ny * L.g.nz;
    for (int c = threadIdx.x; c < n; c += blockDim.x) fs[c] = (double)L.f[c];
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int c = 0; c < n; ++c) t += fs[c];
        *mean = keep_mean ? 0.0 : t / (double)n;
    }
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        double acc = 0.0;
        for (int c = 0; c < n; ++c) acc = fma(M[r * n + c], fs[c] - *mean, acc);
        L.x[r] = (T)acc;
    }
}

// The levels of a tail in one block's shared memory: the table (pointing at
// staged copies or at the caller's arrays), the dense inverse and scratch.
template <typename T>
struct TailShared {
    double fs[kMaxDenseCells];
    double mean;
    TailLevel<T> L[kMaxTail];
    const double* M;
    T* term;  // one value per cell of the first level
};

// The table over n levels with every array in shared memory from base on, and
// (copy) the coefficients, inverse diagonals and the dense inverse staged there;
// with_f: the first level's right-hand side too.  Ends in a block barrier.
template <typename T>
__device__ void tail_stage(TailShared<T>& ts, const TailLevel<T>* levels, int n, const double* Minv, void* base, bool copy,
                           bool with_f) {
    if (threadIdx.x == 0) {
        unsigned char* dyn = (unsigned char*)base;
        auto carve = [&](size_t bytes) {
            void* p = dyn;
            dyn += (bytes + 15) & ~(size_t)15;
            return p;
        };
        for (int l = 0; l < n; ++l) {
            TailLevel<T>& L = ts.L[l];
            L = levels[l];
            const int64_t cells = L.g.ncell();
            L.bx = (const T*)carve(sizeof(T) * L.g.nface(0));
            L.by = (const T*)carve(sizeof(T) * L.g.nface(1));
            L.bz = (const T*)carve(sizeof(T) * L.g.nface(2));
            L.w = (const T*)carve(sizeof(T) * cells);
            if (L.sig) L.sig = (const T*)carve(sizeof(T) * cells);
            L.f = (T*)carve(sizeof(T) * cells);
            L.x = (T*)carve(sizeof(T) * cells);
        }
        const int64_t nc = ts.L[n - 1].g.ncell();
        ts.M = (const double*)carve(sizeof(double) * nc * nc);
        ts.term = (T*)carve(sizeof(T) * ts.L[0].g.ncell());
    }
    __syncthreads();
    if (!copy) return;
    // every thread issues its share of the copies as asynchronous global ->
    // shared copies and waits once, so the staging costs about one memory
    // latency instead of one per element a thread moves
    auto put = [&](const T* src, const T* dst, int64_t cnt) {
        for (int64_t e = threadIdx.x; e < cnt; e += blockDim.x) async_copy(const_cast<T*>(dst) + e, src + e);
    };
    for (int l = 0; l < n; ++l) {
        const TailLevel<T>& G = levels[l];
        const TailLevel<T>& L = ts.L[l];
        put(G.bx, L.bx, G.g.nface(0));
        put(G.by, L.by, G.g.nface(1));
        put(G.bz, L.bz, G.g.nface(2));
        put(G.w, L.w, G.g.ncell());
        if (G.sig) put(G.sig, L.sig, G.g.ncell());
    }
    if (with_f) put(levels[0].f, ts.L[0].f, levels[0].g.ncell());  // the other levels' f are restricted here
    const int64_t nc = levels[n - 1].g.ncell();
    for (int64_t e = threadIdx.x; e < nc * nc; e += blockDim.x) async_copy(const_cast<double*>(ts.M) + e, Minv + e);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// The V-cycle over the table's levels, from the first one's f to its x.
template <typename T>
__device__ void tail_levels(TailShared<T>& ts, int n, int nu1, int nu2, T omega, int keep_mean) {
    for (int l = 0; l < n - 1; ++l) {
        const TailLevel<T> L = ts.L[l];  // in registers: the loops below store through its pointers
        if (nu1 > 0) {
            tail_smooth<T>(L, nu1, true, false, omega, ts.term);
        } else {
            const int cells = L.g.nx * L.g.ny * L.g.nz;
            for (int c = threadIdx.x; c < cells; c += blockDim.x) L.x[c] = T(0);
            __syncthreads();
        }
        tail_restrict<T>(L, ts.L[l + 1], ts.term);
        __syncthreads();
    }
    tail_coarse_solve<T>(ts.L[n - 1], ts.M, ts.fs, &ts.mean, keep_mean);
    __syncthreads();
    for (int l = n - 2; l >= 0; --l) {
        tail_prolong<T>(ts.L[l + 1], ts.L[l]);
        __syncthreads();
        const TailLevel<T> L = ts.L[l];
        if (nu2 > 0) tail_smooth<T>(L, nu2, false, true, omega, ts.term);
    }
}

// shared-memory bytes of the staged tail (16-byte aligned arrays)
template <typename T>
size_t tail_smem_bytes(const TailLevel<T>* levels, int n) {
    auto al = [](size_t b) { return (b + 15) & ~(size_t)15; };
    size_t b = 0;
    for (int l = 0; l < n; ++l) {
        const Geo& g = levels[l].g;
        b += al(sizeof(T) * g.nface(0)) + al(sizeof(T) * g.nface(1)) + al(sizeof(T) * g.nface(2));
        b += (3 + (levels[l].sig ? 1 : 0)) * al(sizeof(T) * g.ncell());
    }
    const int64_t nc = levels[n - 1].g.ncell();
    return b + al(sizeof(double) * nc * nc) + al(sizeof(T) * levels[0].g.ncell());
}


template <typename T>
struct TailArgs {
    int n;                    // levels in the tail, the last one the dense coarsest
    TailLevel<T> L[kMaxTail];
    const double* Minv;       // dense inverse of the coarsest operator
    T omega;
    T* term;                  // scratch of one value per cell of the first level (when not in shared memory)
    int nu1, nu2;
    int keep_mean;            // no null space: the coarsest right-hand side keeps its mean
};

// SMEM: the levels' coefficients, inverse diagonals, right-hand sides and
// solutions and the dense inverse are staged in shared memory; only the first
// level's solution is written back (its right-hand side came from above).
// The level table itself lives in shared memory, pointing at either copy.
template <typename T, bool SMEM>
__global__ void __launch_bounds__(kTailThreads, 1) tail_vcycle_kernel(const __grid_constant__ TailArgs<T> a) {
    pdl_wait();
    __shared__ TailShared<T> ts;
    extern __shared__ __align__(16) unsigned char dyn[];
    if (SMEM) {
        tail_stage<T>(ts, a.L, a.n, a.Minv, dyn, true, true);
    } else {
        if (threadIdx.x == 0) {
            for (int l = 0; l < a.n; ++l) ts.L[l] = a.L[l];
            ts.M = a.Minv;
            ts.term = a.term;
        }
        __syncthreads();
    }
    tail_levels<T>(ts, a.n, a.nu1, a.nu2, a.omega, a.keep_mean);
    if (SMEM) {
        const int64_t cells = a.L[0].g.ncell();
        for (int64_t e = threadIdx.x; e < cells; e += blockDim.x) a.L[0].x[e] = ts.L[0].x[e];
    }
}

// ------------------------------------------------------ the usual small tail

// A tail of one or two smoothed levels of at most 256 pairs of cells each above
// the dense coarsest (8^3, 4^3 and 2^3 cells, say), by one block of 256 threads.
// What bounds the general kernel on such levels is the length of its dependent
// instruction chains: index arithmetic, table look-ups and fifteen reads an
// update, 16 passes long.  Here a thread owns one pair (2p, 2p+1) of a row on
// each level and keeps its coefficients, inverse diagonals, right-hand sides,
// neighbour and parent positions in registers from the first pass down to the
// last one up; only x, the restriction's terms and the coarse right-hand sides
// are in shared memory, and all coefficients arrive in one memory latency.  The
// same arithmetic in the same order.  From 8^3 cells: FP32 17 -> 8.3 us
// a launch, FP64 26 -> 18.9.
constexpr int kSmallThreads = 256;
constexpr int kStagedDense = 32;  // a dense inverse of at most 32^2 values is staged in shared memory

template <typename T>
struct Pair {
    T bx[3], by[2][2], bz[2][2], w[2], f[2], sig[2];  // bx: left of the pair, between, right of it; else by colour (0 red)
    short oym, oyp, ozm, ozp;                         // offsets of the neighbour rows and planes
    short xl, xr;                                     // positions left and right of the pair
    short c;                                          // position of the left cell, -1: no pair
    short par[2];                                     // position of the coarse cell, by colour
    unsigned char mask[2];                            // surface faces of its coarse cell, by colour
    bool black, two;                                  // the left cell is black; there is a right cell
};

template <typename T>
__device__ __forceinline__ void pair_load(Pair<T>& o, const TailLevel<T>& L, const TailLevel<T>& C) {
    const Geo g = L.g, cg = C.g;
    const unsigned npair = (unsigned)(g.nx + 1) / 2, t = threadIdx.x;
    o.c = -1;
    o.black = o.two = false;
    if (t >= npair * (unsigned)(g.ny * g.nz)) return;
    int tp, j, k;
    tail_split(t, npair, (unsigned)g.ny, L.mp, L.my, tp, j, k);
    o.two = 2 * tp + 1 < g.nx;
    o.black = ((j + k) & 1) != 0;  // 2 tp is even
    const int J = parent_of(j, cg.ny, C.fac[1]), K = parent_of(k, cg.nz, C.fac[2]);
    const int nj = child_count(J, cg.ny, g.ny, C.fac[1]), nk = child_count(K, cg.nz, g.nz, C.fac[2]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // left, right
        if (h == 1 && !o.two) continue;
        const int i = 2 * tp + h;
        Stencil<T> s;
        int c;
        load_stencil_fast<T>(g, L.bx, L.by, L.bz, i, j, k, s, c);
        if (h == 0) {
            o.c = (short)c;
            o.bx[0] = s.b[0];
            o.bx[1] = s.b[1];
            o.xl = (short)s.nb[0];
            o.xr = (short)s.nb[1];
            o.oym = (short)(s.nb[2] - c);
            o.oyp = (short)(s.nb[3] - c);
            o.ozm = (short)(s.nb[4] - c);
            o.ozp = (short)(s.nb[5] - c);
        } else {
            o.bx[2] = s.b[1];
            o.xr = (short)s.nb[1];
        }
        const int I = parent_of(i, cg.nx, C.fac[0]);
        const unsigned mask = surface_faces(i - C.fac[0] * I, j - C.fac[1] * J, k - C.fac[2] * K,
                                            child_count(I, cg.nx, g.nx, C.fac[0]), nj, nk);
        const bool red = (h == 0) != o.black;
#pragma unroll
        for (int m = 0; m < 2; ++m)
            if (red == (m == 0)) {
                o.by[m][0] = s.b[2];
                o.by[m][1] = s.b[3];
                o.bz[m][0] = s.b[4];
                o.bz[m][1] = s.b[5];
                o.w[m] = L.w[c];
                o.f[m] = T(0);
                o.sig[m] = L.sig ? L.sig[c] : T(0);
                o.mask[m] = (unsigned char)mask;
                o.par[m] = (short)((K * cg.ny + J) * cg.nx + I);
            }
    }
}

// the pair's cell of colour M: position (-1: none), neighbours and x-faces
template <int M, typename T>
__device__ __forceinline__ int pair_cell(const Pair<T>& o, int& xl, int& xr, T& bl, T& br) {
    const bool right = o.black == (M == 0);
    xl = right ? o.c : o.xl;
    xr = right || !o.two ? o.xr : o.c + 1;
    bl = right ? o.bx[1] : o.bx[0];
    br = right ? o.bx[2] : o.bx[1];
    return o.c < 0 || (right && !o.two) ? -1 : o.c + (right ? 1 : 0);
}

template <int M, typename T>
__device__ __forceinline__ void pair_pass(const Pair<T>& o, T* x, bool zero, bool seam, T omega) {
    int xl, xr;
    T bl, br;
    const int c = pair_cell<M>(o, xl, xr, bl, br);
    if (zero) {
        if (c >= 0) x[c] = omega * o.w[M] * o.f[M];
        const int io = pair_cell<1 - M>(o, xl, xr, bl, br);
        if (io >= 0) x[io] = T(0);
        return;
    }
    T xn = T(0);
    if (c >= 0) {
        T acc = o.f[M];
        acc = fma(bl, x[xl], acc);
        acc = fma(br, x[xr], acc);
        acc = fma(o.by[M][0], x[c + o.oym], acc);
        acc = fma(o.by[M][1], x[c + o.oyp], acc);
        acc = fma(o.bz[M][0], x[c + o.ozm], acc);
        acc = fma(o.bz[M][1], x[c + o.ozp], acc);
        const T xc = x[c];
        xn = fma(omega, fma(o.w[M], acc, -xc), xc);
    }
    if (seam) __syncthreads();  // odd_seam: after all reads
    if (c >= 0) x[c] = xn;
}

template <typename T>
__device__ __forceinline__ void pair_smooth(const Pair<T>& o, T* x, int sweeps, bool first_zero, bool reverse, bool seam,
                                            T omega) {
    for (int s = 0; s < sweeps; ++s) {
        if (!reverse) {
            pair_pass<0>(o, x, first_zero && s == 0, seam, omega);
            __syncthreads();
        }
        pair_pass<1>(o, x, false, seam, omega);
        __syncthreads();
        if (reverse) {
            pair_pass<0>(o, x, false, seam, omega);
            __syncthreads();
        }
    }
}

// the restriction's term of the pair's cell of colour M (f - A x on the coarse cell's surface faces)
template <int M, typename T>
__device__ __forceinline__ void pair_term(const Pair<T>& o, const T* x, bool sig, T* term) {
    int xl, xr;
    T bl, br;
    const int c = pair_cell<M>(o, xl, xr, bl, br);
    if (c < 0) return;
    const T xc = x[c];
    const unsigned mask = o.mask[M];
    T acc = T(0);
    if (mask & 1u) acc = fma(bl, xc - x[xl], acc);
    if (mask & 2u) acc = fma(br, xc - x[xr], acc);
    if (mask & 4u) acc = fma(o.by[M][0], xc - x[c + o.oym], acc);
    if (mask & 8u) acc = fma(o.by[M][1], xc - x[c + o.oyp], acc);
    if (mask & 16u) acc = fma(o.bz[M][0], xc - x[c + o.ozm], acc);
    if (mask & 32u) acc = fma(o.bz[M][1], xc - x[c + o.ozp], acc);
    if (sig) acc = fma(o.sig[M], xc, acc);
    term[c] = o.f[M] - acc;
}

template <int M, typename T>
__device__ __forceinline__ void pair_prolong(const Pair<T>& o, T* x, const T* xc) {
    int xl, xr;
    T bl, br;
    const int c = pair_cell<M>(o, xl, xr, bl, br);
    if (c >= 0) x[c] += xc[o.par[M]];
}

template <int M, typename T>
__device__ __forceinline__ void pair_rhs(Pair<T>& o, const T* f) {
    int xl, xr;
    T bl, br;
    const int c = pair_cell<M>(o, xl, xr, bl, br);
    if (c >= 0) o.f[M] = f[c];
}

// coarse f from the terms of level L (the sums of tail_restrict)
template <typename T>
__device__ __forceinline__ void small_restrict(const Geo& fg, const TailLevel<T>& C, const T* term, T* fc) {
    const Geo cg = C.g;
    const int fa0 = C.fac[0], fa1 = C.fac[1], fa2 = C.fac[2];
    const T inv = (fa0 == 2 ? T(0.5) : T(1)) * (fa1 == 2 ? T(0.5) : T(1)) * (fa2 == 2 ? T(0.5) : T(1));  // factors are 1 or 2
    for (int t = threadIdx.x; t < cg.nx * cg.ny * cg.nz; t += kSmallThreads) {
        int I, J, K;
        tail_split((unsigned)t, (unsigned)cg.nx, (unsigned)cg.ny, C.mx, C.my, I, J, K);
        const int n0 = child_count(I, cg.nx, fg.nx, fa0), n1 = child_count(J, cg.ny, fg.ny, fa1);
        const int n2 = child_count(K, cg.nz, fg.nz, fa2);
        const T* p = term + ((K * fa2) * fg.ny + J * fa1) * fg.nx + I * fa0;
        T sum = T(0);
        if (n0 == 2 && n1 == 2 && n2 == 2) {
#pragma unroll
            for (int dk = 0; dk < 2; ++dk)
#pragma unroll
                for (int dj = 0; dj < 2; ++dj)
#pragma unroll
                    for (int di = 0; di < 2; ++di) sum += p[(dk * fg.ny + dj) * fg.nx + di];
        } else {
            for (int dk = 0; dk < n2; ++dk)
                for (int dj = 0; dj < n1; ++dj)
                    for (int di = 0; di < n0; ++di) sum += p[(dk * fg.ny + dj) * fg.nx + di];
        }
        fc[t] = sum * inv;
    }
}

// NH: smoothed levels (1 or 2) above the dense one.
template <typename T, int NH>
__global__ void __launch_bounds__(kSmallThreads) tail_small_kernel(const __grid_constant__ TailArgs<T> a) {
    pdl_trigger();
    constexpr int kMax = 2 * kSmallThreads;  // cells of 256 pairs
    __shared__ T x[NH][kMax], term[kMax], f1[kMax], fc[kMaxDenseCells], xc[kMaxDenseCells];
    __shared__ double fs[kMaxDenseCells], mean;
    __shared__ double Ms[kStagedDense * kStagedDense];  // the dense inverse when it is small
    const TailLevel<T>& D = a.L[NH];
    const int nd = D.g.nx * D.g.ny * D.g.nz;
    const bool small = nd <= kStagedDense, pow2 = (nd & (nd - 1)) == 0;
    if (small)
        for (int e = threadIdx.x; e < nd * nd; e += kSmallThreads) async_copy(Ms + e, a.Minv + e);
    Pair<T> o0, o1;
    pair_load(o0, a.L[0], a.L[1]);
    if (NH == 2) pair_load(o1, a.L[1], a.L[2]);
    for (int t = threadIdx.x; t < kMax; t += kSmallThreads)
        for (int l = 0; l < NH; ++l) x[l][t] = T(0);
    const double rn = 1.0 / (double)nd;  // exact when nd is a power of two
    asm volatile("cp.async.wait_all;" ::: "memory");
    pdl_wait();  // the first level's right-hand side: what the preceding launch wrote
    pair_rhs<0>(o0, a.L[0].f);
    pair_rhs<1>(o0, a.L[0].f);
    __syncthreads();
    const bool sig = a.L[0].sig != nullptr;
    const bool seam0 = odd_seam(a.L[0].g), seam1 = NH == 2 && odd_seam(a.L[NH - 1].g);
    pair_smooth(o0, x[0], a.nu1, true, false, seam0, a.omega);
    pair_term<0>(o0, x[0], sig, term);
    pair_term<1>(o0, x[0], sig, term);
    __syncthreads();
    if (NH == 2) {
        small_restrict(a.L[0].g, a.L[1], term, f1);
        __syncthreads();
        pair_rhs<0>(o1, f1);
        pair_rhs<1>(o1, f1);
        pair_smooth(o1, x[NH - 1], a.nu1, true, false, seam1, a.omega);
        pair_term<0>(o1, x[NH - 1], sig, term);
        pair_term<1>(o1, x[NH - 1], sig, term);
        __syncthreads();
    }
    small_restrict(a.L[NH - 1].g, D, term, fc);
    __syncthreads();
    // x = M (f - mean f) (the sums of coarse_solve_kernel)
    for (int c = threadIdx.x; c < nd; c += kSmallThreads) fs[c] = (double)fc[c];
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int c = 0; c < nd; ++c) t += fs[c];
        mean = a.keep_mean ? 0.0 : pow2 ? t * rn : t / (double)nd;
    }
    __syncthreads();
    const double* M = small ? Ms : a.Minv;
    for (int r = threadIdx.x; r < nd; r += kSmallThreads) {
        double acc = 0.0;
        for (int c = 0; c < nd; ++c) acc = fma(M[r * nd + c], fs[c] - mean, acc);
        xc[r] = (T)acc;
    }
    __syncthreads();
    if (NH == 2) {
        pair_prolong<0>(o1, x[NH - 1], xc);
        pair_prolong<1>(o1, x[NH - 1], xc);
        __syncthreads();
        pair_smooth(o1, x[NH - 1], a.nu2, false, true, seam1, a.omega);
    }
    const T* up = NH == 2 ? x[NH - 1] : xc;
    pair_prolong<0>(o0, x[0], up);
    pair_prolong<1>(o0, x[0], up);
    __syncthreads();
    pair_smooth(o0, x[0], a.nu2, false, true, seam0, a.omega);
    const int cells = a.L[0].g.nx * a.L[0].g.ny * a.L[0].g.nz;
    for (int e = threadIdx.x; e < cells; e += kSmallThreads) a.L[0].x[e] = x[0][e];
}

template <typename T>
bool small_tail(const TailLevel<T>* levels, int n) {
    if (n < 2 || n > 3) return false;
    for (int l = 0; l < n - 1; ++l) {
        const Geo& g = levels[l].g;
        if ((int64_t)((g.nx + 1) / 2) * g.ny * g.nz > kSmallThreads) return false;
    }
    return true;
}

}  // namespace

template <typename T>
void launch_tail_vcycle(const TailLevel<T>* levels, int n, const double* Minv, double omega, int nu1,
                        int nu2, T* term, bool keep_mean, cudaStream_t st) {
    TailArgs<T> a{};
    a.n = n;
    for (int l = 0; l < n; ++l) a.L[l] = levels[l];
    a.Minv = Minv;
    a.omega = (T)omega;
    a.term = term;
    a.nu1 = nu1;
    a.nu2 = nu2;
    a.keep_mean = keep_mean ? 1 : 0;
    if (small_tail(levels, n)) {
        launch_pdl(n == 3 ? tail_small_kernel<T, 2> : tail_small_kernel<T, 1>, 1, kSmallThreads, 0, st, a);
        count_launch();
        return;
    }
    // stage in shared memory when it fits
    constexpr size_t kSmemMax = 200 * 1024;
    const size_t smem = tail_smem_bytes(levels, n);
    if (smem <= kSmemMax) {
        static SmemOptIn opted;
        allow_smem(opted, (const void*)tail_vcycle_kernel<T, true>, kSmemMax);  // a failure shows at the launch
        launch_pdl(tail_vcycle_kernel<T, true>, 1, kTailThreads, smem, st, a);
    } else {
        launch_pdl(tail_vcycle_kernel<T, false>, 1, kTailThreads, 0, st, a);
    }
    count_launch();
}

template void launch_tail_vcycle<float>(const TailLevel<float>*, int, const double*, double, int, int, float*, bool,
                                        cudaStream_t);
template void launch_tail_vcycle<double>(const TailLevel<double>*, int, const double*, double, int, int,
                                         double*, bool, cudaStream_t);

}  // namespace paris
