// Shared device-side definitions of the projection library: grid geometry,
// face indexing, the 7-point variable-coefficient stencil and deterministic
// block reductions.  Internal header (not part of the C ABI).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace paris {

constexpr int kRedThreads = 256;  // threads of every reducing kernel's block

// One grid level: cells per axis and wall flags.  Cell (i,j,k) lives at
// (k*ny + j)*nx + i; face arrays extend the face axis by one when that axis
// has walls (entries 0 and n are the wall faces).
struct Geo {
    int nx, ny, nz;
    int wx, wy, wz;

    __host__ __device__ int64_t ncell() const { return (int64_t)nx * ny * nz; }
    __host__ __device__ int64_t nface(int axis) const {
        return (int64_t)(nx + (axis == 0 ? wx : 0)) * (ny + (axis == 1 ? wy : 0)) *
               (nz + (axis == 2 ? wz : 0));
    }
    __host__ __device__ int64_t cidx(int i, int j, int k) const {
        return ((int64_t)k * ny + j) * nx + i;
    }
    __host__ __device__ int64_t fx(int i, int j, int k) const {
        return ((int64_t)k * ny + j) * (nx + wx) + i;
    }
    __host__ __device__ int64_t fy(int i, int j, int k) const {
        return ((int64_t)k * (ny + wy) + j) * nx + i;
    }
    __host__ __device__ int64_t fz(int i, int j, int k) const {
        return ((int64_t)k * ny + j) * nx + i;
    }
};

// Children of coarse cell I of cn along an axis of fn fine cells halved
// (f = 2) or kept (f = 1): f of them, three in the last cell of an odd axis.
__host__ __device__ inline int child_count(int I, int cn, int fn, int f) { return I == cn - 1 ? fn - f * I : f; }

// The coarse cell (of cn) that holds fine cell i along such an axis.
__host__ __device__ inline int parent_of(int i, int cn, int f) {
    const int I = i >> (f - 1);
    return I < cn ? I : cn - 1;
}

// A periodic axis of odd length joins cells of one colour across its seam.  There
// a colour pass takes its own colour's values as they were before it: updated
// in place, a cell would meet the neighbour's old or new value depending on the
// order of the threads, and no order is undone by the reversed one, so the V-cycle
// would be neither reproducible nor symmetric (which conjugate gradients need).
__host__ __device__ inline bool odd_seam(const Geo& g) {
    return (!g.wx && (g.nx & 1)) || (!g.wy && (g.ny & 1)) || (!g.wz && (g.nz & 1));
}

// Coefficient set of one level: face arrays and a uniform scale (1/h^2 for
// arrays holding beta itself, 1 for arrays that are already scaled), and an
// optional per-cell diagonal excess sig in the units of the face arrays: the
// operator is  (A x)_c = scale (sum_f beta_f (x_c - x_nb) + sig_c x_c),  the
// form a Dirichlet condition at a cut face takes (Sec. 3.7.5); null: none.
template <typename T>
struct Coef {
    const T* bx;
    const T* by;
    const T* bz;
    T scale;
    const T* sig = nullptr;
};

// Neighbour indices and + face index along one axis of length n.  Along a
// wall axis the missing neighbour is clamped onto the cell itself; its face
// coefficient is forced to zero (Neumann by coefficient zeroing).
struct AxisNb {
    int m, p, fp;   // minus neighbour, plus neighbour, index of the + face
    bool wm, wp;    // minus / plus face is a wall
};

__host__ __device__ inline AxisNb axis_nb(int i, int n, int wall) {
    AxisNb a;
    a.wm = wall && i == 0;
    a.wp = wall && i == n - 1;
    a.m = i > 0 ? i - 1 : (wall ? 0 : n - 1);
    a.p = i + 1 < n ? i + 1 : (wall ? n - 1 : 0);
    a.fp = (i + 1 < n || wall) ? i + 1 : 0;
    return a;
}

// The six face coefficients (unscaled) around cell (i,j,k) and the neighbour
// cell indices, in the order x-, x+, y-, y+, z-, z+.
template <typename T>
struct Stencil {
    T b[6];
    int64_t nb[6];
};

template <typename T>
__device__ inline void load_stencil(const Geo& g, const Coef<T>& cf, int i, int j, int k,
                                    Stencil<T>& s) {
    AxisNb ax = axis_nb(i, g.nx, g.wx);
    AxisNb ay = axis_nb(j, g.ny, g.wy);
    AxisNb az = axis_nb(k, g.nz, g.wz);
    s.b[0] = ax.wm ? T(0) : cf.bx[g.fx(i, j, k)];
    s.b[1] = ax.wp ? T(0) : cf.bx[g.fx(ax.fp, j, k)];
    s.b[2] = ay.wm ? T(0) : cf.by[g.fy(i, j, k)];
    s.b[3] = ay.wp ? T(0) : cf.by[g.fy(i, ay.fp, k)];
    s.b[4] = az.wm ? T(0) : cf.bz[g.fz(i, j, k)];
    s.b[5] = az.wp ? T(0) : cf.bz[g.fz(i, j, az.fp)];
    s.nb[0] = g.cidx(ax.m, j, k);
    s.nb[1] = g.cidx(ax.p, j, k);
    s.nb[2] = g.cidx(i, ay.m, k);
    s.nb[3] = g.cidx(i, ay.p, k);
    s.nb[4] = g.cidx(i, j, az.m);
    s.nb[5] = g.cidx(i, j, az.p);
}

// Coefficient loads from FP16, FP32 or FP64 storage.
__device__ inline float ldc(const __half* p) { return __half2float(*p); }
__device__ inline float ldc(const float* p) { return *p; }
__device__ inline double ldc(const double* p) { return *p; }

// load_stencil for coefficient arrays stored in another type TB (converted to T)
template <typename T, typename TB>
__device__ inline void load_stencil_as(const Geo& g, const TB* bx, const TB* by, const TB* bz,
                                       int i, int j, int k, Stencil<T>& s) {
    AxisNb ax = axis_nb(i, g.nx, g.wx);
    AxisNb ay = axis_nb(j, g.ny, g.wy);
    AxisNb az = axis_nb(k, g.nz, g.wz);
    s.b[0] = ax.wm ? T(0) : (T)ldc(bx + g.fx(i, j, k));
    s.b[1] = ax.wp ? T(0) : (T)ldc(bx + g.fx(ax.fp, j, k));
    s.b[2] = ay.wm ? T(0) : (T)ldc(by + g.fy(i, j, k));
    s.b[3] = ay.wp ? T(0) : (T)ldc(by + g.fy(i, ay.fp, k));
    s.b[4] = az.wm ? T(0) : (T)ldc(bz + g.fz(i, j, k));
    s.b[5] = az.wp ? T(0) : (T)ldc(bz + g.fz(i, j, az.fp));
    s.nb[0] = g.cidx(ax.m, j, k);
    s.nb[1] = g.cidx(ax.p, j, k);
    s.nb[2] = g.cidx(i, ay.m, k);
    s.nb[3] = g.cidx(i, ay.p, k);
    s.nb[4] = g.cidx(i, j, az.m);
    s.nb[5] = g.cidx(i, j, az.p);
}

// Same result as load_stencil_as with 32-bit index arithmetic (valid while
// every face array of the level holds fewer than 2^31 entries): the cell and
// face offsets of the six neighbours follow from the cell offset by
// additions, with wrap-around or clamping at the domain edges.
template <typename T, typename TB>
__device__ inline void load_stencil_fast(const Geo& g, const TB* bx, const TB* by, const TB* bz,
                                         int i, int j, int k, Stencil<T>& s, int& cell) {
    const int nx = g.nx, ny = g.ny, nz = g.nz, pl = nx * ny;
    const int row = k * ny + j;
    const int c = row * nx + i;
    cell = c;
    const bool xlo = i == 0, xhi = i == nx - 1;
    const int fx = row * (nx + g.wx) + i;
    s.b[0] = (g.wx && xlo) ? T(0) : (T)ldc(bx + fx);
    s.b[1] = (g.wx && xhi) ? T(0) : (T)ldc(bx + ((!xhi || g.wx) ? fx + 1 : fx - (nx - 1)));
    s.nb[0] = !xlo ? c - 1 : (g.wx ? c : c + (nx - 1));
    s.nb[1] = !xhi ? c + 1 : (g.wx ? c : c - (nx - 1));
    const bool ylo = j == 0, yhi = j == ny - 1;
    const int fy = (k * (ny + g.wy) + j) * nx + i;
    s.b[2] = (g.wy && ylo) ? T(0) : (T)ldc(by + fy);
    s.b[3] = (g.wy && yhi) ? T(0) : (T)ldc(by + ((!yhi || g.wy) ? fy + nx : fy - (ny - 1) * nx));
    s.nb[2] = !ylo ? c - nx : (g.wy ? c : c + (ny - 1) * nx);
    s.nb[3] = !yhi ? c + nx : (g.wy ? c : c - (ny - 1) * nx);
    const bool zlo = k == 0, zhi = k == nz - 1;
    s.b[4] = (g.wz && zlo) ? T(0) : (T)ldc(bz + c);
    s.b[5] = (g.wz && zhi) ? T(0) : (T)ldc(bz + ((!zhi || g.wz) ? c + pl : c - (nz - 1) * pl));
    s.nb[4] = !zlo ? c - pl : (g.wz ? c : c + (nz - 1) * pl);
    s.nb[5] = !zhi ? c + pl : (g.wz ? c : c - (nz - 1) * pl);
}

// (A x)_c with A = -L: scale * sum_f beta_f (x_c - x_nb)  (difference form,
// which keeps the FP64 residual accurate when x is smooth).
template <typename T>
__device__ inline T apply_A(const Stencil<T>& s, const T* __restrict__ x, T xc, T scale) {
    T acc = s.b[0] * (xc - x[s.nb[0]]);
#pragma unroll
    for (int q = 1; q < 6; ++q) acc = fma(s.b[q], xc - x[s.nb[q]], acc);
    return scale * acc;
}

// The faces of apply_A selected by mask (bit q: face q), in the same order.
// Summed over the children of a coarse cell, A x keeps only the faces on the
// coarse cell's surface (a face between two children enters once from each
// side with opposite signs): the restrictions take those faces only.
template <typename T>
__device__ inline T apply_A_faces(const Stencil<T>& s, const T* __restrict__ x, T xc, T scale, unsigned mask) {
    T acc = T(0);
#pragma unroll
    for (int q = 0; q < 6; ++q)
        if ((mask >> q) & 1u) acc = fma(s.b[q], xc - x[s.nb[q]], acc);
    return scale * acc;
}

// the faces of child (di, dj, dk) of a coarse cell with factors (f0, f1, f2)
// on the coarse cell's surface: - face of the first child along an axis, +
// face of the last
__device__ inline unsigned surface_faces(int di, int dj, int dk, int f0, int f1, int f2) {
    return (di == 0 ? 1u : 0u) | (di == f0 - 1 ? 2u : 0u) | (dj == 0 ? 4u : 0u) | (dj == f1 - 1 ? 8u : 0u) |
           (dk == 0 ? 16u : 0u) | (dk == f2 - 1 ? 32u : 0u);
}

// 1 / sum of the six face coefficients (the red-black sweeps' inverse diagonal)
__device__ inline float rcp_rn(float d) { return __frcp_rn(d); }  // == 1.0f / d
__device__ inline double rcp_rn(double d) { return 1.0 / d; }

template <typename T>
__device__ inline T inv_sum6(const T (&b)[6]) {
    const T d = ((b[0] + b[1]) + (b[2] + b[3])) + (b[4] + b[5]);
    return d > T(0) ? rcp_rn(d) : T(0);
}

// |v| as an integer key: for non-negative doubles (infinities and NaNs
// included) the order of the bit patterns is the numeric order, so running
// maxima of magnitudes and the non-finite test need no FP64 instruction (the
// FP64 pipe runs at 1/64 of the FP32 rate on this GPU).
__device__ inline unsigned long long abs_key(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
}
__device__ inline unsigned key_nonfinite(unsigned long long k) { return k >= 0x7ff0000000000000ULL ? 1u : 0u; }
__device__ inline double key_value(unsigned long long k) { return __longlong_as_double((long long)k); }

// Conversions between FP64 and FP32 with a power-of-two scaling, written
// with integer operations on the IEEE-754 fields: the hardware conversions
// run on the FP64 pipe at about a fifth of its FMA rate on this GPU.
//
// float(v * 2^s): round to nearest, ties to even, for v * 2^s in the FP32
// normal range; smaller values flush to a signed zero (the last half ulp below
// 2^-126 too), larger ones give a signed infinity; infinities stay infinite and
// NaN stays NaN.
__device__ inline float d2f_scaled(double v, int s) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ffu);
    if (e == 0x7ff) return __int_as_float((int)(sign | 0x7f800000u | (((hi & 0xfffffu) | lo) ? 0x400000u : 0u)));
    const int fe = e - 896 + s;  // FP32 biased exponent (FP64 bias 1023, FP32 bias 127)
    if (e == 0 || fe <= 0) return __int_as_float((int)sign);
    if (fe >= 255) return __int_as_float((int)(sign | 0x7f800000u));
    // the 23 leading fraction bits; round on the 29 dropped ones (a carry out
    // of the fraction correctly increments the exponent)
    const unsigned frac = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned rem = lo & 0x1fffffffu;
    unsigned bits = ((unsigned)fe << 23) | frac;
    if (rem > 0x10000000u || (rem == 0x10000000u && (frac & 1u))) bits += 1u;
    return __int_as_float((int)(sign | bits));
}

// (double)v * 2^s, exact for normal v whose scaled value is an FP64 normal
// number; FP32 subnormals flush to a signed zero; infinities and NaN are kept.
__device__ inline double f2d_scaled(float v, int s) {
    const unsigned b = (unsigned)__float_as_int(v);
    const unsigned sign = b & 0x80000000u;
    const int e = (int)((b >> 23) & 0xffu);
    const unsigned frac = b & 0x7fffffu;
    if (e == 0xff) return __hiloint2double((int)(sign | 0x7ff00000u | (frac ? 0x80000u : 0u)), 0);
    const int de = e + 896 + s;  // FP64 biased exponent
    if (e == 0 || de <= 0) return __hiloint2double((int)sign, 0);
    if (de >= 0x7ff) return __hiloint2double((int)(sign | 0x7ff00000u), 0);
    return __hiloint2double((int)(sign | ((unsigned)de << 20) | (frac >> 3)), (int)(frac << 29));
}

// The same conversions with FP32 subnormals kept, as the hardware's, for values
// that no scaling brings to O(1): coefficients, and corrections without a power
// of two of their own.  A heavy fluid's coefficient may be subnormal beside a
// light fluid's normal one, and flushing it would cut its cells off (a 32^3 solve
// with single heavy cells at 5e-39 ended non-finite).  In integers throughout: a
// hardware conversion for the rare values alone is issued for all (the FP32
// copies at 128^3: 24.9 us flushing, 29.5 so, 25.2 as below).
__device__ __forceinline__ float to_f32(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), e = (hi >> 20) & 0x7ffu;
    if (e - 1u >= 896u) return d2f_scaled(v, 0);
    if (e < 873u) return __int_as_float((int)(hi & 0x80000000u));
    const unsigned long long m = ((unsigned long long)__double_as_longlong(v) & 0xfffffffffffffULL) | 0x10000000000000ULL;
    const int s = 926 - (int)e;  // 30 .. 53 bits below a unit of 2^-149
    unsigned n = (unsigned)(m >> s);
    const unsigned long long rem = m & ((1ULL << s) - 1), half = 1ULL << (s - 1);
    if (rem > half || (rem == half && (n & 1u))) ++n;
    return __int_as_float((int)(hi & 0x80000000u | n));
}
__device__ __forceinline__ double to_f64(float v) {
    const unsigned b = (unsigned)__float_as_int(v), f = b & 0x7fffffffu;
    if (f - 1u >= 0x7fffffu) return f2d_scaled(v, 0);
    const int z = __clz((int)f) - 8;  // leading zeros of the fraction's 24 bits
    const unsigned n = f << z, de = 897u - (unsigned)z;  // 1.xxx * 2^(-126 - z)
    return __hiloint2double((int)((b & 0x80000000u) | (de << 20) | ((n & 0x7fffffu) >> 3)), (int)(n << 29));
}

// 1/s for s > 0 without an FP64 division and without FP64<->FP32
// conversions (both run at the FP64 rate, 1/64 of the FP32 rate on this
// GPU): an FP32 estimate is formed from the leading bits of s by re-biasing
// the exponent in integer arithmetic (20 of the 52 fraction bits kept, so
// the estimate is within 2^-20 of s), inverted with the FP32 approximate
// reciprocal (1 ulp), re-biased back into an FP64 y0 with |1 - s y0| < 2^-19.
// One third-order Newton-Raphson step y0 (1 + e + e^2), e = 1 - s y0,
// leaves a truncation error e^3 < 2^-57 relative, below half an ulp, so the
// result is within one ulp of the correctly rounded 1/s.  Values of s
// outside the exponent window [2^-123, 2^117) (or s <= 0, NaN) take the
// FP64 division.
__device__ __forceinline__ bool recip_window(double s) {
    const int hi = __double2hiint(s);
    return !(hi < (900 << 20) || hi >= (1140 << 20));
}
__device__ __forceinline__ double recip_newton(double s) {  // s in the window
    const int hi = __double2hiint(s);
    const float sf = __int_as_float((hi - (896 << 20)) << 3);
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(sf));
    const unsigned yb = (unsigned)__float_as_int(yf);
    const double y0 = __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
    const double e = fma(-s, y0, 1.0);
    return fma(y0, fma(e, e, e), y0);
}
__device__ inline double recip64(double s) {
    if (!recip_window(s)) return 1.0 / s;
    return recip_newton(s);
}

// 1/s correctly rounded: one more step y + (1 - s y) y from a y within one ulp
// gives that for every s whose fraction is not all ones (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor",
// IBM J. Res. Dev. 34, 1990); those take the division.  Two more FP64
// instructions (the viscous set-up at 256^3: 286 -> 345 us a component).
__device__ inline double recip64_rn(double s) {
    const bool ones = ((unsigned)__double2hiint(s) | 0xfff00000u) == 0xffffffffu && __double2loint(s) == -1;
    if (!recip_window(s) || ones) return 1.0 / s;
    const double y = recip_newton(s);
    return fma(fma(-s, y, 1.0), y, y);
}

// a / b for positive a and b: q = a y with y = 1/b to one ulp and one step with
// the exact remainder, q + (a - b q) y, which is within 1.5 ulp times y's relative
// error of a / b before it is rounded.  So the result is the correctly rounded
// quotient unless a / b lies within 2^-51 ulp of the middle between two doubles.
// 6 FP64 instructions; outside the window in which no intermediate over- or
// underflows, the division.
__device__ __forceinline__ double div_pos(double a, double b) {
    const unsigned ha = (unsigned)__double2hiint(a);
    if (ha - (700u << 20) >= (600u << 20) || !recip_window(b)) return a / b;
    const double y = recip_newton(b), q = a * y;
    return fma(fma(-b, q, a), y, q);
}

// p / d for p < 2^31 by the multiplier m = floor(2^32 / d) + 1 of
// fast_div_mul and one correction (the estimate is at most one too large)
inline unsigned fast_div_mul(int d) { return (unsigned)(0x100000000ull / (unsigned)d + 1); }
__device__ __forceinline__ unsigned fast_div(unsigned p, unsigned d, unsigned m) {
    const unsigned q = d == 1 ? p : __umulhi(p, m);
    return q * d > p ? q - 1 : q;
}

// Programmatic dependent launch: a kernel launched with launch_pdl may start
// while the kernel before it on the stream is finishing; it waits here for
// that kernel's completion (and its memory) before touching anything the
// earlier kernel writes.  Without the launch attribute the wait returns at
// once.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the kernel after this one start while this one still runs, as far as
// its pdl_wait(): for grids that leave most of the chip idle, followed by
// kernels with work of their own before the wait.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------ reductions ---

__device__ inline double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ inline double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// An FP32 sum that carries its rounding errors (Knuth's two-sum): the sums of a
// thread that marches through planes, so that their rounding does not grow with
// the planes a block takes: what is left is half an ulp of each term's magnitude,
// where a chain of n fused steps has up to n times that.  Seven FP32 additions a
// term, no FP64 (the product at 250 x 255 x 245: 91 us a launch, 97 with plain
// sums over as many planes, 113 with at most eight).
struct CarriedSum {
    float sum = 0.f, err = 0.f;
    __device__ __forceinline__ void add(float t) {
        const float s = __fadd_rn(sum, t), tp = __fsub_rn(s, sum);
        err = __fadd_rn(err, __fadd_rn(__fsub_rn(sum, __fsub_rn(s, tp)), __fsub_rn(t, tp)));
        sum = s;
    }
    __device__ __forceinline__ double value() const { return (double)sum + (double)err; }
};

// Block reductions.  FP64 runs at 1/64 of the FP32 rate on this GPU, and a
// shuffle tree in every warp is 45 FP64 warp instructions a value: three
// values took 6500 cycles of an SM's FP64 pipe at three blocks per SM.  So
// the threads' values go through shared memory and one warp per value adds
// the eight warps' lanes up and shuffles: 12 FP64 warp instructions.  The
// order is fixed by the thread layout.

// Reduce NV values over a block of kRedThreads threads (ops: 0 = sum,
// 1 = max of values >= 0) and store them as this block's partials at
// partials[NV*block + q] (written by lane 0 of warp q; the block's fence and
// ticket follow in finalize_last_block).
template <int NV>
__device__ inline void block_reduce_store(double (&v)[NV], const int (&op)[NV], double* partials,
                                          int64_t block, int tid) {
    constexpr int kWarps = kRedThreads / 32;
    static_assert(NV <= kWarps, "one warp per value");
    __shared__ double sh[NV][kRedThreads];
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) sh[q][tid] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (wid != q) continue;
        double t = sh[q][lane];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) t = op[q] ? fmax(t, sh[q][32 * w + lane]) : t + sh[q][32 * w + lane];
        t = op[q] ? warp_max(t) : warp_sum(t);
        if (lane == 0) partials[NV * block + q] = t;
    }
}

// Block reduction of NS FP64 sums, one magnitude key (max) and one count,
// stored as the NS + 2 partials (first sum, key_value(max), count, further
// sums) of this block.
template <int NS>
__device__ inline void block_reduce_sums_kc(const double (&sum)[NS], unsigned long long key, unsigned cnt,
                                            double* partials, int64_t block, int tid) {
    __shared__ double sh_s[NS][kRedThreads];
    __shared__ unsigned long long sh_k[kRedThreads / 32];
    __shared__ unsigned sh_c[kRedThreads / 32];
    const unsigned all = 0xffffffffu;
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int q = 0; q < NS; ++q) sh_s[q][tid] = sum[q];
    const unsigned khi = __reduce_max_sync(all, (unsigned)(key >> 32));
    const unsigned klo = __reduce_max_sync(all, (unsigned)(key >> 32) == khi ? (unsigned)key : 0u);
    cnt = __reduce_add_sync(all, cnt);
    if (lane == 0) {
        sh_k[wid] = ((unsigned long long)khi << 32) | klo;
        sh_c[wid] = cnt;
    }
    __syncthreads();
    if (wid != 0) return;
    double t[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        t[q] = sh_s[q][lane];
#pragma unroll
        for (int w = 1; w < kRedThreads / 32; ++w) t[q] += sh_s[q][32 * w + lane];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < NS; ++q) t[q] += __shfl_xor_sync(all, t[q], o);
    if (lane == 0) {
        unsigned long long tk = 0;
        unsigned tc = 0;
        for (int w = 0; w < kRedThreads / 32; ++w) {
            tk = sh_k[w] > tk ? sh_k[w] : tk;
            tc += sh_c[w];
        }
        double* out = partials + (NS + 2) * block;
        out[0] = t[0];
        out[1] = key_value(tk);
        out[2] = (double)tc;
#pragma unroll
        for (int q = 1; q < NS; ++q) out[2 + q] = t[q];
    }
}

// One sum of type S, one magnitude key and one count, stored as the three
// partials (sum, key_value(max), count): an FP32 sum by FP32 shuffles within
// the warps, an FP64 one as above.
template <typename S>
__device__ inline void block_reduce_skc(S sum, unsigned long long key, unsigned cnt, double* partials,
                                        int64_t block, int tid) {
    if constexpr (sizeof(S) == 8) {
        const double one[1] = {sum};
        block_reduce_sums_kc<1>(one, key, cnt, partials, block, tid);
    } else {
        __shared__ double sh_s[kRedThreads / 32];
        __shared__ unsigned long long sh_k[kRedThreads / 32];
        __shared__ unsigned sh_c[kRedThreads / 32];
        const unsigned all = 0xffffffffu;
        const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(all, sum, o);
        const unsigned khi = __reduce_max_sync(all, (unsigned)(key >> 32));
        const unsigned klo = __reduce_max_sync(all, (unsigned)(key >> 32) == khi ? (unsigned)key : 0u);
        cnt = __reduce_add_sync(all, cnt);
        if (lane == 0) {
            sh_s[wid] = (double)sum;
            sh_k[wid] = ((unsigned long long)khi << 32) | klo;
            sh_c[wid] = cnt;
        }
        __syncthreads();
        if (tid == 0) {
            double ts = 0.0;
            unsigned long long tk = 0;
            unsigned tc = 0;
            for (int w = 0; w < kRedThreads / 32; ++w) {
                ts += sh_s[w];
                tk = sh_k[w] > tk ? sh_k[w] : tk;
                tc += sh_c[w];
            }
            partials[3 * block + 0] = ts;
            partials[3 * block + 1] = key_value(tk);
            partials[3 * block + 2] = (double)tc;
        }
    }
}

}  // namespace paris
