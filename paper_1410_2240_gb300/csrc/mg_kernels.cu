// mg_kernels.cu -- CUDA kernels (sm_103a) of the variable-density pressure projection.
//
// Every kernel works on one grid level stored in C order [k][j][i] (x fastest).
// Face arrays hold the LOW face of each cell: bx[c] couples cells c-1 and c in x;
// bx[.][.][0] is the wall (0).  The high wall face is not stored (closed).
// A "live" cell has at least one open face (dinv > 0); other cells (solid or
// isolated) hold p = 0 and are excluded from means and norms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "mg_internal.cuh"

namespace mg {

static std::atomic<unsigned long long> g_launches{0};
unsigned long long launch_count() { return g_launches.load(std::memory_order_relaxed); }
void note_kernel_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

namespace {

inline void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

constexpr int kRowThreads = 128;

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sums of a and b over the block (NT = blockDim.x threads), valid in thread 0.  An FP64 addition holds
// a scheduler's FP64 unit for some 79 cycles whatever the lanes it is for, so the sums are taken with
// few warp-wide additions: every thread stores its pair, one warp per sum adds the warps' values lane by
// lane and then its own lanes (7 + 5 additions a sum for 256 threads, 45 when every warp first added its
// own lanes: 12 us of a 256^3 pass, the whole time of a 128^3 one).
template <int NT, bool TWO = true>
__device__ __forceinline__ void block_sum2(double &a, double &b)
{
    constexpr int W = NT / 32;
    __shared__ double sh[2][NT];
    sh[0][threadIdx.x] = a;
    if (TWO) sh[1][threadIdx.x] = b;
    __syncthreads();
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    double r = 0.0;
    if (w < (TWO ? 2 : 1)) {
        double v[W];
#pragma unroll
        for (int k = 0; k < W; k++) v[k] = sh[w][32 * k + l];
#pragma unroll
        for (int o = W / 2; o > 0; o /= 2)
#pragma unroll
            for (int k = 0; k < o; k++) v[k] += v[k + o];
        r = warp_sum(v[0]);
        if (TWO && w == 1 && l == 0) sh[1][0] = r;  // (lane 0 alone read that word)
    }
    __syncthreads();
    a = r;
    if (TWO) b = sh[1][0];
    __syncthreads();
}
template <int NT>
__device__ __forceinline__ double block_sum(double v)
{
    double none = 0.0;
    block_sum2<NT, false>(v, none);
    return v;
}

// A scalar every thread of a block needs, computed by thread 0 and shared: FP64 divisions and
// square roots of the CG's scalars would otherwise run in every thread, on the FP64 unit these
// passes are bound by (tens of operations per thread, one to two per cell).  f() is called in
// thread 0 only; the value is the one each thread would have computed.
template <typename F>
__device__ __forceinline__ double block_scalar(F f)
{
    __shared__ double v;
    if (threadIdx.x == 0) v = f();
    __syncthreads();
    return v;
}

// Sums the per-block partial pairs in a fixed order (deterministic) into dscal.
__global__ void k_finish2(const double *__restrict__ partials, int nblocks, double *__restrict__ dscal, int slot0,
                          int slot1)
{
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nblocks; i += blockDim.x) {
        a += partials[2 * i];
        b += partials[2 * i + 1];
    }
    block_sum2<kRedThreads>(a, b);
    if (threadIdx.x == 0) {
        if (slot0 >= 0) dscal[slot0] = a;
        if (slot1 >= 0) dscal[slot1] = b;
    }
}

// The end of a grid-wide reduction in the reducing kernel itself: every block stores its pair of
// block sums (valid in thread 0); the last block to finish -- a counter in the word after the
// 2 * kRedBlocks partials, reset by that block -- sums the pairs in k_finish2's order and writes
// dscal[slot0], dscal[slot1] (slots < 0: not written).  The same sums as a separate k_finish2
// launch, one launch fewer.  Returns true in the last block (all its threads).
__device__ bool reduce_finish(double a, double b, double *partials, double *dscal, int slot0, int slot1)
{
    __shared__ bool last;
    unsigned *ctr = reinterpret_cast<unsigned *>(partials + 2 * kRedBlocks);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = a;
        partials[2 * blockIdx.x + 1] = b;
        __threadfence();
        last = atomicAdd(ctr, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double x = 0.0, y = 0.0;
    // two strides per iteration, both loads issued before either sum: half the chain of
    // dependent L2 round trips, the same additions in the same order
    const int nb = (int)gridDim.x;
    for (int i = threadIdx.x; i < nb; i += 2 * blockDim.x) {
        const int i2 = i + (int)blockDim.x;
        const double x0 = __ldcg(partials + 2 * i), y0 = __ldcg(partials + 2 * i + 1);
        const double x1 = i2 < nb ? __ldcg(partials + 2 * i2) : 0.0, y1 = i2 < nb ? __ldcg(partials + 2 * i2 + 1) : 0.0;
        x += x0;
        y += y0;
        if (i2 < nb) {
            x += x1;
            y += y1;
        }
    }
    block_sum2<kRedThreads>(x, y);
    if (threadIdx.x == 0) {
        if (slot0 >= 0) dscal[slot0] = x;
        if (slot1 >= 0) dscal[slot1] = y;
        *ctr = 0u;
    }
    return true;
}

// The last block of a grid to get here (the counter after the partials, reset by that block):
// true in all its threads.  For kernels that need one block to act after every block has read
// something, with nothing to sum.
__device__ bool last_block(double *partials)
{
    __shared__ bool last;
    unsigned *ctr = reinterpret_cast<unsigned *>(partials + 2 * kRedBlocks);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ctr, 1u) == gridDim.x - 1;
        if (last) *ctr = 0u;
    }
    __syncthreads();
    return last;
}

__device__ __forceinline__ void cell_of(unsigned idx, int nx, int ny, int &i, int &j, int &k)
{
    const unsigned t = idx / (unsigned)nx;
    i = (int)(idx - t * (unsigned)nx);
    k = (int)(t / (unsigned)ny);
    j = (int)(t - (unsigned)k * (unsigned)ny);
}

// ---------------------------------------------------------------------------
// Face coefficients (Eq. density, H(phi) = phi; face product (1/rho)*area):
// rho = rho_a + drho*phi, beta = 2/(rho_L + rho_R) on open faces.  Rounded as
// separate IEEE operations (no contraction) so that it is reproducible.
// ---------------------------------------------------------------------------
// Set-up kernels walk kRun cells up a z-column per thread.  A quotient x / den depends on den
// alone, so each keeps its last divisor and quotient and divides again only when the divisor's
// bits change: in a uniform region (pure air, pure water, constant coefficients) that is once
// per run instead of once per cell, and the results are those of dividing every time.
constexpr int kRun = 16;
// a compile-time bool as a value (a generic lambda's case)
template <bool B>
struct BoolTag {
    static constexpr bool value = B;
};
// Kernels that share values along rows (k_face_coeffs, k_phi_grad, k_divergence_flux, k_mom_parts): blocks of at most
// kPhiThreads threads over rows of at most kPhiW cells, kPhiRun planes per block.
constexpr int kPhiW = 256, kPhiThreads = 512, kPhiRun = 8;
constexpr int kMomRun = 2;  // k_mom_parts on grids of medium size

__device__ __forceinline__ bool same_bits(double a, double b)
{
    return __double_as_longlong(a) == __double_as_longlong(b);
}
__device__ __forceinline__ bool same_bits(float a, float b) { return __float_as_int(a) == __float_as_int(b); }

// a / b as a call: the compiler cannot run a call speculatively, so a memo that skips the
// division really skips it (an inlined division is if-converted and runs on every lane, and on
// this part's narrow FP64 unit it costs as much as the rest of the pass)
template <typename T>
__device__ __noinline__ T div_call(T a, T b)
{
    return a / b;
}

// float -> double on the integer pipe.  The hardware conversion issues on the FP64 unit, which
// bounds the CG kernels that widen an FP32 field per cell.  From the IEEE 754 binary32 and binary64
// layouts: the sign is kept, the exponent rebiased (127 -> 1023), the 23-bit fraction shifted into
// the top of the 52-bit one; zeros, infinities and NaNs map field by field.  Subnormal floats (never
// produced by the scaled cycles, but possible) take the hardware conversion.  Exact: every float is
// a double.
__device__ __noinline__ double f2d_slow(float x) { return (double)x; }
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x);
    const unsigned e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
    const unsigned long long sgn = (unsigned long long)(b >> 31) << 63;
    if (e == 0u) return m ? f2d_slow(x) : __longlong_as_double((long long)sgn);
    const unsigned long long ee = (e == 0xffu) ? 0x7ffull : (unsigned long long)(e + 896u);
    return __longlong_as_double((long long)(sgn | (ee << 52) | ((unsigned long long)m << 29)));
}
__device__ __forceinline__ double widen(double x) { return x; }

// x > 0 and x == 0 decided on the integer pipe (an FP64 comparison occupies the FP64 unit, the
// limiting resource of the FP64 passes).  pos_bits(x) equals x > 0 for every x but a NaN with a
// clear sign bit; the coefficients, inverse diagonals and live masks it is applied to are never
// NaN for finite input.  zero_bits(x) equals x == 0 for every x.
__device__ __forceinline__ bool pos_bits(double x) { return __double_as_longlong(x) > 0; }
// x > 0 for every x: a NaN is not (the sums of faces that may hold one)
__device__ __forceinline__ bool pos_number(double x)
{
    return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
// (from its two words: of the 64-bit pattern shifted left the compiler makes an FP64 comparison again)
__device__ __forceinline__ bool zero_bits(double x)
{
    return (((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x)) == 0u;
}
__device__ __forceinline__ bool zero_bits(float x) { return (__float_as_int(x) << 1) == 0; }
// 0 + x: +0 for a zero of either sign
__device__ __forceinline__ double zero_plus(double x) { return zero_bits(x) ? 0.0 : x; }

// ---------------------------------------------------------------------------
// Bounds-check build (-DMGP_CHECK).  Before its loads and stores a kernel checks that every index
// it is about to use, within the guards of its stencil, lies inside the array it indexes
// (nx*ny*nz cells, a colour half, a coarse level); a thread with an index outside skips its
// accesses and records the kernel and the index (the first such record and a count, read by
// mg_check_read).  Nothing traps.  In the normal build MG_CK is the constant true and every check
// folds away.
// ---------------------------------------------------------------------------
enum CheckKernel : unsigned {
    CK_SMOOTH = 1, CK_SMOOTH_SPLIT, CK_SMOOTH_SPLIT4, CK_RESTRICT, CK_RESTRICT_PAIRS, CK_PROLONG, CK_COARSE_SOLVE,
    CK_TAIL, CK_RESID, CK_SPLIT_SLOT, CK_PCG_APPLY, CK_DIVERGENCE, CK_CORRECT, CK_ADJOINT, CK_PHI_GRAD,
    CK_FACE_COEFFS, CK_DIAG_INV, CK_MOMENTUM, CK_LABEL, CK_VOF, CK_NARROW, CK_POW2
};
#ifdef MGP_CHECK
__device__ unsigned long long g_check_first = 0;  // kernel id << 48 | (index & (2^48 - 1)); 0: none
__device__ unsigned long long g_check_count = 0;
__device__ __noinline__ void ck_record(unsigned kid, long long idx)
{
    atomicAdd(&g_check_count, 1ull);
    atomicCAS(&g_check_first, 0ull,
              ((unsigned long long)kid << 48) | ((unsigned long long)idx & 0xffffffffffffull));
}
// [lo, hi] inside [0, n)
__device__ __forceinline__ bool ck_in(long long lo, long long hi, long long n, unsigned kid)
{
    if (lo >= 0 && hi < n) return true;
    ck_record(kid, lo < 0 ? lo : hi);
    return false;
}
#define MG_CK(lo, hi, n, kid) ck_in((long long)(lo), (long long)(hi), (long long)(n), (unsigned)(kid))
#else
#define MG_CK(lo, hi, n, kid) true
#endif
// double -> float, rounded to nearest (ties to even), on the integer pipe: the hardware conversion
// issues on the FP64 unit, the limiting resource of the FP64 passes that hand an FP32 copy to the
// cycles.  From the IEEE 754 layouts: the exponent rebiased (1023 -> 127), the 52-bit fraction cut
// to its top 23 bits and rounded by the 29 bits cut off (above half, or exactly half with an odd
// result, adds one unit; a carry into the exponent is the correct rounding, up to infinity).
// Zeros map exactly; results that would be subnormal, and infinities and NaNs, take the hardware
// conversion.  The check build compares every result with the hardware conversion.
__device__ __noinline__ float d2f_slow(double x) { return __double2float_rn(x); }
__device__ __forceinline__ float narrow(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sgn = (unsigned)(b >> 63) << 31;
    const int e = (int)((b >> 52) & 0x7ffull);
    const unsigned long long m = b & 0xfffffffffffffull;
    float f;
    if (e == 0 && m == 0) {
        f = __uint_as_float(sgn);
    } else if (e - 896 <= 0 || e - 896 >= 255) {
        f = d2f_slow(x);
    } else {
        const unsigned mant = (unsigned)(m >> 29), rest = (unsigned)(m & 0x1fffffffull);
        unsigned u = sgn | ((unsigned)(e - 896) << 23) | mant;
        if (rest > 0x10000000u || (rest == 0x10000000u && (mant & 1u))) u += 1u;
        f = __uint_as_float(u);
    }
#ifdef MGP_CHECK
    if (__float_as_uint(f) != __float_as_uint(__double2float_rn(x)) && !(isnan(x) && isnan(f)))
        ck_record(CK_NARROW, (long long)(b >> 16));
#endif
    return f;
}

// Products that only some lanes or launches need, as calls: the compiler cannot run a call
// speculatively, so a branch around one is not if-converted into an FP64 instruction that every
// warp issues (predicated off, it still occupies the FP64 unit).
__device__ __noinline__ double dmul_call(double x, double f) { return __dmul_rn(x, f); }
__device__ __noinline__ double dadd_call(double x, double y) { return __dadd_rn(x, y); }
__device__ __noinline__ double sq_mul_call(double b, double g) { return __dmul_rn(__dmul_rn(b, b), g); }

// x * f for f = 2^e, bit for bit the product __dmul_rn(x, f), on the integer pipe where x and the
// product are normal numbers: e added to the exponent field (the FP64 unit is the limiting
// resource of the FP64 set-up and projection passes).  Zeros stay what they are (f > 0); subnormals,
// infinities, NaNs and products outside the normal range take the multiply (a call).  The check build compares every
// result with the multiply.
__device__ __forceinline__ double mul_pow2(double x, double f, int e)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int ex = (hi >> 20) & 0x7ff;
    double y;
    if ((unsigned)(ex - 1) < 2046u && (unsigned)(ex + e - 1) < 2046u)
        y = __hiloint2double(hi + e * (1 << 20), lo);
    else if ((((unsigned)hi << 1) | (unsigned)lo) == 0u)
        y = x;
    else
        y = dmul_call(x, f);
#ifdef MGP_CHECK
    if (__double_as_longlong(y) != __double_as_longlong(__dmul_rn(x, f)) && !isnan(x))
        ck_record(CK_POW2, (long long)((unsigned long long)__double_as_longlong(x) >> 16));
#endif
    return y;
}
// -x, exactly, on the integer pipe (a negation that no operand takes is an FP64 addition)
__device__ __forceinline__ double neg_bits(double x)
{
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
// the product with a power-of-two factor (ok: f = 2^e) or any other (ok = 0: a multiply)
__device__ __forceinline__ double mul_s2(double x, const Scale2 &s) { return s.ok ? mul_pow2(x, s.f, s.e) : dmul_call(x, s.f); }

// cell c = (i, j, k) and the neighbours its guards admit (i > 0: c - 1, i < nx - 1: c + 1, ...)
// inside the nx*ny*nz cells
__device__ __forceinline__ bool ck_cell(long long c, int i, int j, int k, int nx, int ny, int nz, unsigned kid)
{
    const long long n = (long long)nx * ny * nz, sxy = (long long)nx * ny;
    (void)n;
    (void)sxy;
    return MG_CK(c, c, n, kid) && (i == 0 || MG_CK(c - 1, c - 1, n, kid)) &&
           (i >= nx - 1 || MG_CK(c + 1, c + 1, n, kid)) && (j == 0 || MG_CK(c - nx, c - nx, n, kid)) &&
           (j >= ny - 1 || MG_CK(c + nx, c + nx, n, kid)) && (k == 0 || MG_CK(c - sxy, c - sxy, n, kid)) &&
           (k >= nz - 1 || MG_CK(c + sxy, c + sxy, n, kid));
}

// planes per thread: kRun, or as few (at least two) as leave four blocks per SM on the small levels, where the
// walk's length is the kernel's (64^3: 14 us with 16 planes)
inline int run_planes(int nx, int ny, int nz)
{
    int run = kRun;
    while (run > 2 && (size_t)((nx + kRowThreads - 1) / kRowThreads) * ny * ((nz + run - 1) / run) < 4 * 152) run /= 2;
    return run;
}
inline dim3 run_grid(int nx, int ny, int nz)
{
    const int run = run_planes(nx, ny, nz);
    return dim3((unsigned)((nx + kRowThreads - 1) / kRowThreads), (unsigned)ny, (unsigned)((nz + run - 1) / run));
}

// beta_f = 2 / (rho_L + rho_R), rho = rho_a + drho phi (each operation rounded separately); 0 on
// walls and on faces touching a solid cell.  Blocks as k_phi_grad's: each cell's density is formed once
// (shared memory, two buffers by plane parity) and taken by the cells after it along x and y; at the
// block's left edge and first row the neighbour's is formed again, the density below is carried up the
// run.  5 FP64 operations per cell and a division where the divisor changes, instead of 9: 0.42 ms at
// 256^3 (0.52 ms), 128^3 90 us (98 us), 32^3 14 us (28 us, in fewer and larger blocks).
template <bool SOLID>
__global__ void __launch_bounds__(kPhiThreads, 2)
k_face_coeffs(int nx, int ny, int nz, int run, const double *__restrict__ phi, const uint8_t *__restrict__ solid,
              double rho_a, double drho, double den_w, double q_w, double *__restrict__ bx, double *__restrict__ by,
              double *__restrict__ bz)
{
    __shared__ double sh[2][kPhiThreads];
    const int W = blockDim.x, R = blockDim.y;
    const int i = blockIdx.x * W + threadIdx.x, j = blockIdx.y * R + threadIdx.y;
    const int t = threadIdx.y * W + threadIdx.x;
    const bool in = i < nx && j < ny;
    const int k0 = blockIdx.z * run, k1 = min(k0 + run, nz);
    const size_t sxy = (size_t)nx * ny;
    auto rho = [&](double f) { return __dadd_rn(rho_a, __dmul_rn(drho, f)); };
    // the edges' densities, as calls (no FP64 instruction for the warps inside)
    auto rho_edge = [&](double f) { return dadd_call(rho_a, dmul_call(drho, f)); };
    // divisor memo per face direction, from the divisor and quotient of water on
    double dx_last = den_w, qx_last = q_w, dy_last = den_w, qy_last = q_w, dz_last = den_w, qz_last = q_w;
    size_t c = in ? (size_t)k0 * sxy + (size_t)j * nx + i : 0;
    bool s_below = false;
    double r_below = 0.0;
    if (in && k0 > 0) {
        s_below = SOLID && solid[c - sxy];
        r_below = rho(phi[c - sxy]);
    }
    // a cell's inputs (phi and the solid flags of the cell and its x- and y- neighbours), all loaded at
    // once; the next cell's are loaded before this one's faces are formed and stored
    const bool ex = threadIdx.x == 0 && i > 0, ey = threadIdx.y == 0 && j > 0;
    struct In {
        double pc, px, py;
        bool sc, sx, sy;
    };
    auto load = [&](size_t cc) {
        In v{};
        if (!in) return v;
        v.pc = phi[cc];
        if (ex) v.px = phi[cc - 1];
        if (ey) v.py = phi[cc - nx];
        if (SOLID) {
            v.sc = solid[cc];
            v.sx = i > 0 && solid[cc - 1];
            v.sy = j > 0 && solid[cc - nx];
        }
        return v;
    };
    In cur = load(c);
    for (int k = k0; k < k1; k++, c += sxy) {
        const In nxt = k + 1 < k1 ? load(c + sxy) : cur;
        const double rc = rho(cur.pc);
        double *const buf = sh[k & 1];
        buf[t] = rc;
        __syncthreads();  // one barrier per plane: a buffer is written again two planes later
        if (in && MG_CK(c, c, (long long)sxy * nz, CK_FACE_COEFFS)) {
            double v = 0.0;
            if (i > 0 && !cur.sc && !cur.sx) {
                const double den = __dadd_rn(ex ? rho_edge(cur.px) : buf[t - 1], rc);
                if (!same_bits(den, dx_last)) {
                    dx_last = den;
                    qx_last = div_call(2.0, den);
                }
                v = qx_last;
            }
            bx[c] = v;
            v = 0.0;
            if (j > 0 && !cur.sc && !cur.sy) {
                const double den = __dadd_rn(ey ? rho_edge(cur.py) : buf[t - W], rc);
                if (!same_bits(den, dy_last)) {
                    dy_last = den;
                    qy_last = div_call(2.0, den);
                }
                v = qy_last;
            }
            by[c] = v;
            v = 0.0;
            if (k > 0 && !cur.sc && !s_below) {
                const double den = __dadd_rn(r_below, rc);
                if (!same_bits(den, dz_last)) {
                    dz_last = den;
                    qz_last = div_call(2.0, den);
                }
                v = qz_last;
            }
            bz[c] = v;
        }
        s_below = cur.sc;
        r_below = rc;
        cur = nxt;
    }
}

// dinv = 1 / (sum of the six face coefficients), summed x-, x+, y-, y+, z-, z+; 0 if none is
// open.  Optionally (op != null) the CG operator's arrays scaled by `scale` = h^-2: op->dinv =
// scale * sum, op->bx/by/bz = scale * the faces (mul_s2: the products, on the integer pipe when
// h^-2 is a power of two).  kRun cells per thread with the divisor memo above.
template <typename T>
// open (optional): per cell the open bits of its three low faces (x 1, y 2, z 4), kept from the
// last call; where they change, *changed = 1 (the fluid regions must be labelled again)
__global__ void k_diag_inv(int nx, int ny, int nz, int run, const T *__restrict__ bx, const T *__restrict__ by,
                           const T *__restrict__ bz, T *__restrict__ dinv, LevelArrays<T> op, Scale2 scale,
                           uint8_t *__restrict__ open, double *__restrict__ changed)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= nx) return;
    const int k0 = blockIdx.z * run, k1 = min(k0 + run, nz);
    const size_t sxy = (size_t)nx * ny;
    T s_last = T(1), q_last = T(1);
    size_t c = (size_t)k0 * sxy + (size_t)j * nx + i;
    T bz_lo = bz[c];
    // a cell's loads at once; the next cell's issued before this one's stores
    struct In {
        T x0, x1, y0, y1, zh;
        uint8_t ob;
    };
    auto load = [&](size_t cc, int kk) {
        In v;
        v.x0 = bx[cc];
        v.x1 = (i < nx - 1) ? bx[cc + 1] : T(0);
        v.y0 = by[cc];
        v.y1 = (j < ny - 1) ? by[cc + nx] : T(0);
        v.zh = (kk < nz - 1) ? bz[cc + sxy] : T(0);
        v.ob = open ? open[cc] : 0;
        return v;
    };
    In cur = load(c, k0);
    for (int k = k0; k < k1; k++, c += sxy) {
        const In nxt = k + 1 < k1 ? load(c + sxy, k + 1) : cur;
        const T bz_hi = cur.zh;
        T s = cur.x0;
        s += cur.x1;
        s += cur.y0;
        s += cur.y1;
        s += bz_lo;
        s += bz_hi;
        if (op.dinv) {
            op.dinv[c] = mul_s2(s, scale);
            op.bx[c] = mul_s2(cur.x0, scale);
            op.by[c] = mul_s2(cur.y0, scale);
            op.bz[c] = mul_s2(bz_lo, scale);
        }
        if (open) {
            const uint8_t bits = (uint8_t)((pos_bits(cur.x0) ? 1 : 0) | (pos_bits(cur.y0) ? 2 : 0) | (pos_bits(bz_lo) ? 4 : 0));
            if (cur.ob != bits) {
                open[c] = bits;
                *changed = 1.0;
            }
        }
        cur = nxt;
        bz_lo = bz_hi;
        T q = T(0);
        if (pos_number(s)) {
            if (!same_bits(s, s_last)) {
                s_last = s;
                q_last = div_call(T(1), s);
            }
            q = q_last;
        }
        dinv[c] = q;
    }
}

// Coarse face coefficient = mean of the 2x2 coplanar fine faces it covers.
__global__ void k_restrict_coeffs(int nx, int ny, int nz, const double *__restrict__ bx,
                                  const double *__restrict__ by, const double *__restrict__ bz,
                                  double *__restrict__ cbx, double *__restrict__ cby, double *__restrict__ cbz)
{
    const int NX = nx / 2, NY = ny / 2;
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y, K = blockIdx.z;
    if (I >= NX) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t f = (size_t)(2 * K) * sxy + (size_t)(2 * J) * nx + 2 * I;  // fine cell (2I, 2J, 2K)
    const size_t C = ((size_t)K * NY + J) * NX + I;
    cbx[C] = 0.25 * (((bx[f] + bx[f + nx]) + bx[f + sxy]) + bx[f + sxy + nx]);
    cby[C] = 0.25 * (((by[f] + by[f + 1]) + by[f + sxy]) + by[f + sxy + 1]);
    cbz[C] = 0.25 * (((bz[f] + bz[f + 1]) + bz[f + nx]) + bz[f + nx + 1]);
}

// Inverse diagonal of a smoothing update: FP64 levels use the stored 1/sum(beta); FP32 levels
// form 1/sum from the six face coefficients already loaded (sum in the order of k_diag_inv),
// which saves reading dinv.
template <typename T>
__device__ __forceinline__ T inv_diag(T stored, T bxl, T bxh, T byl, T byh, T bzl, T bzh)
{
    if (sizeof(T) == 8) return stored;
    const T sum = ((((bxl + bxh) + byl) + byh) + bzl) + bzh;
    return sum > T(0) ? T(1) / sum : T(0);
}

// ---------------------------------------------------------------------------
// Red-black Gauss-Seidel, one colour ((i+j+k) mod 2 == colour).  Each thread
// owns the one cell of that colour in an x-pair of a row:
//     p_c = dinv_c * (sum_f beta_f p_nb - h^2 b_c),  faces x-,x+,y-,y+,z-,z+,
// products accumulated with fused multiply-adds in that order; in FP32 from 0 with the right-hand
// side last, in FP64 from -h^2 b_c: h^2 b is an exponent shift on the integer pipe where h is a power of
// two, so an update is 7 FP64 operations instead of 8 (the pass is bound by them).
// ---------------------------------------------------------------------------
// the right-hand side's factor: h^2, and as a Scale2 (FP64)
template <typename T>
struct GsScale {
    T h2;
    Scale2 s;
};
template <typename T>
GsScale<T> gs_scale(T h2)
{
    return GsScale<T>{h2, scale2((double)h2)};
}
// what the products are added to, a product added, and the update from the sum.  The FP64 sum is kept with
// its sign turned round, h^2 b - sum beta p (the same roundings): a negation of its own would be an FP64
// addition, those of a product's factors are free.
__device__ __forceinline__ double gs_start(double b, const GsScale<double> &g) { return mul_s2(b, g.s); }
__device__ __forceinline__ float gs_start(float, const GsScale<float> &) { return 0.f; }
// the same with the kind of the factor known to the kernel (POW2; FP32: not asked): a product that is none of the shift's
// is a multiplication in place, where gs_start makes a call
template <bool POW2>
__device__ __forceinline__ double gs_start_of(double b, const GsScale<double> &g)
{
    return POW2 ? mul_pow2(b, g.s.f, g.s.e) : __dmul_rn(b, g.s.f);
}
template <bool POW2>
__device__ __forceinline__ float gs_start_of(float, const GsScale<float> &) { return 0.f; }
__device__ __forceinline__ double gs_add(double beta, double p, double s) { return fma(beta, -p, s); }
__device__ __forceinline__ float gs_add(float beta, float p, float s) { return fmaf(beta, p, s); }
__device__ __forceinline__ double gs_update(double s, double, double d, const GsScale<double> &) { return -d * s; }
__device__ __forceinline__ float gs_update(float s, float b, float d, const GsScale<float> &g) { return d * fmaf(-g.h2, b, s); }

// ZERO: the iterate is zero (the first pass of a cycle from a zero guess): the products with it are
// zeros, so only b and the inverse diagonal are read.  Both precisions take 1/sum from dinv (in FP32 the
// hierarchy stores exactly inv_diag's value).  ROWS (the finest FP64 level, and coarse levels from kRecCells64 and
// kRecCells32 cells on): rows with a record (launch_row_records) take the faces and the inverse diagonal from it, the
// same values: in FP64 24 bytes per cell and pass instead of 56, since a pass that loads the faces is bound by HBM (0.139 ms at 256^3) as
// much as by the FP64 unit (0.132 ms at 8 operations, 0.115 at 7).  Sweep at 256^3, FP64: 0.271 ms with
// 8 operations and every face loaded, 0.257 with 7 and the short zero pass, 0.231 with the records
// too (the average over the passes of a cycle from zero); 128^3 40.6 -> 34.2 us.
// Where h is no power of two an update is 8 operations, the eighth in a call: V-cycle at 256^3 1.55 ms, 1.67 with h = 1/30 (2.09 with
// both before).  FP32 coarse levels: kRecCells32 has both sides.
// GATE: a pass queued before the host knows whether the iteration has ended: it stores nothing unless the squared
// residual norm *gate.rr is finite and above gate.limit (both compared as integers: not negative).
template <typename T, bool ZERO, bool ROWS, bool GATE = false>
__global__ void k_smooth(int nx, int ny, int nz, GsScale<T> gs, LevelArrays<T> L, const T *__restrict__ b,
                         T *__restrict__ p, int colour, const T *__restrict__ rec, Gate gate)
{
    bool go = true;
    if constexpr (GATE) {
        const long long rr = __double_as_longlong(*gate.rr);
        go = rr > __double_as_longlong(gate.limit) && rr < 0x7ff0000000000000ll;
    }
    const int j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + colour) & 1);
    if (i >= nx || j >= ny) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_SMOOTH)) return;
    const T bc = b[c];
    if (ZERO) {
        p[c] = gs_update(gs_start(bc, gs), bc, L.dinv[c], gs);
        return;
    }
    const bool xl = i > 0, xh = i < nx - 1, yl = j > 0, yh = j < ny - 1, zl = k > 0, zh = k < nz - 1;
    // the neighbours are loaded before the row's record is known, so a row with one waits for one round trip
    const T pxl = xl ? p[c - 1] : T(0), pxh = xh ? p[c + 1] : T(0);
    const T pyl = yl ? p[c - nx] : T(0), pyh = yh ? p[c + nx] : T(0);
    const T pzl = zl ? p[c - sxy] : T(0), pzh = zh ? p[c + sxy] : T(0);
    T bxl, bxh, byl, byh, bzl, bzh, d;
    bool loaded = false;
    if constexpr (ROWS) {
        using V2 = std::conditional_t<sizeof(T) == 8, double2, float2>;
        const T *r = rec + 8 * ((size_t)k * ny + j);
        const V2 v0 = *reinterpret_cast<const V2 *>(r);
        if (!zero_bits(v0.x)) {
            const V2 v1 = *reinterpret_cast<const V2 *>(r + 2);
            bxl = bxh = v0.x;
            byl = byh = v0.y;
            bzl = v1.x;
            bzh = v1.y;
            // an address, not a branch: lanes apart at a wall would run the update's last product twice
            d = r[xl && xh ? 4 : 5];
            loaded = true;
        }
    }
    if (!loaded) {
        bxl = L.bx[c];
        bxh = xh ? L.bx[c + 1] : T(0);
        byl = L.by[c];
        byh = yh ? L.by[c + nx] : T(0);
        bzl = L.bz[c];
        bzh = zh ? L.bz[c + sxy] : T(0);
        d = L.dinv[c];
    }
    T s = gs_start(bc, gs);
    if (xl) s = gs_add(bxl, pxl, s);
    if (xh) s = gs_add(bxh, pxh, s);
    if (yl) s = gs_add(byl, pyl, s);
    if (yh) s = gs_add(byh, pyh, s);
    if (zl) s = gs_add(bzl, pzl, s);
    if (zh) s = gs_add(bzh, pzh, s);
    const T v = gs_update(s, bc, d, gs);
    if (go) p[c] = v;
}

// The first red pass of a cycle from zero and the black pass after it in one launch (FP32 levels below the
// finest), where another red pass follows (nu1 >= 2): that pass replaces every red value without reading it, so the first ones,
// a product of b and the inverse diagonal each, are formed by the black cells beside them and not stored.
// Same operations in the same order as the two passes.  These levels are bound by launches and latency:
// FP32 32^3 2.7 us (5.1 in two launches), 64^3 3.7 (6.0), 128^3 10.2 (13.6).  FP64 levels keep the two
// passes: 13 operations per cell instead of 8 on the unit that bounds them (the coarse-grid correction of 64^3
// was 1.9 us faster, of 160^3 6 us slower, solves 0.1 %).
__global__ void k_smooth_first(int nx, int ny, int nz, float h2, LevelArrays<float> L, const float *__restrict__ b,
                               float *__restrict__ p)
{
    const int j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + 1) & 1);
    if (i >= nx || j >= ny) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_SMOOTH)) return;
    const bool in[6] = {i > 0, i < nx - 1, j > 0, j < ny - 1, k > 0, k < nz - 1};
    const size_t nb[6] = {c - 1, c + 1, c - nx, c + nx, c - sxy, c + sxy};
    float bn[6], dn[6], beta[6];
    const float bc = b[c], d = L.dinv[c];
#pragma unroll
    for (int f = 0; f < 6; f++) {
        bn[f] = in[f] ? b[nb[f]] : 0.f;
        dn[f] = in[f] ? L.dinv[nb[f]] : 0.f;
        const float *a = f < 2 ? L.bx : (f < 4 ? L.by : L.bz);
        beta[f] = in[f] ? a[(f & 1) ? nb[f] : c] : 0.f;
    }
    const GsScale<float> gs{h2, Scale2{}};
    float s = gs_start(bc, gs);
#pragma unroll
    for (int f = 0; f < 6; f++)
        if (in[f]) s = gs_add(beta[f], gs_update(gs_start(bn[f], gs), bn[f], dn[f], gs), s);
    p[c] = gs_update(s, bc, d, gs);
}

// the row records of a level, one warp per row (as k_uniform_rows)
template <typename T>
__global__ void k_row_records(int nx, int ny, int nz, const T *__restrict__ bx, const T *__restrict__ by,
                              const T *__restrict__ bz, T *__restrict__ rec)
{
    const int lane = threadIdx.x & 31, r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= ny * nz) return;
    const int j = r % ny, k = r / ny;
    const size_t sxy = (size_t)nx * ny, c0 = (size_t)r * nx;
    const bool inner = nx > 1 && j > 0 && k > 0 && j < ny - 1 && k < nz - 1;
    T vx = T(0), vy = T(0), vzl = T(0), vzh = T(0);
    if (inner) {
        vx = bx[c0 + 1];
        vy = by[c0];
        vzl = bz[c0];
        vzh = bz[c0 + sxy];
    }
    bool ok = inner && pos_bits((double)vx) && pos_bits((double)vy) && pos_bits((double)vzl) && pos_bits((double)vzh);
    if (ok)  // warp-uniform
        for (int i = lane; i < nx; i += 32) {
            const size_t c = c0 + i;
            const bool cell = (i == 0 || same_bits(bx[c], vx)) & same_bits(by[c], vy) & same_bits(by[c + nx], vy) &
                              same_bits(bz[c], vzl) & same_bits(bz[c + sxy], vzh);
            ok = ok & cell;
        }
    ok = __all_sync(0xffffffffu, ok);
    if (lane != 0) return;
    T *r8 = rec + 8 * (size_t)r;
    T i6 = T(0), i5 = T(0);
    if (ok) {
        i6 = div_call(T(1), ((((vx + vx) + vy) + vy) + vzl) + vzh);
        i5 = div_call(T(1), (((vx + vy) + vy) + vzl) + vzh);
    }
    r8[0] = ok ? vx : T(0);
    r8[1] = ok ? vy : T(0);
    r8[2] = ok ? vzl : T(0);
    r8[3] = ok ? vzh : T(0);
    r8[4] = i6;
    r8[5] = i5;
}

// Colour-split layout (Split in mg_internal.cuh): slot of natural cell c in a row of parity
// q = (j + k) & 1, whose colour is (c & 1) ^ q (rows start at even indices).
__device__ __forceinline__ size_t split_slot(size_t c, int q, size_t half)
{
    return (((int)(c & 1) ^ q) ? half : 0) + (c >> 1);
}
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv &f)
{
    const unsigned t = __umulhi(n, f.mult);
    return (t + ((n - t) >> f.s1)) >> f.s2;
}
// parity (j + k) & 1 of the row holding natural index c
__device__ __forceinline__ int row_parity(unsigned c, const Split &sp)
{
    const unsigned row = fdiv(c, sp.fnx), k = fdiv(row, sp.fny), j = row - k * (unsigned)sp.ny;
    return (int)((j + k) & 1u);
}

// Uniform rows.  Away from the interface and the body, every face coefficient around an x-row of
// cells holds one value (pure air or pure water).  urow[k*ny + j] = that value v when the row is
// interior (0 < j < ny-1, 0 < k < nz-1) and every face of every cell of row (j,k) except the two x-walls (bx at i = 0 and the high face of i = nx-1,
// both walls, stored as 0) equals v bitwise, else 0; one warp per row.  A pass that reads urow[r]
// != 0 takes its face values from it instead of loading them: the same values, so the same results.
// On a grid stretched in z the metric factors differ per axis, and a row away from the interface
// holds four values instead: vx on its x-faces, vy on its low and high y-faces, vzl on its low and
// vzh on its high z-faces.  arow[r] (optional) = {vx, vy, vzl, vzh} for such a "banded" row, else
// zeros.  uinv[r] (optional) = the inverse diagonals of such a row's cells {inside, at an x-wall} (left as it
// is for other rows).  count[0] and count[1] (optional) receive the numbers of uniform rows and of banded rows
// that are not uniform.
__global__ void k_uniform_rows(int nx, int ny, int nz, const float *__restrict__ bx, const float *__restrict__ by,
                               const float *__restrict__ bz, float *__restrict__ urow, float4 *__restrict__ arow,
                               float2 *__restrict__ uinv, unsigned *__restrict__ count)
{
    const int warps = blockDim.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * warps + (threadIdx.x >> 5);
    if (r >= ny * nz) return;
    const int j = r % ny, k = r / ny;
    const size_t sxy = (size_t)nx * ny, c0 = (size_t)r * nx;
    const bool inner = j > 0 && k > 0 && j < ny - 1 && k < nz - 1;
    const float vy = by[c0], vx = nx > 1 ? bx[c0 + 1] : vy, vzl = bz[c0], vzh = inner ? bz[c0 + sxy] : 0.f;
    const int bxv = __float_as_int(vx), byv = __float_as_int(vy), bzl = __float_as_int(vzl),
              bzh = __float_as_int(vzh);
    bool ok = inner && vx > 0.f && vy > 0.f && vzl > 0.f && vzh > 0.f;
    if (ok)  // warp-uniform; the loads of a lane's cells are independent of one another
        for (int i = lane; i < nx; i += 32) {
            const size_t c = c0 + i;
            const bool cell = (i == 0 || __float_as_int(bx[c]) == bxv) & (__float_as_int(by[c]) == byv) &
                              (__float_as_int(by[c + nx]) == byv) & (__float_as_int(bz[c]) == bzl) &
                              (__float_as_int(bz[c + sxy]) == bzh);
            ok = ok & cell;
        }
    ok = __all_sync(0xffffffffu, ok);
    if (lane == 0) {
        const bool uni = ok && bxv == byv && bzl == byv && bzh == byv;
        urow[r] = uni ? vy : 0.f;
        if (arow) arow[r] = ok ? make_float4(vx, vy, vzl, vzh) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (uinv && ok)
            uinv[r] = make_float2(1.f / (((((vx + vx) + vy) + vy) + vzl) + vzh), 1.f / ((((vx + vy) + vy) + vzl) + vzh));
        if (count && ok) atomicAdd(&count[uni ? 0 : 1], 1u);
    }
}

// One colour of red-black Gauss-Seidel on the colour-split layout (FP32, all dims even): the
// cell's six neighbours are the other colour's slots m-1+(i&1), m+(i&1), m -+ nx/2, m -+ nx*ny/2
// (m = c >> 1), read contiguously; b and the result are the own colour's slot m.  A pass moves
// the face coefficients (none on uniform rows), half of p and half of b instead of all of p and
// b.  Same arithmetic, in the same order, as k_smooth<float>.  Used where nx % 8 != 0
// (k_smooth_split4 otherwise).
__global__ void k_smooth_split(int nx, int ny, int nz, float h2, LevelArrays<float> L, const float *__restrict__ b,
                               float *__restrict__ p, int colour, const float *__restrict__ urow, int rev, int zero)
{
    const int j = rev ? ny - 1 - (int)blockIdx.y : (int)blockIdx.y, k = rev ? nz - 1 - (int)blockIdx.z : (int)blockIdx.z;
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + colour) & 1);
    if (i >= nx) return;
    const size_t sxy = (size_t)nx * ny, half = sxy * nz / 2;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    const size_t m = c >> 1, hx = nx / 2, hxy = sxy / 2;
    const float *__restrict__ o = p + (colour ? 0 : half);  // the other colour
    const int odd = i & 1;
    const size_t own = (colour ? half : 0) + m;
    if (!(ck_cell((long long)c, i, j, k, nx, ny, nz, CK_SMOOTH_SPLIT) && MG_CK(m, m, half, CK_SMOOTH_SPLIT) &&
          (i == 0 || MG_CK(m - 1 + odd, m - 1 + odd, half, CK_SMOOTH_SPLIT)) &&
          (i >= nx - 1 || MG_CK(m + odd, m + odd, half, CK_SMOOTH_SPLIT)) &&
          (j == 0 || MG_CK((long long)m - (long long)hx, m, half, CK_SMOOTH_SPLIT)) &&
          (j >= ny - 1 || MG_CK(m, m + hx, half, CK_SMOOTH_SPLIT)) &&
          (k == 0 || MG_CK((long long)m - (long long)hxy, m, half, CK_SMOOTH_SPLIT)) &&
          (k >= nz - 1 || MG_CK(m, m + hxy, half, CK_SMOOTH_SPLIT))))
        return;
    // the neighbours and b are loaded before the row's uniform value is known, so a uniform row
    // waits for one memory round trip, not two
    const float v = urow ? urow[(size_t)k * ny + j] : 0.f;
    // zero: the iterate is zero (first pass of a cycle from a zero guess), nothing to read
    const float pxm = (!zero && i > 0) ? o[m - 1 + odd] : 0.f, pxp = (!zero && i < nx - 1) ? o[m + odd] : 0.f;
    const float pym = (!zero && j > 0) ? o[m - hx] : 0.f, pyp = (!zero && j < ny - 1) ? o[m + hx] : 0.f;
    const float pzm = (!zero && k > 0) ? o[m - hxy] : 0.f, pzp = (!zero && k < nz - 1) ? o[m + hxy] : 0.f;
    const float bv = b[own];
    float bxl, bxh, byl, byh, bzl, bzh;
    if (v != 0.f) {  // uniform row: the stored values, x-walls 0
        bxl = i > 0 ? v : 0.f;
        bxh = i < nx - 1 ? v : 0.f;
        byl = byh = bzl = bzh = v;
    } else {
        bxl = L.bx[c];
        bxh = (i < nx - 1) ? L.bx[c + 1] : 0.f;
        byl = L.by[c];
        byh = (j < ny - 1) ? L.by[c + nx] : 0.f;
        bzl = L.bz[c];
        bzh = (k < nz - 1) ? L.bz[c + sxy] : 0.f;
    }
    float s = 0.f;
    if (i > 0) s = fmaf(bxl, pxm, s);
    if (i < nx - 1) s = fmaf(bxh, pxp, s);
    if (j > 0) s = fmaf(byl, pym, s);
    if (j < ny - 1) s = fmaf(byh, pyp, s);
    if (k > 0) s = fmaf(bzl, pzm, s);
    if (k < nz - 1) s = fmaf(bzh, pzp, s);
    p[own] = inv_diag<float>(0.f, bxl, bxh, byl, byh, bzl, bzh) * fmaf(-h2, bv, s);
}

// The same colour pass, four consecutive cells of the colour per thread (nx % 8 == 0): the cells'
// slots mb..mb+3 are float4-aligned in the colour-split arrays, so the x-neighbours (one float4
// and one scalar), the y and z neighbours, b and the results move as float4.  Four independent
// updates per thread keep more loads in flight than one, which the pass needs once uniform rows
// have removed most of its bytes.  Each cell's arithmetic is k_smooth_split's, in its order.
// OFF = (j + k + colour) & 1, the x offset of the colour in the row (uniform across a warp).
// BAND: the row's record is {vx, vy, vzl, vzh} of a banded row (all four equal on a uniform row,
// zeros elsewhere), else {v, v, v, v} from urow.  A row with a record is interior (0 < j < ny-1,
// 0 < k < nz-1: k_uniform_rows), so its update needs no y or z wall tests, which keeps the
// record path short; the neighbours are loaded before the record is known, under the wall tests
// any row needs.  Rows without a record take their faces from S, the colour-split copies of the
// face arrays: a cell's low faces are the own colour's slots, its high faces the low faces of its
// +x, +y and +z neighbours, i.e. the other colour's slots of its x-neighbour (as for p), mb + hx
// and mb + hxy; six float4 and one scalar, each value used.
// A record's two inverse diagonals are read from uinv (k_uniform_rows), and only a row's first cell (OFF = 0) or its
// last one (OFF = 1) can lie at an x-wall: without the two divisions and eight wall tests per thread a sweep
// takes 56.9 us at 256^3 instead of 59.4, 192x160x224 27.9 (31.6), 320x192x128 35.3 (39.5), 128^3 15.3 (16.7).  The
// pass waits for its loads (half of the issue slots are used): 67 % of the copy rate at 256^3.  More warps
// in fewer registers (48, 40: spills) take 12 and 20 % longer.
// ROWS: 1 where a warp lies in one row (OFF_ is then the row's offset), 0 where it may hold several
// rows of both parities (off: this thread's; selected per value, so that the warp does not run the
// two parities one after the other).
template <int ROWS, int OFF_, bool BAND, bool ZERO>
__device__ __forceinline__ void split4_body(int nx, int ny, int nz, float h2, const LevelArrays<float> &S,
                                            const float *__restrict__ b, float *__restrict__ p, int colour, float4 rv,
                                            float2 iv, int g, int j, int k, int off, const float *__restrict__ dinv)
{
    const int OFF = ROWS ? OFF_ : off;
    const float v = rv.x;
    const int G = nx / 8;
    const bool wl = !OFF && g == 0, wh = OFF && g == G - 1;  // the first cell, the last cell at an x-wall
    const size_t sxy = (size_t)nx * ny, half = sxy * nz / 2, hx = nx / 2, hxy = sxy / 2;
    const size_t mb = ((size_t)k * sxy + (size_t)j * nx) / 2 + 4 * g;
    const float *__restrict__ o = p + (colour ? 0 : half);
    float *own = p + (colour ? half : 0);
    const float *bo = b + (colour ? half : 0);
    const size_t so = colour ? half : 0, sn = colour ? 0 : half;  // own and other colour in S
    {
        const long long n = (long long)sxy * nz, m = (long long)mb;
        (void)n;
        (void)m;
        if (!(MG_CK(m, m + 3, half, CK_SMOOTH_SPLIT4) &&
              (OFF ? (g >= G - 1 || MG_CK(m + 4, m + 4, half, CK_SMOOTH_SPLIT4))
                   : (g == 0 || MG_CK(m - 1, m - 1, half, CK_SMOOTH_SPLIT4))) &&
              (j == 0 || MG_CK(m - (long long)hx, m - (long long)hx + 3, half, CK_SMOOTH_SPLIT4)) &&
              (j >= ny - 1 || MG_CK(m + hx, m + hx + 3, half, CK_SMOOTH_SPLIT4)) &&
              (k == 0 || MG_CK(m - (long long)hxy, m - (long long)hxy + 3, half, CK_SMOOTH_SPLIT4)) &&
              (k >= nz - 1 || MG_CK(m + hxy, m + hxy + 3, half, CK_SMOOTH_SPLIT4)) &&
              (v != 0.f || (MG_CK(so + m, so + m + 3, n, CK_SMOOTH_SPLIT4) &&
                            MG_CK(sn + m, sn + m + 3 + ((OFF && g < G - 1) ? 1 : 0), n, CK_SMOOTH_SPLIT4) &&
                            (j >= ny - 1 || MG_CK(sn + m + hx, sn + m + hx + 3, n, CK_SMOOTH_SPLIT4)) &&
                            (k >= nz - 1 || MG_CK(sn + m + hxy, sn + m + hxy + 3, n, CK_SMOOTH_SPLIT4))))))
            return;
    }
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    // ZERO: the other colour is zero (first pass of a cycle from a zero guess), nothing to read
    const float4 ox = ZERO ? zero4 : *reinterpret_cast<const float4 *>(o + mb);
    const float oxe = ZERO ? 0.f : (OFF ? ((g < G - 1) ? o[mb + 4] : 0.f) : ((g > 0) ? o[mb - 1] : 0.f));
    const float4 oym = (!ZERO && j > 0) ? *reinterpret_cast<const float4 *>(o + mb - hx) : zero4;
    const float4 oyp = (!ZERO && j < ny - 1) ? *reinterpret_cast<const float4 *>(o + mb + hx) : zero4;
    const float4 ozm = (!ZERO && k > 0) ? *reinterpret_cast<const float4 *>(o + mb - hxy) : zero4;
    const float4 ozp = (!ZERO && k < nz - 1) ? *reinterpret_cast<const float4 *>(o + mb + hxy) : zero4;
    // b of this colour is read next a sweep later: loaded evict-first, so that it leaves L2 to the
    // iterate the next pass reads
    const float4 bv = __ldcs(reinterpret_cast<const float4 *>(bo + mb));
    // the x-neighbours of the four cells: slots mb-1+OFF .. mb+2+OFF and mb+OFF .. mb+3+OFF
    const float xm[4] = {OFF ? ox.x : oxe, OFF ? ox.y : ox.x, OFF ? ox.z : ox.y, OFF ? ox.w : ox.z};
    const float xp[4] = {xm[1], xm[2], xm[3], OFF ? oxe : ox.w};
    const float oy0[4] = {oym.x, oym.y, oym.z, oym.w}, oy1[4] = {oyp.x, oyp.y, oyp.z, oyp.w};
    const float oz0[4] = {ozm.x, ozm.y, ozm.z, ozm.w}, oz1[4] = {ozp.x, ozp.y, ozp.z, ozp.w};
    const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
    float out[4];
    if (ZERO && v == 0.f) {
        // the products are zeros: 1/sum as the hierarchy stores it (natural order: this colour's are every
        // second value of the eight) instead of the six faces it is the inverse of
        const float4 d0 = *reinterpret_cast<const float4 *>(dinv + 2 * mb), d1 = *reinterpret_cast<const float4 *>(dinv + 2 * mb + 4);
        const float dd[4] = {OFF ? d0.y : d0.x, OFF ? d0.w : d0.z, OFF ? d1.y : d1.x, OFF ? d1.w : d1.z};
#pragma unroll
        for (int t = 0; t < 4; t++) out[t] = dd[t] * fmaf(-h2, bb[t], 0.f);
    } else if (v != 0.f) {
        // a row with a record: the diagonal is 6v, or 5v at an x-wall (the sums of inv_diag, in its
        // order: 0 + v = v + 0 = v), on a banded row the same with vx, vy, vzl, vzh in their places; both inverses
        // come with the record
        const float vx = BAND ? rv.x : v, vy = BAND ? rv.y : v, vzl = BAND ? rv.z : v, vzh = BAND ? rv.w : v;
#pragma unroll
        for (int t = 0; t < 4; t++) {
            float s = 0.f;
            if (!(t == 0 && wl)) s = fmaf(vx, xm[t], s);
            if (!(t == 3 && wh)) s = fmaf(vx, xp[t], s);
            s = fmaf(vy, oy0[t], s);
            s = fmaf(vy, oy1[t], s);
            s = fmaf(vzl, oz0[t], s);
            s = fmaf(vzh, oz1[t], s);
            const float d = ((t == 0 && wl) || (t == 3 && wh)) ? iv.y : iv.x;
            out[t] = d * fmaf(-h2, bb[t], s);
        }
    } else {
        const float4 xl = *reinterpret_cast<const float4 *>(S.bx + so + mb);
        const float4 yl = *reinterpret_cast<const float4 *>(S.by + so + mb);
        const float4 zl = *reinterpret_cast<const float4 *>(S.bz + so + mb);
        const float4 xh = *reinterpret_cast<const float4 *>(S.bx + sn + mb);
        const float xe = (OFF && g < G - 1) ? S.bx[sn + mb + 4] : 0.f;
        const float4 yh = (j < ny - 1) ? *reinterpret_cast<const float4 *>(S.by + sn + mb + hx) : zero4;
        const float4 zh = (k < nz - 1) ? *reinterpret_cast<const float4 *>(S.bz + sn + mb + hxy) : zero4;
        // high x-faces: the other colour's slots mb+OFF .. mb+3+OFF, the x-neighbours' low faces
        const float fxl[4] = {xl.x, xl.y, xl.z, xl.w};
        const float fxh[4] = {OFF ? xh.y : xh.x, OFF ? xh.z : xh.y, OFF ? xh.w : xh.z, OFF ? xe : xh.w};
        const float fyl[4] = {yl.x, yl.y, yl.z, yl.w}, fyh[4] = {yh.x, yh.y, yh.z, yh.w};
        const float fzl[4] = {zl.x, zl.y, zl.z, zl.w}, fzh[4] = {zh.x, zh.y, zh.z, zh.w};
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const float bxl = fxl[t], bxh = fxh[t];  // (xe is 0 at the wall)
            const float byl = fyl[t], byh = fyh[t], bzl = fzl[t], bzh = fzh[t];
            float s = 0.f;
            if (!(t == 0 && wl)) s = fmaf(bxl, xm[t], s);
            if (!(t == 3 && wh)) s = fmaf(bxh, xp[t], s);
            if (j > 0) s = fmaf(byl, oy0[t], s);
            if (j < ny - 1) s = fmaf(byh, oy1[t], s);
            if (k > 0) s = fmaf(bzl, oz0[t], s);
            if (k < nz - 1) s = fmaf(bzh, oz1[t], s);
            out[t] = inv_diag<float>(0.f, bxl, bxh, byl, byh, bzl, bzh) * fmaf(-h2, bb[t], s);
        }
    }
    *reinterpret_cast<float4 *>(own + mb) = make_float4(out[0], out[1], out[2], out[3]);
}
template <bool BAND, bool ZERO, int ROWS>
__global__ void k_smooth_split4(int nx, int ny, int nz, float h2, LevelArrays<float> S, const float *__restrict__ b,
                                float *__restrict__ p, int colour, const float *__restrict__ urow,
                                const float4 *__restrict__ arow, const float2 *__restrict__ uinv, int rev,
                                const float *__restrict__ dinv)
{
    // rev: the blocks take the planes (and rows) in descending order, so that a pass that follows
    // an ascending one starts on the data that pass touched last (still in L2)
    const int g = blockIdx.x * blockDim.x + threadIdx.x;  // (blockDim.x = 32 where ROWS = 1)
    const int by = rev ? (int)gridDim.y - 1 - (int)blockIdx.y : (int)blockIdx.y;
    // the planes of the four quarters interleaved in the block order (0, nz/4, nz/2, 3nz/4, 1, ...):
    // the rows without a record gather in a band of planes (an interface), and interleaving runs
    // their face-loading blocks alongside blocks of record rows instead of all together
    const int zb = rev ? (int)gridDim.z - 1 - (int)blockIdx.z : (int)blockIdx.z;
    const int qz = nz / 4;
    const int k = (nz & 3) ? zb : (zb & 3) * qz + (zb >> 2);
    const int j = by * blockDim.y + threadIdx.y;
    if (g >= nx / 8 || j >= ny) return;
    float4 rv;
    if (BAND) {
        rv = arow[(size_t)k * ny + j];
    } else {
        const float v = urow ? urow[(size_t)k * ny + j] : 0.f;
        rv = make_float4(v, v, v, v);
    }
    const float2 iv = uinv ? uinv[(size_t)k * ny + j] : make_float2(0.f, 0.f);
    const int off = (j + k + colour) & 1;
    if (!ROWS) split4_body<0, 0, BAND, ZERO>(nx, ny, nz, h2, S, b, p, colour, rv, iv, g, j, k, off, dinv);
    else if (off) split4_body<1, 1, BAND, ZERO>(nx, ny, nz, h2, S, b, p, colour, rv, iv, g, j, k, 1, dinv);
    else split4_body<1, 0, BAND, ZERO>(nx, ny, nz, h2, S, b, p, colour, rv, iv, g, j, k, 0, dinv);
}

// FP64 residuals for the solver's convergence checks: f(c, (j + k) & 1, r, p_c) for every cell.  The blocks
// take tasks of 256 columns by `run` planes; a thread walks up its column and takes the difference to the cell
// below from the step before (its negative, exactly): 12 FP64 operations for a residual instead of 13, two
// loads less (with the norm, 59 us at 128^3, 68 us with one thread per cell and the sum of p in the same pass).
// r = b - h^-2 sum_f beta_f (p_nb - p_c), summed x-, x+, y-, y+, z-, z+: differences of neighbouring p first, so a
// large smooth offset in p (a hydrostatic pressure) cancels before any product.  Where p and its in-domain neighbours are
// all zero (bitwise, either sign) every product beta (0 - 0) is a signed zero, the sum stays +0
// and the residual is b[c] exactly (for finite coefficients): the test runs on the integer
// pipe and skips the FP64 arithmetic, which dominates this pass on a zero initial guess.
struct ResidGrid {
    unsigned colblocks, tasks;  // blocks of 256 columns; times the runs of planes
    int run;
    FastDiv fcb, fnx;
};
template <typename F>
__device__ __forceinline__ void resid_columns(int nx, int ny, int nz, double ih2, const LevelArrays<double> &L,
                                              const double *__restrict__ b, const double *__restrict__ p,
                                              const ResidGrid &g, F f)
{
    const unsigned sxy = (unsigned)nx * ny;
    for (unsigned task = blockIdx.x; task < g.tasks; task += gridDim.x) {
        const unsigned ch = fdiv(task, g.fcb), col = (task - ch * g.colblocks) * kRedThreads + threadIdx.x;
        if (col >= sxy) continue;
        const int j = (int)fdiv(col, g.fnx), i = (int)(col - (unsigned)j * nx);
        const int k0 = (int)ch * g.run, k1 = min(k0 + g.run, nz);
        const bool xl = i > 0, xh = i < nx - 1, yl = j > 0, yh = j < ny - 1;
        size_t c = (size_t)k0 * sxy + col;
        double pc = p[c], bz = L.bz[c], pzl = k0 > 0 ? p[c - sxy] : 0.0, dz = 0.0;
        if (k0 > 0) dz = pc - pzl;
        for (int k = k0; k < k1; k++, c += sxy) {
            const bool zh = k < nz - 1;
            if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_RESID)) break;
            const double pxl = xl ? p[c - 1] : 0.0, pxh = xh ? p[c + 1] : 0.0, pyl = yl ? p[c - nx] : 0.0,
                         pyh = yh ? p[c + nx] : 0.0, pzh = zh ? p[c + sxy] : 0.0, bc = b[c];
            const double bzh = zh ? L.bz[c + sxy] : 0.0;
            const unsigned long long z = __double_as_longlong(pc) | __double_as_longlong(pxl) | __double_as_longlong(pxh) |
                                         __double_as_longlong(pyl) | __double_as_longlong(pyh) |
                                         __double_as_longlong(pzl) | __double_as_longlong(pzh);
            double r = bc, dzh = 0.0;
            if ((z << 1) != 0ull) {
                const double bxl = L.bx[c], bxh = xh ? L.bx[c + 1] : 0.0, byl = L.by[c], byh = yh ? L.by[c + nx] : 0.0;
                double s = 0.0;
                if (xl) s = fma(bxl, pxl - pc, s);
                if (xh) s = fma(bxh, pxh - pc, s);
                if (yl) s = fma(byl, pyl - pc, s);
                if (yh) s = fma(byh, pyh - pc, s);
                if (k > 0) s = fma(bz, -dz, s);
                if (zh) {
                    dzh = pzh - pc;
                    s = fma(bzh, dzh, s);
                }
                r = fma(-s, ih2, bc);
            }
            f(c, (j + k) & 1, r, pc);
            dz = dzh;
            pzl = pc;
            pc = pzh;
            bz = bzh;
        }
    }
}

template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

// Residual and cell-centred full weighting: coarse b = the mean of the 8 children's residuals.  Their
// sum is sum(b) - h^-2 sum over the 24 outer faces of the 2x2x2 block of beta (p_out - p_in): the 12
// faces inside it enter the two cells they join with opposite signs and cancel.  Half the products
// of forming the 8 residuals (7 FP64 operations per fine cell instead of 14; the FP64 pass is bound
// by them), half the face loads, and no rounding left of the inner fluxes.  Opposite faces of a row are
// added in turn, so the running sum stays a difference of fluxes.  (Leaving out the black children,
// whose residuals the pass before has made zero, is no option: their rounding residuals balance
// the red ones', and the coarse grids amplify what is left by the density ratio; an FP32 cycle from
// a nonzero iterate was 6e-5 off.)
// Children are read as x-pairs (aligned: even nx, 16-byte aligned arrays).  SPLIT: p and b colour by
// colour (FP32 finest level; half: a colour's cells), a pair's colours in the order of the row's
// parity.
template <typename T, bool SPLIT>
__device__ __forceinline__ void restrict_box(int I, int J, int K, int nx, int ny, int nz, T ih2,
                                             const LevelArrays<T> &L, const T *b, const T *p, T *bc, size_t half)
{
    using P2 = typename Pair<T>::type;
    const int NX = nx / 2, NY = ny / 2;
    const size_t sxy = (size_t)nx * ny;
    const size_t C = ((size_t)K * NY + J) * NX + I, c0 = (size_t)(2 * K) * sxy + (size_t)(2 * J) * nx + 2 * I;
    const bool xlo = I > 0, xhi = 2 * I + 2 < nx, ylo = J > 0, yhi = 2 * J + 2 < ny, zlo = K > 0, zhi = 2 * K + 2 < nz;
    if (!(MG_CK(C, C, (long long)NX * NY * (nz / 2), CK_RESTRICT) &&
          MG_CK((long long)c0 - (zlo ? (long long)sxy : 0), c0 + (zhi ? 2 : 1) * sxy + nx + 1, (long long)sxy * nz,
                CK_RESTRICT) &&
          MG_CK((long long)c0 - (ylo ? nx : 0) - (xlo ? 1 : 0), c0 + sxy + (yhi ? 2 : 1) * (size_t)nx + (xhi ? 2 : 1),
                (long long)sxy * nz, CK_RESTRICT)))
        return;
    auto pair = [](const T *a, size_t c) { return *reinterpret_cast<const P2 *>(a + c); };
    // pair and value of p or b in a row of parity q
    auto pair_q = [&](const T *a, size_t c, int q) {
        if (!SPLIT) return pair(a, c);
        P2 v;
        v.x = a[(q ? half : 0) + (c >> 1)];
        v.y = a[(q ? 0 : half) + (c >> 1)];
        return v;
    };
    auto val_q = [&](const T *a, size_t c, int q) { return SPLIT ? a[split_slot(c, q, half)] : a[c]; };
    // every load first: on the small levels the pass is one round trip to L2 long
    P2 pc[2][2], fy[2][2], fz[2][2], py[2][2], pz[2][2];  // [dk][dj]
    T xl[2][2], xh[2][2], pxl[2][2], pxh[2][2], sb = T(0);
#pragma unroll
    for (int dk = 0; dk < 2; dk++)
#pragma unroll
        for (int dj = 0; dj < 2; dj++) {
            const int q = dj ^ dk;
            const size_t c = c0 + dk * sxy + (size_t)dj * nx;
            const bool hy = dj ? yhi : ylo, hz = dk ? zhi : zlo;  // the outer neighbour exists
            const size_t cy = dj ? c + nx : c - nx, cz = dk ? c + sxy : c - sxy;
            P2 none;  // an absent outer neighbour: a closed face
            none.x = none.y = T(0);
            pc[dk][dj] = pair_q(p, c, q);
            xl[dk][dj] = xlo ? L.bx[c] : T(0);
            xh[dk][dj] = xhi ? L.bx[c + 2] : T(0);
            pxl[dk][dj] = xlo ? val_q(p, c - 1, q) : T(0);
            pxh[dk][dj] = xhi ? val_q(p, c + 2, q) : T(0);
            fy[dk][dj] = hy ? pair(L.by, dj ? cy : c) : none;
            py[dk][dj] = hy ? pair_q(p, cy, q ^ 1) : none;
            fz[dk][dj] = hz ? pair(L.bz, dk ? cz : c) : none;
            pz[dk][dj] = hz ? pair_q(p, cz, q ^ 1) : none;
            const P2 bb = pair_q(b, c, q);
            sb += bb.x + bb.y;
        }
    T s = T(0);
#pragma unroll
    for (int dk = 0; dk < 2; dk++)
#pragma unroll
        for (int dj = 0; dj < 2; dj++) {
            const P2 v = pc[dk][dj];
            s = fma(xl[dk][dj], pxl[dk][dj] - v.x, s);
            s = fma(xh[dk][dj], pxh[dk][dj] - v.y, s);
            s = fma(fy[dk][dj].x, py[dk][dj].x - v.x, s);
            s = fma(fy[dk][dj].y, py[dk][dj].y - v.y, s);
            s = fma(fz[dk][dj].x, pz[dk][dj].x - v.x, s);
            s = fma(fz[dk][dj].y, pz[dk][dj].y - v.y, s);
        }
    bc[C] = T(0.125) * fma(-s, ih2, sb);
}

template <typename T, bool SPLIT>
__global__ void k_restrict(int nx, int ny, int nz, T ih2, LevelArrays<T> L, const T *__restrict__ b,
                           const T *__restrict__ p, T *__restrict__ bc, size_t half)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y, K = blockIdx.z;
    if (I >= nx / 2 || J >= ny / 2) return;
    restrict_box<T, SPLIT>(I, J, K, nx, ny, nz, ih2, L, b, p, bc, half);
}

// restrict_box on the colour-split finest FP32 level with nx % 8 == 0, two coarse cells along x per
// thread: the even and the odd cells of a row's four children are pairs of consecutive slots of the
// two colours.  A row with a record ({v, v, v, v} from urow, or {vx, vy, vzl, vzh} of a banded row)
// takes its outer faces from it, the others load them from S, the colour-split faces, as in
// k_smooth_split4.  The pass is bound by instruction issue and load latency; see launch_restrict for
// what it measures.
template <bool BAND>
__global__ void k_restrict4(int nx, int ny, int nz, float ih2, LevelArrays<float> S, const float *__restrict__ b,
                            const float *__restrict__ p, float *__restrict__ bc, const float *__restrict__ urow,
                            const float4 *__restrict__ arow, int rev)
{
    const int NX = nx / 2, NY = ny / 2, NZ = nz / 2;
    const int I = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const int Jb = blockIdx.y * blockDim.y + threadIdx.y;
    const int J = rev ? NY - 1 - Jb : Jb;
    // coarse planes of the four quarters interleaved in the block order, as in the colour passes
    const int zb = rev ? NZ - 1 - (int)blockIdx.z : (int)blockIdx.z;
    const int K = (NZ & 3) ? zb : (zb & 3) * (NZ / 4) + (zb >> 2);
    if (I >= NX || Jb >= NY) return;
    const size_t hx = nx / 2, hxy = (size_t)nx * ny / 2, half = hxy * nz;
    const size_t m0 = (size_t)(2 * K) * hxy + (size_t)(2 * J) * hx + I;  // slot of the block's first row
    const bool xlo = I > 0, xhi = I + 2 < NX, ylo = J > 0, yhi = J < NY - 1, zlo = K > 0, zhi = K < NZ - 1;
    {
        const long long m = (long long)m0, h = (long long)hxy, x = (long long)hx;
        (void)m;
        (void)h;
        (void)x;
        if (!(MG_CK(m - (zlo ? h : 0), m + (zhi ? 2 : 1) * h + x + 1, half, CK_RESTRICT_PAIRS) &&
              MG_CK(m - (ylo ? x : 0) - (xlo ? 1 : 0), m + h + (yhi ? 2 : 1) * x + (xhi ? 2 : 1), half, CK_RESTRICT_PAIRS)))
            return;
    }
    auto ld2 = [](const float *a, size_t m) { return *reinterpret_cast<const float2 *>(a + m); };
    const float2 zero2 = make_float2(0.f, 0.f);
    float2 ev[2][2], od[2][2], ye[2][2], yo[2][2], ze[2][2], zo[2][2], sb = zero2;  // [dk][dj]
    float xm[2][2], xp[2][2];
    float4 rec[2][2];
#pragma unroll
    for (int dk = 0; dk < 2; dk++)
#pragma unroll
        for (int dj = 0; dj < 2; dj++) {
            const int q = dj ^ dk;
            const size_t m = m0 + dk * hxy + dj * hx, row = (size_t)(2 * K + dk) * ny + 2 * J + dj;
            const float *pe = p + (q ? half : 0), *po = p + (q ? 0 : half);  // even and odd cells of the row
            if (BAND) {
                rec[dk][dj] = arow[row];
            } else {
                const float v = urow[row];
                rec[dk][dj] = make_float4(v, v, v, v);
            }
            ev[dk][dj] = ld2(pe, m);
            od[dk][dj] = ld2(po, m);
            xm[dk][dj] = xlo ? po[m - 1] : 0.f;
            xp[dk][dj] = xhi ? pe[m + 2] : 0.f;
            const bool hy = dj ? yhi : ylo, hz = dk ? zhi : zlo;  // the outer neighbour rows exist
            const size_t my = dj ? m + hx : m - hx, mz = dk ? m + hxy : m - hxy;
            ye[dk][dj] = hy ? ld2(po, my) : zero2;  // (the parity of the row beside is the other one)
            yo[dk][dj] = hy ? ld2(pe, my) : zero2;
            ze[dk][dj] = hz ? ld2(po, mz) : zero2;
            zo[dk][dj] = hz ? ld2(pe, mz) : zero2;
            const float2 b0 = ld2(b, m), b1 = ld2(b + half, m);
            sb.x += b0.x + b1.x;
            sb.y += b0.y + b1.y;
        }
    float2 s = zero2;
#pragma unroll
    for (int dk = 0; dk < 2; dk++)
#pragma unroll
        for (int dj = 0; dj < 2; dj++) {
            const int q = dj ^ dk;
            const size_t m = m0 + dk * hxy + dj * hx;
            const float4 rv = rec[dk][dj];
            float x0, x1, x2;  // x-faces before, between and after the two coarse cells
            float2 fye, fyo, fze, fzo;
            if (rv.x != 0.f) {
                x0 = xlo ? rv.x : 0.f;
                x1 = rv.x;
                x2 = xhi ? rv.x : 0.f;
                fye = fyo = make_float2(rv.y, rv.y);
                fze = fzo = dk ? make_float2(rv.w, rv.w) : make_float2(rv.z, rv.z);
            } else {
                const size_t e = q ? half : 0, o = q ? 0 : half;  // even and odd cells of the row
                const float2 xf = ld2(S.bx + e, m);
                x0 = xlo ? xf.x : 0.f;
                x1 = xf.y;
                x2 = xhi ? S.bx[e + m + 2] : 0.f;
                if (dj) {  // the low faces of the row above
                    fye = yhi ? ld2(S.by + o, m + hx) : zero2;
                    fyo = yhi ? ld2(S.by + e, m + hx) : zero2;
                } else {
                    fye = ld2(S.by + e, m);
                    fyo = ld2(S.by + o, m);
                }
                if (dk) {
                    fze = zhi ? ld2(S.bz + o, m + hxy) : zero2;
                    fzo = zhi ? ld2(S.bz + e, m + hxy) : zero2;
                } else {
                    fze = ld2(S.bz + e, m);
                    fzo = ld2(S.bz + o, m);
                }
            }
            const float2 E = ev[dk][dj], O = od[dk][dj];
            s.x = fmaf(x0, xm[dk][dj] - E.x, s.x);
            s.x = fmaf(x1, E.y - O.x, s.x);
            s.y = fmaf(x1, O.x - E.y, s.y);
            s.y = fmaf(x2, xp[dk][dj] - O.y, s.y);
            s.x = fmaf(fye.x, ye[dk][dj].x - E.x, s.x);
            s.x = fmaf(fyo.x, yo[dk][dj].x - O.x, s.x);
            s.y = fmaf(fye.y, ye[dk][dj].y - E.y, s.y);
            s.y = fmaf(fyo.y, yo[dk][dj].y - O.y, s.y);
            s.x = fmaf(fze.x, ze[dk][dj].x - E.x, s.x);
            s.x = fmaf(fzo.x, zo[dk][dj].x - O.x, s.x);
            s.y = fmaf(fze.y, ze[dk][dj].y - E.y, s.y);
            s.y = fmaf(fzo.y, zo[dk][dj].y - O.y, s.y);
        }
    *reinterpret_cast<float2 *>(bc + ((size_t)K * NY + J) * NX + I) =
        make_float2(0.125f * fmaf(-s.x, ih2, sb.x), 0.125f * fmaf(-s.y, ih2, sb.y));
}

// Trilinear cell-centred prolongation added to p (cells with no open face keep p): weights 3/4
// (parent) and 1/4 (next coarse cell on the fine cell's side) per axis; that index clamps at
// walls.  One thread per coarse cell handles its 2x2x2 children as four x-pairs: the 3x3x3 coarse
// neighbourhood is loaded once and every fine load is issued before the dead-cell test, so a
// thread keeps 8 pair loads in flight (one load per thread, then a dependent one, leaves the pass
// bound by memory latency).  A child's 8 products w_z w_y w_x e are summed with fma, z outermost
// and x innermost, the parent before the neighbour on each axis.  p and dinv are aligned to a
// pair (16-byte aligned arrays, even nx).
// the trilinear corrections of coarse cell (I,J,K)'s 8 children, corr[dz][dy][dx]
template <typename T>
__device__ __forceinline__ void prolong_corr(int I, int J, int K, int NX, int NY, int NZ, const T *ec, T corr[2][2][2])
{
    // neighbourhood index 0 = lower neighbour (clamped), 1 = parent, 2 = upper neighbour (clamped)
    const int Is[3] = {max(I - 1, 0), I, min(I + 1, NX - 1)};
    const int Js[3] = {max(J - 1, 0), J, min(J + 1, NY - 1)};
    const int Ks[3] = {max(K - 1, 0), K, min(K + 1, NZ - 1)};
    if (!(MG_CK(((long long)Ks[0] * NY + Js[0]) * NX + Is[0], ((long long)Ks[2] * NY + Js[2]) * NX + Is[2],
                (long long)NX * NY * NZ, CK_PROLONG))) {
        for (int q = 0; q < 8; q++) (&corr[0][0][0])[q] = T(0);
        return;
    }
    T e[3][3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int bb = 0; bb < 3; bb++)
#pragma unroll
            for (int d = 0; d < 3; d++) e[a][bb][d] = ec[((size_t)Ks[a] * NY + Js[bb]) * NX + Is[d]];
    const T w[2] = {T(0.75), T(0.25)};
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++)
#pragma unroll
            for (int dx = 0; dx < 2; dx++) {
                // parent first, then the neighbour on the child's side
                const int ka[2] = {1, dz ? 2 : 0}, jb[2] = {1, dy ? 2 : 0}, id[2] = {1, dx ? 2 : 0};
                T s = T(0);
#pragma unroll
                for (int a = 0; a < 2; a++)
#pragma unroll
                    for (int bb = 0; bb < 2; bb++)
#pragma unroll
                        for (int d = 0; d < 2; d++) s = fma(w[a] * w[bb] * w[d], e[ka[a]][jb[bb]][id[d]], s);
                corr[dz][dy][dx] = s;
            }
}

// urow (optional, the finest FP32 level): a fine row with a uniform value has every cell live, so
// its inverse diagonals are not read
template <typename T, bool SPLIT>
__global__ void k_prolong(int nx, int ny, int nz, const T *__restrict__ ec, const T *__restrict__ dinv,
                          T *__restrict__ p, size_t half, const float *__restrict__ urow)
{
    using P2 = typename Pair<T>::type;
    const int NX = nx / 2, NY = ny / 2, NZ = nz / 2;
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    // on the colour-split finest level, coarse planes of the four quarters interleaved in the block
    // order, as in its colour passes and restriction
    const int zb = blockIdx.z;
    const int K = (SPLIT && (NZ & 3) == 0) ? (zb & 3) * (NZ / 4) + (zb >> 2) : zb;
    if (I >= NX || J >= NY) return;
    {
        const long long n = (long long)nx * ny * nz;
        const long long c0 = ((long long)(2 * K) * ny + 2 * J) * nx + 2 * I;
        const long long c1 = ((long long)(2 * K + 1) * ny + 2 * J + 1) * nx + 2 * I + 1;
        (void)n;
        (void)c0;
        (void)c1;
        if (!(MG_CK(c0, c1, n, CK_PROLONG) && (!SPLIT || MG_CK(c0 >> 1, c1 >> 1, (long long)half, CK_PROLONG))))
            return;
    }
    P2 dv[2][2], pv[2][2];
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            const size_t c = ((size_t)(2 * K + dz) * ny + (2 * J + dy)) * nx + 2 * I;
            if (urow && urow[(size_t)(2 * K + dz) * ny + 2 * J + dy] != 0.f) {
                dv[dz][dy].x = T(1);
                dv[dz][dy].y = T(1);
            } else {
                dv[dz][dy] = *reinterpret_cast<const P2 *>(dinv + c);
            }
            if (SPLIT) {  // the pair's two colours at slot c >> 1 of each half
                const size_t m = c >> 1;
                const bool q = (2 * J + dy + 2 * K + dz) & 1;
                pv[dz][dy].x = p[(q ? half : 0) + m];
                pv[dz][dy].y = p[(q ? 0 : half) + m];
            } else {
                pv[dz][dy] = *reinterpret_cast<const P2 *>(p + c);
            }
        }
    T corr[2][2][2];
    prolong_corr<T>(I, J, K, NX, NY, NZ, ec, corr);
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            T out[2];
#pragma unroll
            for (int dx = 0; dx < 2; dx++) {
                const T dval = dx ? dv[dz][dy].y : dv[dz][dy].x;
                const T pold = dx ? pv[dz][dy].y : pv[dz][dy].x;
                out[dx] = zero_bits(dval) ? pold : pold + corr[dz][dy][dx];
            }
            const size_t c = ((size_t)(2 * K + dz) * ny + (2 * J + dy)) * nx + 2 * I;
            if (SPLIT) {
                const size_t m = c >> 1;
                const bool q = (2 * J + dy + 2 * K + dz) & 1;
                p[(q ? half : 0) + m] = out[0];
                p[(q ? 0 : half) + m] = out[1];
            } else {
                P2 o;
                o.x = out[0];
                o.y = out[1];
                *reinterpret_cast<P2 *>(p + c) = o;
            }
        }
}

// The correction of one red child: the fma chain of prolong_corr for child (dz, dy, dx), from e(a, b, d),
// the coarse value at neighbourhood index a, b, d (0 lower, 1 parent, 2 upper)
template <typename T, typename E>
__device__ __forceinline__ T prolong_child(int dz, int dy, int dx, E e)
{
    const T w[2] = {T(0.75), T(0.25)};
    const int ka[2] = {1, dz ? 2 : 0}, jb[2] = {1, dy ? 2 : 0}, id[2] = {1, dx ? 2 : 0};
    T s = T(0);
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int bb = 0; bb < 2; bb++)
#pragma unroll
            for (int d = 0; d < 2; d++) s = fma(w[a] * w[bb] * w[d], e(ka[a], jb[bb], id[d]), s);
    return s;
}

// Prolongation where a black pass follows (every cycle with nu2 >= 1: the way up starts with the
// black colour).  That pass replaces each black value from the red ones without reading it, so only
// the four red children of a coarse cell are corrected: half the loads, stores and arithmetic, and
// the same iterate after the black pass.  p, dinv natural or, SPLIT, p colour by colour.
template <typename T, bool SPLIT>
__device__ __forceinline__ void prolong_red(int I, int J, int K, int nx, int ny, int nz, const T *ec, const T *dinv,
                                            T *p)
{
    const int NX = nx / 2, NY = ny / 2, NZ = nz / 2;
    const int Is[3] = {max(I - 1, 0), I, min(I + 1, NX - 1)};
    const int Js[3] = {max(J - 1, 0), J, min(J + 1, NY - 1)};
    const int Ks[3] = {max(K - 1, 0), K, min(K + 1, NZ - 1)};
    const size_t sxy = (size_t)nx * ny, c0 = (size_t)(2 * K) * sxy + (size_t)(2 * J) * nx + 2 * I;
    if (!(MG_CK(((long long)Ks[0] * NY + Js[0]) * NX + Is[0], ((long long)Ks[2] * NY + Js[2]) * NX + Is[2],
                (long long)NX * NY * NZ, CK_PROLONG) &&
          MG_CK(c0, c0 + sxy + nx + 1, (long long)sxy * nz, CK_PROLONG)))
        return;
    T pv[2][2], dv[2][2];
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            const size_t c = c0 + dz * sxy + (size_t)dy * nx + (dz ^ dy);
            pv[dz][dy] = p[SPLIT ? c >> 1 : c];
            dv[dz][dy] = dinv[c];
        }
    T e[3][3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int bb = 0; bb < 3; bb++)
#pragma unroll
            for (int d = 0; d < 3; d++) e[a][bb][d] = ec[((size_t)Ks[a] * NY + Js[bb]) * NX + Is[d]];
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            const size_t c = c0 + dz * sxy + (size_t)dy * nx + (dz ^ dy);
            const T corr = prolong_child<T>(dz, dy, dz ^ dy, [&](int a, int bb, int d) { return e[a][bb][d]; });
            if (!zero_bits(dv[dz][dy])) p[SPLIT ? c >> 1 : c] = pv[dz][dy] + corr;
        }
}

template <typename T, bool SPLIT>
__global__ void k_prolong_red(int nx, int ny, int nz, const T *__restrict__ ec, const T *__restrict__ dinv,
                              T *__restrict__ p)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y, K = blockIdx.z;
    if (I >= nx / 2 || J >= ny / 2) return;
    prolong_red<T, SPLIT>(I, J, K, nx, ny, nz, ec, dinv, p);
}

// prolong_red on the colour-split finest FP32 level with nx % 8 == 0, two coarse cells along x per
// thread: the 3 x 3 coarse rows are loaded as a pair and the value on either side (27 loads for two
// coarse cells), the red children as pairs of slots.  Rows with a record (rows[r * stride] != 0)
// have no dead cell, the others read dinv.
__global__ void k_prolong_red4(int nx, int ny, int nz, const float *__restrict__ ec, const float *__restrict__ dinv,
                               float *__restrict__ p, const float *__restrict__ rows, int stride)
{
    const int NX = nx / 2, NY = ny / 2, NZ = nz / 2;
    const int I = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x), J = blockIdx.y * blockDim.y + threadIdx.y;
    const int zb = blockIdx.z;
    const int K = (NZ & 3) ? zb : (zb & 3) * (NZ / 4) + (zb >> 2);  // plane quarters interleaved
    if (I >= NX || J >= NY) return;
    const size_t hx = nx / 2, hxy = (size_t)nx * ny / 2;
    const size_t m0 = (size_t)(2 * K) * hxy + (size_t)(2 * J) * hx + I;
    const int Js[3] = {max(J - 1, 0), J, min(J + 1, NY - 1)};
    const int Ks[3] = {max(K - 1, 0), K, min(K + 1, NZ - 1)};
    const int il = max(I - 1, 0), ih = min(I + 2, NX - 1);
    if (!(MG_CK(m0, m0 + hxy + hx + 1, (long long)hxy * nz, CK_PROLONG) &&
          MG_CK(((long long)Ks[0] * NY + Js[0]) * NX + il, ((long long)Ks[2] * NY + Js[2]) * NX + ih,
                (long long)NX * NY * NZ, CK_PROLONG)))
        return;
    float2 pv[2][2];
    float rec[2][2];
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            pv[dz][dy] = *reinterpret_cast<const float2 *>(p + m0 + dz * hxy + dy * hx);
            rec[dz][dy] = rows[((size_t)(2 * K + dz) * ny + 2 * J + dy) * stride];
        }
    float e[3][3][4];  // [K][J][I - 1 .. I + 2]
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int bb = 0; bb < 3; bb++) {
            const float *r = ec + ((size_t)Ks[a] * NY + Js[bb]) * NX;
            const float2 mid = *reinterpret_cast<const float2 *>(r + I);
            e[a][bb][0] = r[il];
            e[a][bb][1] = mid.x;
            e[a][bb][2] = mid.y;
            e[a][bb][3] = r[ih];
        }
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            const size_t m = m0 + dz * hxy + dy * hx;
            float2 v = pv[dz][dy];
            const float c0 = prolong_child<float>(dz, dy, dz ^ dy, [&](int a, int bb, int d) { return e[a][bb][d]; });
            const float c1 = prolong_child<float>(dz, dy, dz ^ dy, [&](int a, int bb, int d) { return e[a][bb][d + 1]; });
            bool l0 = true, l1 = true;
            if (rec[dz][dy] == 0.f) {
                l0 = !zero_bits(dinv[2 * m + (dz ^ dy)]);
                l1 = !zero_bits(dinv[2 * m + 2 + (dz ^ dy)]);
            }
            if (l0) v.x += c0;
            if (l1) v.y += c1;
            *reinterpret_cast<float2 *>(p + m) = v;
        }
}

// The prolongation and the black pass after it in one launch (FP32 levels below the finest).  The red
// pass that follows replaces every red value from the black ones without reading it, so the corrected red
// values are needed by this black pass alone: each black cell corrects its six red neighbours itself and no
// red value is written, so no thread reads what another writes.  Along an axis the neighbour within
// the black cell's coarse cell o is the child on the far side (its other coarse cell q), the one outside the near
// child of the coarse cell t, so 20 of the 3 x 3 x 3 coarse values serve all six.  A dead red cell is
// corrected too: its faces are 0.  Same operations in the same order as k_prolong_red and k_smooth.
// These levels are bound by launches and latency (four black cells per thread, a coarse cell's, was no
// faster than the two launches: too few warps): 32^3 3.1 us (5.4 in two launches), 64^3 4.2 us (6.1).  Every red value is
// corrected six times, so larger levels keep the two launches: 128^3 15.6 us against 12.4, and of 80^3
// or 96 x 80 x 80 the coarse-grid correction is 1 to 2 us slower (kUpCells lies at 64^3).
__global__ void k_prolong_black(int nx, int ny, int nz, float h2, LevelArrays<float> L, const float *__restrict__ b,
                                const float *__restrict__ ec, float *__restrict__ p)
{
    const int j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + 1) & 1);
    if (i >= nx || j >= ny) return;
    const int NX = nx / 2, NY = ny / 2, NZ = nz / 2;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    // coarse indices along an axis: 0 the cell's own, 1 on its near side, 2 on its far side
    auto index = [](int v, int n, int out[3]) {
        const int o = v >> 1, lo = max(o - 1, 0), hi = min(o + 1, n - 1);
        out[0] = o;
        out[1] = (v & 1) ? hi : lo;
        out[2] = (v & 1) ? lo : hi;
    };
    int X[3], Y[3], Z[3];
    index(i, NX, X);
    index(j, NY, Y);
    index(k, NZ, Z);
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_PROLONG) ||
        !MG_CK(((long long)min(Z[1], Z[2]) * NY + min(Y[1], Y[2])) * NX + min(X[1], X[2]),
               ((long long)max(Z[1], Z[2]) * NY + max(Y[1], Y[2])) * NX + max(X[1], X[2]), (long long)NX * NY * NZ,
               CK_PROLONG))
        return;
    const bool xl = i > 0, xh = i < nx - 1, yl = j > 0, yh = j < ny - 1, zl = k > 0, zh = k < nz - 1;
    const float pxl = xl ? p[c - 1] : 0.f, pxh = xh ? p[c + 1] : 0.f;
    const float pyl = yl ? p[c - nx] : 0.f, pyh = yh ? p[c + nx] : 0.f;
    const float pzl = zl ? p[c - sxy] : 0.f, pzh = zh ? p[c + sxy] : 0.f;
    const float bc = b[c], d = L.dinv[c], bxl = L.bx[c], byl = L.by[c], bzl = L.bz[c];
    const float bxh = xh ? L.bx[c + 1] : 0.f, byh = yh ? L.by[c + nx] : 0.f, bzh = zh ? L.bz[c + sxy] : 0.f;
    float e[3][3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int bb = 0; bb < 3; bb++)
#pragma unroll
            for (int m = 0; m < 3; m++)
                if ((a == 2) + (bb == 2) + (m == 2) <= 1) e[a][bb][m] = ec[((size_t)Z[a] * NY + Y[bb]) * NX + X[m]];
    // the correction of a neighbour along `axis` (0 x, 1 y, 2 z), inside the coarse cell or not
    auto corr = [&](int axis, bool inside) {
        const float w[2] = {0.75f, 0.25f};
        float s = 0.f;
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int bb = 0; bb < 2; bb++)
#pragma unroll
                for (int m = 0; m < 2; m++) {
                    const int v = axis == 0 ? m : (axis == 1 ? bb : a), u = inside ? 2 * v : 1 - v;  // (o, q) or (t, o)
                    s = fmaf(w[a] * w[bb] * w[m], e[axis == 2 ? u : a][axis == 1 ? u : bb][axis == 0 ? u : m], s);
                }
        return s;
    };
    const float xi = corr(0, true), xo = corr(0, false), yi = corr(1, true), yo = corr(1, false), zi = corr(2, true),
                zo = corr(2, false);
    const bool ox = i & 1, oy = j & 1, oz = k & 1;  // the inside neighbour is the lower one
    float s = 0.f;
    if (xl) s = fmaf(bxl, pxl + (ox ? xi : xo), s);
    if (xh) s = fmaf(bxh, pxh + (ox ? xo : xi), s);
    if (yl) s = fmaf(byl, pyl + (oy ? yi : yo), s);
    if (yh) s = fmaf(byh, pyh + (oy ? yo : yi), s);
    if (zl) s = fmaf(bzl, pzl + (oz ? zi : zo), s);
    if (zh) s = fmaf(bzh, pzh + (oz ? zo : zi), s);
    p[c] = d * fmaf(-h2, bc, s);
}

// ---------------------------------------------------------------------------
// Fused red-black sweep: both colours in one pass over HBM.
//
// The CTA owns a TX x TY tile of columns and a chunk of z-planes and marches up
// the chunk with a two-plane wavefront: at step s it updates the FIRST colour on
// plane s, then the SECOND colour on plane s-1 (whose first-colour neighbours on
// planes s-2, s-1 and s are final by then).  It reads the iterate from p_old and
// writes every cell of its tile to p_new, so CTAs never see each other's writes:
// the first colour on a one-cell ring around the tile (and on one plane below
// and above the chunk) is recomputed from p_old, exactly as the neighbouring CTA
// computes it.  Per cell the arithmetic is that of k_smooth, so the result is
// bit-identical to two colour passes.  Threads: one per column of the tile plus a
// two-cell halo; ring 2 only loads, ring 1 also updates the first colour.
// Shared memory holds three rotating planes of (p, bx, by): the x+ and y+ face
// coefficients of a cell are its neighbour's low faces.
// ---------------------------------------------------------------------------
template <typename T, bool POW2, int TX, int TY>
__global__ void __launch_bounds__((TX + 4) * (TY + 4))
k_rb_sweep(int nx, int ny, int nz, int zc, GsScale<T> gs, LevelArrays<T> L, const T *__restrict__ b,
           const T *__restrict__ p_old, T *__restrict__ p_new, int first)
{
    constexpr int W = TX + 4, H = TY + 4;
    __shared__ T sp[3][H][W];
    __shared__ T sbx[3][H][W];
    __shared__ T sby[3][H][W];
    const int lx = threadIdx.x % W, ly = threadIdx.x / W;
    const int i = blockIdx.x * TX + lx - 2, j = blockIdx.y * TY + ly - 2;
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
    const bool dom = (i >= 0 && i < nx && j >= 0 && j < ny);
    const bool ring1 = dom && lx >= 1 && lx <= TX + 2 && ly >= 1 && ly <= TY + 2;
    const bool inner = dom && lx >= 2 && lx < TX + 2 && ly >= 2 && ly < TY + 2;
    const size_t sxy = (size_t)nx * ny;
    const size_t col = dom ? (size_t)j * nx + i : 0;
    const int second = first ^ 1;
    const bool xlo = i > 0, xhi = i < nx - 1, ylo = j > 0, yhi = j < ny - 1;

    // column registers: iterate at planes s-2 .. s+1, coefficients at planes s-1 .. s+1
    T q_m2 = T(0), q_m1 = T(0), q_0 = T(0), q_p1 = T(0);
    T bx_m1 = T(0), by_m1 = T(0), bz_m1 = T(0), di_m1 = T(0), b_m1 = T(0);
    T bx_0 = T(0), by_0 = T(0), bz_0 = T(0), di_0 = T(0), b_0 = T(0);
    T bx_p1 = T(0), by_p1 = T(0), bz_p1 = T(0), di_p1 = T(0), b_p1 = T(0);

    auto load_plane = [&](int z, T &q, T &bxv, T &byv, T &bzv, T &div, T &bv) {
        q = bxv = byv = bzv = div = bv = T(0);
        if (!dom || z < 0 || z >= nz) return;
        const size_t c = (size_t)z * sxy + col;
        q = p_old[c];
        bxv = L.bx[c];
        byv = L.by[c];
        if (ring1) {
            bzv = L.bz[c];
            if (sizeof(T) == 8) div = L.dinv[c];
            bv = b[c];
        }
    };
    // prologue: planes z0-2 (iterate only) and z0-1
    {
        T t0, t1, t2, t3, t4;
        load_plane(z0 - 2, q_m1, t0, t1, t2, t3, t4);
        load_plane(z0 - 1, q_0, bx_0, by_0, bz_0, di_0, b_0);
    }
    int cur = 0;
    for (int s = z0 - 1; s <= z1; s++) {
        const int prv = (cur + 2) % 3;  // buffer of plane s-1
        load_plane(s + 1, q_p1, bx_p1, by_p1, bz_p1, di_p1, b_p1);
        sp[cur][ly][lx] = q_0;
        sbx[cur][ly][lx] = bx_0;
        sby[cur][ly][lx] = by_0;
        __syncthreads();
        // first colour on plane s
        if (ring1 && s >= 0 && s < nz && ((i + j + s) & 1) == first) {
            const T bxh = xhi ? sbx[cur][ly][lx + 1] : T(0), byh = yhi ? sby[cur][ly + 1][lx] : T(0);
            const T bzh = (s < nz - 1) ? bz_p1 : T(0);
            T acc = gs_start_of<POW2>(b_0, gs);
            if (xlo) acc = gs_add(bx_0, sp[cur][ly][lx - 1], acc);
            if (xhi) acc = gs_add(bxh, sp[cur][ly][lx + 1], acc);
            if (ylo) acc = gs_add(by_0, sp[cur][ly - 1][lx], acc);
            if (yhi) acc = gs_add(byh, sp[cur][ly + 1][lx], acc);
            if (s > 0) acc = gs_add(bz_0, q_m1, acc);
            if (s < nz - 1) acc = gs_add(bz_p1, q_p1, acc);
            q_0 = gs_update(acc, b_0, inv_diag<T>(di_0, bx_0, bxh, by_0, byh, bz_0, bzh), gs);
            sp[cur][ly][lx] = q_0;
        }
        __syncthreads();
        // second colour on plane s-1, then plane s-1 is final for this tile
        const int z = s - 1;
        if (inner && z >= z0 && z < z1) {
            if (((i + j + z) & 1) == second) {
                const T bxh = xhi ? sbx[prv][ly][lx + 1] : T(0), byh = yhi ? sby[prv][ly + 1][lx] : T(0);
                const T bzh = (z < nz - 1) ? bz_0 : T(0);
                T acc = gs_start_of<POW2>(b_m1, gs);
                if (xlo) acc = gs_add(bx_m1, sp[prv][ly][lx - 1], acc);
                if (xhi) acc = gs_add(bxh, sp[prv][ly][lx + 1], acc);
                if (ylo) acc = gs_add(by_m1, sp[prv][ly - 1][lx], acc);
                if (yhi) acc = gs_add(byh, sp[prv][ly + 1][lx], acc);
                if (z > 0) acc = gs_add(bz_m1, q_m2, acc);
                if (z < nz - 1) acc = gs_add(bz_0, q_0, acc);
                q_m1 = gs_update(acc, b_m1, inv_diag<T>(di_m1, bx_m1, bxh, by_m1, byh, bz_m1, bzh), gs);
            }
            p_new[(size_t)z * sxy + col] = q_m1;
        }
        q_m2 = q_m1; q_m1 = q_0; q_0 = q_p1;
        bx_m1 = bx_0; by_m1 = by_0; bz_m1 = bz_0; di_m1 = di_0; b_m1 = b_0;
        bx_0 = bx_p1; by_0 = by_p1; bz_0 = bz_p1; di_0 = di_p1; b_0 = b_p1;
        cur = (cur + 1) % 3;
    }
}

// Exact coarsest-grid solve e = M b with the dense minimum-norm inverse M (FP64 always).
// One warp per row (coalesced row reads, shuffle reduction); b staged in shared memory.
template <typename T>
__global__ void k_coarse_solve(int n, const double *__restrict__ M, const T *__restrict__ b, T *__restrict__ e)
{
    extern __shared__ double sb[];
    for (int i = threadIdx.x; i < n; i += blockDim.x) sb[i] = (double)b[i];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    for (int r = blockIdx.x * warps + warp; r < n; r += gridDim.x * warps) {
        if (!MG_CK((long long)r * n, (long long)r * n + n - 1, (long long)n * n, CK_COARSE_SOLVE)) continue;
        const double *row = M + (size_t)r * n;
        double s = 0.0;
        for (int q = lane; q < n; q += 32) s = fma(row[q], sb[q], s);
        s = warp_sum(s);
        if (lane == 0) e[r] = (T)s;
    }
}

// ---------------------------------------------------------------------------
// Coarse tail: one thread-block cluster runs all of a V-cycle from a level of some 10^4 cells down, the
// exact solve on the coarsest grid included, in one launch.  A pass over such a level is far shorter
// than a launch: as a graph of launches each of its ~10 passes took 1.5 us, and in one CTA, as the
// tail ran before, a level of 16^3 cells was bound by that SM's instruction issue (FP32) or FP64 unit.
// Here the levels live in the shared memory of the cluster's CTAs:
//   * a level's planes are dealt out in slabs of P = ceil(nz / CTAs), stored colour by colour, so
//     that a pass reads consecutive words;
//   * a thread keeps the coefficients of its cells (at most kTailCells of each colour) in registers
//     for all sweeps of a level, and a pass is six loads of the other colour, the update and a store;
//   * the planes beside the slab are read from the neighbour CTA's shared memory (distributed shared
//     memory, ~440 cycles), and a pass ends with a cluster barrier (~500 cycles): these two are what
//     a pass takes, whatever the level;
//   * restriction and prolongation read the planes they need wherever these are;
//   * every CTA gathers the coarsest right-hand side and computes some of the inverse's rows.
// A neighbour beyond a wall is another cell of that colour, or a zero of the row of zeros before and after each
// colour's cells, with a zero coefficient: an update has no wall tests, the product is a zero.
// The arithmetic of a cell is that of the kernels of the larger levels, in their order, so the
// results are those of a launch per pass.  What it measures: launch_tail.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const __grid_constant__ TailArgs<T> a)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *const sm = reinterpret_cast<T *>(smem_raw);
    const int rank = (int)cl.block_rank(), ncta = (int)cl.num_blocks();
    const int tid = threadIdx.x, nthr = kTailThreads, top = a.nlev - 1;

    // the slabs of every level: p = 0, faces and inverse diagonals, the top level's b
    for (int l = 0; l < top; l++) {
        const TailLevel<T> &v = a.lev[l];
        const int z0 = rank * v.P, nk = max(0, min(v.nz - z0, v.P));
        const unsigned hx = v.nx / 2, hxy = hx * v.ny, H = v.P * hxy + hx, HZ = H + hxy;
        const unsigned total = (unsigned)nk * 2 * hxy, plane = 2 * hxy;
        const size_t g0 = (size_t)z0 * plane;
        for (unsigned c = tid; c < 2 * H + hx; c += nthr) sm[v.op - hx + c] = T(0);
        for (unsigned c = tid; c < total + plane; c += nthr) {  // the plane above for its low z-faces
            const bool own = c < total;
            if (!own && (nk == 0 || z0 + nk >= v.nz)) break;
            if (!MG_CK(g0 + c, g0 + c, (long long)plane * v.nz, CK_TAIL)) break;
            const unsigned row = fdiv(c, v.fnx), i = c - row * v.nx, kl = fdiv(row, v.fny), j = row - kl * v.ny;
            const unsigned q = (i + j + kl + z0) & 1u, m = c >> 1;
            sm[v.oz + q * HZ + m] = v.L.bz[g0 + c];
            if (own) {
                sm[v.ox + q * H + m] = v.L.bx[g0 + c];
                sm[v.oy + q * H + m] = v.L.by[g0 + c];
                sm[v.od + q * H + m] = v.L.dinv[g0 + c];
                if (l == 0) sm[v.ob + q * H + m] = v.L.b[g0 + c];
            }
        }
    }
    cl.sync();

    // n sweeps on level v, colour `first` first; zero: the level's p is zero (a first red pass reads
    // no neighbour)
    auto sweeps = [&](const TailLevel<T> &v, int n, unsigned first, bool zero) {
        if (n == 0) return;
        const int z0 = rank * v.P, nk = max(0, min(v.nz - z0, v.P));
        const unsigned hx = v.nx / 2, hxy = hx * v.ny, H = v.P * hxy + hx, HZ = H + hxy, total = nk * hxy;
        T *const p = sm + v.op;
        const T *const below = rank > 0 ? cl.map_shared_rank(p, rank - 1) + (v.P - 1) * hxy : p;
        const T *const above = rank + 1 < ncta ? cl.map_shared_rank(p, rank + 1) : p;
        T fxl[kTailCells][2], fxh[kTailCells][2], fyl[kTailCells][2], fyh[kTailCells][2], fzl[kTailCells][2],
            fzh[kTailCells][2], fd[kTailCells][2], fb[kTailCells][2];
        const GsScale<T> gs{v.h2, v.sh2};
        const T *zl[kTailCells], *zh[kTailCells];  // the planes below and above (colour 0)
        unsigned odd[kTailCells];                   // (j + k) & 1
#pragma unroll
        for (int e = 0; e < kTailCells; e++) {
            const unsigned t = tid + e * nthr;
            odd[e] = 0;
            zl[e] = zh[e] = p;
            if (t >= total) continue;
            const unsigned row = fdiv(t, v.fhx), u = t - row * hx, kl = fdiv(row, v.fny), j = row - kl * v.ny;
            const unsigned k = z0 + kl, t0 = t - kl * hxy;
            odd[e] = (j + k) & 1u;
            zl[e] = k == 0 ? p + t : (kl > 0 ? p + t - hxy : below + t0);
            zh[e] = k + 1 == (unsigned)v.nz ? p + t : (kl + 1 < (unsigned)v.P ? p + t + hxy : above + t0);
#pragma unroll
            for (unsigned q = 0; q < 2; q++) {
                const unsigned off = odd[e] ^ q, i = 2 * u + off, o = q ^ 1u;
                fxl[e][q] = i > 0 ? sm[v.ox + q * H + t] : T(0);
                fxh[e][q] = i + 1 < (unsigned)v.nx ? sm[v.ox + o * H + t + off] : T(0);
                fyl[e][q] = j > 0 ? sm[v.oy + q * H + t] : T(0);
                fyh[e][q] = j + 1 < (unsigned)v.ny ? sm[v.oy + o * H + t + hx] : T(0);
                fzl[e][q] = k > 0 ? sm[v.oz + q * HZ + t] : T(0);
                fzh[e][q] = k + 1 < (unsigned)v.nz ? sm[v.oz + o * HZ + t + hxy] : T(0);
                fd[e][q] = sm[v.od + q * H + t];
                fb[e][q] = sm[v.ob + q * H + t];
            }
        }
        auto pass = [&](auto colour) {
            constexpr unsigned q = decltype(colour)::value, o = q ^ 1u;
#pragma unroll
            for (int e = 0; e < kTailCells; e++) {
                const unsigned t = tid + e * nthr;
                if (t >= total) break;
                T s = gs_start(fb[e][q], gs);
                if (!zero) {
                    const T *const ot = p + o * H + t, *const ox = ot + (odd[e] ^ q);
                    s = gs_add(fxl[e][q], ox[-1], s);
                    s = gs_add(fxh[e][q], ox[0], s);
                    s = gs_add(fyl[e][q], *(ot - hx), s);
                    s = gs_add(fyh[e][q], *(ot + hx), s);
                    s = gs_add(fzl[e][q], zl[e][o * H], s);
                    s = gs_add(fzh[e][q], zh[e][o * H], s);
                }
                p[q * H + t] = gs_update(s, fb[e][q], fd[e][q], gs);
            }
            zero = false;
            cl.sync();
        };
        for (int it = 0; it < n; it++) {
            if (first == 0) {
                pass(std::integral_constant<unsigned, 0>{});
                pass(std::integral_constant<unsigned, 1>{});
            } else {
                pass(std::integral_constant<unsigned, 1>{});
                pass(std::integral_constant<unsigned, 0>{});
            }
        }
    };
    // base of plane k of an array at offset o of level v, in the shared memory that holds it
    auto plane_of = [&](const TailLevel<T> &v, unsigned o, unsigned k, unsigned stride) {
        const unsigned r = fdiv(k, v.fP);
        return cl.map_shared_rank(sm + o, r) + (k - r * v.P) * stride;
    };
    // where cell (I, J) of a plane of level v sits (the coarsest level is kept in natural order)
    auto slot = [&](const TailLevel<T> &v, bool last, unsigned I, unsigned J, unsigned K) {
        const unsigned hx = v.nx / 2;
        return last ? J * v.nx + I : ((I + J + K) & 1u) * (v.P * hx * v.ny + hx) + J * hx + (I >> 1);
    };

    // descent: nu1 sweeps red then black, restriction (restrict_box)
    for (int l = 0; l < top; l++) {
        const TailLevel<T> &v = a.lev[l], &w = a.lev[l + 1];
        sweeps(v, a.nu1, 0, true);
        const bool last = l + 1 == top;
        const unsigned hx = v.nx / 2, hxy = hx * v.ny, H = v.P * hxy + hx, HZ = H + hxy;
        const int Z0 = rank * w.P, nK = max(0, min(w.nz - Z0, w.P));
        const unsigned NX = w.nx, NY = w.ny, total = (unsigned)nK * NX * NY, stride_w = last ? NX * NY : NX / 2 * NY;
        for (unsigned t = tid; t < total; t += nthr) {
            const unsigned row = fdiv(t, w.fnx), I = t - row * NX, Kl = fdiv(row, w.fny), J = row - Kl * NY;
            const unsigned K = Z0 + Kl;
            T s = T(0), sb = T(0);
#pragma unroll
            for (unsigned dk = 0; dk < 2; dk++) {
                const unsigned k = 2 * K + dk;
                const T *const p = plane_of(v, v.op, k, hxy), *const b = plane_of(v, v.ob, k, hxy);
                const T *const X = plane_of(v, v.ox, k, hxy), *const Y = plane_of(v, v.oy, k, hxy);
                const T *const Z = plane_of(v, v.oz, k, hxy) + (dk ? hxy : 0);
                const bool hz = dk ? k + 1 < (unsigned)v.nz : k > 0;
                const T *const pz = hz ? plane_of(v, v.op, dk ? k + 1 : k - 1, hxy) : p;
#pragma unroll
                for (unsigned dj = 0; dj < 2; dj++) {
                    const unsigned j = 2 * J + dj, q = dj ^ dk, e = j * hx + I;  // q: colour of the even cell
                    const unsigned E = q * H + e, O = (q ^ 1u) * H + e;
                    const T pe = p[E], po = p[O];
                    if (I > 0) s = fma(X[E], p[O - 1] - pe, s);
                    if (I + 1 < hx) s = fma(X[E + 1], p[E + 1] - po, s);
                    if (dj ? j + 1 < (unsigned)v.ny : j > 0) {
                        const T fe = dj ? Y[O + hx] : Y[E], fo = dj ? Y[E + hx] : Y[O];
                        s = fma(fe, (dj ? p[O + hx] : p[O - hx]) - pe, s);
                        s = fma(fo, (dj ? p[E + hx] : p[E - hx]) - po, s);
                    }
                    if (hz) {
                        const unsigned ZE = q * HZ + e, ZO = (q ^ 1u) * HZ + e;
                        s = fma(Z[dk ? ZO : ZE], pz[O] - pe, s);
                        s = fma(Z[dk ? ZE : ZO], pz[E] - po, s);
                    }
                    sb += b[E] + b[O];
                }
            }
            sm[w.ob + Kl * stride_w + slot(w, last, I, J, K)] = T(0.125) * fma(-s, v.ih2, sb);
        }
        cl.sync();
    }

    // the coarsest grid: e = M b, a row per warp (k_coarse_solve)
    {
        const TailLevel<T> &w = a.lev[top];
        const unsigned NXY = w.nx * w.ny, n = NXY * w.nz;
        double *const sb = reinterpret_cast<double *>(smem_raw + a.sb_bytes);
        for (unsigned t = tid; t < n; t += nthr) {
            const unsigned K = fdiv(fdiv(t, w.fnx), w.fny);
            sb[t] = (double)plane_of(w, w.ob, K, NXY)[t - K * NXY];
        }
        __syncthreads();
        const unsigned warps = nthr / 32, lane = tid & 31;
        for (unsigned r = rank * warps + tid / 32; r < n; r += ncta * warps) {
            if (!MG_CK((long long)r * n, (long long)r * n + n - 1, (long long)n * n, CK_COARSE_SOLVE)) continue;
            const double *row = a.M + (size_t)r * n;
            double s = 0.0;
            for (unsigned q = lane; q < n; q += 32) s = fma(row[q], sb[q], s);
            s = warp_sum(s);
            const unsigned K = fdiv(fdiv(r, w.fnx), w.fny);
            if (lane == 0) plane_of(w, w.op, K, NXY)[r - K * NXY] = (T)s;
        }
        cl.sync();
    }

    // ascent: prolongation (of the red cells alone where a black pass follows), nu2 sweeps black then red
    for (int l = top - 1; l >= 0; l--) {
        const TailLevel<T> &v = a.lev[l], &w = a.lev[l + 1];
        const bool last = l + 1 == top;
        const int z0 = rank * v.P, nk = max(0, min(v.nz - z0, v.P));
        const unsigned hx = v.nx / 2, hxy = hx * v.ny, H = v.P * hxy + hx, total = nk * hxy;
        const unsigned stride_w = last ? w.nx * w.ny : w.nx / 2 * w.ny;
        for (unsigned q = 0; q < (a.nu2 >= 1 ? 1u : 2u); q++)
            for (unsigned t = tid; t < total; t += nthr) {
                const unsigned row = fdiv(t, v.fhx), u = t - row * hx, kl = fdiv(row, v.fny), j = row - kl * v.ny;
                const unsigned k = z0 + kl, i = 2 * u + ((j + k + q) & 1u);
                // parent and the neighbour on the cell's side, clamped at the walls
                auto next = [](unsigned f, int n) {
                    return (f & 1u) ? min((f >> 1) + 1, (unsigned)n - 1) : ((f >> 1) ? (f >> 1) - 1 : 0u);
                };
                const unsigned Ks[2] = {k >> 1, next(k, w.nz)}, Js[2] = {j >> 1, next(j, w.ny)},
                               Is[2] = {i >> 1, next(i, w.nx)};
                const T wt[2] = {T(0.75), T(0.25)};
                T s = T(0);
#pragma unroll
                for (int z = 0; z < 2; z++) {
                    const T *const e = plane_of(w, w.op, Ks[z], stride_w);
#pragma unroll
                    for (int y = 0; y < 2; y++)
#pragma unroll
                        for (int x = 0; x < 2; x++)
                            s = fma(wt[z] * wt[y] * wt[x], e[slot(w, last, Is[x], Js[y], Ks[z])], s);
                }
                if (!zero_bits(sm[v.od + q * H + t])) sm[v.op + q * H + t] += s;
            }
        cl.sync();
        sweeps(v, a.nu2, 1, false);
    }

    // the top level's correction (every remote read of this CTA's memory lies before the last barrier)
    {
        const TailLevel<T> &v = a.lev[0];
        const int z0 = rank * v.P, nk = max(0, min(v.nz - z0, v.P));
        const unsigned hx = v.nx / 2, hxy = hx * v.ny, H = v.P * hxy + hx, total = (unsigned)nk * 2 * hxy;
        const size_t g0 = (size_t)z0 * 2 * hxy;
        for (unsigned c = tid; c < total; c += nthr) {
            const unsigned row = fdiv(c, v.fnx), i = c - row * v.nx, kl = fdiv(row, v.fny), j = row - kl * v.ny;
            if (!MG_CK(g0 + c, g0 + c, (long long)2 * hxy * v.nz, CK_TAIL)) break;
            v.L.p[g0 + c] = sm[v.op + ((i + j + kl + z0) & 1u) * H + (c >> 1)];
        }
    }
}

// ---------------------------------------------------------------------------
// Fine-level reductions (FP64, grid-stride, per-block partial pairs)
// ---------------------------------------------------------------------------
// The passes below read one or two arrays once.  Each thread takes two pairs of cells per iteration, all
// loads issued first: at one cell per iteration their five blocks per SM left HBM at half its rate.
// load(v) returns what pair v (cells 2v and 2v + 1) needs, use(v, that) works on it; the last cell of an odd n is cell(n - 1).
template <typename Load, typename Use, typename Cell>
__device__ __forceinline__ void stream_pairs(unsigned n, Load load, Use use, Cell cell)
{
    const unsigned n2 = n / 2, stride = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
    for (unsigned v = t; v < n2; v += 2 * stride) {
        const unsigned w = v + stride;
        const bool two = w < n2;
        const auto a = load(v), b = load(two ? w : v);
        use(v, a);
        if (two) use(w, b);
    }
    if ((n & 1u) && t == 0) cell(n - 1);
}
struct Pair2 {
    double2 x, y;
};

__global__ void k_count_live(unsigned n, const double *__restrict__ dinv, double *__restrict__ partials, double *dscal)
{
    unsigned a = 0;  // counted in integers: the FP64 unit would bound the pass
    const double2 *d2 = reinterpret_cast<const double2 *>(dinv);
    stream_pairs(
        n, [&](unsigned v) { return d2[v]; },
        [&](unsigned, const double2 &d) { a += (pos_bits(d.x) ? 1u : 0u) + (pos_bits(d.y) ? 1u : 0u); },
        [&](unsigned c) { a += pos_bits(dinv[c]) ? 1u : 0u; });
    reduce_finish(block_sum<kRedThreads>((double)a), 0.0, partials, dscal, S_NLIVE, -1);
}

// sum of v over the live cells into dscal[slot] (the rhs of a solve, or its p)
__global__ void k_sum_live(unsigned n, const double *__restrict__ v, const double *__restrict__ dinv,
                           double *__restrict__ partials, double *dscal, int slot)
{
    double a = 0.0;
    const double2 *v2 = reinterpret_cast<const double2 *>(v), *d2 = reinterpret_cast<const double2 *>(dinv);
    stream_pairs(
        n, [&](unsigned i) { return Pair2{v2[i], d2[i]}; },
        [&](unsigned, const Pair2 &q) {
            a += pos_bits(q.y.x) ? q.x.x : 0.0;
            a += pos_bits(q.y.y) ? q.x.y : 0.0;
        },
        [&](unsigned c) { a += pos_bits(dinv[c]) ? v[c] : 0.0; });
    reduce_finish(block_sum<kRedThreads>(a), 0.0, partials, dscal, slot, -1);
}

// pass 2: b0 = rhs - mean on live cells, 0 elsewhere; partial ||b0||^2
__global__ void k_rhs_center(unsigned n, const double *__restrict__ rhs, const double *__restrict__ dinv,
                             double *__restrict__ b0, double *dscal, double *__restrict__ partials)
{
    const double mean = block_scalar([&] { return dscal[S_SUM_B] / dscal[S_NLIVE]; });
    double a = 0.0;
    const double2 *r2 = reinterpret_cast<const double2 *>(rhs), *d2 = reinterpret_cast<const double2 *>(dinv);
    double2 *b2 = reinterpret_cast<double2 *>(b0);
    auto one = [&](double x, double d) {
        const double v = pos_bits(d) ? x - mean : 0.0;
        a = fma(v, v, a);
        return v;
    };
    stream_pairs(
        n, [&](unsigned i) { return Pair2{r2[i], d2[i]}; },
        [&](unsigned i, const Pair2 &q) {
            const double vx = one(q.x.x, q.y.x), vy = one(q.x.y, q.y.y);
            b2[i] = make_double2(vx, vy);
        },
        [&](unsigned c) { b0[c] = one(rhs[c], dinv[c]); });
    reduce_finish(block_sum<kRedThreads>(a), 0.0, partials, dscal, S_NB2, -1);
}

// ||b - A p||^2; SUM: and the sum of p over the live cells (resid_sums_p)
template <bool SUM>
__global__ void k_resid_norm(int nx, int ny, int nz, double ih2, LevelArrays<double> L,
                             const double *__restrict__ b, const double *__restrict__ p, double *__restrict__ partials,
                             double *dscal, ResidGrid g)
{
    double rr = 0.0, sum = 0.0;
    resid_columns(nx, ny, nz, ih2, L, b, p, g, [&](size_t c, int, double r, double pc) {
        rr = fma(r, r, rr);
        if (SUM && pos_bits(L.dinv[c])) sum += pc;
    });
    block_sum2<kRedThreads, SUM>(rr, sum);
    reduce_finish(rr, sum, partials, dscal, S_RR, SUM ? S_SUM_P : -1);
}

// p -= mean of p over live cells (mean = dscal[S_SUM_P] / dscal[S_NLIVE]); dead cells 0
__global__ void k_sub_mean_p(unsigned n, const double *__restrict__ dinv, double *__restrict__ p,
                             const double *__restrict__ dscal)
{
    const double mean = block_scalar([&] { return dscal[S_SUM_P] / dscal[S_NLIVE]; });
    const double2 *d2 = reinterpret_cast<const double2 *>(dinv);
    double2 *p2 = reinterpret_cast<double2 *>(p);
    auto one = [&](double x, double d) { return pos_bits(d) ? x - mean : 0.0; };
    stream_pairs(
        n, [&](unsigned i) { return Pair2{p2[i], d2[i]}; },
        [&](unsigned i, const Pair2 &q) { p2[i] = make_double2(one(q.x.x, q.y.x), one(q.x.y, q.y.y)); },
        [&](unsigned c) { p[c] = one(p[c], dinv[c]); });
}

// Mixed refinement: r = b - A p in FP64, stored as FP32 r / scale_in; partial ||r||^2.
template <bool SUM>
__global__ void k_resid_cast(int nx, int ny, int nz, double ih2, LevelArrays<double> L,
                             const double *__restrict__ b, const double *__restrict__ p, float *__restrict__ r32,
                             double *dscal, int scale_in, int scale_out, double *__restrict__ partials, size_t half,
                             ResidGrid g)
{
    const double inv_scale = block_scalar([&] { return 1.0 / dscal[scale_in]; });
    double rr = 0.0, sum = 0.0;
    resid_columns(nx, ny, nz, ih2, L, b, p, g, [&](size_t c, int q, double r, double pc) {
        rr = fma(r, r, rr);
        if (SUM && pos_bits(L.dinv[c])) sum += pc;
        const size_t slot = half ? split_slot(c, q, half) : c;
        if (MG_CK(slot, slot, (long long)nx * ny * nz, CK_SPLIT_SLOT)) r32[slot] = narrow(r * inv_scale);
    });
    block_sum2<kRedThreads, SUM>(rr, sum);
    // the last block also sets the next scale: the RMS of this residual over the live cells (1 if 0)
    if (reduce_finish(rr, sum, partials, dscal, S_RR, SUM ? S_SUM_P : -1) && threadIdx.x == 0 && scale_out >= 0) {
        const double rms = sqrt(dscal[S_RR] / dscal[S_NLIVE]);
        dscal[scale_out] = (rms > 0.0 && isfinite(rms)) ? rms : 1.0;
    }
}

__global__ void k_scale_from_nb2(double *dscal, int slot)
{
    const double rms = sqrt(dscal[S_NB2] / dscal[S_NLIVE]);
    dscal[slot] = (rms > 0.0 && isfinite(rms)) ? rms : 1.0;
}

// p += scale * e32 (the FP32 cycle leaves e32 = 0 on dead cells, so no mask is read); e32 in
// the layout (half, nx, ny)
__global__ void k_accumulate(unsigned n, const float *__restrict__ e32, double *__restrict__ p,
                             const double *__restrict__ dscal, int scale_slot, Split sp)
{
    const double s = dscal[scale_slot];
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        const size_t e = sp.half ? split_slot(idx, row_parity(idx, sp), sp.half) : idx;
        if (!MG_CK(e, e, (long long)n, CK_SPLIT_SLOT)) continue;
        p[idx] = fma(s, widen(e32[e]), p[idx]);
    }
}

// The FP32 copy of one level: the narrowed faces (natural layout; on the finest level with a
// colour-split layout, also in that layout, sf != null) and 1/sum of the narrowed faces, summed
// in k_diag_inv's order with its divisor memo (so the value k_diag_inv gives on the narrowed
// faces), from one read of the FP64 faces.  Grid and runs as k_diag_inv.
__global__ void k_level_f32(int nx, int ny, int nz, int run, const double *__restrict__ bx, const double *__restrict__ by,
                            const double *__restrict__ bz, LevelArrays<float> out, LevelArrays<float> sf,
                            size_t half)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= nx) return;
    const int k0 = blockIdx.z * run, k1 = min(k0 + run, nz);
    const size_t sxy = (size_t)nx * ny;
    float s_last = 1.0f, q_last = 1.0f;
    size_t c = (size_t)k0 * sxy + (size_t)j * nx + i;
    float bz_lo = narrow(bz[c]);
    // a cell's loads at once; the next cell's issued before this one's stores
    struct In {
        double x0, x1, y0, y1, zh;
    };
    auto load = [&](size_t cc, int kk) {
        In v;
        v.x0 = bx[cc];
        v.x1 = (i < nx - 1) ? bx[cc + 1] : 0.0;
        v.y0 = by[cc];
        v.y1 = (j < ny - 1) ? by[cc + nx] : 0.0;
        v.zh = (kk < nz - 1) ? bz[cc + sxy] : 0.0;
        return v;
    };
    In cur = load(c, k0);
    for (int k = k0; k < k1; k++, c += sxy) {
        const In nxt = k + 1 < k1 ? load(c + sxy, k + 1) : cur;
        const float bz_hi = narrow(cur.zh);
        const float x = narrow(cur.x0), y = narrow(cur.y0);
        out.bx[c] = x;
        out.by[c] = y;
        out.bz[c] = bz_lo;
        if (sf.bx) {
            const size_t e = split_slot(c, (j + k) & 1, half);
            sf.bx[e] = x;
            sf.by[e] = y;
            sf.bz[e] = bz_lo;
        }
        float t = x;
        t += narrow(cur.x1);
        t += y;
        t += narrow(cur.y1);
        t += bz_lo;
        t += bz_hi;
        bz_lo = bz_hi;
        cur = nxt;
        float q = 0.0f;
        if (t > 0.0f) {
            if (!same_bits(t, s_last)) {
                s_last = t;
                q_last = div_call(1.0f, t);
            }
            q = q_last;
        }
        out.dinv[c] = q;
    }
}

// FP64 natural-order field <-> the finest FP32 field in the layout sp (one FP32 V-cycle on a
// caller's FP64 rhs and iterate)
__global__ void k_to_f32_layout(unsigned n, const double *__restrict__ src, float *__restrict__ dst, Split sp)
{
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x)
    {
        const size_t e = sp.half ? split_slot(idx, row_parity(idx, sp), sp.half) : idx;
        if (MG_CK(e, e, (long long)n, CK_SPLIT_SLOT)) dst[e] = narrow(src[idx]);
    }
}
__global__ void k_from_f32_layout(unsigned n, const float *__restrict__ src, double *__restrict__ dst, Split sp)
{
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x)
    {
        const size_t e = sp.half ? split_slot(idx, row_parity(idx, sp), sp.half) : idx;
        if (MG_CK(e, e, (long long)n, CK_SPLIT_SLOT)) dst[idx] = widen(src[e]);
    }
}

// ---------------------------------------------------------------------------
// Projection (Eq. poisson1 right-hand side; Eq. runge1 correction) and adjoint
// ---------------------------------------------------------------------------
__global__ void k_divergence(int nx, int ny, int nz, Scale2 scale, const double *__restrict__ bx,
                             const double *__restrict__ by, const double *__restrict__ bz,
                             const double *__restrict__ ux, const double *__restrict__ uy,
                             const double *__restrict__ uz, double *__restrict__ rhs)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= nx) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_DIVERGENCE)) return;
    // every load first (a velocity's load does not wait for its face's coefficient)
    const bool xh = i < nx - 1, yh = j < ny - 1, zh = k < nz - 1;
    const double bx0 = bx[c], bx1 = xh ? bx[c + 1] : 0.0, by0 = by[c], by1 = yh ? by[c + nx] : 0.0;
    const double bz0 = bz[c], bz1 = zh ? bz[c + sxy] : 0.0;
    const double ux0 = ux[c], ux1 = xh ? ux[c + 1] : 0.0, uy0 = uy[c], uy1 = yh ? uy[c + nx] : 0.0;
    const double uz0 = uz[c], uz1 = zh ? uz[c + sxy] : 0.0;
    double d = pos_bits(bx1) ? zero_plus(ux1) : 0.0;
    if (pos_bits(bx0)) d -= ux0;
    if (pos_bits(by1)) d += uy1;
    if (pos_bits(by0)) d -= uy0;
    if (pos_bits(bz1)) d += uz1;
    if (pos_bits(bz0)) d -= uz0;
    rhs[c] = mul_s2(d, scale);  // scale * d
}

// ---------------------------------------------------------------------------
// Fractional face areas (Body Boundary Conditions section, Eq. integral2).  psi is given at the
// nodes ((nz+1) x (ny+1) x (nx+1), > 0 outside the body).  A face is split into four triangles
// about its centre (psi there = the mean of the four corners), psi is linear on each, and the open
// fraction is the mean of the triangles' fractions where psi > 0; a triangle with one corner f > 0
// and two g1, g2 <= 0 has f^2 / ((f - g1)(f - g2)), one with two corners > 0 and one g <= 0 has
// 1 - g^2 / ((g - f1)(g - f2)).  Each operation rounded separately.
// ---------------------------------------------------------------------------
__device__ double tri_open(double a, double b, double c)
{
    const bool pa = pos_bits(a), pb = pos_bits(b), pc = pos_bits(c);
    const int np = (int)pa + (int)pb + (int)pc;
    if (np == 0) return 0.0;
    if (np == 3) return 1.0;
    if (np == 1) {
        const double f = pa ? a : (pb ? b : c);
        const double g1 = pa ? b : a, g2 = pc ? b : c;
        return div_call(__dmul_rn(f, f), __dmul_rn(__dsub_rn(f, g1), __dsub_rn(f, g2)));
    }
    const double g = !pa ? a : (!pb ? b : c);
    const double f1 = !pa ? b : a, f2 = !pc ? b : c;
    return __dsub_rn(1.0, div_call(__dmul_rn(g, g), __dmul_rn(__dsub_rn(g, f1), __dsub_rn(g, f2))));
}

// corners in cyclic order around the face: f00, f10, f11, f01
__device__ double face_open(double f00, double f10, double f01, double f11)
{
    const double fc = __dmul_rn(__dadd_rn(__dadd_rn(f00, f10), __dadd_rn(f01, f11)), 0.25);
    const double t0 = tri_open(f00, f10, fc), t1 = tri_open(f10, f11, fc);
    const double t2 = tri_open(f11, f01, fc), t3 = tri_open(f01, f00, fc);
    return __dmul_rn(__dadd_rn(__dadd_rn(__dadd_rn(t0, t1), t2), t3), 0.25);
}

// open fractions of the low faces of every cell; wall faces 0
__global__ void k_face_areas(int nx, int ny, int nz, const double *__restrict__ psi, double *__restrict__ ax,
                             double *__restrict__ ay, double *__restrict__ az)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= nx) return;
    const size_t NX = (size_t)nx + 1, NXY = NX * ((size_t)ny + 1);
    auto P = [&](int ii, int jj, int kk) { return psi[(size_t)kk * NXY + (size_t)jj * NX + (size_t)ii]; };
    const size_t c = ((size_t)k * ny + j) * nx + i;
    ax[c] = i == 0 ? 0.0 : face_open(P(i, j, k), P(i, j + 1, k), P(i, j, k + 1), P(i, j + 1, k + 1));
    ay[c] = j == 0 ? 0.0 : face_open(P(i, j, k), P(i + 1, j, k), P(i, j, k + 1), P(i + 1, j, k + 1));
    az[c] = k == 0 ? 0.0 : face_open(P(i, j, k), P(i + 1, j, k), P(i, j + 1, k), P(i + 1, j + 1, k));
}

// Stretched grids: cell widths hx[i], hy[j], hz[k].  Eq. integral2 times the cell volume on the
// index grid (unit spacing): beta_idx = beta / d with d the distance between the two cell centres,
// area = the face's two widths times the open fraction (frac, or 1); walls 0.  Each operation
// rounded separately.
// On small grids one thread per cell, every face divided where it stands: the launch is a round trip to memory and a
// division long (launch_stretched_metrics has the line).
__global__ void k_stretched_metrics_cells(int nx, int ny, int nz, const double *__restrict__ hx,
                                          const double *__restrict__ hy, const double *__restrict__ hz,
                                          LevelArrays<double> beta, LevelArrays<double> frac, LevelArrays<double> bout,
                                          LevelArrays<double> aout)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const size_t c = ((size_t)k * ny + j) * nx + i;
    if (i == 0) {
        bout.bx[c] = 0.0;
        aout.bx[c] = 0.0;
    } else {
        const double d = __dmul_rn(0.5, __dadd_rn(hx[i - 1], hx[i]));
        bout.bx[c] = div_call(beta.bx[c], d);
        aout.bx[c] = __dmul_rn(__dmul_rn(hy[j], hz[k]), frac.bx ? frac.bx[c] : 1.0);
    }
    if (j == 0) {
        bout.by[c] = 0.0;
        aout.by[c] = 0.0;
    } else {
        const double d = __dmul_rn(0.5, __dadd_rn(hy[j - 1], hy[j]));
        bout.by[c] = div_call(beta.by[c], d);
        aout.by[c] = __dmul_rn(__dmul_rn(hx[i], hz[k]), frac.by ? frac.by[c] : 1.0);
    }
    if (k == 0) {
        bout.bz[c] = 0.0;
        aout.bz[c] = 0.0;
    } else {
        const double d = __dmul_rn(0.5, __dadd_rn(hz[k - 1], hz[k]));
        bout.bz[c] = div_call(beta.bz[c], d);
        aout.bz[c] = __dmul_rn(__dmul_rn(hx[i], hy[j]), frac.bz ? frac.bz[c] : 1.0);
    }
}

// On larger grids: bound by the FP64 unit if every face divides (some 42 operations per cell).  Threads walk up z in runs of RUN
// planes: x and y distances are fixed, so a quotient is kept until beta changes; the z distance
// changes with every plane, so the block tabulates the quotients of two values of beta_z for
// its planes (one division of one warp), the ones found at its first cell's bottom and top, and only cells with
// another value divide.  Areas fully open are not multiplied by 1.  192x160x224: 0.461 -> 0.178 ms.
template <int RUN>
__global__ void k_stretched_metrics(int nx, int ny, int nz, const double *__restrict__ hx,
                                    const double *__restrict__ hy, const double *__restrict__ hz,
                                    LevelArrays<double> beta, LevelArrays<double> frac, LevelArrays<double> bout,
                                    LevelArrays<double> aout)
{
    __shared__ double zq[2][RUN], zref[2];
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    const int k0 = blockIdx.z * RUN, k1 = min(k0 + RUN, nz);
    const size_t sxy = (size_t)nx * ny;
    if (t < 2 * RUN) {
        const size_t c0 = (size_t)(blockIdx.y * blockDim.y) * nx + (size_t)blockIdx.x * blockDim.x;  // the block's first cell
        const int m = t / RUN, k = k0 + t % RUN;
        const double r = beta.bz[c0 + (size_t)(m ? k1 - 1 : k0) * sxy];
        if (k > 0 && k < nz) zq[m][t % RUN] = div_call(r, __dmul_rn(0.5, __dadd_rn(hz[k - 1], hz[k])));
        if (t % RUN == 0) zref[m] = r;
    }
    __syncthreads();
    if (i >= nx || j >= ny) return;
    const double wx = hx[i], wy = hy[j], wxy = __dmul_rn(wx, wy);
    const double dx = i ? __dmul_rn(0.5, __dadd_rn(hx[i - 1], wx)) : 1.0;
    const double dy = j ? __dmul_rn(0.5, __dadd_rn(hy[j - 1], wy)) : 1.0;
    const double r0 = zref[0], r1 = zref[1];
    // (0 / d is 0 where the widths are positive; they are not checked)
    double bx_last = 0.0, qx = pos_number(dx) ? 0.0 : div_call(0.0, dx);
    double by_last = 0.0, qy = pos_number(dy) ? 0.0 : div_call(0.0, dy);
    auto area = [&](double w, double f) { return same_bits(f, 1.0) ? w : dmul_call(w, f); };
    size_t c = (size_t)k0 * sxy + (size_t)j * nx + i;
    for (int k = k0; k < k1; k++, c += sxy) {
        const double b0 = beta.bx[c], b1 = beta.by[c], b2 = beta.bz[c], wz = hz[k];
        const double f0 = frac.bx ? frac.bx[c] : 1.0, f1 = frac.by ? frac.by[c] : 1.0, f2 = frac.bz ? frac.bz[c] : 1.0;
        if (!same_bits(b0, bx_last)) {
            bx_last = b0;
            qx = div_call(b0, dx);
        }
        if (!same_bits(b1, by_last)) {
            by_last = b1;
            qy = div_call(b1, dy);
        }
        double qz = 0.0;
        if (k > 0) {
            if (same_bits(b2, r0)) qz = zq[0][k - k0];
            else if (same_bits(b2, r1)) qz = zq[1][k - k0];
            else qz = div_call(b2, dmul_call(0.5, dadd_call(hz[k - 1], wz)));
        }
        bout.bx[c] = i ? qx : 0.0;
        bout.by[c] = j ? qy : 0.0;
        bout.bz[c] = qz;
        aout.bx[c] = i ? area(__dmul_rn(wy, wz), f0) : 0.0;
        aout.by[c] = j ? area(__dmul_rn(wx, wz), f1) : 0.0;
        aout.bz[c] = k ? area(wxy, f2) : 0.0;
    }
}

// ---------------------------------------------------------------------------
// The Runge-Kutta time step (Numerical Time Integration section).  R = the body force, -g on the
// open z-faces (beta_z > 0), 0 elsewhere; each operation rounded separately in the order written.
// ---------------------------------------------------------------------------
// out = (a + b) + dt R   (b null: a + dt R)
__global__ void k_rk_combine(size_t n, LevelArrays<double> a, LevelArrays<double> b, LevelArrays<double> r, double dt,
                             LevelArrays<double> out)
{
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
        const double sx = b.bx ? __dadd_rn(a.bx[c], b.bx[c]) : a.bx[c];
        const double sy = b.by ? __dadd_rn(a.by[c], b.by[c]) : a.by[c];
        const double sz = b.bz ? __dadd_rn(a.bz[c], b.bz[c]) : a.bz[c];
        out.bx[c] = __dadd_rn(sx, __dmul_rn(dt, r.bx[c]));
        out.by[c] = __dadd_rn(sy, __dmul_rn(dt, r.by[c]));
        out.bz[c] = __dadd_rn(sz, __dmul_rn(dt, r.bz[c]));
    }
}

// ---------------------------------------------------------------------------
// Momentum right-hand side R_i of Eq. navi without the pressure gradient and the sub-grid
// stress: R_i = -d/dx_j (u_j u_i) + (1/rho_f)/Re d/dx_j (2 mu S_ij) - delta_i3 g, with mu from
// Eq. density and 1/rho_f the face coefficient.  Second-order central conservative MAC form:
// u_i u_i at the cell centres (mean of the cell's two i-faces), u_j u_i at the edges (means of
// the two j-faces and of the two i-faces meeting there), 2 mu S_ii at the centres, 2 mu S_ij at
// the edges (mu: mean of the four cells around the edge, in cell-index order), each divergence
// the difference of the two values bracketing the face over h.  Free-slip walls: normal velocity
// 0 (the stored wall face, or the unstored high wall), tangential velocity mirrored into the
// ghost row; closed faces get R = 0.  Separately rounded operations in a fixed order.
//
// Two passes.  k_mom_parts computes, once per cell, the quantities every face shares: for each
// axis a the centre flux C_a = U_a^2 (U_a the cell's mean a-velocity) and stress T_a = 2 mu
// dU_a/dx_a, and for each plane (a, b), a < b, at the cell's low edge the flux F_ab = (mean u_b)
// (mean u_a) and the shear S_ab = mu_edge (du_a/dx_b + du_b/dx_a).  k_mom_combine forms each
// open face's R from the values bracketing it.  A face's F_ab and S_ab are the same numbers
// whichever of the four faces at the edge uses them (the product and the sum commute exactly), so
// R is bitwise the per-face evaluation, with a third of its FP64 operations.
//
// Both passes are bound by the FP64 unit, so what is not an addition or a general product stays off it:
// the halvings, doublings and quarterings, and the products with 1/h where h is a power of two (POW2), are exponent shifts
// on the integer pipe; a cell's viscosity is formed once per block (shared memory) instead of by each of the
// seven cells that use it; the terms a call leaves out (CONV, VISC) are not formed, their share of R
// being a zero.  FP64 operations per cell: about 85 (106 where h is no power of two), 134 with all of that on the
// FP64 unit.  At 256^3: 2.79 ms (4.23 ms), convective terms alone 1.03 ms, viscous alone 1.84 ms, gravity alone
// 0.08 ms (4.23 ms each); 251x190x133 1.35 ms (1.64 ms).
// ---------------------------------------------------------------------------
struct MomArgs {
    int nx, ny, nz;
    Scale2 ih;
    double mu_air, dmu, inv_re, g;
    const double *phi;
    LevelArrays<double> beta, u, r;
    double *w;  // 12 arrays of n: C_x, C_y, C_z, T_x, T_y, T_z, F_xy, F_xz, F_yz, S_xy, S_xz, S_yz
};

__device__ __forceinline__ int clamp_idx(int v, int hi) { return v < 0 ? 0 : (v > hi ? hi : v); }

// x / h as the product with 1/h
template <bool POW2>
__device__ __forceinline__ double mom_ih(const MomArgs &m, double x)
{
    return POW2 ? mul_pow2(x, m.ih.f, m.ih.e) : __dmul_rn(x, m.ih.f);
}

// velocity of axis AX on its face (i, j, k): 0 at the high wall of its own axis, the other two
// indices mirrored into the domain
template <int AX>
__device__ __forceinline__ double mom_vel(const MomArgs &m, int i, int j, int k)
{
    if ((AX == 0 && i >= m.nx) || (AX == 1 && j >= m.ny) || (AX == 2 && k >= m.nz)) return 0.0;
    i = clamp_idx(i, m.nx - 1);
    j = clamp_idx(j, m.ny - 1);
    k = clamp_idx(k, m.nz - 1);
    const double *u = AX == 0 ? m.u.bx : (AX == 1 ? m.u.by : m.u.bz);
    return u[((size_t)k * m.ny + j) * m.nx + i];
}

// viscosity of cell (i, j, k), the indices mirrored into the domain
__device__ __forceinline__ double mom_mu(const MomArgs &m, int i, int j, int k)
{
    i = clamp_idx(i, m.nx - 1);
    j = clamp_idx(j, m.ny - 1);
    k = clamp_idx(k, m.nz - 1);
    return __dadd_rn(m.mu_air, __dmul_rn(m.dmu, m.phi[((size_t)k * m.ny + j) * m.nx + i]));
}

// centre flux and stress of axis A at cell (i, j, k) (mu: the cell's viscosity) into their arrays at c
template <int A, bool CONV, bool VISC, bool POW2>
__device__ __forceinline__ void mom_centre(const MomArgs &m, size_t n, size_t c, int i, int j, int k, double mu)
{
    constexpr int ai = A == 0, aj = A == 1, ak = A == 2;
    const double u0 = mom_vel<A>(m, i, j, k), u1 = mom_vel<A>(m, i + ai, j + aj, k + ak);
    if (CONV) {
        const double U = mul_pow2(__dadd_rn(u0, u1), 0.5, -1);
        m.w[A * n + c] = __dmul_rn(U, U);
    }
    if (VISC) m.w[(3 + A) * n + c] = __dmul_rn(mul_pow2(mu, 2.0, 1), mom_ih<POW2>(m, __dsub_rn(u1, u0)));
}

// flux and shear of plane (A, B), A < B, at the low edge of cell (i, j, k); mc, ma, mb, mab: the
// viscosities of the cell and of its neighbours below along A, along B, along both
template <int A, int B, bool CONV, bool VISC, bool POW2>
__device__ __forceinline__ void mom_edge(const MomArgs &m, size_t n, size_t c, int i, int j, int k, double mc, double ma,
                                         double mb, double mab)
{
    constexpr int ai = A == 0, aj = A == 1, ak = A == 2, bi = B == 0, bj = B == 1, bk = B == 2;
    constexpr int slot = A + B - 1;  // xy, xz, yz
    const double ua0 = mom_vel<A>(m, i - bi, j - bj, k - bk), ua1 = mom_vel<A>(m, i, j, k);
    const double ub0 = mom_vel<B>(m, i - ai, j - aj, k - ak), ub1 = mom_vel<B>(m, i, j, k);
    if (CONV)
        m.w[(6 + slot) * n + c] =
            __dmul_rn(mul_pow2(__dadd_rn(ub0, ub1), 0.5, -1), mul_pow2(__dadd_rn(ua0, ua1), 0.5, -1));
    if (VISC) {
        const double me = mul_pow2(__dadd_rn(__dadd_rn(__dadd_rn(mab, mb), ma), mc), 0.25, -2);
        m.w[(9 + slot) * n + c] =
            __dmul_rn(me, __dadd_rn(mom_ih<POW2>(m, __dsub_rn(ua1, ua0)), mom_ih<POW2>(m, __dsub_rn(ub1, ub0))));
    }
}

// the viscosities a cell's terms use: its own and those of the cells below it along x, y, z, xy, xz and yz
struct MomMu {
    double c, x, y, z, xy, xz, yz;
};

// the fluxes and stresses of a cell
template <bool CONV, bool VISC, bool POW2>
__device__ __forceinline__ void mom_cell(const MomArgs &m, size_t n, size_t c, int i, int j, int k, const MomMu &mu)
{
    mom_centre<0, CONV, VISC, POW2>(m, n, c, i, j, k, mu.c);
    mom_centre<1, CONV, VISC, POW2>(m, n, c, i, j, k, mu.c);
    mom_centre<2, CONV, VISC, POW2>(m, n, c, i, j, k, mu.c);
    // in cell-index order: the cell below along both axes, below along the higher axis, below along
    // the lower axis, the cell itself
    mom_edge<0, 1, CONV, VISC, POW2>(m, n, c, i, j, k, mu.c, mu.x, mu.y, mu.xy);
    mom_edge<0, 2, CONV, VISC, POW2>(m, n, c, i, j, k, mu.c, mu.x, mu.z, mu.xz);
    mom_edge<1, 2, CONV, VISC, POW2>(m, n, c, i, j, k, mu.c, mu.y, mu.z, mu.yz);
}

// one thread per cell, which forms the viscosities it uses itself: where there are none to share (no viscous
// term), on small grids and on those whose rows leave the sharing blocks' lanes idle
template <bool CONV, bool VISC, bool POW2>
__global__ void k_mom_parts_cells(MomArgs m)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    if (i >= m.nx || j >= m.ny) return;
    const size_t n = (size_t)m.nx * m.ny * m.nz, c = ((size_t)k * m.ny + j) * m.nx + i;
    if (!MG_CK(c, c, (long long)n, CK_MOMENTUM)) return;
    MomMu mu{};
    if (VISC)
        mu = MomMu{mom_mu(m, i, j, k),         mom_mu(m, i - 1, j, k),     mom_mu(m, i, j - 1, k),    mom_mu(m, i, j, k - 1),
                   mom_mu(m, i - 1, j - 1, k), mom_mu(m, i - 1, j, k - 1), mom_mu(m, i, j - 1, k - 1)};
    mom_cell<CONV, VISC, POW2>(m, n, c, i, j, k, mu);
}

// blocks as k_phi_grad's (W x R threads, at most kPhiThreads, RUN planes up z); the viscosities of a plane
// of the block, with those of the row and the column before it, in one of three buffers by plane
// (a buffer is written again three planes later: one barrier per plane)
template <bool CONV, bool POW2, int RUN>
__global__ void k_mom_parts(MomArgs m)
{
    __shared__ double sh[3][kPhiThreads + kPhiW + 4];  // (R + 1) (W + 1): at most 3 x 257
    const int W = blockDim.x, R = blockDim.y, tx = threadIdx.x, ty = threadIdx.y;
    const int i = blockIdx.x * W + tx, j = blockIdx.y * R + ty;
    const bool in = i < m.nx && j < m.ny;
    const int k0 = blockIdx.z * RUN, k1 = min(k0 + RUN, m.nz);
    const size_t n = (size_t)m.nx * m.ny * m.nz;
    const int P = W + 1, at = (ty + 1) * P + tx + 1;
    // the viscosities of plane k (mirrored into the domain) into a buffer; a row or column before the first is
    // the first itself
    auto plane = [&](int k, double *buf) {
        if (!in) return;
        const double mc = mom_mu(m, i, j, k);
        buf[at] = mc;
        if (ty == 0) buf[at - P] = j > 0 ? mom_mu(m, i, j - 1, k) : mc;
        if (tx == 0) {
            buf[at - 1] = i > 0 ? mom_mu(m, i - 1, j, k) : mc;
            if (ty == 0) buf[0] = i > 0 || j > 0 ? mom_mu(m, i - 1, j - 1, k) : mc;
        }
    };
    plane(k0 - 1, sh[(k0 + 2) % 3]);
    for (int k = k0; k < k1; k++) {
        double *const b = sh[k % 3], *const bl = sh[(k + 2) % 3];
        plane(k, b);
        __syncthreads();
        const MomMu mu{b[at], b[at - 1], b[at - P], bl[at], b[at - P - 1], bl[at - 1], bl[at - P]};
        const size_t c = ((size_t)k * m.ny + j) * m.nx + i;
        if (!in || !MG_CK(c, c, (long long)n, CK_MOMENTUM)) continue;
        mom_cell<CONV, true, POW2>(m, n, c, i, j, k, mu);
    }
}

// R of face A at cell (i, j, k) = c, i.e. from the values at c, at the cell before it along A and, for the
// tangential axes, at c and the cell after it (edge values past the last cell lie on a high wall: zero flux
// and shear, the wall's normal velocity and the mirrored tangential one)
template <int A, bool CONV, bool VISC, bool POW2>
__device__ __forceinline__ double mom_face(const MomArgs &m, size_t n, int i, int j, int k, size_t c, double beta)
{
    const size_t step[3] = {1, (size_t)m.nx, (size_t)m.nx * m.ny};
    const bool last[3] = {i + 1 >= m.nx, j + 1 >= m.ny, k + 1 >= m.nz};
    const size_t cm = c - step[A];
    double conv = 0.0, visc = 0.0;
    if (CONV) conv = mom_ih<POW2>(m, __dsub_rn(m.w[A * n + c], m.w[A * n + cm]));
    if (VISC) visc = __dsub_rn(m.w[(3 + A) * n + c], m.w[(3 + A) * n + cm]);
#pragma unroll
    for (int B = 0; B < 3; B++) {
        if (B == A) continue;
        const int slot = A + B - 1;  // xy, xz, yz
        if (CONV) {
            const double *F = m.w + (6 + slot) * n;
            const double F0 = F[c], F1 = last[B] ? 0.0 : F[c + step[B]];
            conv = __dadd_rn(conv, mom_ih<POW2>(m, __dsub_rn(F1, F0)));
        }
        if (VISC) {
            const double *S = m.w + (9 + slot) * n;
            const double S0 = S[c], S1 = last[B] ? 0.0 : S[c + step[B]];
            visc = __dadd_rn(visc, __dsub_rn(S1, S0));
        }
    }
    double r = CONV ? neg_bits(conv) : 0.0;
    // (without the viscous term the sum is with a zero: +0 for a zero of either sign, as r + 0)
    if (VISC) r = __dadd_rn(r, __dmul_rn(__dmul_rn(m.inv_re, beta), mom_ih<POW2>(m, visc)));
    else if (zero_bits(r)) r = 0.0;
    if (A == 2) r = __dsub_rn(r, m.g);
    return r;
}

// one thread per cell: R on its three low faces
template <bool CONV, bool VISC, bool POW2>
__global__ void k_mom_combine(MomArgs m)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    if (i >= m.nx || j >= m.ny) return;
    const size_t n = (size_t)m.nx * m.ny * m.nz, c = ((size_t)k * m.ny + j) * m.nx + i;
    if (!MG_CK(c, c, (long long)n, CK_MOMENTUM)) return;
    const double bx = m.beta.bx[c], by = m.beta.by[c], bz = m.beta.bz[c];
    // an open face is interior (its low neighbour exists), so c - e_a is a cell
    m.r.bx[c] = (i > 0 && pos_bits(bx)) ? mom_face<0, CONV, VISC, POW2>(m, n, i, j, k, c, bx) : 0.0;
    m.r.by[c] = (j > 0 && pos_bits(by)) ? mom_face<1, CONV, VISC, POW2>(m, n, i, j, k, c, by) : 0.0;
    m.r.bz[c] = (k > 0 && pos_bits(bz)) ? mom_face<2, CONV, VISC, POW2>(m, n, i, j, k, c, bz) : 0.0;
}

// out = 0.5 (a + b)   (b null: 0.5 a)
__global__ void k_half(size_t n, LevelArrays<double> a, LevelArrays<double> b, LevelArrays<double> out)
{
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
        out.bx[c] = __dmul_rn(0.5, b.bx ? __dadd_rn(a.bx[c], b.bx[c]) : a.bx[c]);
        out.by[c] = __dmul_rn(0.5, b.by ? __dadd_rn(a.by[c], b.by[c]) : a.by[c]);
        out.bz[c] = __dmul_rn(0.5, b.bz ? __dadd_rn(a.bz[c], b.bz[c]) : a.bz[c]);
    }
}

// phi_out = phi - s * sum over open faces of +-u_f phi_up(f)  (s = dt / h; first-order upwind, the
// order x+, x-, y+, y-, z+, z-; closed faces carry no flux)
__global__ void k_vof_upwind(int nx, int ny, int nz, double s, LevelArrays<double> mask, LevelArrays<double> u,
                             const double *__restrict__ phi, double *__restrict__ phi_out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= nx) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_VOF)) return;
    auto upw = [&](double uf, size_t lo, size_t hi) { return __dmul_rn(uf, pos_bits(uf) ? phi[lo] : phi[hi]); };
    double d = 0.0;
    if (i < nx - 1 && pos_bits(mask.bx[c + 1])) d = __dadd_rn(d, upw(u.bx[c + 1], c, c + 1));
    if (pos_bits(mask.bx[c])) d = __dsub_rn(d, upw(u.bx[c], c - 1, c));
    if (j < ny - 1 && pos_bits(mask.by[c + nx])) d = __dadd_rn(d, upw(u.by[c + nx], c, c + nx));
    if (pos_bits(mask.by[c])) d = __dsub_rn(d, upw(u.by[c], c - nx, c));
    if (k < nz - 1 && pos_bits(mask.bz[c + sxy])) d = __dadd_rn(d, upw(u.bz[c + sxy], c, c + sxy));
    if (pos_bits(mask.bz[c])) d = __dsub_rn(d, upw(u.bz[c], c - sxy, c));
    phi_out[c] = __dsub_rn(phi[c], __dmul_rn(s, d));
}

// the operator's coefficient of a face: area * 1/rho where the area is > 0, else 0
__global__ void k_area_coeffs(size_t n, LevelArrays<double> area, LevelArrays<double> beta, LevelArrays<double> out)
{
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
        out.bx[c] = pos_bits(area.bx[c]) ? __dmul_rn(area.bx[c], beta.bx[c]) : 0.0;
        out.by[c] = pos_bits(area.by[c]) ? __dmul_rn(area.by[c], beta.by[c]) : 0.0;
        out.bz[c] = pos_bits(area.bz[c]) ? __dmul_rn(area.bz[c], beta.bz[c]) : 0.0;
    }
}

// u_f = u*_f - dt beta_f (p_c - p_nb) / h on open low faces; closed faces copy u*.
// x / h, rounded once: a multiply by ih = 1/h when h is a power of two (then x * (1/h) is exact
// and equal to the quotient; mul_pow2), an IEEE division otherwise
__device__ __forceinline__ double div_h(double x, double h, const Scale2 &ih)
{
    return ih.ok ? mul_pow2(x, ih.f, ih.e) : div_call(x, h);
}

// The face is open where b > 0; its coefficient is val (1/rho when b holds area * 1/rho), or b
// itself when val is null.
// DT2: dt is a power of two (1 by default), its product an exponent shift: 9 FP64 operations per cell
// instead of 12, 0.291 ms at 256^3 instead of 0.385
template <bool DT2>
__global__ void k_correct(int nx, int ny, int nz, Scale2 dt, double h, Scale2 ih,
                          const double *__restrict__ bx, const double *__restrict__ by, const double *__restrict__ bz,
                          const double *__restrict__ p, const double *ux0, const double *uy0, const double *uz0,
                          double *ux, double *uy, double *uz, LevelArrays<double> val)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= nx) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_CORRECT)) return;
    // every load first; each face's update formed and kept where the face is open (the same
    // operations as forming it there alone)
    const double pc = p[c], pxl = i > 0 ? p[c - 1] : 0.0, pyl = j > 0 ? p[c - nx] : 0.0;
    const double pzl = k > 0 ? p[c - sxy] : 0.0;
    const double b0 = bx[c], b1 = by[c], b2 = bz[c];
    const double u0 = ux0[c], u1 = uy0[c], u2 = uz0[c];
    const double v0 = val.bx ? val.bx[c] : b0, v1 = val.by ? val.by[c] : b1, v2 = val.bz ? val.bz[c] : b2;
    auto upd = [&](double u, double bv, double pn) {
        const double db = DT2 ? mul_pow2(bv, dt.f, dt.e) : __dmul_rn(dt.f, bv);
        return __dsub_rn(u, div_h(__dmul_rn(db, __dsub_rn(pc, pn)), h, ih));
    };
    ux[c] = (i > 0 && pos_bits(b0)) ? upd(u0, v0, pxl) : u0;
    uy[c] = (j > 0 && pos_bits(b1)) ? upd(u1, v1, pyl) : u1;
    uz[c] = (k > 0 && pos_bits(b2)) ? upd(u2, v2, pzl) : u2;
}

// The flux through face f along axis a: a product B_f w_f (the adjoint's right-hand side D(beta w)), or w_f (u_f - v_f) with w
// the face's area (null: 1) and v the body velocity (null: none); each operation rounded once.  edge: the same as calls,
// so that the warps without a face to form again skip their FP64 instructions.
struct FluxMul {
    LevelArrays<double> B, w;
    __device__ double operator()(int a, size_t f) const { return __dmul_rn(ax(B, a)[f], ax(w, a)[f]); }
    __device__ double edge(int a, size_t f) const { return dmul_call(ax(B, a)[f], ax(w, a)[f]); }
    static __device__ const double *ax(const LevelArrays<double> &v, int a) { return a == 0 ? v.bx : (a == 1 ? v.by : v.bz); }
};
struct FluxArea {
    LevelArrays<double> area, u, v;
    __device__ double operator()(int a, size_t f) const
    {
        const double *A = FluxMul::ax(area, a), *V = FluxMul::ax(v, a);
        double d = FluxMul::ax(u, a)[f];
        if (V) d = __dsub_rn(d, V[f]);
        return A ? __dmul_rn(A[f], d) : d;
    }
    __device__ double edge(int a, size_t f) const
    {
        const double *A = FluxMul::ax(area, a), *V = FluxMul::ax(v, a);
        double d = FluxMul::ax(u, a)[f];
        if (V) d = dadd_call(d, -V[f]);
        return A ? dmul_call(A[f], d) : d;
    }
};

// With areas or a body velocity on small grids: a thread per cell, each of its faces' fluxes formed where it stands
// (launch_divergence_area has the lines).
__global__ void k_divergence_area(int nx, int ny, int nz, Scale2 scale, LevelArrays<double> mask,
                                  LevelArrays<double> area, LevelArrays<double> u, LevelArrays<double> v,
                                  double *__restrict__ rhs)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_DIVERGENCE)) return;
    auto flux = [&](const double *a, const double *uu, const double *vv, size_t f) {
        const double du = vv ? __dsub_rn(uu[f], vv[f]) : uu[f];
        return a ? __dmul_rn(a[f], du) : du;
    };
    double d = 0.0;
    if (i < nx - 1 && pos_bits(mask.bx[c + 1])) d = __dadd_rn(d, flux(area.bx, u.bx, v.bx, c + 1));
    if (pos_bits(mask.bx[c])) d = __dsub_rn(d, flux(area.bx, u.bx, v.bx, c));
    if (j < ny - 1 && pos_bits(mask.by[c + nx])) d = __dadd_rn(d, flux(area.by, u.by, v.by, c + nx));
    if (pos_bits(mask.by[c])) d = __dsub_rn(d, flux(area.by, u.by, v.by, c));
    if (k < nz - 1 && pos_bits(mask.bz[c + sxy])) d = __dadd_rn(d, flux(area.bz, u.bz, v.bz, c + sxy));
    if (pos_bits(mask.bz[c])) d = __dsub_rn(d, flux(area.bz, u.bz, v.bz, c));
    rhs[c] = mul_s2(d, scale);
}

// rhs_c = scale * the sum over the open faces of c (L's coefficient > 0) of +- the flux, x+ added
// and x- subtracted, then y, then z (as k_divergence).  Blocks as k_phi_grad: each face's
// flux formed once, the x+ and y+ ones taken from the neighbours through shared memory (formed
// again only at the block's right edge and top row), the z+ one carried up the column.  With areas and
// no body velocity 10 FP64 operations per cell instead of 13 (192x160x224: 0.247 -> 0.170 ms).  RUN planes per block.
template <int RUN, typename F>
__global__ void k_divergence_flux(int nx, int ny, int nz, Scale2 scale, LevelArrays<double> L, F flux,
                                  double *__restrict__ rhs)
{
    __shared__ double sh[2][2][kPhiThreads];  // [plane parity][x- / y- flux][thread]
    const int W = blockDim.x, R = blockDim.y;
    const int i = blockIdx.x * W + threadIdx.x, j = blockIdx.y * R + threadIdx.y;
    const int t = threadIdx.y * W + threadIdx.x;
    const bool in = i < nx && j < ny;
    const int k0 = blockIdx.z * RUN, k1 = min(k0 + RUN, nz);
    const size_t sxy = (size_t)nx * ny;
    size_t c = in ? (size_t)k0 * sxy + (size_t)j * nx + i : 0;
    const bool ok0 = in && ck_cell((long long)c, i, j, k0, nx, ny, nz, CK_DIVERGENCE);
    double tz_lo = ok0 ? flux(2, c) : 0.0;
    bool oz_lo = ok0 && pos_bits(L.bz[c]);
    for (int k = k0; k < k1; k++, c += sxy) {
        const bool ok = in && ck_cell((long long)c, i, j, k, nx, ny, nz, CK_DIVERGENCE);
        double tx = 0.0, ty = 0.0, tz_hi = 0.0;
        bool ox0 = false, ox1 = false, oy0 = false, oy1 = false, oz1 = false;
        if (ok) {
            tx = flux(0, c);
            ty = flux(1, c);
            ox0 = pos_bits(L.bx[c]);
            oy0 = pos_bits(L.by[c]);
            ox1 = i < nx - 1 && pos_bits(L.bx[c + 1]);
            oy1 = j < ny - 1 && pos_bits(L.by[c + nx]);
            if (k < nz - 1) {
                tz_hi = flux(2, c + sxy);
                oz1 = pos_bits(L.bz[c + sxy]);
            }
        }
        double(*buf)[kPhiThreads] = sh[k & 1];
        buf[0][t] = tx;
        buf[1][t] = ty;
        __syncthreads();  // one barrier per plane: a buffer is written again two planes later
        if (ok) {
            double tx_hi = 0.0, ty_hi = 0.0;
            if (i < nx - 1) tx_hi = threadIdx.x < W - 1 ? buf[0][t + 1] : flux.edge(0, c + 1);
            if (j < ny - 1) ty_hi = threadIdx.y < R - 1 ? buf[1][t + W] : flux.edge(1, c + nx);
            double d = ox1 ? zero_plus(tx_hi) : 0.0;
            if (ox0) d = __dsub_rn(d, tx);
            if (oy1) d = __dadd_rn(d, ty_hi);
            if (oy0) d = __dsub_rn(d, ty);
            if (oz1) d = __dadd_rn(d, tz_hi);
            if (oz_lo) d = __dsub_rn(d, tz_lo);
            rhs[c] = mul_s2(d, scale);  // scale * d
        }
        tz_lo = tz_hi;
        oz_lo = oz1;
    }
}

// grad_u = w - G q (open faces) / w (closed);  grad_beta = dt (G p)((G q) - w) (open) / 0 (closed)
// has_a: the face's open area a multiplies G q (fractional areas)
template <bool DT2>
__device__ __forceinline__ void adj_face(double b, double pc, double pn, double qc, double qn, double w, double h,
                                         const Scale2 &ih, const Scale2 &dt, bool has_a, double a, double &gu,
                                         double &gb)
{
    double gq = div_h(__dsub_rn(qc, qn), h, ih);
    const double gp = div_h(__dsub_rn(pc, pn), h, ih);
    if (has_a) gq = dmul_call(a, gq);
    const double go = __dsub_rn(w, gq);
    // (Gq - w) is -gu exactly: a rounded difference changes sign with its operands' order
    const double bo = __dmul_rn(DT2 ? mul_pow2(gp, dt.f, dt.e) : __dmul_rn(dt.f, gp), -go);
    const bool open = pos_bits(b);
    gu = open ? go : w;
    gb = open ? bo : 0.0;
}

// DT2: as for k_correct (12 FP64 operations per cell instead of 15, 0.392 ms at 256^3 instead of 0.487)
template <bool DT2>
__global__ void k_adjoint_faces(int nx, int ny, int nz, double h, Scale2 ih, Scale2 dt,
                                const double *__restrict__ bx,
                                const double *__restrict__ by, const double *__restrict__ bz,
                                const double *__restrict__ p, const double *__restrict__ q,
                                const double *__restrict__ wx, const double *__restrict__ wy,
                                const double *__restrict__ wz, double *gux, double *guy, double *guz, double *gbx,
                                double *gby, double *gbz, LevelArrays<double> area)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= nx) return;
    const size_t sxy = (size_t)nx * ny;
    const size_t c = (size_t)k * sxy + (size_t)j * nx + i;
    if (!ck_cell((long long)c, i, j, k, nx, ny, nz, CK_ADJOINT)) return;
    // every load first
    const double pc = p[c], qc = q[c];
    const double pxl = i > 0 ? p[c - 1] : 0.0, qxl = i > 0 ? q[c - 1] : 0.0;
    const double pyl = j > 0 ? p[c - nx] : 0.0, qyl = j > 0 ? q[c - nx] : 0.0;
    const double pzl = k > 0 ? p[c - sxy] : 0.0, qzl = k > 0 ? q[c - sxy] : 0.0;
    const double b0 = bx[c], b1 = by[c], b2 = bz[c], w0 = wx[c], w1 = wy[c], w2 = wz[c];
    const double a0 = area.bx ? area.bx[c] : 1.0, a1 = area.by ? area.by[c] : 1.0, a2 = area.bz ? area.bz[c] : 1.0;
    double gu, gb;
    adj_face<DT2>(b0, pc, pxl, qc, qxl, w0, h, ih, dt, area.bx != nullptr, a0, gu, gb);
    gux[c] = gu;
    if (gbx) gbx[c] = gb;
    adj_face<DT2>(b1, pc, pyl, qc, qyl, w1, h, ih, dt, area.by != nullptr, a1, gu, gb);
    guy[c] = gu;
    if (gby) gby[c] = gb;
    adj_face<DT2>(b2, pc, pzl, qc, qzl, w2, h, ih, dt, area.bz != nullptr, a2, gu, gb);
    guz[c] = gu;
    if (gbz) gbz[c] = gb;
}

// grad_phi_c = -(drho/2) sum over the six faces of beta_f^2 grad_beta_f (order x-,x+,y-,y+,z-,z+).
// A block of W x R threads covers R rows of W cells (W: nx rounded up to a warp multiple, at most
// kPhiW) and walks kPhiRun planes up z.  Each face's product (beta_f beta_f) grad_beta_f is formed
// once: every cell forms those of its x- and y- faces and of the z- face of the cell above; the
// x+ and y+ products are the neighbours' (shared memory, two buffers by plane parity), formed again
// only at the block's right edge and top row, and the z+ product is carried up as the next cell's
// z- product.  The same products summed in the same order as forming all six per cell (0 + t is
// t but for -0; NaN payloads aside).
__global__ void k_phi_grad(int nx, int ny, int nz, double neg_half_drho, const double *__restrict__ bx,
                           const double *__restrict__ by, const double *__restrict__ bz,
                           const double *__restrict__ gbx, const double *__restrict__ gby,
                           const double *__restrict__ gbz, double *__restrict__ gphi)
{
    __shared__ double sh[2][2][kPhiThreads];  // [plane parity][x- / y- product][thread]
    const int W = blockDim.x, R = blockDim.y;
    const int i = blockIdx.x * W + threadIdx.x, j = blockIdx.y * R + threadIdx.y;
    const int t = threadIdx.y * W + threadIdx.x;
    const bool in = i < nx && j < ny;
    const int k0 = blockIdx.z * kPhiRun, k1 = min(k0 + kPhiRun, nz);
    const size_t sxy = (size_t)nx * ny;
    auto prod = [](double b, double g) { return __dmul_rn(__dmul_rn(b, b), g); };
    size_t c = in ? (size_t)k0 * sxy + (size_t)j * nx + i : 0;
    const bool ok0 = in && ck_cell((long long)c, i, j, k0, nx, ny, nz, CK_PHI_GRAD);
    double tz_lo = ok0 ? prod(bz[c], gbz[c]) : 0.0;
    for (int k = k0; k < k1; k++, c += sxy) {
        const bool ok = in && ck_cell((long long)c, i, j, k, nx, ny, nz, CK_PHI_GRAD);
        double tx = 0.0, ty = 0.0, tz_hi = 0.0;
        if (ok) {
            tx = prod(bx[c], gbx[c]);
            ty = prod(by[c], gby[c]);
            if (k < nz - 1) tz_hi = prod(bz[c + sxy], gbz[c + sxy]);
        }
        double(*buf)[kPhiThreads] = sh[k & 1];
        buf[0][t] = tx;
        buf[1][t] = ty;
        __syncthreads();  // one barrier per plane: a buffer is written again two planes later
        if (ok) {
            double tx_hi = 0.0, ty_hi = 0.0;
            if (i < nx - 1) tx_hi = threadIdx.x < W - 1 ? buf[0][t + 1] : sq_mul_call(bx[c + 1], gbx[c + 1]);
            if (j < ny - 1) ty_hi = threadIdx.y < R - 1 ? buf[1][t + W] : sq_mul_call(by[c + nx], gby[c + nx]);
            double s = zero_plus(tx);
            if (i < nx - 1) s = __dadd_rn(s, tx_hi);
            s = __dadd_rn(s, ty);
            if (j < ny - 1) s = __dadd_rn(s, ty_hi);
            s = __dadd_rn(s, tz_lo);
            if (k < nz - 1) s = __dadd_rn(s, tz_hi);
            gphi[c] = __dmul_rn(neg_half_drho, s);
        }
        tz_lo = tz_hi;
    }
}

// ---------------------------------------------------------------------------
// Multigrid-preconditioned CG (flexible form).  FP64 Krylov vectors; the
// preconditioned vector z is FP64 (plain FP64 solves) or s * e32 with the FP32
// cycle's output e32 and the scale s the FP32 right-hand side was divided by.
// Device scalars (Scal): S_RZ <r,z>, S_RZN / S_RZO new <r,z> and <r,z_old>,
// S_SIGMA <d, A d>, S_RR ||r||^2.
// ---------------------------------------------------------------------------

// *flag |= 1 if any p[i] is nonzero (either sign of zero counts as zero); the caller clears it
__global__ void k_nonzero(unsigned n, const double *__restrict__ p, unsigned *__restrict__ flag)
{
    bool any = false;
    const double2 *p2 = reinterpret_cast<const double2 *>(p);
    stream_pairs(
        n, [&](unsigned v) { return p2[v]; }, [&](unsigned, const double2 &x) { any |= !zero_bits(x.x) || !zero_bits(x.y); },
        [&](unsigned c) { any |= !zero_bits(p[c]); });
    if (__syncthreads_or(any) && threadIdx.x == 0) atomicOr(flag, 1u);
}

// r = b - A p (FP64, resid_columns).  Optionally r32 = r / scale, scale = RMS of b (first pass) written to scale_slot.
// pnz (optional): the k_nonzero flag of p; 0 means p is zero everywhere, and each cell's
// residual is then b exactly with no stencil loaded: the same values for a fraction of the loads (the
// first residual of a solve from a zero guess), streamed as pairs of cells in a loop that holds no stencil
// arithmetic at all (a select inside one loop would still issue it)
__global__ void k_pcg_resid(int nx, int ny, int nz, double ih2, LevelArrays<double> L, const double *__restrict__ b,
                            const double *__restrict__ p, double *__restrict__ r, float *__restrict__ r32,
                            double *__restrict__ dscal, int scale_slot, double *__restrict__ partials, Split sp,
                            ResidGrid g, const unsigned *__restrict__ pnz)
{
    const bool pzero = pnz && *pnz == 0u;
    const unsigned n = (unsigned)nx * ny * nz;
    const double inv_scale = block_scalar([&] {
        if (!r32) return 1.0;
        const double rms = sqrt(dscal[S_NB2] / dscal[S_NLIVE]);
        const double sc = (rms > 0.0 && isfinite(rms)) ? rms : 1.0;
        if (blockIdx.x == 0) dscal[scale_slot] = sc;
        return 1.0 / sc;
    });
    double rr = 0.0, sum = 0.0;
    if (pzero) {
        const double2 *b2 = reinterpret_cast<const double2 *>(b);
        double2 *r2 = reinterpret_cast<double2 *>(r);
        stream_pairs(
            n, [&](unsigned v) { return b2[v]; },
            [&](unsigned v, const double2 &x) {
                r2[v] = x;
                if (r32) {
                    const float f0 = narrow(x.x * inv_scale), f1 = narrow(x.y * inv_scale);
                    if (sp.half) {  // the pair's colours at slot v of each half
                        const int q = row_parity(2 * v, sp);
                        r32[(q ? sp.half : 0) + v] = f0;
                        r32[(q ? 0 : sp.half) + v] = f1;
                    } else {
                        reinterpret_cast<float2 *>(r32)[v] = make_float2(f0, f1);
                    }
                }
                rr = fma(x.x, x.x, rr);
                rr = fma(x.y, x.y, rr);
            },
            [&](unsigned c) {  // (an odd number of cells is never colour-split)
                r[c] = b[c];
                if (r32) r32[c] = narrow(b[c] * inv_scale);
                rr = fma(b[c], b[c], rr);
            });
    } else {
        resid_columns(nx, ny, nz, ih2, L, b, p, g, [&](size_t c, int q, double v, double pc) {
            r[c] = v;
            if (r32) {
                const size_t slot = sp.half ? split_slot(c, q, sp.half) : c;
                if (MG_CK(slot, slot, (long long)n, CK_SPLIT_SLOT)) r32[slot] = narrow(v * inv_scale);
            }
            rr = fma(v, v, rr);
            if (pos_bits(L.dinv[c])) sum += pc;
        });
    }
    block_sum2<kRedThreads>(rr, sum);
    reduce_finish(rr, sum, partials, dscal, S_RR, S_SUM_P);
}

// <r, z> and <r, z_old> with z = sz * Z, z_old = so * Zo (Z double: scales 1)
template <typename Z>
__global__ void k_pcg_dots(unsigned n, const double *__restrict__ r, const Z *__restrict__ z, const Z *__restrict__ zo,
                           double *dscal, int sz_slot, int so_slot, double *__restrict__ partials)
{
    const double sz = sz_slot >= 0 ? dscal[sz_slot] : 1.0;
    const double so = so_slot >= 0 ? dscal[so_slot] : 1.0;
    double a = 0.0, c = 0.0;
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        const double rv = r[idx];
        a = fma(rv, (double)z[idx], a);
        if (zo) c = fma(rv, (double)zo[idx], c);
    }
    block_sum2<kRedThreads>(a, c);
    reduce_finish(a * sz, c * so, partials, dscal, S_RZN, S_RZO);
}

// Mixed-precision variant: <r, z> = sr sz <r32, e32> from the FP32 copy r32 = r / sr that the
// preconditioner read.  Products and short per-thread sums are FP32, block sums FP64: the CG
// scalars need only the accuracy of the FP32 preconditioner they weigh.
__global__ void k_pcg_dots32(unsigned n, const float *__restrict__ r32, const float *__restrict__ z,
                             const float *__restrict__ zo, double *dscal, int sr_slot, int sz_slot,
                             int so_slot, double *__restrict__ partials)
{
    const double sr = dscal[sr_slot];
    double a = 0.0, c = 0.0;
    const unsigned n4 = n / 4, stride = gridDim.x * blockDim.x;
    const float4 *r4 = reinterpret_cast<const float4 *>(r32);
    const float4 *z4 = reinterpret_cast<const float4 *>(z);
    const float4 *o4 = reinterpret_cast<const float4 *>(zo);
    // widened on the integer pipe (exact, as the conversion instruction, which runs on the FP64 unit)
    auto dot4 = [](float4 x, float4 y) { return widen(fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, x.x * y.x)))); };
    // float4 groups v and v + stride per iteration, all loads issued first; the sums in the same
    // order as one group per iteration
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < n4; v += 2 * stride) {
        const unsigned w = v + stride;
        const bool has_w = w < n4;
        const float4 rv = r4[v], zv = z4[v], rw = has_w ? r4[w] : zero4, zw = has_w ? z4[w] : zero4;
        const float4 ov = zo ? o4[v] : zero4, ow = (zo && has_w) ? o4[w] : zero4;
        a += dot4(rv, zv);
        if (zo) c += dot4(rv, ov);
        if (has_w) {
            a += dot4(rw, zw);
            if (zo) c += dot4(rw, ow);
        }
    }
    for (unsigned idx = 4 * n4 + blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += stride) {
        a += widen(r32[idx] * z[idx]);
        if (zo) c += widen(r32[idx] * zo[idx]);
    }
    block_sum2<kRedThreads>(a, c);
    a = a * sr * dscal[sz_slot];
    c = c * (so_slot >= 0 ? sr * dscal[so_slot] : 0.0);
    reduce_finish(a, c, partials, dscal, S_RZN, S_RZO);
}

// The search direction d = sz Z + beta d_old, beta = (<r,z> - <r,z_old>) / <r_old, z_old> (first:
// beta = 0), with z = sz Z the preconditioned residual, is kept divided by its z's scale: D = d / sz
// = Z + (beta so / sz) D_old (so: the scale of D_old), one FP64 operation per cell.  The CG
// update then moves p and r by <r,z> / (sz <D, A D>) times D and A D (k_pcg_update), the same
// step.  Without scales (sz_slot, so_slot < 0) D = d.
template <typename Z>
__global__ void k_pcg_dir(unsigned n, const Z *__restrict__ z, double *__restrict__ d, double *dscal,
                          int sz_slot, int so_slot, int first, Split sp, double *__restrict__ partials)
{
    const double beta = block_scalar([&] {
        return first ? 0.0
                     : (dscal[S_RZN] - dscal[S_RZO]) / dscal[S_RZ] *
                           (so_slot >= 0 ? dscal[so_slot] / dscal[sz_slot] : 1.0);
    });
    const unsigned n2 = n / 2, stride = gridDim.x * blockDim.x;
    double2 *d2 = reinterpret_cast<double2 *>(d);
    // the two Z indices of pair v (colour-split Z: the pair's colours sit at slot v of each half)
    auto zidx = [&](unsigned v, size_t &i0, size_t &i1) {
        i0 = 2 * (size_t)v;
        i1 = 2 * (size_t)v + 1;
        if (sp.half) {
            const int q = row_parity(2 * v, sp);
            i0 = (q ? sp.half : 0) + v;
            i1 = (q ? 0 : sp.half) + v;
            return MG_CK(i0, i0, (long long)n, CK_SPLIT_SLOT) && MG_CK(i1, i1, (long long)n, CK_SPLIT_SLOT);
        }
        return true;
    };
    // pairs v and v + stride per iteration, both pairs' loads issued before either update
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < n2; v += 2 * stride) {
        const unsigned w = v + stride;
        const bool has_w = w < n2;
        size_t a0, a1, b0 = 0, b1 = 0;
        const bool ok_v = zidx(v, a0, a1), ok_w = has_w && zidx(w, b0, b1);
        const Z za0 = ok_v ? z[a0] : Z(0), za1 = ok_v ? z[a1] : Z(0);
        const Z zb0 = ok_w ? z[b0] : Z(0), zb1 = ok_w ? z[b1] : Z(0);
        double2 dv = (first || !ok_v) ? make_double2(0.0, 0.0) : d2[v];
        double2 dw = (first || !ok_w) ? make_double2(0.0, 0.0) : d2[w];
        if (ok_v) {
            dv.x = fma(beta, dv.x, widen(za0));
            dv.y = fma(beta, dv.y, widen(za1));
            d2[v] = dv;
        }
        if (ok_w) {
            dw.x = fma(beta, dw.x, widen(zb0));
            dw.y = fma(beta, dw.y, widen(zb1));
            d2[w] = dw;
        }
    }
    for (unsigned idx = 2 * n2 + blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += stride)
        d[idx] = fma(beta, first ? 0.0 : d[idx], widen(z[idx]));
    // every block has read <r, z> above: the last one moves the new <r, z> into its place
    if (last_block(partials) && threadIdx.x == 0) dscal[S_RZ] = dscal[S_RZN];
}

// Jacobi preconditioner: z = (scale * dinv) * r, dead cells 0
__global__ void k_jacobi(unsigned n, double scale, const double *__restrict__ dinv, const double *__restrict__ r,
                         double *__restrict__ z)
{
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x)
        z[idx] = (scale * dinv[idx]) * r[idx];
}

// q = A d and <d, q>, with A d = sum_f (h^-2 beta_f) d_nb - (h^-2 diag) d_c on arrays pre-scaled
// by h^-2 (L, diag; exact for a power-of-two h): 8 FP64 operations per cell instead of 15 for the
// difference form.  Its rounding error is larger for smooth d (relative ~1e-12 at 256^3), which
// only perturbs the recursive residual; convergence is confirmed on the true residual in
// difference form.
__global__ void k_pcg_apply(int nx, int ny, int nz, LevelArrays<double> L, const double *__restrict__ diag,
                            const double *__restrict__ d, double *__restrict__ q, double *__restrict__ partials,
                            double *dscal)
{
    const unsigned n = (unsigned)nx * ny * nz;
    const size_t sxy = (size_t)nx * ny;
    double dq = 0.0;
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        int i, j, k;
        cell_of(idx, nx, ny, i, j, k);
        if (!ck_cell(idx, i, j, k, nx, ny, nz, CK_PCG_APPLY)) continue;
        const double dc = d[idx];
        double s = -diag[idx] * dc;
        if (i > 0) s = fma(L.bx[idx], d[idx - 1], s);
        if (i < nx - 1) s = fma(L.bx[idx + 1], d[idx + 1], s);
        if (j > 0) s = fma(L.by[idx], d[idx - nx], s);
        if (j < ny - 1) s = fma(L.by[idx + nx], d[idx + nx], s);
        if (k > 0) s = fma(L.bz[idx], d[idx - sxy], s);
        if (k < nz - 1) s = fma(L.bz[idx + sxy], d[idx + sxy], s);
        const double qv = s;
        q[idx] = qv;
        dq = fma(dc, qv, dq);
    }
    reduce_finish(block_sum<kRedThreads>(dq), 0.0, partials, dscal, S_SIGMA, -1);
}

// alpha = <r,z>/<d,Ad>; p += alpha d; r -= alpha q; ||r||^2; optionally r32 = r / scale with
// scale = RMS of the previous residual (written to scale_slot).  Two elements per iteration.
__global__ void k_pcg_update(unsigned n, const double *__restrict__ d, const double *__restrict__ q,
                             double *__restrict__ p, double *__restrict__ r, float *__restrict__ r32,
                             double *dscal, int scale_slot, int sd_slot, double *__restrict__ partials,
                             Split sp)
{
    // d holds D = (direction) / sd (k_pcg_dir): alpha = <r,z> / <d, A d> times sd
    const double alpha =
        block_scalar([&] { return dscal[S_RZ] / (dscal[S_SIGMA] * (sd_slot >= 0 ? dscal[sd_slot] : 1.0)); });
    const double inv_scale = block_scalar([&] {
        if (!r32) return 1.0;
        const double rms = sqrt(dscal[S_RR] / dscal[S_NLIVE]);
        const double sc = (rms > 0.0 && isfinite(rms)) ? rms : 1.0;
        if (blockIdx.x == 0) dscal[scale_slot] = sc;
        return 1.0 / sc;
    });
    const float inv_scale32 = (float)inv_scale;
    double rr = 0.0;
    const unsigned n2 = n / 2, stride = gridDim.x * blockDim.x;
    const double2 *d2 = reinterpret_cast<const double2 *>(d);
    const double2 *q2 = reinterpret_cast<const double2 *>(q);
    double2 *p2 = reinterpret_cast<double2 *>(p);
    double2 *rv2 = reinterpret_cast<double2 *>(r);
    float2 *r32v = reinterpret_cast<float2 *>(r32);
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < n2; v += stride) {
        const double2 dv = d2[v], qv = q2[v];
        double2 pv = p2[v], rv = rv2[v];
        pv.x = fma(alpha, dv.x, pv.x);
        pv.y = fma(alpha, dv.y, pv.y);
        rv.x = fma(-alpha, qv.x, rv.x);
        rv.y = fma(-alpha, qv.y, rv.y);
        p2[v] = pv;
        rv2[v] = rv;
        if (r32) {
            const float r0 = narrow(rv.x) * inv_scale32, r1 = narrow(rv.y) * inv_scale32;
            if (sp.half) {  // colour-split r32: the pair's colours at slot v of each half
                const int qp = row_parity(2 * v, sp);
                r32[(qp ? sp.half : 0) + v] = r0;
                r32[(qp ? 0 : sp.half) + v] = r1;
            } else {
                r32v[v] = make_float2(r0, r1);
            }
        }
        rr = fma(rv.x, rv.x, rr);
        rr = fma(rv.y, rv.y, rr);
    }
    for (unsigned idx = 2 * n2 + blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += stride) {
        p[idx] = fma(alpha, d[idx], p[idx]);
        const double rv = fma(-alpha, q[idx], r[idx]);
        r[idx] = rv;
        if (r32) r32[idx] = narrow(rv) * inv_scale32;
        rr = fma(rv, rv, rr);
    }
    reduce_finish(block_sum<kRedThreads>(rr), 0.0, partials, dscal, S_RR, -1);
}


// ---------------------------------------------------------------------------
// Connected components of the live cells (cells joined by open faces) and the mean removal of
// the Neumann problem per component (Eq. neumann with Eq. pois: A is singular with one constant
// per component in its null space, so the rhs is projected to zero mean on each component and p
// is pinned to zero mean on each).  Union-find over x-runs:
//   1. each live cell points to the first cell of its run of cells joined by open x-faces;
//   2. each open y- or z-face joins the roots of its two cells (the larger root is hooked under
//      the smaller with atomicMin; a hook that finds the root hooked meanwhile continues with the
//      new parent), except where the face to the left already joined the same two runs;
//   3. every cell takes its root; a root is the smallest cell index of its component.
// Every parent has a smaller index than its child, so the pointers form no cycle and every loop
// below ends; each is still bounded by kCcBudget steps and reports exceeding it in *err.
// ---------------------------------------------------------------------------
constexpr unsigned kCcBudget = 1u << 26;

__device__ __forceinline__ int cc_load(const int *label, int x)
{
    if (!MG_CK(x, x, 0x7fffffffll, CK_LABEL)) return x;
    return *(const volatile int *)(label + x);
}

__device__ __forceinline__ int cc_find(const int *label, int x, unsigned &budget)
{
    int y = cc_load(label, x);
    while (y != x && budget) {
        budget--;
        x = y;
        y = cc_load(label, x);
    }
    return x;
}

__device__ void cc_union(int *label, int a, int b, unsigned *err)
{
    unsigned budget = kCcBudget;
    a = cc_find(label, a, budget);
    b = cc_find(label, b, budget);
    while (a != b && budget) {
        budget--;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(label + b, a);
        if (old == b) return;  // b was a root: now under a
        // b had been hooked under old meanwhile (and is now under min(old, a)): join old and a
        b = cc_find(label, old, budget);
        a = cc_find(label, a, budget);
    }
    if (a != b) atomicOr(err, 1u);
}

// step 1: one warp per x-row; label = first cell of the run (-1 on dead cells)
__global__ void k_cc_rows(int nx, int ny, int nz, const double *__restrict__ dinv, const double *__restrict__ bx,
                          int *__restrict__ label)
{
    const unsigned lane = threadIdx.x & 31u;
    const size_t row = (size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= (size_t)ny * nz) return;  // uniform across the warp
    const size_t base = row * (size_t)nx;
    int carry = -1;
    for (int i0 = 0; i0 < nx; i0 += 32) {
        const int i = i0 + (int)lane;
        const bool in = i < nx;
        const size_t c = base + (size_t)i;
        const bool live = in && pos_bits(dinv[c]);
        const bool join = live && i > 0 && pos_bits(bx[c]);
        const unsigned starts = __ballot_sync(0xffffffffu, live && !join);
        const unsigned m = starts & (0xffffffffu >> (31u - lane));
        const int start = m ? (int)(base + (size_t)i0 + (31 - __clz((int)m))) : carry;
        if (in) label[c] = live ? start : -1;
        carry = __shfl_sync(0xffffffffu, start, 31);
    }
}

// step 2: join the runs across open y- and z-faces
__global__ void k_cc_merge(int nx, int ny, int nz, const double *__restrict__ bx, const double *__restrict__ by,
                           const double *__restrict__ bz, int *label, unsigned *err)
{
    const unsigned n = (unsigned)nx * ny * nz;
    const unsigned sxy = (unsigned)nx * ny;
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        int i, j, k;
        cell_of(idx, nx, ny, i, j, k);
        // the run continues from the left (its own low x-face open)
        const bool left = i > 0 && pos_bits(bx[idx]);
        if (j > 0 && pos_bits(by[idx])) {
            // implied when the cell to the left is in this run, its y-face is open and its
            // neighbour is in the neighbour's run
            const bool implied = left && pos_bits(by[idx - 1]) && pos_bits(bx[idx - nx]);
            if (!implied) cc_union(label, (int)idx, (int)(idx - nx), err);
        }
        if (k > 0 && pos_bits(bz[idx])) {
            const bool implied = left && pos_bits(bz[idx - 1]) && pos_bits(bx[idx - sxy]);
            if (!implied) cc_union(label, (int)idx, (int)(idx - sxy), err);
        }
    }
}

// step 3: every live cell takes its root; count[0] += number of roots
__global__ void k_cc_flatten(unsigned n, int *label, unsigned *count, unsigned *err)
{
    unsigned roots = 0;
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        const int l = label[idx];
        if (l < 0) continue;
        unsigned budget = kCcBudget;
        const int r = cc_find(label, l, budget);
        if (!budget) atomicOr(err, 1u);
        label[idx] = r;
        roots += (r == (int)idx);
    }
    roots = __reduce_add_sync(0xffffffffu, roots);
    if ((threadIdx.x & 31u) == 0 && roots) atomicAdd(count, roots);
}

// the roots (one per component) in any order
__global__ void k_cc_roots(unsigned n, const int *__restrict__ label, int *__restrict__ roots, unsigned *slot,
                           unsigned cap)
{
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x)
        if (label[idx] == (int)idx) {
            const unsigned q = atomicAdd(slot, 1u);
            if (q < cap) roots[q] = (int)idx;
        }
}

// root -> component number (its rank among the sorted roots)
__global__ void k_cc_compact(unsigned n, int *__restrict__ label, const int *__restrict__ roots, int ncomp)
{
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        const int r = label[idx];
        if (r < 0) continue;
        int lo = 0, hi = ncomp - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (roots[mid] < r) lo = mid + 1;
            else hi = mid;
        }
        label[idx] = lo;
    }
}

// per-component sums of v (v null: of 1, the cell counts) over the live cells: each thread sums
// kCcChunk consecutive cells and adds to the component total once per change of component (a
// domain's cells mostly share one)
constexpr unsigned kCcChunk = 64;
__global__ void k_comp_sums(unsigned n, const double *__restrict__ v, const int *__restrict__ comp,
                            double *__restrict__ sums)
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned c0 = t * kCcChunk; c0 < n; c0 += stride * kCcChunk) {
        int cur = -1;
        double acc = 0.0;
        const unsigned c1 = min(n, c0 + kCcChunk);
        for (unsigned c = c0; c < c1; c++) {
            const int id = comp[c];
            if (id < 0) continue;
            if (id != cur) {
                if (cur >= 0) atomicAdd(sums + cur, acc);
                cur = id;
                acc = 0.0;
            }
            acc += v ? v[c] : 1.0;
        }
        if (cur >= 0) atomicAdd(sums + cur, acc);
    }
}

// The same sums in a fixed order (bitwise reproducible), eight components per pass: per-block
// sums of the components g0 .. g0+7 into part[q * gridDim.x + block], then summed over the blocks
__global__ void k_comp_sums8(unsigned n, const double *__restrict__ v, const int *__restrict__ comp, int g0,
                             double *__restrict__ part)
{
    double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        const int q = comp[idx] - g0;
        if ((unsigned)q < 8u) {
            const double x = v ? v[idx] : 1.0;
#pragma unroll
            for (int r = 0; r < 8; r++)
                if (q == r) acc[r] += x;
        }
    }
#pragma unroll
    for (int r = 0; r < 8; r++) {
        const double t = block_sum<kRedThreads>(acc[r]);
        if (threadIdx.x == 0) part[r * gridDim.x + blockIdx.x] = t;
    }
}
__global__ void k_comp_finish8(const double *__restrict__ part, int nblocks, int g0, int ncomp,
                               double *__restrict__ sums)
{
    for (int r = 0; r < 8; r++) {
        double a = 0.0;
        for (int i = threadIdx.x; i < nblocks; i += blockDim.x) a += part[r * nblocks + i];
        a = block_sum<kRedThreads>(a);
        if (threadIdx.x == 0 && g0 + r < ncomp) sums[g0 + r] = a;
    }
}

// out = v - its component's mean on live cells, 0 elsewhere; partial sums of out^2 and of v
__global__ void k_comp_center(unsigned n, const double *__restrict__ v, const int *__restrict__ comp,
                              const double *__restrict__ sums, const double *__restrict__ cnt,
                              double *__restrict__ out, double *__restrict__ partials)
{
    double a = 0.0, b = 0.0;
    for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        const int id = comp[idx];
        double o = 0.0;
        if (id >= 0) {
            o = v[idx] - sums[id] / cnt[id];
            b += v[idx];
        }
        out[idx] = o;
        a += o * o;
    }
    block_sum2<kRedThreads>(a, b);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = a;
        partials[2 * blockIdx.x + 1] = b;
    }
}

// 1/h as a Scale2 for div_h: ok when h is a power of two (h = 2^(ex-1), 1/h = 2^(1-ex) exactly)
inline Scale2 inv_scale2(double h)
{
    int ex;
    const bool ok = std::frexp(h, &ex) == 0.5;
    return Scale2{1.0 / h, 1 - ex, ok ? 1 : 0};
}

inline dim3 row_grid(int threads_x, int ny, int nz)
{
    return dim3((unsigned)((threads_x + kRowThreads - 1) / kRowThreads), (unsigned)ny, (unsigned)nz);
}

// Blocks of kRowThreads threads over rows of threads_x threads each: x the next power of two >=
// threads_x (at most kRowThreads), the rest of the block over consecutive rows, so that a coarse
// level's short rows (32 or 64 threads) do not leave most of each block idle.  Kernels launched so
// take their row from blockIdx.y * blockDim.y + threadIdx.y and skip rows past the last.
inline dim3 row_block2(int threads_x)
{
    int bx = 1;
    while (bx < threads_x && bx < kRowThreads) bx *= 2;
    return dim3((unsigned)bx, (unsigned)(kRowThreads / bx));
}
inline dim3 row_grid2(int threads_x, int ny, int nz)
{
    const dim3 b = row_block2(threads_x);
    return dim3((unsigned)((threads_x + b.x - 1) / b.x), (unsigned)((ny + b.y - 1) / b.y), (unsigned)nz);
}

// Blocks of the kernels that share values along rows: W x R threads, a row or, beyond kPhiW cells, an equal part of
// one, rounded up to whole warps, by as many rows as fit, and `run` planes.  (In parts of kPhiW a row of 300 cells left 41 % of
// the lanes idle: face coefficients of 300x48x49 105 us, 67 so.)
inline void row_share_grid(Dims d, dim3 &grid, dim3 &block, int run = kPhiRun, int threads = kPhiThreads)
{
    const int parts = (d.nx + kPhiW - 1) / kPhiW, W = ((d.nx + parts - 1) / parts + 31) / 32 * 32;
    const int R = std::max(1, std::min(threads / W, d.ny));
    grid = dim3((unsigned)((d.nx + W - 1) / W), (unsigned)((d.ny + R - 1) / R), (unsigned)((d.nz + run - 1) / run));
    block = dim3((unsigned)W, (unsigned)R);
}

// Blocks of the finest FP32 level's kernels that take several cells along x per thread (rows of G threads):
// 32 threads by 4 rows where G is a multiple of 32, else G cut into equal parts of at most 32 threads
// by as many rows as make up to 128 threads, so that short rows do not leave lanes idle (at nx = 128 a
// colour pass had 16 threads per row and ran half of each warp: 19.5 us per sweep, 16.5 us so; 192x160x224
// 34.9 -> 31.8 us, 320x192x128 44.9 -> 39.6 us).  Rows of 32 threads keep the colour pass's body per row
// parity: with the parity selected per value a sweep took 10 % longer at 256^3.
inline dim3 pair_block(int G)
{
    const int parts = (G + 31) / 32, x = (G + parts - 1) / parts;
    return dim3((unsigned)x, (unsigned)(128 / x));
}
inline dim3 pair_grid(int G, int rows, int planes, dim3 block)
{
    return dim3((unsigned)((G + block.x - 1) / block.x), (unsigned)((rows + block.y - 1) / block.y), (unsigned)planes);
}

// Blocks of the grid-stride reductions: at most five per SM, so that the grid is one wave (the operator
// of the CG holds six blocks per SM by its registers) and its end reads few partials, and on small
// grids at least four cells per thread beyond two blocks per SM.  CG operator + update + dots and
// direction, mixed: 241 + 182 + 100 us at 256^3 with 16 blocks per SM, 241 + 177 + 92 us with five,
// 238 + 175 + 96 with four; 128^3: 45 + 38 + 36 us with 16, 39 + 31 + 26 with five; 64^3: 14 + 15 + 18 us with up to 16,
// 12 + 14 + 16 with two.
inline unsigned red_grid(size_t n)
{
    const size_t b = (n + kRedThreads - 1) / kRedThreads, sm = 152;
    return (unsigned)std::max<size_t>(1, std::min({b, std::max(2 * sm, b / 4), 5 * sm}));
}
// Tasks of the residual kernels, one per block: the shortest runs of planes that need no more than kRedBlocks blocks
// (many short tasks even out over the SMs), of two at least where that leaves four blocks per SM
inline ResidGrid resid_grid(Dims d)
{
    ResidGrid g;
    g.colblocks = (unsigned)(((size_t)d.nx * d.ny + kRedThreads - 1) / kRedThreads);
    g.run = 1;
    auto tasks = [&](int run) { return (size_t)g.colblocks * ((d.nz + run - 1) / run); };
    if (tasks(2) >= 4 * 152) g.run = 2;
    while (tasks(g.run) > (size_t)kRedBlocks && g.run < d.nz) g.run++;
    g.tasks = (unsigned)tasks(g.run);
    g.fcb = make_fastdiv(g.colblocks);
    g.fnx = make_fastdiv((unsigned)d.nx);
    return g;
}
inline unsigned resid_blocks(const ResidGrid &g) { return std::min(g.tasks, (unsigned)kRedBlocks); }
// Blocks of the vector passes without a reduction and of the FP64 CG's dots and direction, which
// stream and have no FP64 arithmetic to hide latency behind: eight per SM (FP64 CG vectors at 256^3: 129 us, 138 us with
// five, 133 us with 16).
inline unsigned vec_grid(size_t n)
{
    const size_t b = (n + kRedThreads - 1) / kRedThreads;
    return (unsigned)std::max<size_t>(1, std::min<size_t>(b, 8 * 152));
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_face_coeffs(Dims d, const double *phi, const uint8_t *solid, double rho_a, double drho,
                               double *bx, double *by, double *bz, cudaStream_t s)
{
    note_launch();
    // the largest blocks and the longest runs that leave two blocks per SM
    int run = kRun, threads = kPhiThreads;
    dim3 grid, block;
    for (;;) {
        row_share_grid(d, grid, block, run, threads);
        if ((size_t)grid.x * grid.y * grid.z >= 2 * 152 || (run <= 2 && threads <= 128)) break;
        if (threads > 128) threads /= 2;
        else run /= 2;
    }
    const double rho_w = rho_a + drho, den_w = rho_w + rho_w, q_w = 2.0 / den_w;  // the kernel's for phi = 1
    if (solid)
        k_face_coeffs<true><<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, run, phi, solid, rho_a, drho, den_w, q_w, bx, by, bz);
    else
        k_face_coeffs<false><<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, run, phi, nullptr, rho_a, drho, den_w, q_w, bx, by,
                                                    bz);
    return cudaGetLastError();
}

cudaError_t launch_jacobi(size_t n, double scale, const double *dinv, const double *r, double *z, cudaStream_t s)
{
    note_launch();
    k_jacobi<<<vec_grid(n), kRedThreads, 0, s>>>((unsigned)n, scale, dinv, r, z);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_diag_inv(Dims d, const T *bx, const T *by, const T *bz, T *dinv, cudaStream_t s,
                            const LevelArrays<T> *op, T scale, uint8_t *open, double *changed)
{
    note_launch();
    k_diag_inv<T><<<run_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(d.nx, d.ny, d.nz, run_planes(d.nx, d.ny, d.nz), bx, by, bz, dinv,
                                                                      op ? *op : LevelArrays<T>{},
                                                                      scale2((double)scale), open, changed);
    return cudaGetLastError();
}
template cudaError_t launch_diag_inv<double>(Dims, const double *, const double *, const double *, double *,
                                             cudaStream_t, const LevelArrays<double> *, double, uint8_t *, double *);

cudaError_t launch_level_f32(Dims d, const LevelArrays<double> &L, LevelArrays<float> &out, cudaStream_t s,
                             LevelArrays<float> *sf, Split sp)
{
    note_launch();
    const bool split = sf && sf->bx && sp.half;
    k_level_f32<<<run_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(d.nx, d.ny, d.nz, run_planes(d.nx, d.ny, d.nz), L.bx, L.by, L.bz, out,
                                                                     split ? *sf : LevelArrays<float>{},
                                                                     split ? sp.half : 0);
    return cudaGetLastError();
}

cudaError_t launch_restrict_coeffs(Dims f, const double *bx, const double *by, const double *bz, double *cbx,
                                   double *cby, double *cbz, cudaStream_t s)
{
    note_launch();
    k_restrict_coeffs<<<row_grid(f.nx / 2, f.ny / 2, f.nz / 2), kRowThreads, 0, s>>>(f.nx, f.ny, f.nz, bx, by, bz, cbx,
                                                                                      cby, cbz);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_smooth(Dims d, T h2, const LevelArrays<T> &L, const T *b, T *p, int colour, cudaStream_t s,
                          bool zero, const T *rec, Gate gate)
{
    note_launch();
    const dim3 g = row_grid2((d.nx + 1) / 2, d.ny, d.nz), blk = row_block2((d.nx + 1) / 2);
    const GsScale<T> gs = gs_scale<T>(h2);
    auto go = [&](auto zer, auto rows, auto gated) {
        k_smooth<T, decltype(zer)::value, decltype(rows)::value, decltype(gated)::value>
            <<<g, blk, 0, s>>>(d.nx, d.ny, d.nz, gs, L, b, p, colour, rec, gate);
    };
    const BoolTag<true> yes;
    const BoolTag<false> no;
    if (gate.rr) {  // (FP64, from an iterate)
        if (sizeof(T) != 8 || zero) return cudaErrorInvalidValue;
        if constexpr (sizeof(T) == 8) {
            if (rec) go(no, yes, yes);
            else go(no, no, yes);
        }
    } else if (zero) go(yes, no, no);
    else if (rec) go(no, yes, no);
    else go(no, no, no);
    return cudaGetLastError();
}
template cudaError_t launch_smooth<double>(Dims, double, const LevelArrays<double> &, const double *, double *, int,
                                           cudaStream_t, bool, const double *, Gate);
template cudaError_t launch_smooth<float>(Dims, float, const LevelArrays<float> &, const float *, float *, int,
                                          cudaStream_t, bool, const float *, Gate);

cudaError_t launch_smooth_first(Dims d, float h2, const LevelArrays<float> &L, const float *b, float *p, cudaStream_t s)
{
    note_launch();
    const dim3 g = row_grid2((d.nx + 1) / 2, d.ny, d.nz), blk = row_block2((d.nx + 1) / 2);
    k_smooth_first<<<g, blk, 0, s>>>(d.nx, d.ny, d.nz, h2, L, b, p);
    return cudaGetLastError();
}

cudaError_t launch_prolong_black(Dims f, float h2, const LevelArrays<float> &L, const float *b, const float *ec, float *p,
                                 cudaStream_t s)
{
    note_launch();
    const dim3 g = row_grid2(f.nx / 2, f.ny, f.nz), blk = row_block2(f.nx / 2);
    k_prolong_black<<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, h2, L, b, ec, p);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_row_records(Dims d, const LevelArrays<T> &L, T *rec, cudaStream_t s)
{
    const int rows = d.ny * d.nz, warps = 8;
    note_launch();
    k_row_records<T><<<(rows + warps - 1) / warps, 32 * warps, 0, s>>>(d.nx, d.ny, d.nz, L.bx, L.by, L.bz, rec);
    return cudaGetLastError();
}
template cudaError_t launch_row_records<double>(Dims, const LevelArrays<double> &, double *, cudaStream_t);
template cudaError_t launch_row_records<float>(Dims, const LevelArrays<float> &, float *, cudaStream_t);

cudaError_t launch_smooth_split(Dims d, float h2, const LevelArrays<float> &L, const float *b, float *p, int colour,
                                cudaStream_t s, const float *urow, const float4 *arow, const float2 *uinv, int rev,
                                bool zero, const LevelArrays<float> *S)
{
    note_launch();
    if (d.nx % 8 == 0) {  // four cells per thread
        if (!S || !S->bx || !S->by || !S->bz || (urow && !uinv)) return cudaErrorInvalidValue;
        const dim3 block = pair_block(d.nx / 8), grid = pair_grid(d.nx / 8, d.ny, d.nz, block);
        auto go = [&](auto band, auto zer, auto rows) {
            k_smooth_split4<decltype(band)::value, decltype(zer)::value, decltype(rows)::value ? 1 : 0>
                <<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, h2, *S, b, p, colour, urow, arow, uinv, rev, L.dinv);
        };
        auto go_rows = [&](auto band, auto zer) {
            if (block.x == 32) go(band, zer, BoolTag<true>{});
            else go(band, zer, BoolTag<false>{});
        };
        if (arow) {
            if (zero) go_rows(BoolTag<true>{}, BoolTag<true>{});
            else go_rows(BoolTag<true>{}, BoolTag<false>{});
        } else {
            if (zero) go_rows(BoolTag<false>{}, BoolTag<true>{});
            else go_rows(BoolTag<false>{}, BoolTag<false>{});
        }
    } else {
        k_smooth_split<<<row_grid(d.nx / 2, d.ny, d.nz), kRowThreads, 0, s>>>(d.nx, d.ny, d.nz, h2, L, b, p, colour,
                                                                              urow, rev, zero ? 1 : 0);
    }
    return cudaGetLastError();
}

cudaError_t launch_uniform_rows(Dims d, const float *bx, const float *by, const float *bz, float *urow,
                                cudaStream_t s, float4 *arow, float2 *uinv, unsigned *count)
{
    const int rows = d.ny * d.nz, warps = 8;
    note_launch();
    k_uniform_rows<<<(rows + warps - 1) / warps, 32 * warps, 0, s>>>(d.nx, d.ny, d.nz, bx, by, bz, urow, arow,
                                                                      uinv, count);
    return cudaGetLastError();
}

// 256^3, FP32 finest level: 35.0 us (58.9 us with all 8 residuals formed, one coarse cell per thread);
// 128^3 natural: 5.8 us (9.3), 32^3: 2.5 us (3.6).  FP64 at 128^3: 31.4 us against 57 us, 29 us of it
// the FP64 unit's.
template <typename T>
cudaError_t launch_restrict(Dims f, T ih2, const LevelArrays<T> &L, const T *b, const T *p, T *bc, cudaStream_t s,
                            Split sp, const float *urow, const float4 *arow, int rev, const LevelArrays<T> *S)
{
    note_launch();
    const dim3 g = row_grid2(f.nx / 2, f.ny / 2, f.nz / 2), blk = row_block2(f.nx / 2);
    if constexpr (std::is_same<T, float>::value) {
        if (sp.half && f.nx % 8 == 0) {
            if (!S || !S->bx || !urow) return cudaErrorInvalidValue;
            const dim3 b4 = pair_block(f.nx / 4), g4 = pair_grid(f.nx / 4, f.ny / 2, f.nz / 2, b4);
            if (arow)
                k_restrict4<true><<<g4, b4, 0, s>>>(f.nx, f.ny, f.nz, ih2, *S, b, p, bc, urow, arow, rev);
            else
                k_restrict4<false><<<g4, b4, 0, s>>>(f.nx, f.ny, f.nz, ih2, *S, b, p, bc, urow, nullptr, rev);
            return cudaGetLastError();
        }
        if (sp.half) {
            k_restrict<T, true><<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, ih2, L, b, p, bc, sp.half);
            return cudaGetLastError();
        }
    } else if (sp.half) {
        return cudaErrorInvalidValue;  // FP64 fields are never split
    }
    k_restrict<T, false><<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, ih2, L, b, p, bc, 0);
    return cudaGetLastError();
}
template cudaError_t launch_restrict<double>(Dims, double, const LevelArrays<double> &, const double *, const double *,
                                             double *, cudaStream_t, Split, const float *, const float4 *, int,
                                             const LevelArrays<double> *);
template cudaError_t launch_restrict<float>(Dims, float, const LevelArrays<float> &, const float *, const float *,
                                            float *, cudaStream_t, Split, const float *, const float4 *, int,
                                            const LevelArrays<float> *);

// 256^3, FP32 finest level: 19.4 us (35.3 us correcting all 8 children, one coarse cell per thread);
// 128^3: 5.5 us (6.3).  FP64 at 128^3: 19.0 us, bound by the FP64 unit (36 operations per coarse cell,
// 72 for all children).
template <typename T>
cudaError_t launch_prolong_red(Dims f, const T *ec, const T *dinv, T *p, cudaStream_t s, Split sp, const float *urow,
                               const float4 *arow)
{
    note_launch();
    const dim3 g = row_grid2(f.nx / 2, f.ny / 2, f.nz / 2), blk = row_block2(f.nx / 2);
    if constexpr (std::is_same<T, float>::value) {
        if (sp.half && f.nx % 8 == 0) {
            if (!urow) return cudaErrorInvalidValue;
            const dim3 b4 = pair_block(f.nx / 4), g4 = pair_grid(f.nx / 4, f.ny / 2, f.nz / 2, b4);
            k_prolong_red4<<<g4, b4, 0, s>>>(f.nx, f.ny, f.nz, ec, dinv, p, arow ? &arow->x : urow, arow ? 4 : 1);
            return cudaGetLastError();
        }
        if (sp.half) {
            k_prolong_red<T, true><<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, ec, dinv, p);
            return cudaGetLastError();
        }
    } else if (sp.half) {
        return cudaErrorInvalidValue;  // FP64 fields are never split
    }
    k_prolong_red<T, false><<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, ec, dinv, p);
    return cudaGetLastError();
}
template cudaError_t launch_prolong_red<double>(Dims, const double *, const double *, double *, cudaStream_t, Split,
                                                const float *, const float4 *);
template cudaError_t launch_prolong_red<float>(Dims, const float *, const float *, float *, cudaStream_t, Split,
                                               const float *, const float4 *);

template <typename T>
cudaError_t launch_prolong(Dims f, const T *ec, const T *dinv, T *p, cudaStream_t s, Split sp, const float *urow)
{
    note_launch();
    const dim3 g = row_grid2(f.nx / 2, f.ny / 2, f.nz / 2), blk = row_block2(f.nx / 2);
    if constexpr (std::is_same<T, float>::value) {
        if (sp.half) {
            k_prolong<T, true><<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, ec, dinv, p, sp.half, urow);
            return cudaGetLastError();
        }
    } else if (sp.half) {
        return cudaErrorInvalidValue;  // FP64 fields are never split
    }
    k_prolong<T, false><<<g, blk, 0, s>>>(f.nx, f.ny, f.nz, ec, dinv, p, 0, sizeof(T) == 4 ? urow : nullptr);
    return cudaGetLastError();
}
template cudaError_t launch_prolong<double>(Dims, const double *, const double *, double *, cudaStream_t, Split,
                                            const float *);
template cudaError_t launch_prolong<float>(Dims, const float *, const float *, float *, cudaStream_t, Split,
                                           const float *);

// Tiles of 32 x 8 columns; z-chunks sized so that the grid has about 4 CTAs per SM.
template <typename T>
cudaError_t launch_rb_sweep(Dims d, T h2, const LevelArrays<T> &L, const T *b, const T *p_old, T *p_new, int first,
                            cudaStream_t s)
{
    constexpr int TX = 32, TY = 8;
    const int tx = (d.nx + TX - 1) / TX, ty = (d.ny + TY - 1) / TY;
    const int want = 4 * 152;
    int chunks = (want + tx * ty - 1) / (tx * ty);
    int zc = (d.nz + chunks - 1) / chunks;
    if (zc < 8) zc = 8;
    if (zc > d.nz) zc = d.nz;
    const dim3 grid((unsigned)tx, (unsigned)ty, (unsigned)((d.nz + zc - 1) / zc));
    note_launch();
    // (FP64, h no power of two: 256^3, V-cycle of 2 + 2 such sweeps: 4.09 ms, 4.47 with gs_start's call per cell)
    const GsScale<T> gs = gs_scale<T>(h2);
    if (sizeof(T) == 4 || gs.s.ok)
        k_rb_sweep<T, true, TX, TY><<<grid, (TX + 4) * (TY + 4), 0, s>>>(d.nx, d.ny, d.nz, zc, gs, L, b, p_old, p_new, first);
    else if constexpr (sizeof(T) == 8)
        k_rb_sweep<T, false, TX, TY><<<grid, (TX + 4) * (TY + 4), 0, s>>>(d.nx, d.ny, d.nz, zc, gs, L, b, p_old, p_new, first);
    return cudaGetLastError();
}
template cudaError_t launch_rb_sweep<double>(Dims, double, const LevelArrays<double> &, const double *,
                                             const double *, double *, int, cudaStream_t);
template cudaError_t launch_rb_sweep<float>(Dims, float, const LevelArrays<float> &, const float *, const float *,
                                            float *, int, cudaStream_t);

template <typename T>
cudaError_t launch_coarse_solve(int n, const double *M, const T *b, T *e, cudaStream_t s)
{
    const int rows_per_cta = 8;  // one warp per row
    note_launch();
    k_coarse_solve<T><<<(n + rows_per_cta - 1) / rows_per_cta, 32 * rows_per_cta, (size_t)n * sizeof(double), s>>>(n, M, b,
                                                                                                                e);
    return cudaGetLastError();
}
// a launch of k_tail on a cluster
inline void tail_config(int ctas, size_t smem, cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at)
{
    cfg = cudaLaunchConfig_t{};
    at = cudaLaunchAttribute{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
}

// CTAs of the largest cluster (16, else 8) that the current device holds with kTailSmem bytes each, 0 if
// neither: a property of the device, asked once for each (the query takes some 80 us).
// The kernel's shared-memory limit and its cluster opt-in belong to the function, so every context and thread of a
// device shares them: they are set here, by each mg_setup before the context's first launch, always to the same values, and
// never by a launch.  (A limit set to a context's own need fails another thread's larger launch between the two.)
template <typename T>
int tail_ctas()
{
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];  // 1 + the answer
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    cudaError_t e = cudaFuncSetAttribute(k_tail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const bool wide = cudaFuncSetAttribute(k_tail<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (dev < kDevices && known[dev].load() > 0) return known[dev].load() - 1;
    int n = 0;
    for (int ctas : {16, 8}) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at;
        int clusters = 0;
        tail_config(ctas, kTailSmem, cfg, at);
        if ((wide || ctas <= 8) && cudaOccupancyMaxActiveClusters(&clusters, k_tail<T>, &cfg) == cudaSuccess &&
            clusters >= 1) {
            n = ctas;
            break;
        }
    }
    cudaGetLastError();
    if (dev < kDevices) known[dev].store(n + 1);
    return n;
}
template int tail_ctas<double>();
template int tail_ctas<float>();

// Coarse-grid correction below a grid, us (a launch per pass -> this kernel -> one CTA with its fields in
// L1, two launches and the exact solve between, as it was): 32^3 FP32 35 -> 21 (35), FP64 45 -> 27 (86);
// 64^3 FP32 47 -> 35 (50), FP64 64 -> 48 (111); 192x160x224 FP32 92 -> 87 (96).  With a coarsest grid of
// 512 cells, whose inverse 16 SMs apply in the time of the launches saved: 116 -> 116 (125) FP32.
template <typename T>
cudaError_t launch_tail(const TailArgs<T> &a, cudaStream_t s)
{
    if (a.nlev < 2 || a.nlev > kTailMaxLevels || a.ctas < 1 || a.smem > kTailSmem) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    tail_config(a.ctas, a.smem, cfg, at);
    cfg.stream = s;
    note_launch();
    return cudaLaunchKernelEx(&cfg, k_tail<T>, a);
}
template cudaError_t launch_tail<double>(const TailArgs<double> &, cudaStream_t);
template cudaError_t launch_tail<float>(const TailArgs<float> &, cudaStream_t);

template cudaError_t launch_coarse_solve<double>(int, const double *, const double *, double *, cudaStream_t);
template cudaError_t launch_coarse_solve<float>(int, const double *, const float *, float *, cudaStream_t);

cudaError_t launch_components(Dims d, const double *dinv, const double *bx, const double *by, const double *bz,
                              int *label, unsigned *ctr, cudaStream_t s)
{
    const unsigned n = (unsigned)d.n();
    cudaError_t e = cudaMemsetAsync(ctr, 0, 2 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const size_t rows = (size_t)d.ny * d.nz;
    note_launch();
    k_cc_rows<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(d.nx, d.ny, d.nz, dinv, bx, label);
    note_launch();
    k_cc_merge<<<vec_grid(n), kRedThreads, 0, s>>>(d.nx, d.ny, d.nz, bx, by, bz, label, ctr + 1);
    note_launch();
    k_cc_flatten<<<vec_grid(n), kRedThreads, 0, s>>>(n, label, ctr, ctr + 1);
    return cudaGetLastError();
}

cudaError_t launch_component_roots(size_t n, const int *label, int *roots, unsigned *slot, unsigned cap,
                                   cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(slot, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    note_launch();
    k_cc_roots<<<vec_grid(n), kRedThreads, 0, s>>>((unsigned)n, label, roots, slot, cap);
    return cudaGetLastError();
}

cudaError_t launch_component_compact(size_t n, int *label, const int *sorted_roots, int ncomp, double *cnt,
                                     double *part, cudaStream_t s)
{
    note_launch();
    k_cc_compact<<<vec_grid(n), kRedThreads, 0, s>>>((unsigned)n, label, sorted_roots, ncomp);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_comp_sums(n, nullptr, label, ncomp, cnt, part, s);
}

cudaError_t launch_comp_sums(size_t n, const double *v, const int *comp, int ncomp, double *sums, double *part,
                             cudaStream_t s)
{
    if (ncomp <= kCompOrdered) {  // fixed order, eight components per pass
        const unsigned g = red_grid(n);
        for (int g0 = 0; g0 < ncomp; g0 += 8) {
            note_launch();
            k_comp_sums8<<<g, kRedThreads, 0, s>>>((unsigned)n, v, comp, g0, part);
            note_launch();
            k_comp_finish8<<<1, kRedThreads, 0, s>>>(part, (int)g, g0, ncomp, sums);
        }
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(sums, 0, (size_t)ncomp * sizeof(double), s);
    if (e != cudaSuccess) return e;
    const unsigned threads = (unsigned)((n + kCcChunk - 1) / kCcChunk);
    note_launch();
    k_comp_sums<<<vec_grid(threads), kRedThreads, 0, s>>>((unsigned)n, v, comp, sums);
    return cudaGetLastError();
}

cudaError_t launch_comp_center(size_t n, const double *v, const int *comp, int ncomp, double *sums,
                               const double *cnt, double *out, double *partials, double *dscal, int slot_sq,
                               int slot_sum, cudaStream_t s, double *part)
{
    cudaError_t e = launch_comp_sums(n, v, comp, ncomp, sums, part, s);
    if (e != cudaSuccess) return e;
    const unsigned g = red_grid(n);
    note_launch();
    k_comp_center<<<g, kRedThreads, 0, s>>>((unsigned)n, v, comp, sums, cnt, out, partials);
    note_launch();
    k_finish2<<<1, kRedThreads, 0, s>>>(partials, (int)g, dscal, slot_sq, slot_sum);
    return cudaGetLastError();
}

cudaError_t launch_count_live(Dims d, const double *dinv, double *partials, double *dscal, cudaStream_t s)
{
    const unsigned g = vec_grid(d.n());
    note_launch();
    k_count_live<<<g, kRedThreads, 0, s>>>((unsigned)d.n(), dinv, partials, dscal);
    return cudaGetLastError();
}

cudaError_t launch_rhs_prepare(Dims d, const double *rhs, const double *dinv, double *b0, double *partials,
                               double *dscal, cudaStream_t s)
{
    const unsigned g = vec_grid(d.n());
    note_launch();
    k_sum_live<<<g, kRedThreads, 0, s>>>((unsigned)d.n(), rhs, dinv, partials, dscal, S_SUM_B);
    note_launch();
    k_rhs_center<<<g, kRedThreads, 0, s>>>((unsigned)d.n(), rhs, dinv, b0, dscal, partials);
    return cudaGetLastError();
}

cudaError_t launch_resid_norm(Dims d, double ih2, const LevelArrays<double> &L, const double *b, const double *p,
                              double *partials, double *dscal, cudaStream_t s)
{
    const ResidGrid g = resid_grid(d);
    note_launch();
    if (resid_sums_p(d.n()))
        k_resid_norm<true><<<resid_blocks(g), kRedThreads, 0, s>>>(d.nx, d.ny, d.nz, ih2, L, b, p, partials, dscal, g);
    else
        k_resid_norm<false><<<resid_blocks(g), kRedThreads, 0, s>>>(d.nx, d.ny, d.nz, ih2, L, b, p, partials, dscal, g);
    return cudaGetLastError();
}

cudaError_t launch_sum_p(Dims d, const double *dinv, const double *p, double *partials, double *dscal, cudaStream_t s)
{
    note_launch();
    k_sum_live<<<vec_grid(d.n()), kRedThreads, 0, s>>>((unsigned)d.n(), p, dinv, partials, dscal, S_SUM_P);
    return cudaGetLastError();
}

cudaError_t launch_sub_mean_p(Dims d, const double *dinv, double *p, const double *dscal, cudaStream_t s)
{
    note_launch();
    k_sub_mean_p<<<vec_grid(d.n()), kRedThreads, 0, s>>>((unsigned)d.n(), dinv, p, dscal);
    return cudaGetLastError();
}

cudaError_t launch_resid_cast(Dims d, double ih2, const LevelArrays<double> &L, const double *b, const double *p,
                              float *r32, double *partials, double *dscal, int scale_in, int scale_out,
                              cudaStream_t s, Split sp)
{
    const ResidGrid g = resid_grid(d);
    if (scale_in < 0) {  // first pass: scale from ||b0||
        scale_in = S_SCALE0;
        note_launch();
        k_scale_from_nb2<<<1, 1, 0, s>>>(dscal, scale_in);
    }
    note_launch();
    auto go = [&](auto sum) {
        k_resid_cast<decltype(sum)::value><<<resid_blocks(g), kRedThreads, 0, s>>>(
            d.nx, d.ny, d.nz, ih2, L, b, p, r32, dscal, scale_in, scale_out, partials, sp.half, g);
    };
    if (resid_sums_p(d.n())) go(BoolTag<true>{});
    else go(BoolTag<false>{});
    return cudaGetLastError();
}

cudaError_t launch_to_f32_layout(size_t n, const double *src, float *dst, cudaStream_t s, Split sp)
{
    note_launch();
    k_to_f32_layout<<<vec_grid(n), kRedThreads, 0, s>>>((unsigned)n, src, dst, sp);
    return cudaGetLastError();
}

cudaError_t launch_from_f32_layout(size_t n, const float *src, double *dst, cudaStream_t s, Split sp)
{
    note_launch();
    k_from_f32_layout<<<vec_grid(n), kRedThreads, 0, s>>>((unsigned)n, src, dst, sp);
    return cudaGetLastError();
}

cudaError_t launch_accumulate(Dims d, const double *dinv, const float *e32, double *p, const double *dscal,
                              int scale_slot, cudaStream_t s, Split sp)
{
    note_launch();
    (void)dinv;
    k_accumulate<<<vec_grid(d.n()), kRedThreads, 0, s>>>((unsigned)d.n(), e32, p, dscal, scale_slot, sp);
    return cudaGetLastError();
}

cudaError_t launch_divergence(Dims d, double scale, const double *bx, const double *by, const double *bz,
                              const double *ux, const double *uy, const double *uz, double *rhs, cudaStream_t s)
{
    note_launch();
    k_divergence<<<row_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(d.nx, d.ny, d.nz, scale2(scale), bx, by, bz, ux, uy, uz,
                                                                     rhs);
    return cudaGetLastError();
}

cudaError_t launch_correct(Dims d, double dt, double h, const double *bx, const double *by, const double *bz,
                           const double *p, const double *ux0, const double *uy0, const double *uz0, double *ux,
                           double *uy, double *uz, cudaStream_t s, const LevelArrays<double> *val)
{
    note_launch();
    const Scale2 dt2 = scale2(dt);
    auto go = [&](auto tag) {
        k_correct<decltype(tag)::value><<<row_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(
            d.nx, d.ny, d.nz, dt2, h, inv_scale2(h), bx, by, bz, p, ux0, uy0, uz0, ux, uy, uz,
            val ? *val : LevelArrays<double>{});
    };
    if (dt2.ok) go(BoolTag<true>{});
    else go(BoolTag<false>{});
    return cudaGetLastError();
}

cudaError_t launch_face_areas(Dims d, const double *psi, double *ax, double *ay, double *az, cudaStream_t s)
{
    note_launch();
    k_face_areas<<<row_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(d.nx, d.ny, d.nz, psi, ax, ay, az);
    return cudaGetLastError();
}

cudaError_t launch_stretched_metrics(Dims d, const double *hx, const double *hy, const double *hz,
                                    const LevelArrays<double> &beta, const LevelArrays<double> &frac,
                                    const LevelArrays<double> &bout, const LevelArrays<double> &aout, cudaStream_t s)
{
    note_launch();
    // Per cell below 600,000 cells, in runs of 4 planes below 1.2 M and of kRun above: a block walks its run one plane after the
    // other, 30 us for 16 planes however few blocks there are.  Per cell, 4 and 16 planes (z stretched, waves; us): 16^3 4.9, 13, 32;
    // 32^3 6, 16, 36; 64^3 23, 28, 45; 224x56x40 38, 40, 56; 80^3 45, 42, 54; 88^3 55, 48, 57; 96^3 65, 52, 61; 500x500x4 68, 65, 65;
    // 112^3 114, 80, 92; 128^3 148, 100, 114; 192x160x224 473, 254, 211; 256^3 1143, 553, 451.
    const dim3 blk = row_block2(d.nx);
    auto grid = [&](int run) {
        return dim3((d.nx + blk.x - 1) / blk.x, (d.ny + blk.y - 1) / blk.y, (d.nz + run - 1) / run);
    };
    auto go = [&](auto tag) {
        constexpr int R = decltype(tag)::value;
        k_stretched_metrics<R><<<grid(R), blk, 0, s>>>(d.nx, d.ny, d.nz, hx, hy, hz, beta, frac, bout, aout);
    };
    const dim3 g1 = grid(1), g4 = grid(4);  // (a grid's z extent is at most 65535)
    if (d.n() < 600000 && g1.z <= 65535)
        k_stretched_metrics_cells<<<g1, blk, 0, s>>>(d.nx, d.ny, d.nz, hx, hy, hz, beta, frac, bout, aout);
    else if (d.n() < 1200000 && g4.z <= 65535) go(std::integral_constant<int, 4>{});
    else go(std::integral_constant<int, kRun>{});
    return cudaGetLastError();
}

cudaError_t launch_rk_combine(size_t n, const LevelArrays<double> &a, const LevelArrays<double> &b,
                              const LevelArrays<double> &r, double dt, const LevelArrays<double> &out, cudaStream_t s)
{
    note_launch();
    k_rk_combine<<<vec_grid(n), kRedThreads, 0, s>>>(n, a, b, r, dt, out);
    return cudaGetLastError();
}

cudaError_t launch_momentum_rhs(Dims d, double h, const double *phi, double mu_air, double mu_water, double inv_re,
                                double g, int convect, const LevelArrays<double> &beta, const LevelArrays<double> &u,
                                const LevelArrays<double> &r, double *work, cudaStream_t s)
{
    MomArgs m;
    m.nx = d.nx;
    m.ny = d.ny;
    m.nz = d.nz;
    m.ih = scale2(1.0 / h);
    m.mu_air = mu_air;
    m.dmu = mu_water - mu_air;
    m.inv_re = inv_re;
    m.g = g;
    m.phi = phi;
    m.beta = beta;
    m.u = u;
    m.r = r;
    m.w = work;
    const dim3 g2 = row_grid2(d.nx, d.ny, d.nz), blk = row_block2(d.nx);
    // Where the viscosities are shared (k_mom_parts): not below 70,000 cells and not in rows of less than 20 cells, which
    // leave a warp's lanes idle; in runs of two planes by 128 threads (or a row) below 3 M cells, of kPhiRun by kPhiThreads above.  Both
    // passes with all terms, h a power of two; per cell, 2 and 8 planes, us: 16^3 10, 15, 65; 32^3 13, 16, 68; 48^3 33, 32, 76; 64^3 56, 51,
    // 86; 80^3 121, 117, 157; 96^3 169, 163, 180; 128^3 390, 364, 390; 192x160x224 1260, 1177, 1212; 256^3 3040, 2854, 2767; narrow rows:
    // 16x16x1024 56, 76, 84; 2x600x600 144, 1087, 1101; 33x65x129 104, 97, 106; 33x300x300 1060 and, in 8 planes, 993.  Without the viscous term per cell throughout:
    // 64^3 25, 25, 36; 256^3 1269, 1270, 1289.
    const bool two = d.n() < 3000000;
    dim3 pg, pb;
    row_share_grid(d, pg, pb, two ? kMomRun : kPhiRun, two ? 128 : kPhiThreads);
    const bool share = d.n() >= 70000 && d.nx >= 20;
    auto go = [&](auto conv, auto visc, auto pow2) {
        constexpr bool C = decltype(conv)::value, V = decltype(visc)::value, P = decltype(pow2)::value;
        if constexpr (C || V) {
            note_launch();
            if (!V || !share) k_mom_parts_cells<C, V, P><<<g2, blk, 0, s>>>(m);
            else if (two) k_mom_parts<C, P, kMomRun><<<pg, pb, 0, s>>>(m);
            else k_mom_parts<C, P, kPhiRun><<<pg, pb, 0, s>>>(m);
        }
        note_launch();
        k_mom_combine<C, V, P><<<g2, blk, 0, s>>>(m);
    };
    auto go_p = [&](auto conv, auto visc) {
        // (few cells wait for their chain of operations, on which the exponent shift is the longer one: 16^3 10.2 us, 9.4)
        if (m.ih.ok && d.n() >= 30000) go(conv, visc, BoolTag<true>{});
        else go(conv, visc, BoolTag<false>{});
    };
    const BoolTag<true> yes;
    const BoolTag<false> no;
    if (convect && inv_re != 0.0) go_p(yes, yes);
    else if (convect) go_p(yes, no);
    else if (inv_re != 0.0) go_p(no, yes);
    else go(no, no, yes);
    return cudaGetLastError();
}

cudaError_t launch_half(size_t n, const LevelArrays<double> &a, const LevelArrays<double> &b,
                        const LevelArrays<double> &out, cudaStream_t s)
{
    note_launch();
    k_half<<<vec_grid(n), kRedThreads, 0, s>>>(n, a, b, out);
    return cudaGetLastError();
}

cudaError_t launch_vof_upwind(Dims d, double s_dt_h, const LevelArrays<double> &mask, const LevelArrays<double> &u,
                              const double *phi, double *phi_out, cudaStream_t s)
{
    note_launch();
    k_vof_upwind<<<row_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(d.nx, d.ny, d.nz, s_dt_h, mask, u, phi, phi_out);
    return cudaGetLastError();
}

cudaError_t launch_area_coeffs(size_t n, const LevelArrays<double> &area, const LevelArrays<double> &beta,
                               const LevelArrays<double> &out, cudaStream_t s)
{
    note_launch();
    k_area_coeffs<<<vec_grid(n), kRedThreads, 0, s>>>(n, area, beta, out);
    return cudaGetLastError();
}

cudaError_t launch_divergence_area(Dims d, double scale, const LevelArrays<double> &mask,
                                   const LevelArrays<double> &area, const LevelArrays<double> &u,
                                   const LevelArrays<double> &v, double *rhs, cudaStream_t s)
{
    note_launch();
    const Scale2 sc = scale2(scale);
    // Per cell below 150,000 cells, runs of two planes below 5 M and of kPhiRun above: a block walks its run one plane after the
    // other behind a barrier each.  Per cell, 2 and 8 planes (areas, dt = 1; us): 16^3 3.5, 5.9, 18; 32^3 3.8, 5.9, 18; 512x16x16 6.5,
    // 6.5, 20; 16x512x16 6.6, 9.1, 18; 48^3 7.7, 6.1, 18; 64^3 11, 9.1, 18; 80^3 23, 19, 28; 96^3 32, 27, 28; 128^3 73, 58, 73; 160^3
    // 140, 112, 123; 192x160x224 230, 173, 169; 256^3 550, 422, 400.
    if (d.n() < 150000) {
        k_divergence_area<<<row_grid2(d.nx, d.ny, d.nz), row_block2(d.nx), 0, s>>>(d.nx, d.ny, d.nz, sc, mask, area, u, v,
                                                                                    rhs);
        return cudaGetLastError();
    }
    dim3 grid, block;
    const FluxArea flux{area, u, v};
    if (d.n() < 5000000) {
        row_share_grid(d, grid, block, 2);
        k_divergence_flux<2><<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, sc, mask, flux, rhs);
    } else {
        row_share_grid(d, grid, block);
        k_divergence_flux<kPhiRun><<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, sc, mask, flux, rhs);
    }
    return cudaGetLastError();
}

cudaError_t launch_divergence_mul(Dims d, double scale, const LevelArrays<double> &L, const LevelArrays<double> &B,
                                  const double *wx, const double *wy, const double *wz, double *rhs, cudaStream_t s)
{
    note_launch();
    dim3 grid, block;
    row_share_grid(d, grid, block);
    LevelArrays<double> w{};
    w.bx = const_cast<double *>(wx);
    w.by = const_cast<double *>(wy);
    w.bz = const_cast<double *>(wz);
    k_divergence_flux<kPhiRun><<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, scale2(scale), L, FluxMul{B, w}, rhs);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_faces(Dims d, double h, double dt, const double *bx, const double *by, const double *bz,
                                 const double *p, const double *q, const double *wx, const double *wy,
                                 const double *wz, double *gux, double *guy, double *guz, double *gbx, double *gby,
                                 double *gbz, cudaStream_t s, const LevelArrays<double> *area)
{
    note_launch();
    const Scale2 dt2 = scale2(dt);
    auto go = [&](auto tag) {
        k_adjoint_faces<decltype(tag)::value><<<row_grid(d.nx, d.ny, d.nz), kRowThreads, 0, s>>>(
            d.nx, d.ny, d.nz, h, inv_scale2(h), dt2, bx, by, bz, p, q, wx, wy, wz, gux, guy, guz, gbx, gby, gbz,
            area ? *area : LevelArrays<double>{});
    };
    if (dt2.ok) go(BoolTag<true>{});
    else go(BoolTag<false>{});
    return cudaGetLastError();
}

cudaError_t launch_phi_grad(Dims d, double neg_half_drho, const double *bx, const double *by, const double *bz,
                            const double *gbx, const double *gby, const double *gbz, double *gphi, cudaStream_t s)
{
    note_launch();
    dim3 grid, block;
    row_share_grid(d, grid, block);
    k_phi_grad<<<grid, block, 0, s>>>(d.nx, d.ny, d.nz, neg_half_drho, bx, by, bz, gbx, gby, gbz, gphi);
    return cudaGetLastError();
}


cudaError_t launch_pcg_resid(Dims d, double ih2, const LevelArrays<double> &L, const double *b, const double *p,
                             double *r, float *r32, double *partials, double *dscal, int scale_slot, cudaStream_t s,
                             Split sp, unsigned *pnz)
{
    if (pnz) {  // is p zero everywhere?
        cudaError_t e = cudaMemsetAsync(pnz, 0, sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
        note_launch();
        k_nonzero<<<vec_grid(d.n()), kRedThreads, 0, s>>>((unsigned)d.n(), p, pnz);
    }
    const ResidGrid g = resid_grid(d);
    note_launch();
    k_pcg_resid<<<resid_blocks(g), kRedThreads, 0, s>>>(d.nx, d.ny, d.nz, ih2, L, b, p, r, r32, dscal, scale_slot,
                                                                   partials, sp, g, pnz);
    return cudaGetLastError();
}

template <typename Z>
cudaError_t launch_pcg_dots(size_t n, const double *r, const Z *z, const Z *zo, double *partials, double *dscal,
                            int sz_slot, int so_slot, cudaStream_t s)
{
    const unsigned g = vec_grid(n);
    note_launch();
    k_pcg_dots<Z><<<g, kRedThreads, 0, s>>>((unsigned)n, r, z, zo, dscal, sz_slot, so_slot, partials);
    return cudaGetLastError();
}
cudaError_t launch_pcg_dots32(size_t n, const float *r32, const float *z, const float *zo, double *partials,
                              double *dscal, int sr_slot, int sz_slot, int so_slot, cudaStream_t s)
{
    const unsigned g = red_grid(n);
    note_launch();
    k_pcg_dots32<<<g, kRedThreads, 0, s>>>((unsigned)n, r32, z, zo, dscal, sr_slot, sz_slot, so_slot, partials);
    return cudaGetLastError();
}
template cudaError_t launch_pcg_dots<double>(size_t, const double *, const double *, const double *, double *,
                                             double *, int, int, cudaStream_t);
template cudaError_t launch_pcg_dots<float>(size_t, const double *, const float *, const float *, double *, double *,
                                            int, int, cudaStream_t);

template <typename Z>
cudaError_t launch_pcg_dir(size_t n, const Z *z, double *d, double *dscal, int sz_slot, int so_slot, int first,
                           cudaStream_t s, Split sp, double *partials)
{
    if (sp.half && sizeof(Z) != 4) return cudaErrorInvalidValue;  // FP64 fields are never split
    if (so_slot >= 0 && sz_slot < 0) return cudaErrorInvalidValue;
    note_launch();
    k_pcg_dir<Z><<<sizeof(Z) == 8 ? vec_grid(n) : red_grid(n), kRedThreads, 0, s>>>((unsigned)n, z, d, dscal, sz_slot, so_slot, first, sp, partials);
    return cudaGetLastError();
}
template cudaError_t launch_pcg_dir<double>(size_t, const double *, double *, double *, int, int, int, cudaStream_t,
                                            Split, double *);
template cudaError_t launch_pcg_dir<float>(size_t, const float *, double *, double *, int, int, int, cudaStream_t,
                                           Split, double *);

cudaError_t launch_pcg_apply(Dims d, const LevelArrays<double> &op, const double *dv, double *q, double *partials,
                             double *dscal, cudaStream_t s)
{
    const unsigned g = red_grid(d.n());
    note_launch();
    k_pcg_apply<<<g, kRedThreads, 0, s>>>(d.nx, d.ny, d.nz, op, op.dinv, dv, q, partials, dscal);
    return cudaGetLastError();
}

cudaError_t launch_pcg_update(size_t n, const double *dv, const double *q, double *p, double *r, float *r32,
                              double *partials, double *dscal, int scale_slot, int sd_slot, cudaStream_t s, Split sp)
{
    const unsigned g = red_grid(n);
    if (sd_slot >= 0 && sd_slot == scale_slot) return cudaErrorInvalidValue;  // read and written by the kernel
    note_launch();
    k_pcg_update<<<g, kRedThreads, 0, s>>>((unsigned)n, dv, q, p, r, r32, dscal, scale_slot, sd_slot, partials, sp);
    return cudaGetLastError();
}

int check_read(unsigned long long *first, unsigned long long *count)
{
#ifdef MGP_CHECK
    cudaError_t e = cudaMemcpyFromSymbol(first, g_check_first, sizeof *first);
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(count, g_check_count, sizeof *count);
    const unsigned long long zero = 0;
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_check_first, &zero, sizeof zero);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_check_count, &zero, sizeof zero);
    return e == cudaSuccess ? 1 : -1;
#else
    *first = 0;
    *count = 0;
    return 0;
#endif
}

}  // namespace mg
