// mg_api.cu -- C ABI of the GB300 variable-density pressure projection (host side).
//
// Owns the multigrid hierarchy (one mg_ctx per set of face coefficients), drives
// the V-cycles on the caller's stream, and computes the dense minimum-norm inverse
// of the coarsest grid's operator on the host in FP64 (one banded Cholesky
// factorisation per connected component).
#include <cuda_runtime.h>
#include <omp.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <memory>
#include <string>
#include <type_traits>
#include <vector>

#include "mg_internal.cuh"

using mg::Dims;
using mg::LevelArrays;

namespace {

thread_local std::string g_err;

int fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

#define CK(call)                                                                                     \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ != cudaSuccess)                                                                       \
            return fail(e_ == cudaErrorMemoryAllocation ? MG_ERR_OOM : MG_ERR_CUDA, "%s: %s (%s:%d)", \
                        #call, cudaGetErrorString(e_), __FILE__, __LINE__);                          \
    } while (0)

#define CKS(expr)              \
    do {                       \
        int s_ = (expr);       \
        if (s_ != MG_OK) return s_; \
    } while (0)

}  // namespace

namespace mg {
void set_last_error(const char *msg) { g_err = msg; }
}  // namespace mg

// The coarse tail of a context in one precision: its first level (-1: none) and the kernel's
// arguments but for that level's b and p
template <typename T>
struct TailPlan {
    int first = -1;
    mg::TailArgs<T> a{};
};

struct mg_ctx {
    mg_grid g{};
    mg_opts o{};
    cudaStream_t s = nullptr;
    int nlev = 0;
    std::vector<Dims> dims;
    std::vector<double> hs;
    std::vector<LevelArrays<double>> L64;
    std::vector<LevelArrays<float>> L32;
    TailPlan<double> tail64;
    TailPlan<float> tail32;
    std::vector<double *> palt64;  // second iterate buffer per level for fused sweeps (null if unused)
    std::vector<float *> palt32;
    // conjugate-gradient vectors (krylov = 1): FP64 r, d, q; z, z_old (FP64 cycles) or a
    // second FP32 cycle output (mixed cycles)
    double *kr = nullptr, *kd = nullptr, *kq = nullptr, *kz = nullptr, *kzo = nullptr;
    // CG operator on the finest grid: h^-2 beta in bx/by/bz and h^-2 sum(beta) in dinv
    LevelArrays<double> kop;
    float *ke_alt = nullptr;
    // layout of the finest FP32 iterate / right-hand side (L32[0].p, L32[0].b, ke_alt): colour-split
    // for the per-colour smoother in mixed precision, natural otherwise
    mg::Split split0;
    // fractional face areas (mg_set_face_areas): the open fractions, and 1/rho on the faces as given
    // to mg_setup / mg_update (the operator then uses area * 1/rho); the body velocity on the faces
    // (mg_set_body_velocity)
    bool has_area = false, has_vb = false;
    LevelArrays<double> karea, kbeta, kvb;
    // the time step's scratch (mg_rk2_step): face coefficients of the two stages, u~, u*, phi*
    LevelArrays<double> rk_b1, rk_b2, rk_ut, rk_us, rk_r;
    double *rk_phis = nullptr;
    double *rk_work = nullptr;  // the momentum terms' per-cell fluxes and stresses
    // row records of the levels whose colour passes take them (null elsewhere; rec_level)
    std::vector<double *> rec64;
    std::vector<float *> rec32;
    float *urow0 = nullptr;  // uniform-row values of the finest FP32 level (with split0)
    // banded-row records of the finest FP32 level (with split0 and nx % 8 == 0), the two row
    // counts of the last hierarchy build, and whether its sweeps use the records (more banded
    // rows than uniform ones: a stretched grid)
    float4 *arow0 = nullptr;
    float2 *uinv0 = nullptr;  // the inverse diagonals of the rows with a record, inside and at an x-wall
    unsigned *rowcnt = nullptr;
    // the finest FP32 face arrays in the colour-split layout (with split0 and nx % 8 == 0), read
    // by the colour passes on rows without a record
    LevelArrays<float> sf0;
    bool banded = false;
    // connected regions of the live fine cells: their number; for more than one, each live cell's
    // region number (cc_label, the union-find labels otherwise), the cells per region (device
    // cc_cnt, host hcnt) and the per-region sums of the current solve (cc_sum, host hsum)
    int ncomp = 1, ncomp_raw = 0;
    int *cc_label = nullptr, *cc_roots = nullptr;
    uint8_t *open_bits = nullptr;  // open low faces of each fine cell at the last labelling
    unsigned *cc_ctr = nullptr;
    unsigned *pnz = nullptr;  // the zero test of a solve's initial guess
    double *cc_sum = nullptr, *cc_cnt = nullptr, *cc_part = nullptr;
    std::vector<double> hcnt, hsum;
    bool incompat = false;      // the current solve's rhs failed the compatibility test
    double incompat_mean = 0.0, incompat_rms = 0.0;
    double *b0 = nullptr;       // compatible fine rhs of the current solve
    double *rhs_tmp = nullptr;  // projection / adjoint right-hand side
    double *qbuf = nullptr;     // adjoint solution when the caller passes none
    double *M = nullptr;        // coarsest dense inverse (device, ncoarse^2)
    int ncoarse = 0;
    double *partials = nullptr; // reduction partials
    double *dscal = nullptr;    // device scalars (mg::Scal)
    double *hscal = nullptr;    // pinned host mirror of dscal
    // pinned staging of the coarsest grid's inverse: its three face arrays (3 ncoarse), the
    // inverse (ncoarse^2), then the two row counters of the finest uniform / banded rows
    double *hcoarse = nullptr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    cudaEvent_t ev_h = nullptr;  // the coarsest faces and the scalars reached the host
    // the coarse-grid correction of one V-cycle (everything below the finest level) as a
    // CUDA graph per precision, captured on first use on a private stream
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t coarse_graph[2] = {nullptr, nullptr};  // [0] FP64, [1] FP32
    unsigned long long coarse_graph_kernels[2] = {0, 0};   // kernel nodes per graph (launch counter)
    bool capturing = false;
    float ms_setup = 0.f;
    double nlive = 0.0;
    std::vector<void *> allocs;
    // profiling (opts.profile): event pairs recorded around finest-grid kernels
    std::vector<cudaEvent_t> pev;
    std::vector<int> pgroup;
    size_t pused = 0;

    template <typename T>
    int alloc(T **p, size_t n)
    {
        void *q = nullptr;
        cudaError_t e = cudaMalloc(&q, n * sizeof(T) + 16);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(MG_ERR_OOM, "cudaMalloc of %zu bytes failed: %s", n * sizeof(T), cudaGetErrorString(e));
        }
        allocs.push_back(q);
        *p = (T *)q;
        return MG_OK;
    }
    ~mg_ctx()
    {
        for (void *q : allocs) cudaFree(q);
        if (hscal) cudaFreeHost(hscal);
        if (hcoarse) cudaFreeHost(hcoarse);
        if (ev_h) cudaEventDestroy(ev_h);
        if (ev0) cudaEventDestroy(ev0);
        if (ev1) cudaEventDestroy(ev1);
        for (cudaEvent_t e : pev) cudaEventDestroy(e);
        for (cudaGraphExec_t g : coarse_graph)
            if (g) cudaGraphExecDestroy(g);
        if (cap_stream) cudaStreamDestroy(cap_stream);
    }
};

namespace {

// every device array starts on a 16-byte boundary (the kernels move aligned pairs); null passes
bool aligned16(std::initializer_list<const void *> ptrs)
{
    for (const void *q : ptrs)
        if (reinterpret_cast<uintptr_t>(q) % 16 != 0) return false;
    return true;
}

// most disconnected fluid regions a context handles (per-region sums and counts: 1 MB)
constexpr int kMaxRegions = 1 << 16;

bool forces_ok(const mg_forces *f)
{
    return f && std::isfinite(f->g) && std::isfinite(f->inv_re) && f->inv_re >= 0.0 && std::isfinite(f->mu_air) &&
           f->mu_air >= 0.0 && std::isfinite(f->mu_water) && f->mu_water >= 0.0;
}

bool grid_ok(const mg_grid *g)
{
    return g && g->nx >= 1 && g->ny >= 1 && g->nz >= 1 && g->h > 0.0 && std::isfinite(g->h) &&
           (double)g->nx * g->ny * g->nz < 2147483647.0;
}

// dot product with four partial sums (lets the compiler keep several FMA chains in flight)
inline double dot4(const double *a, const double *b, int n)
{
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int q = 0;
    for (; q + 4 <= n; q += 4) {
        s0 += a[q] * b[q];
        s1 += a[q + 1] * b[q + 1];
        s2 += a[q + 2] * b[q + 2];
        s3 += a[q + 3] * b[q + 3];
    }
    for (; q < n; q++) s0 += a[q] * b[q];
    return (s0 + s1) + (s2 + s3);
}

// ---------------------------------------------------------------------------
// Coarsest-grid dense inverse (host, FP64): the Moore-Penrose inverse of the operator A, for each
// connected component of >= 2 cells from one banded Cholesky factorisation; isolated cells get
// zero rows and columns.
//
// With the cells numbered along the grid's longest axis last, L = -A on a component couples cells at most a
// cross-section of the grid apart: a band of some n^(2/3).  L + a e e^T (e: one of its cells, a: 100 mean
// diagonal entries) is positive definite with the same band, and for a right-hand side of zero sum its
// solution is L's that is zero at that cell; so with X its inverse, L^+ = P X P, P = I - 1 1^T / m.
// That takes n^2 bandwidth products for the columns of X instead of the n^3 of a dense
// factorisation (of the matrix shifted by a multiple of 1 1^T, as it was): 512 cells 2.55 -> 0.46 ms on 16 Arm
// cores, 360 cells 1.11 -> 0.28 ms, 216 cells 0.43 -> 0.14 ms, 64 cells 58 -> 28 us.  Its error against 113 bits is
// below 1e-14 (relative, density ratio 1000): layered air and water 5e-16 to 3e-15 (dense: 2e-14 to
// 1e-12), a smooth interface 6e-16 to 4e-15 (3e-16 to 4e-14), random densities 8e-16 to 7e-15 (4e-16 to 1e-14).
// ---------------------------------------------------------------------------
constexpr int kInvCols = 8;  // columns of X solved together (the loops over them are the vector loops)

int coarse_inverse(int nx, int ny, int nz, double h, const double *bx, const double *by, const double *bz, double *M)
{
    const int n = nx * ny * nz;
    const double ih2 = 1.0 / (h * h);
    const int dim[3] = {nx, ny, nz}, stride[3] = {1, nx, nx * ny};
    const double *face[3] = {bx, by, bz};
    // conductance of the low face of cell c along an axis; 0 where closed or on the wall (a NaN is neither)
    auto low = [&](int c, const int *idx, int ax) {
        return idx[ax] > 0 && !(face[ax][c] <= 0.0) ? face[ax][c] * ih2 : 0.0;
    };
    // cells in an order with the longest axis slowest: pos[c] and its inverse
    int ax[3] = {0, 1, 2};
    std::sort(ax, ax + 3, [&](int a, int b) { return dim[a] != dim[b] ? dim[a] < dim[b] : a < b; });
    std::vector<int> order;
    order.reserve(n);
    for (int w = 0; w < dim[ax[2]]; w++)
        for (int v = 0; v < dim[ax[1]]; v++)
            for (int u = 0; u < dim[ax[0]]; u++) order.push_back(u * stride[ax[0]] + v * stride[ax[1]] + w * stride[ax[2]]);
    // the couplings of each cell: its low faces (to c - stride) and, mirrored, its high ones
    std::vector<std::array<double, 6>> g(n, std::array<double, 6>{});
    for (int c = 0; c < n; c++) {
        const int idx[3] = {c % nx, (c / nx) % ny, c / (nx * ny)};
        for (int a = 0; a < 3; a++) {
            const double v = low(c, idx, a);
            if (v == 0.0) continue;
            g[c][2 * a] = v;
            g[c - stride[a]][2 * a + 1] = v;
        }
    }
    auto neighbour = [&](int c, int f) { return (f & 1) ? c + stride[f / 2] : c - stride[f / 2]; };
    std::fill(M, M + (size_t)n * n, 0.0);
    std::vector<int> comp(n, -1), pos(n, 0), mem, stack;
    for (int s0 = 0, cid = 0; s0 < n; s0++) {
        if (comp[s0] >= 0) continue;
        stack.assign(1, s0);
        comp[s0] = cid;
        int m = 0;
        while (!stack.empty()) {
            const int c = stack.back();
            stack.pop_back();
            m++;
            for (int f = 0; f < 6; f++)
                if (g[c][f] != 0.0 && comp[neighbour(c, f)] < 0) {
                    comp[neighbour(c, f)] = cid;
                    stack.push_back(neighbour(c, f));
                }
        }
        const int id = cid++;
        if (m < 2) continue;
        mem.clear();
        for (int c : order)
            if (comp[c] == id) {
                pos[c] = (int)mem.size();
                mem.push_back(c);
            }
        int bw = 0;
        double tr = 0.0;
        for (int c : mem)
            for (int f = 0; f < 6; f++)
                if (g[c][f] != 0.0) {
                    bw = std::max(bw, std::abs(pos[c] - pos[neighbour(c, f)]));
                    tr += g[c][f];
                }
        if (!std::isfinite(tr)) return fail(MG_ERR_ARG, "coarsest-grid operator is not finite");
        // banded S = L + a e e^T, row i at S[i * (bw + 1)], S[i][d] = S(i, i - bw + d); the cell e is the
        // best connected one
        const int ld = bw + 1;
        std::vector<double> S((size_t)m * ld, 0.0), T((size_t)m * ld, 0.0);
        int e = 0;
        for (int i = 0; i < m; i++) {
            const int c = mem[i];
            double d = 0.0;
            for (int f = 0; f < 6; f++) {
                if (g[c][f] == 0.0) continue;
                d += g[c][f];
                const int j = pos[neighbour(c, f)];
                if (j < i) S[(size_t)i * ld + bw - (i - j)] = -g[c][f];
            }
            S[(size_t)i * ld + bw] = d;
            if (d > S[(size_t)e * ld + bw]) e = i;
        }
        S[(size_t)e * ld + bw] += 100.0 * (tr / m);
        // Cholesky in place (C lower), rows in turn
        for (int i = 0; i < m; i++) {
            double *ri = &S[(size_t)i * ld];
            for (int j = std::max(0, i - bw); j <= i; j++) {
                const double *rj = &S[(size_t)j * ld];
                const int k0 = std::max({0, i - bw, j - bw});  // the columns both rows hold
                const double v = ri[bw - (i - j)] - dot4(ri + bw - (i - k0), rj + bw - (j - k0), j - k0);
                if (j < i) {
                    ri[bw - (i - j)] = v / rj[bw];
                } else {
                    if (!(v > 0.0)) return fail(MG_ERR_ARG, "coarsest-grid operator is not semi-definite");
                    ri[bw] = std::sqrt(v);
                }
            }
        }
        // its transpose, T[i][d] = C(i + d, i)
        for (int i = 0; i < m; i++)
            for (int j = std::max(0, i - bw); j <= i; j++) T[(size_t)j * ld + (i - j)] = S[(size_t)i * ld + bw - (i - j)];
        // X = S^-1 into M, kInvCols columns at a time: C w = e_j, then C^T x = w from below up to the diagonal;
        // X is symmetric, so column j below the diagonal is also row j beyond it
        const int groups = (m + kInvCols - 1) / kInvCols;
        std::vector<double> r(m);
        double all = 0.0;
        // a part per thread, none of it read before it is written (clearing one per thread of a large host, most of them
        // without a group of columns, took longer than the columns)
        const int team = m > 128 ? std::min(omp_get_max_threads(), groups) : 1;
        const std::unique_ptr<double[]> work(new double[(size_t)team * m * kInvCols]);
#pragma omp parallel num_threads(team)
        {
            double *const W = work.get() + (size_t)omp_get_thread_num() * m * kInvCols;  // rows j0 .. m - 1
#pragma omp for schedule(dynamic, 1)
            for (int gr = 0; gr < groups; gr++) {
                const int j0 = gr * kInvCols, nc = std::min(kInvCols, m - j0);
                for (int i = j0; i < m; i++) {
                    double acc[kInvCols];
                    for (int q = 0; q < kInvCols; q++) acc[q] = i == j0 + q ? 1.0 : 0.0;
                    const double *ci = &S[(size_t)i * ld];
                    const int k0 = std::max(j0, i - bw);
                    const double *w = &W[(size_t)(k0 - j0) * kInvCols];
                    for (int k = k0; k < i; k++, w += kInvCols) {
                        const double f = ci[bw - (i - k)];
                        for (int q = 0; q < kInvCols; q++) acc[q] -= f * w[q];
                    }
                    double *wi = &W[(size_t)(i - j0) * kInvCols];
                    for (int q = 0; q < kInvCols; q++) wi[q] = acc[q] / ci[bw];
                }
                for (int i = m - 1; i >= j0; i--) {
                    double acc[kInvCols];
                    double *wi = &W[(size_t)(i - j0) * kInvCols];
                    for (int q = 0; q < kInvCols; q++) acc[q] = wi[q];
                    const double *ti = &T[(size_t)i * ld];
                    const int d1 = std::min(m - 1 - i, bw);
                    const double *x = wi + kInvCols;
                    for (int d = 1; d <= d1; d++, x += kInvCols) {
                        const double f = ti[d];
                        for (int q = 0; q < kInvCols; q++) acc[q] -= f * x[q];
                    }
                    for (int q = 0; q < kInvCols; q++) wi[q] = acc[q] / ti[0];
                }
                for (int q = 0; q < nc; q++) {
                    double *row = M + (size_t)mem[j0 + q] * n;
                    for (int i = j0 + q; i < m; i++) row[mem[i]] = W[(size_t)(i - j0) * kInvCols + q];
                }
            }
            // the lower triangle from the upper one, and the rows' means
#pragma omp for schedule(static)
            for (int i = 0; i < m; i++) {
                double *row = M + (size_t)mem[i] * n, s = 0.0;
                for (int j = 0; j < i; j++) row[mem[j]] = M[(size_t)mem[j] * n + mem[i]];
                for (int j = 0; j < m; j++) s += row[mem[j]];
                r[i] = s / m;
            }
#pragma omp single
            {
                for (int i = 0; i < m; i++) all += r[i];
                all /= m;
            }
            // A^+ = -P X P
#pragma omp for schedule(static)
            for (int i = 0; i < m; i++) {
                double *row = M + (size_t)mem[i] * n;
                for (int j = 0; j < m; j++) row[mem[j]] = -((row[mem[j]] - r[i]) - (r[j] - all));
            }
        }
    }
    return MG_OK;
}

template <typename T>
int level_alloc(mg_ctx *c, LevelArrays<T> &L, size_t n, bool with_bp)
{
    CKS(c->alloc(&L.bx, n));
    CKS(c->alloc(&L.by, n));
    CKS(c->alloc(&L.bz, n));
    CKS(c->alloc(&L.dinv, n));
    if (with_bp) {
        CKS(c->alloc(&L.b, n));
        CKS(c->alloc(&L.p, n));
    }
    return MG_OK;
}

// Profiling: an event pair around one finest-grid kernel launch (no-op unless enabled).
struct ProfScope {
    mg_ctx *c;
    int slot = -1;
    ProfScope(mg_ctx *c_, int group, bool on) : c(c_)
    {
        if (!on || !c->o.profile || c->capturing || c->pused + 2 > c->pev.size()) return;
        slot = (int)c->pused;
        c->pused += 2;
        c->pgroup[slot / 2] = group;
        cudaEventRecord(c->pev[slot], c->s);
    }
    ~ProfScope()
    {
        if (slot >= 0) cudaEventRecord(c->pev[slot + 1], c->s);
    }
};

// ---------------------------------------------------------------------------
// V-cycle on level l (p updated in place): pre-smooth nu1 x (red, black),
// residual + restriction, coarse correction (recursion or exact solve),
// prolongation, post-smooth nu2 x (black, red).
// ---------------------------------------------------------------------------
template <typename T>
T *palt_of(mg_ctx *c, int l);
template <>
double *palt_of<double>(mg_ctx *c, int l) { return c->palt64.empty() ? nullptr : c->palt64[l]; }
template <>
float *palt_of<float>(mg_ctx *c, int l) { return c->palt32.empty() ? nullptr : c->palt32[l]; }

template <typename T>
const TailPlan<T> &tail_of(const mg_ctx *c);
template <>
const TailPlan<double> &tail_of<double>(const mg_ctx *c) { return c->tail64; }
template <>
const TailPlan<float> &tail_of<float>(const mg_ctx *c) { return c->tail32; }

// fused sweeps pay off on levels with at least one full 32 x 8 tile and 8 planes
bool fused_level(const Dims &d) { return d.nx >= 32 && d.ny >= 8 && d.nz >= 8; }

template <typename T>
const T *rec_of(const mg_ctx *c, int l);
template <>
const double *rec_of<double>(const mg_ctx *c, int l) { return c->rec64.empty() ? nullptr : c->rec64[l]; }
template <>
const float *rec_of<float>(const mg_ctx *c, int l) { return c->rec32.empty() ? nullptr : c->rec32[l]; }

template <typename T>
bool use_fused(const mg_ctx *c, int l)
{
    if (!fused_level(c->dims[l]) || l == c->nlev - 1) return false;
    if (c->o.smoother == 2) return true;
    if (c->o.smoother == 3) return sizeof(T) == 4;
    return false;  // auto and 1: one pass per colour (the measured fastest on GB300)
}

// FP32 levels in auto mode sweep with the TMA-staged kernel where its layout allows
template <typename T>
bool tma_level(const mg_ctx *c, int l)
{
    return sizeof(T) == 4 && c->o.smoother == 3 && mg::tma_sweep_supported(c->dims[l]);
}
inline cudaError_t launch_sweep_tma(Dims d, float h2, const LevelArrays<float> &L, const float *b, const float *pold,
                                    float *pnew, int first, double *dscal, cudaStream_t s)
{
    return mg::launch_rb_sweep_tma(d, h2, L, b, pold, pnew, first, dscal, s);
}
inline cudaError_t launch_sweep_tma(Dims, double, const LevelArrays<double> &, const double *, const double *,
                                    double *, int, double *, cudaStream_t)
{
    return cudaErrorNotSupported;  // FP64 levels never take this path
}

template <typename T>
int coarse_correction_graph(mg_ctx *c, const std::vector<LevelArrays<T>> &L);

// The coarse tail in precision T: its first level (the largest below the finest and above the coarsest
// whose slabs, with those of all levels below, fit in the shared memory of a cluster's CTAs; -1 if
// none, or if the coarsest grid is larger than a cluster should solve) and its layout.
template <typename T>
int tail_layout(const mg_ctx *c, const std::vector<LevelArrays<T>> &L, int ctas, mg::TailArgs<T> &a)
{
    if (c->ncoarse > mg::kTailCoarse) return -1;
    for (int l = 1; l + 1 < c->nlev; l++) {
        if (c->nlev - l > mg::kTailMaxLevels || c->dims[l].n() > mg::kTailCellsMax) continue;
        a.nlev = c->nlev - l;
        a.ctas = ctas;
        size_t n = 0;  // elements per CTA
        bool fits = true;
        for (int q = 0; q < a.nlev; q++) {
            const Dims d = c->dims[l + q];
            mg::TailLevel<T> &v = a.lev[q];
            v.nx = d.nx;
            v.ny = d.ny;
            v.nz = d.nz;
            v.P = (d.nz + ctas - 1) / ctas;
            v.h2 = (T)(c->hs[l + q] * c->hs[l + q]);
            v.ih2 = (T)(1.0 / (c->hs[l + q] * c->hs[l + q]));
            v.sh2 = mg::scale2((double)v.h2);
            v.L = L[l + q];
            v.fnx = mg::make_fastdiv((unsigned)d.nx);
            v.fhx = mg::make_fastdiv((unsigned)std::max(d.nx / 2, 1));
            v.fny = mg::make_fastdiv((unsigned)d.ny);
            v.fP = mg::make_fastdiv((unsigned)v.P);
            const size_t plane = (size_t)d.nx * d.ny, slab = plane * v.P;
            const bool smoothed = q + 1 < a.nlev;
            fits = fits && (!smoothed || slab <= 2 * (size_t)mg::kTailCells * mg::kTailThreads);
            unsigned *const off[6] = {&v.op, &v.ob, &v.ox, &v.oy, &v.oz, &v.od};
            for (int f = 0; f < (smoothed ? 6 : 2); f++) {
                const size_t pad = smoothed && f == 0 ? d.nx / 2 : 0;  // the row of zeros before p
                *off[f] = (unsigned)std::min<size_t>(n + pad, 0xffffffffu);
                n += slab + pad + (smoothed ? d.nx : 0) + (f == 4 ? plane : 0);  // and after each colour
            }
        }
        n = (n * sizeof(T) + 15) / 16 * 16;
        a.sb_bytes = (unsigned)std::min<size_t>(n, 0xffffffffu);
        a.smem = n + (size_t)c->ncoarse * sizeof(double);
        if (fits && a.smem <= mg::kTailSmem) return l;
    }
    return -1;
}

template <typename T>
int tail_start(const mg_ctx *c, const std::vector<LevelArrays<T>> &L, mg::TailArgs<T> &a)
{
    const int ctas = c->o.coarse_tail ? mg::tail_ctas<T>() : 0;
    return ctas > 0 ? tail_layout<T>(c, L, ctas, a) : -1;
}

// zero: p is taken as zero on entry (a cycle from a zero guess): the coarsest solve overwrites it,
// the coarse tail zeroes it in its kernel, and the per-colour passes start with a pass that reads
// no iterate, so no separate clearing pass is needed (the fused sweeps and nu1 = 0 clear it first)
// again: the last thing done to p was a cycle with this b.  Its last pass was the red one of a
// post-smoothing sweep, so this cycle's first red pass would compute the red values that stand there
// from the same black ones: it is left out (the same iterate bit for bit, one of the finest level's
// 2 (nu1 + nu2) passes less)
// part: the cycle in two calls, the first making its first `stop` pre-smoothing passes alone, the second
// the rest after those `done` (colour passes; a cycle of fused sweeps is not divided); gate: for the first call's
// passes from an iterate (FP64, natural layout)
struct CyclePart {
    int done = 0, stop = -1;
    mg::Gate gate = {};
};
template <typename T>
int vcycle(mg_ctx *c, const std::vector<LevelArrays<T>> &L, int l, const T *b, T *p, bool zero = false,
           bool again = false, CyclePart part = {})
{
    cudaStream_t s = c->s;
    const Dims d = c->dims[l];
    if (l == c->nlev - 1) {
        CK(mg::launch_coarse_solve<T>(c->ncoarse, c->M, b, p, s));
        return MG_OK;
    }
    const TailPlan<T> &tail = tail_of<T>(c);
    if (l == tail.first && zero) {  // this level and all below: one cluster, one launch
        mg::TailArgs<T> a = tail.a;
        a.lev[0].L.b = const_cast<T *>(b);
        a.lev[0].L.p = p;
        CK(mg::launch_tail<T>(a, s));
        return MG_OK;
    }
    const T h2 = (T)(c->hs[l] * c->hs[l]);
    const T ih2 = (T)(1.0 / (c->hs[l] * c->hs[l]));
    const bool fine = (l == 0);
    const bool fused = use_fused<T>(c, l) && palt_of<T>(c, l) != nullptr;
    const mg::Split sp = (sizeof(T) == 4 && l == 0) ? c->split0 : mg::Split{};
    const float *urow = (sizeof(T) == 4 && l == 0) ? c->urow0 : nullptr;
    const float4 *arow = (sizeof(T) == 4 && l == 0 && c->banded) ? c->arow0 : nullptr;
    const float2 *uinv = (sizeof(T) == 4 && l == 0) ? c->uinv0 : nullptr;
    const T *rec = rec_of<T>(c, l);
    T *cur = p, *alt = palt_of<T>(c, l);
    // plane order of the finest colour passes (pass_order = 1): each group of passes alternates
    // descending, ascending, ... so that every pass starts on the planes its predecessor (or the
    // prolongation, ascending) touched last, which are still in L2; the restriction that follows
    // the last (ascending) pre-smoothing pass runs descending
    const bool alternate = c->o.pass_order == 1 && sp.half;
    int npass = 0;
    // the first pass reads no iterate when p starts at zero; otherwise clear p first
    const bool zpass = zero && !fused && c->o.nu1 >= 1;
    if (zero && !zpass) CK(cudaMemsetAsync(p, 0, d.n() * sizeof(T), s));
    // two passes as one launch where the red values between them are not needed again
    const bool both = zpass && !fine && c->o.nu1 >= 2 && sizeof(T) == 4;
    const bool up = sizeof(T) == 4 && !fine && !fused && c->o.nu2 >= 1 && d.n() <= mg::kUpCells;
    const bool skip = again && !fused && c->o.nu1 >= 1 && c->o.nu2 >= 1;  // the first red pass
    // one colour pass; zp: p is zero
    auto pass = [&](int colour, bool zp) -> int {
        if (sp.half) {
            if constexpr (std::is_same<T, float>::value)
                CK(mg::launch_smooth_split(d, h2, L[l], b, cur, colour, s, urow, arow, uinv, alternate ? (npass + 1) & 1 : 0, zp,
                                           &c->sf0));
        } else {
            CK(mg::launch_smooth<T>(d, h2, L[l], b, cur, colour, s, zp, rec, part.gate));
        }
        npass++;
        return MG_OK;
    };
    // one red-black sweep, `first` colour first
    auto sweep = [&](int first) -> int {
        ProfScope ps(c, MG_PROF_SMOOTH, fine);
        if (!fused) {
            CKS(pass(first, false));
            return pass(first ^ 1, false);
        }
        if (tma_level<T>(c, l))
            CK(launch_sweep_tma(d, h2, L[l], b, cur, alt, first, c->dscal, s));
        else
            CK(mg::launch_rb_sweep<T>(d, h2, L[l], b, cur, alt, first, s));
        std::swap(cur, alt);
        return MG_OK;
    };
    for (int it = 0; it < c->o.nu1; it++) {
        if (fused) {
            CKS(sweep(0));
            continue;
        }
        ProfScope ps(c, MG_PROF_SMOOTH, fine && !(skip && it == 0));  // (a lone black pass is no sweep)
        for (int colour = 0; colour < 2; colour++) {
            const int m = 2 * it + colour;
            if (both && m < 2) {
                if constexpr (std::is_same<T, float>::value)
                    if (m == 0) CK(mg::launch_smooth_first(d, h2, L[l], b, cur, s));
                continue;
            }
            if (m < part.done) npass++;
            else if ((m > 0 || !skip) && (part.stop < 0 || m < part.stop)) CKS(pass(colour, m == 0 && zpass));
        }
    }
    if (part.stop >= 0) return MG_OK;
    const LevelArrays<T> &C = L[l + 1];
    {
        ProfScope ps(c, MG_PROF_RESTRICT, fine);
        // descending after an ascending last pass (an even number of passes, the last ascending)
        const int rrev = alternate && npass > 0 && (npass & 1) == 0 ? 1 : 0;
        const LevelArrays<T> *S = nullptr;
        if constexpr (std::is_same<T, float>::value) S = l == 0 ? &c->sf0 : nullptr;
        CK(mg::launch_restrict<T>(d, ih2, L[l], b, cur, C.b, s, sp, urow, arow, rrev, S));
    }
    npass = 0;
    {
        ProfScope ps(c, MG_PROF_COARSE, fine);
        if (fine && c->o.coarse_graph && !c->capturing)
            CKS(coarse_correction_graph<T>(c, L));
        else
            CKS(vcycle<T>(c, L, l + 1, C.b, C.p, true));
    }
    {
        ProfScope ps(c, MG_PROF_PROLONG, fine);
        if (up) {
            if constexpr (std::is_same<T, float>::value)
                CK(mg::launch_prolong_black(d, h2, L[l], b, C.p, cur, s));
        } else if (c->o.nu2 >= 1)  // a black pass follows: the red cells alone
            CK(mg::launch_prolong_red<T>(d, C.p, L[l].dinv, cur, s, sp, urow, arow));
        else
            CK(mg::launch_prolong<T>(d, C.p, L[l].dinv, cur, s, sp, urow));
    }
    for (int it = 0; it < c->o.nu2; it++) {
        if (up && it == 0) CKS(pass(0, false));
        else CKS(sweep(1));
    }
    if (cur != p) CK(cudaMemcpyAsync(p, cur, d.n() * sizeof(T), cudaMemcpyDeviceToDevice, s));
    return MG_OK;
}

// The coarse-grid correction of a V-cycle on the finest level: zero the level-1
// correction, V-cycle levels 1..coarsest.  Its buffers are the context's own, so one
// captured graph per precision serves every call; it is launched on the caller's stream.
template <typename T>
int coarse_correction_graph(mg_ctx *c, const std::vector<LevelArrays<T>> &L)
{
    const int slot = sizeof(T) == 4 ? 1 : 0;
    if (!c->coarse_graph[slot]) {
        if (!c->cap_stream) CK(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
        cudaStream_t user = c->s;
        c->s = c->cap_stream;
        c->capturing = true;
        cudaGraph_t g = nullptr;
        int st = MG_OK;
        const unsigned long long k0 = mg::launch_count();
        cudaError_t e = cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            st = [&]() -> int {
                CKS(vcycle<T>(c, L, 1, L[1].b, L[1].p, true));
                return MG_OK;
            }();
            e = cudaStreamEndCapture(c->cap_stream, &g);
        }
        c->s = user;
        c->capturing = false;
        c->coarse_graph_kernels[slot] = mg::launch_count() - k0;
        if (st != MG_OK) {
            if (g) cudaGraphDestroy(g);
            return st;
        }
        if (e != cudaSuccess) return fail(MG_ERR_CUDA, "coarse-grid graph capture failed: %s", cudaGetErrorString(e));
        e = cudaGraphInstantiate(&c->coarse_graph[slot], g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            c->coarse_graph[slot] = nullptr;
            return fail(MG_ERR_CUDA, "coarse-grid graph instantiation failed: %s", cudaGetErrorString(e));
        }
    }
    CK(cudaGraphLaunch(c->coarse_graph[slot], c->s));
    for (unsigned long long k = 0; k < c->coarse_graph_kernels[slot]; k++) mg::note_kernel_launch();
    return MG_OK;
}

// read the device scalars into the pinned mirror (one stream sync); report a kernel whose
// bounded wait expired
int check_scalars(mg_ctx *c);
int read_scalars(mg_ctx *c)
{
    CK(cudaMemcpyAsync(c->hscal, c->dscal, mg::S_COUNT * sizeof(double), cudaMemcpyDeviceToHost, c->s));
    CK(cudaStreamSynchronize(c->s));
    return check_scalars(c);
}
// the same in two steps, with work queued between them that the host does not wait for
int queue_scalars(mg_ctx *c)
{
    CK(cudaMemcpyAsync(c->hscal, c->dscal, mg::S_COUNT * sizeof(double), cudaMemcpyDeviceToHost, c->s));
    CK(cudaEventRecord(c->ev_h, c->s));
    return MG_OK;
}
int wait_scalars(mg_ctx *c)
{
    CK(cudaEventSynchronize(c->ev_h));
    return check_scalars(c);
}

// the scalars just read: report a kernel whose bounded wait expired (and clear its flag)
int check_scalars(mg_ctx *c)
{
    if (c->hscal[mg::S_ERR] != 0.0) {
        CK(cudaMemsetAsync(c->dscal + mg::S_ERR, 0, sizeof(double), c->s));
        return fail(MG_ERR_CUDA, "a pipelined smoothing kernel's bounded wait expired (data not delivered)");
    }
    return MG_OK;
}

void stats_begin(mg_stats *st)
{
    if (!st) return;
    st->cycles = 0;
    st->rel_resid = 0.0;
    st->rhs_norm = 0.0;
    st->rhs_mean_removed = 0.0;
    for (double &v : st->resid_hist) v = 0.0;
}

// The compatible right-hand side b0 of a solve (Eq. neumann with Eq. pois: one constant per
// connected fluid region spans A's null space, so b is solvable only with zero sum on each): the
// rhs minus its mean on each region, 0 on dead cells; dscal gets S_SUM_B (the sum over the live
// cells) and S_NB2 (||b0||^2).  The region sums go to the host with the next read_scalars.
int prepare_rhs(mg_ctx *c, const double *rhs)
{
    const Dims d = c->dims[0];
    if (c->ncomp > 1) {
        CK(mg::launch_comp_center(d.n(), rhs, c->cc_label, c->ncomp, c->cc_sum, c->cc_cnt, c->b0, c->partials,
                                  c->dscal, mg::S_NB2, mg::S_SUM_B, c->s, c->cc_part));
        c->hsum.resize(c->ncomp);
        CK(cudaMemcpyAsync(c->hsum.data(), c->cc_sum, c->ncomp * sizeof(double), cudaMemcpyDeviceToHost, c->s));
    } else {
        CK(mg::launch_rhs_prepare(d, rhs, c->L64[0].dinv, c->b0, c->partials, c->dscal, c->s));
    }
    return MG_OK;
}

// After the first read_scalars of a solve: the rhs is incompatible when the mean it had on some
// region exceeds kIncompatible times its RMS over the live cells (both before the removal):
// sum b^2 = ||b0||^2 + sum over regions of (cells x mean^2).
constexpr double kIncompatible = 1e-8;
void check_compatible(mg_ctx *c)
{
    c->incompat = false;
    const double n = c->nlive, nb2 = c->hscal[mg::S_NB2];
    if (!(n > 0.0) || !std::isfinite(nb2)) return;
    double worst = 0.0, sq = nb2;
    if (c->ncomp > 1) {
        for (int m = 0; m < c->ncomp; m++) {
            const double mean = c->hsum[m] / c->hcnt[m];
            sq += c->hcnt[m] * mean * mean;
            worst = std::max(worst, std::fabs(mean));
        }
    } else {
        const double mean = c->hscal[mg::S_SUM_B] / n;
        sq += n * mean * mean;
        worst = std::fabs(mean);
    }
    const double rms = std::sqrt(sq / n);
    c->incompat = worst > kIncompatible * rms;
    c->incompat_mean = worst;
    c->incompat_rms = rms;
}

// a solve that converged on an incompatible rhs reports it (p is the solution for the rhs with
// its region means removed)
int final_status(mg_ctx *c, int status)
{
    if (status == MG_OK && c->incompat)
        return fail(MG_ERR_INCOMPATIBLE,
                    "right-hand side incompatible with the Neumann problem: mean %.3e on a fluid region against an "
                    "RMS of %.3e; the mean of each region was removed and the solve converged",
                    c->incompat_mean, c->incompat_rms);
    return status;
}

// p -= its mean over each fluid region (live cells), dead cells 0; with one region the mean is
// dscal[S_SUM_P] / nlive, from the last residual pass or (sum) summed here
int remove_p_mean(mg_ctx *c, double *p, bool sum)
{
    const Dims d = c->dims[0];
    if (c->ncomp > 1)
        CK(mg::launch_comp_center(d.n(), p, c->cc_label, c->ncomp, c->cc_sum, c->cc_cnt, p, c->partials, c->dscal,
                                  -1, -1, c->s, c->cc_part));
    else {
        if (sum) CK(mg::launch_sum_p(d, c->L64[0].dinv, p, c->partials, c->dscal, c->s));
        CK(mg::launch_sub_mean_p(d, c->L64[0].dinv, p, c->dscal, c->s));
    }
    return MG_OK;
}

// Colour passes of the next cycle to queue before the host waits for a residual: the GPU would stand idle for the
// copy, the host's wait and the next launch, some 13 us an iteration (a tenth of one at 64^3).  As many as take some
// 20 us (a pass moves about three values per cell at 4 TB/s), at least one; none where the cycle is not
// made of colour passes or is timed by parts.  Anything from 10 to 40 us gives the same: mixed CG solves of 32^3, 64^3, 96^3 and 128^3
// with none ahead 1176, 1820, 2280 and 3074 us, with 5 us of passes 1152, 1805, 2259, 3027, 10 us 1140, 1777, 2251, 3025, 20 us 1145,
// 1782, 2260, 3023, 40 us 1145, 1777, 2266, 3056.
int passes_ahead(const mg_ctx *c)
{
    const bool mixed = c->o.prec == MG_MIXED;
    if (c->o.profile || c->nlev < 2 || c->o.nu1 < 1 || (mixed ? use_fused<float>(c, 0) : use_fused<double>(c, 0))) return 0;
    const double pass_us = std::max(3.0, (double)c->dims[0].n() * (mixed ? 4 : 8) * 3.0 / 4e6);
    return std::max(1, std::min(2 * c->o.nu1, (int)(20.0 / pass_us)));
}

int solve_impl(mg_ctx *c, const double *rhs, double *p, double tol, mg_stats *st)
{
    cudaStream_t s = c->s;
    const Dims d = c->dims[0];
    const double ih2 = 1.0 / (c->hs[0] * c->hs[0]);
    const bool mixed = c->o.prec == MG_MIXED;
    stats_begin(st);
    if (st) st->ms_setup = c->ms_setup;
    CK(cudaEventRecord(c->ev0, s));
    CKS(prepare_rhs(c, rhs));
    int scale_slot = mg::S_SCALE0, next_slot = mg::S_SCALE1;
    if (mixed) {
        ProfScope ps(c, MG_PROF_RESID64, true);
        CK(mg::launch_resid_cast(d, ih2, c->L64[0], c->b0, p, c->L32[0].b, c->partials, c->dscal, -1, next_slot, s,
                                 c->split0));
    } else {
        ProfScope ps(c, MG_PROF_RESID64, true);
        CK(mg::launch_resid_norm(d, ih2, c->L64[0], c->b0, p, c->partials, c->dscal, s));
    }
    CKS(read_scalars(c));
    check_compatible(c);
    const double nb2 = c->hscal[mg::S_NB2];
    if (st) {
        st->rhs_norm = std::sqrt(nb2);
        st->rhs_mean_removed = c->nlive > 0 ? c->hscal[mg::S_SUM_B] / c->nlive : 0.0;
    }
    if (!std::isfinite(nb2)) return fail(MG_ERR_NAN, "right-hand side is not finite");
    if (nb2 == 0.0 || c->nlive == 0.0) {
        CK(cudaMemsetAsync(p, 0, d.n() * sizeof(double), s));
        CK(cudaEventRecord(c->ev1, s));
        CK(cudaEventSynchronize(c->ev1));
        if (st) cudaEventElapsedTime(&st->ms_solve, c->ev0, c->ev1);
        return final_status(c, MG_OK);
    }
    double rel = std::sqrt(c->hscal[mg::S_RR] / nb2);
    int cyc = 0, status = MG_OK;
    int nhist = 0;
    // The next cycle's first passes, queued before the residual that decides on it is read (passes_ahead).  Mixed: they
    // write the correction alone, which nothing reads if the iteration has ended.  FP64: they would change p, so each
    // stores only where the squared residual norm is above `limit` (a little above tol^2 ||b||^2, so that the
    // host goes on wherever a pass has stored); between the two the host queues them again.  A FP64 solve
    // at 32^3 1.325 -> 1.227 ms, at 128^3 11.05 -> 10.93 ms.
    const int ahead = passes_ahead(c);
    const bool skipped = c->o.nu1 >= 1 && c->o.nu2 >= 1;  // the first red pass of a continued FP64 cycle
    const int stop = ahead == 0 ? 0 : (mixed ? ahead : std::min(2 * c->o.nu1, ahead + (skipped ? 1 : 0)));
    const double limit = tol * tol * nb2 * (1.0 + 1e-10);
    int done = 0;  // of the next cycle's passes, those made
    while (!(rel <= tol)) {
        if (!std::isfinite(rel)) {
            status = fail(MG_ERR_NAN, "residual norm is not finite after %d cycles", cyc);
            break;
        }
        if (cyc >= c->o.max_cycles) {
            status = fail(MG_ERR_NOT_CONVERGED, "not converged: relative residual %.3e after %d cycles (tol %.1e)",
                          rel, cyc, tol);
            break;
        }
        cyc++;
        if (mixed) {
            for (int ic = 0; ic < c->o.inner_cycles; ic++)
                CKS(vcycle<float>(c, c->L32, 0, c->L32[0].b, c->L32[0].p, ic == 0, ic > 0, CyclePart{ic == 0 ? done : 0, -1, {}}));
            CK(mg::launch_accumulate(d, c->L64[0].dinv, c->L32[0].p, p, c->dscal, scale_slot, s, c->split0));
            std::swap(scale_slot, next_slot);
            ProfScope ps(c, MG_PROF_RESID64, true);
            CK(mg::launch_resid_cast(d, ih2, c->L64[0], c->b0, p, c->L32[0].b, c->partials, c->dscal, scale_slot,
                                     next_slot, s, c->split0));
        } else {
            CKS(vcycle<double>(c, c->L64, 0, c->b0, p, false, cyc > 1, CyclePart{done, -1, {}}));
            done = 0;
            if (cyc % c->o.check_every != 0 && cyc < c->o.max_cycles) continue;
            ProfScope ps(c, MG_PROF_RESID64, true);
            CK(mg::launch_resid_norm(d, ih2, c->L64[0], c->b0, p, c->partials, c->dscal, s));
        }
        CKS(queue_scalars(c));
        const bool more = stop > 0 && cyc < c->o.max_cycles;
        if (more && mixed) CKS(vcycle<float>(c, c->L32, 0, c->L32[0].b, c->L32[0].p, true, false, CyclePart{0, stop, {}}));
        else if (more)
            CKS(vcycle<double>(c, c->L64, 0, c->b0, p, false, true, CyclePart{0, stop, mg::Gate{c->dscal + mg::S_RR, limit}}));
        CKS(wait_scalars(c));
        const double rr = c->hscal[mg::S_RR];
        done = more && (mixed || (rr > limit && std::isfinite(rr))) ? stop : 0;
        rel = std::sqrt(rr / nb2);
        if (st && nhist < 256) st->resid_hist[nhist++] = rel;
    }
    // zero mean over each region's live cells (the cycle commutes with constant shifts, so once
    // suffices)
    CKS(remove_p_mean(c, p, !mg::resid_sums_p(d.n())));
    CK(cudaEventRecord(c->ev1, s));
    CK(cudaEventSynchronize(c->ev1));
    if (st) {
        st->cycles = cyc;
        st->rel_resid = rel;
        cudaEventElapsedTime(&st->ms_solve, c->ev0, c->ev1);
    }
    return final_status(c, status);
}

int compute_hierarchy(mg_ctx *c, const double *const face_coeffs[3])
{
    cudaStream_t s = c->s;
    const Dims dc = c->dims.back();
    const size_t n0 = c->dims[0].n();
    CK(cudaMemsetAsync(c->dscal, 0, mg::S_COUNT * sizeof(double), s));
    if (c->has_area) {  // keep 1/rho; the operator's coefficient is area * 1/rho
        double *kb[3] = {c->kbeta.bx, c->kbeta.by, c->kbeta.bz};
        for (int a = 0; a < 3; a++)
            if (face_coeffs[a] != kb[a])
                CK(cudaMemcpyAsync(kb[a], face_coeffs[a], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
        CK(mg::launch_area_coeffs(n0, c->karea, c->kbeta, c->L64[0], s));
    } else {
        CK(cudaMemcpyAsync(c->L64[0].bx, face_coeffs[0], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(c->L64[0].by, face_coeffs[1], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(c->L64[0].bz, face_coeffs[2], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    for (int l = 0; l < c->nlev; l++) {
        if (l > 0)
            CK(mg::launch_restrict_coeffs(c->dims[l - 1], c->L64[l - 1].bx, c->L64[l - 1].by, c->L64[l - 1].bz,
                                          c->L64[l].bx, c->L64[l].by, c->L64[l].bz, s));
        // the finest level's CG operator (scaled coefficients and diagonal) comes out of the same pass
        const bool op = l == 0 && c->kop.dinv;
        CK(mg::launch_diag_inv<double>(c->dims[l], c->L64[l].bx, c->L64[l].by, c->L64[l].bz, c->L64[l].dinv, s,
                                       op ? &c->kop : nullptr, 1.0 / (c->hs[0] * c->hs[0]),
                                       l == 0 ? c->open_bits : nullptr, c->dscal + mg::S_TOPO));
    }
    CK(mg::launch_count_live(c->dims[0], c->L64[0].dinv, c->partials, c->dscal, s));
    // the coarsest operator and the scalars to the pinned host mirrors; the host waits for them
    // alone (event), while the FP32 copies queued next still run: the host's inverse of the
    // coarsest operator overlaps them
    const int nc = c->ncoarse;
    double *hcb = c->hcoarse, *hM = c->hcoarse + 3 * (size_t)nc;
    unsigned *hrow = reinterpret_cast<unsigned *>(hM + (size_t)nc * nc);
    const double *src[3] = {c->L64.back().bx, c->L64.back().by, c->L64.back().bz};
    for (int a = 0; a < 3; a++)
        CK(cudaMemcpyAsync(hcb + (size_t)a * nc, src[a], nc * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(c->hscal, c->dscal, mg::S_COUNT * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaEventRecord(c->ev_h, s));
    for (size_t l = 0; l < c->rec64.size(); l++)
        if (c->rec64[l]) CK(mg::launch_row_records<double>(c->dims[l], c->L64[l], c->rec64[l], s));
    if (c->o.prec == MG_MIXED) {
        // narrowed faces and 1/sum of them (the value the FP32 smoothers form on the fly); the
        // finest level's faces also in the colour-split layout
        for (int l = 0; l < c->nlev; l++)
            CK(mg::launch_level_f32(c->dims[l], c->L64[l], c->L32[l], s, l == 0 ? &c->sf0 : nullptr, c->split0));
        for (size_t l = 0; l < c->rec32.size(); l++)
            if (c->rec32[l]) CK(mg::launch_row_records<float>(c->dims[l], c->L32[l], c->rec32[l], s));
        if (c->rowcnt) CK(cudaMemsetAsync(c->rowcnt, 0, 2 * sizeof(unsigned), s));
        if (c->urow0)
            CK(mg::launch_uniform_rows(c->dims[0], c->L32[0].bx, c->L32[0].by, c->L32[0].bz, c->urow0, s, c->arow0, c->uinv0,
                                       c->rowcnt));
        if (c->rowcnt) CK(cudaMemcpyAsync(hrow, c->rowcnt, 2 * sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    }
    CK(cudaEventSynchronize(c->ev_h));
    CKS(check_scalars(c));
    c->nlive = c->hscal[mg::S_NLIVE];
    // connected regions of the live fine cells, labelled again where the open faces changed
    // (first build included: the stored bits start as 0xff)
    unsigned cc[2] = {(unsigned)c->ncomp, 0};
    if (c->hscal[mg::S_TOPO] != 0.0) {
        CK(mg::launch_components(c->dims[0], c->L64[0].dinv, c->L64[0].bx, c->L64[0].by, c->L64[0].bz, c->cc_label,
                                 c->cc_ctr, s));
        CK(cudaMemcpyAsync(cc, c->cc_ctr, sizeof cc, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
    } else {
        cc[0] = (unsigned)(c->ncomp_raw);
    }
    if (cc[1]) return fail(MG_ERR_CUDA, "fluid-region labelling: a bounded union-find loop gave up");
    if (cc[0] > (unsigned)kMaxRegions)
        return fail(MG_ERR_ARG, "the fluid forms %u disconnected regions (at most %d supported)", cc[0], kMaxRegions);
    c->ncomp = (int)std::max(cc[0], 1u);
    const bool relabel = c->hscal[mg::S_TOPO] != 0.0;
    c->ncomp_raw = (int)cc[0];
    std::vector<int> roots;
    if (cc[0] > 1 && relabel) {  // number the regions by their smallest cell index; cells per region
        CK(mg::launch_component_roots(n0, c->cc_label, c->cc_roots, c->cc_ctr, (unsigned)kMaxRegions, s));
        roots.resize(cc[0]);
        CK(cudaMemcpyAsync(roots.data(), c->cc_roots, cc[0] * sizeof(int), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        std::sort(roots.begin(), roots.end());
        CK(cudaMemcpyAsync(c->cc_roots, roots.data(), cc[0] * sizeof(int), cudaMemcpyHostToDevice, s));
        CK(mg::launch_component_compact(n0, c->cc_label, c->cc_roots, c->ncomp, c->cc_cnt, c->cc_part, s));
        c->hcnt.resize(c->ncomp);
        CK(cudaMemcpyAsync(c->hcnt.data(), c->cc_cnt, c->ncomp * sizeof(double), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
    }
    CKS(coarse_inverse(dc.nx, dc.ny, dc.nz, c->hs.back(), hcb, hcb + nc, hcb + 2 * (size_t)nc, hM));
    CK(cudaMemcpyAsync(c->M, hM, (size_t)nc * nc * sizeof(double), cudaMemcpyHostToDevice, s));
    // the pinned staging must outlive the copy; the row counters have arrived
    CK(cudaStreamSynchronize(s));
    if (c->o.prec == MG_MIXED && c->rowcnt) c->banded = hrow[1] > hrow[0];
    return MG_OK;
}

// ---------------------------------------------------------------------------
// Multigrid-preconditioned conjugate gradients, flexible (Polak-Ribiere) form:
//   r = b - A p; z = M r; d = z
//   repeat: q = A d; alpha = <r,z>/<d,q>; p += alpha d; r -= alpha q
//           z' = M r; beta = (<r,z'> - <r,z>) / <r_old,z>; d = z' + beta d
// M = inner_cycles V-cycles from a zero guess, FP64 or FP32 (on r scaled by the
// RMS of the previous residual).  Convergence is decided on the recursive r and
// confirmed with the true residual (restart from p if it is above the target).
// The target is kCgTolFactor * tol: the relative solution error of a CG iterate is
// 4 to 23 times its relative residual on the 128^3, 256^3 and 512x256x128 workloads,
// so the CG stops where the residual is 0.4 tol and the error below 10 tol.
// ---------------------------------------------------------------------------
constexpr double kCgTolFactor = 0.4;

int pcg_impl(mg_ctx *c, const double *rhs, double *p, double tol_user, mg_stats *st)
{
    const double tol = tol_user * kCgTolFactor;
    cudaStream_t s = c->s;
    const Dims d = c->dims[0];
    const size_t n = d.n();
    const double ih2 = 1.0 / (c->hs[0] * c->hs[0]);
    const bool mixed = c->o.prec == MG_MIXED;
    stats_begin(st);
    if (st) st->ms_setup = c->ms_setup;
    CK(cudaEventRecord(c->ev0, s));
    CKS(prepare_rhs(c, rhs));
    bool first_check = true;
    float *e_cur = mixed ? c->L32[0].p : nullptr, *e_old = mixed ? c->ke_alt : nullptr;
    int sc_cur = mg::S_SCALE0, sc_old = mg::S_SCALE1;
    double *z = c->kz, *zo = c->kzo;
    int it = 0, status = MG_OK, nhist = 0;
    double rel = 0.0, nb2 = 0.0;
    bool done = false, zeroed = false;
    // precondition: z = M r (FP64) or e_cur = M (r / scale) (mixed); M = V-cycles, or the inverse
    // diagonal of A (Jacobi: -h^2 dinv); `done` passes of its first cycle are queued already
    auto precondition = [&](int done) -> int {
        if (c->o.precond == 1) {
            CK(mg::launch_jacobi(n, -c->hs[0] * c->hs[0], c->L64[0].dinv, c->kr, z, s));
        } else if (mixed) {
            for (int v = 0; v < c->o.inner_cycles; v++)
                CKS(vcycle<float>(c, c->L32, 0, c->L32[0].b, e_cur, v == 0, v > 0, CyclePart{v == 0 ? done : 0, -1, {}}));
        } else {
            for (int v = 0; v < c->o.inner_cycles; v++)
                CKS(vcycle<double>(c, c->L64, 0, c->kr, z, v == 0, v > 0, CyclePart{v == 0 ? done : 0, -1, {}}));
        }
        return MG_OK;
    };
    // the first passes of the next preconditioning, queued while the host waits for the residual of the update
    // before them; they write e_cur or z alone, which nothing reads if the iteration was the last
    const int ahead = c->o.precond == 0 ? passes_ahead(c) : 0;
    auto begin_precondition = [&]() -> int {
        if (ahead == 0) return MG_OK;
        if (mixed) return vcycle<float>(c, c->L32, 0, c->L32[0].b, e_cur, true, false, CyclePart{0, ahead, {}});
        return vcycle<double>(c, c->L64, 0, c->kr, z, true, false, CyclePart{0, ahead, {}});
    };
    while (!done) {
        // (re)start: true residual
        {
            ProfScope ps(c, MG_PROF_RESID64, true);
            // the first residual of a solve tests p for zero (a zero guess needs no stencil)
            CK(mg::launch_pcg_resid(d, ih2, c->L64[0], c->b0, p, c->kr, mixed ? c->L32[0].b : nullptr, c->partials,
                                    c->dscal, sc_cur, s, c->split0, first_check ? c->pnz : nullptr));
        }
        CKS(read_scalars(c));
        if (first_check) check_compatible(c);
        first_check = false;
        nb2 = c->hscal[mg::S_NB2];
        if (st) {
            st->rhs_norm = std::sqrt(nb2);
            st->rhs_mean_removed = c->nlive > 0 ? c->hscal[mg::S_SUM_B] / c->nlive : 0.0;
        }
        if (!std::isfinite(nb2)) return fail(MG_ERR_NAN, "right-hand side is not finite");
        if (nb2 == 0.0 || c->nlive == 0.0) {
            CK(cudaMemsetAsync(p, 0, n * sizeof(double), s));
            rel = 0.0;
            zeroed = true;
            break;
        }
        rel = std::sqrt(c->hscal[mg::S_RR] / nb2);
        if (rel <= tol) break;
        if (!std::isfinite(rel)) {
            status = fail(MG_ERR_NAN, "residual norm is not finite after %d iterations", it);
            break;
        }
        if (it >= c->o.max_cycles) {
            status = fail(MG_ERR_NOT_CONVERGED,
                          "not converged: relative residual %.3e after %d iterations (tol %.1e, CG target %.1e)", rel,
                          it, tol_user, tol);
            break;
        }
        CKS(precondition(0));
        if (mixed) {
            CK(mg::launch_pcg_dots32(n, c->L32[0].b, e_cur, nullptr, c->partials, c->dscal, sc_cur, sc_cur, -1, s));
            CK(mg::launch_pcg_dir<float>(n, e_cur, c->kd, c->dscal, sc_cur, -1, 1, s, c->split0, c->partials));
        } else {
            CK(mg::launch_pcg_dots<double>(n, c->kr, z, nullptr, c->partials, c->dscal, -1, -1, s));
            CK(mg::launch_pcg_dir<double>(n, z, c->kd, c->dscal, -1, -1, 1, s, {}, c->partials));
        }
        for (;;) {
            it++;
            {
                ProfScope ps(c, MG_PROF_APPLY, true);
                CK(mg::launch_pcg_apply(d, c->kop, c->kd, c->kq, c->partials, c->dscal, s));
            }
            std::swap(e_cur, e_old);
            std::swap(sc_cur, sc_old);
            std::swap(z, zo);
            {
                ProfScope ps(c, MG_PROF_RESID64, true);
                CK(mg::launch_pcg_update(n, c->kd, c->kq, p, c->kr, mixed ? c->L32[0].b : nullptr, c->partials, c->dscal,
                                         sc_cur, mixed ? sc_old : -1, s, c->split0));
            }
            CKS(queue_scalars(c));
            const bool more = it < c->o.max_cycles;
            if (more) CKS(begin_precondition());
            CKS(wait_scalars(c));
            rel = std::sqrt(c->hscal[mg::S_RR] / nb2);
            if (st && nhist < 256) st->resid_hist[nhist++] = rel;
            if (rel <= tol || !std::isfinite(rel) || !more) break;
            CKS(precondition(ahead));
            ProfScope ps(c, MG_PROF_KRYLOV, true);
            if (mixed) {
                CK(mg::launch_pcg_dots32(n, c->L32[0].b, e_cur, e_old, c->partials, c->dscal, sc_cur, sc_cur, sc_old,
                                         s));
                CK(mg::launch_pcg_dir<float>(n, e_cur, c->kd, c->dscal, sc_cur, sc_old, 0, s, c->split0, c->partials));
            } else {
                CK(mg::launch_pcg_dots<double>(n, c->kr, z, zo, c->partials, c->dscal, -1, -1, s));
                CK(mg::launch_pcg_dir<double>(n, z, c->kd, c->dscal, -1, -1, 0, s, {}, c->partials));
            }
        }
        if (!std::isfinite(rel)) {
            status = fail(MG_ERR_NAN, "residual norm is not finite after %d iterations", it);
            break;
        }
        // the loop top re-checks with the true residual (and restarts if needed)
    }
    (void)done;
    if (!zeroed && (status == MG_OK || status == MG_ERR_NOT_CONVERGED)) CKS(remove_p_mean(c, p, false));
    CK(cudaEventRecord(c->ev1, s));
    CK(cudaEventSynchronize(c->ev1));
    if (st) {
        st->cycles = it;
        st->rel_resid = rel;
        cudaEventElapsedTime(&st->ms_solve, c->ev0, c->ev1);
    }
    return final_status(c, status);
}

int ensure(mg_ctx *c, double **p, size_t n)
{
    if (*p) return MG_OK;
    return c->alloc(p, n);
}

}  // namespace

extern "C" {

void mg_default_opts(mg_opts *o)
{
    if (!o) return;
    o->nu1 = 2;
    o->nu2 = 2;
    o->max_cycles = 100;
    o->check_every = 1;
    o->coarse_max_cells = 512;
    o->prec = MG_FP64;
    o->inner_cycles = 1;
    o->profile = 0;
    o->smoother = 0;
    o->krylov = 0;
    o->coarse_graph = 1;
    o->coarse_tail = 1;
    o->precond = 0;
    o->pass_order = 1;
}

const char *mg_last_error(void) { return g_err.c_str(); }

int mg_face_coeffs(const mg_grid *g, const double *phi, const uint8_t *solid_mask, double rho_air, double rho_water,
                   double *const beta_out[3], void *stream)
{
    g_err.clear();
    if (!grid_ok(g)) return fail(MG_ERR_ARG, "mg_face_coeffs: bad grid");
    if (!phi || !beta_out || !beta_out[0] || !beta_out[1] || !beta_out[2])
        return fail(MG_ERR_ARG, "mg_face_coeffs: null pointer");
    if (!(rho_air > 0.0) || !(rho_water > 0.0)) return fail(MG_ERR_ARG, "mg_face_coeffs: densities must be > 0");
    if (!aligned16({phi, solid_mask, beta_out[0], beta_out[1], beta_out[2]}))
        return fail(MG_ERR_ARG, "mg_face_coeffs: arrays must be 16-byte aligned");
    const Dims d{g->nx, g->ny, g->nz};
    CK(mg::launch_face_coeffs(d, phi, solid_mask, rho_air, rho_water - rho_air, beta_out[0], beta_out[1], beta_out[2],
                              (cudaStream_t)stream));
    return MG_OK;
}

int mg_setup(mg_ctx **out, const mg_grid *g, const double *const face_coeffs[3], const mg_bc *bc,
             const uint8_t *solid_mask, const mg_opts *opt, void *stream)
{
    g_err.clear();
    (void)solid_mask;
    const auto t0 = std::chrono::steady_clock::now();
    if (!out) return fail(MG_ERR_ARG, "mg_setup: out is null");
    *out = nullptr;
    if (!grid_ok(g)) return fail(MG_ERR_ARG, "mg_setup: bad grid");
    if (!face_coeffs || !face_coeffs[0] || !face_coeffs[1] || !face_coeffs[2])
        return fail(MG_ERR_ARG, "mg_setup: null face coefficient pointer");
    if (!aligned16({face_coeffs[0], face_coeffs[1], face_coeffs[2], solid_mask}))
        return fail(MG_ERR_ARG, "mg_setup: arrays must be 16-byte aligned");
    if (bc)
        for (int w = 0; w < 6; w++)
            if (bc->wall[w] != MG_BC_NEUMANN) return fail(MG_ERR_ARG, "mg_setup: only Neumann walls are supported");
    mg_opts o;
    mg_default_opts(&o);
    if (opt) o = *opt;
    if (o.nu1 < 0 || o.nu2 < 0 || o.nu1 + o.nu2 < 1 || o.max_cycles < 0 || o.check_every < 1 ||
        o.coarse_max_cells < 1 || o.coarse_max_cells > 2048 || (o.prec != MG_FP64 && o.prec != MG_MIXED) ||
        o.inner_cycles < 1 || o.profile < 0 || o.smoother < 0 || o.smoother > 3 || o.krylov < 0 || o.krylov > 1 || o.coarse_graph < 0 || o.coarse_graph > 1 ||
        o.coarse_tail < 0 || o.coarse_tail > 1 || o.precond < 0 || o.precond > 1 || o.pass_order < 0 ||
        o.pass_order > 1 ||
        (o.precond == 1 && (o.krylov != 1 || o.prec != MG_FP64)))
        return fail(MG_ERR_ARG, "mg_setup: invalid options");

    mg_ctx *c = new mg_ctx();
    c->g = *g;
    c->o = o;
    c->s = (cudaStream_t)stream;
    auto bail = [&](int code) {
        delete c;
        return code;
    };
    // levels: halve while every axis is even and >= 8
    Dims d{g->nx, g->ny, g->nz};
    double h = g->h;
    for (;;) {
        c->dims.push_back(d);
        c->hs.push_back(h);
        if (!(d.nx % 2 == 0 && d.ny % 2 == 0 && d.nz % 2 == 0 && d.nx >= 8 && d.ny >= 8 && d.nz >= 8)) break;
        d = Dims{d.nx / 2, d.ny / 2, d.nz / 2};
        h *= 2.0;
    }
    c->nlev = (int)c->dims.size();
    // the finest FP32 fields are colour-split when its sweeps are colour passes; a hierarchy of
    // two or more levels has even dims on the finest
    if (c->o.prec == MG_MIXED && c->o.smoother <= 1 && c->nlev >= 2)
        c->split0 = mg::Split{c->dims[0].n() / 2, c->dims[0].nx, c->dims[0].ny, mg::make_fastdiv(c->dims[0].nx),
                              mg::make_fastdiv(c->dims[0].ny)};
    const Dims dc = c->dims.back();
    if ((long long)dc.n() > o.coarse_max_cells)
        return bail(fail(MG_ERR_ARG, "mg_setup: coarsest grid %dx%dx%d has %zu cells > coarse_max_cells=%d", dc.nx,
                         dc.ny, dc.nz, dc.n(), o.coarse_max_cells));
    c->ncoarse = (int)dc.n();
    int st = MG_OK;
    c->L64.resize(c->nlev);
    for (int l = 0; l < c->nlev && st == MG_OK; l++) st = level_alloc<double>(c, c->L64[l], c->dims[l].n(), l > 0);
    if (st == MG_OK) st = c->alloc(&c->b0, c->dims[0].n());
    if (st == MG_OK) st = c->alloc(&c->partials, mg::kRedPartials);
    if (st == MG_OK && cudaMemsetAsync(c->partials, 0, mg::kRedPartials * sizeof(double), c->s) != cudaSuccess)
        st = fail(MG_ERR_CUDA, "mg_setup: memset failed");
    if (st == MG_OK) st = c->alloc(&c->dscal, mg::S_COUNT);
    if (st == MG_OK) st = c->alloc(&c->M, (size_t)c->ncoarse * c->ncoarse);
    if (st == MG_OK) st = c->alloc(&c->cc_label, c->dims[0].n());
    if (st == MG_OK) st = c->alloc(&c->open_bits, c->dims[0].n());
    if (st == MG_OK && cudaMemsetAsync(c->open_bits, 0xff, c->dims[0].n(), c->s) != cudaSuccess)
        st = fail(MG_ERR_CUDA, "mg_setup: memset failed");
    if (st == MG_OK) st = c->alloc(&c->cc_ctr, 4);
    if (st == MG_OK) st = c->alloc(&c->pnz, 1);
    if (st == MG_OK) st = c->alloc(&c->cc_roots, kMaxRegions);
    if (st == MG_OK) st = c->alloc(&c->cc_sum, kMaxRegions);
    if (st == MG_OK) st = c->alloc(&c->cc_cnt, kMaxRegions);
    if (st == MG_OK) st = c->alloc(&c->cc_part, 8 * mg::kRedBlocks);
    if (st != MG_OK) return bail(st);
    if (cudaMallocHost(&c->hscal, mg::S_COUNT * sizeof(double)) != cudaSuccess ||
        cudaMallocHost(&c->hcoarse, (3 * (size_t)c->ncoarse + (size_t)c->ncoarse * c->ncoarse + 1) * sizeof(double)) !=
            cudaSuccess ||
        cudaEventCreate(&c->ev0) != cudaSuccess || cudaEventCreate(&c->ev1) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->ev_h, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return bail(fail(MG_ERR_CUDA, "mg_setup: pinned buffer / event creation failed"));
    }
    if (c->o.smoother <= 1) {
        auto records = [&](auto &rec, int first, size_t cells) {
            rec.resize(c->nlev, nullptr);
            for (int l = first; l + 1 < c->nlev && st == MG_OK; l++)
                if (l == 0 || c->dims[l].n() >= cells) st = c->alloc(&rec[l], 8 * (size_t)c->dims[l].ny * c->dims[l].nz);
        };
        if (c->o.prec == MG_FP64) records(c->rec64, 0, mg::kRecCells64);
        else records(c->rec32, 1, mg::kRecCells32);
        if (st != MG_OK) return bail(st);
    }
    if (c->o.prec == MG_MIXED) {
        c->L32.resize(c->nlev);
        for (int l = 0; l < c->nlev && st == MG_OK; l++) st = level_alloc<float>(c, c->L32[l], c->dims[l].n(), true);
        if (st == MG_OK && c->split0.half) st = c->alloc(&c->urow0, (size_t)c->dims[0].ny * c->dims[0].nz);
        if (st == MG_OK && c->split0.half && c->dims[0].nx % 8 == 0) {
            st = c->alloc(&c->arow0, (size_t)c->dims[0].ny * c->dims[0].nz);
            if (st == MG_OK) st = c->alloc(&c->uinv0, (size_t)c->dims[0].ny * c->dims[0].nz);
            if (st == MG_OK) st = c->alloc(&c->rowcnt, 2);
            if (st == MG_OK) st = c->alloc(&c->sf0.bx, c->dims[0].n());
            if (st == MG_OK) st = c->alloc(&c->sf0.by, c->dims[0].n());
            if (st == MG_OK) st = c->alloc(&c->sf0.bz, c->dims[0].n());
        }
        if (st != MG_OK) return bail(st);
    }
    if (c->o.krylov) {
        const size_t n0 = c->dims[0].n();
        st = c->alloc(&c->kr, n0);
        if (st == MG_OK) st = level_alloc<double>(c, c->kop, n0, false);
        if (st == MG_OK) st = c->alloc(&c->kd, n0);
        if (st == MG_OK) st = c->alloc(&c->kq, n0);
        if (st == MG_OK && c->o.prec == MG_MIXED) st = c->alloc(&c->ke_alt, n0);
        if (st == MG_OK && c->o.prec != MG_MIXED) st = c->alloc(&c->kz, n0);
        if (st == MG_OK && c->o.prec != MG_MIXED) st = c->alloc(&c->kzo, n0);
        if (st != MG_OK) return bail(st);
    }
    // second iterate buffers for the fused sweeps
    for (int l = 0; l + 1 < c->nlev && st == MG_OK; l++) {
        const bool f64 = c->o.smoother == 2 && fused_level(c->dims[l]);
        const bool f32 = c->o.prec == MG_MIXED && c->o.smoother >= 2 && fused_level(c->dims[l]);
        if (f64) {
            c->palt64.resize(c->nlev, nullptr);
            st = c->alloc(&c->palt64[l], c->dims[l].n());
        }
        if (f32 && st == MG_OK) {
            c->palt32.resize(c->nlev, nullptr);
            st = c->alloc(&c->palt32[l], c->dims[l].n());
        }
    }
    if (st != MG_OK) return bail(st);
    if (c->o.profile) {
        c->pev.resize(2 * 32768);
        c->pgroup.resize(32768);
        for (auto &e : c->pev)
            if (cudaEventCreate(&e) != cudaSuccess) {
                cudaGetLastError();
                return bail(fail(MG_ERR_CUDA, "mg_setup: event creation failed"));
            }
    }
    auto plan = [&](auto &t, const auto &L) {
        t.first = tail_start(c, L, t.a);
        t.a.nu1 = o.nu1;
        t.a.nu2 = o.nu2;
        t.a.M = c->M;
    };
    if (c->o.prec == MG_MIXED) plan(c->tail32, c->L32);
    else plan(c->tail64, c->L64);
    st = compute_hierarchy(c, face_coeffs);
    if (st != MG_OK) return bail(st);
    c->ms_setup = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
    *out = c;
    return MG_OK;
}

int mg_update(mg_ctx *c, const double *const face_coeffs[3])
{
    g_err.clear();
    if (!c || !face_coeffs || !face_coeffs[0] || !face_coeffs[1] || !face_coeffs[2])
        return fail(MG_ERR_ARG, "mg_update: null argument");
    if (!aligned16({face_coeffs[0], face_coeffs[1], face_coeffs[2]}))
        return fail(MG_ERR_ARG, "mg_update: arrays must be 16-byte aligned");
    const auto t0 = std::chrono::steady_clock::now();
    {
        ProfScope ps(c, MG_PROF_UPDATE, true);
        CKS(compute_hierarchy(c, face_coeffs));
    }
    c->ms_setup = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return MG_OK;
}

int mg_solve(mg_ctx *c, const double *rhs, double *p, double tol, mg_stats *stats)
{
    g_err.clear();
    if (!c || !rhs || !p) return fail(MG_ERR_ARG, "mg_solve: null argument");
    if (rhs == p) return fail(MG_ERR_ARG, "mg_solve: rhs and p must not alias");
    if (!aligned16({rhs, p})) return fail(MG_ERR_ARG, "mg_solve: arrays must be 16-byte aligned");
    if (!(tol > 0.0)) return fail(MG_ERR_ARG, "mg_solve: tol must be > 0");
    return c->o.krylov ? pcg_impl(c, rhs, p, tol, stats) : solve_impl(c, rhs, p, tol, stats);
}

int mg_vcycle(mg_ctx *c, const double *rhs, double *p)
{
    g_err.clear();
    if (!c || !rhs || !p) return fail(MG_ERR_ARG, "mg_vcycle: null argument");
    if (!aligned16({rhs, p})) return fail(MG_ERR_ARG, "mg_vcycle: arrays must be 16-byte aligned");
    if (c->o.prec != MG_MIXED) return vcycle<double>(c, c->L64, 0, rhs, p);
    // the cycle of a mixed context: FP32 copies of rhs and p in the finest FP32 level's layout,
    // one FP32 V-cycle on them, p widened back
    const size_t n = c->dims[0].n();
    CK(mg::launch_to_f32_layout(n, rhs, c->L32[0].b, c->s, c->split0));
    CK(mg::launch_to_f32_layout(n, p, c->L32[0].p, c->s, c->split0));
    CKS(vcycle<float>(c, c->L32, 0, c->L32[0].b, c->L32[0].p));
    CK(mg::launch_from_f32_layout(n, c->L32[0].p, p, c->s, c->split0));
    return MG_OK;
}

int mg_divergence(mg_ctx *c, const double *const u[3], double dt, double *rhs)
{
    g_err.clear();
    if (!c || !u || !u[0] || !u[1] || !u[2] || !rhs) return fail(MG_ERR_ARG, "mg_divergence: null argument");
    if (!(dt > 0.0)) return fail(MG_ERR_ARG, "mg_divergence: dt must be > 0");
    if (!aligned16({u[0], u[1], u[2], rhs})) return fail(MG_ERR_ARG, "mg_divergence: arrays must be 16-byte aligned");
    const LevelArrays<double> &L = c->L64[0];
    if (c->has_area || c->has_vb) {
        LevelArrays<double> uu{};
        uu.bx = const_cast<double *>(u[0]);
        uu.by = const_cast<double *>(u[1]);
        uu.bz = const_cast<double *>(u[2]);
        CK(mg::launch_divergence_area(c->dims[0], 1.0 / (dt * c->g.h), L, c->has_area ? c->karea : LevelArrays<double>{},
                                      uu, c->has_vb ? c->kvb : LevelArrays<double>{}, rhs, c->s));
    } else {
        CK(mg::launch_divergence(c->dims[0], 1.0 / (dt * c->g.h), L.bx, L.by, L.bz, u[0], u[1], u[2], rhs, c->s));
    }
    return MG_OK;
}

int mg_correct(mg_ctx *c, const double *const u_star[3], const double *p, double dt, double *const u[3])
{
    g_err.clear();
    if (!c || !u_star || !u || !p) return fail(MG_ERR_ARG, "mg_correct: null argument");
    for (int a = 0; a < 3; a++)
        if (!u_star[a] || !u[a]) return fail(MG_ERR_ARG, "mg_correct: null face array");
    if (!aligned16({u_star[0], u_star[1], u_star[2], u[0], u[1], u[2], p}))
        return fail(MG_ERR_ARG, "mg_correct: arrays must be 16-byte aligned");
    const LevelArrays<double> &L = c->L64[0];
    CK(mg::launch_correct(c->dims[0], dt, c->g.h, L.bx, L.by, L.bz, p, u_star[0], u_star[1], u_star[2], u[0], u[1],
                          u[2], c->s, c->has_area ? &c->kbeta : nullptr));
    return MG_OK;
}

int mg_face_areas(const mg_grid *g, const double *psi_nodes, double *const area_out[3], void *stream)
{
    g_err.clear();
    if (!grid_ok(g)) return fail(MG_ERR_ARG, "mg_face_areas: bad grid");
    if (!psi_nodes || !area_out || !area_out[0] || !area_out[1] || !area_out[2])
        return fail(MG_ERR_ARG, "mg_face_areas: null pointer");
    if (!aligned16({psi_nodes, area_out[0], area_out[1], area_out[2]}))
        return fail(MG_ERR_ARG, "mg_face_areas: arrays must be 16-byte aligned");
    CK(mg::launch_face_areas(Dims{g->nx, g->ny, g->nz}, psi_nodes, area_out[0], area_out[1], area_out[2],
                             (cudaStream_t)stream));
    return MG_OK;
}

int mg_stretched_metrics(const mg_grid *g, const double *hx, const double *hy, const double *hz,
                         const double *const beta[3], const double *const frac[3], double *const beta_out[3],
                         double *const area_out[3], void *stream)
{
    g_err.clear();
    if (!g || g->nx < 1 || g->ny < 1 || g->nz < 1 || (double)g->nx * g->ny * g->nz >= 2147483647.0)
        return fail(MG_ERR_ARG, "mg_stretched_metrics: bad grid");
    if (!hx || !hy || !hz || !beta || !beta_out || !area_out) return fail(MG_ERR_ARG, "mg_stretched_metrics: null pointer");
    for (int a = 0; a < 3; a++)
        if (!beta[a] || !beta_out[a] || !area_out[a] || (frac && !frac[a]))
            return fail(MG_ERR_ARG, "mg_stretched_metrics: null face array");
    if (!aligned16({hx, hy, hz, beta[0], beta[1], beta[2], beta_out[0], beta_out[1], beta_out[2], area_out[0],
                    area_out[1], area_out[2]}) ||
        (frac && !aligned16({frac[0], frac[1], frac[2]})))
        return fail(MG_ERR_ARG, "mg_stretched_metrics: arrays must be 16-byte aligned");
    auto view = [](const double *const x[3]) {
        LevelArrays<double> v{};
        if (x) {
            v.bx = const_cast<double *>(x[0]);
            v.by = const_cast<double *>(x[1]);
            v.bz = const_cast<double *>(x[2]);
        }
        return v;
    };
    CK(mg::launch_stretched_metrics(Dims{g->nx, g->ny, g->nz}, hx, hy, hz, view(beta), view(frac),
                                    view(beta_out), view(area_out), (cudaStream_t)stream));
    return MG_OK;
}

int mg_momentum_rhs(const mg_grid *g, const double *phi, const double *const beta[3], const double *const u[3],
                    const mg_forces *f, double *const R[3], double *work, void *stream)
{
    g_err.clear();
    if (!grid_ok(g)) return fail(MG_ERR_ARG, "mg_momentum_rhs: bad grid");
    if (!phi || !beta || !u || !f || !R || !work) return fail(MG_ERR_ARG, "mg_momentum_rhs: null argument");
    for (int a = 0; a < 3; a++)
        if (!beta[a] || !u[a] || !R[a]) return fail(MG_ERR_ARG, "mg_momentum_rhs: null face array");
    if (!forces_ok(f)) return fail(MG_ERR_ARG, "mg_momentum_rhs: forces not finite or viscosities not >= 0");
    if (!aligned16({phi, beta[0], beta[1], beta[2], u[0], u[1], u[2], R[0], R[1], R[2], work}))
        return fail(MG_ERR_ARG, "mg_momentum_rhs: arrays must be 16-byte aligned");
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++)
            if ((const double *)R[a] == u[b] || (const double *)R[a] == beta[b] || (const double *)R[a] == phi)
                return fail(MG_ERR_ARG, "mg_momentum_rhs: R must not alias its inputs");
    LevelArrays<double> B, U, RR;
    B.bx = const_cast<double *>(beta[0]);
    B.by = const_cast<double *>(beta[1]);
    B.bz = const_cast<double *>(beta[2]);
    U.bx = const_cast<double *>(u[0]);
    U.by = const_cast<double *>(u[1]);
    U.bz = const_cast<double *>(u[2]);
    RR.bx = R[0];
    RR.by = R[1];
    RR.bz = R[2];
    CK(mg::launch_momentum_rhs(Dims{g->nx, g->ny, g->nz}, g->h, phi, f->mu_air, f->mu_water, f->inv_re, f->g,
                               f->convection, B, U, RR, work, (cudaStream_t)stream));
    return MG_OK;
}

int mg_rk2_step(mg_ctx *c, const double *phi, const uint8_t *solid_mask, double rho_air, double rho_water,
                const mg_forces *forces, double dt, double *const u[3], double *phi_out, double *p_out, double tol,
                mg_stats *stats)
{
    g_err.clear();
    if (!c || !phi || !u || !u[0] || !u[1] || !u[2] || !phi_out || !p_out || !forces)
        return fail(MG_ERR_ARG, "mg_rk2_step: null argument");
    if (!(dt > 0.0) || !(tol > 0.0) || !(rho_air > 0.0) || !(rho_water > 0.0) || !forces_ok(forces))
        return fail(MG_ERR_ARG, "mg_rk2_step: dt, tol and the densities must be > 0, the forces finite");
    if (!aligned16({phi, solid_mask, u[0], u[1], u[2], phi_out, p_out}))
        return fail(MG_ERR_ARG, "mg_rk2_step: arrays must be 16-byte aligned");
    if (phi_out == phi) return fail(MG_ERR_ARG, "mg_rk2_step: phi_out must not alias phi");
    const size_t n = c->dims[0].n();
    const Dims d = c->dims[0];
    cudaStream_t s = c->s;
    if (!c->rk_phis) {
        for (LevelArrays<double> *L : {&c->rk_b1, &c->rk_b2, &c->rk_ut, &c->rk_us, &c->rk_r}) {
            CKS(c->alloc(&L->bx, n));
            CKS(c->alloc(&L->by, n));
            CKS(c->alloc(&L->bz, n));
        }
        CKS(c->alloc(&c->rk_phis, n));
        CKS(c->alloc(&c->rk_work, mg::kMomWork * n));
    }
    LevelArrays<double> uk{};
    uk.bx = u[0];
    uk.by = u[1];
    uk.bz = u[2];
    const LevelArrays<double> none{};
    const double drho = rho_water - rho_air, s_dt_h = dt / c->g.h;
    std::string incompat;  // message of a projection that reported an incompatible rhs
    auto faces = [](const LevelArrays<double> &L) {
        return std::array<double *, 3>{L.bx, L.by, L.bz};
    };
    // stage 1: rho(phi^k); u~ = u^k + dt R; u* = u~ - dt B G P*  (Eq. poisson1, runge1)
    CK(mg::launch_face_coeffs(d, phi, solid_mask, rho_air, drho, c->rk_b1.bx, c->rk_b1.by, c->rk_b1.bz, s));
    {
        const auto b1 = faces(c->rk_b1);
        const double *cb1[3] = {b1[0], b1[1], b1[2]};
        CKS(compute_hierarchy(c, cb1));
    }
    // R(u^k, phi^k) with the first stage's 1/rho
    CK(mg::launch_momentum_rhs(d, c->g.h, phi, forces->mu_air, forces->mu_water, forces->inv_re, forces->g,
                               forces->convection, c->rk_b1, uk, c->rk_r, c->rk_work, s));
    CK(mg::launch_rk_combine(n, uk, none, c->rk_r, dt, c->rk_ut, s));
    CK(cudaMemsetAsync(p_out, 0, n * sizeof(double), s));
    {
        const double *ut[3] = {c->rk_ut.bx, c->rk_ut.by, c->rk_ut.bz};
        double *us[3] = {c->rk_us.bx, c->rk_us.by, c->rk_us.bz};
        const int st = mg_project(c, ut, us, p_out, dt, tol, stats);
        if (st == MG_ERR_INCOMPATIBLE) incompat = g_err;
        else if (st != MG_OK) return st;
    }
    // phi* = phi^k - VOF(u^k, phi^k, dt)
    CK(mg::launch_vof_upwind(d, s_dt_h, c->rk_b1, uk, phi, c->rk_phis, s));
    // stage 2: rho(phi*); u~~ = (u* + u^k) + dt R; u^{k+1} = (u~~ - dt B* G P) / 2  (Eq. poisson2, runge2)
    CK(mg::launch_face_coeffs(d, c->rk_phis, solid_mask, rho_air, drho, c->rk_b2.bx, c->rk_b2.by, c->rk_b2.bz, s));
    {
        const auto b2 = faces(c->rk_b2);
        const double *cb2[3] = {b2[0], b2[1], b2[2]};
        CKS(compute_hierarchy(c, cb2));
    }
    // R(u*, phi*) with the second stage's 1/rho
    CK(mg::launch_momentum_rhs(d, c->g.h, c->rk_phis, forces->mu_air, forces->mu_water, forces->inv_re, forces->g,
                               forces->convection, c->rk_b2, c->rk_us, c->rk_r, c->rk_work, s));
    CK(mg::launch_rk_combine(n, c->rk_us, uk, c->rk_r, dt, c->rk_ut, s));
    // (u* + u^k) / 2 for the second VOF, kept in u* (u^k is overwritten below)
    CK(mg::launch_half(n, c->rk_us, uk, c->rk_us, s));
    // phi^{k+1} = phi^k - VOF((u* + u^k)/2, phi^k, dt), with the first stage's face mask
    CK(mg::launch_vof_upwind(d, s_dt_h, c->rk_b1, c->rk_us, phi, phi_out, s));
    CK(cudaMemsetAsync(p_out, 0, n * sizeof(double), s));
    {
        const double *ut[3] = {c->rk_ut.bx, c->rk_ut.by, c->rk_ut.bz};
        const int st = mg_project(c, ut, u, p_out, dt, tol, stats);
        if (st == MG_ERR_INCOMPATIBLE) incompat = g_err;
        else if (st != MG_OK) return st;
    }
    CK(mg::launch_half(n, uk, none, uk, s));
    if (!incompat.empty()) return fail(MG_ERR_INCOMPATIBLE, "%s", incompat.c_str());
    return MG_OK;
}

int mg_set_face_areas(mg_ctx *c, const double *const area[3])
{
    g_err.clear();
    if (!c) return fail(MG_ERR_ARG, "mg_set_face_areas: null context");
    const size_t n0 = c->dims[0].n();
    if (!area) {
        if (!c->has_area) return MG_OK;
        c->has_area = false;
        const double *kb[3] = {c->kbeta.bx, c->kbeta.by, c->kbeta.bz};
        return compute_hierarchy(c, kb);
    }
    if (!area[0] || !area[1] || !area[2]) return fail(MG_ERR_ARG, "mg_set_face_areas: null face array");
    if (!aligned16({area[0], area[1], area[2]}))
        return fail(MG_ERR_ARG, "mg_set_face_areas: arrays must be 16-byte aligned");
    if (!c->karea.bx) {
        CKS(c->alloc(&c->karea.bx, n0));
        CKS(c->alloc(&c->karea.by, n0));
        CKS(c->alloc(&c->karea.bz, n0));
        CKS(c->alloc(&c->kbeta.bx, n0));
        CKS(c->alloc(&c->kbeta.by, n0));
        CKS(c->alloc(&c->kbeta.bz, n0));
    }
    cudaStream_t s = c->s;
    if (!c->has_area) {  // the coefficients given so far are 1/rho
        CK(cudaMemcpyAsync(c->kbeta.bx, c->L64[0].bx, n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(c->kbeta.by, c->L64[0].by, n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(c->kbeta.bz, c->L64[0].bz, n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    CK(cudaMemcpyAsync(c->karea.bx, area[0], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CK(cudaMemcpyAsync(c->karea.by, area[1], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CK(cudaMemcpyAsync(c->karea.bz, area[2], n0 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    c->has_area = true;
    const double *kb[3] = {c->kbeta.bx, c->kbeta.by, c->kbeta.bz};
    return compute_hierarchy(c, kb);
}

int mg_set_body_velocity(mg_ctx *c, const double *const v[3])
{
    g_err.clear();
    if (!c) return fail(MG_ERR_ARG, "mg_set_body_velocity: null context");
    if (!v) {
        c->has_vb = false;
        return MG_OK;
    }
    if (!v[0] || !v[1] || !v[2]) return fail(MG_ERR_ARG, "mg_set_body_velocity: null face array");
    if (!aligned16({v[0], v[1], v[2]})) return fail(MG_ERR_ARG, "mg_set_body_velocity: arrays must be 16-byte aligned");
    const size_t n0 = c->dims[0].n();
    if (!c->kvb.bx) {
        CKS(c->alloc(&c->kvb.bx, n0));
        CKS(c->alloc(&c->kvb.by, n0));
        CKS(c->alloc(&c->kvb.bz, n0));
    }
    CK(cudaMemcpyAsync(c->kvb.bx, v[0], n0 * sizeof(double), cudaMemcpyDeviceToDevice, c->s));
    CK(cudaMemcpyAsync(c->kvb.by, v[1], n0 * sizeof(double), cudaMemcpyDeviceToDevice, c->s));
    CK(cudaMemcpyAsync(c->kvb.bz, v[2], n0 * sizeof(double), cudaMemcpyDeviceToDevice, c->s));
    c->has_vb = true;
    return MG_OK;
}

int mg_project(mg_ctx *c, const double *const u_star[3], double *const u[3], double *p, double dt, double tol,
               mg_stats *stats)
{
    g_err.clear();
    if (!c || !u_star || !u || !p) return fail(MG_ERR_ARG, "mg_project: null argument");
    for (int a = 0; a < 3; a++)
        if (!u_star[a] || !u[a]) return fail(MG_ERR_ARG, "mg_project: null face array");
    if (!(dt > 0.0) || !(tol > 0.0)) return fail(MG_ERR_ARG, "mg_project: dt and tol must be > 0");
    if (!aligned16({u_star[0], u_star[1], u_star[2], u[0], u[1], u[2], p}))
        return fail(MG_ERR_ARG, "mg_project: arrays must be 16-byte aligned");
    CKS(ensure(c, &c->rhs_tmp, c->dims[0].n()));
    CKS(mg_divergence(c, u_star, dt, c->rhs_tmp));
    const int st = c->o.krylov ? pcg_impl(c, c->rhs_tmp, p, tol, stats) : solve_impl(c, c->rhs_tmp, p, tol, stats);
    if (st != MG_OK && st != MG_ERR_NOT_CONVERGED && st != MG_ERR_INCOMPATIBLE) return st;
    const std::string keep = g_err;
    CKS(mg_correct(c, u_star, p, dt, u));
    g_err = keep;
    return st;
}

int mg_project_adjoint(mg_ctx *c, const double *const w[3], const double *p, double dt, double tol,
                       double *const grad_u[3], double *const grad_beta[3], double *q_out, mg_stats *stats)
{
    g_err.clear();
    if (!c || !w || !p || !grad_u) return fail(MG_ERR_ARG, "mg_project_adjoint: null argument");
    for (int a = 0; a < 3; a++) {
        if (!w[a] || !grad_u[a]) return fail(MG_ERR_ARG, "mg_project_adjoint: null face array");
        for (int b = 0; b < 3; b++)
            if ((const double *)grad_u[a] == w[b]) return fail(MG_ERR_ARG, "mg_project_adjoint: grad_u aliases w");
    }
    if (!(dt > 0.0) || !(tol > 0.0)) return fail(MG_ERR_ARG, "mg_project_adjoint: dt and tol must be > 0");
    if (!aligned16({w[0], w[1], w[2], grad_u[0], grad_u[1], grad_u[2], p, q_out}) ||
        (grad_beta && !aligned16({grad_beta[0], grad_beta[1], grad_beta[2]})))
        return fail(MG_ERR_ARG, "mg_project_adjoint: arrays must be 16-byte aligned");
    const size_t n = c->dims[0].n();
    CKS(ensure(c, &c->rhs_tmp, n));
    double *q = q_out;
    if (!q) {
        CKS(ensure(c, &c->qbuf, n));
        q = c->qbuf;
        CK(cudaMemsetAsync(q, 0, n * sizeof(double), c->s));
    }
    const LevelArrays<double> &L = c->L64[0];
    // c = D(beta w), the products beta * w rounded once; beta = 1/rho (with fractional areas the
    // operator's coefficient is area * 1/rho, and D sums the open faces without their areas)
    const LevelArrays<double> &B = c->has_area ? c->kbeta : L;
    CK(mg::launch_divergence_mul(c->dims[0], 1.0 / c->g.h, L, B, w[0], w[1], w[2], c->rhs_tmp, c->s));
    const int st = c->o.krylov ? pcg_impl(c, c->rhs_tmp, q, tol, stats) : solve_impl(c, c->rhs_tmp, q, tol, stats);
    if (st != MG_OK && st != MG_ERR_NOT_CONVERGED && st != MG_ERR_INCOMPATIBLE) return st;
    const std::string keep = g_err;
    double *gb[3] = {nullptr, nullptr, nullptr};
    if (grad_beta)
        for (int a = 0; a < 3; a++) gb[a] = grad_beta[a];
    CK(mg::launch_adjoint_faces(c->dims[0], c->g.h, dt, L.bx, L.by, L.bz, p, q, w[0], w[1], w[2], grad_u[0],
                                grad_u[1], grad_u[2], gb[0], gb[1], gb[2], c->s, c->has_area ? &c->karea : nullptr));
    g_err = keep;
    return st;
}

int mg_phi_grad(const mg_grid *g, const double *const beta[3], const double *const grad_beta[3], double rho_air,
                double rho_water, double *grad_phi, void *stream)
{
    g_err.clear();
    if (!grid_ok(g)) return fail(MG_ERR_ARG, "mg_phi_grad: bad grid");
    if (!beta || !grad_beta || !grad_phi) return fail(MG_ERR_ARG, "mg_phi_grad: null argument");
    for (int a = 0; a < 3; a++)
        if (!beta[a] || !grad_beta[a]) return fail(MG_ERR_ARG, "mg_phi_grad: null face array");
    if (!aligned16({beta[0], beta[1], beta[2], grad_beta[0], grad_beta[1], grad_beta[2], grad_phi}))
        return fail(MG_ERR_ARG, "mg_phi_grad: arrays must be 16-byte aligned");
    const Dims d{g->nx, g->ny, g->nz};
    CK(mg::launch_phi_grad(d, -0.5 * (rho_water - rho_air), beta[0], beta[1], beta[2], grad_beta[0], grad_beta[1],
                           grad_beta[2], grad_phi, (cudaStream_t)stream));
    return MG_OK;
}

int mg_num_levels(const mg_ctx *c) { return c ? c->nlev : 0; }

int mg_level_dims(const mg_ctx *c, int level, int dims[3])
{
    if (!c || !dims || level < 0 || level >= c->nlev) return fail(MG_ERR_ARG, "mg_level_dims: bad level");
    dims[0] = c->dims[level].nx;
    dims[1] = c->dims[level].ny;
    dims[2] = c->dims[level].nz;
    return MG_OK;
}

int mg_level_array(mg_ctx *c, int level, int which, double *out)
{
    g_err.clear();
    if (!c || !out || level < 0 || level >= c->nlev || which < 0 || which > 3)
        return fail(MG_ERR_ARG, "mg_level_array: bad argument");
    if (!aligned16({out})) return fail(MG_ERR_ARG, "mg_level_array: out must be 16-byte aligned");
    const LevelArrays<double> &L = c->L64[level];
    const double *src = which == 0 ? L.bx : which == 1 ? L.by : which == 2 ? L.bz : L.dinv;
    CK(cudaMemcpyAsync(out, src, c->dims[level].n() * sizeof(double), cudaMemcpyDeviceToDevice, c->s));
    return MG_OK;
}

uint64_t mg_kernel_launches(void) { return (uint64_t)mg::launch_count(); }

int mg_check_read(int *enabled, uint64_t *first, uint64_t *count)
{
    g_err.clear();
    if (!enabled || !first || !count) return fail(MG_ERR_ARG, "mg_check_read: null argument");
    unsigned long long f = 0, n = 0;
    const int r = mg::check_read(&f, &n);
    if (r < 0) return fail(MG_ERR_CUDA, "mg_check_read: reading the check record failed");
    *enabled = r;
    *first = f;
    *count = n;
    return MG_OK;
}

int mg_profile_read(mg_ctx *c, int group, int *count, double *ms_total)
{
    g_err.clear();
    if (!c || group < 0 || group >= MG_PROF_GROUPS) return fail(MG_ERR_ARG, "mg_profile_read: bad argument");
    int n = 0;
    double tot = 0.0;
    for (size_t i = 0; i + 1 < c->pused; i += 2) {
        if (c->pgroup[i / 2] != group) continue;
        float ms = 0.f;
        CK(cudaEventElapsedTime(&ms, c->pev[i], c->pev[i + 1]));
        tot += ms;
        n++;
    }
    if (count) *count = n;
    if (ms_total) *ms_total = tot;
    return MG_OK;
}

void mg_profile_reset(mg_ctx *c)
{
    if (c) c->pused = 0;
}

void mg_destroy(mg_ctx *c)
{
    if (!c) return;
    if (c->s) cudaStreamSynchronize(c->s);
    else cudaDeviceSynchronize();
    delete c;
}

}  // extern "C"
