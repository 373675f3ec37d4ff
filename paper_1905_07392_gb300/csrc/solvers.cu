// Linear solvers of one step: the cell-centred projection (Poisson), the
// three semi-implicit viscous Helmholtz solves and the nodal projection
// (paper Sec. "Numerical algorithm": geometric multigrid for EB systems with a
// Krylov method at the bottom).
//
// Every solve is conjugate gradients in FP64 preconditioned by one symmetric
// multigrid V-cycle: red-black Gauss-Seidel (red first on the way down, black
// first on the way up) for the 7-point cell-centred operators, a degree-3
// Chebyshev-Jacobi smoother for the 27-point nodal operator, averaging /
// full-weighting restriction, piecewise-constant / trilinear prolongation and
// an exact dense solve at the bottom.  The V-cycle runs in FP64 or FP32
// (EBV_FP32_REFINE); residuals, Krylov vectors and solution accumulation stay
// FP64, so FP32 only enters as a preconditioner.  Dot products use fixed-order
// block partials, so results are bitwise reproducible run to run.
#include <math.h>
#include <vector>

#include <cooperative_groups.h>

#include "ebv_internal.cuh"
#include "tma.cuh"
#include "fpbits.cuh"

namespace ebv {

// Device scalars of a solve (c->scal).  S_ALPHA = rz/pq and S_BETA = rz/rz_old
// are formed once, by the reduction that completes their last operand
// (kRedAlpha, kRedBeta), S_ISIG = 1/S_SIG where S_SIG is set: an FP64 division
// costs about twenty FP64-pipe slots, and with 2 FP64 lanes per SM the vector
// kernels spent most of their time on the same quotient in every thread
// (k_cg_update32 on 64^3: 9.3 us with it, 1.8 us without; 256^3: 28.5 -> 26.4;
// k_cg_pupdate32 on 64^3: 6.9 -> 1.8 us; FP64 k_cg_pupdate on 128^3: 10.8 -> 6.0).
enum { S_BB = 0, S_RR = 1, S_RZ = 2, S_RZOLD = 3, S_PQ = 4, S_REL = 16, S_PREV = 17, S_T2 = 18, S_SIG = 19,
       S_ISIG = 20, S_ALPHA = 21, S_BETA = 22 };

// ===========================================================================
// Reductions
// ===========================================================================
namespace {

// What a reduction does with its sum besides storing it.
enum { kRedSum = 0, kRedAlpha = 1, kRedBeta = 2 };

template <int kThreads>
__device__ inline double block_sum(double v)
{
    __shared__ double sm[kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = threadIdx.x < kThreads / 32 ? sm[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;
}

// block_sum<256> in fewer FP64 instructions: every warp's five shuffle steps
// are additions of all its lanes, so two warps add four threads' values each
// first (17 warp instructions on the FP64 pipe for 45).
__device__ inline double block_sum_flat(double v)
{
    __shared__ double sm[256];
    const int t = threadIdx.x;
    sm[t] = v;
    __syncthreads();
    if (t < 64) {
        v = (sm[t] + sm[t + 64]) + (sm[t + 128] + sm[t + 192]);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (t == 32) sm[255] = v;   // (read by its own warp before the shuffles)
    }
    __syncthreads();
    return t == 0 ? v + sm[255] : 0.0;
}

__device__ inline int block_linear() { return (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x; }

// The solvers run one system, or the three velocity components' viscous
// systems side by side: same grid and faces, own diagonals, vectors, scalars
// and loop control.  Launches on a component axis do the work of three (the
// levels that cannot fill the GPU cost launches and latency, not work: two
// steps at 64^3 21.3 ms with the components one after another, 17.1 ms
// together; viscous solves on 192 x 160 x 224 14.8 and 11.6 ms); each
// component's operations, and so its results, are those of a solve alone, and
// a component that has converged is frozen while the others go on.  3-D
// kernels carry the component in blockIdx.z (component-major), the others in
// blockIdx.y.
constexpr int kMaxComp = 3;
template <class T>
struct V3 {
    T *p[kMaxComp] = {};
    V3() = default;
    __host__ __device__ V3(T *a, T *b, T *c) : p{a, b, c} {}
    template <class U>
    __host__ __device__ V3(const V3<U> &o) : p{o.p[0], o.p[1], o.p[2]} {}
};
template <class T>
inline V3<T> one(T *p)
{
    return V3<T>(p, nullptr, nullptr);
}
// component and plane-block of a 3-D launch of nzb blocks per component
struct CompZ {
    int comp, z;
    __device__ explicit CompZ(int nzb)
    {
        comp = (int)blockIdx.z >= nzb ? ((int)blockIdx.z >= 2 * nzb ? 2 : 1) : 0;
        z = (int)blockIdx.z - comp * nzb;
    }
    __device__ int linear() const { return (z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x; }
};
// act: the loop condition word of component 0 (the others C_LEN apart), or
// null where every component runs
__device__ inline bool comp_off(const int *act, int comp) { return act && act[comp * C_LEN] == 0; }
constexpr int kScalLen = 32;                        // device scalars per component
constexpr size_t kPartLen = (size_t)1 << 20;        // doubles in c->part
constexpr size_t kPartComp = kPartLen / kMaxComp;   // of these per component when three run together
// joint control words, behind the components' own
enum { J_OUT = kMaxComp * C_LEN, J_IN, J_IT, J_NOUT };
__device__ inline int thread_linear() { return (threadIdx.z * blockDim.y + threadIdx.y) * blockDim.x + threadIdx.x; }

// 3-D blocks of 256 threads: block sum keyed on the linear thread index.
__device__ inline double block_sum3(double v)
{
    __shared__ double sm[8];
    const int t = thread_linear();
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t & 31) == 0) sm[t >> 5] = v;
    __syncthreads();
    double r = 0.0;
    if (t < 32) {
        r = t < 8 ? sm[t] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    return r;
}

// Block sum of per-thread partials of type T, returned in FP64.  FP64 keeps
// FP64 throughout (block_sum3).  FP32 partials are summed in FP32 within the
// warp (32 terms) and in FP64 across warps: FP64 arithmetic is scarce on this
// GPU, and per-cell FP64 work in a kernel that streams FP32 data made FP64 the
// bound of the FP32 operator apply.
template <class T>
__device__ inline double block_sum3_t(T v)
{
    if constexpr (sizeof(T) == 8) {
        return block_sum3(v);
    } else {
        __shared__ double sm[8];
        const int t = thread_linear();
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((t & 31) == 0) sm[t >> 5] = (double)v;
        __syncthreads();
        double r = 0.0;
        if (t < 32) {
            r = t < 8 ? sm[t] : 0.0;
            for (int o = 4; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
        }
        return r;
    }
}

// Block sum of FP32 partials of eight terms each, as wide as block_sum3_t's of
// two: FP32 over groups of 8 lanes (64 terms, seven additions deep with the
// thread's own), FP64 over the block's 32 groups.
__device__ inline double block_sum8(float v)
{
    __shared__ double sm[32];
    const int t = thread_linear();
    for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t & 7) == 0) sm[t >> 3] = (double)v;
    __syncthreads();
    double r = 0.0;
    if (t < 32) {
        r = sm[t];
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    return r;
}

// A term of a dot product that is summed in FP64: the product rounded in its
// operands' precision.
__device__ inline double dot_term(float a, float b) { return f32_to_f64(a * b); }
__device__ inline double dot_term(double a, double b) { return a * b; }

// Sum of n block partials in a fixed order, over a cluster of kRedCtas
// blocks: block q sums the slice [q n / kRedCtas, (q + 1) n / kRedCtas)
// (strided over its threads, then its block sum) and stores that sum in
// block 0's shared memory; after the cluster barrier block 0 adds the
// kRedCtas sums in rank order.  FP64 additions issue at about one per SM and
// cycle on this GPU, so a single block spent up to 16 us on the 32,768
// partials of a 256^3 refinement residual; the cluster spreads them over
// kRedCtas SMs.  The barrier is the hardware cluster barrier (no spin).
constexpr int kRedCtas = 8, kRedThreads = 512;
__global__ void __cluster_dims__(kRedCtas, 1, 1) __launch_bounds__(kRedThreads)
    k_reduce_final(const double *part, int n, double *out, double *scal, int post, const int *act)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ double csum[kRedCtas];
    cl.barrier_arrive();   // (no block's shared memory is written before that block runs)
    const int comp = blockIdx.y;
    part += comp * kPartComp;
    out += comp * kScalLen;
    scal += comp * kScalLen;
    const bool off = comp_off(act, comp);
    const int q = (int)cl.block_rank();
    const int lo = (int)((long long)n * q / kRedCtas), hi = (int)((long long)n * (q + 1) / kRedCtas);
    double v = 0.0;
    for (int s = lo + threadIdx.x; s < hi; s += kRedThreads) v += part[s];
    v = block_sum<kRedThreads>(v);
    cl.barrier_wait();
    if (threadIdx.x == 0) *cl.map_shared_rank(&csum[q], 0) = v;
    cl.sync();
    if (q == 0 && threadIdx.x == 0 && !off) {
        double t = 0.0;
        for (int r = 0; r < kRedCtas; r++) t += csum[r];
        *out = t;
        if (post == kRedAlpha) scal[S_ALPHA] = scal[S_RZ] / t;   // t = p.q
        if (post == kRedBeta) scal[S_BETA] = t / scal[S_RZOLD];  // t = r.z (unused by a first iteration)
    }
}

// k_reduce_final for at most kRedSmall partials: one small block per component.
// The sum of few terms is latency -- of the shuffle steps, which every warp
// takes through the FP64 pipe, and of the cluster's barriers (64^3, three
// components: 3.2 us over a cluster, 1.8 us so).
constexpr int kRedSmall = 1024, kRedSmallThreads = 128;
__device__ inline double small_sum(const double *part, int n, int t, double *sm)
{
    // t: 0 .. kRedSmallThreads - 1; sm: one word per warp; valid in t = 0
    double v = 0.0;
    for (int s = t; s < n; s += kRedSmallThreads) v += part[s];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t & 31) == 0) sm[t >> 5] = v;
    __syncthreads();
    return t == 0 ? (sm[0] + sm[1]) + (sm[2] + sm[3]) : 0.0;
}
__global__ void __launch_bounds__(kRedSmallThreads) k_reduce_small(const double *part, int n, double *out, double *scal,
                                                                   int post, const int *act)
{
    __shared__ double sm[kRedSmallThreads / 32];
    const int comp = blockIdx.y;
    part += comp * kPartComp;
    out += comp * kScalLen;
    scal += comp * kScalLen;
    const bool off = comp_off(act, comp);
    // the quotient's other operand, loaded meanwhile
    const double other = post == kRedAlpha ? scal[S_RZ] : (post == kRedBeta ? scal[S_RZOLD] : 0.0);
    const double t = small_sum(part, n, threadIdx.x, sm);
    if (threadIdx.x == 0 && !off) {
        *out = t;
        if (post == kRedAlpha) scal[S_ALPHA] = other / t;
        if (post == kRedBeta) scal[S_BETA] = t / other;
    }
}

__global__ void __launch_bounds__(256) k_dot(V3<const double> av, V3<const double> bv, int n,
                                             double *__restrict__ part)
{
    const double *__restrict__ a = av.p[blockIdx.y], *__restrict__ b = bv.p[blockIdx.y];
    part += blockIdx.y * kPartComp;
    double v = 0.0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        v += a[s] * b[s];
    v = block_sum<256>(v);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
}

}  // namespace

static void launch_reduce(Ctx *c, int nc, const double *part, int n, double *out, int post, const int *act)
{
    if (n <= kRedSmall)
        EBV_LAUNCH(c, k_reduce_small, dim3(1, nc), dim3(kRedSmallThreads), 0, part, n, out, c->scal, post, act);
    else
        EBV_LAUNCH(c, k_reduce_final, dim3(kRedCtas, nc), dim3(kRedThreads), 0, part, n, out, c->scal, post, act);
}
ebv_status reduce_sum(Ctx *c, const double *part, int nblocks, double *out_dev)
{
    launch_reduce(c, 1, part, nblocks, out_dev, kRedSum, nullptr);
    return EBV_OK;
}
// A sum of every component's partials into its scalar S; r.z and p.q of a CG
// iteration with the quotient they complete.
static void reduce_comp(Ctx *c, int nc, int nblocks, int S, int post = kRedSum, const int *act = nullptr,
                        const double *part = nullptr)
{
    launch_reduce(c, nc, part ? part : c->part, nblocks, c->scal + S, post, act);
}

namespace {

// ===========================================================================
// Cell-centred operator  (A x)_i = extra_i x_i + sum_faces beta_f (x_i - x_nb)
// (face coefficients include the box faces; x_nb = 0 outside the box).
// Each level stores extra (for coarsening) and the full diagonal
// diag = extra + sum of the 6 face coefficients (for the smoother and apply).
// ===========================================================================

// Cell-centred operator of one level: diagonal (precision T) and face
// coefficients (storage F, widened to T when read).
template <class T, class F = T>
struct CcOp {
    GridD g;
    const T *diag;
    const F *bx, *by, *bz;
    const T *dinv = nullptr;   // V-cycle operator: 1/diag (0 where diag <= 0)
};
// The operators of the components: one set of faces, their own diagonals.
template <class T, class F = T>
struct CcOp3 {
    CcOp<T, F> A;
    const T *diag[kMaxComp], *dinv[kMaxComp];
    __device__ CcOp<T, F> op(int comp) const
    {
        CcOp<T, F> B = A;
        B.diag = diag[comp];
        B.dinv = dinv[comp];
        return B;
    }
};
// The V-cycle's operator: in FP32 its faces are stored in BF16 (half the
// bytes of the face arrays every colour pass reads whole); the Krylov
// operator it preconditions keeps FP32 faces (CcOp<T>).  Built with
// EBV_VCYCLE_FP32_FACES (a measurement variant of the library, not the
// default) the V-cycle reads the FP32 faces instead, with the diagonal
// formed from them unrounded; everything else is the same code.
template <class T> struct VFace { using type = T; };
#ifdef EBV_VCYCLE_FP32_FACES
template <> struct VFace<float> { using type = float; };
constexpr bool kVcycleBf16 = false;
#else
template <> struct VFace<float> { using type = __nv_bfloat16; };
constexpr bool kVcycleBf16 = true;
#endif
template <class T> using VOp = CcOp<T, typename VFace<T>::type>;
template <class T> using VOp3 = CcOp3<T, typename VFace<T>::type>;

// Array layout of the cell-centred multigrid, by precision.  FP64 arrays are
// in the natural order (x fastest).  FP32 arrays -- the coefficients of every
// level, the V-cycle vectors and the inner Krylov vectors of the refinement
// solver -- are "row-split": within every x-row the even-i entries come first,
// then the odd-i ones.  A colour of a red-black pass then reads and writes
// contiguous half-rows (the cells of one colour in a row all have the same
// parity of i) instead of every other word of every sector; only the x-face
// coefficients are still read whole.  Rows keep their length and place, so
// neighbours in y and z are at the same offsets as in the natural order.
__host__ __device__ inline int spos(int m, int i) { return (i & 1) ? ((m + 1) >> 1) + (i >> 1) : (i >> 1); }
template <class T>
__host__ __device__ inline int cix(const GridD &g, int i, int j, int k)
{
    return (k * g.ny + j) * g.nx + (sizeof(T) == 4 ? spos(g.nx, i) : i);
}
template <class T>
__host__ __device__ inline int fidxT(const GridD &g, int d, int i, int j, int k)
{
    if (d == 0) return (k * g.ny + j) * (g.nx + 1) + (sizeof(T) == 4 ? spos(g.nx + 1, i) : i);
    if (d == 1) return (k * (g.ny + 1) + j) * g.nx + (sizeof(T) == 4 ? spos(g.nx, i) : i);
    return (k * g.ny + j) * g.nx + (sizeof(T) == 4 ? spos(g.nx, i) : i);
}

// Positions of cell (i,j,k), of its two x-neighbours and of its six faces in
// the level's layout (cix / fidxT), from the start of its row.  Row-split
// (FP32): with t = i/2 the even cells of a row sit at rc + t and the odd ones
// at rc + h + t (h = ceil(nx/2), rc the row's start), so the x-neighbours of
// an even cell are odd cells t-1 and t and those of an odd cell even cells t
// and t+1; x-face rows (nx+1 faces, hf = ceil((nx+1)/2)) start at rc + k ny + j.
// Natural order (FP64): the plain offsets.  In both, a y-face row is the cell
// row shifted by k nx and a z-face row the cell row itself.
struct CellPos {
    int c, xw, xe, fx0, fx1, fy0, fy1, fz0, fz1;
};
template <class T>
__device__ inline CellPos cell_pos(const GridD &g, int i, int j, int k)
{
    CellPos p;
    const int rc = (k * g.ny + j) * g.nx;
    if constexpr (sizeof(T) == 4) {
        const int t = i >> 1, odd = i & 1, h = (g.nx + 1) >> 1, hf = (g.nx + 2) >> 1;
        const int rf = rc + k * g.ny + j;
        p.c = rc + (odd ? h + t : t);
        p.xw = rc + (odd ? t : h + t - 1);
        p.xe = rc + (odd ? t + 1 : h + t);
        p.fx0 = rf + (odd ? hf + t : t);
        p.fx1 = rf + (odd ? t + 1 : hf + t);
    } else {
        p.c = rc + i;
        p.xw = p.c - 1;
        p.xe = p.c + 1;
        p.fx0 = rc + k * g.ny + j + i;
        p.fx1 = p.fx0 + 1;
    }
    p.fy0 = p.c + k * g.nx;
    p.fy1 = p.fy0 + g.nx;
    p.fz0 = p.c;
    p.fz1 = p.c + g.nx * g.ny;
    return p;
}

// off = init + sum beta x_nb.  A residual b - (diag x - sum) in FP64 starts its
// chain from b - diag x: seven multiply-adds instead of eight operations, in
// kernels that the FP64 pipe bounds (the three components' residual on 256^3
// 622 -> 553 us).
template <class T, class F>
__device__ inline void cc_row(const CcOp<T, F> &A, int i, int j, int k, const T *__restrict__ x,
                              T &diag, T &off, T init = T(0))
{
    const GridD &g = A.g;
    const CellPos p = cell_pos<T>(g, i, j, k);
    const int c = p.c;
    const T bxl = T(A.bx[p.fx0]), bxh = T(A.bx[p.fx1]);
    const T byl = T(A.by[p.fy0]), byh = T(A.by[p.fy1]);
    const T bzl = T(A.bz[p.fz0]), bzh = T(A.bz[p.fz1]);
    diag = A.diag[c];
    T s = init;
    if (i > 0) s += bxl * x[p.xw];
    if (i < g.nx - 1) s += bxh * x[p.xe];
    if (j > 0) s += byl * x[c - g.nx];
    if (j < g.ny - 1) s += byh * x[c + g.nx];
    if (k > 0) s += bzl * x[c - g.nx * g.ny];
    if (k < g.nz - 1) s += bzh * x[c + g.nx * g.ny];
    off = s;
}

// One colour of Gauss-Seidel in place: x_i = (b_i + sum beta x_nb) / diag for
// the cells of colour `color` ((i+j+k) mod 2); with zero_start the other
// colour reads as 0 (the sweep starts from x = 0) and x is not read.
// Thread (t, j, kk) owns the x-pair (2t, 2t+1) of row j on planes
// GS_PZ kk .. GS_PZ kk + GS_PZ - 1 and updates the cell of colour `color` in
// each: every lane works.  All operands of its GS_PZ updates are loaded before
// any result is stored (the updated cells are never read in the same pass), so
// the loads of all of them are in flight together.
// kCorr: the pass that follows the coarse-grid correction.  Since a pass
// never reads the old value of the cells it updates, prolongation (x += the
// coarse correction xc of the parent cell, on uncovered cells) is folded into
// the neighbour reads: x_nb + xc(parent(nb)), the very sums a separate
// prolongation kernel would store.  A covered neighbour's face coefficient is
// 0, so adding to it changes nothing either.
constexpr int GS_PZ = 2;

// The Gauss-Seidel value of cell (i,j,k): (b + sum beta x_nb) / diag, 0 on
// cells with no diagonal (see k_cc_gs for kCorr and zero_start), formed with
// the stored inverse diagonal: an FP64 division is about twenty FP64-pipe
// operations, three times the rest of the cell (a 128^3 FP64 colour pass took
// 33.7 us with it, 16.8 without).
template <class T, bool kCorr>
__device__ inline T gs_cell(const VOp<T> &A, const T *__restrict__ x, const T *__restrict__ b, int i, int j,
                            int k, int zero_start, const T *__restrict__ xc, const GridD &gc)
{
    const GridD &g = A.g;
    const int sy = g.nx, sz = g.nx * g.ny;
    const CellPos p = cell_pos<T>(g, i, j, k);
    const int c = p.c;
    const T di = A.dinv[c], bc = b[c];
    T off = sizeof(T) == 8 ? bc : T(0);   // (FP64: the chain starts from b, one operation less)
    if (!zero_start) {
        const T bxl = T(A.bx[p.fx0]), bxh = T(A.bx[p.fx1]);
        const T byl = T(A.by[p.fy0]), byh = T(A.by[p.fy1]);
        const T bzl = T(A.bz[p.fz0]), bzh = T(A.bz[p.fz1]);
        auto cor = [&](int ii, int jj, int kq) -> T {
            return kCorr ? xc[cix<T>(gc, ii >> 1, jj >> 1, kq >> 1)] : T(0);
        };
        const T xw = i > 0 ? (kCorr ? x[p.xw] + cor(i - 1, j, k) : x[p.xw]) : T(0);
        const T xe = i < g.nx - 1 ? (kCorr ? x[p.xe] + cor(i + 1, j, k) : x[p.xe]) : T(0);
        const T xs = j > 0 ? (kCorr ? x[c - sy] + cor(i, j - 1, k) : x[c - sy]) : T(0);
        const T xn = j < g.ny - 1 ? (kCorr ? x[c + sy] + cor(i, j + 1, k) : x[c + sy]) : T(0);
        const T xd = k > 0 ? (kCorr ? x[c - sz] + cor(i, j, k - 1) : x[c - sz]) : T(0);
        const T xu = k < g.nz - 1 ? (kCorr ? x[c + sz] + cor(i, j, k + 1) : x[c + sz]) : T(0);
        if (i > 0) off += bxl * xw;
        if (i < g.nx - 1) off += bxh * xe;
        if (j > 0) off += byl * xs;
        if (j < g.ny - 1) off += byh * xn;
        if (k > 0) off += bzl * xd;
        if (k < g.nz - 1) off += bzh * xu;
    }
    return (sizeof(T) == 8 ? off : bc + off) * di;
}

// kDot (the last pass of a V-cycle on the finest level): also block partials
// of b.x over both cells of every x-pair -- the updated one and its partner of
// the other colour, which this pass does not change -- i.e. r.z of the
// preconditioned CG, without a separate pass over both vectors.
template <class T, bool kCorr = false, bool kDot = false>
__global__ void __launch_bounds__(256) k_cc_gs(VOp3<T> A3, V3<T> xv, V3<const T> bv, int nzb, const int *act,
                                               int color, int zero_start, V3<const T> xcv = V3<const T>(),
                                               GridD gc = GridD(), double *__restrict__ part = nullptr)
{
    const CompZ cz(nzb);
    if (comp_off(act, cz.comp)) return;
    const VOp<T> A = A3.op(cz.comp);
    T *__restrict__ x = xv.p[cz.comp];
    const T *__restrict__ b = bv.p[cz.comp], *__restrict__ xc = xcv.p[cz.comp];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int kk = cz.z * blockDim.z + threadIdx.z;
    const GridD &g = A.g;
    const bool own = 2 * t < g.nx && j < g.ny;
    if (!kDot && !own) return;   // (with kDot every thread reaches the block sum)
    T val[GS_PZ];
    int cc[GS_PZ];
#pragma unroll
    for (int h = 0; h < GS_PZ; h++) {
        const int k = GS_PZ * kk + h;
        const int i = 2 * t + ((j + k + color) & 1);
        cc[h] = -1;
        val[h] = T(0);
        if (!own || k >= g.nz || i >= g.nx) continue;
        cc[h] = cix<T>(g, i, j, k);
        val[h] = gs_cell<T, kCorr>(A, x, b, i, j, k, zero_start, xc, gc);
    }
    T dot = T(0);
#pragma unroll
    for (int h = 0; h < GS_PZ; h++) {
        if (zero_start) {
            const int k = GS_PZ * kk + h;
            const int io = 2 * t + 1 - ((j + k + color) & 1);
            if (k < g.nz && io < g.nx) x[cix<T>(g, io, j, k)] = T(0);
        }
        if (cc[h] >= 0) x[cc[h]] = val[h];
        if constexpr (kDot) {
            const int k = GS_PZ * kk + h;
            const int io = 2 * t + 1 - ((j + k + color) & 1);
            if (cc[h] >= 0) dot += b[cc[h]] * val[h];
            if (own && k < g.nz && io < g.nx) {
                const int co = cix<T>(g, io, j, k);
                dot += b[co] * x[co];
            }
        }
    }
    if constexpr (kDot) {
        const double sdot = block_sum3_t<T>(dot);
        if (thread_linear() == 0) part[cz.comp * kPartComp + cz.linear()] = sdot;
    }
}

// The colour pass of k_cc_gs (plain form: no coarse correction, no r.z) for
// FP32 levels whose rows split into half-rows of a multiple of 4 cells (nx a
// multiple of 8): a thread updates 4 consecutive cells of its colour in one
// half-row of each of its kPz planes.  The row-split layout makes b, 1/diag,
// the y and z neighbours (the other colour at the same half-row position in
// the adjacent rows), the y and z faces and the result 16-byte (FP32) or
// 8-byte (BF16) vectors; the x neighbours are the other half-row's 4 values
// plus one beyond, the x faces 8 scalars.  Per cell the same operations in
// the same order as gs_cell, so the result is bit for bit that of k_cc_gs.
template <class F>
__device__ inline void load4(const F *p, float v[4])
{
    if constexpr (sizeof(F) == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const uint2 q = *reinterpret_cast<const uint2 *>(p);
        const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162 *>(&q.x);
        const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162 *>(&q.y);
        v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
    }
}

// kPz = 1 asks for 5 resident blocks per SM (at most 51 registers), kPz = 2
// for 4: one plane per thread and more warps, or two and more loads per warp.
// kCorr: the pass after the coarse-grid correction, as in k_cc_gs (each
// neighbour value plus its parent's coarse correction xc, level gc); its
// coarse rows in registers ask for 3 resident blocks per SM.
template <int kPz, bool kCorr = false>
__global__ void __launch_bounds__(256, kCorr ? 3 : (kPz == 1 ? 5 : 4)) k_cc_gs4(VOp3<float> A3, V3<float> xv,
                                                                 V3<const float> bv, int nzb, const int *act, int color,
                                                                 int zero_start, V3<const float> xcv = V3<const float>(),
                                                                 GridD gc = GridD())
{
    using F = typename VFace<float>::type;
    const CompZ cz(nzb);
    if (comp_off(act, cz.comp)) return;
    const VOp<float> A = A3.op(cz.comp);
    float *__restrict__ x = xv.p[cz.comp];
    const float *__restrict__ b = bv.p[cz.comp], *__restrict__ xc = xcv.p[cz.comp];
    const GridD &g = A.g;
    const int hx = g.nx >> 1;
    const int t0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int kb = (cz.z * blockDim.z + threadIdx.z) * kPz;
    if (t0 >= hx || j >= g.ny) return;
    const int sy = g.nx, sz = g.nx * g.ny;
    float val[kPz][4];
    int pos[kPz], oth[kPz];
#pragma unroll
    for (int h = 0; h < kPz; h++) {
        const int k = kb + h;
        pos[h] = -1;
        if (k >= g.nz) continue;
        const int par = (color + j + k) & 1;            // i parity of this row's cells of the colour
        const int rc = (k * g.ny + j) * g.nx;
        const int c = rc + (par ? hx : 0) + t0;         // own half-row, cells t0 .. t0+3
        const int o = rc + (par ? 0 : hx) + t0;         // the other half-row, same positions
        pos[h] = c;
        oth[h] = o;
        float bc[4], di[4];
        load4(b + c, bc);
        load4(A.dinv + c, di);
        float off[4] = {0.f, 0.f, 0.f, 0.f};
        if (!zero_start) {
            float xo[4], xs[4], xn[4], xd[4], xu[4], fy0[4], fy1[4], fz0[4], fz1[4];
            load4(x + o, xo);
            const float xb = par ? (t0 + 4 < hx ? x[o + 4] : 0.f) : (t0 > 0 ? x[o - 1] : 0.f);
            if (j > 0) load4(x + c - sy, xs);
            if (j < g.ny - 1) load4(x + c + sy, xn);
            if (k > 0) load4(x + c - sz, xd);
            if (k < g.nz - 1) load4(x + c + sz, xu);
            load4(A.by + c + k * g.nx, fy0);
            load4(A.by + c + k * g.nx + g.nx, fy1);
            load4(A.bz + c, fz0);
            load4(A.bz + c + sz, fz1);
            const int rf = rc + k * g.ny + j, hf = (g.nx + 2) >> 1;
            // kCorr: the parents of the 4 cells' neighbours are the coarse cells
            // t0-1 .. t0+4 of the parent row and t0 .. t0+3 of the rows of the y
            // and z neighbours' parents; in the coarse row-split layout the even
            // and odd ones of t0 .. t0+3 are two 8-byte pairs of each row
            float cw[6] = {}, cs[4] = {}, cn[4] = {}, cd[4] = {}, cu[4] = {};
            if constexpr (kCorr) {
                const int hxc = gc.nx >> 1, tc = t0 >> 1;
                auto row4 = [&](int J, int K, float *o) {
                    const float *r0 = xc + (K * gc.ny + J) * gc.nx;
                    const float2 ev = *reinterpret_cast<const float2 *>(r0 + tc);
                    const float2 od = *reinterpret_cast<const float2 *>(r0 + hxc + tc);
                    o[0] = ev.x; o[1] = od.x; o[2] = ev.y; o[3] = od.y;
                };
                row4(j >> 1, k >> 1, cw + 1);
                const float *r0 = xc + ((k >> 1) * gc.ny + (j >> 1)) * gc.nx;
                cw[0] = t0 > 0 ? r0[hxc + tc - 1] : 0.f;          // coarse t0 - 1 (odd)
                cw[5] = t0 + 4 < gc.nx ? r0[tc + 2] : 0.f;         // coarse t0 + 4 (even)
                if (j > 0) row4((j - 1) >> 1, k >> 1, cs);
                if (j < g.ny - 1) row4((j + 1) >> 1, k >> 1, cn);
                if (k > 0) row4(j >> 1, (k - 1) >> 1, cd);
                if (k < g.nz - 1) row4(j >> 1, (k + 1) >> 1, cu);
            }
#pragma unroll
            for (int m = 0; m < 4; m++) {
                const int t = t0 + m, i = 2 * t + par;
                const float bxl = float(A.bx[rf + (par ? hf + t : t)]);
                const float bxh = float(A.bx[rf + (par ? t + 1 : hf + t)]);
                float xw = par ? xo[m] : (m ? xo[m - 1] : xb);
                float xe = par ? (m < 3 ? xo[m + 1] : xb) : xo[m];
                float ys = xs[m], yn = xn[m], zd = xd[m], zu = xu[m];
                if constexpr (kCorr) {
                    // parent of i - 1 is coarse t - 1 + par, of i + 1 coarse t + par
                    if (i > 0) xw = xw + (par ? cw[m + 1] : cw[m]);
                    if (i < g.nx - 1) xe = xe + (par ? cw[m + 2] : cw[m + 1]);
                    if (j > 0) ys = ys + cs[m];
                    if (j < g.ny - 1) yn = yn + cn[m];
                    if (k > 0) zd = zd + cd[m];
                    if (k < g.nz - 1) zu = zu + cu[m];
                }
                float s = 0.f;
                if (i > 0) s += bxl * xw;
                if (i < g.nx - 1) s += bxh * xe;
                if (j > 0) s += fy0[m] * ys;
                if (j < g.ny - 1) s += fy1[m] * yn;
                if (k > 0) s += fz0[m] * zd;
                if (k < g.nz - 1) s += fz1[m] * zu;
                off[m] = s;
            }
        }
#pragma unroll
        for (int m = 0; m < 4; m++) val[h][m] = (bc[m] + off[m]) * di[m];
    }
#pragma unroll
    for (int h = 0; h < kPz; h++) {
        if (pos[h] < 0) continue;
        if (zero_start) *reinterpret_cast<float4 *>(x + oth[h]) = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4 *>(x + pos[h]) = make_float4(val[h][0], val[h][1], val[h][2], val[h][3]);
    }
}
inline bool gs4_ok(const GridD &g) { return (g.nx & 7) == 0; }
inline dim3 gs4_grid(const GridD &g, dim3 bk, int pz)
{
    const int nq = (g.nx >> 1) / 4, nzg = (g.nz + pz - 1) / pz;
    return dim3((nq + bk.x - 1) / bk.x, (g.ny + bk.y - 1) / bk.y, (nzg + bk.z - 1) / bk.z);
}
// a 3-D grid for nc components
inline dim3 comp_grid(dim3 g, int nc) { return dim3(g.x, g.y, g.z * nc); }
inline void launch_gs4(cudaStream_t st, dim3 bk, int pz, const VOp3<float> &A, V3<float> x, V3<const float> b, int color,
                       int zs)
{
    const dim3 gr = gs4_grid(A.A.g, bk, pz);
    if (pz == 1) k_cc_gs4<1><<<gr, bk, 0, st>>>(A, x, b, gr.z, nullptr, color, zs);
    else k_cc_gs4<2><<<gr, bk, 0, st>>>(A, x, b, gr.z, nullptr, color, zs);
}

// ---------------------------------------------------------------------------
// A whole red-black sweep in one pass (FP32 levels with nx a multiple of 16):
// the cells of colour c0 from the old values of the other colour, then the
// other colour from the new c0 values, read from x_in and written to x_out
// (the two passes in place give the same values, bit for bit: each cell is
// formed by the same operations in the same order as in gs_cell).
//
// A block owns a tile of RB_TX x RB_TY cells of every plane of a chunk of
// planes [z0, z1) and marches it in z.  Step m forms the first colour on
// plane m over the tile and a one-cell ring around it (the ring's values are
// the neighbours of the tile's second-colour cells; neighbouring blocks form
// them too), keeping three planes of these in shared memory, then the second
// colour on plane m-1 and writes plane m-1 (both colours).  Every operand
// comes in by TMA tile loads two steps ahead, completed on mbarriers: x (tile
// + 2-cell ring), b and 1/diag (tile + 1-cell ring), and the x, y and z face
// coefficients -- the x faces from a copy whose rows are padded to 16-byte
// strides (bxp: even faces then odd faces, each half RB_HXP(nx) long), since
// the stored rows hold nx + 1 entries.  No global load is left inside a
// step.  Per sweep every array is read once from DRAM (the rings come from
// L2) and x written once: 22 bytes per cell with BF16 faces instead of 28
// for two colour passes.
//
// Out-of-range tile coordinates load as zeros and the cells there are
// skipped; a neighbour outside the box is not read (the same tests as in
// gs_cell).  Each wait on a load is bounded (spin cycles of clock64); a wait
// that gives up sets E_TIMEOUT in ctl[C_ERR], waits (bounded) for the loads
// still in flight and ends the block, so the solve stops with that status
// instead of hanging.
// kZero: x_in is zero (not read).  kCorr: the first colour reads
// x_in + the coarse correction of the neighbour's parent (prolongation
// folded in, as in k_cc_gs); the coarse planes of the tile's parents come by
// TMA too (a RB_KW x 2 x RB_KR box per coarse plane, a three-slot ring, one
// new plane every other step), and each cell reads its four distinct parent
// values (its own parent and, per axis, the next coarse cell on the
// neighbour's side) once.  The first colour's results keep only that
// colour's half of each row.  kDot: also the partial b.x_out of every
// (plane, tile), part[plane * ntiles + tile], summed over the same cells in
// the same order as k_cc_gs2_dot, which forms them with the colour passes:
// in FP32 over a thread's cells and within the warp, in FP64 over the warps
// (FP64 arithmetic is scarce on this GPU: FP64 warp sums made each plane's
// partial cost more than the plane's loads).
constexpr int RB_TX = 64;                 // tile cells along x
constexpr int RB_HW = RB_TX / 2;          // half-row positions per tile
constexpr int RB_TY = 16;                 // tile rows
constexpr int RB_THREADS = RB_TY * (RB_HW / 2);   // one thread per 2 positions of a tile row
constexpr int RB_XW = RB_HW + 8;          // x / cell box width (FP32): 4 positions each side
constexpr int RB_FW = RB_HW + 16;         // face box width: 8 positions each side
constexpr int RB_XR = RB_TY + 4;          // rows of the x box
constexpr int RB_CR = RB_TY + 2;          // rows of the cell boxes (b, 1/diag, x and z faces, results)
constexpr int RB_YR = RB_TY + 3;          // rows of the y-face box
constexpr int RB_NBAR = 3;                // mbarriers (steps in flight + 1)
constexpr int RB_KW = 24;                 // coarse box width (half-row positions of the coarse level)
constexpr int RB_KR = RB_TY / 2 + 2;      // coarse box rows
static_assert(RB_THREADS == 256, "one thread per 2 positions of each tile row");
// half-row length of the padded x-face copy: nx/2 + 1 even faces, rounded up to 8
__host__ __device__ inline int rb_hxp(int nx) { return ((nx / 2 + 1) + 7) / 8 * 8; }

constexpr int al128(int b) { return (b + 127) / 128 * 128; }
template <class F>
struct RbSmem {
    static constexpr int bX = RB_XW * 2 * RB_XR * 4, bC = RB_XW * 2 * RB_CR * 4;
    static constexpr int bY = RB_FW * 2 * RB_YR * (int)sizeof(F), bZ = RB_FW * 2 * RB_CR * (int)sizeof(F);
    static constexpr int bR = RB_XW * RB_CR * 4, bK = RB_KW * 2 * RB_KR * 4;
    static constexpr int kX = al128(bX), kC = al128(bC), kY = al128(bY), kZ = al128(bZ);
    static constexpr int kR = al128(bR), kK = al128(bK);
    // x: planes m-1, m, m+1 and one ahead; b, 1/diag, x and y faces: m-1, m
    // and one ahead; z faces: face planes m-1 .. m+1 and one ahead; results
    // of the first colour (only its half of each row): planes m-2 .. m;
    // coarse correction (kCorr): coarse planes (m-1)/2 .. (m+1)/2 and one ahead
    static constexpr int oX = 0, oB = oX + 4 * kX, oD = oB + 3 * kC, oY = oD + 3 * kC, oZ = oY + 3 * kY;
    static constexpr int oXF = oZ + 4 * kZ, oR = oXF + 3 * kZ, oK = oR + 3 * kR, oBar = oK + 3 * kK;
    static constexpr int oMisc = oBar + 64;
    static constexpr int bytes = oMisc + 128;
};

template <class F>
struct RbArgs {
    GridD g;                // this level
    V3<float> xout;
    double *part;           // kDot partials
    int *ctl;
    const int *act;
    int nzb;                // chunks per component
    int c0, kz;             // first colour, planes per chunk
    long long spin;         // bound of one wait, clock64 cycles
};

struct RbMaps {
    struct Comp {
        CUtensorMap x, b, d, xc;   // xc: the coarse correction (kCorr)
    };
    CUtensorMap fx, fy, fz;
    Comp v[kMaxComp];
};

// Coarse planes step q loads (kCorr): step m needs coarse planes (m-1)/2 ..
// (m+1)/2 (floor division); the first step loads both of its, every later
// step the plane (m+1)/2 when it is new (m+1 even).  With three ring slots a
// load never lands on a slot a step in flight still reads.
__device__ inline int rb_coarse_count(int q, int m) { return q == 0 ? 2 : (((m + 1) & 1) == 0 ? 1 : 0); }

template <class F>
__device__ inline void rb_issue(unsigned char *sm, uint64_t *bar, int q, int m0, int p0, int y0, bool zero,
                                bool corr, const RbMaps &tm, const RbMaps::Comp &tc)
{
    using S = RbSmem<F>;
    const int m = m0 + q;
    uint64_t *b = bar + q % RB_NBAR;
    uint32_t bytes = 2 * S::bC + S::bY + 2 * S::bZ;
    if (!zero) bytes += (q == 0 ? 3 : 1) * S::bX;
    if (q == 0) bytes += S::bZ;
    if (corr) bytes += rb_coarse_count(q, m) * S::bK;
    mbar_arrive_expect_tx(b, bytes);
    if (corr) {
        const int nk = rb_coarse_count(q, m), cfirst = q == 0 ? ((m - 1) >> 1) : ((m + 1) >> 1);
        for (int t = 0; t < nk; t++) {
            const int C = cfirst + t;
            tma_load_4d(sm + S::oK + ((C + 3) % 3) * S::kK, &tc.xc, p0 / 2 - 4, 0, y0 / 2 - 1, C, b);
        }
    }
    if (!zero) {
        if (q == 0) {
            tma_load_4d(sm + S::oX + ((m - 1 + 8) & 3) * S::kX, &tc.x, p0 - 4, 0, y0 - 2, m - 1, b);
            tma_load_4d(sm + S::oX + ((m + 8) & 3) * S::kX, &tc.x, p0 - 4, 0, y0 - 2, m, b);
        }
        tma_load_4d(sm + S::oX + ((m + 1 + 8) & 3) * S::kX, &tc.x, p0 - 4, 0, y0 - 2, m + 1, b);
    }
    const int sb = (m + 3) % 3;
    tma_load_4d(sm + S::oB + sb * S::kC, &tc.b, p0 - 4, 0, y0 - 1, m, b);
    tma_load_4d(sm + S::oD + sb * S::kC, &tc.d, p0 - 4, 0, y0 - 1, m, b);
    tma_load_4d(sm + S::oY + sb * S::kY, &tm.fy, p0 - 8, 0, y0 - 1, m, b);
    tma_load_4d(sm + S::oXF + sb * S::kZ, &tm.fx, p0 - 8, 0, y0 - 1, m, b);
    if (q == 0) tma_load_4d(sm + S::oZ + ((m + 8) & 3) * S::kZ, &tm.fz, p0 - 8, 0, y0 - 1, m, b);
    tma_load_4d(sm + S::oZ + ((m + 1 + 8) & 3) * S::kZ, &tm.fz, p0 - 8, 0, y0 - 1, m + 1, b);
}

// Two consecutive face coefficients from shared memory (4- or 8-byte aligned) as floats.
template <class F>
__device__ inline float2 ld2f(const F *p)
{
    if constexpr (sizeof(F) == 4) {
        return *reinterpret_cast<const float2 *>(p);
    } else {
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162 *>(p);
        return make_float2(__low2float(v), __high2float(v));
    }
}

template <class F, bool kZero, bool kCorr, bool kDot>
__global__ void __launch_bounds__(RB_THREADS, 2)
    k_cc_rb_sweep(const __grid_constant__ RbMaps tm, const RbArgs<F> a)
{
    using S = RbSmem<F>;
    extern __shared__ __align__(128) unsigned char sm[];
    const GridD &g = a.g;
    const int hx = g.nx >> 1;
    const int p0 = blockIdx.x * RB_HW, y0 = blockIdx.y * RB_TY;
    const CompZ cz(a.nzb);
    const int z0 = cz.z * a.kz, z1 = min(g.nz, z0 + a.kz);
    if (z0 >= z1 || comp_off(a.act, cz.comp)) return;
    const RbMaps::Comp &tc = tm.v[cz.comp];
    int *const ctl = a.ctl + cz.comp * C_LEN;
    float *const xout = a.xout.p[cz.comp];
    const int tid = threadIdx.x, c1 = 1 - a.c0;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + S::oBar);
    int *flag = reinterpret_cast<int *>(sm + S::oMisc);
    double *wsum = reinterpret_cast<double *>(sm + S::oMisc + 16);
    const int m0 = z0 - 1, nstep = z1 - z0 + 2;
    auto X = [&](int pl) { return reinterpret_cast<const float *>(sm + S::oX + ((pl + 8) & 3) * S::kX); };
    auto Bv = [&](int pl) { return reinterpret_cast<const float *>(sm + S::oB + ((pl + 3) % 3) * S::kC); };
    auto Dv = [&](int pl) { return reinterpret_cast<const float *>(sm + S::oD + ((pl + 3) % 3) * S::kC); };
    auto FX = [&](int pl) { return reinterpret_cast<const F *>(sm + S::oXF + ((pl + 3) % 3) * S::kZ); };
    auto FY = [&](int pl) { return reinterpret_cast<const F *>(sm + S::oY + ((pl + 3) % 3) * S::kY); };
    auto FZ = [&](int pl) { return reinterpret_cast<const F *>(sm + S::oZ + ((pl + 8) & 3) * S::kZ); };
    // results of the first colour: row r, position q of that row's first-colour half
    auto R = [&](int pl) { return reinterpret_cast<float *>(sm + S::oR + ((pl + 3) % 3) * S::kR); };
    // the staged coarse correction (kCorr): coarse plane K, the entry of
    // coarse cell I in box row rw (a row offset from cor_row)
    auto Kpl = [&](int K) { return reinterpret_cast<const float *>(sm + S::oK + ((K + 3) % 3) * S::kK); };
    auto cor_row = [&](int J) { return (J - (y0 / 2 - 1)) * 2 * RB_KW; };
    auto cor_col = [&](int I) { return (I & 1) * RB_KW + (I >> 1) - (p0 / 2 - 4); };
    if (smem_u32(sm) & 127) {   // tile destinations must be 128-byte aligned: report, load nothing
        if (tid == 0) atomicCAS(ctl + C_ERR, 0, E_SMEM);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < RB_NBAR; s++) mbar_init(bar + s, 1);
        *flag = 0;
        mbar_fence_init();
    }
    __syncthreads();
    if (tid == 0) {
        rb_issue<F>(sm, bar, 0, m0, p0, y0, kZero, kCorr, tm, tc);
        rb_issue<F>(sm, bar, 1, m0, p0, y0, kZero, kCorr, tm, tc);
    }
    // second colour and output: thread -> positions pq, pq+1 of both halves of tile row r
    const int r = tid >> 4, pq = p0 + 2 * (tid & 15);
    const int j2 = y0 + r;
    const bool own = j2 < g.ny && pq < hx;
    for (int q = 0; q < nstep; q++) {
        const int m = m0 + q;
        if (!mbar_wait_bounded(bar + q % RB_NBAR, (q / RB_NBAR) & 1, a.spin)) atomicExch(flag, 1);
        // first colour on plane m over the tile (two positions per thread)
        // and its one-cell ring (82 cells)
        if (m >= 0 && m < g.nz) {
            const float *X0 = X(m - 1), *X1 = X(m), *X2 = X(m + 1), *Bm = Bv(m), *Dm = Dv(m);
            const F *Fx = FX(m), *Fy = FY(m), *Fz0 = FZ(m), *Fz1 = FZ(m + 1);
            float *Rm = R(m);
            const int k = m;
            // coarse planes of the parents (k >> 1) and of the other z neighbour
            const float *Kk = nullptr, *Ko = nullptr;
            if (kCorr) {
                Kk = Kpl(k >> 1);
                Ko = Kpl((k >> 1) - 1 + 2 * (k & 1));
            }
            auto XI = [&](const float *Xp, int rr, int h2, int qq) { return Xp[(rr * 2 + h2) * RB_XW + qq]; };
            // one cell (i = 2p + h, j) of box row r1: the operations of gs_cell
            auto cell = [&](int r1, int j, int h, int p) {
                const int i = 2 * p + h, qx = p - p0 + 4, qf = p - p0 + 8;
                const int cc = (r1 * 2 + h) * RB_XW + qx;
                float off = 0.f;
                if (!kZero) {
                    const int rx = r1 + 1;
                    // x faces i (lo) and i + 1 (hi): even faces in half 0, odd in half 1
                    const float bxl = float(Fx[(r1 * 2 + h) * RB_FW + qf]);
                    const float bxh = float(Fx[(r1 * 2 + 1 - h) * RB_FW + qf + h]);
                    const float fy0 = float(Fy[(r1 * 2 + h) * RB_FW + qf]);
                    const float fy1 = float(Fy[((r1 + 1) * 2 + h) * RB_FW + qf]);
                    const float fz0 = float(Fz0[(r1 * 2 + h) * RB_FW + qf]);
                    const float fz1 = float(Fz1[(r1 * 2 + h) * RB_FW + qf]);
                    float xw = h ? XI(X1, rx, 0, qx) : XI(X1, rx, 1, qx - 1);
                    float xe = h ? XI(X1, rx, 0, qx + 1) : XI(X1, rx, 1, qx);
                    float xs = XI(X1, rx - 1, h, qx), xn = XI(X1, rx + 1, h, qx);
                    float xd = XI(X0, rx, h, qx), xu = XI(X2, rx, h, qx);
                    if (kCorr) {
                        // the neighbours' parents: this cell's (I = p, J, K) or, one
                        // per axis, the next coarse cell on the neighbour's side
                        const int rj = cor_row(j >> 1), ro = cor_row((j >> 1) - 1 + 2 * (j & 1));
                        const float co = Kk[rj + cor_col(p)], cx = Kk[rj + cor_col(h ? p + 1 : p - 1)];
                        const float cy = Kk[ro + cor_col(p)], cz = Ko[rj + cor_col(p)];
                        if (i > 0) xw = xw + (h ? co : cx);
                        if (i < g.nx - 1) xe = xe + (h ? cx : co);
                        if (j > 0) xs = xs + ((j & 1) ? co : cy);
                        if (j < g.ny - 1) xn = xn + ((j & 1) ? cy : co);
                        if (k > 0) xd = xd + ((k & 1) ? co : cz);
                        if (k < g.nz - 1) xu = xu + ((k & 1) ? cz : co);
                    }
                    if (i > 0) off += bxl * xw;
                    if (i < g.nx - 1) off += bxh * xe;
                    if (j > 0) off += fy0 * xs;
                    if (j < g.ny - 1) off += fy1 * xn;
                    if (k > 0) off += fz0 * xd;
                    if (k < g.nz - 1) off += fz1 * xu;
                }
                Rm[r1 * RB_XW + qx] = (Bm[cc] + off) * Dm[cc];
            };
            {   // the tile: positions p, p + 1 of row y0 + r, paired shared-memory loads
                const int j = y0 + r, h = (a.c0 + j + m) & 1, p = pq;
                if (own) {
                    const int r1 = r + 1, rx = r1 + 1, qx = p - p0 + 4, qf = p - p0 + 8;
                    const int ch = (r1 * 2 + h) * RB_XW + qx, cx = (rx * 2 + h) * RB_XW + qx;
                    const int co = (rx * 2 + 1 - h) * RB_XW + qx;   // the other half, same positions
                    const float2 bb = *reinterpret_cast<const float2 *>(Bm + ch);
                    const float2 dd = *reinterpret_cast<const float2 *>(Dm + ch);
                    float v[2];
                    if (!kZero) {
                        const float2 xs = *reinterpret_cast<const float2 *>(X1 + cx - 2 * RB_XW);
                        const float2 xn = *reinterpret_cast<const float2 *>(X1 + cx + 2 * RB_XW);
                        const float2 xd = *reinterpret_cast<const float2 *>(X0 + cx);
                        const float2 xu = *reinterpret_cast<const float2 *>(X2 + cx);
                        const float2 xo = *reinterpret_cast<const float2 *>(X1 + co);
                        // h = 1: neighbours (p, p+1 | p+1, p+2) of half 0; h = 0: (p-1, p | p, p+1) of half 1
                        const float xb = h ? X1[co + 2] : X1[co - 1];
                        const float xw2[2] = {h ? xo.x : xb, h ? xo.y : xo.x};
                        const float xe2[2] = {h ? xo.y : xo.x, h ? xb : xo.y};
                        const float2 fxl = ld2f(Fx + (r1 * 2 + h) * RB_FW + qf);
                        const float fxh0 = float(Fx[(r1 * 2 + 1 - h) * RB_FW + qf + h]);
                        const float fxh1 = float(Fx[(r1 * 2 + 1 - h) * RB_FW + qf + h + 1]);
                        const float2 fy0 = ld2f(Fy + (r1 * 2 + h) * RB_FW + qf);
                        const float2 fy1 = ld2f(Fy + ((r1 + 1) * 2 + h) * RB_FW + qf);
                        const float2 fz0 = ld2f(Fz0 + (r1 * 2 + h) * RB_FW + qf);
                        const float2 fz1 = ld2f(Fz1 + (r1 * 2 + h) * RB_FW + qf);
                        const float bxl[2] = {fxl.x, fxl.y}, bxh[2] = {fxh0, fxh1};
                        const float ys0[2] = {fy0.x, fy0.y}, ys1[2] = {fy1.x, fy1.y};
                        const float zs0[2] = {fz0.x, fz0.y}, zs1[2] = {fz1.x, fz1.y};
                        const float vs[2] = {xs.x, xs.y}, vn[2] = {xn.x, xn.y}, vd[2] = {xd.x, xd.y};
                        const float vu[2] = {xu.x, xu.y}, bv[2] = {bb.x, bb.y}, dv[2] = {dd.x, dd.y};
                        // the parents of the neighbours of cells 2(p+e)+h: coarse cells
                        // p+e (co) and, per axis, the next one on the neighbour's side
                        float co[2] = {0.f, 0.f}, cx[2] = {0.f, 0.f}, cy[2] = {0.f, 0.f}, cz[2] = {0.f, 0.f};
                        if (kCorr) {
                            const int rj = cor_row(j >> 1), ro = cor_row((j >> 1) - 1 + 2 * (j & 1));
                            const int i0 = cor_col(p), i1 = cor_col(p + 1);
                            co[0] = Kk[rj + i0];
                            co[1] = Kk[rj + i1];
                            const float ce = Kk[rj + cor_col(h ? p + 2 : p - 1)];
                            cx[0] = h ? co[1] : ce;
                            cx[1] = h ? ce : co[0];
                            cy[0] = Kk[ro + i0];
                            cy[1] = Kk[ro + i1];
                            cz[0] = Ko[rj + i0];
                            cz[1] = Ko[rj + i1];
                        }
#pragma unroll
                        for (int e = 0; e < 2; e++) {
                            const int i = 2 * (p + e) + h;
                            float xw = xw2[e], xe = xe2[e], xs_ = vs[e], xn_ = vn[e], xd_ = vd[e], xu_ = vu[e];
                            if (kCorr) {
                                if (i > 0) xw = xw + (h ? co[e] : cx[e]);
                                if (i < g.nx - 1) xe = xe + (h ? cx[e] : co[e]);
                                if (j > 0) xs_ = xs_ + ((j & 1) ? co[e] : cy[e]);
                                if (j < g.ny - 1) xn_ = xn_ + ((j & 1) ? cy[e] : co[e]);
                                if (k > 0) xd_ = xd_ + ((k & 1) ? co[e] : cz[e]);
                                if (k < g.nz - 1) xu_ = xu_ + ((k & 1) ? cz[e] : co[e]);
                            }
                            float off = 0.f;
                            if (i > 0) off += bxl[e] * xw;
                            if (i < g.nx - 1) off += bxh[e] * xe;
                            if (j > 0) off += ys0[e] * xs_;
                            if (j < g.ny - 1) off += ys1[e] * xn_;
                            if (k > 0) off += zs0[e] * xd_;
                            if (k < g.nz - 1) off += zs1[e] * xu_;
                            v[e] = (bv[e] + off) * dv[e];
                        }
                    } else {
                        v[0] = (bb.x + 0.f) * dd.x;
                        v[1] = (bb.y + 0.f) * dd.y;
                    }
                    *reinterpret_cast<float2 *>(Rm + r1 * RB_XW + qx) = make_float2(v[0], v[1]);
                }
            }
            // the ring: item t = tid / 3 of every third thread, spread over all warps
            const int t = tid / 3;
            if (tid % 3 == 0 && t < 2 * (RB_HW + 1) + RB_TY) {
                int r1, p;
                const int w = t < RB_HW + 1 ? t : t - (RB_HW + 1);
                if (t < 2 * (RB_HW + 1)) {
                    r1 = t < RB_HW + 1 ? 0 : RB_CR - 1;
                    const int j = y0 - 1 + r1, h = (a.c0 + j + m) & 1;
                    p = (h ? p0 - 1 : p0) + w;
                } else {
                    r1 = t - 2 * (RB_HW + 1) + 1;
                    const int j = y0 - 1 + r1, h = (a.c0 + j + m) & 1;
                    p = h ? p0 - 1 : p0 + RB_HW;
                }
                const int j = y0 - 1 + r1, h = (a.c0 + j + m) & 1;
                if (j >= 0 && j < g.ny && p >= 0 && p < hx) cell(r1, j, h, p);
            }
        }
        __syncthreads();
        if (*flag) {
            // a load did not arrive in time: record it, let the loads in
            // flight land (bounded) and stop this block
            if (tid == 0) {
                atomicCAS(ctl + C_ERR, 0, E_TIMEOUT);
                for (int s = q; s < min(nstep, q + 2); s++)
                    mbar_wait_bounded(bar + s % RB_NBAR, (s / RB_NBAR) & 1, kRbDrainCycles);
            }
            return;
        }
        // second colour on plane mm = m - 1, and the plane's output
        const int mm = m - 1;
        if (q >= 2) {
            float dsum = 0.f;   // (a thread's 4 cells, then the warp: FP32; the 8 warps: FP64)
            if (own) {
                const float *Rc = R(mm), *Bm = Bv(mm);
                const int rc = r + 1, qx = pq - p0 + 4, h2 = (c1 + j2 + mm) & 1;
                float s2[2], s1[2];   // second colour (computed), first colour (from R)
                {
                    const float *Rl = R(mm - 1), *Rh = R(mm + 1), *Dm = Dv(mm);
                    const F *Fx = FX(mm), *Fy = FY(mm), *Fz0 = FZ(mm), *Fz1 = FZ(mm + 1);
                    const int k = mm, j = j2, hh = h2, qf = qx + 4;
                    const int ch = (rc * 2 + hh) * RB_XW + qx, cr = rc * RB_XW + qx;
                    // paired loads: own half (b, 1/diag), and the first colour's results:
                    // the y and z neighbours (rows rc -+ 1, planes mm -+ 1) and the x
                    // neighbours (row rc) -- each row's first-colour half
                    const float2 bb = *reinterpret_cast<const float2 *>(Bm + ch);
                    const float2 dd = *reinterpret_cast<const float2 *>(Dm + ch);
                    const float2 xs = *reinterpret_cast<const float2 *>(Rc + cr - RB_XW);
                    const float2 xn = *reinterpret_cast<const float2 *>(Rc + cr + RB_XW);
                    const float2 xd = *reinterpret_cast<const float2 *>(Rl + cr);
                    const float2 xu = *reinterpret_cast<const float2 *>(Rh + cr);
                    const float2 xo = *reinterpret_cast<const float2 *>(Rc + cr);
                    const float xb = hh ? Rc[cr + 2] : Rc[cr - 1];
                    const float xw2[2] = {hh ? xo.x : xb, hh ? xo.y : xo.x};
                    const float xe2[2] = {hh ? xo.y : xo.x, hh ? xb : xo.y};
                    const float2 fxl = ld2f(Fx + (rc * 2 + hh) * RB_FW + qf);
                    const float bxh[2] = {float(Fx[(rc * 2 + 1 - hh) * RB_FW + qf + hh]),
                                          float(Fx[(rc * 2 + 1 - hh) * RB_FW + qf + hh + 1])};
                    const float2 fy0 = ld2f(Fy + (rc * 2 + hh) * RB_FW + qf);
                    const float2 fy1 = ld2f(Fy + ((rc + 1) * 2 + hh) * RB_FW + qf);
                    const float2 fz0 = ld2f(Fz0 + (rc * 2 + hh) * RB_FW + qf);
                    const float2 fz1 = ld2f(Fz1 + (rc * 2 + hh) * RB_FW + qf);
                    const float bxl[2] = {fxl.x, fxl.y}, ys0[2] = {fy0.x, fy0.y}, ys1[2] = {fy1.x, fy1.y};
                    const float zs0[2] = {fz0.x, fz0.y}, zs1[2] = {fz1.x, fz1.y};
                    const float vs[2] = {xs.x, xs.y}, vn[2] = {xn.x, xn.y}, vd[2] = {xd.x, xd.y};
                    const float vu[2] = {xu.x, xu.y}, bv[2] = {bb.x, bb.y}, dv[2] = {dd.x, dd.y};
                    s1[0] = xo.x;
                    s1[1] = xo.y;
#pragma unroll
                    for (int e = 0; e < 2; e++) {
                        const int i = 2 * (pq + e) + hh;
                        float off = 0.f;
                        if (i > 0) off += bxl[e] * xw2[e];
                        if (i < g.nx - 1) off += bxh[e] * xe2[e];
                        if (j > 0) off += ys0[e] * vs[e];
                        if (j < g.ny - 1) off += ys1[e] * vn[e];
                        if (k > 0) off += zs0[e] * vd[e];
                        if (k < g.nz - 1) off += zs1[e] * vu[e];
                        s2[e] = (bv[e] + off) * dv[e];
                    }
                }
                float v[2][2];
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    v[0][e] = h2 ? s1[e] : s2[e];
                    v[1][e] = h2 ? s2[e] : s1[e];
                }
                float *o = xout + (size_t)(mm * g.ny + j2) * g.nx + pq;
                *reinterpret_cast<float2 *>(o) = make_float2(v[0][0], v[0][1]);
                *reinterpret_cast<float2 *>(o + hx) = make_float2(v[1][0], v[1][1]);
                if constexpr (kDot) {
                    float d = 0.f;
#pragma unroll
                    for (int h = 0; h < 2; h++)
#pragma unroll
                        for (int e = 0; e < 2; e++) d += Bm[(rc * 2 + h) * RB_XW + qx + e] * v[h][e];
                    dsum = d;
                }
            }
            if constexpr (kDot) {
                for (int o = 16; o > 0; o >>= 1) dsum += __shfl_down_sync(0xffffffffu, dsum, o);
                if ((tid & 31) == 0) wsum[tid >> 5] = (double)dsum;
            }
        }
        __syncthreads();
        // the plane's partial from the warp sums (FP64) in warp 1, so that
        // thread 0 issues the next loads at once
        if (kDot && q >= 2 && tid == 32) {
            double s = 0.0;
            for (int w = 0; w < RB_THREADS / 32; w++) s += wsum[w];
            a.part[cz.comp * kPartComp + (size_t)mm * (gridDim.x * gridDim.y) + blockIdx.y * gridDim.x + blockIdx.x] = s;
        }
        if (tid == 0 && q + 2 < nstep) {
            fence_proxy_async();
            rb_issue<F>(sm, bar, q + 2, m0, p0, y0, kZero, kCorr, tm, tc);
        }
    }
}

// The padded copy of the x-face coefficients that k_cc_rb_sweep loads: per
// row, the nx/2 + 1 even faces then, from position rb_hxp(nx), the nx/2 odd
// ones (zeros in the padding), converted as the V-cycle's copy is.
template <class F>
__global__ void k_xface_pad(GridD g, const float *__restrict__ bf, F *__restrict__ out)
{
    const int hxp = rb_hxp(g.nx), hf = g.nx / 2 + 1, hx = g.nx / 2;
    const long long n = 2LL * hxp * g.ny * g.nz;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const int pos = (int)(s % hxp);
        const long long rh = s / hxp;
        const int half = (int)(rh & 1);
        const long long row = rh >> 1;
        const long long rf = row * (g.nx + 1);
        float v = 0.f;
        if (half == 0 && pos < hf) v = bf[rf + pos];
        if (half == 1 && pos < hx) v = bf[rf + hf + pos];
        if constexpr (sizeof(F) == 2) out[s] = __float2bfloat16_rn(v);
        else out[s] = v;
    }
}

// The fused sweep's face type: the V-cycle's.
using RbF = typename VFace<float>::type;

// The second colour pass of a sweep (colour c1, plain) together with the
// (plane, tile) partials of b.x that k_cc_rb_sweep<kDot> forms: the same
// threads (positions pq, pq+1 of both halves of a tile row), cells, order
// and sums, so the colour passes end with the fused sweep's r.z bit for bit.
// Each c1 cell is formed by the operations of gs_cell; the other colour is
// read (unchanged by this pass) for the partial.  A block covers
// kGs2Planes planes of its tile (the loads of all of them in flight
// together), each plane's partial reduced on its own.  Grid (tiles x,
// tiles y, ceil(nz / kGs2Planes)).
constexpr int kGs2Planes = 4;
__global__ void __launch_bounds__(RB_THREADS) k_cc_gs2_dot(VOp3<float> A3, V3<float> xv, V3<const float> bv, int nzb,
                                                            const int *act, int c1, double *__restrict__ part)
{
    const CompZ cz(nzb);
    if (comp_off(act, cz.comp)) return;
    const VOp<float> A = A3.op(cz.comp);
    float *__restrict__ x = xv.p[cz.comp];
    const float *__restrict__ b = bv.p[cz.comp];
    part += cz.comp * kPartComp;
    __shared__ double wsum[kGs2Planes][RB_THREADS / 32];
    const GridD &g = A.g;
    const int tid = threadIdx.x, hx = g.nx >> 1, hf = (g.nx + 2) >> 1;
    const int r = tid >> 4;
    const int j = blockIdx.y * RB_TY + r, pq = blockIdx.x * RB_HW + 2 * (tid & 15);
    const int sy = g.nx, sz = g.nx * g.ny;
    float dsum[kGs2Planes];
#pragma unroll
    for (int pl = 0; pl < kGs2Planes; pl++) {
        const int k = cz.z * kGs2Planes + pl;
        dsum[pl] = 0.f;
        if (j >= g.ny || pq >= hx || k >= g.nz) continue;
        const int h2 = (c1 + j + k) & 1;
        const int rc = (k * g.ny + j) * g.nx;
        const int c = rc + (h2 ? hx : 0) + pq, o = rc + (h2 ? 0 : hx) + pq;
        const float2 bb = *reinterpret_cast<const float2 *>(b + c);
        const float2 bo = *reinterpret_cast<const float2 *>(b + o);
        const float2 di = *reinterpret_cast<const float2 *>(A.dinv + c);
        const float2 xo = *reinterpret_cast<const float2 *>(x + o);
        const float xb = h2 ? (pq + 2 < hx ? x[o + 2] : 0.f) : (pq > 0 ? x[o - 1] : 0.f);
        float2 xs = make_float2(0.f, 0.f), xn = xs, xd = xs, xu = xs;
        if (j > 0) xs = *reinterpret_cast<const float2 *>(x + c - sy);
        if (j < g.ny - 1) xn = *reinterpret_cast<const float2 *>(x + c + sy);
        if (k > 0) xd = *reinterpret_cast<const float2 *>(x + c - sz);
        if (k < g.nz - 1) xu = *reinterpret_cast<const float2 *>(x + c + sz);
        const float2 fy0 = ld2f(A.by + c + k * g.nx), fy1 = ld2f(A.by + c + k * g.nx + g.nx);
        const float2 fz0 = ld2f(A.bz + c), fz1 = ld2f(A.bz + c + sz);
        const float xw2[2] = {h2 ? xo.x : xb, h2 ? xo.y : xo.x};
        const float xe2[2] = {h2 ? xo.y : xo.x, h2 ? xb : xo.y};
        const float ys0[2] = {fy0.x, fy0.y}, ys1[2] = {fy1.x, fy1.y}, zs0[2] = {fz0.x, fz0.y}, zs1[2] = {fz1.x, fz1.y};
        const float vs[2] = {xs.x, xs.y}, vn[2] = {xn.x, xn.y}, vd[2] = {xd.x, xd.y}, vu[2] = {xu.x, xu.y};
        const float bv[2] = {bb.x, bb.y}, dv[2] = {di.x, di.y};
        const int rf = rc + k * g.ny + j;
        float s2[2];
#pragma unroll
        for (int e = 0; e < 2; e++) {
            const int t = pq + e, i = 2 * t + h2;
            const float bxl = float(A.bx[rf + (h2 ? hf + t : t)]);
            const float bxh = float(A.bx[rf + (h2 ? t + 1 : hf + t)]);
            float off = 0.f;
            if (i > 0) off += bxl * xw2[e];
            if (i < g.nx - 1) off += bxh * xe2[e];
            if (j > 0) off += ys0[e] * vs[e];
            if (j < g.ny - 1) off += ys1[e] * vn[e];
            if (k > 0) off += zs0[e] * vd[e];
            if (k < g.nz - 1) off += zs1[e] * vu[e];
            s2[e] = (bv[e] + off) * dv[e];
        }
        *reinterpret_cast<float2 *>(x + c) = make_float2(s2[0], s2[1]);
        // b.x over the 4 cells, half 0 then half 1, as k_cc_rb_sweep<kDot>
        const float b0[2] = {h2 ? bo.x : bb.x, h2 ? bo.y : bb.y}, b1[2] = {h2 ? bb.x : bo.x, h2 ? bb.y : bo.y};
        const float v0[2] = {h2 ? xo.x : s2[0], h2 ? xo.y : s2[1]}, v1[2] = {h2 ? s2[0] : xo.x, h2 ? s2[1] : xo.y};
        float d = 0.f;
        d += b0[0] * v0[0];
        d += b0[1] * v0[1];
        d += b1[0] * v1[0];
        d += b1[1] * v1[1];
        dsum[pl] = d;
    }
    // per warp in FP32, across the 8 warps in FP64 (as k_cc_rb_sweep<kDot>)
#pragma unroll
    for (int pl = 0; pl < kGs2Planes; pl++) {
        float v = dsum[pl];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) wsum[pl][tid >> 5] = (double)v;
    }
    __syncthreads();
    if (tid < kGs2Planes) {
        const int k = cz.z * kGs2Planes + tid;
        if (k < g.nz) {
            double s = 0.0;
            for (int w = 0; w < RB_THREADS / 32; w++) s += wsum[tid][w];
            part[(size_t)k * (gridDim.x * gridDim.y) + blockIdx.y * gridDim.x + blockIdx.x] = s;
        }
    }
}

// Residual of the 8 children of coarse cell (I,J,K), averaged.
template <class T>
__device__ inline T rr_cell(const VOp<T> &A, const T *__restrict__ x, const T *__restrict__ b, int I, int J,
                            int K)
{
    // child by child with the layout's index functions: with the children's
    // parities known after unrolling these fold to row offsets in few
    // registers (this kernel is latency-bound: occupancy counts more).
    // Only the 4 red children ((i+j+k) even) are summed: the restriction
    // follows pre-smoothing whose last pass updated every black cell from its
    // current neighbours, so a black cell's residual is 0 up to rounding.
    const GridD &g = A.g;
    T s = 0;
#pragma unroll
    for (int o = 0; o < 8; o++) {
        if (__popc(o) & 1) continue;   // black child
        const int i = 2 * I + (o & 1), j = 2 * J + ((o >> 1) & 1), k = 2 * K + ((o >> 2) & 1);
        const int c = cix<T>(g, i, j, k);
        const T bxl = T(A.bx[fidxT<T>(g, 0, i, j, k)]), bxh = T(A.bx[fidxT<T>(g, 0, i + 1, j, k)]);
        const T byl = T(A.by[fidxT<T>(g, 1, i, j, k)]), byh = T(A.by[fidxT<T>(g, 1, i, j + 1, k)]);
        const T bzl = T(A.bz[fidxT<T>(g, 2, i, j, k)]), bzh = T(A.bz[fidxT<T>(g, 2, i, j, k + 1)]);
        T off = sizeof(T) == 8 ? b[c] - A.diag[c] * x[c] : T(0);
        if (i > 0) off += bxl * x[cix<T>(g, i - 1, j, k)];
        if (i < g.nx - 1) off += bxh * x[cix<T>(g, i + 1, j, k)];
        if (j > 0) off += byl * x[c - g.nx];
        if (j < g.ny - 1) off += byh * x[c + g.nx];
        if (k > 0) off += bzl * x[c - g.nx * g.ny];
        if (k < g.nz - 1) off += bzh * x[c + g.nx * g.ny];
        s += sizeof(T) == 8 ? off : b[c] - (A.diag[c] * x[c] - off);
    }
    return s * T(0.125);
}

// Residual of the 8 children, averaged into the coarse right-hand side.
template <class T>
__global__ void __launch_bounds__(256) k_cc_resid_restrict(VOp3<T> A3, V3<const T> x, V3<const T> b, GridD gc,
                                                           V3<T> bc, int nzb, const int *act)
{
    const CompZ cz(nzb);
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = cz.z * blockDim.z + threadIdx.z;
    if (I >= gc.nx || J >= gc.ny || K >= gc.nz || comp_off(act, cz.comp)) return;
    bc.p[cz.comp][cix<T>(gc, I, J, K)] = rr_cell<T>(A3.op(cz.comp), x.p[cz.comp], b.p[cz.comp], I, J, K);
}

// k_cc_resid_restrict for FP32 levels with nx a multiple of 8: a thread
// forms coarse cells I0 .. I0+3 (I0 = 4t) of coarse row (J, K).  Their red
// children lie in one half of each of the 4 fine rows (2J+jj, 2K+kk) -- the
// half of parity (j + k) & 1 -- at the consecutive positions I0 .. I0+3, so
// x, b, the diagonal, the y and z neighbours and faces are 16-byte (8-byte
// BF16) vectors, as in k_cc_gs4.  Children and operations in the order of
// rr_cell (rows (2J,2K), (2J+1,2K), (2J,2K+1), (2J+1,2K+1)), so the results
// are the same bits; the coarse values go out as two 8-byte pairs (even and
// odd coarse cells are the two halves of the coarse row).  Bound by load
// latency: capped at 64 registers (from 75) for four blocks per SM, 16 %
// faster at 256^3.
__global__ void __launch_bounds__(256, 4) k_cc_rr4(VOp3<float> A3, V3<const float> xv, V3<const float> bv, GridD gc,
                                               V3<float> bcv, int nzb, const int *act)
{
    const CompZ cz(nzb);
    if (comp_off(act, cz.comp)) return;
    const VOp<float> A = A3.op(cz.comp);
    const float *__restrict__ x = xv.p[cz.comp], *__restrict__ b = bv.p[cz.comp];
    float *__restrict__ bc = bcv.p[cz.comp];
    const GridD &g = A.g;
    const int hx = g.nx >> 1, hf = (g.nx + 2) >> 1;
    const int I0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = cz.z * blockDim.z + threadIdx.z;
    if (I0 >= gc.nx || J >= gc.ny || K >= gc.nz) return;
    const int sy = g.nx, sz = g.nx * g.ny;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kk = 0; kk < 2; kk++)
#pragma unroll
        for (int jj = 0; jj < 2; jj++) {
            const int j = 2 * J + jj, k = 2 * K + kk, h = (j + k) & 1;
            const int rc = (k * g.ny + j) * g.nx;
            const int c = rc + (h ? hx : 0) + I0, o = rc + (h ? 0 : hx) + I0;
            float xc4[4], bb[4], dg[4], xo[4], xs[4], xn[4], xd[4], xu[4], fy0[4], fy1[4], fz0[4], fz1[4];
            load4(x + c, xc4);
            load4(b + c, bb);
            load4(A.diag + c, dg);
            load4(x + o, xo);
            const float xb = h ? (I0 + 4 < hx ? x[o + 4] : 0.f) : (I0 > 0 ? x[o - 1] : 0.f);
            if (j > 0) load4(x + c - sy, xs);
            if (j < g.ny - 1) load4(x + c + sy, xn);
            if (k > 0) load4(x + c - sz, xd);
            if (k < g.nz - 1) load4(x + c + sz, xu);
            load4(A.by + c + k * g.nx, fy0);
            load4(A.by + c + k * g.nx + g.nx, fy1);
            load4(A.bz + c, fz0);
            load4(A.bz + c + sz, fz1);
            const int rf = rc + k * g.ny + j;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int t = I0 + e, i = 2 * t + h;
                const float bxl = float(A.bx[rf + (h ? hf + t : t)]);
                const float bxh = float(A.bx[rf + (h ? t + 1 : hf + t)]);
                const float xw = h ? xo[e] : (e ? xo[e - 1] : xb);
                const float xe = h ? (e < 3 ? xo[e + 1] : xb) : xo[e];
                float off = 0.f;
                if (i > 0) off += bxl * xw;
                if (i < g.nx - 1) off += bxh * xe;
                if (j > 0) off += fy0[e] * xs[e];
                if (j < g.ny - 1) off += fy1[e] * xn[e];
                if (k > 0) off += fz0[e] * xd[e];
                if (k < g.nz - 1) off += fz1[e] * xu[e];
                acc[e] += bb[e] - (dg[e] * xc4[e] - off);
            }
        }
    const int hxc = gc.nx >> 1;
    float *row = bc + (K * gc.ny + J) * gc.nx;
    *reinterpret_cast<float2 *>(row + (I0 >> 1)) = make_float2(acc[0] * 0.125f, acc[2] * 0.125f);
    *reinterpret_cast<float2 *>(row + hxc + (I0 >> 1)) = make_float2(acc[1] * 0.125f, acc[3] * 0.125f);
}

// Rediscretised coarse operator: face coefficient = (sum of the 4 fine faces) / 16,
// extra = sum over uncovered children / 8 (identity where all children are covered).
template <class T>
__global__ void k_cc_coarsen(GridD gf, const T *__restrict__ ef, const T *__restrict__ bxf,
                             const T *__restrict__ byf, const T *__restrict__ bzf,
                             const uint8_t *__restrict__ covf, GridD gc, const uint8_t *__restrict__ covc,
                             T *__restrict__ ec, T *__restrict__ bxc, T *__restrict__ byc,
                             T *__restrict__ bzc)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = blockIdx.z * blockDim.z + threadIdx.z;
    if (I > gc.nx || J > gc.ny || K > gc.nz) return;
    if (I < gc.nx && J < gc.ny && K < gc.nz) {
        const int C = cix<T>(gc, I, J, K);
        if (covc[cidx(gc, I, J, K)]) {
            ec[C] = T(1);
        } else {
            T s = 0;
            for (int o = 0; o < 8; o++) {
                const int i = 2 * I + (o & 1), j = 2 * J + ((o >> 1) & 1), k = 2 * K + ((o >> 2) & 1);
                if (!covf[cidx(gf, i, j, k)]) s += ef[cix<T>(gf, i, j, k)];
            }
            ec[C] = s * T(0.125);
        }
    }
    const T *bf[3] = {bxf, byf, bzf};
    T *bcs[3] = {bxc, byc, bzc};
    const int m[3] = {gc.nx, gc.ny, gc.nz};
    for (int d = 0; d < 3; d++) {
        int id[3] = {I, J, K};
        bool ok = true;
        for (int e = 0; e < 3; e++) ok &= (e == d) ? id[e] <= m[e] : id[e] < m[e];
        if (!ok) continue;
        int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
        T s = 0;
        for (int q1 = 0; q1 < 2; q1++)
            for (int q2 = 0; q2 < 2; q2++) {
                int f[3] = {2 * I, 2 * J, 2 * K};
                f[t1] += q1;
                f[t2] += q2;
                s += bf[d][fidxT<T>(gf, d, f[0], f[1], f[2])];
            }
        bcs[d][fidxT<T>(gc, d, I, J, K)] = s * T(0.0625);
    }
}

// diag = extra + the six face coefficients of the cell, for each of nvar
// variants of the operator: a face on box side s counts for variant q only if
// bit s of side mask q (bits 6q .. 6q+5 of masks) is set.  Sums in the same
// order for every variant, so a variant with all bits set is the plain sum.
// kRound: the faces as the V-cycle stores them (rounded to BF16), so that its
// operator keeps diag = extra + sum of its own faces.
template <class T, bool kRound = false>
__global__ void k_cc_make_diag(GridD g, const T *__restrict__ extra, const T *__restrict__ bx,
                               const T *__restrict__ by, const T *__restrict__ bz, int nvar, unsigned masks,
                               T *__restrict__ d0, T *__restrict__ d1, T *__restrict__ d2,
                               T *__restrict__ i0 = nullptr, T *__restrict__ i1 = nullptr,
                               T *__restrict__ i2 = nullptr)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i >= g.nx || j >= g.ny || k >= g.nz) return;
    const int c = cix<T>(g, i, j, k);
    const T e = extra[c];
    T f[6] = {bx[fidxT<T>(g, 0, i, j, k)], bx[fidxT<T>(g, 0, i + 1, j, k)],
              by[fidxT<T>(g, 1, i, j, k)], by[fidxT<T>(g, 1, i, j + 1, k)],
              bz[fidxT<T>(g, 2, i, j, k)], bz[fidxT<T>(g, 2, i, j, k + 1)]};
    if constexpr (kRound) {
#pragma unroll
        for (int t = 0; t < 6; t++) f[t] = __bfloat162float(__float2bfloat16_rn(f[t]));
    }
    // box side of each face, -1 for a face between two cells
    const int sd[6] = {i == 0 ? 0 : -1, i == g.nx - 1 ? 1 : -1, j == 0 ? 2 : -1,
                       j == g.ny - 1 ? 3 : -1, k == 0 ? 4 : -1, k == g.nz - 1 ? 5 : -1};
    T *out[3] = {d0, d1, d2};
    T *inv[3] = {i0, i1, i2};
    // away from the box sides the variants agree: one sum (and one quotient)
    const bool side = i == 0 || i == g.nx - 1 || j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1;
    T s = e, si = T(0);
    for (int q = 0; q < nvar; q++) {
        if (q == 0 || side) {
            const unsigned m = masks >> (6 * q);
            s = e;
#pragma unroll
            for (int t = 0; t < 6; t++) s += (sd[t] < 0 || ((m >> sd[t]) & 1u)) ? f[t] : T(0);
            if (inv[q]) si = s > T(0) ? T(1) / s : T(0);
        }
        out[q][c] = s;
        if (inv[q]) inv[q][c] = si;
    }
}

__global__ void k_cov_coarsen(GridD gf, const uint8_t *covf, GridD gc, uint8_t *covc)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = blockIdx.z * blockDim.z + threadIdx.z;
    if (I >= gc.nx || J >= gc.ny || K >= gc.nz) return;
    int all = 1;
    for (int o = 0; o < 8; o++)
        all &= covf[cidx(gf, 2 * I + (o & 1), 2 * J + ((o >> 1) & 1), 2 * K + ((o >> 2) & 1))];
    covc[cidx(gc, I, J, K)] = (uint8_t)all;
}

__global__ void k_cov_from_flag(int n, const uint8_t *flag, uint8_t *cov)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        cov[s] = flag[s] == 0;
}

template <class S, class D>
__global__ void k_convert(const S *__restrict__ a, D *__restrict__ b, int n)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        b[s] = (D)a[s];
}

// FP64 natural-order array of cells (d < 0) or of faces of normal d -> FP32
// row-split copy, a thread per element by row (found from a flat index by two
// divisions it took 80 us at 256^3; 68 us here, 12 bytes a cell).
__global__ void __launch_bounds__(256) k_to_split(GridD g, int d, const double *__restrict__ a, float *__restrict__ b,
                           const double *__restrict__ sig = nullptr)
{
    const int mx = g.nx + (d == 0), my = g.ny + (d == 1), mz = g.nz + (d == 2);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i >= mx || j >= my || k >= mz) return;
    const double sc = sig ? *sig : 1.0;
    b[d < 0 ? cix<float>(g, i, j, k) : fidxT<float>(g, d, i, j, k)] = f64_to_f32_pow2(a[(k * my + j) * mx + i], sc);
}
inline dim3 split_grid(const GridD &g, int d)
{
    return grid3(g.nx + (d == 0), g.ny + (d == 1), g.nz + (d == 2));
}

// r = sig * a in FP32 (the refinement solver's first residual, natural order)
__global__ void k_to32_scaled(const double *__restrict__ a, float *__restrict__ b, int n,
                              const double *__restrict__ sig)
{
    const double sc = *sig;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        b[s] = f64_to_f32_pow2(a[s], sc);
}

// FP32 face coefficients -> the V-cycle's BF16 copy (same layout)
__global__ void k_to_bf16(const float *__restrict__ a, __nv_bfloat16 *__restrict__ b, int n)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        b[s] = __float2bfloat16_rn(a[s]);
}


// Level-0 coefficients of the cell-centred projection: beta = a_f / h^2,
// 2 a_f / h^2 on outflow faces (phi = 0 there), 0 on other box faces.
__global__ void k_mac_coeffs(GridD g, const uint8_t *__restrict__ flag, const double *__restrict__ ax,
                             const double *__restrict__ ay, const double *__restrict__ az,
                             double *__restrict__ extra, double *__restrict__ bx, double *__restrict__ by,
                             double *__restrict__ bz)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i > g.nx || j > g.ny || k > g.nz) return;
    const double h2 = g.h * g.h;
    if (i < g.nx && j < g.ny && k < g.nz) {
        int c = cidx(g, i, j, k);
        extra[c] = flag[c] ? 0.0 : 1.0;
    }
    const double *A[3] = {ax, ay, az};
    double *B[3] = {bx, by, bz};
    int id[3] = {i, j, k};
#pragma unroll
    for (int d = 0; d < 3; d++) {
        bool ok = true;
#pragma unroll
        for (int e = 0; e < 3; e++) ok &= (e == d) ? id[e] <= dimn(g, e) : id[e] < dimn(g, e);
        if (!ok) continue;
        int f = fidx(g, d, i, j, k);
        if (id[d] == 0 || id[d] == dimn(g, d)) {
            int side = 2 * d + (id[d] != 0);
            B[d][f] = (g.bc[side] == EBV_OUTFLOW || pin_face(g, d, i, j, k)) ? 2.0 * A[d][f] / h2 : 0.0;
        } else {
            B[d][f] = A[d][f] / h2;
        }
    }
}

// Level-0 coefficients of the viscous solves (Eq. implicit-viscous,
// alpha-weighted), shared by the three velocity components:
//   extra = rho alpha + dt eta A_EB / (h^2 delta), delta = max(-n.b, delta_min)
//   beta  = dt a_f eta_f / h^2, eta_f the mean of the two cells; on a box face
//           2 dt a_f eta / h^2, the coefficient of a Dirichlet condition there.
// A box face enters the diagonal of component q only where the side is a
// Dirichlet side for q (k_cc_make_diag's side masks); its value enters the
// right-hand side (k_visc_rhs).
__global__ void __launch_bounds__(256) k_visc_coeffs(GridD g, GeomD geo, ParamsD p, const double *__restrict__ eta,
                              const double *__restrict__ dtp, double *__restrict__ extra,
                              double *__restrict__ bx, double *__restrict__ by, double *__restrict__ bz)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i > g.nx || j > g.ny || k > g.nz) return;
    const double h2 = g.h * g.h, dt = dtp[DT_DT];
    const double dth2 = dtp[DT_DTH2];  // dt / h^2
    const int N3 = geo.ncell;
    const double *A[3] = {geo.ax, geo.ay, geo.az};
    double *B[3] = {bx, by, bz};
    int id[3] = {i, j, k};
#pragma unroll
    for (int d = 0; d < 3; d++) {
        bool ok = true;
#pragma unroll
        for (int e = 0; e < 3; e++) ok &= (e == d) ? id[e] <= dimn(g, e) : id[e] < dimn(g, e);
        if (!ok) continue;
        int f = fidx(g, d, i, j, k);
        double a = A[d][f];
        if (id[d] == 0 || id[d] == dimn(g, d)) {
            int cc[3] = {i, j, k};
            cc[d] -= id[d] != 0;
            B[d][f] = __double2hiint(a) > 0 ? 2.0 * dth2 * a * eta[cidx(g, cc[0], cc[1], cc[2])] : 0.0;
        } else {
            int lo[3] = {i, j, k};
            lo[d] -= 1;
            // dt/h^2 a eta_f, the mean's 1/2 taken with dt (exact); a > 0 on the integer pipe
            const double es = eta[cidx(g, lo[0], lo[1], lo[2])] + eta[cidx(g, i, j, k)];
            B[d][f] = __double2hiint(a) > 0 ? (0.5 * dth2) * a * es : 0.0;
        }
    }
    if (i >= g.nx || j >= g.ny || k >= g.nz) return;
    const int c = cidx(g, i, j, k);
    if (geo.flag[c] == 0) {
        extra[c] = 1.0;
        return;
    }
    double e = p.rho * geo.alpha[c];
    if (geo.flag[c] == 2 && geo.area[c] > 0.0) {
        double nb = 0.0;
        for (int q = 0; q < 3; q++) nb += geo.nrm[q * N3 + c] * geo.bcen[q * N3 + c];
        double del = -nb > p.delta_min ? -nb : p.delta_min;
        e += dt * eta[c] * geo.area[c] / (h2 * del);
    }
    extra[c] = e;
}

// Right-hand sides of the three viscous solves: alpha psi plus, for each box
// face of the cell on a Dirichlet side of the component, its coefficient
// (k_visc_coeffs) times the boundary value; faces are read at the box sides only.
__global__ void k_visc_rhs(GridD g, GeomD geo, const double *__restrict__ psi, const double *__restrict__ bx,
                           const double *__restrict__ by, const double *__restrict__ bz, double *__restrict__ b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i >= g.nx || j >= g.ny || k >= g.nz) return;
    const int c = cidx(g, i, j, k), N3 = geo.ncell;
    if (geo.flag[c] == 0) {
        for (int q = 0; q < 3; q++) b[q * N3 + c] = 0.0;
        return;
    }
    const bool side = i == 0 || i == g.nx - 1 || j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1;
    const double al = geo.alpha[c];
    const double *B[3] = {bx, by, bz};
    const int id[3] = {i, j, k};
#pragma unroll
    for (int q = 0; q < 3; q++) {
        double rb = 0.0, val;
        if (side)
            for (int d = 0; d < 3; d++)
                for (int hs = 0; hs < 2; hs++) {
                    if (id[d] != (hs ? dimn(g, d) - 1 : 0)) continue;
                    int fi[3] = {i, j, k};
                    fi[d] += hs;
                    if (side_dirichlet(g, 2 * d + hs, q, &val)) rb += B[d][fidx(g, d, fi[0], fi[1], fi[2])] * val;
                }
        b[q * N3 + c] = al * psi[q * N3 + c] + rb;
    }
}

// q = A p (level 0) and block partials of p.q in FP64 (per thread and warp
// in T, see block_sum3_t).  Each thread handles planes 2kk and 2kk+1 of
// column (i, j).  With kRes (FP64) instead the residual r = b - A p, stored
// as an FP32 row-split vector, with block partials of |r|^2 (the refinement
// solver's true residual in one pass; |r|^2 only decides convergence, so it
// is summed from the stored FP32 values, per thread and warp in FP32).
template <class T, bool kRes = false>
__global__ void __launch_bounds__(256) k_cc_apply_dot(CcOp3<T> A3, V3<const T> pv, V3<T> qv, double *__restrict__ part,
                                                      int nzb, const int *act, V3<const T> bv = V3<const T>(),
                                                      V3<float> rv = V3<float>(), const double *__restrict__ sig = nullptr)
{
    const CompZ cz(nzb);
    if (comp_off(act, cz.comp)) return;
    const CcOp<T> A = A3.op(cz.comp);
    const T *__restrict__ p = pv.p[cz.comp], *__restrict__ b = bv.p[cz.comp];
    T *__restrict__ q = qv.p[cz.comp];
    float *__restrict__ r32 = rv.p[cz.comp];
    const double sc = (kRes && sig) ? sig[cz.comp * kScalLen] : 1.0;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int kk = cz.z * blockDim.z + threadIdx.z;
    T v = 0;
    float vr = 0.0f;
    if (i < A.g.nx && j < A.g.ny) {
        T y[2], pc[2];
        int cc[2] = {-1, -1};
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int k = 2 * kk + h;
            if (k >= A.g.nz) continue;
            T diag, off;
            cc[h] = cix<T>(A.g, i, j, k);
            pc[h] = p[cc[h]];
            if constexpr (kRes) {
                cc_row(A, i, j, k, p, diag, y[h], b[cc[h]] - A.diag[cc[h]] * pc[h]);
            } else {
                cc_row(A, i, j, k, p, diag, off);
                y[h] = diag * pc[h] - off;
            }
        }
#pragma unroll
        for (int h = 0; h < 2; h++)
            if (cc[h] >= 0) {
                if constexpr (kRes) {
                    const float r = f64_to_f32_pow2(y[h], sc);
                    r32[cix<float>(A.g, i, j, 2 * kk + h)] = r;
                    vr += r * r;
                } else {
                    q[cc[h]] = y[h];
                    v += pc[h] * y[h];
                }
            }
    }
    const double vs = kRes ? block_sum3_t<float>(vr) : block_sum3_t<T>(v);
    if (thread_linear() == 0) part[cz.comp * kPartComp + cz.linear()] = vs;
}

// k_cc_apply_dot<float> for levels with nx a multiple of 8: a thread forms
// q = A p at 4 consecutive cells of one half-row (half h = tx / nq) in each of
// two planes, with 16-byte loads as in k_cc_gs4 (the x faces, rows of nx + 1,
// as scalars), and adds p.q of its 8 cells to its block's partial (block_sum8).
// Each q is formed as in cc_row; the partial sums are grouped by this kernel's
// fixed block shape (kApply4X x Y x Z).  (A cap of 48 registers, for five blocks per SM,
// measures no faster than 64 registers and four blocks.)
constexpr int kApply4X = 16, kApply4Y = 8, kApply4Z = 2;
// The vectorised apply and restriction serve grids where they launch at least
// this many blocks (two per SM of 152); smaller grids keep one cell per thread.
constexpr long long kVecMinBlocks = 304;
__global__ void __launch_bounds__(256) k_cc_apply4(CcOp3<float> A3, V3<const float> pv, V3<float> qv,
                                                  double *__restrict__ part, int nzb, const int *act)
{
    const CompZ cz(nzb);
    if (comp_off(act, cz.comp)) return;
    const CcOp<float> A = A3.op(cz.comp);
    const float *__restrict__ p = pv.p[cz.comp];
    float *__restrict__ q = qv.p[cz.comp];
    const GridD &g = A.g;
    const int hx = g.nx >> 1, hf = (g.nx + 2) >> 1, nq = hx >> 2;
    const int tx = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int kk = cz.z * blockDim.z + threadIdx.z;
    const int sy = g.nx, sz = g.nx * g.ny;
    float v[4] = {0.f, 0.f, 0.f, 0.f};   // per position: two terms, as a thread of k_cc_apply_dot
    if (tx < 2 * nq && j < g.ny) {
        const int h = tx / nq, t0 = 4 * (tx - h * nq);
#pragma unroll
        for (int hp = 0; hp < 2; hp++) {
            const int k = 2 * kk + hp;
            if (k >= g.nz) continue;
            const int rc = (k * g.ny + j) * g.nx;
            const int c = rc + (h ? hx : 0) + t0, o = rc + (h ? 0 : hx) + t0;
            float pc[4], dg[4], xo[4], xs[4], xn[4], xd[4], xu[4], fy0[4], fy1[4], fz0[4], fz1[4], y[4];
            load4(p + c, pc);
            load4(A.diag + c, dg);
            load4(p + o, xo);
            const float xb = h ? (t0 + 4 < hx ? p[o + 4] : 0.f) : (t0 > 0 ? p[o - 1] : 0.f);
            if (j > 0) load4(p + c - sy, xs);
            if (j < g.ny - 1) load4(p + c + sy, xn);
            if (k > 0) load4(p + c - sz, xd);
            if (k < g.nz - 1) load4(p + c + sz, xu);
            load4(A.by + c + k * g.nx, fy0);
            load4(A.by + c + k * g.nx + g.nx, fy1);
            load4(A.bz + c, fz0);
            load4(A.bz + c + sz, fz1);
            const int rf = rc + k * g.ny + j;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int t = t0 + e, i = 2 * t + h;
                const float bxl = A.bx[rf + (h ? hf + t : t)];
                const float bxh = A.bx[rf + (h ? t + 1 : hf + t)];
                const float xw = h ? xo[e] : (e ? xo[e - 1] : xb);
                const float xe = h ? (e < 3 ? xo[e + 1] : xb) : xo[e];
                float off = 0.f;
                if (i > 0) off += bxl * xw;
                if (i < g.nx - 1) off += bxh * xe;
                if (j > 0) off += fy0[e] * xs[e];
                if (j < g.ny - 1) off += fy1[e] * xn[e];
                if (k > 0) off += fz0[e] * xd[e];
                if (k < g.nz - 1) off += fz1[e] * xu[e];
                y[e] = dg[e] * pc[e] - off;
                v[e] += pc[e] * y[e];
            }
            *reinterpret_cast<float4 *>(q + c) = make_float4(y[0], y[1], y[2], y[3]);
        }
    }
    const double vs = block_sum8((v[0] + v[1]) + (v[2] + v[3]));
    if (thread_linear() == 0) part[cz.comp * kPartComp + cz.linear()] = vs;
}
inline dim3 apply4_grid(const GridD &g)
{
    const int nq2 = 2 * ((g.nx >> 1) >> 2), nzh = (g.nz + 1) / 2;
    return dim3((nq2 + kApply4X - 1) / kApply4X, (g.ny + kApply4Y - 1) / kApply4Y, (nzh + kApply4Z - 1) / kApply4Z);
}

// ===========================================================================
// Nodal operator (alpha-weighted trilinear stiffness, unit coefficient):
//   (A x)_a = h sum_{cells c at a} alpha_c sum_{nodes b of c, active} K(a,b) x_b
// with K(a,b) = 1/3, 0, -1/12, -1/12 for corners differing in 0, 1, 2, 3
// coordinates.
// ===========================================================================

// node kinds: inactive, active with all 8 cells full (so interior), other active
enum { ND_OFF = 0, ND_REG = 1, ND_IRR = 2 };
__constant__ double kQ1[4] = {1.0 / 3.0, 0.0, -1.0 / 12.0, -1.0 / 12.0};

template <class T>
struct NdOp {
    GridD g;               // cell dims
    T h;                   // g.h in the operator's precision
    const T *alpha;        // cells
    const uint8_t *act;    // nodes
    const uint8_t *kind;   // per node: ND_OFF, ND_REG (all 8 cells full) or ND_IRR
};

// Row of the nodal operator at node (i,j,k), assembled in stencil form.  With
// a[r][q][p] the volume fraction of the cell (i-1+p, j-1+q, k-1+r) (0 outside
// the box), the element matrix gives: centre (1/3) sum a; axis neighbours 0;
// each face-diagonal neighbour -(sum of the two cells sharing that edge)/12;
// each body-diagonal neighbour -(the one cell between them)/12.  Inactive
// neighbours hold x = 0 in every vector the solvers pass here.
// Sums of the 12 face-diagonal (fd) and 8 body-diagonal (bd) neighbours of
// interior node n.
template <class T>
__device__ inline void nd_regular_sums(const GridD &g, const T *__restrict__ x, int n, T &fd, T &bd)
{
    const T *xc = x + n;
    const int sy = g.nx + 1, sz = (g.nx + 1) * (g.ny + 1);
    fd = xc[1 + sy] + xc[-1 + sy] + xc[1 - sy] + xc[-1 - sy] + xc[1 + sz] + xc[-1 + sz] + xc[1 - sz] +
         xc[-1 - sz] + xc[sy + sz] + xc[-sy + sz] + xc[sy - sz] + xc[-sy - sz];
    bd = xc[1 + sy + sz] + xc[-1 + sy + sz] + xc[1 - sy + sz] + xc[-1 - sy + sz] + xc[1 + sy - sz] +
         xc[-1 + sy - sz] + xc[1 - sy - sz] + xc[-1 - sy - sz];
}

template <class T>
__device__ inline void nd_row(const NdOp<T> &A, int i, int j, int k, const T *__restrict__ x, T &diag,
                              T &ax)
{
    const GridD &g = A.g;
    const int NXn = g.nx + 1, NYn = g.ny + 1;
    if (A.kind[nidx(g, i, j, k)] == ND_REG) {
        // all 8 cells full (so the node is interior): the constant stencil
        // 8/3 at the centre, -1/6 on the 12 face diagonals, -1/12 on the 8
        // body diagonals (times h)
        T fd, bd;
        nd_regular_sums(g, x, nidx(g, i, j, k), fd, bd);
        const T hh = A.h;
        diag = hh * T(8.0 / 3.0);
        ax = diag * x[nidx(g, i, j, k)] - hh * T(1.0 / 12.0) * (T(2) * fd + bd);
        return;
    }
    T a[2][2][2];
    T sa = 0;
#pragma unroll
    for (int r = 0; r < 2; r++)
#pragma unroll
        for (int q = 0; q < 2; q++)
#pragma unroll
            for (int p = 0; p < 2; p++) {
                int ci = i - 1 + p, cj = j - 1 + q, ck = k - 1 + r;
                T v = inbox(g, ci, cj, ck) ? A.alpha[cidx(g, ci, cj, ck)] : T(0);
                a[r][q][p] = v;
                sa += v;
            }
    const int n0 = nidx(g, i, j, k);
    auto X = [&](int di, int dj, int dk) -> T {
        int ii = i + di, jj = j + dj, kk = k + dk;
        if ((unsigned)ii > (unsigned)g.nx || (unsigned)jj > (unsigned)g.ny || (unsigned)kk > (unsigned)g.nz)
            return T(0);
        return x[n0 + di + dj * NXn + dk * NXn * NYn];
    };
    T s = 0;
    // face diagonals in the xy, xz and yz planes
#pragma unroll
    for (int q = 0; q < 2; q++)
#pragma unroll
        for (int p = 0; p < 2; p++) {
            s += (a[0][q][p] + a[1][q][p]) * X(2 * p - 1, 2 * q - 1, 0);
            s += (a[q][0][p] + a[q][1][p]) * X(2 * p - 1, 0, 2 * q - 1);
            s += (a[q][p][0] + a[q][p][1]) * X(0, 2 * p - 1, 2 * q - 1);
        }
    // body diagonals
#pragma unroll
    for (int r = 0; r < 2; r++)
#pragma unroll
        for (int q = 0; q < 2; q++)
#pragma unroll
            for (int p = 0; p < 2; p++) s += a[r][q][p] * X(2 * p - 1, 2 * q - 1, 2 * r - 1);
    const T hh = A.h;
    diag = hh * sa * T(1.0 / 3.0);
    ax = diag * x[n0] - hh * T(1.0 / 12.0) * s;
}

// One Chebyshev step: r = b - A x_in; d = cd d + cr D^-1 r; x_out = x_in + d.
// Node by node, on the levels that do not take the plane march.
template <class T>
__global__ void __launch_bounds__(256) k_nd_cheb(NdOp<T> A, const T *__restrict__ xin, T *__restrict__ xout,
                                                 T *__restrict__ dvec, const T *__restrict__ b, T cd, T cr)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    const GridD &g = A.g;
    if (i > g.nx || j > g.ny || k > g.nz) return;
    const int n = nidx(g, i, j, k);
    // the node's own operands are loaded before any branch on them
    const uint8_t on = A.act[n];
    const T bn = b[n], xn = xin[n], dold = dvec[n];
    if (!on) {
        xout[n] = T(0);
        dvec[n] = T(0);
        return;
    }
    T diag, ax;
    nd_row(A, i, j, k, xin, diag, ax);
    T r = bn - ax;
    T dn = (cd != T(0) ? cd * dold : T(0)) + cr * r / diag;
    dvec[n] = dn;
    xout[n] = xn + dn;
}

// The first step from x = 0, d = 0: x = d = cr D^-1 b, a constant times b on
// regular nodes; only the others sum their cells' fractions.  Streams 16 bytes
// per thread and array (arrays from cudaMalloc), then the tail (FP32 256^3: as
// part of k_nd_cheb 130 us, eight fractions and a division per node; 55 us so).
template <class T>
__global__ void __launch_bounds__(128) k_nd_cheb0(NdOp<T> A, T *__restrict__ x, T *__restrict__ d, const T *__restrict__ b,
                                                  T cr, T crd, int nn)
{
    const GridD &g = A.g;   // (crd = cr / regular diagonal)
    auto other = [&](int n, T bn) -> T {   // an active node that is not regular
        const int NX = g.nx + 1, NY = g.ny + 1, i = n % NX, j = (n / NX) % NY, k = n / (NX * NY);
        T a[8];
#pragma unroll
        for (int oc = 0; oc < 8; oc++) {
            const int ci = i - 1 + (oc & 1), cj = j - 1 + ((oc >> 1) & 1), ck = k - 1 + ((oc >> 2) & 1);
            a[oc] = inbox(g, ci, cj, ck) ? A.alpha[cidx(g, ci, cj, ck)] : T(0);
        }
        const T dsum = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
        return cr * bn / (A.h * dsum * T(1.0 / 3.0));
    };
    constexpr int W = 16 / sizeof(T);
    const int nv = nn / W, t0 = blockIdx.x * blockDim.x + threadIdx.x, st = gridDim.x * blockDim.x;
    for (int s = t0; s < nv; s += st) {
        T v[W];
        uint8_t kd[W];
        if constexpr (W == 4) {
            const float4 q = reinterpret_cast<const float4 *>(b)[s];
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
            const uchar4 c = reinterpret_cast<const uchar4 *>(A.kind)[s];
            kd[0] = c.x; kd[1] = c.y; kd[2] = c.z; kd[3] = c.w;
        } else {
            const double2 q = reinterpret_cast<const double2 *>(b)[s];
            v[0] = q.x; v[1] = q.y;
            const uchar2 c = reinterpret_cast<const uchar2 *>(A.kind)[s];
            kd[0] = c.x; kd[1] = c.y;
        }
#pragma unroll
        for (int u = 0; u < W; u++)
            v[u] = kd[u] == ND_REG ? crd * v[u] : (kd[u] == ND_OFF ? T(0) : other(W * s + u, v[u]));
        if constexpr (W == 4) {
            const float4 q = make_float4(v[0], v[1], v[2], v[3]);
            reinterpret_cast<float4 *>(x)[s] = q;
            reinterpret_cast<float4 *>(d)[s] = q;
        } else {
            const double2 q = make_double2(v[0], v[1]);
            reinterpret_cast<double2 *>(x)[s] = q;
            reinterpret_cast<double2 *>(d)[s] = q;
        }
    }
    for (int n = W * nv + t0; n < nn; n += st) {
        const T v = A.kind[n] == ND_REG ? crd * b[n] : (A.kind[n] == ND_OFF ? T(0) : other(n, b[n]));
        x[n] = v;
        d[n] = v;
    }
}

// ---- nodal passes in plane-sum form (levels with node kinds) ------------------------
// On a regular node the row is 8/3 x - (2 fd + bd) / 12 with fd, bd the sums of
// the 12 face- and 8 body-diagonal neighbours.  Per plane let A = the four axis
// neighbours within the plane, B = its four diagonals and C = 2 A + B; then
//   2 fd + bd = 2 B_k + C_{k-1} + C_{k+1}.
// A block of NT_X x NT_Y threads owns as many node columns and marches kz
// planes: each plane of x (with its one-node halo) is staged in shared memory
// while the next plane's loads are in flight (two buffers: the one written at
// plane kk was last read at plane kk - 2, before every thread passed plane
// kk - 1's barrier), B and C stay in registers, and the node operands are
// fetched one plane ahead.  Interior nodes only (1 .. n-1: with the box faces
// the tiles of a 2^q grid would be almost empty in their last row and column);
// the box faces and the interior nodes that are active but not regular (cut
// cells) are listed once per geometry and take the general row nd_row in the
// first blocks of the same launch, so no warp of the march diverges into it.
// kz is the largest of 16, 8, 4, 2 that still gives four blocks per SM.  (A
// form without shared memory -- a warp per 32 columns x 4 rows, x neighbours by
// shuffle -- was as fast on small grids and half as fast on 256^3: 169 us for
// 89, its loads per plane bound by their latency at 16 warps per SM.)  Modes:
//   ND_CHEB   one Chebyshev step, as k_nd_cheb (out = x_out, d updated);
//   ND_RESID  out = b - A x, as k_nd_resid;
//   ND_APPLY  out = A x (x on inactive nodes) with block partials of x.out;
//   ND_RES32  r = b - A x (b - x on inactive nodes) in T, stored to the FP32
//             vector out32, with block partials of |r|^2 (the refinement
//             solver's true residual; T = double).
// The sums are associated differently from the one-node kernels.  Measured per
// Chebyshev step, against 16 planes per block at every size, box faces
// included, and the listed nodes in a launch of their own: FP64 32^3 25.3 + 6.2
// -> 6.1 us, 128^3 106 + 14.4 -> 86.7 us (FP64-pipe bound: 14 operations per
// node, of 17), its 64^3 level (one node per thread before) 18.7 -> 10 us; FP32
// 64^3 8.0 + 2.9 -> 4.2 us, 256^3 89 + 10.4 -> 89.7 us (HBM).
enum { ND_CHEB = 0, ND_RESID = 1, ND_APPLY = 2, ND_RES32 = 3 };
constexpr int NT_X = 32, NT_Y = 8, NT_T = NT_X * NT_Y;
constexpr int NT_W = NT_X + 2, NT_H = NT_Y + 2, NT_N = NT_W * NT_H;
constexpr int NT_SLOTS = (NT_N + NT_T - 1) / NT_T;
constexpr int kKindNodes = 4096;   // coarse levels with at least this many nodes take the march too

// Launch of a pass: blocks of listed nodes first, then of tiles.
struct NdShape {
    int ntx, nty, kz, nlb, blocks;
};
inline NdShape nd_shape(const GridD &g, int nlist)
{
    NdShape s;
    const int mz = g.nz - 1;   // interior nodes along z
    s.ntx = (g.nx - 1 + NT_X - 1) / NT_X;
    s.nty = (g.ny - 1 + NT_Y - 1) / NT_Y;
    s.kz = 16;
    while (s.kz > 2 && (long long)s.ntx * s.nty * ((mz + s.kz - 1) / s.kz) < 4 * 152) s.kz /= 2;
    s.nlb = (nlist + NT_T - 1) / NT_T;
    s.blocks = s.nlb + s.ntx * s.nty * ((mz + s.kz - 1) / s.kz);
    return s;
}

// Constants of a pass on regular nodes, formed on the host (a division per
// thread cost as much as the node's row where a block marches few planes):
// diagonal, h / 12, and of the Chebyshev step cd, cr, cr / diagonal and that
// times the other two.
template <class T>
struct NdCoef {
    T cd, cr, dreg, h12, crd, c0, c1;
};
template <class T>
inline NdCoef<T> nd_coef(T h, T cd, T cr)
{
    NdCoef<T> k;
    k.cd = cd;
    k.cr = cr;
    k.dreg = h * T(8.0 / 3.0);
    k.h12 = h * T(1.0 / 12.0);
    k.crd = cr / k.dreg;
    k.c0 = k.crd * k.dreg;
    k.c1 = k.crd * k.h12;
    return k;
}

template <class T, int kMode>
__global__ void __launch_bounds__(NT_T) k_nd_pass(NdOp<T> A, NdShape sh, const int *__restrict__ list, int nlist,
                                                          const T *__restrict__ xin, T *__restrict__ out,
                                                          T *__restrict__ dvec, const T *__restrict__ b, NdCoef<T> ck,
                                                          double *__restrict__ part, float *__restrict__ out32,
                                                          const double *__restrict__ sig)
{
    const T cd = ck.cd, cr = ck.cr;
    const double sc = (kMode == ND_RES32 && sig) ? *sig : 1.0;
    const GridD &g = A.g;
    const int NX = g.nx + 1, NY = g.ny + 1, tid = threadIdx.x;
    T v = 0;          // ND_APPLY: this thread's part of x.out; ND_RES32: of |r|^2 on the listed nodes
    float vr = 0.0f;  // ND_RES32: its part of |r|^2 in the march, from the stored FP32 values too
    const bool listed = (int)blockIdx.x < sh.nlb;
    if (listed) {
        const int t = blockIdx.x * NT_T + tid;
        if (t < nlist) {
            const int n = list[t];
            const int i = n % NX, j = (n / NX) % NY, k = n / (NX * NY);
            const bool on = A.act[n] != 0;
            const T x0 = xin[n], bn = kMode != ND_APPLY ? b[n] : T(0);
            T diag = T(1), ax = x0;
            if (on) nd_row(A, i, j, k, xin, diag, ax);
            if (kMode == ND_CHEB) {
                const T dn = on ? (cd != T(0) ? cd * dvec[n] : T(0)) + cr * (bn - ax) / diag : T(0);
                dvec[n] = dn;
                out[n] = on ? x0 + dn : T(0);
            }
            if (kMode == ND_RESID) out[n] = on ? bn - ax : T(0);
            if (kMode == ND_APPLY) { out[n] = ax; v = x0 * ax; }
            if (kMode == ND_RES32) {
                const float r = f64_to_f32_pow2(bn - ax, sc);
                out32[n] = r;
                v = T(r) * T(r);
            }
        }
    } else {
        __shared__ T sx[2][NT_H][NT_W];
        const int tile = (int)blockIdx.x - sh.nlb, bx = tile % sh.ntx, tq = tile / sh.ntx, by = tq % sh.nty, bz = tq / sh.nty;
        const int sy = NX, sz = NX * NY, tx = tid & 31, ty = tid >> 5;
        const int i0 = 1 + bx * NT_X, j0 = 1 + by * NT_Y, k0 = 1 + bz * sh.kz;
        const int i = i0 + tx, j = j0 + ty;
        const bool col = i < g.nx && j < g.ny;
        const int kend = min(k0 + sh.kz, g.nz);   // nodes k0 .. kend-1; planes k0-1 .. kend
        // halo-tile slots of this thread: offset within a plane, -1 outside the box
        int soff[NT_SLOTS];
#pragma unroll
        for (int u = 0; u < NT_SLOTS; u++) {
            const int sl = tid + u * NT_T;
            const int rr = sl / NT_W, qq = sl - rr * NT_W;
            const int gi = i0 - 1 + qq, gj = j0 - 1 + rr;
            soff[u] = (sl < NT_N && gi < NX && gj < NY) ? gj * sy + gi : -1;
        }
        T pre[NT_SLOTS];
        auto fetch = [&](int kk) {
#pragma unroll
            for (int u = 0; u < NT_SLOTS; u++) pre[u] = soff[u] >= 0 ? xin[kk * sz + soff[u]] : T(0);
        };
        const T dreg = ck.dreg, h12 = ck.h12, crd = ck.crd, c0 = ck.c0, c1 = ck.c1;
        T Cm = 0, C0 = 0, B0 = 0, X0 = 0, b_c = 0, d_c = 0, b_n = 0, d_n = 0;
        int kd_c = -1, kd_n = -1;   // node kind, -1: no node of this block
        fetch(k0 - 1);
        for (int kk = k0 - 1; kk <= kend; kk++) {
            T(*S)[NT_W] = sx[kk & 1];
#pragma unroll
            for (int u = 0; u < NT_SLOTS; u++) {
                const int sl = tid + u * NT_T;
                if (sl < NT_N) (&S[0][0])[sl] = pre[u];
            }
            if (kk < kend) fetch(kk + 1);
            // operands of node kk, finalised at the next plane
            kd_n = -1;
            if (col && kk >= k0 && kk < kend) {
                const int n = kk * sz + j * sy + i;
                kd_n = A.kind[n];
                if (kMode != ND_APPLY) b_n = b[n];
                if (kMode == ND_CHEB) d_n = dvec[n];
            }
            __syncthreads();
            const T xc = S[ty + 1][tx + 1];
            const T An = (S[ty + 1][tx] + S[ty + 1][tx + 2]) + (S[ty][tx + 1] + S[ty + 2][tx + 1]);
            const T Bn = (S[ty][tx] + S[ty][tx + 2]) + (S[ty + 2][tx] + S[ty + 2][tx + 2]);
            const T Cn = T(2) * An + Bn;
            const int n = (kk - 1) * sz + j * sy + i;
            if (kd_c == ND_OFF) {
                if (kMode == ND_CHEB) { out[n] = T(0); dvec[n] = T(0); }
                if (kMode == ND_RESID) out[n] = T(0);
                if (kMode == ND_APPLY) { out[n] = X0; v += X0 * X0; }
                if (kMode == ND_RES32) {
                    const float r = f64_to_f32_pow2(b_c - X0, sc);
                    out32[n] = r;
                    vr += r * r;
                }
            } else if (kd_c == ND_REG) {
                const T t = T(2) * B0 + (Cm + Cn);   // 2 fd + bd
                if (kMode == ND_CHEB) {
                    const T dn = (cd != T(0) ? cd * d_c : T(0)) + crd * b_c - c0 * X0 + c1 * t;
                    dvec[n] = dn;
                    out[n] = X0 + dn;
                } else {
                    // (a residual as two multiply-adds on b)
                    if (kMode == ND_RESID) out[n] = (b_c - dreg * X0) + h12 * t;
                    if (kMode == ND_APPLY) {
                        const T ax = dreg * X0 - h12 * t;
                        out[n] = ax;
                        v += X0 * ax;
                    }
                    if (kMode == ND_RES32) {
                        const float r = f64_to_f32_pow2((b_c - dreg * X0) + h12 * t, sc);
                        out32[n] = r;
                        vr += r * r;
                    }
                }
            }
            Cm = C0; C0 = Cn; B0 = Bn; X0 = xc;
            kd_c = kd_n; b_c = b_n; d_c = d_n;
        }
    }
    if constexpr (kMode == ND_APPLY || kMode == ND_RES32) {
        const double vs = kMode == ND_RES32 && !listed ? block_sum3_t<float>(vr) : block_sum3_t<T>(v);
        if (tid == 0) part[blockIdx.x] = vs;
    }
}

template <class T>
__global__ void __launch_bounds__(256) k_nd_resid(NdOp<T> A, const T *__restrict__ x, const T *__restrict__ b,
                                                  T *__restrict__ r)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    const GridD &g = A.g;
    if (i > g.nx || j > g.ny || k > g.nz) return;
    const int n = nidx(g, i, j, k);
    if (!A.act[n]) { r[n] = T(0); return; }
    T diag, ax;
    nd_row(A, i, j, k, x, diag, ax);
    r[n] = b[n] - ax;
}

// Full weighting (transpose of trilinear prolongation), line by line and plane
// by plane (27 guarded and weighted terms one by one before: 13.5 -> 8.4 us on
// average over the launched levels of 256^3).
template <class T>
__global__ void k_nd_restrict(GridD gf, const T *__restrict__ rf, GridD gc, const uint8_t *__restrict__ actc,
                              T *__restrict__ bc)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = blockIdx.z * blockDim.z + threadIdx.z;
    if (I > gc.nx || J > gc.ny || K > gc.nz) return;
    const int N = nidx(gc, I, J, K);
    const int sy = gf.nx + 1, sz = (gf.nx + 1) * (gf.ny + 1);
    const T *q = rf + nidx(gf, 2 * I, 2 * J, 2 * K);
    const int im = I > 0 ? -1 : 0, ip = 2 * I < gf.nx ? 1 : 0, jm = J > 0 ? -sy : 0, jp = 2 * J < gf.ny ? sy : 0;
    const int km = K > 0 ? -sz : 0, kp = 2 * K < gf.nz ? sz : 0;
    const T hf = T(0.5);
    T s;
    if constexpr (sizeof(T) == 8) {   // fewest operations (guarded reads: 9.1 us on 128^3, 12.5 with the weights)
        auto line = [&](const T *p) { return p[0] + hf * ((im ? p[im] : T(0)) + (ip ? p[ip] : T(0))); };
        auto plane = [&](const T *p) { return line(p) + hf * ((jm ? line(p + jm) : T(0)) + (jp ? line(p + jp) : T(0))); };
        s = plane(q) + hf * ((km ? plane(q + km) : T(0)) + (kp ? plane(q + kp) : T(0)));
    } else {                          // unguarded reads, weight 0 outside (8.4 us on 256^3, 12.4 guarded)
        const T um = im ? hf : T(0), up = ip ? hf : T(0), vm = jm ? hf : T(0), vp = jp ? hf : T(0);
        const T wm = km ? hf : T(0), wp = kp ? hf : T(0);
        auto line = [&](const T *p) { return p[0] + (um * p[im] + up * p[ip]); };
        auto plane = [&](const T *p) { return line(p) + (vm * line(p + jm) + vp * line(p + jp)); };
        s = plane(q) + (wm * plane(q + km) + wp * plane(q + kp));
    }
    bc[N] = actc[N] ? s : T(0);
}

// xout = xin + trilinear interpolation of the coarse correction (active nodes).
// A thread forms nodes (i, j, 2K) and (i, j, 2K + 1) from the coarse planes K and
// K + 1; along x the two coarse neighbours are the same one at even i, so the
// lanes of a row run the same instructions (a branch per term and one node per
// thread before: 27.4 -> 14.0 us on average over the levels of 256^3).
template <class T>
__global__ void k_nd_prolong(GridD gf, const uint8_t *__restrict__ actf, GridD gc, const T *__restrict__ xc,
                             const T *__restrict__ xin, T *__restrict__ xout)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = blockIdx.z * blockDim.z + threadIdx.z;
    if (i > gf.nx || j > gf.ny || K > gc.nz) return;
    const int n0 = nidx(gf, i, j, 2 * K), sz = (gf.nx + 1) * (gf.ny + 1);
    const int cy = gc.nx + 1, cz = (gc.nx + 1) * (gc.ny + 1);
    const bool up = K < gc.nz;   // (node plane 2K + 1 exists)
    const uint8_t on0 = actf[n0], on1 = up ? actf[n0 + sz] : 0;
    const T x0 = xin[n0], x1 = up ? xin[n0 + sz] : T(0);
    const T *c = xc + nidx(gc, i >> 1, j >> 1, K);
    const int pi = i & 1, pj = j & 1;
    // four times the interpolation within a coarse plane
    auto plane = [&](const T *q) {
        T s = q[0] + q[pi];
        if (pj) s += q[cy] + q[cy + pi];
        return pj ? s : T(2) * s;
    };
    const T s0 = plane(c), s1 = up ? plane(c + cz) : T(0);
    xout[n0] = on0 ? x0 + T(0.25) * s0 : T(0);
    if (up) xout[n0 + sz] = on1 ? x1 + T(0.125) * (s0 + s1) : T(0);
}
inline dim3 prolong_grid(const GridD &gf, const GridD &gc) { return grid3(gf.nx + 1, gf.ny + 1, gc.nz + 1); }

__global__ void k_nd_alpha_coarsen(GridD gf, const double *__restrict__ af, GridD gc, double *__restrict__ ac)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = blockIdx.z * blockDim.z + threadIdx.z;
    if (I >= gc.nx || J >= gc.ny || K >= gc.nz) return;
    double s = 0.0;
    for (int o = 0; o < 8; o++)
        s += af[cidx(gf, 2 * I + (o & 1), 2 * J + ((o >> 1) & 1), 2 * K + ((o >> 2) & 1))];
    ac[cidx(gc, I, J, K)] = 0.125 * s;
}

__global__ void k_nd_kind(GridD g, const double *__restrict__ alpha, const uint8_t *__restrict__ act,
                          uint8_t *__restrict__ kind)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i > g.nx || j > g.ny || k > g.nz) return;
    bool all = true;
    for (int oc = 0; oc < 8; oc++) {
        int ci = i - 1 + (oc & 1), cj = j - 1 + ((oc >> 1) & 1), ck = k - 1 + ((oc >> 2) & 1);
        if (!inbox(g, ci, cj, ck) || alpha[cidx(g, ci, cj, ck)] != 1.0) all = false;
    }
    const int n = nidx(g, i, j, k);
    kind[n] = !act[n] ? ND_OFF : (all ? ND_REG : ND_IRR);
}

__global__ void k_nd_active(GridD g, const double *__restrict__ alpha, uint8_t *__restrict__ act)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i > g.nx || j > g.ny || k > g.nz) return;
    int id[3] = {i, j, k};
    bool dir = pin_node(g, i, j, k);
    for (int d = 0; d < 3; d++) {
        if (id[d] == 0 && g.bc[2 * d] == EBV_OUTFLOW) dir = true;
        if (id[d] == dimn(g, d) && g.bc[2 * d + 1] == EBV_OUTFLOW) dir = true;
    }
    bool any = false;
    for (int oc = 0; oc < 8; oc++) {
        int ci = i - 1 + (oc & 1), cj = j - 1 + ((oc >> 1) & 1), ck = k - 1 + ((oc >> 2) & 1);
        if (inbox(g, ci, cj, ck) && alpha[cidx(g, ci, cj, ck)] > 0.0) any = true;
    }
    act[nidx(g, i, j, k)] = (!dir && any) ? 1 : 0;
}

// ===========================================================================
// Dense bottom solve
// ===========================================================================

// Edge of the padded bottom matrix: nb rounded up to whole pivot blocks, the
// rows past nb those of the identity.
constexpr int kGjB = 16;
__host__ __device__ inline int gj_pad(int nb) { return (nb + kGjB - 1) / kGjB * kGjB; }
// doubles of scratch per matrix: two copies and two pivot-block inverses
inline size_t gj_scratch(int nb) { return 2 * (size_t)gj_pad(nb) * gj_pad(nb) + 2 * kGjB * kGjB; }

// Bottom matrices of the variants of one operator (blockIdx.y; they differ in
// the diagonal), one block per row: np x np, natural numbering.
template <class T>
struct BottomDiag {
    const T *d[3];
};
template <class T>
__global__ void __launch_bounds__(128) k_cc_bottom_assemble(VOp<T> A, BottomDiag<T> D, double *__restrict__ M, int nb,
                                                            size_t mstride)
{
    const GridD &g = A.g;
    const int r = blockIdx.x, np = gridDim.x;
    double *row = M + blockIdx.y * mstride + (size_t)r * np;
    for (int s = threadIdx.x; s < np; s += blockDim.x) row[s] = (s == r) ? 1.0 : 0.0;
    __syncthreads();
    if (threadIdx.x || r >= nb) return;
    int i = r % g.nx, j = (r / g.nx) % g.ny, k = r / (g.nx * g.ny);
    double bxl = (double)T(A.bx[fidxT<T>(g, 0, i, j, k)]), bxh = (double)T(A.bx[fidxT<T>(g, 0, i + 1, j, k)]);
    double byl = (double)T(A.by[fidxT<T>(g, 1, i, j, k)]), byh = (double)T(A.by[fidxT<T>(g, 1, i, j + 1, k)]);
    double bzl = (double)T(A.bz[fidxT<T>(g, 2, i, j, k)]), bzh = (double)T(A.bz[fidxT<T>(g, 2, i, j, k + 1)]);
    double diag = (double)D.d[blockIdx.y][cix<T>(g, i, j, k)];
    row[r] = diag > 0.0 ? diag : 1.0;
    if (i > 0) row[r - 1] = -bxl;
    if (i < g.nx - 1) row[r + 1] = -bxh;
    if (j > 0) row[r - g.nx] = -byl;
    if (j < g.ny - 1) row[r + g.nx] = -byh;
    if (k > 0) row[r - g.nx * g.ny] = -bzl;
    if (k < g.nz - 1) row[r + g.nx * g.ny] = -bzh;
}

__global__ void __launch_bounds__(128) k_nd_bottom_assemble(GridD g, const double *__restrict__ alpha,
                                                            const uint8_t *__restrict__ act, double *__restrict__ M,
                                                            int nb)
{
    const int r = blockIdx.x, np = gridDim.x;
    double *row = M + (size_t)r * np;
    for (int s = threadIdx.x; s < np; s += blockDim.x) row[s] = 0.0;
    __syncthreads();
    if (threadIdx.x) return;
    if (r >= nb || !act[r]) { row[r] = 1.0; return; }
    int i = r % (g.nx + 1), j = (r / (g.nx + 1)) % (g.ny + 1), k = r / ((g.nx + 1) * (g.ny + 1));
    for (int oc = 0; oc < 8; oc++) {
        int ci = i - 1 + (oc & 1), cj = j - 1 + ((oc >> 1) & 1), ck = k - 1 + ((oc >> 2) & 1);
        if (!inbox(g, ci, cj, ck)) continue;
        double al = alpha[cidx(g, ci, cj, ck)];
        if (!(al > 0.0)) continue;
        int oa = (i - ci) | ((j - cj) << 1) | ((k - ck) << 2);
        for (int ob = 0; ob < 8; ob++) {
            int n = nidx(g, ci + (ob & 1), cj + ((ob >> 1) & 1), ck + ((ob >> 2) & 1));
            if (!act[n]) continue;
            row[n] += g.h * al * kQ1[__popc(oa ^ ob)];
        }
    }
}

// Inverse of an SPD matrix in place by Gauss-Jordan elimination with pivot
// blocks of kGjB rows (no pivoting needed), for up to three matrices of one
// size at once.  With P = A_KK^-1, one step replaces
//   A_KK by P, A_Kj by P A_Kj, A_iK by -A_iK P, A_ij by A_ij - A_iK P A_Kj.
// One launch per step over tiles of TE x TE entries, from one copy of the
// matrix into the other; the tile that forms the next step's diagonal block
// also inverts it, and the last step writes the unpadded inverse.  The work
// is nb^3 FP64 multiply-adds and one SM does two per cycle: one block per
// matrix on the augmented [A | I] (the form before) took 0.23 ms for 64
// unknowns, 0.84 ms for 105 and 6.0 ms for 210; over the tiles 50, 90 and 247 us
// (about 10 us a step, two thirds of it the next block's inverse).  Tiles of 32
// where 16 x 16 ones would make more than two waves (each tile forms
// A_iK P itself, a third of the work at 32 and half of it at 16).
struct GjArgs {
    const double *src[3];
    double *dst[3];
    double *piv[3];      // two kGjB x kGjB inverses each: this step's and the next one's
    int np, ldo, nout;   // padded size; leading dimension and size of the output
    int K;               // pivot block
};

// a (kGjB x kGjB, shared) := its inverse; 256 threads, one entry each.
__device__ inline void gj_invert_block(double (*a)[kGjB + 1], double *sc)
{
    const int r = threadIdx.x / kGjB, c = threadIdx.x % kGjB;
    for (int k = 0; k < kGjB; k++) {
        __syncthreads();
        if (threadIdx.x == 0) *sc = 1.0 / a[k][k];
        __syncthreads();
        const double p = *sc, f = a[r][k], q = a[k][c], v = a[r][c];
        __syncthreads();
        if (r == k) a[r][c] = (c == k) ? p : q * p;
        else a[r][c] = (c == k) ? -f * p : v - f * (q * p);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256) k_gj_first(GjArgs a)
{
    __shared__ double d[kGjB][kGjB + 1];
    __shared__ double sc;
    const int r = threadIdx.x / kGjB, c = threadIdx.x % kGjB, q = blockIdx.x;
    d[r][c] = a.src[q][(size_t)r * a.np + c];
    gj_invert_block(d, &sc);
    a.piv[q][threadIdx.x] = d[r][c];
}

template <int TE>
__global__ void __launch_bounds__(256) k_gj_step(GjArgs a)
{
    constexpr int B = kGjB, NE = TE * TE / 256;
    __shared__ double sl[TE][B + 1], sr[B][TE + 1], sp[B][B + 1], sc[TE][B + 1];
    __shared__ double inv;
    const int q = blockIdx.z, np = a.np, K0 = a.K * B;
    const int I0 = blockIdx.y * TE, J0 = blockIdx.x * TE, tid = threadIdx.x;
    const double *A = a.src[q];
    for (int e = tid; e < TE * B; e += 256) {
        const int r = e / B, c = e % B;
        sl[r][c] = I0 + r < np ? A[(size_t)(I0 + r) * np + K0 + c] : 0.0;
        const int r2 = e / TE, c2 = e % TE;
        sr[r2][c2] = J0 + c2 < np ? A[(size_t)(K0 + r2) * np + J0 + c2] : 0.0;
    }
    const double *P = a.piv[q] + (a.K & 1) * B * B;
    sp[tid / B][tid % B] = P[tid];
    __syncthreads();
    // the row factors: A_iK P, and -P for the pivot rows themselves
    for (int e = tid; e < TE * B; e += 256) {
        const int r = e / B, c = e % B, pr = I0 + r - K0;
        double v = 0.0;
        if (pr >= 0 && pr < B) {
            v = -sp[pr][c];
        } else {
#pragma unroll
            for (int k = 0; k < B; k++) v += sl[r][k] * sp[k][c];
        }
        sc[r][c] = v;
    }
    __syncthreads();
    const int N1 = K0 + B;   // first row of the next pivot block
    double out[NE];
#pragma unroll
    for (int u = 0; u < NE; u++) {
        const int e = tid + 256 * u, r = e / TE, c = e % TE, i = I0 + r, j = J0 + c;
        const bool pr = i >= K0 && i < K0 + B, pc = j >= K0 && j < K0 + B;
        double v;
        if (pc) {
            v = -sc[r][j - K0];
        } else {
            v = (pr || i >= np || j >= np) ? 0.0 : A[(size_t)i * np + j];
#pragma unroll
            for (int k = 0; k < B; k++) v -= sc[r][k] * sr[k][c];
        }
        out[u] = v;
        if (i < a.nout && j < a.nout) a.dst[q][(size_t)i * a.ldo + j] = v;
    }
    // the next step's diagonal block and its inverse
    if (N1 < np && N1 >= I0 && N1 < I0 + TE && N1 >= J0 && N1 < J0 + TE) {
#pragma unroll
        for (int u = 0; u < NE; u++) {
            const int e = tid + 256 * u, r = I0 + e / TE - N1, c = J0 + e % TE - N1;
            if (r >= 0 && r < B && c >= 0 && c < B) sp[r][c] = out[u];
        }
        gj_invert_block(sp, &inv);
        a.piv[q][((a.K + 1) & 1) * B * B + tid] = sp[tid / B][tid % B];
    }
}

// inv_q := the inverse of matrix q (assembled in M + q gj_scratch(nb)).
void bottom_invert(Ctx *c, double *M, int nb, int nmat, double *const *inv)
{
    const int np = gj_pad(nb), ns = np / kGjB;
    GjArgs a;
    a.np = np;
    for (int q = 0; q < 3; q++) {
        double *m = M + (size_t)std::min(q, nmat - 1) * gj_scratch(nb);
        a.src[q] = m;
        a.dst[q] = nullptr;
        a.piv[q] = m + 2 * (size_t)np * np;
    }
    EBV_LAUNCH(c, k_gj_first, dim3(nmat), dim3(256), 0, a);
    const bool big = (long long)ns * ns * nmat > 2 * 152;
    for (int K = 0; K < ns; K++) {
        const bool last = K + 1 == ns;
        a.K = K;
        a.ldo = last ? nb : np;
        a.nout = last ? nb : np;
        for (int q = 0; q < nmat; q++) {
            double *m = M + (size_t)q * gj_scratch(nb);
            a.src[q] = m + (size_t)(K & 1) * np * np;
            a.dst[q] = last ? inv[q] : m + (size_t)((K + 1) & 1) * np * np;
        }
        if (big) EBV_LAUNCH(c, k_gj_step<32>, dim3((np + 31) / 32, (np + 31) / 32, nmat), dim3(256), 0, a);
        else EBV_LAUNCH(c, k_gj_step<16>, dim3(ns, ns, nmat), dim3(256), 0, a);
    }
}

// x = inv b; the dense system is numbered in the natural order, the
// vectors of a row-split (FP32 cell-centred) level are mapped through g.
__device__ inline int bottom_pos(const GridD &g, int split, int r)
{
    if (!split) return r;
    return cix<float>(g, r % g.nx, (r / g.nx) % g.ny, r / (g.nx * g.ny));
}
// One warp per row, eight rows per block: a row's products are FP64-pipe work
// and a serial chain for one thread (125 unknowns: 13-25 us for one block with
// a thread per row, 2-4 us so).
template <class T>
__global__ void __launch_bounds__(256) k_bottom_solve(V3<const double> inv, int nb, V3<const T> b, V3<T> x, GridD g,
                                                      int split)
{
    const int c = blockIdx.y, r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= nb) return;
    const double *row = inv.p[c] + (size_t)r * nb;
    double s = 0.0;
    for (int q = lane; q < nb; q += 32) s += row[q] * (double)b.p[c][bottom_pos(g, split, q)];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) x.p[c][bottom_pos(g, split, r)] = (T)s;
}

// ---- the coarse end of the cell-centred V-cycle in one cluster -------------------
// Levels that cannot fill the GPU cost more in launch latency than in work.
// One cluster of kCvCtas blocks runs the V-cycle from such a level down to the
// bottom and back.  Its top one or two levels (nd) are cut into slabs of
// planes, one per block; the next smoothed level, at most 512 cells, is
// smoothed by every block for itself (a cluster barrier per pass would cost
// more than the pass); the bottom system is multiplied by its inverse.  Every
// array lives in shared memory: per cell one record (six face coefficients,
// masked at the box sides, and the inverse diagonal: 16 bytes with BF16
// faces, one load), right-hand side and x, and per x-pair its position and
// that of its parent, so a pass does no index arithmetic.  x is row-split with
// one halo plane on either side of the slab, which the blocks write for each
// other (distributed shared memory) before the hardware cluster barrier that
// ends the pass.  Per cell the operations and their order are those of gs_cell
// and rr_cell (a box side's coefficient is 0 here, which adds an exact 0); the
// coarse correction is added to the cells of the colour that the first pass
// reads, the sums a prolongation kernel would store.  The passes are small
// loops on purpose: unrolled over slots held in registers they ran as fast
// when cached, but their instructions came from DRAM at every launch on large
// grids (72 us instead of 37 at 128^3).
//
// Measured per V-cycle: levels up to 32^3 in FP32 28 us at 64^3 and 29 us at
// 128^3, against 36 and 40 us for one 1024-thread block that took the levels up
// to 16^3 and recomputed every index, plus 24 us for the launches on the 32^3
// level (about 6 us are loading, 1.1 us a pass over a 4,096-cell slab, 0.5 us
// one over 512 cells with its cluster barrier).  FP64, levels up to 16^3: 26 us
// against 63 (one SM's FP64 pipe bound it).  nd = 2 stays FP32: FP64 records
// of a 4,096-cell slab do not fit in shared memory.  512 threads: 1,024 measured
// 5 % slower.
constexpr int kCvCtas = 8, kCvThreads = 512, kCvMax = 4;
constexpr int kCoarseCells = 4096;    // largest top level with nd = 1
constexpr int kCvTopCells = 32768;    // with nd = 2 (FP32)
constexpr int kCvSmem = 225 * 1024;
template <class T> struct CvLoad { static constexpr int n = sizeof(T) == 4 ? 2 : 1; };   // x-pairs whose operands a thread loads together
struct CvLayout {
    int x[3], rec[3], b[3], dg[3], info[3], cpos[3], res, bs, bi, xb, ps, total;
};
template <class T>
struct CoarseVC {
    int n;                    // levels handled; the last is the bottom
    int nd;                   // of these, cut into slabs
    int split_z;              // slabs of z planes, else of y planes
    int na;                   // blocks that own a slab (ranks 0 .. na-1)
    VOp3<T> A3[kCvMax];
    V3<T> x;                  // top level
    V3<const T> b;
    V3<const double> binv;    // bottom inverses (natural numbering)
    int nb;
    double *part;             // block partials of b.x, or null
    CvLayout L;               // shared-memory offsets (cv_layout)
};
// planes along the split direction, and rows in the other one
__host__ __device__ inline int cv_np(const GridD &g, int split_z) { return split_z ? g.nz : g.ny; }
__host__ __device__ inline int cv_no(const GridD &g, int split_z) { return split_z ? g.ny : g.nz; }
// first plane of rank r's slab on level l (slabs nest: a coarse plane's two
// fine planes belong to the same block)
__host__ __device__ inline int cv_s0(int np_nd, int na, int nd, int l, int r) { return (np_nd * r / na) << (nd - l); }
// planes of the largest slab on level l
__host__ __device__ inline int cv_plmax(int np_nd, int na, int nd, int l) { return ((np_nd + na - 1) / na) << (nd - l); }

// One cell's coefficients in shared memory: faces x-, x+, y-, y+, z-, z+ (0 at
// the box sides) and the inverse diagonal.
template <class F, class T>
struct CvRec {
    T f[6], di, pad;
    __device__ void set(const F *g, T d)
    {
        for (int q = 0; q < 6; q++) f[q] = T(g[q]);
        di = d;
    }
    __device__ void get(T *g, T &d) const
    {
        for (int q = 0; q < 6; q++) g[q] = f[q];
        d = di;
    }
    __device__ void get_di(T &d) const { d = di; }
};
template <>
struct __align__(16) CvRec<__nv_bfloat16, float> {
    uint4 v;
    __device__ void set(const __nv_bfloat16 *g, float d)
    {
        auto two = [&](int q) {
            return (unsigned)__bfloat16_as_ushort(g[q]) | ((unsigned)__bfloat16_as_ushort(g[q + 1]) << 16);
        };
        v = make_uint4(two(0), two(2), two(4), __float_as_uint(d));
    }
    __device__ void get(float *g, float &d) const
    {
        const uint4 w = v;
        const unsigned u[3] = {w.x, w.y, w.z};
#pragma unroll
        for (int q = 0; q < 3; q++) {   // a BF16 is the high half of the FP32 of the same value
            g[2 * q] = __uint_as_float(u[q] << 16);
            g[2 * q + 1] = __uint_as_float(u[q] & 0xffff0000u);
        }
        d = __uint_as_float(w.w);
    }
    __device__ void get_di(float &d) const { d = __uint_as_float(v.w); }
};

// One level in shared memory: offsets in bytes (the same in every block) and
// shape.  info per x-pair: position of its even cell, then the flags kCvPar
// ((j+k) odd), kCvLo / kCvHi (on the slab's first / last plane); cpos: the
// position of its parent one level down.
constexpr int kCvParBit = 28, kCvPar = 1 << kCvParBit, kCvLo = 1 << 29, kCvHi = 1 << 30, kCvPos = kCvPar - 1;
struct CvLevel {
    int x, rec, b, dg, info, cpos;
    int nx, h, no, plane, sy, sz, s0, pl, pairs, cap;
    int lo_rank, hi_rank, dlo, dhi;   // where the slab's end planes go too (-1: nowhere), and the position shift
};
constexpr int kCvBiMax = 32 * 1024;   // the block's rows of the bottom inverse are staged up to this size
template <class T>
inline CvLayout cv_layout(const CoarseVC<T> &D)
{
    using Rec = CvRec<typename VFace<T>::type, T>;
    CvLayout o;
    int at = 0;
    auto take = [&](int bytes) { const int q = at; at += (bytes + 15) & ~15; return q; };
    const int npd = cv_np(D.A3[D.nd].A.g, D.split_z);
    for (int l = 0; l + 1 < D.n; l++) {
        const GridD &g = D.A3[l].A.g;
        const int plane = cv_no(g, D.split_z) * g.nx, pl = l < D.nd ? cv_plmax(npd, D.na, D.nd, l) : npd;
        o.x[l] = take((pl + 2) * plane * (int)sizeof(T));
        o.rec[l] = take(pl * plane * (int)sizeof(Rec));
        o.b[l] = take(pl * plane * (int)sizeof(T));
        o.dg[l] = take(pl * plane / 2 * (int)sizeof(T));
        o.info[l] = take(pl * plane / 2 * 4);
        o.cpos[l] = take(pl * plane / 2 * 4);
        if (l == 0) o.res = take(pl * plane * (int)sizeof(T));
    }
    o.bs = take(D.nb * 8);
    const int rows = (D.nb + D.na - 1) / D.na;
    o.bi = rows * D.nb * 8 <= kCvBiMax ? take(rows * D.nb * 8) : -1;
    o.xb = take(D.nb * (int)sizeof(T));
    o.ps = take(kCvThreads / 32 * 8);
    o.total = at;
    return o;
}

// One block's view while it works on a level.
template <class T>
struct CvView {
    using Rec = CvRec<typename VFace<T>::type, T>;
    T *x;
    const Rec *rec;      // [colour][pair]
    const T *b;          // [colour][pair]
    const int *info, *cpos;
    T *lo, *hi;   // the neighbouring blocks' x, shifted to this block's positions, or null
    int h, sy, sz, pairs, cap;   // cap: slots per colour
    // sum of face times neighbour of the cell at p whose x- neighbour is at w
    // (its x+ neighbour is the next word of the other half-row)
    // (FP64: added to init, as gs_cell's chain)
    __device__ T off(const Rec &r, int p, int w, T &di, T init) const
    {
        T f[6];
        r.get(f, di);
        const T xw = x[w], xe = x[w + 1], xs = x[p - sy], xn = x[p + sy], xd = x[p - sz], xu = x[p + sz];
        T s = sizeof(T) == 8 ? init + f[0] * xw : f[0] * xw;
        s += f[1] * xe;
        s += f[2] * xs;
        s += f[3] * xn;
        s += f[4] * xd;
        s += f[5] * xu;
        return s;
    }
    __device__ void put(int p, T v, int in) const
    {
        x[p] = v;
        if ((in & kCvLo) && lo) lo[p] = v;
        if ((in & kCvHi) && hi) hi[p] = v;
    }
    // one colour pass (two slots at a time, loads before stores: a pass never
    // reads the cells it writes); from_zero: the other colour is 0
    __device__ void pass(int c, bool from_zero) const
    {
        for (int m = threadIdx.x; m < pairs; m += 2 * kCvThreads) {
            T v[2];
            int in[2], p[2];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int mu = m + u * kCvThreads;
                if (u && mu >= pairs) continue;
                in[u] = info[mu];
                const T bb = b[c * cap + mu];
                const int base = in[u] & kCvPos;
                const bool q = ((in[u] >> kCvParBit) ^ c) & 1;   // the cell of colour c is the pair's odd one
                p[u] = base + (q ? h : 0);
                T di, o = sizeof(T) == 8 ? bb : T(0);
                if (from_zero) rec[c * cap + mu].get_di(di);
                else o = off(rec[c * cap + mu], p[u], base + (q ? 0 : h - 1), di, bb);
                v[u] = (sizeof(T) == 8 ? o : bb + o) * di;
            }
            put(p[0], v[0], in[0]);
            if (m + kCvThreads < pairs) put(p[1], v[1], in[1]);
        }
    }
    // x += the parent's coarse correction on the even-coloured cells
    __device__ void correct(const T *xc) const
    {
        for (int m = threadIdx.x; m < pairs; m += kCvThreads) {
            const int in = info[m], p = (in & kCvPos) + ((in & kCvPar) ? h : 0);
            put(p, x[p] + xc[cpos[m]], in);
        }
    }
};

template <class T>
__global__ void __cluster_dims__(kCvCtas, 1, 1) __launch_bounds__(kCvThreads, 1)
    k_cc_coarse_vcycle(const __grid_constant__ CoarseVC<T> D)
{
    namespace cg = cooperative_groups;
    using F = typename VFace<T>::type;
    using Rec = CvRec<F, T>;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char cvsm[];
    __shared__ CvLevel lv[3];
    const int comp = blockIdx.y, tid = threadIdx.x, rank = (int)cl.block_rank(), na = D.na, split_z = D.split_z, nd = D.nd;
    const int npd = cv_np(D.A3[nd].A.g, split_z), nl = D.n - 1;   // nl smoothed levels
    const bool act = rank < na;
    const CvLayout &L = D.L;
    if (tid < nl) {
        const int l = tid;
        const GridD &g = D.A3[l].A.g;
        const bool slab = l < nd;
        CvLevel v;
        v.x = L.x[l]; v.rec = L.rec[l]; v.b = L.b[l]; v.dg = L.dg[l]; v.info = L.info[l]; v.cpos = L.cpos[l];
        v.nx = g.nx; v.h = g.nx >> 1; v.no = cv_no(g, split_z); v.plane = v.no * g.nx;
        v.sy = split_z ? g.nx : v.plane;
        v.sz = split_z ? v.plane : g.nx;
        v.s0 = slab && act ? cv_s0(npd, na, nd, l, rank) : 0;
        v.pl = !act ? 0 : (slab ? cv_s0(npd, na, nd, l, rank + 1) - v.s0 : npd);
        v.pairs = v.pl * v.no * v.h;
        v.cap = (slab ? cv_plmax(npd, na, nd, l) : npd) * v.no * v.h;   // (offsets are the same in every block)
        v.lo_rank = slab && act && rank > 0 ? rank - 1 : -1;
        v.hi_rank = slab && act && rank + 1 < na ? rank + 1 : -1;
        v.dlo = v.lo_rank >= 0 ? (v.s0 - cv_s0(npd, na, nd, l, rank - 1)) * v.plane : 0;
        v.dhi = -v.pl * v.plane;
        lv[l] = v;
    }
    __syncthreads();
    // halo planes and cells not yet written meet zero coefficients only, but
    // must be finite
    for (int l = 0; l < nl; l++) {
        T *x = reinterpret_cast<T *>(cvsm + lv[l].x);
        for (int q = tid; q < (lv[l].pl + 2) * lv[l].plane; q += kCvThreads) x[q] = T(0);
    }
    // every level's records in one loop (level by level their load latencies
    // added up); kU pairs' loads before their use, a slot past the end loads
    // the first pair again
    constexpr int kU = CvLoad<T>::n;
    const int n0 = lv[0].pairs, n1 = n0 + (nl > 1 ? lv[1].pairs : 0), n2 = n1 + (nl > 2 ? lv[2].pairs : 0);
    for (int m0 = tid; m0 < n2; m0 += kU * kCvThreads) {
        F f[kU][11];
        T d[kU][3], bb[kU][2];
        int ts[kU], os[kU], ss[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const int m = m0 + u * kCvThreads < n2 ? m0 + u * kCvThreads : 0;
            const int l = m < n0 ? 0 : (m < n1 ? 1 : 2), ml = m - (l == 0 ? 0 : (l == 1 ? n0 : n1));
            const VOp<T> &A = D.A3[l].A;
            const int r = ml / lv[l].h;
            ts[u] = ml - r * lv[l].h;
            ss[u] = r / lv[l].no;
            os[u] = r - ss[u] * lv[l].no;
            const int j = split_z ? os[u] : lv[l].s0 + ss[u], k = split_z ? lv[l].s0 + ss[u] : os[u];
            const CellPos p0 = cell_pos<T>(A.g, 2 * ts[u], j, k), p1 = cell_pos<T>(A.g, 2 * ts[u] + 1, j, k);
            f[u][0] = A.bx[p0.fx0];
            f[u][1] = A.bx[p0.fx1];
            f[u][2] = A.bx[p1.fx1];
            f[u][3] = A.by[p0.fy0];
            f[u][4] = A.by[p0.fy1];
            f[u][5] = A.by[p1.fy0];
            f[u][6] = A.by[p1.fy1];
            f[u][7] = A.bz[p0.fz0];
            f[u][8] = A.bz[p0.fz1];
            f[u][9] = A.bz[p1.fz0];
            f[u][10] = A.bz[p1.fz1];
            d[u][0] = D.A3[l].dinv[comp][p0.c];
            d[u][1] = D.A3[l].dinv[comp][p1.c];
            d[u][2] = D.A3[l].diag[comp][((j + k) & 1) ? p1.c : p0.c];
            if (l == 0) {
                bb[u][0] = D.b.p[comp][p0.c];
                bb[u][1] = D.b.p[comp][p1.c];
            }
        }
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const int m = m0 + u * kCvThreads;
            if (m >= n2) continue;
            const int l = m < n0 ? 0 : (m < n1 ? 1 : 2), ml = m - (l == 0 ? 0 : (l == 1 ? n0 : n1));
            const CvLevel &v = lv[l];
            const GridD &g = D.A3[l].A.g, &gc = D.A3[l + 1].A.g;
            const int t = ts[u], o = os[u], sl = ss[u];
            const int j = split_z ? o : v.s0 + sl, k = split_z ? v.s0 + sl : o, c0 = (j + k) & 1;   // colour of the even cell
            int *info = reinterpret_cast<int *>(cvsm + v.info), *cpos = reinterpret_cast<int *>(cvsm + v.cpos);
            info[ml] = ((sl + 1) * v.plane + o * v.nx + t) | (c0 ? kCvPar : 0) | (sl == 0 ? kCvLo : 0) |
                       (sl == v.pl - 1 ? kCvHi : 0);
            // parent: one level down row-split with a halo plane, or the bottom in natural order
            const int cs0 = l + 1 < nd ? lv[l + 1].s0 : 0;
            cpos[ml] = l + 1 == nl ? ((k >> 1) * gc.ny + (j >> 1)) * gc.nx + t
                                   : ((((v.s0 + sl) >> 1) - cs0 + 1) * (v.no >> 1) + (o >> 1)) * gc.nx + spos(gc.nx, t);
            const F z = F(0.0f);
            const bool j0 = j == 0, j1 = j == g.ny - 1, k0 = k == 0, k1 = k == g.nz - 1;
            const F fe[6] = {t == 0 ? z : f[u][0], f[u][1], j0 ? z : f[u][3], j1 ? z : f[u][4], k0 ? z : f[u][7],
                             k1 ? z : f[u][8]};
            const F fo[6] = {f[u][1], t == v.h - 1 ? z : f[u][2], j0 ? z : f[u][5], j1 ? z : f[u][6], k0 ? z : f[u][9],
                             k1 ? z : f[u][10]};
            Rec *rec = reinterpret_cast<Rec *>(cvsm + v.rec);
            rec[c0 * v.cap + ml].set(fe, d[u][0]);
            rec[(1 - c0) * v.cap + ml].set(fo, d[u][1]);
            reinterpret_cast<T *>(cvsm + v.dg)[ml] = d[u][2];   // of the even-coloured cell, for its residual
            if (l == 0) {
                T *b = reinterpret_cast<T *>(cvsm + v.b);
                b[c0 * v.cap + ml] = bb[u][0];
                b[(1 - c0) * v.cap + ml] = bb[u][1];
            }
        }
    }
    // this block's rows of the bottom inverse: staged, or on their way into L2
    const int br0 = D.nb * min(rank, na) / na, br1 = D.nb * min(rank + 1, na) / na;
    {
        const double *src = D.binv.p[comp] + (size_t)br0 * D.nb;
        const int n = (br1 - br0) * D.nb;
        if (L.bi >= 0) {
            double *bi = reinterpret_cast<double *>(cvsm + L.bi);
            for (int q = tid; q < n; q += kCvThreads) bi[q] = src[q];
        } else {
            for (int q = tid * 16; q < n; q += 16 * kCvThreads) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(src + q));
        }
    }
    cl.sync();

    T *res = reinterpret_cast<T *>(cvsm + L.res), *xb = reinterpret_cast<T *>(cvsm + L.xb);
    double *bs = reinterpret_cast<double *>(cvsm + L.bs), *ps = reinterpret_cast<double *>(cvsm + L.ps);
    auto view = [&](int l) {
        const CvLevel &v = lv[l];
        CvView<T> w;
        w.x = reinterpret_cast<T *>(cvsm + v.x);
        w.rec = reinterpret_cast<const Rec *>(cvsm + v.rec);
        w.b = reinterpret_cast<const T *>(cvsm + v.b);
        w.info = reinterpret_cast<const int *>(cvsm + v.info);
        w.cpos = reinterpret_cast<const int *>(cvsm + v.cpos);
        w.lo = v.lo_rank >= 0 ? cl.map_shared_rank(w.x, v.lo_rank) + v.dlo : nullptr;
        w.hi = v.hi_rank >= 0 ? cl.map_shared_rank(w.x, v.hi_rank) + v.dhi : nullptr;
        w.h = v.h; w.sy = v.sy; w.sz = v.sz; w.pairs = v.pairs; w.cap = v.cap;
        return w;
    };
    auto bar = [&](int l) {
        if (l < nd) cl.sync();
        else __syncthreads();
    };
    // Down (dir 0): two sweeps from zero, red first; up (dir 1): the coarse
    // correction, then two sweeps, black first.  Nobody reads the last pass's
    // halo, so it writes none (the other blocks may have ended by then: every
    // remote write is followed by a cluster barrier that its target takes
    // part in) and needs no cluster barrier.
    auto smooth = [&](int l, int dir, const T *xc) {
        CvView<T> w = view(l);
        if (dir == 0) w.pass(0, true);
        else w.correct(xc);
        bar(l);
#pragma unroll 1
        for (int it = dir == 0 ? 1 : 0; it < 4; it++) {
            const bool last = dir == 1 && it == 3;
            if (last) w.lo = w.hi = nullptr;
            w.pass((it & 1) ^ dir, false);
            if (last) __syncthreads();
            else bar(l);
        }
    };
#pragma unroll 1
    for (int l = 0; l < nl; l++) {
        if (l < nd || act) {
            smooth(l, 0, nullptr);
            // residuals of the even-coloured cells, then their averages over
            // the children in rr_cell's order
            {
                const CvView<T> w = view(l);
                const T *dg = reinterpret_cast<const T *>(cvsm + lv[l].dg);
                for (int m = tid; m < w.pairs; m += kCvThreads) {
                    const int in = w.info[m], base = in & kCvPos, p = base + ((in & kCvPar) ? w.h : 0);
                    T di;
                    const T o = w.off(w.rec[m], p, base + ((in & kCvPar) ? 0 : w.h - 1), di, w.b[m] - dg[m] * w.x[p]);
                    res[p - lv[l].plane] = sizeof(T) == 8 ? o : w.b[m] - (dg[m] * w.x[p] - o);
                }
            }
            __syncthreads();
            const GridD &gc = D.A3[l + 1].A.g;
            const CvLevel &v = lv[l];
            const int noc = v.no >> 1, nc = (v.pl >> 1) * noc * gc.nx;
            for (int m = tid; m < nc; m += kCvThreads) {
                const int r = m / gc.nx, I = m - r * gc.nx, S = r / noc, O = r - S * noc;
                T s = 0;
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    if (__popc(e) & 1) continue;
                    const int dj = (e >> 1) & 1, dk = e >> 2;
                    const int o = 2 * O + (split_z ? dj : dk), sl = 2 * S + (split_z ? dk : dj);
                    s += res[(sl * v.no + o) * v.nx + ((e & 1) ? v.h : 0) + I];
                }
                s *= T(0.125);
                // to the next level: its right-hand side (this block's slab, or
                // every active block's copy), or the bottom's in natural order
                const int Sg = (v.s0 >> 1) + S;
                if (l + 1 < nl) {
                    T *bq = reinterpret_cast<T *>(cvsm + lv[l + 1].b);
                    const bool own = l + 1 < nd || l >= nd;
                    const int Sl = own ? S : Sg, col = (I + O + (v.s0 >> 1) + S) & 1;   // colour of (I, O, Sg)
                    const int at = col * lv[l + 1].cap + (Sl * noc + O) * (gc.nx >> 1) + (I >> 1);
                    if (own) bq[at] = s;
                    else
                        for (int a = 0; a < na; a++) cl.map_shared_rank(bq, a)[at] = s;
                } else {
                    const int at = (split_z ? Sg * gc.ny + O : O * gc.ny + Sg) * gc.nx + I;
                    if (l >= nd) bs[at] = (double)s;
                    else
                        for (int a = 0; a < na; a++) cl.map_shared_rank(bs, a)[at] = (double)s;
                }
            }
        }
        // (the next level's right-hand side comes from other blocks where it stops being cut)
        if (l + 1 == nd) cl.sync();
        else __syncthreads();
    }
    // bottom: x = inv b, each block its share of the rows (FP64: one SM would
    // take nb^2 / 2 cycles), 16 lanes per row, the result to every block
    {
        const double *bi = L.bi >= 0 ? reinterpret_cast<const double *>(cvsm + L.bi) : D.binv.p[comp] + (size_t)br0 * D.nb;
        const int nr = act ? br1 - br0 : 0, g = tid & 15;
        for (int rr = tid >> 4; rr < (nr + 1) / 2 * 2; rr += kCvThreads / 16) {   // (whole warps)
            double sum = 0.0;
            if (rr < nr) {
                const double *row = bi + (size_t)rr * D.nb;
#pragma unroll 4
                for (int q = g; q < D.nb; q += 16) sum += row[q] * bs[q];
            }
            for (int o = 8; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o, 16);
            if (g == 0 && rr < nr)
                for (int a = 0; a < na; a++) cl.map_shared_rank(xb, a)[br0 + rr] = (T)sum;
        }
        cl.sync();
    }
#pragma unroll 1
    for (int l = nl - 1; l >= 0; l--)
        if (l < nd || act) smooth(l, 1, l == nl - 1 ? xb : reinterpret_cast<const T *>(cvsm + lv[l + 1].x));
    // the top level's x, and b.x over the block's cells (FP32 products, FP64 sums: a block has few cells)
    double dot = 0.0;
    {
        const GridD &g = D.A3[0].A.g;
        const CvView<T> w = view(0);
        const CvLevel &v = lv[0];
        for (int m = tid; m < w.pairs; m += kCvThreads) {
            const int r = m / v.h, t = m - r * v.h, sl = r / v.no, o = r - sl * v.no;
            const int j = split_z ? o : v.s0 + sl, k = split_z ? v.s0 + sl : o, p = (w.info[m] & kCvPos);
            const int c0 = (w.info[m] & kCvPar) ? 1 : 0;   // colour of the even cell
            const T x0 = w.x[p], x1 = w.x[p + v.h];
            D.x.p[comp][cix<T>(g, 2 * t, j, k)] = x0;
            D.x.p[comp][cix<T>(g, 2 * t + 1, j, k)] = x1;
            if (D.part) dot += dot_term(w.b[c0 * w.cap + m], x0) + dot_term(w.b[(1 - c0) * w.cap + m], x1);
        }
    }
    if (D.part) {
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_down_sync(0xffffffffu, dot, o);
        if ((tid & 31) == 0) ps[tid >> 5] = dot;
        __syncthreads();
        if (tid == 0) {
            double sum = 0.0;
            for (int q = 0; q < kCvThreads / 32; q++) sum += ps[q];
            D.part[comp * kPartComp + rank] = sum;
        }
    }
}

// Which levels of the hierarchy the cluster kernel takes: fills the shape of D
// and returns its top level, or -1 (no smoothed level fits: the bottom alone).
// By the level sizes only: the largest top level whose slabs fit in shared
// memory.  The finest level of a grid above 16^3 keeps its own kernels: its
// last sweep forms r.z, and the whole GPU's sweeps of 32^3 cells (4.3 us each)
// take about as long as eight blocks'.
template <class T>
int cv_plan(const CcHier &H, CoarseVC<T> &D)
{
    const int Lb = H.L - 1;
    for (int l0 = 0; l0 < Lb; l0++) {
        const int cells = ncell(H.lv[l0].g);
        const int nd = cells <= kCoarseCells ? 1 : 2, n = Lb - l0 + 1;
        if (nd == 2 && (l0 == 0 || sizeof(T) != 4 || cells > kCvTopCells)) continue;
        if (n < nd + 1 || n > nd + 2) continue;
        for (int q = 0; q < n; q++) D.A3[q].A.g = H.lv[l0 + q].g;
        const GridD &gd = D.A3[nd].A.g;   // the first level that is not cut
        D.n = n;
        D.nd = nd;
        D.split_z = gd.nz >= gd.ny;
        D.na = std::min(kCvCtas, cv_np(gd, D.split_z));
        D.nb = H.nb;
        if (n == nd + 2 && ncell(gd) > 512) continue;
        D.L = cv_layout(D);
        if (D.L.total <= kCvSmem) return l0;
    }
    return -1;
}

// ---- the coarse end of the nodal V-cycle in one cluster --------------------------
// Below a level of at most kNcNodes nodes a nodal V-cycle is ten launches per
// level of two to four microseconds each.  One cluster of kNcCtas blocks runs
// that level and all below it: every smoothed level in slabs of node planes
// (nested: a coarse plane K belongs to the block of fine plane 2K), the vectors,
// cell fractions and node records in shared memory, the planes at a slab's ends
// written to the neighbouring blocks before the cluster barrier that ends a
// step, and the bottom rows shared out.  Steps and per-node operations are those
// of k_nd_cheb, k_nd_resid, k_nd_restrict and k_nd_prolong.  Every remote write
// is followed by a cluster barrier that its target takes part in.
// kNcNodes: FP32 a 16^3-cell level; FP64 an 8^3-cell one (of a 17^3-node level
// the FP64 operations alone take eight SMs 5 us a step, a launch over the whole
// GPU 4).  Per V-cycle 31 us in FP32 for 19 launches of 2.2-3.8 us and their
// gaps (two steps at 64^3 15.1 -> 14.6 ms), 25 us in FP64 for ten of 2-5 us
// (64^3 gradient, 12-instance sweep: 3.5 and 2.8 % faster).  A step over 600
// nodes of the 17^3 level takes 1.5 us, half of it instruction issue.
constexpr int kNcCtas = 8, kNcThreads = 512, kNcMax = 4, kNcSmem = 200 * 1024;
template <class T> struct NcNodes { static constexpr int n = sizeof(T) == 4 ? 8192 : 1024; };
struct NcLayout {
    int x[kNcMax], t[kNcMax], d[kNcMax], b[kNcMax], dg[kNcMax], di[kNcMax], al[kNcMax], rec[kNcMax], bs, xb, total;
};
template <class T>
struct NdCoarse {
    int n;                 // levels; the last is the bottom
    int na;                // blocks that own a slab
    NdOp<T> A[kNcMax];
    T *x;
    const T *b;
    const double *binv;
    int nb;
    T cd[3], cr[3];
    NcLayout L;
};
// first node plane of rank r's slab on smoothed level l of ns (npb: planes of
// the last smoothed level)
__host__ __device__ inline int nc_s0(int npb, int na, int ns, int l, int np, int r)
{
    return r >= na ? np : (npb * r / na) << (ns - 1 - l);
}
template <class T>
inline NcLayout nc_layout(const NdCoarse<T> &D)
{
    NcLayout o;
    int at = 0;
    auto take = [&](size_t bytes) { const int q = at; at += (int)((bytes + 15) & ~(size_t)15); return q; };
    const int ns = D.n - 1, npb = D.A[ns - 1].g.nz + 1;
    for (int l = 0; l < ns; l++) {
        const GridD &g = D.A[l].g;
        const int P = (g.nx + 1) * (g.ny + 1), np = g.nz + 1;
        int pl = 0;
        for (int r = 0; r < D.na; r++)
            pl = std::max(pl, nc_s0(npb, D.na, ns, l, np, r + 1) - nc_s0(npb, D.na, ns, l, np, r));
        o.x[l] = take((size_t)(pl + 2) * P * sizeof(T));
        o.t[l] = take((size_t)(pl + 2) * P * sizeof(T));
        o.d[l] = take((size_t)pl * P * sizeof(T));
        o.b[l] = take((size_t)pl * P * sizeof(T));
        o.dg[l] = take((size_t)pl * P * sizeof(T));
        o.di[l] = take((size_t)pl * P * sizeof(T));
        o.al[l] = take((size_t)(pl + 1) * g.nx * g.ny * sizeof(T));
        o.rec[l] = take((size_t)pl * P * 4);
    }
    o.bs = take((size_t)D.nb * 8);
    o.xb = take((size_t)D.nb * sizeof(T));
    o.total = at;
    return o;
}
// node record: i, j, plane within the slab (10 bits each), kind (2)
__device__ inline int nc_rec(int i, int j, int sl, int kind) { return i | (j << 10) | (sl << 20) | (kind << 30); }

struct NcLevel {
    int NX, NY, P, nx, ny, s0, pl, np, nodes;
    int nreg, nirr;   // listed nodes: records rec[0 .. nreg), and from the array's end
    int lo_rank, hi_rank, dlo, dhi;
};

template <class T>
__global__ void __cluster_dims__(kNcCtas, 1, 1) __launch_bounds__(kNcThreads)
    k_nd_coarse(const __grid_constant__ NdCoarse<T> D)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char ncsm[];
    __shared__ NcLevel lv[kNcMax];
    const int tid = threadIdx.x, rank = (int)cl.block_rank(), na = D.na, ns = D.n - 1;
    const bool act = rank < na;
    const NcLayout &L = D.L;
    const int npb = D.A[ns - 1].g.nz + 1;
    if (tid < ns) {
        const GridD &g = D.A[tid].g;
        NcLevel v;
        v.nx = g.nx; v.ny = g.ny; v.NX = g.nx + 1; v.NY = g.ny + 1; v.P = v.NX * v.NY; v.np = g.nz + 1;
        v.s0 = act ? nc_s0(npb, na, ns, tid, v.np, rank) : 0;
        v.pl = act ? nc_s0(npb, na, ns, tid, v.np, rank + 1) - v.s0 : 0;
        v.nodes = v.pl * v.P;
        v.nreg = v.nirr = 0;
        v.lo_rank = act && rank > 0 ? rank - 1 : -1;
        v.hi_rank = act && rank + 1 < na ? rank + 1 : -1;
        v.dlo = v.lo_rank >= 0 ? (v.s0 - nc_s0(npb, na, ns, tid, v.np, rank - 1)) * v.P : 0;
        v.dhi = -v.pl * v.P;
        lv[tid] = v;
    }
    __syncthreads();
    auto arr = [&](int off) { return reinterpret_cast<T *>(ncsm + off); };
    for (int l = 0; l < ns; l++) {
        NcLevel &v = lv[l];
        const NdOp<T> &A = D.A[l];
        T *x = arr(L.x[l]), *t = arr(L.t[l]), *b = arr(L.b[l]), *d = arr(L.d[l]), *al = arr(L.al[l]);
        int *rec = reinterpret_cast<int *>(ncsm + L.rec[l]);
        // (halo planes outside the box and inactive nodes stay 0)
        for (int q = tid; q < v.nodes + 2 * v.P; q += kNcThreads) x[q] = t[q] = T(0);
        // cell planes s0 - 1 .. s0 + pl - 1
        const int cp = v.nx * v.ny;
        for (int q = tid; q < (v.pl + 1) * cp && act; q += kNcThreads) {
            const int ck = v.s0 - 1 + q / cp;
            al[q] = ck >= 0 && ck < A.g.nz ? A.alpha[ck * cp + q % cp] : T(0);
        }
        for (int q = tid; q < v.nodes; q += kNcThreads) {
            const int sl = q / v.P, r = q - sl * v.P, j = r / v.NX, i = r - j * v.NX;
            const int n = v.s0 * v.P + q;
            // regular nodes from the front, the others from the back: a warp of
            // a step then takes one of the two rows (their order is of no
            // consequence, a node's result depends on no other of the step)
            const int kind = A.kind[n];
            if (kind == ND_REG) rec[atomicAdd(&v.nreg, 1)] = nc_rec(i, j, sl, kind);
            if (kind == ND_IRR) rec[v.nodes - 1 - atomicAdd(&v.nirr, 1)] = nc_rec(i, j, sl, kind);
            d[q] = T(0);
            if (l == 0) b[q] = D.b[n];
        }
    }
    __syncthreads();
    // f(q, w) for every active node of level l, records w
    auto each = [&](int l, auto &&f) {
        const NcLevel &v = lv[l];
        const int *rec = reinterpret_cast<const int *>(ncsm + L.rec[l]);
        const int np32 = (v.nreg + 31) & ~31, n = np32 + v.nirr;
        for (int m = tid; m < n; m += kNcThreads) {
            if (m >= v.nreg && m < np32) continue;
            const int w = m < v.nreg ? rec[m] : rec[v.nodes - 1 - (m - np32)];
            f(((w >> 20) & 1023) * v.P + ((w >> 10) & 1023) * v.NX + (w & 1023), w);
        }
    };
    // diagonals, once per V-cycle (an FP64 division and a sum of eight per node)
    for (int l = 0; l < ns; l++) {
        const NcLevel &v = lv[l];
        const T *al = arr(L.al[l]), h = D.A[l].h;
        T *dg = arr(L.dg[l]), *di = arr(L.di[l]);
        each(l, [&](int q, int w) {
            const int i = w & 1023, j = (w >> 10) & 1023, sl = (w >> 20) & 1023;
            T sa = T(8);
            if ((unsigned)w >> 30 == ND_IRR) {
                T a8[8];
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    const int ci = i - 1 + (e & 1), cj = j - 1 + ((e >> 1) & 1);
                    a8[e] = (unsigned)ci < (unsigned)v.nx && (unsigned)cj < (unsigned)v.ny
                                ? al[((sl + (e >> 2)) * v.ny + cj) * v.nx + ci] : T(0);
                }
                sa = ((a8[0] + a8[1]) + (a8[2] + a8[3])) + ((a8[4] + a8[5]) + (a8[6] + a8[7]));
            }
            const T g = h * sa * T(1.0 / 3.0);
            dg[q] = g;
            di[q] = T(1) / g;
        });
    }
    cl.sync();

    // row of node q (record w) on x, as nd_row, its sums as trees (the FP64
    // chains were the time of a step)
    auto row = [&](const NcLevel &v, const T *al, T h, const T *x, int q, int w, T diag) -> T {
        const int i = w & 1023, j = (w >> 10) & 1023, sl = (w >> 20) & 1023;
        const T *xc = x + q + v.P;
        const int sy = v.NX, sz = v.P;
        T s;
        if ((unsigned)w >> 30 == ND_REG) {
            const T b0 = (xc[1 + sy] + xc[-1 + sy]) + (xc[1 - sy] + xc[-1 - sy]);
            const T am = (xc[1 - sz] + xc[-1 - sz]) + (xc[sy - sz] + xc[-sy - sz]);
            const T ap = (xc[1 + sz] + xc[-1 + sz]) + (xc[sy + sz] + xc[-sy + sz]);
            const T bm = (xc[1 + sy - sz] + xc[-1 + sy - sz]) + (xc[1 - sy - sz] + xc[-1 - sy - sz]);
            const T bp = (xc[1 + sy + sz] + xc[-1 + sy + sz]) + (xc[1 - sy + sz] + xc[-1 - sy + sz]);
            s = T(2) * (b0 + (am + ap)) + (bm + bp);
        } else {
            // per cell its fraction times its three face-diagonal and one
            // body-diagonal neighbours (outside the box the fraction is 0; the
            // index is clamped to the node itself there)
            T pr[8];
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const int ex = e & 1, ey = (e >> 1) & 1, ez = e >> 2, ci = i - 1 + ex, cj = j - 1 + ey;
                const bool in = (unsigned)ci < (unsigned)v.nx && (unsigned)cj < (unsigned)v.ny;
                const T a = in ? al[((sl + ez) * v.ny + cj) * v.nx + ci] : T(0);
                const int ox = in ? 2 * ex - 1 : 0, oy = in ? (2 * ey - 1) * sy : 0, oz = in ? (2 * ez - 1) * sz : 0;
                pr[e] = a * ((xc[ox + oy] + xc[ox + oz]) + (xc[oy + oz] + xc[ox + oy + oz]));
            }
            s = ((pr[0] + pr[1]) + (pr[2] + pr[3])) + ((pr[4] + pr[5]) + (pr[6] + pr[7]));
        }
        return diag * xc[0] - h * T(1.0 / 12.0) * s;
    };
    // own value at node q, and the copies in the neighbours' halo planes
    auto put = [&](const NcLevel &v, T *x, T *lo, T *hi, int q, T val) {
        const int p = q + v.P;
        x[p] = val;
        if (lo && q < v.P) lo[p + v.dlo] = val;
        if (hi && q >= v.nodes - v.P) hi[p + v.dhi] = val;
    };
    // one Chebyshev step src -> dst (zero: src and the direction are 0)
    auto cheb = [&](int l, const T *src, T *dst, int step, bool zero, bool halo) {
        const NcLevel &v = lv[l];
        const T h = D.A[l].h, cd = D.cd[step], cr = D.cr[step];
        const T *b = arr(L.b[l]), *al = arr(L.al[l]), *dg = arr(L.dg[l]), *di = arr(L.di[l]);
        T *d = arr(L.d[l]);
        T *lo = halo && v.lo_rank >= 0 ? cl.map_shared_rank(dst, v.lo_rank) : nullptr;
        T *hi = halo && v.hi_rank >= 0 ? cl.map_shared_rank(dst, v.hi_rank) : nullptr;
        each(l, [&](int q, int w) {
            T r = b[q];
            if (!zero) r -= row(v, al, h, src, q, w, dg[q]);
            T dn = cr * (r * di[q]);
            if (!zero && cd != T(0)) dn += cd * d[q];
            d[q] = dn;
            put(v, dst, lo, hi, q, zero ? dn : src[q + v.P] + dn);
        });
    };
#pragma unroll 1
    for (int l = 0; l < ns; l++) {
        const NcLevel &v = lv[l];
        T *x = arr(L.x[l]), *t = arr(L.t[l]);
        cheb(l, x, x, 0, true, true);
        cl.sync();
        cheb(l, x, t, 1, false, true);
        cl.sync();
        cheb(l, t, x, 2, false, true);
        cl.sync();
        {   // residual into t (0 on inactive nodes, as t is there)
            const T h = D.A[l].h;
            const T *b = arr(L.b[l]), *al = arr(L.al[l]), *dg = arr(L.dg[l]);
            T *lo = v.lo_rank >= 0 ? cl.map_shared_rank(t, v.lo_rank) : nullptr;
            T *hi = v.hi_rank >= 0 ? cl.map_shared_rank(t, v.hi_rank) : nullptr;
            each(l, [&](int q, int w) { put(v, t, lo, hi, q, b[q] - row(v, al, h, x, q, w, dg[q])); });
        }
        cl.sync();
        // full weighting: coarse planes K with 2 K in the slab
        const GridD &gc = D.A[l + 1].g;
        const int CX = gc.nx + 1, CP = CX * (gc.ny + 1);
        const int K0 = (v.s0 + 1) >> 1, K1 = act ? (v.s0 + v.pl + 1) >> 1 : K0;
        for (int m = tid; m < (K1 - K0) * CP; m += kNcThreads) {
            const int K = K0 + m / CP, r = m % CP, J = r / CX, I = r - J * CX;
            // (planes outside the box hold 0; an index outside a row or plane is
            // clamped to the centre and its weight is 0)
            const uint8_t on = D.A[l + 1].act[K * CP + r];
            const T *tc = t + (2 * K - v.s0 + 1) * v.P + 2 * J * v.NX + 2 * I;
            const int im = I > 0 ? -1 : 0, ip = 2 * I < v.nx ? 1 : 0, jm = J > 0 ? -v.NX : 0, jp = 2 * J < v.ny ? v.NX : 0;
            const T wm = I > 0 ? T(0.5) : T(0), wp = ip ? T(0.5) : T(0), vm = J > 0 ? T(0.5) : T(0), vp = jp ? T(0.5) : T(0);
            auto line = [&](const T *q) { return q[0] + (wm * q[im] + wp * q[ip]); };
            auto plane = [&](const T *q) { return line(q) + (vm * line(q + jm) + vp * line(q + jp)); };
            T sum = plane(tc) + T(0.5) * (plane(tc - v.P) + plane(tc + v.P));
            if (!on) sum = T(0);
            if (l + 1 < ns) arr(L.b[l + 1])[K * CP + r - lv[l + 1].s0 * CP] = sum;
            else {
                double *bs = reinterpret_cast<double *>(ncsm + L.bs);
                for (int a = 0; a < na; a++) cl.map_shared_rank(bs, a)[K * CP + r] = (double)sum;
            }
        }
        if (l + 1 < ns) __syncthreads();
        else cl.sync();
    }
    {   // bottom: x = inv b, this block's share of the rows, 16 lanes per row, to every block
        const double *bs = reinterpret_cast<const double *>(ncsm + L.bs);
        T *xb = arr(L.xb);
        const int r0 = D.nb * min(rank, na) / na, nr = D.nb * min(rank + 1, na) / na - r0, g = tid & 15;
        for (int rr = tid >> 4; rr < (nr + 1) / 2 * 2; rr += kNcThreads / 16) {
            double sum = 0.0;
            if (rr < nr) {
                const double *rw = D.binv + (size_t)(r0 + rr) * D.nb;
#pragma unroll 4
                for (int q = g; q < D.nb; q += 16) sum += rw[q] * bs[q];
            }
            for (int o = 8; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o, 16);
            if (g == 0 && rr < nr)
                for (int a = 0; a < na; a++) cl.map_shared_rank(xb, a)[r0 + rr] = (T)sum;
        }
        cl.sync();
    }
#pragma unroll 1
    for (int l = ns - 1; l >= 0; l--) {
        const NcLevel &v = lv[l];
        T *x = arr(L.x[l]), *t = arr(L.t[l]);
        const GridD &gc = D.A[l + 1].g;
        const int CX = gc.nx + 1, CP = CX * (gc.ny + 1);
        // coarse correction, at plane K: the bottom's whole array, or the
        // slab with its halo (fine planes 2c .. reach coarse plane c' of the next slab)
        const T *xc = l + 1 < ns ? arr(L.x[l + 1]) + (1 - lv[l + 1].s0) * CP : arr(L.xb);
        {
            T *lo = v.lo_rank >= 0 ? cl.map_shared_rank(t, v.lo_rank) : nullptr;
            T *hi = v.hi_rank >= 0 ? cl.map_shared_rank(t, v.hi_rank) : nullptr;
            each(l, [&](int q, int w) {
                const int i = w & 1023, j = (w >> 10) & 1023, k = v.s0 + ((w >> 20) & 1023);
                const int pi = i & 1, pj = j & 1, pk = k & 1;
                const T *c0 = xc + (k >> 1) * CP + (j >> 1) * CX + (i >> 1);
                // the two coarse neighbours along each axis (the same one twice at even positions)
                const int oj = pj ? CX : 0, ok = pk ? CP : 0;
                const T s0 = (c0[0] + c0[pi]) + (c0[oj] + c0[oj + pi]);
                const T s1 = (c0[ok] + c0[ok + pi]) + (c0[ok + oj] + c0[ok + oj + pi]);
                put(v, t, lo, hi, q, x[q + v.P] + T(0.125) * (s0 + s1));
            });
        }
        cl.sync();
        cheb(l, t, x, 0, false, true);
        cl.sync();
        cheb(l, x, t, 1, false, true);
        cl.sync();
        // (the top level's last step is read by nobody else: no remote write
        // without a barrier after it)
        cheb(l, t, x, 2, false, l > 0);
        if (l > 0) cl.sync();
        else __syncthreads();
    }
    {
        const NcLevel &v = lv[0];
        const T *x = arr(L.x[0]);
        for (int q = tid; q < v.nodes; q += kNcThreads) D.x[v.s0 * v.P + q] = x[q + v.P];
    }
}

// Which levels of the nodal hierarchy the cluster kernel takes: fills the shape
// of D and returns its top level, or -1 (the bottom alone).  By the sizes only.
template <class T>
int nc_plan(const NdHier &H, NdCoarse<T> &D)
{
    const int Lb = H.L - 1;
    for (int l0 = 0; l0 < Lb; l0++) {
        const int n = Lb - l0 + 1;
        if (n > kNcMax || nnode(H.lv[l0].g) > NcNodes<T>::n) continue;
        const GridD &g = H.lv[l0].g;
        if (g.nx >= 1023 || g.ny >= 1023 || g.nz >= 1023) continue;   // (record fields)
        for (int q = 0; q < n; q++) D.A[q].g = H.lv[l0 + q].g;
        D.n = n;
        D.nb = H.nb;
        D.na = std::min(kNcCtas, H.lv[Lb - 1].g.nz + 1);
        D.L = nc_layout(D);
        if (D.L.total <= kNcSmem) return l0;
    }
    return -1;
}

// ===========================================================================
// Krylov glue
// ===========================================================================

// Scale of the refinement solver's FP32 residuals: a power of two near 1/|b|
// (1 when |b| is 0 or not finite), so that corrections of right-hand sides far
// below 1 (down to round-off) do not underflow in FP32.  Multiplying by a
// power of two is exact, so in the usual range every FP32 operation gives
// the same bits as without it.  The FP64 norms are scaled alike.
__global__ void k_set_sigma(double *scal, int nc, int x_zero)
{
    if ((int)threadIdx.x >= nc) return;
    scal += threadIdx.x * kScalLen;
    const double bb = scal[S_BB];
    double sig = 1.0;
    if (bb > 0.0 && isfinite(bb)) sig = ldexp(1.0, -ilogb(sqrt(bb)));
    scal[S_SIG] = sig;
    scal[S_ISIG] = 1.0 / sig;   // exact: a power of two
    scal[S_BB] = bb * sig * sig;
    if (x_zero) scal[S_RR] = scal[S_BB];
}

// Writes a loop condition: the control word (polled by the host in eager
// mode) and, inside a captured graph, the conditional node's handle.
__device__ inline void set_cond(int *ctl, int slot, int v, cudaGraphConditionalHandle h, int use_h)
{
    ctl[slot] = v;
    if (use_h) cudaGraphSetConditional(h, v ? 1u : 0u);
}

// Opens the CG loop of the coming pass: of the components whose pass runs.
__global__ void k_inner_begin(int *ctl, int nc, cudaGraphConditionalHandle h, int use_h)
{
    if (threadIdx.x) return;
    for (int q = 0; q < nc; q++) ctl[q * C_LEN + C_COND_IN] = ctl[q * C_LEN + C_COND_OUT];
    set_cond(ctl, J_IN, 1, h, use_h);
}

__global__ void k_solve_begin(int *ctl, int nc)
{
    if (threadIdx.x) return;
    for (int q = 0; q < nc; q++) {
        int *c = ctl + q * C_LEN;
        c[C_IT] = 0; c[C_K] = 0; c[C_NOUT] = 0; c[C_STALL] = 0; c[C_ERR] = 0; c[C_ZERO] = 0;
        c[C_COND_OUT] = 1;
    }
    ctl[J_IT] = 0;
    ctl[J_NOUT] = 0;
}

// After a true residual (S_RR = |b - A x|^2, S_BB = |b|^2): record the
// relative residual and decide whether another CG pass (FP64 path: a
// restart; refinement path: one correction solve) runs.  Passes are capped
// at max_pass, iterations at maxit; a non-finite norm stops with E_NAN; b = 0
// flags x for zeroing.  For refinement, the inner target and stall state of
// the coming correction solve are set here.
__global__ void k_outer_check(double *scal0, int *ctl0, int nc, double tol, int maxit, int max_pass, int refine,
                              double inner_drop, cudaGraphConditionalHandle h, int use_h)
{
    // a lane per component
    int go = 0;
    const int q = threadIdx.x;
    double *scal = scal0 + q * kScalLen;
    int *ctl = ctl0 + q * C_LEN;
    if (q < nc && ctl[C_COND_OUT]) {   // (else this component's solve has ended)
        const double bb = scal[S_BB], rr = scal[S_RR];
        if (ctl[C_ERR] == 0) {
            if (!isfinite(rr) || !isfinite(bb)) {
                ctl[C_ERR] = E_NAN;
            } else if (bb == 0.0) {
                ctl[C_ZERO] = 1;
                scal[S_REL] = 0.0;
            } else {
                const double rel = sqrt(rr / bb);
                scal[S_REL] = rel;
                go = rel > tol && ctl[C_IT] < maxit && ctl[C_NOUT] < max_pass;
                if (go && refine) {
                    const double f = fmax(inner_drop, 0.5 * tol / rel);
                    scal[S_T2] = rr * f * f;
                    scal[S_PREV] = rr;
                    ctl[C_STALL] = 0;
                }
            }
        }
        ctl[C_NOUT]++;
        ctl[C_K] = 0;
        ctl[C_COND_OUT] = go;
    }
    const int any = __any_sync(0xffffffffu, go);
    if (q == 0) {
        ctl0[J_NOUT]++;
        set_cond(ctl0, J_OUT, any, h, use_h);
    }
}

// After one CG iteration (S_RR = recursive residual norm^2).  FP64 path:
// continue while |r|/|b| > tol/2.  Refinement path: continue until the
// correction's residual is below its target, or it has stalled (three
// iterations in a row that do not cut |r|^2 by 4: the FP32 round-off floor).
__device__ inline int inner_check(double *scal, int *ctl, double tol, int maxit, int refine)
{
    scal[S_RZOLD] = scal[S_RZ];
    ctl[C_IT]++;
    ctl[C_K]++;
    const double rr = scal[S_RR];
    int go = 1;
    if (!isfinite(rr)) {
        if (ctl[C_ERR] == 0) ctl[C_ERR] = E_NAN;   // (the first error word stands)
        go = 0;
    } else if (!refine) {
        go = sqrt(rr / scal[S_BB]) > 0.5 * tol;
    } else if (rr <= scal[S_T2]) {
        go = 0;
    } else {
        if (rr > 0.25 * scal[S_PREV]) {
            if (++ctl[C_STALL] >= 3) go = 0;
        } else {
            ctl[C_STALL] = 0;
        }
        scal[S_PREV] = rr;
    }
    if (ctl[C_IT] >= maxit || ctl[C_ERR]) go = 0;   // (an error word set by a kernel ends the solve)
    ctl[C_COND_IN] = go;
    return go;
}

// S_RR = the sum of the update's n block partials, then the same decision
// (one launch instead of a reduction and a check), per component: 128 threads
// sum, a lane of the first warp decides; the loop goes on while one component
// does.  (With 1024 threads per component's sum and one thread for the three
// decisions the FP64 shuffle steps and the chains of loads took 5.8 us for
// three components at 64^3; 3.2 us so.)
__global__ void __launch_bounds__(kMaxComp * kRedSmallThreads) k_reduce_inner_check(const double *part, int n, double *scal,
                                                                                  int *ctl, int nc, double tol, int maxit,
                                                                                  int refine,
                                                                                  cudaGraphConditionalHandle h, int use_h)
{
    __shared__ double sm[kMaxComp][kRedSmallThreads / 32], sum[kMaxComp];
    const int q = threadIdx.x / kRedSmallThreads, t = threadIdx.x % kRedSmallThreads;
    const double v = small_sum(part + q * kPartComp, n, t, sm[q]);
    if (t == 0) sum[q] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    int go = 0;
    if ((int)threadIdx.x < nc && ctl[threadIdx.x * C_LEN + C_COND_IN]) {
        const int c = threadIdx.x;
        scal[c * kScalLen + S_RR] = sum[c];
        go = inner_check(scal + c * kScalLen, ctl + c * C_LEN, tol, maxit, refine);
    }
    const int any = __any_sync(0xffffffffu, go);
    if (threadIdx.x == 0) {
        ctl[J_IT]++;
        set_cond(ctl, J_IN, any, h, use_h);
    }
}

// End of a solve: per-slot statistics, and the step's first failure
// (100 x error + slot) kept in C_STEPERR.
// The launch accounting of the joint loops goes to the first component's slot.
__global__ void k_solve_end(const double *scal0, int *ctl0, int nc, double tol, double *sstat, int slot0)
{
    if (threadIdx.x) return;
    for (int q = 0; q < nc; q++) {
        const double *scal = scal0 + q * kScalLen;
        int *ctl = ctl0 + q * C_LEN;
        const int slot = slot0 + q;
        const double rel = scal[S_REL];
        sstat[3 * slot] = ctl[C_IT];
        sstat[3 * slot + 1] = rel;
        sstat[3 * slot + 2] = ctl[C_NOUT];
        int e = ctl[C_ERR];
        if (e == 0 && !(rel <= tol)) e = E_NOTCONV;
        if (e) ctl[C_ERR] = e;
        if (e && ctl0[C_STEPERR] == 0) ctl0[C_STEPERR] = 100 * e + slot;
    }
    sstat[kSstatAcc + 2 * slot0] += ctl0[J_IT];
    sstat[kSstatAcc + 2 * slot0 + 1] += ctl0[J_NOUT] - 1;
}

__global__ void k_zero_if(V3<double> xv, int n, const int *ctl)
{
    if (!ctl[blockIdx.y * C_LEN + C_ZERO]) return;
    double *x = xv.p[blockIdx.y];
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) x[s] = 0.0;
}

__global__ void __launch_bounds__(256) k_resid_init(V3<const double> bv, V3<const double> qv, V3<double> rv, int n,
                                                    double *__restrict__ part, const int *act)
{
    const int comp = blockIdx.y;
    if (comp_off(act, comp)) return;
    const double *__restrict__ b = bv.p[comp], *__restrict__ q = qv.p[comp];
    double *__restrict__ r = rv.p[comp];
    part += comp * kPartComp;
    double v = 0.0, w = 0.0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        double rs = b[s] - q[s];
        r[s] = rs;
        v += rs * rs;
        w += b[s] * b[s];
    }
    v = block_sum<256>(v);
    w = block_sum<256>(w);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = v;
        part[gridDim.x + blockIdx.x] = w;
    }
}

__global__ void __launch_bounds__(256) k_cg_update(V3<double> xv, V3<double> rv, V3<const double> pv,
                                                   V3<const double> qv, const double *__restrict__ scal, int n,
                                                   double *__restrict__ part, const int *act)
{
    const int comp = blockIdx.y;
    if (comp_off(act, comp)) return;
    double *__restrict__ x = xv.p[comp], *__restrict__ r = rv.p[comp];
    const double *__restrict__ p = pv.p[comp], *__restrict__ q = qv.p[comp];
    scal += comp * kScalLen;
    part += comp * kPartComp;
    const double a = scal[S_ALPHA];
    double v = 0.0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        x[s] += a * p[s];
        double rs = r[s] - a * q[s];
        r[s] = rs;
        v += rs * rs;
    }
    v = block_sum<256>(v);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
}

__global__ void k_cg_pupdate(V3<double> pv, V3<const double> zv, const double *__restrict__ scal, int n,
                             const int *__restrict__ ctl, const int *act)
{
    const int comp = blockIdx.y;
    if (comp_off(act, comp)) return;
    double *__restrict__ p = pv.p[comp];
    const double *__restrict__ z = zv.p[comp];
    scal += comp * kScalLen;
    ctl += comp * C_LEN;
    const int first = ctl[C_K] == 0;
    const double beta = first ? 0.0 : scal[S_BETA];
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        p[s] = first ? z[s] : z[s] + beta * p[s];
}

// --- refinement: FP64 residual into an FP32 vector, FP32 inner CG, FP64 update.
// Per-thread sums of the FP32 kernels stay FP32 (a few dozen terms), block and
// final sums are FP64.

// Below kWideDot elements a thread's elements would take four FP32 additions
// where a thread per element takes none: there the FP32 products are summed in
// FP64 (275 k elements 0.4 us of the FP64 pipe); from there on a thread of the
// largest grid sums four or more of them either way.
constexpr int kWideDot = 4 * 256 * kReduceBlocks;
__global__ void __launch_bounds__(256) k_dot32(V3<const float> av, V3<const float> bv, int n, double *__restrict__ part)
{
    const float *__restrict__ a = av.p[blockIdx.y], *__restrict__ b = bv.p[blockIdx.y];
    part += blockIdx.y * kPartComp;
    float v = 0.0f;
    double dv = 0.0;
    const bool wide = n < kWideDot;
    const int n4 = n >> 2, t0 = blockIdx.x * blockDim.x + threadIdx.x, st = gridDim.x * blockDim.x;
    const float4 *a4 = reinterpret_cast<const float4 *>(a), *b4 = reinterpret_cast<const float4 *>(b);
    for (int s = t0; s < n4; s += st) {
        const float4 u = a4[s], w = b4[s];
        if (wide) {
            dv += (dot_term(u.x, w.x) + dot_term(u.y, w.y)) + (dot_term(u.z, w.z) + dot_term(u.w, w.w));
        } else {
            v += u.x * w.x;
            v += u.y * w.y;
            v += u.z * w.z;
            v += u.w * w.w;
        }
    }
    for (int s = 4 * n4 + t0; s < n; s += st) {
        if (wide) dv += dot_term(a[s], b[s]);
        else v += a[s] * b[s];
    }
    if (!wide) dv = (double)v;
    dv = block_sum_flat(dv);
    if (threadIdx.x == 0) part[blockIdx.x] = dv;
}

// r -= a q with a = rz/pq, partials of r.r.  (The solution update e += a p
// of the same iteration is deferred to the next k_cg_pupdate32, which reads
// p anyway, and after the last iteration to k_add32to64*.)
__global__ void __launch_bounds__(256) k_cg_update32(V3<float> rv, V3<const float> qv,
                                                     const double *__restrict__ scal, int n,
                                                     double *__restrict__ part, const int *act)
{
    const int comp = blockIdx.y;
    if (comp_off(act, comp)) return;
    float *__restrict__ r = rv.p[comp];
    const float *__restrict__ q = qv.p[comp];
    scal += comp * kScalLen;
    part += comp * kPartComp;
    const float a = (float)scal[S_ALPHA];
    float v = 0.0f;
    // 16-byte vectors (the arrays come from cudaMalloc), then the n % 4 tail:
    // four independent loads per thread keep enough bytes in flight
    const int n4 = n >> 2, t0 = blockIdx.x * blockDim.x + threadIdx.x, st = gridDim.x * blockDim.x;
    float4 *r4 = reinterpret_cast<float4 *>(r);
    const float4 *q4 = reinterpret_cast<const float4 *>(q);
    for (int s = t0; s < n4; s += st) {
        float4 rs = r4[s];
        const float4 qs = q4[s];
        rs.x = rs.x - a * qs.x;
        rs.y = rs.y - a * qs.y;
        rs.z = rs.z - a * qs.z;
        rs.w = rs.w - a * qs.w;
        r4[s] = rs;
        v += rs.x * rs.x;
        v += rs.y * rs.y;
        v += rs.z * rs.z;
        v += rs.w * rs.w;
    }
    for (int s = 4 * n4 + t0; s < n; s += st) {
        const float rs = r[s] - a * q[s];
        r[s] = rs;
        v += rs * rs;
    }
    double dv = block_sum<256>((double)v);
    if (threadIdx.x == 0) part[blockIdx.x] = dv;
}

// Iteration k of the FP32 CG: p = z (k = 0) or z + beta p, beta = rz/rz_old;
// for k >= 1 first the previous iteration's solution update with the old p,
// e = a p (k = 1) or e + a p, a = rz_old/pq (that iteration's step).
__global__ void k_cg_pupdate32(V3<float> pv3, V3<float> ev3, V3<const float> zv3, const double *__restrict__ scal, int n,
                               const int *__restrict__ ctl, const int *act)
{
    const int comp = blockIdx.y;
    if (comp_off(act, comp)) return;
    float *__restrict__ p = pv3.p[comp], *__restrict__ e = ev3.p[comp];
    const float *__restrict__ z = zv3.p[comp];
    scal += comp * kScalLen;
    ctl += comp * C_LEN;
    const int k = ctl[C_K];
    const float beta = k == 0 ? 0.0f : (float)scal[S_BETA];
    const float a = k == 0 ? 0.0f : (float)scal[S_ALPHA];   // of the iteration before
    // one element (each lane of a vector, and the tail)
    auto upd = [&](float &pv, float &ev, float zv) {
        if (k == 0) {
            pv = zv;
        } else {
            const float po = pv;
            ev = k == 1 ? a * po : ev + a * po;
            pv = zv + beta * po;
        }
    };
    // 16-byte vectors (cudaMalloc'd arrays), then the n % 4 tail
    const int n4 = n >> 2, t0 = blockIdx.x * blockDim.x + threadIdx.x, st = gridDim.x * blockDim.x;
    float4 *p4 = reinterpret_cast<float4 *>(p), *e4 = reinterpret_cast<float4 *>(e);
    const float4 *z4 = reinterpret_cast<const float4 *>(z);
    for (int s = t0; s < n4; s += st) {
        const float4 zv = z4[s];
        float4 pv = k == 0 ? zv : p4[s];
        float4 ev = k >= 2 ? e4[s] : make_float4(0.f, 0.f, 0.f, 0.f);
        upd(pv.x, ev.x, zv.x);
        upd(pv.y, ev.y, zv.y);
        upd(pv.z, ev.z, zv.z);
        upd(pv.w, ev.w, zv.w);
        p4[s] = pv;
        if (k >= 1) e4[s] = ev;
    }
    for (int s = 4 * n4 + t0; s < n; s += st) {
        float pv = k == 0 ? z[s] : p[s], ev = k >= 2 ? e[s] : 0.f;
        upd(pv, ev, z[s]);
        p[s] = pv;
        if (k >= 1) e[s] = ev;
    }
}

// After the last of the correction solve's k = ctl[C_K] iterations: its
// deferred solution update (a = rz_old/pq of that iteration) as in
// k_cg_pupdate32, then the FP64 solution x += e.
__device__ inline float final_e(const float *__restrict__ e, const float *__restrict__ p, float a, int k, int s)
{
    return k == 1 ? a * p[s] : e[s] + a * p[s];
}

__global__ void k_add32to64(double *__restrict__ x, const float *__restrict__ e, const float *__restrict__ p,
                            const double *__restrict__ scal, const int *__restrict__ ctl, int n)
{
    const int k = ctl[C_K];
    const float a = (float)scal[S_ALPHA];
    const double isig = scal[S_ISIG];
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        x[s] += f32_to_f64(final_e(e, p, a, k, s)) * isig;
}

// k_add32to64 with e and p FP32 row-split vectors.  A thread owns one column
// and kAddPz planes, all loads before the stores: no division by the row
// length per cell, and one FP64 operation (the FMA; the widening is integer
// work, f32_to_f64).  64^3: 9.8 -> 4.1 us; 256^3 83 us (81 before), 4.9 TB/s
// of its 24 bytes per cell.
constexpr int kAddPz = 4;
inline dim3 add_grid(const GridD &g)
{
    return dim3((g.nx + 31) / 32, (g.ny + 7) / 8, (g.nz + kAddPz - 1) / kAddPz);
}
__global__ void __launch_bounds__(256) k_add32to64_split(GridD g, V3<double> xv3, V3<const float> ev3,
                                                         V3<const float> pv3, const double *__restrict__ scal,
                                                         const int *__restrict__ ctl, int nzb, const int *act)
{
    const CompZ cz(nzb);
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k0 = cz.z * kAddPz;
    if (i >= g.nx || j >= g.ny || comp_off(act, cz.comp)) return;
    double *__restrict__ x = xv3.p[cz.comp];
    const float *__restrict__ e = ev3.p[cz.comp], *__restrict__ p = pv3.p[cz.comp];
    scal += cz.comp * kScalLen;
    ctl += cz.comp * C_LEN;
    const int kit = ctl[C_K];
    const float a = (float)scal[S_ALPHA];
    const double isig = scal[S_ISIG];
    double xv[kAddPz];
    float ev[kAddPz];
#pragma unroll
    for (int q = 0; q < kAddPz; q++) {
        if (k0 + q >= g.nz) continue;
        xv[q] = x[cidx(g, i, j, k0 + q)];
        ev[q] = final_e(e, p, a, kit, cix<float>(g, i, j, k0 + q));
    }
#pragma unroll
    for (int q = 0; q < kAddPz; q++)
        if (k0 + q < g.nz) x[cidx(g, i, j, k0 + q)] = xv[q] + f32_to_f64(ev[q]) * isig;
}

__global__ void k_fill(double *a, int n, double v)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) a[s] = v;
}

__global__ void k_zero_inactive(int n, const uint8_t *__restrict__ act, double *__restrict__ x)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
        if (!act[s]) x[s] = 0.0;
}

inline dim3 cgrid(const GridD &g) { return grid3(g.nx, g.ny, g.nz); }
inline dim3 ngrid(const GridD &g) { return grid3(g.nx + 1, g.ny + 1, g.nz + 1); }
inline int nblocks3(dim3 b) { return b.x * b.y * b.z; }

// The Krylov operator of level L (FP32: level 0 only, FP32 faces, diag_a).
template <class T>
CcOp<T> ccop(const CcLevel &L)
{
    CcOp<T> A;
    A.g = L.g;
    if constexpr (sizeof(T) == 8) {
        A.diag = (const T *)L.diag_d; A.bx = (const T *)L.bf_d[0]; A.by = (const T *)L.bf_d[1]; A.bz = (const T *)L.bf_d[2];
    } else {
        A.diag = (const T *)L.diag_a; A.bx = (const T *)L.bf_f[0]; A.by = (const T *)L.bf_f[1]; A.bz = (const T *)L.bf_f[2];
    }
    return A;
}

// The V-cycle operator of level L (FP32: BF16 faces, diag_f).
template <class T>
VOp<T> vop(const CcLevel &L)
{
    VOp<T> A;
    A.g = L.g;
    if constexpr (sizeof(T) == 8) {
        A.diag = (const T *)L.diag_d; A.bx = (const T *)L.bf_d[0]; A.by = (const T *)L.bf_d[1]; A.bz = (const T *)L.bf_d[2];
        A.dinv = (const T *)L.diag_f;   // (the block of diag_f and dinv_f: see CcLevel)
    } else {
        A.diag = (const T *)L.diag_f;
        if constexpr (kVcycleBf16) {
            A.bx = L.bf_h[0]; A.by = L.bf_h[1]; A.bz = L.bf_h[2];
        } else {
            A.bx = (const typename VFace<T>::type *)L.bf_f[0];
            A.by = (const typename VFace<T>::type *)L.bf_f[1];
            A.bz = (const typename VFace<T>::type *)L.bf_f[2];
        }
        A.dinv = (const T *)L.dinv_f;
    }
    return A;
}

// The operators of level l for nc components: the selected variant, or all
// three (component q takes variant q).
template <class T>
CcOp3<T> ccop3(const CcHier &H, int nc)
{
    CcOp3<T> O;
    O.A = ccop<T>(H.lv[0]);
    for (int q = 0; q < kMaxComp; q++) {
        O.dinv[q] = nullptr;
        if (nc == 1) O.diag[q] = O.A.diag;
        else if constexpr (sizeof(T) == 8) O.diag[q] = (const T *)H.vdiag_d[q][0];
        else O.diag[q] = (const T *)H.vdiag_a[q];
    }
    return O;
}
template <class T>
VOp3<T> vop3(const CcHier &H, int l, int nc)
{
    VOp3<T> O;
    O.A = vop<T>(H.lv[l]);
    for (int q = 0; q < kMaxComp; q++) {
        O.diag[q] = O.A.diag;
        O.dinv[q] = O.A.dinv;
        if (nc == 1) continue;
        if constexpr (sizeof(T) == 8) {
            O.diag[q] = (const T *)H.vdiag_d[q][l];
            O.dinv[q] = (const T *)H.vdiag_f[q][l];
        } else {
            O.diag[q] = (const T *)H.vdiag_f[q][l];
            O.dinv[q] = (const T *)H.vdinv_f[q][l];
        }
    }
    return O;
}
// vector of every component: the first has its own arrays, the others theirs in
// the carved scratch (carve_components)
template <class T>
V3<T> comp_vec(Ctx *c, void *first, int kind, int l)
{
    return V3<T>((T *)first, (T *)c->cvec[0][kind][l], (T *)c->cvec[1][kind][l]);
}

// diagonals of every variant of level l from its extra and faces, in precision
// T (FP32: the V-cycle's, from the faces rounded as it stores them).
// inv (FP64): also the inverse diagonals, which the FP64 V-cycle reads.
template <class T>
void cc_make_diag(Ctx *c, CcHier &H, int l, bool inv = false)
{
    const CcLevel &L = H.lv[l];
    unsigned masks = 0;
    for (int q = 0; q < H.nvar; q++) masks |= (H.side_mask[q] & 0x3fu) << (6 * q);
    if constexpr (sizeof(T) == 8)
        EBV_LAUNCH(c, k_cc_make_diag<double>, cgrid(L.g), block3(), 0, L.g, L.extra_d, L.bf_d[0], L.bf_d[1],
                   L.bf_d[2], H.nvar, masks, H.vdiag_d[0][l], H.vdiag_d[1][l], H.vdiag_d[2][l],
                   inv ? (double *)H.vdiag_f[0][l] : nullptr, inv ? (double *)H.vdiag_f[1][l] : nullptr,
                   inv ? (double *)H.vdiag_f[2][l] : nullptr);
    else
        EBV_LAUNCH(c, (k_cc_make_diag<float, kVcycleBf16>), cgrid(L.g), block3(), 0, L.g, L.extra_f, L.bf_f[0], L.bf_f[1],
                   L.bf_f[2], H.nvar, masks, H.vdiag_f[0][l], H.vdiag_f[1][l], H.vdiag_f[2][l], H.vdinv_f[0][l],
                   H.vdinv_f[1][l], H.vdinv_f[2][l]);
}

// The V-cycle's BF16 copy of the FP32 faces of level L, and the padded copy
// of its x faces that the fused sweep loads (in the V-cycle's face type).
inline void cc_faces_bf16(Ctx *c, CcLevel &L)
{
    if (L.bxp)
        EBV_LAUNCH(c, k_xface_pad<RbF>, dim3(kReduceBlocks), dim3(256), 0, L.g, L.bf_f[0], (RbF *)L.bxp);
    if constexpr (!kVcycleBf16) return;
    for (int d = 0; d < 3; d++) {
        const int n = nface(L.g, d);
        EBV_LAUNCH(c, k_to_bf16, dim3(std::min(kReduceBlocks, (n + 255) / 256)), dim3(256), 0, L.bf_f[d], L.bf_h[d], n);
    }
}

template <class T>
NdOp<T> ndop(const NdLevel &L)
{
    NdOp<T> A;
    A.g = L.g;
    A.h = (T)L.g.h;
    if constexpr (sizeof(T) == 8) A.alpha = (const T *)L.alpha_d;
    else A.alpha = (const T *)L.alpha_f;
    A.act = L.act;
    A.kind = L.kind;
    return A;
}

// ---------------------------------------------------------------------------
// V-cycles
// ---------------------------------------------------------------------------

// Profiling labels of the colour passes per precision and level (level 0 is
// HBM-bound; the coarse levels are latency- and launch-bound): plain passes
// (from zero or not), the pass after the coarse correction, and the pass
// that also forms r.z; and of the residual-restriction per level.
static const char *const kGsName[2][8] = {
    {"cc_gs_colour_pass<double> L0", "cc_gs_colour_pass<double> L1", "cc_gs_colour_pass<double> L2",
     "cc_gs_colour_pass<double> L3", "cc_gs_colour_pass<double> L4", "cc_gs_colour_pass<double> L5",
     "cc_gs_colour_pass<double> L6", "cc_gs_colour_pass<double> L7+"},
    {"cc_gs_colour_pass<float> L0", "cc_gs_colour_pass<float> L1", "cc_gs_colour_pass<float> L2",
     "cc_gs_colour_pass<float> L3", "cc_gs_colour_pass<float> L4", "cc_gs_colour_pass<float> L5",
     "cc_gs_colour_pass<float> L6", "cc_gs_colour_pass<float> L7+"}};
static const char *const kGsCorrName[2][8] = {
    {"cc_gs_correction_pass<double> L0", "cc_gs_correction_pass<double> L1", "cc_gs_correction_pass<double> L2",
     "cc_gs_correction_pass<double> L3", "cc_gs_correction_pass<double> L4", "cc_gs_correction_pass<double> L5",
     "cc_gs_correction_pass<double> L6", "cc_gs_correction_pass<double> L7+"},
    {"cc_gs_correction_pass<float> L0", "cc_gs_correction_pass<float> L1", "cc_gs_correction_pass<float> L2",
     "cc_gs_correction_pass<float> L3", "cc_gs_correction_pass<float> L4", "cc_gs_correction_pass<float> L5",
     "cc_gs_correction_pass<float> L6", "cc_gs_correction_pass<float> L7+"}};
static const char *const kGsDotName[2] = {"cc_gs_rz_pass<double> L0", "cc_gs_rz_pass<float> L0"};
static const char *const kRrName[2][4] = {
    {"cc_residual_restrict<double> L0", "cc_residual_restrict<double> L1", "cc_residual_restrict<double> L2",
     "cc_residual_restrict<double> L3+"},
    {"cc_residual_restrict<float> L0", "cc_residual_restrict<float> L1", "cc_residual_restrict<float> L2",
     "cc_residual_restrict<float> L3+"}};

// Two red-black Gauss-Seidel sweeps in place (the first from x = 0 when
// zero_start), each as two colour passes.
inline dim3 gs_grid(const GridD &g, dim3 bk)
{
    const int nzg = (g.nz + GS_PZ - 1) / GS_PZ;
    return dim3(((g.nx + 1) / 2 + bk.x - 1) / bk.x, (g.ny + bk.y - 1) / bk.y, (nzg + bk.z - 1) / bk.z);
}
inline dim3 ch_grid(const GridD &g, dim3 bk)
{
    return dim3((g.nx + 1 + bk.x - 1) / bk.x, (g.ny + 1 + bk.y - 1) / bk.y, (g.nz + 1 + bk.z - 1) / bk.z);
}


// ---- the fused sweep on the host: where it applies, tensor maps, shape -----
enum { RB_ZERO = 0, RB_PLAIN = 1, RB_CORR = 2, RB_DOT = 3 };

inline int rb_ntiles(const GridD &g) { return ((g.nx / 2 + RB_HW - 1) / RB_HW) * ((g.ny + RB_TY - 1) / RB_TY); }

// FP32 levels whose half-rows are whole multiples of 8 positions (16-byte TMA
// strides for the BF16 face rows); their r.z partials are per (plane, tile).
inline bool rb_fusable(const GridD &g)
{
    return g.nx % 16 == 0 && g.nx >= 16 && (size_t)rb_ntiles(g) * g.nz <= kPartLen;
}

// Tensor map of one array of the level, by box kind: 0 x (FP32 cells, tile +
// 2 rows each side), 1 FP32 cells (tile + 1 row), 2 y faces, 3 z faces, 4 the
// padded x faces, 5 the coarse correction (g the coarse level: the parents
// of the tile and its ring); the array viewed as (half-row position, half,
// row, plane).
bool rb_map(Ctx *c, const void *p, int kind, const GridD &g, CUtensorMap *out)
{
    if (!p) return false;
    for (const auto &e : c->tma)
        if (e.p == p && e.kind == kind && e.nx == g.nx && e.ny == g.ny && e.nz == g.nz) {
            *out = e.m;
            return true;
        }
    const bool face = kind >= 2 && kind <= 4;
    const uint64_t es = face ? sizeof(RbF) : 4;
    const uint64_t hx = kind == 4 ? (uint64_t)rb_hxp(g.nx) : (uint64_t)g.nx / 2;
    const uint64_t rows = kind == 2 ? g.ny + 1 : g.ny, planes = kind == 3 ? g.nz + 1 : g.nz;
    const uint64_t dims[4] = {hx, 2, rows, planes};
    const uint64_t st[3] = {hx * es, 2 * hx * es, rows * 2 * hx * es};
    const uint32_t box[4] = {(uint32_t)(kind == 5 ? RB_KW : (face ? RB_FW : RB_XW)), 2u,
                             (uint32_t)(kind == 0 ? RB_XR : (kind == 2 ? RB_YR : (kind == 5 ? RB_KR : RB_CR))), 1u};
    const CUtensorMapDataType ty = (face && sizeof(RbF) == 2) ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                              : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    Ctx::TmaEntry e;
    e.p = p;
    e.kind = kind;
    e.nx = g.nx;
    e.ny = g.ny;
    e.nz = g.nz;
    if (!tma_encode_4d(&e.m, ty, const_cast<void *>(p), dims, st, box)) return false;
    c->tma.push_back(e);
    *out = e.m;
    return true;
}

// Shared-memory limit of the fused sweeps on the context's device (raised by
// setup_solvers: the attribute belongs to the device, and a context on another
// one, or a second thread, must not find it half set), and the blocks of one
// that are resident on it at once.
cudaError_t rb_setup(Ctx *c)
{
    const int sb = RbSmem<RbF>::bytes;
    const cudaFuncAttribute smem_max = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_cc_rb_sweep<RbF, false, false, false>, smem_max, sb);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cc_rb_sweep<RbF, true, false, false>, smem_max, sb);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cc_rb_sweep<RbF, false, true, false>, smem_max, sb);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cc_rb_sweep<RbF, false, false, true>, smem_max, sb);
    int dev = 0, sms = 0, per = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cc_rb_sweep<RbF, false, false, false>, RB_THREADS, sb);
    c->rb_res = std::max(1, per) * std::max(1, sms);
    return e;
}

// Planes per chunk of a block: the fewest waves of resident blocks times the
// steps of one block (its planes and the two of the chunk's start).
int rb_kz(const Ctx *c, const GridD &g, int nc = 1)
{
    const long long nt = (long long)nc * rb_ntiles(g), res = c->rb_res;
    long long best = -1;
    int bkz = g.nz;
    for (int nc = 1; nc <= g.nz; nc++) {
        const int kz = (g.nz + nc - 1) / nc, ncr = (g.nz + kz - 1) / kz;
        const long long cost = ((nt * ncr + res - 1) / res) * (kz + 2);
        if (best < 0 || cost < best) {
            best = cost;
            bkz = kz;
        }
    }
    return bkz;
}

// One fused sweep (maps already encoded by rb_maps).
void rb_launch(Ctx *c, const char *name, const GridD &g, const RbMaps &tm, V3<float> xout, int c0, int mode,
               double *part, int kz = 0, int nc = 1, const int *act = nullptr)
{
    RbArgs<RbF> a;
    a.g = g;
    a.xout = xout;
    a.part = part;
    a.ctl = c->ctl;
    a.act = act;
    a.c0 = c0;
    a.kz = kz > 0 ? kz : rb_kz(c, g, nc);
    a.nzb = (g.nz + a.kz - 1) / a.kz;
    a.spin = spin_limit();
    const dim3 gr((g.nx / 2 + RB_HW - 1) / RB_HW, (g.ny + RB_TY - 1) / RB_TY, a.nzb * nc);
    // algorithmic bytes: x written, x read (not from zero), b, 1/diag, three
    // faces, the coarse correction (1/8 word per cell)
    const double nb = (double)nc * ncell(g) * (4.0 + (mode == RB_ZERO ? 0.0 : 4.0) + 8.0 + 3.0 * sizeof(RbF) +
                                          (mode == RB_CORR ? 0.5 : 0.0));
    const int sb = RbSmem<RbF>::bytes;
    switch (mode) {
    case RB_ZERO:
        EBV_LAUNCH_P(c, name, nb, (k_cc_rb_sweep<RbF, true, false, false>), gr, dim3(RB_THREADS), sb, tm, a);
        break;
    case RB_CORR:
        EBV_LAUNCH_P(c, name, nb, (k_cc_rb_sweep<RbF, false, true, false>), gr, dim3(RB_THREADS), sb, tm, a);
        break;
    case RB_DOT:
        EBV_LAUNCH_P(c, name, nb, (k_cc_rb_sweep<RbF, false, false, true>), gr, dim3(RB_THREADS), sb, tm, a);
        break;
    default:
        EBV_LAUNCH_P(c, name, nb, (k_cc_rb_sweep<RbF, false, false, false>), gr, dim3(RB_THREADS), sb, tm, a);
    }
}

const char *const kRbName[8] = {"cc_rb_sweep<float> L0", "cc_rb_sweep<float> L1", "cc_rb_sweep<float> L2",
                                "cc_rb_sweep<float> L3", "cc_rb_sweep<float> L4", "cc_rb_sweep<float> L5",
                                "cc_rb_sweep<float> L6", "cc_rb_sweep<float> L7+"};

// Two red-black sweeps' worth of smoothing is two calls; this is one sweep
// pair as the V-cycle uses it: sweep 1 (from zero, or after the coarse
// correction) then sweep 2 (plain, or with r.z partials).
// dot_part: the last pass also writes partials of b.x -- per (plane, tile)
// (k_cc_rb_sweep<kDot> or k_cc_gs2_dot) on levels the fused sweep applies
// to, else per block of k_cc_gs<kDot>; returns their number (0 without
// dot_part).  FP32 levels with nx a multiple of 16 can run each sweep as one
// fused pass (x -> t -> x) or as two colour passes, with the same results bit
// for bit: ebv_set_fused_sweep picks the passes (0), the faster of the two as
// timed when the solvers are set up (1, the default) or the fused pass (2).
template <class T>
int cc_smooth2(Ctx *c, const CcHier &H, int l, int nc, const int *act, V3<T> x, V3<T> t, V3<const T> b, bool red_first,
               bool zero_start, V3<const T> xc = V3<const T>(), const GridD *gc = nullptr, double *dot_part = nullptr)
{
    const CcLevel &L = H.lv[l];
    const VOp3<T> A = vop3<T>(H, l, nc);
    const int c0 = red_first ? 0 : 1;
    const GridD &g = L.g;
    const bool corr = gc != nullptr;
    bool tiles = false;   // r.z partials per (plane, tile)
    if constexpr (sizeof(T) == 4) {
        if (rb_fusable(g)) {
            tiles = true;
            RbMaps m1, m2;
            // each kind of sweep (from zero, plain, after the coarse correction,
            // with r.z) was timed on its own against its colour passes
            const int mode = fused_sweep_mode();
            const int k1 = zero_start ? RB_ZERO : (corr ? RB_CORR : RB_PLAIN), k2 = dot_part ? RB_DOT : RB_PLAIN;
            // (the pair runs x -> t -> x fused, or in place as passes: one form for
            // both; timed with one component, for the joint solves too)
            const bool faster = L.rb_ms[k1][0] + L.rb_ms[k2][0] < L.rb_ms[k1][1] + L.rb_ms[k2][1];
            bool use = (mode == 2 || (mode == 1 && faster)) && rb_map(c, L.bxp, 4, g, &m1.fx) &&
                       rb_map(c, A.A.by, 2, g, &m1.fy) && rb_map(c, A.A.bz, 3, g, &m1.fz);
            m2.fx = m1.fx;
            m2.fy = m1.fy;
            m2.fz = m1.fz;
            for (int q = 0; q < nc && use; q++) {
                RbMaps::Comp &v1 = m1.v[q], &v2 = m2.v[q];
                use = rb_map(c, x.p[q], 0, g, &v1.x) && rb_map(c, t.p[q], 0, g, &v2.x) &&
                      rb_map(c, b.p[q], 1, g, &v1.b) && rb_map(c, A.dinv[q], 1, g, &v1.d);
                v2.b = v1.b;
                v2.d = v1.d;
                v1.xc = v2.xc = v1.b;   // (read by the correction sweep only)
                if (use && k1 == RB_CORR) use = rb_map(c, xc.p[q], 5, *gc, &v1.xc);
            }
            if (use) {
                const char *nm = kRbName[l < 7 ? l : 7];
                const int kz = nc == 1 ? L.rb_kz : 0;   // (the timed chunking is that of one component)
                rb_launch(c, nm, g, m1, t, c0, k1, nullptr, kz, nc, act);
                rb_launch(c, nm, g, m2, x, c0, k2, dot_part, kz, nc, act);
                return dot_part ? rb_ntiles(g) * g.nz : 0;
            }
        }
    }
    // algorithmic bytes of one colour pass: half of one sweep's x read and
    // write, b, diagonal and 3 face coefficients (in their storage type)
    const double nb = nc * 0.5 * ((4.0 * sizeof(T) + 3.0 * sizeof(typename VFace<T>::type)) * (double)ncell(g));
    // threads: x-pairs x rows x groups of GS_PZ planes, in the level's block shape
    const dim3 bk = L.gs_blk, gr = gs_grid(g, bk);
    const char *name = kGsName[sizeof(T) == 4][l < 7 ? l : 7];
    const V3<const T> none = V3<const T>();
    for (int s = 0; s < 2; s++) {
        const int z = (s == 0 && zero_start) ? 1 : 0;
        // the plain passes of FP32 levels with half-rows of a multiple of 4
        // cells take the vectorised form (same results)
        auto plain = [&](int color, int zs) {
            if constexpr (sizeof(T) == 4) {
                if (gs4_ok(g)) {
                    const dim3 g4 = gs4_grid(g, L.gs4_blk, L.gs4_pz);
                    if (L.gs4_pz == 1)
                        EBV_LAUNCH_P(c, name, nb, (k_cc_gs4<1>), comp_grid(g4, nc), L.gs4_blk, 0, A, x, b, g4.z, act,
                                     color, zs);
                    else
                        EBV_LAUNCH_P(c, name, nb, (k_cc_gs4<2>), comp_grid(g4, nc), L.gs4_blk, 0, A, x, b, g4.z, act,
                                     color, zs);
                    return;
                }
            }
            EBV_LAUNCH_P(c, name, nb, (k_cc_gs<T, false>), comp_grid(gr, nc), bk, 0, A, x, b, gr.z, act, color, zs, none,
                         GridD());
        };
        if (s == 0 && corr) {  // the first pass after the coarse-grid correction (+ the coarse array)
            const char *nmc = kGsCorrName[sizeof(T) == 4][l < 7 ? l : 7];
            const double nbc = nb + nc * 0.125 * sizeof(T) * (double)ncell(g);
            bool done = false;
            if constexpr (sizeof(T) == 4) {
                if (gs4_ok(g)) {   // vectorised, same results
                    const dim3 g4 = gs4_grid(g, L.gs4_blk, L.gs4_pz);
                    if (L.gs4_pz == 1)
                        EBV_LAUNCH_P(c, nmc, nbc, (k_cc_gs4<1, true>), comp_grid(g4, nc), L.gs4_blk, 0, A, x, b, g4.z,
                                     act, c0, z, xc, *gc);
                    else
                        EBV_LAUNCH_P(c, nmc, nbc, (k_cc_gs4<2, true>), comp_grid(g4, nc), L.gs4_blk, 0, A, x, b, g4.z,
                                     act, c0, z, xc, *gc);
                    done = true;
                }
            }
            if (!done)
                EBV_LAUNCH_P(c, nmc, nbc, (k_cc_gs<T, true>), comp_grid(gr, nc), bk, 0, A, x, b, gr.z, act, c0, z, xc,
                             *gc);
        }
        else
            plain(c0, z);
        if (s == 1 && dot_part && tiles) {
            // the fused sweep's r.z partials, per (plane, tile), with the last pass
            if constexpr (sizeof(T) == 4) {
                const dim3 gt((g.nx / 2 + RB_HW - 1) / RB_HW, (g.ny + RB_TY - 1) / RB_TY,
                              (g.nz + kGs2Planes - 1) / kGs2Planes);
                EBV_LAUNCH_P(c, kGsDotName[1], nb, k_cc_gs2_dot, comp_grid(gt, nc), dim3(RB_THREADS), 0, A, x, b, gt.z,
                             act, 1 - c0, dot_part);
                return rb_ntiles(g) * g.nz;
            }
        } else if (s == 1 && dot_part) {
            // fixed block shape: the grouping of its partial sums must not
            // follow the autotuned shape, or results would depend on timing
            const dim3 gd = gs_grid(g, block3());
            EBV_LAUNCH_P(c, kGsDotName[sizeof(T) == 4], nb, (k_cc_gs<T, false, true>), comp_grid(gd, nc), block3(), 0, A,
                         x, b, gd.z, act, 1 - c0, 0, none, GridD(), dot_part);
        } else {
            plain(1 - c0, 0);
        }
    }
    if (!dot_part) return 0;
    const dim3 gd = gs_grid(g, block3());
    return (int)(gd.x * gd.y * gd.z);
}

// One V-cycle x0 = M b0.  dot_part: the finest level's last pass (or the
// cluster kernel, where it takes that level) also writes block partials of
// b0.x0; returns their number (0 with a single level, or without dot_part).
template <class T>
int cc_vcycle(Ctx *c, CcHier &H, int nc, const int *act, V3<const T> b0, V3<T> x0, double *dot_part = nullptr)
{
    const int Lb = H.L - 1;
    // levels l0 .. Lb run in one cluster
    CoarseVC<T> D;
    const int lc = cv_plan<T>(H, D), l0 = lc < 0 ? Lb : lc;
    auto X = [&](int l) { return l ? comp_vec<T>(c, c->lx[l], Ctx::CV_X, l) : x0; };
    auto B = [&](int l) { return l ? V3<const T>(comp_vec<T>(c, c->lb[l], Ctx::CV_B, l)) : b0; };
    auto Tv = [&](int l) { return comp_vec<T>(c, c->lt[l], Ctx::CV_T, l); };
    for (int l = 0; l < l0; l++) {
        const CcLevel &L = H.lv[l];
        cc_smooth2<T>(c, H, l, nc, act, X(l), Tv(l), B(l), true, true);
        const CcLevel &Lc = H.lv[l + 1];
        const V3<T> bc = comp_vec<T>(c, c->lb[l + 1], Ctx::CV_B, l + 1);
        // x, b, diagonal, 3 faces (storage type) read, 1/8 word written
        const double nbr = nc * ((3.0 + 1.0 / 8.0) * sizeof(T) + 3.0 * sizeof(typename VFace<T>::type)) * (double)ncell(L.g);
        const char *nmr = kRrName[sizeof(T) == 4][l < 3 ? l : 3];
        bool vec = false;
        if constexpr (sizeof(T) == 4) {
            const dim3 bk(8, 8, 4), gr((Lc.g.nx / 4 + bk.x - 1) / bk.x, (Lc.g.ny + bk.y - 1) / bk.y,
                                        (Lc.g.nz + bk.z - 1) / bk.z);
            // four coarse cells per thread, vector loads (same results), where
            // that still gives two blocks per SM (small levels keep the scalar kernel)
            if (gs4_ok(L.g) && (long long)gr.x * gr.y * gr.z * nc >= kVecMinBlocks) {
                EBV_LAUNCH_P(c, nmr, nbr, k_cc_rr4, comp_grid(gr, nc), bk, 0, vop3<float>(H, l, nc), X(l), B(l), Lc.g, bc,
                             gr.z, act);
                vec = true;
            }
        }
        if (!vec) {
            const dim3 gr = cgrid(Lc.g);
            EBV_LAUNCH_P(c, nmr, nbr, k_cc_resid_restrict<T>, comp_grid(gr, nc), block3(), 0, vop3<T>(H, l, nc), X(l),
                         B(l), Lc.g, bc, gr.z, act);
        }
    }
    V3<const double> binv = one<const double>(H.binv);
    if (nc > 1)
        for (int q = 0; q < nc; q++) binv.p[q] = H.vbinv[q];
    if (l0 < Lb) {
        for (int q = 0; q < D.n; q++) D.A3[q] = vop3<T>(H, l0 + q, nc);
        D.x = X(l0);
        D.b = B(l0);
        D.binv = binv;
        D.nb = H.nb;
        D.part = l0 == 0 ? dot_part : nullptr;
        const size_t bytes = D.L.total;
        const char *nm = sizeof(T) == 4 ? "cc_coarse_vcycle<float>" : "cc_coarse_vcycle<double>";
        EBV_LAUNCH_P(c, nm, 0.0, k_cc_coarse_vcycle<T>, dim3(kCvCtas, nc), dim3(kCvThreads), bytes, D);
        if (l0 == 0) return dot_part ? kCvCtas : 0;
    } else {
        EBV_LAUNCH(c, k_bottom_solve<T>, dim3((H.nb + 7) / 8, nc), dim3(256), 0, binv, H.nb, B(Lb), X(Lb), H.lv[Lb].g,
                   (int)(sizeof(T) == 4));
    }
    for (int l = l0 - 1; l >= 0; l--) {
        // prolongation folded into the first colour pass of the post-smoothing
        const int nd = cc_smooth2<T>(c, H, l, nc, act, X(l), Tv(l), B(l), false, false, X(l + 1), &H.lv[l + 1].g,
                                     l == 0 ? dot_part : nullptr);
        if (l == 0) return nd;
    }
    return 0;
}

// Chebyshev coefficients on [lam_max / 8, lam_max] of D^-1 A, degree 3.
struct ChebCoef { double cd[3], cr[3]; };
inline ChebCoef cheb_coef(double lmax)
{
    const double lmin = lmax / 8.0;
    const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin), sigma = theta / delta;
    ChebCoef k;
    double rho0 = 1.0 / sigma;
    k.cd[0] = 0.0;
    k.cr[0] = 1.0 / theta;
    for (int s = 1; s < 3; s++) {
        double rho1 = 1.0 / (2.0 * sigma - rho0);
        k.cd[s] = rho1 * rho0;
        k.cr[s] = 2.0 * rho1 / delta;
        rho0 = rho1;
    }
    return k;
}

// Three Chebyshev steps on A x = b, ending in x.  From zero: (0) -> x -> t -> x.
// Otherwise the start is in t: t -> x -> t -> x.  d is the level's direction.
// A nodal pass on a level that marches: one launch for the listed nodes and
// the march; block partials per block of the launch.
template <class T, int kMode>
void nd_pass(Ctx *c, const NdLevel &L, const char *name, double nbytes, const T *xin, T *out, T *d, const T *b, T cd, T cr,
             double *part, float *out32 = nullptr, const double *sig = nullptr)
{
    const NdShape sh = nd_shape(L.g, L.nirr);
    EBV_LAUNCH_P(c, name, nbytes, (k_nd_pass<T, kMode>), dim3(sh.blocks), dim3(NT_T), 0, ndop<T>(L), sh, L.irr,
                 L.nirr, xin, out, d, b, nd_coef<T>((T)L.g.h, cd, cr), part, out32, sig);
}
// partial sums written by nd_pass on level L
inline int nd_pass_parts(const NdLevel &L) { return nd_shape(L.g, L.nirr).blocks; }

template <class T>
void nd_smooth(Ctx *c, const NdLevel &L, int l, T *x, T *t, const T *b, bool zero_start)
{
    NdOp<T> A = ndop<T>(L);
    ChebCoef k = cheb_coef(L.lam_max);
    T *d = (T *)c->ld[l];
    T *src = zero_start ? x : t, *dst = x;
    for (int s = 0; s < 3; s++) {
        // per node: x in/out, d in/out, b, alpha of one cell (the first step
        // from zero reads only b and alpha and writes d, x)
        const bool z0 = s == 0 && zero_start;
        const double nb = (z0 ? 4.0 : 6.0) * sizeof(T) * (double)nnode(L.g);
        if (z0)
            EBV_LAUNCH_P(c, sizeof(T) == 4 ? "nodal_chebyshev_first<float>" : "nodal_chebyshev_first<double>", nb,
                         k_nd_cheb0<T>,
                         dim3(std::min(8 * kReduceBlocks, (nnode(L.g) / (16 / (int)sizeof(T)) + 127) / 128 + 1)), dim3(128),
                         0, A, dst, d, b, (T)k.cr[s], nd_coef<T>((T)L.g.h, T(0), (T)k.cr[s]).crd, nnode(L.g));
        else if (L.march)   // plane-sum form
            nd_pass<T, ND_CHEB>(c, L,
                                   sizeof(T) == 4 ? (l ? "nodal_chebyshev_step<float> L1+" : "nodal_chebyshev_step<float> L0")
                                                  : (l ? "nodal_chebyshev_step<double> L1+" : "nodal_chebyshev_step<double> L0"),
                                   nb, src, dst, d, b, (T)k.cd[s], (T)k.cr[s], nullptr);
        else
            EBV_LAUNCH_P(c, sizeof(T) == 4 ? "nodal_chebyshev_step<float>" : "nodal_chebyshev_step<double>", nb,
                         k_nd_cheb<T>, ch_grid(L.g, L.ch_blk), L.ch_blk, 0, A, src, dst, d, b, (T)k.cd[s],
                         (T)k.cr[s]);
        src = dst;
        dst = (dst == x) ? t : x;
    }
}

template <class T>
void nd_vcycle(Ctx *c, NdHier &H, const T *b0, T *x0)
{
    const int Lb = H.L - 1;
    // levels l0 .. Lb run in one cluster
    NdCoarse<T> D;
    const int lc = nc_plan<T>(H, D), l0 = lc < 0 ? Lb : lc;
    for (int l = 0; l < l0; l++) {
        const NdLevel &L = H.lv[l];
        T *x = l ? (T *)c->lx[l] : x0;
        const T *b = l ? (const T *)c->lb[l] : b0;
        nd_smooth<T>(c, L, l, x, (T *)c->lt[l], b, true);
        if (L.march)
            nd_pass<T, ND_RESID>(c, L, l ? "nodal_residual L1+" : "nodal_residual L0", 0.0, x, (T *)c->lr[l], nullptr, b,
                                 T(0), T(0), nullptr);
        else
            EBV_LAUNCH(c, k_nd_resid<T>, ngrid(L.g), block3(), 0, ndop<T>(L), x, b, (T *)c->lr[l]);
        const NdLevel &Lc = H.lv[l + 1];
        EBV_LAUNCH(c, k_nd_restrict<T>, ngrid(Lc.g), block3(), 0, L.g, (const T *)c->lr[l], Lc.g, Lc.act,
                   (T *)c->lb[l + 1]);
    }
    {
        T *x = l0 ? (T *)c->lx[l0] : x0;
        const T *b = l0 ? (const T *)c->lb[l0] : b0;
        if (l0 < Lb) {
            for (int q = 0; q < D.n; q++) D.A[q] = ndop<T>(H.lv[l0 + q]);
            D.x = x;
            D.b = b;
            D.binv = H.binv;
            const ChebCoef k = cheb_coef(H.lv[l0].lam_max);   // (2 on every level)
            for (int q = 0; q < 3; q++) {
                D.cd[q] = (T)k.cd[q];
                D.cr[q] = (T)k.cr[q];
            }
            EBV_LAUNCH_P(c, sizeof(T) == 4 ? "nodal_coarse_vcycle<float>" : "nodal_coarse_vcycle<double>", 0.0,
                         k_nd_coarse<T>, dim3(kNcCtas), dim3(kNcThreads), D.L.total, D);
        } else {
            EBV_LAUNCH(c, k_bottom_solve<T>, dim3((H.nb + 7) / 8), dim3(256), 0, one<const double>(H.binv), H.nb,
                       one<const T>(b), one(x), H.lv[Lb].g, 0);
        }
    }
    for (int l = l0 - 1; l >= 0; l--) {
        const NdLevel &L = H.lv[l];
        T *x = l ? (T *)c->lx[l] : x0;
        const T *b = l ? (const T *)c->lb[l] : b0;
        // t = x + P x_coarse, then smooth from t back into x
        EBV_LAUNCH(c, k_nd_prolong<T>, prolong_grid(L.g, H.lv[l + 1].g), block3(), 0, L.g, L.act, H.lv[l + 1].g,
                   (const T *)c->lx[l + 1], x, (T *)c->lt[l]);
        nd_smooth<T>(c, L, l, x, (T *)c->lt[l], b, false);
    }
}

// ---------------------------------------------------------------------------
// Preconditioned conjugate gradients
// ---------------------------------------------------------------------------

// act: the loop condition words that gate a kernel's components (see comp_off),
// given where skipping an ended component saves more than the word's load costs
struct Problem {
    int nc = 1;                                // components solved together
    virtual ~Problem() {}
    virtual int n() const = 0;
    virtual int apply_blocks() const = 0;      // partial sums written by apply_dot
    virtual int apply_blocks32() const { return apply_blocks(); }   // by apply_dot32
    virtual int resid_blocks() const { return apply_blocks(); }     // by resid32
    // q = A p with block partials of p.q in c->part, in FP64 or FP32
    virtual void apply_dot(Ctx *c, V3<const double> p, V3<double> q, const int *act) = 0;
    virtual void apply_dot32(Ctx *c, V3<const float> p, V3<float> q, const int *act) = 0;
    // z = one V-cycle applied to r, in FP64, or in FP32 possibly leaving block
    // partials of r.z in c->part: returns their number, 0 if it did not
    virtual void precond(Ctx *c, V3<const double> r, V3<double> z, const int *act) = 0;
    virtual int precond32_dot(Ctx *c, V3<const float> r, V3<float> z, const int *act) = 0;
    // FP64 <-> FP32 vectors of the refinement solver (the FP32 side in the
    // layout of the problem's FP32 multigrid): r = b - A x in FP64 with
    // resid_blocks() block partials of |r|^2 in c->part; x += e
    virtual void resid32(Ctx *c, V3<const double> b, V3<const double> x, V3<float> r, const int *act) = 0;
    virtual void to32(Ctx *c, V3<const double> b, V3<float> r) = 0;   // r = b in the FP32 layout
    // x += e + the deferred last step of the correction solve (search direction p)
    virtual void add32(Ctx *c, V3<double> x, V3<const float> e, V3<const float> p, const int *act) = 0;
};

inline int vblocks(int n) { return std::min(kReduceBlocks, (n + 255) / 256); }
// for the FP32 CG kernels, whose threads take four elements at a time
inline int v4blocks(int n) { return std::min(kReduceBlocks, (n / 4 + 255) / 256 + 1); }

// A loop whose condition is decided on the device.  Eager mode: next()
// reads the condition word back (one synchronisation per pass).  Capture
// mode: the first next() adds a conditional WHILE node after the work issued
// so far and redirects the context's stream into the node's body graph; the
// second ends the body capture.  The kernel that sets the condition before
// the loop and the last kernel of the body take (h, use_h).
struct DevLoop {
    Ctx *c;
    int slot;
    cudaGraphConditionalHandle h = 0;
    int use_h = 0;
    int pass = 0;
    cudaStream_t saved = nullptr, body = nullptr;
    long long l0 = 0;
    int inner_count = 0;   // launches of a nested loop's body (capture mode)

    DevLoop(Ctx *c_, int slot_) : c(c_), slot(slot_)
    {
        if (!c->capturing) return;
        cudaStreamCaptureStatus st;
        cudaGraph_t g = nullptr;
        if (cudaStreamGetCaptureInfo(c->stream, &st, nullptr, &g) != cudaSuccess ||
            st != cudaStreamCaptureStatusActive ||
            cudaGraphConditionalHandleCreate(&h, g, 0, 0) != cudaSuccess) {
            if (c->cap_err.empty()) c->cap_err = "conditional handle";
            return;
        }
        use_h = 1;
    }

    bool next()
    {
        if (!c->capturing) {
            if (cudaMemcpyAsync(c->ctl_host + slot, c->ctl + slot, sizeof(int), cudaMemcpyDeviceToHost,
                                c->stream) != cudaSuccess ||
                cudaStreamSynchronize(c->stream) != cudaSuccess)
                return false;
            return c->ctl_host[slot] != 0;
        }
        if (pass == 0) {
            pass = 1;
            if (!use_h || c->cap_depth + 1 >= 4) {
                if (c->cap_err.empty()) c->cap_err = "loop nesting";
                return false;
            }
            cudaStreamCaptureStatus st;
            cudaGraph_t g = nullptr;
            const cudaGraphNode_t *deps = nullptr;
            size_t nd = 0;
            cudaGraphNodeParams np = {};
            np.type = cudaGraphNodeTypeConditional;
            np.conditional.handle = h;
            np.conditional.type = cudaGraphCondTypeWhile;
            np.conditional.size = 1;
            cudaGraphNode_t node;
            if (cudaStreamGetCaptureInfo(c->stream, &st, nullptr, &g, &deps, nullptr, &nd) != cudaSuccess ||
                cudaGraphAddNode(&node, g, deps, nullptr, nd, &np) != cudaSuccess ||
                cudaStreamUpdateCaptureDependencies(c->stream, &node, nullptr, 1,
                                                    cudaStreamSetCaptureDependencies) != cudaSuccess) {
                if (c->cap_err.empty()) c->cap_err = "conditional node";
                return false;
            }
            body = c->cap_stream[++c->cap_depth];
            if (cudaStreamBeginCaptureToGraph(body, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                              cudaStreamCaptureModeRelaxed) != cudaSuccess) {
                c->cap_depth--;
                if (c->cap_err.empty()) c->cap_err = "body capture";
                return false;
            }
            saved = c->stream;
            c->stream = body;
            l0 = c->launches;
            return true;
        }
        if (pass == 1) {
            pass = 2;
            cudaGraph_t gb = nullptr;
            if (cudaStreamEndCapture(body, &gb) != cudaSuccess && c->cap_err.empty()) c->cap_err = "body end";
            c->stream = saved;
            c->cap_depth--;
        }
        return false;
    }
    // launches captured in the body (valid after the loop in capture mode)
    int body_launches() const { return (int)(c->launches - l0); }
};

// Issues the end-of-solve kernels and, in eager mode, reads the solve's
// statistics and status back.
ebv_status finish_solve(Ctx *c, int nc, V3<double> x, int n, int *iters, double *res)
{
    EBV_LAUNCH(c, k_zero_if, dim3(vblocks(n), nc), dim3(256), 0, x, n, c->ctl);
    EBV_LAUNCH(c, k_solve_end, dim3(1), dim3(32), 0, c->scal, c->ctl, nc, c->prm.tol, c->sstat, c->cur_slot);
    if (c->capturing) {
        for (int q = 0; q < nc; q++) {
            if (iters) iters[q] = 0;
            if (res) res[q] = 0.0;
        }
        return EBV_OK;
    }
    const int s0 = c->cur_slot;
    EBV_CUDA_TRY(c, cudaMemcpyAsync(c->sstat_host + 3 * s0, c->sstat + 3 * s0, 3 * nc * sizeof(double),
                                    cudaMemcpyDeviceToHost, c->stream));
    EBV_CUDA_TRY(c, cudaMemcpyAsync(c->ctl_host, c->ctl, nc * C_LEN * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    EBV_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    for (int q = 0; q < nc; q++) {
        if (iters) iters[q] = (int)c->sstat_host[3 * (s0 + q)];
        if (res) res[q] = c->sstat_host[3 * (s0 + q) + 1];
    }
    for (int q = 0; q < nc; q++) {
        const int e = c->ctl_host[q * C_LEN + C_ERR], s = s0 + q;
        if (e == E_NAN) return c->fail(EBV_ERR_NAN, "non-finite residual (solve slot " + std::to_string(s) + ")");
        if (e == E_SMEM)
            return c->fail(EBV_ERR_CUDA, "shared memory of the fused sweep not 128-byte aligned (solve slot " +
                                             std::to_string(s) + ")");
        if (e == E_TIMEOUT)
            return c->fail(EBV_ERR_TIMEOUT, "a bounded wait in the smoother gave up (solve slot " + std::to_string(s) + ")");
        if (e == E_NOTCONV)
            return c->fail(EBV_ERR_NOT_CONVERGED, "linear solve did not reach the tolerance (solve slot " +
                                                      std::to_string(s) + ", relative residual " +
                                                      std::to_string(c->sstat_host[3 * s + 1]) + ", " +
                                                      std::to_string((int)c->sstat_host[3 * s]) + " iterations)");
    }
    return EBV_OK;
}

// Grids of at least this many cells skip the ended components of a joint solve
// in every kernel; on smaller ones the condition word's load (half a
// microsecond before each kernel's first) costs more than the redundant work,
// which only rewrites scratch vectors.
// (For one grid at a time: in a batch the redundant work takes SMs that other
// instances wait for, which was not measured.)
constexpr int kGateCells = 1 << 20;

// Preconditioned CG in FP64, restarted from the true residual whenever the
// recursive one has dropped below tol/2 but the true one is still above tol
// (at most 20 passes).
ebv_status pcg(Ctx *c, Problem &P, V3<const double> b, V3<double> x, int *iters, double *res)
{
    const int n = P.n(), nc = P.nc;
    const double tol = c->prm.tol;
    const int maxit = c->prm.max_iters;
    const V3<double> r = comp_vec<double>(c, c->kr, Ctx::CV_K, 0), z = comp_vec<double>(c, c->kz, Ctx::CV_K, 1),
                     p = comp_vec<double>(c, c->kp, Ctx::CV_K, 2), q = comp_vec<double>(c, c->kq, Ctx::CV_K, 3);
    const int *in = nc > 1 ? c->ctl + C_COND_IN : nullptr, *out = nc > 1 ? c->ctl + C_COND_OUT : nullptr;
    const int *gin = n >= kGateCells ? in : nullptr;
    const dim3 gv(vblocks(n), nc);
    auto true_residual = [&]() {
        P.apply_dot(c, x, q, out);
        EBV_LAUNCH(c, k_resid_init, gv, dim3(256), 0, b, q, r, n, c->part, out);
        reduce_comp(c, nc, vblocks(n), S_RR, kRedSum, out);
        reduce_comp(c, nc, vblocks(n), S_BB, kRedSum, out, c->part + vblocks(n));
    };
    EBV_LAUNCH(c, k_solve_begin, dim3(1), dim3(32), 0, c->ctl, nc);
    DevLoop outer(c, J_OUT);
    true_residual();
    EBV_LAUNCH(c, k_outer_check, dim3(1), dim3(32), 0, c->scal, c->ctl, nc, tol, maxit, 20, 0, 0.0, outer.h,
               outer.use_h);
    int inner_count = 0;
    while (outer.next()) {
        DevLoop inner(c, J_IN);
        EBV_LAUNCH(c, k_inner_begin, dim3(1), dim3(32), 0, c->ctl, nc, inner.h, inner.use_h);
        while (inner.next()) {
            P.precond(c, r, z, gin);
            EBV_LAUNCH(c, k_dot, gv, dim3(256), 0, r, z, n, c->part);
            reduce_comp(c, nc, vblocks(n), S_RZ, kRedBeta, in);
            EBV_LAUNCH(c, k_cg_pupdate, gv, dim3(256), 0, p, z, c->scal, n, c->ctl, in);
            P.apply_dot(c, p, q, gin);
            reduce_comp(c, nc, P.apply_blocks(), S_PQ, kRedAlpha, in);
            EBV_LAUNCH(c, k_cg_update, gv, dim3(256), 0, x, r, p, q, c->scal, n, c->part, in);
            EBV_LAUNCH(c, k_reduce_inner_check, dim3(1), dim3(nc * kRedSmallThreads), 0, c->part, vblocks(n), c->scal, c->ctl, nc, tol,
                       maxit, 0, inner.h, inner.use_h);
        }
        inner_count = inner.body_launches();
        true_residual();
        EBV_LAUNCH(c, k_outer_check, dim3(1), dim3(32), 0, c->scal, c->ctl, nc, tol, maxit, 20, 0, 0.0, outer.h,
                   outer.use_h);
    }
    if (c->capturing)
        c->loop_recs.push_back({c->cur_slot, outer.body_launches() - inner_count, inner_count});
    if (!c->cap_err.empty() && c->capturing) return c->fail(EBV_ERR_CUDA, "graph capture: " + c->cap_err);
    return finish_solve(c, nc, x, n, iters, res);
}

// Iterative refinement for the FP32 path: the residual r = b - A x and the
// solution update x += e are FP64; each correction e solves A e = r with
// conjugate gradients run entirely in FP32 (vectors, operator with FP32
// coefficients, V-cycle) until its residual drops by `inner_drop` (or it
// stalls), so FP64 arithmetic is spent once per refinement step instead of in
// every Krylov iteration.  At most 60 corrections.
ebv_status pcg_refine(Ctx *c, Problem &P, V3<const double> b, V3<double> x, int *iters, double *res, bool x_zero)
{
    const int n = P.n(), nc = P.nc;
    const double tol = c->prm.tol;
    const int maxit = c->prm.max_iters;
    const double inner_drop = refine_inner_drop();
    const V3<float> r = comp_vec<float>(c, c->kr32, Ctx::CV_K, 0), z = comp_vec<float>(c, c->kz32, Ctx::CV_K, 1),
                    p = comp_vec<float>(c, c->kp32, Ctx::CV_K, 2), q = comp_vec<float>(c, c->kq32, Ctx::CV_K, 3),
                    e = comp_vec<float>(c, c->ke32, Ctx::CV_K, 4);
    const int *in = nc > 1 ? c->ctl + C_COND_IN : nullptr, *out = nc > 1 ? c->ctl + C_COND_OUT : nullptr;
    const int *gin = n >= kGateCells ? in : nullptr;
    const dim3 gv(vblocks(n), nc), g4(v4blocks(n), nc);
    // x_zero: the first residual is b itself (its norm is |b|^2, reduced below)
    bool first_is_b = x_zero;
    auto true_residual = [&]() {
        if (first_is_b) {
            first_is_b = false;
            P.to32(c, b, r);
            return;
        }
        P.resid32(c, b, x, r, out);
        reduce_comp(c, nc, P.resid_blocks(), S_RR, kRedSum, out);
    };
    EBV_LAUNCH(c, k_solve_begin, dim3(1), dim3(32), 0, c->ctl, nc);
    EBV_LAUNCH(c, k_dot, gv, dim3(256), 0, b, b, n, c->part);
    reduce_comp(c, nc, vblocks(n), S_BB);
    EBV_LAUNCH(c, k_set_sigma, dim3(1), dim3(32), 0, c->scal, nc, x_zero ? 1 : 0);
    DevLoop outer(c, J_OUT);
    true_residual();
    EBV_LAUNCH(c, k_outer_check, dim3(1), dim3(32), 0, c->scal, c->ctl, nc, tol, maxit, 60, 1, inner_drop, outer.h,
               outer.use_h);
    int inner_count = 0;
    while (outer.next()) {
        DevLoop inner(c, J_IN);
        EBV_LAUNCH(c, k_inner_begin, dim3(1), dim3(32), 0, c->ctl, nc, inner.h, inner.use_h);
        while (inner.next()) {
            const int nd = P.precond32_dot(c, r, z, gin);
            if (!nd) EBV_LAUNCH(c, k_dot32, g4, dim3(256), 0, r, z, n, c->part);
            reduce_comp(c, nc, nd ? nd : v4blocks(n), S_RZ, kRedBeta, in);
            EBV_LAUNCH(c, k_cg_pupdate32, g4, dim3(256), 0, p, e, z, c->scal, n, c->ctl, in);
            P.apply_dot32(c, p, q, gin);
            reduce_comp(c, nc, P.apply_blocks32(), S_PQ, kRedAlpha, in);
            EBV_LAUNCH(c, k_cg_update32, g4, dim3(256), 0, r, q, c->scal, n, c->part, in);
            EBV_LAUNCH(c, k_reduce_inner_check, dim3(1), dim3(nc * kRedSmallThreads), 0, c->part, v4blocks(n), c->scal, c->ctl, nc, tol,
                       maxit, 1, inner.h, inner.use_h);
        }
        inner_count = inner.body_launches();
        P.add32(c, x, e, p, out);
        true_residual();
        EBV_LAUNCH(c, k_outer_check, dim3(1), dim3(32), 0, c->scal, c->ctl, nc, tol, maxit, 60, 1, inner_drop,
                   outer.h, outer.use_h);
    }
    if (c->capturing)
        c->loop_recs.push_back({c->cur_slot, outer.body_launches() - inner_count, inner_count});
    if (!c->cap_err.empty() && c->capturing) return c->fail(EBV_ERR_CUDA, "graph capture: " + c->cap_err);
    return finish_solve(c, nc, x, n, iters, res);
}

struct CcProblem : Problem {
    CcHier *H;
    int n() const override { return ncell(H->lv[0].g); }
    // two planes per thread
    dim3 agrid() const { const GridD &g = H->lv[0].g; return grid3(g.nx, g.ny, (g.nz + 1) / 2); }
    int apply_blocks() const override { return nblocks3(agrid()); }
    void apply_dot(Ctx *c, V3<const double> p, V3<double> q, const int *act) override
    {
        // p, diagonal, 3 faces, q: 6 words per cell
        const dim3 gr = agrid();
        EBV_LAUNCH_P(c, "cc_apply_fp64", nc * 48.0 * n(), k_cc_apply_dot<double>, comp_grid(gr, nc), block3(), 0,
                     ccop3<double>(*H, nc), p, q, c->part, gr.z, act);
    }
    // FP32 levels with nx a multiple of 8 large enough for two blocks per SM:
    // the vectorised apply.  By the operator, not by the components at hand
    // (the viscous one has three, solved together or one after another), so a
    // joint solve sums p.q as each component's own would
    bool vec32() const
    {
        return gs4_ok(H->lv[0].g) && H->nvar * nblocks3(apply4_grid(H->lv[0].g)) >= kVecMinBlocks;
    }
    int apply_blocks32() const override { return vec32() ? nblocks3(apply4_grid(H->lv[0].g)) : apply_blocks(); }
    void apply_dot32(Ctx *c, V3<const float> p, V3<float> q, const int *act) override
    {
        const dim3 g4 = apply4_grid(H->lv[0].g), gr = agrid();
        if (vec32())
            EBV_LAUNCH_P(c, "cc_apply_fp32", nc * 24.0 * n(), k_cc_apply4, comp_grid(g4, nc),
                         dim3(kApply4X, kApply4Y, kApply4Z), 0, ccop3<float>(*H, nc), p, q, c->part, g4.z, act);
        else
            EBV_LAUNCH_P(c, "cc_apply_fp32", nc * 24.0 * n(), k_cc_apply_dot<float>, comp_grid(gr, nc), block3(), 0,
                         ccop3<float>(*H, nc), p, q, c->part, gr.z, act);
    }
    void precond(Ctx *c, V3<const double> r, V3<double> z, const int *act) override
    {
        cc_vcycle<double>(c, *H, nc, act, r, z);
    }
    int precond32_dot(Ctx *c, V3<const float> r, V3<float> z, const int *act) override
    {
        return cc_vcycle<float>(c, *H, nc, act, r, z, c->part);
    }
    void resid32(Ctx *c, V3<const double> b, V3<const double> x, V3<float> r, const int *act) override
    {
        // x, diagonal, 3 faces, b read, r (FP32) written: 6.5 words per cell
        const dim3 gr = agrid();
        EBV_LAUNCH_P(c, "cc_resid_fp64", nc * 52.0 * n(), (k_cc_apply_dot<double, true>), comp_grid(gr, nc), block3(), 0,
                     ccop3<double>(*H, nc), x, V3<double>(), c->part, gr.z, act, b, r, c->scal + S_SIG);
    }
    void add32(Ctx *c, V3<double> x, V3<const float> e, V3<const float> p, const int *act) override
    {
        const dim3 gr = add_grid(H->lv[0].g);
        EBV_LAUNCH(c, k_add32to64_split, comp_grid(gr, nc), dim3(32, 8), 0, H->lv[0].g, x, e, p, c->scal, c->ctl, gr.z,
                   act);
    }
    void to32(Ctx *c, V3<const double> b, V3<float> r) override
    {
        for (int q = 0; q < nc; q++)
            EBV_LAUNCH(c, k_to_split, split_grid(H->lv[0].g, -1), block3(), 0, H->lv[0].g, -1, b.p[q], r.p[q],
                       c->scal + q * kScalLen + S_SIG);
    }
};

struct NdProblem : Problem {
    NdHier *H;
    int n() const override { return nnode(H->lv[0].g); }
    int apply_blocks() const override { return nd_pass_parts(H->lv[0]); }
    void apply_dot(Ctx *c, V3<const double> p, V3<double> q, const int *) override
    {
        // p read, q written, act and reg flags: 2.25 words per node
        nd_pass<double, ND_APPLY>(c, H->lv[0], "nodal_apply_fp64", 18.0 * n(), p.p[0], q.p[0], nullptr, nullptr, 0.0,
                                       0.0, c->part);
    }
    void apply_dot32(Ctx *c, V3<const float> p, V3<float> q, const int *) override
    {
        nd_pass<float, ND_APPLY>(c, H->lv[0], "nodal_apply_fp32", 12.0 * n(), p.p[0], q.p[0], nullptr, nullptr, 0.0f,
                                    0.0f, c->part);
    }
    void precond(Ctx *c, V3<const double> r, V3<double> z, const int *) override
    {
        nd_vcycle<double>(c, *H, r.p[0], z.p[0]);
    }
    int precond32_dot(Ctx *c, V3<const float> r, V3<float> z, const int *) override
    {
        nd_vcycle<float>(c, *H, r.p[0], z.p[0]);
        return 0;
    }
    void resid32(Ctx *c, V3<const double> b, V3<const double> x, V3<float> r, const int *) override
    {
        // x, b read, r (FP32) written, act and reg flags: 5.25 words per node
        nd_pass<double, ND_RES32>(c, H->lv[0], "nodal_resid_fp64", 22.0 * n(), x.p[0], nullptr, nullptr, b.p[0], 0.0,
                                       0.0, c->part, r.p[0], c->scal + S_SIG);
    }
    void add32(Ctx *c, V3<double> x, V3<const float> e, V3<const float> p, const int *) override
    {
        EBV_LAUNCH(c, k_add32to64, dim3(vblocks(n())), dim3(256), 0, x.p[0], e.p[0], p.p[0], c->scal, c->ctl, n());
    }
    void to32(Ctx *c, V3<const double> b, V3<float> r) override
    {
        EBV_LAUNCH(c, k_to32_scaled, dim3(vblocks(n())), dim3(256), 0, b.p[0], r.p[0], n(), c->scal + S_SIG);
    }
};

// x_zero: x holds zeros on entry (lets the refinement solver skip its first
// operator application)
ebv_status solve(Ctx *c, Problem &P, V3<const double> b, V3<double> x, int *iters, double *res, bool x_zero = false)
{
    if (c->prm.precision != EBV_FP64) return pcg_refine(c, P, b, x, iters, res, x_zero);
    return pcg(c, P, b, x, iters, res);
}

// The level and Krylov vectors of components 1 and 2 in precision T, carved
// from the cell gradients c->G and the face fluxes c->ff: explicit-term scratch
// that nothing reads during a solve (9 and more than 9 cell fields; about 8.6
// of each size are needed).  Sets c->joint: whether three components fit, and
// their partial sums in c->part.
template <class T>
void carve_components(Ctx *c)
{
    const CcHier &H = c->visc;
    const size_t N3 = ncell(c->g);
    char *base[2] = {(char *)c->G, (char *)c->ff};
    const size_t len[2] = {9 * N3 * 8, 3 * (size_t)(nface(c->g, 0) + nface(c->g, 1) + nface(c->g, 2)) * 8};
    bool ok = true;
    for (int q = 0; q < 2; q++) {
        size_t at = 0;
        auto take = [&](size_t n) -> void * {
            void *p = base[q] + at;
            at += (n * sizeof(T) + 255) / 256 * 256;
            if (at > len[q]) ok = false;
            return p;
        };
        for (int kind = 0; kind < Ctx::CV_KINDS; kind++)
            for (int l = 0; l < kMaxLevels; l++) c->cvec[q][kind][l] = nullptr;
        for (int k = 0; k < 5; k++) c->cvec[q][Ctx::CV_K][k] = take(N3);
        for (int l = 0; l < H.L; l++) {
            const size_t n = ncell(H.lv[l].g);
            c->cvec[q][Ctx::CV_T][l] = take(n);
            if (l == 0) continue;
            c->cvec[q][Ctx::CV_X][l] = take(n);
            c->cvec[q][Ctx::CV_B][l] = take(n);
        }
    }
    CcProblem P;
    P.H = &c->visc;
    P.nc = kMaxComp;
    const GridD &g = c->g;
    const dim3 gd = gs_grid(g, block3());
    const size_t tiles = rb_fusable(g) ? (size_t)rb_ntiles(g) * g.nz : 0;
    const size_t parts = std::max<size_t>(std::max(std::max(P.apply_blocks(), P.apply_blocks32()), nblocks3(gd)),
                                          std::max<size_t>(2 * kReduceBlocks, tiles));
    c->joint = ok && parts <= kPartComp;
}

// Coarse levels of a cell-centred hierarchy whose level-0 FP64 coefficients
// are set: the diagonals of every variant, in FP32 also the level-0 Krylov
// operator and on every level the V-cycle's BF16 faces with the diagonal (and
// its inverse) formed from them; then the bottom inverses of all variants.
ebv_status cc_finish_hierarchy(Ctx *c, CcHier &H, bool fp32)
{
    CcLevel &L0 = H.lv[0];
    cc_make_diag<double>(c, H, 0, !fp32);
    if (fp32) {
        // level 0 in FP32: the Krylov operator (the FP64 diagonal rounded),
        // then the V-cycle's BF16 faces and the diagonal formed from them
        const int n = ncell(L0.g);
        EBV_LAUNCH(c, k_to_split, split_grid(L0.g, -1), block3(), 0, L0.g, -1, L0.extra_d, L0.extra_f);
        for (int q = 0; q < H.nvar; q++)
            EBV_LAUNCH(c, k_to_split, split_grid(L0.g, -1), block3(), 0, L0.g, -1, H.vdiag_d[q][0], H.vdiag_a[q]);
        for (int d = 0; d < 3; d++)
            EBV_LAUNCH(c, k_to_split, split_grid(L0.g, d), block3(), 0, L0.g, d, L0.bf_d[d], L0.bf_f[d]);
        cc_faces_bf16(c, L0);
        cc_make_diag<float>(c, H, 0);
    }
    for (int l = 0; l + 1 < H.L; l++) {
        CcLevel &F = H.lv[l], &Cc = H.lv[l + 1];
        dim3 gr = grid3(Cc.g.nx + 1, Cc.g.ny + 1, Cc.g.nz + 1);
        if (fp32) {
            EBV_LAUNCH(c, k_cc_coarsen<float>, gr, block3(), 0, F.g, F.extra_f, F.bf_f[0], F.bf_f[1], F.bf_f[2], F.cov,
                       Cc.g, Cc.cov, Cc.extra_f, Cc.bf_f[0], Cc.bf_f[1], Cc.bf_f[2]);
            cc_faces_bf16(c, Cc);
            cc_make_diag<float>(c, H, l + 1);
        } else {
            EBV_LAUNCH(c, k_cc_coarsen<double>, gr, block3(), 0, F.g, F.extra_d, F.bf_d[0], F.bf_d[1], F.bf_d[2],
                       F.cov, Cc.g, Cc.cov, Cc.extra_d, Cc.bf_d[0], Cc.bf_d[1], Cc.bf_d[2]);
            cc_make_diag<double>(c, H, l + 1, true);
        }
    }
    const int lb = H.L - 1;
    const dim3 ga(gj_pad(H.nb), H.nvar);
    if (fp32) {
        BottomDiag<float> D = {{H.vdiag_f[0][lb], H.vdiag_f[1][lb], H.vdiag_f[2][lb]}};
        EBV_LAUNCH(c, k_cc_bottom_assemble<float>, ga, dim3(128), 0, vop<float>(H.lv[lb]), D, H.bmat, H.nb,
                   gj_scratch(H.nb));
    } else {
        BottomDiag<double> D = {{H.vdiag_d[0][lb], H.vdiag_d[1][lb], H.vdiag_d[2][lb]}};
        EBV_LAUNCH(c, k_cc_bottom_assemble<double>, ga, dim3(128), 0, vop<double>(H.lv[lb]), D, H.bmat, H.nb,
                   gj_scratch(H.nb));
    }
    bottom_invert(c, H.bmat, H.nb, H.nvar, H.vbinv);
    select_variant(H, 0);
    return EBV_OK;
}

// Level dimensions: halve while every dimension is even and the level has
// more than 64 cells (cell-centred) / 125 nodes (nodal).
int plan_levels(const GridD &g0, GridD *out, bool nodal)
{
    int L = 0;
    GridD g = g0;
    out[L++] = g;
    while (L < kMaxLevels) {
        long long sz = nodal ? (long long)(g.nx + 1) * (g.ny + 1) * (g.nz + 1) : (long long)g.nx * g.ny * g.nz;
        if (sz <= (nodal ? 125 : 64)) break;
        if ((g.nx & 1) || (g.ny & 1) || (g.nz & 1)) break;
        g.nx /= 2; g.ny /= 2; g.nz /= 2;
        g.h *= 2.0;
        g.ih *= 0.5;
        out[L++] = g;
    }
    return L;
}

template <class T>
T *dalloc(size_t n, cudaError_t &e)
{
    T *p = nullptr;
    cudaError_t r = dev_malloc((void **)&p, n * sizeof(T));
    if (r != cudaSuccess) e = r;
    return p;
}

}  // namespace

// ===========================================================================
// Set-up and public solver entry points
// ===========================================================================

ebv_status setup_solvers(Ctx *c)
{
    const GridD &g = c->g;
    cudaError_t e = cudaSuccess;
    // dynamic shared memory of the cluster kernels (per device: set for each context)
    const cudaFuncAttribute smem_max = cudaFuncAttributeMaxDynamicSharedMemorySize;
    EBV_CUDA_TRY(c, cudaFuncSetAttribute(k_cc_coarse_vcycle<float>, smem_max, kCvSmem));
    EBV_CUDA_TRY(c, cudaFuncSetAttribute(k_cc_coarse_vcycle<double>, smem_max, kCvSmem));
    EBV_CUDA_TRY(c, cudaFuncSetAttribute(k_nd_coarse<float>, smem_max, kNcSmem));
    EBV_CUDA_TRY(c, cudaFuncSetAttribute(k_nd_coarse<double>, smem_max, kNcSmem));
    EBV_CUDA_TRY(c, rb_setup(c));
    GridD gl[kMaxLevels];
    // cell-centred hierarchies (projection and viscous)
    int L = plan_levels(g, gl, false);
    long long nbc = (long long)gl[L - 1].nx * gl[L - 1].ny * gl[L - 1].nz;
    if (nbc > kBottomMax) return c->fail(EBV_ERR_INVALID, "grid cannot be coarsened to a small bottom level");
    CcHier *hs[2] = {&c->mac, &c->visc};
    // the projection operator has one variant; the viscous one a variant per
    // velocity component, whose diagonals take the box faces of its Dirichlet sides
    c->mac.nvar = 1;
    c->mac.side_mask[0] = 0x3fu;
    c->visc.nvar = 3;
    for (int q = 0; q < 3; q++) {
        unsigned m = 0;
        double val;
        for (int sd = 0; sd < 6; sd++)
            if (side_dirichlet(g, sd, q, &val)) m |= 1u << sd;
        c->visc.side_mask[q] = m;
    }
    for (CcHier *H : hs) {
        H->L = L;
        H->nb = (int)nbc;
        for (int l = 0; l < L; l++) {
            CcLevel &Lv = H->lv[l];
            Lv.g = gl[l];
            size_t nc = ncell(gl[l]);
            Lv.extra_d = dalloc<double>(nc, e);
            Lv.extra_f = dalloc<float>(nc, e);
            for (int q = 0; q < H->nvar; q++) {
                H->vdiag_d[q][l] = dalloc<double>(nc, e);
                const size_t np = (nc + 31) / 32 * 32;   // (keeps dinv_f 128-byte aligned)
                H->vdiag_f[q][l] = dalloc<float>(2 * np, e);
                H->vdinv_f[q][l] = H->vdiag_f[q][l] ? H->vdiag_f[q][l] + np : nullptr;
                if (l == 0) H->vdiag_a[q] = dalloc<float>(nc, e);
            }
            for (int d = 0; d < 3; d++) {
                Lv.bf_d[d] = dalloc<double>(nface(gl[l], d), e);
                Lv.bf_f[d] = dalloc<float>(nface(gl[l], d), e);
                Lv.bf_h[d] = dalloc<__nv_bfloat16>(nface(gl[l], d), e);
            }
            if (rb_fusable(gl[l]))
                Lv.bxp = dalloc<RbF>((size_t)2 * rb_hxp(gl[l].nx) * gl[l].ny * gl[l].nz, e);
            if (H == &c->mac) Lv.cov = dalloc<uint8_t>(nc, e);
            else Lv.cov = c->mac.lv[l].cov;
        }
        for (int q = 0; q < H->nvar; q++) H->vbinv[q] = dalloc<double>((size_t)nbc * nbc, e);
        H->bmat = dalloc<double>((size_t)H->nvar * gj_scratch((int)nbc), e);
        select_variant(*H, 0);
    }
    // nodal hierarchy
    GridD gn[kMaxLevels];
    int Ln = plan_levels(g, gn, true);
    long long nbn = (long long)(gn[Ln - 1].nx + 1) * (gn[Ln - 1].ny + 1) * (gn[Ln - 1].nz + 1);
    if (nbn > kBottomMax) return c->fail(EBV_ERR_INVALID, "grid cannot be coarsened to a small nodal bottom");
    c->nd.L = Ln;
    c->nd.nb = (int)nbn;
    for (int l = 0; l < Ln; l++) {
        NdLevel &Lv = c->nd.lv[l];
        Lv.g = gn[l];
        size_t nc = ncell(gn[l]);
        Lv.alpha_d = l ? dalloc<double>(nc, e) : c->alpha;
        Lv.alpha_f = dalloc<float>(nc, e);
        Lv.act = dalloc<uint8_t>(nnode(gn[l]), e);
        // the plane march: the finest level, and the coarse ones large enough
        // that it is the faster form
        Lv.march = l == 0 || nnode(gn[l]) >= kKindNodes;
        Lv.kind = dalloc<uint8_t>(nnode(gn[l]), e);
        Lv.lam_max = 2.0;
    }
    c->nd.binv = dalloc<double>((size_t)nbn * nbn, e);
    c->nd.bmat = dalloc<double>(gj_scratch((int)nbn), e);
    // level vectors: large enough for nodes of that level (>= cells)
    int Lmax = std::max(L, Ln);
    for (int l = 0; l < Lmax; l++) {
        const GridD &gg = l < Ln ? gn[l] : gl[l];
        size_t m = (size_t)nnode(gg);
        c->lx[l] = dalloc<double>(m, e);
        c->lb[l] = dalloc<double>(m, e);
        c->lr[l] = dalloc<double>(m, e);
        c->ld[l] = dalloc<double>(m, e);
        c->lt[l] = dalloc<double>(m, e);
    }
    if (e != cudaSuccess)
        return c->fail(e == cudaErrorMemoryAllocation ? EBV_ERR_OOM : EBV_ERR_CUDA,
                       std::string("allocation: ") + cudaGetErrorString(e));
    return EBV_OK;
}

// Geometry-dependent solver data: projection coefficients, coverage, nodal
// volume fractions and active nodes, both bottom inverses.
ebv_status autotune_shapes(Ctx *c);

ebv_status setup_geometry_solvers(Ctx *c)
{
    const GridD &g = c->g;
    // coverage per level
    EBV_LAUNCH(c, k_cov_from_flag, dim3(vblocks(ncell(g))), dim3(256), 0, ncell(g), c->flag, c->mac.lv[0].cov);
    for (int l = 0; l + 1 < c->mac.L; l++)
        EBV_LAUNCH(c, k_cov_coarsen, cgrid(c->mac.lv[l + 1].g), block3(), 0, c->mac.lv[l].g, c->mac.lv[l].cov,
                   c->mac.lv[l + 1].g, c->mac.lv[l + 1].cov);
    // projection operator
    CcLevel &M0 = c->mac.lv[0];
    EBV_LAUNCH(c, k_mac_coeffs, grid3(g.nx + 1, g.ny + 1, g.nz + 1), block3(), 0, g, c->flag, c->ax, c->ay, c->az,
               M0.extra_d, M0.bf_d[0], M0.bf_d[1], M0.bf_d[2]);
    // its levels and bottom inverse in the precision the solves use (the two
    // share the blocks of the inverse diagonals, and the inverse)
    ebv_status s = cc_finish_hierarchy(c, c->mac, c->prm.precision != EBV_FP64);
    if (s != EBV_OK) return s;
    // nodal
    NdHier &N = c->nd;
    for (int l = 0; l < N.L; l++) {
        NdLevel &Lv = N.lv[l];
        if (l) EBV_LAUNCH(c, k_nd_alpha_coarsen, cgrid(Lv.g), block3(), 0, N.lv[l - 1].g, N.lv[l - 1].alpha_d, Lv.g,
                          Lv.alpha_d);
        int nc = ncell(Lv.g);
        EBV_LAUNCH(c, (k_convert<double, float>), dim3(vblocks(nc)), dim3(256), 0, Lv.alpha_d, Lv.alpha_f, nc);
        EBV_LAUNCH(c, k_nd_active, ngrid(Lv.g), block3(), 0, Lv.g, Lv.alpha_d, Lv.act);
        EBV_LAUNCH(c, k_nd_kind, ngrid(Lv.g), block3(), 0, Lv.g, Lv.alpha_d, Lv.act, Lv.kind);
    }
    for (int l = 0; l < N.L; l++) {
        // levels that march: the nodes that take the general row, in
        // ascending order -- the box faces, and inside the active nodes that
        // are not regular
        NdLevel &Lv = N.lv[l];
        if (!Lv.march) continue;
        const GridD &gl = Lv.g;
        const int nn = nnode(gl);
        std::vector<uint8_t> kind(nn);
        EBV_CUDA_TRY(c, cudaMemcpyAsync(kind.data(), Lv.kind, nn, cudaMemcpyDeviceToHost, c->stream));
        EBV_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        std::vector<int> irr;
        for (int k = 0, n = 0; k <= gl.nz; k++)
            for (int j = 0; j <= gl.ny; j++) {
                const bool row = k == 0 || k == gl.nz || j == 0 || j == gl.ny;
                for (int i = 0; i <= gl.nx; i++, n++)
                    if (row || i == 0 || i == gl.nx || kind[n] == ND_IRR) irr.push_back(n);
            }
        if (Lv.irr) cudaFree(Lv.irr);
        Lv.irr = nullptr;
        Lv.nirr = (int)irr.size();
        if (Lv.nirr) {
            EBV_CUDA_TRY(c, dev_malloc((void **)&Lv.irr, irr.size() * sizeof(int)));
            EBV_CUDA_TRY(c, cudaMemcpy(Lv.irr, irr.data(), irr.size() * sizeof(int), cudaMemcpyHostToDevice));
        }
    }
    const NdLevel &B = N.lv[N.L - 1];
    EBV_LAUNCH(c, k_nd_bottom_assemble, dim3(gj_pad(N.nb)), dim3(128), 0, B.g, B.alpha_d, B.act, N.bmat, N.nb);
    bottom_invert(c, N.bmat, N.nb, 1, &N.binv);
    EBV_CUDA_TRY(c, cudaGetLastError());
    if (c->prm.precision != EBV_FP64) carve_components<float>(c);
    else carve_components<double>(c);
    return autotune_shapes(c);
}

// Launch-shape autotuner.  For every level that launches them it times each
// candidate block shape of the colour pass (on the projection operator) and of
// the node-by-node Chebyshev step, on zeroed scratch vectors in the precision
// the solves use, and keeps the fastest; the viscous hierarchy shares the shapes of the
// projection hierarchy (same level sizes).  The smoothers' results do not
// depend on the shape: every update of a pass reads only values that the
// pass does not write (the one pass that also sums r.z keeps the default
// shape, so its partial sums are grouped the same way).
template <class T>
ebv_status autotune_shapes_t(Ctx *c)
{
    static const dim3 cand[] = {dim3(32, 4, 2), dim3(32, 8, 1), dim3(32, 2, 4), dim3(16, 8, 2),
                                dim3(64, 4, 1), dim3(64, 2, 2), dim3(16, 16, 1), dim3(128, 2, 1)};
    const int nc = (int)(sizeof(cand) / sizeof(cand[0]));
    T *x = (T *)(sizeof(T) == 4 ? (void *)c->kz32 : (void *)c->kz);
    T *y = (T *)(sizeof(T) == 4 ? (void *)c->kp32 : (void *)c->kp);
    T *d = (T *)(sizeof(T) == 4 ? (void *)c->kq32 : (void *)c->kq);
    T *b = (T *)(sizeof(T) == 4 ? (void *)c->kr32 : (void *)c->kr);
    for (T *v : {x, y, d, b}) EBV_CUDA_TRY(c, cudaMemsetAsync(v, 0, c->vec_len * sizeof(T), c->stream));
    cudaEvent_t e0, e1;
    EBV_CUDA_TRY(c, cudaEventCreate(&e0));
    EBV_CUDA_TRY(c, cudaEventCreate(&e1));
    auto time_it = [&](auto launch) -> float {
        launch();
        cudaEventRecord(e0, c->stream);
        for (int r = 0; r < 4; r++) launch();
        cudaEventRecord(e1, c->stream);
        float ms = 1e30f;
        if (cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    // (levels inside a cluster kernel launch neither; of these the ones that the
    // fused sweep applies to are timed all the same, for ebv_sweep_timing)
    CoarseVC<T> D;
    const int lc = cv_plan<T>(c->mac, D), cl0 = lc < 0 ? c->mac.L - 1 : lc;
    for (int l = 0; l < c->mac.L; l++) {
        CcLevel &L = c->mac.lv[l];
        if (l >= cl0 && !(sizeof(T) == 4 && rb_fusable(L.g) && gs4_ok(L.g))) continue;
        const VOp3<T> A = vop3<T>(c->mac, l, 1);
        const V3<T> xv = one(x);
        const V3<const T> bv = one<const T>(b), dv = one<const T>(d);
        float best = 1e30f;
        for (int q = 0; q < nc; q++) {
            const dim3 bk = cand[q], gr = gs_grid(L.g, bk);
            float ms = time_it([&]() {
                k_cc_gs<T, false><<<gr, bk, 0, c->stream>>>(A, xv, bv, gr.z, nullptr, 0, 0, V3<const T>(), GridD());
            });
            if (ms < best) { best = ms; L.gs_blk = bk; }
        }
        c->visc.lv[l].gs_blk = L.gs_blk;
        if constexpr (sizeof(T) == 4) {
            // the vectorised pass: a thread covers 4 cells of a half-row, so
            // narrow blocks suit the levels whose rows are short
            static const dim3 c4[] = {dim3(32, 4, 2), dim3(32, 8, 1), dim3(16, 8, 2), dim3(16, 16, 1),
                                      dim3(8, 16, 2), dim3(8, 32, 1), dim3(4, 32, 2), dim3(4, 16, 4)};
            if (gs4_ok(L.g)) {
                float best4 = 1e30f;
                for (int pz = 1; pz <= 2; pz++)
                    for (const dim3 &bk : c4) {
                        if (bk.x > 2 * (unsigned)((L.g.nx >> 3) + 1)) continue;   // no block wider than twice a row
                        float ms = time_it([&]() { launch_gs4(c->stream, bk, pz, A, xv, bv, 0, 0); });
                        if (ms < best4) { best4 = ms; L.gs4_blk = bk; L.gs4_pz = pz; }
                    }
                c->visc.lv[l].gs4_blk = L.gs4_blk;
                c->visc.lv[l].gs4_pz = L.gs4_pz;
            }
            // the fused one-pass sweep against its two colour passes (same
            // results), per kind of sweep: the faster serves it in switch mode 1
            RbMaps m;
            for (int q = 0; q < 4; q++) L.rb_ms[q][0] = 1e30f, L.rb_ms[q][1] = 0.f;
            if (!c->batched && rb_fusable(L.g) && gs4_ok(L.g) && rb_map(c, x, 0, L.g, &m.v[0].x) &&
                rb_map(c, b, 1, L.g, &m.v[0].b) && rb_map(c, A.dinv[0], 1, L.g, &m.v[0].d) &&
                rb_map(c, L.bxp, 4, L.g, &m.fx) && rb_map(c, A.A.by, 2, L.g, &m.fy) &&
                rb_map(c, A.A.bz, 3, L.g, &m.fz)) {
                const long long nl = c->launches;
                // planes per block: the model's choice, the most planes that
                // still fill one wave, and half that (results do not depend on it)
                const int nt = rb_ntiles(L.g), res = c->rb_res, nz = L.g.nz;
                const int wave = std::max(1, res / std::max(1, nt));   // chunks per wave
                const int kzc[3] = {rb_kz(c, L.g), (nz + wave - 1) / wave, (nz + 2 * wave - 1) / (2 * wave)};
                float best = 1e30f;
                for (int kz : kzc) {
                    const float ms = time_it(
                        [&]() { rb_launch(c, "autotune", L.g, m, one(y), 0, RB_PLAIN, nullptr, kz); });
                    if (ms < best) { best = ms; L.rb_kz = kz; }
                }
                // the correction sweep reads a coarse array: a zeroed vector with the next level's dims
                const bool has_c = l + 1 < c->mac.L;
                const GridD gc = has_c ? c->mac.lv[l + 1].g : GridD();
                const dim3 gt((L.g.nx / 2 + RB_HW - 1) / RB_HW, (L.g.ny + RB_TY - 1) / RB_TY,
                              (L.g.nz + kGs2Planes - 1) / kGs2Planes);
                const dim3 bk = L.gs_blk, grc = gs_grid(L.g, bk);
                for (int kind = 0; kind < 4; kind++) {
                    if (kind == RB_CORR && !has_c) continue;   // (no correction sweep on the last level)
                    RbMaps mk = m;
                    mk.v[0].xc = m.v[0].b;
                    if (kind == RB_CORR && !rb_map(c, d, 5, gc, &mk.v[0].xc)) continue;
                    const float ms_f = time_it([&]() {
                        rb_launch(c, "autotune", L.g, mk, one(y), 0, kind, kind == RB_DOT ? c->part : nullptr, L.rb_kz);
                    });
                    const float ms_p = time_it([&]() {
                        if (kind == RB_CORR) {
                            const dim3 g4 = gs4_grid(L.g, L.gs4_blk, L.gs4_pz);
                            if (L.gs4_pz == 1)
                                k_cc_gs4<1, true><<<g4, L.gs4_blk, 0, c->stream>>>(A, xv, bv, g4.z, nullptr, 0, 0, dv, gc);
                            else
                                k_cc_gs4<2, true><<<g4, L.gs4_blk, 0, c->stream>>>(A, xv, bv, g4.z, nullptr, 0, 0, dv, gc);
                        }
                        else
                            launch_gs4(c->stream, L.gs4_blk, L.gs4_pz, A, xv, bv, 0, kind == RB_ZERO ? 1 : 0);
                        if (kind == RB_DOT)
                            k_cc_gs2_dot<<<gt, RB_THREADS, 0, c->stream>>>(A, xv, bv, gt.z, nullptr, 1, c->part);
                        else launch_gs4(c->stream, L.gs4_blk, L.gs4_pz, A, xv, bv, 1, 0);
                    });
                    L.rb_ms[kind][0] = ms_f;
                    L.rb_ms[kind][1] = ms_p;
                }
                c->launches = nl;
            }
            for (int q = 0; q < 4; q++) c->visc.lv[l].rb_ms[q][0] = L.rb_ms[q][0], c->visc.lv[l].rb_ms[q][1] = L.rb_ms[q][1];
            c->visc.lv[l].rb_kz = L.rb_kz;
        }
    }
    ChebCoef k = cheb_coef(2.0);
    NdCoarse<T> DN;
    const int ln = nc_plan<T>(c->nd, DN), nl0 = ln < 0 ? c->nd.L - 1 : ln;
    for (int l = 0; l < nl0; l++) {
        NdLevel &L = c->nd.lv[l];
        if (L.march) continue;   // (takes k_nd_pass)
        NdOp<T> A = ndop<T>(L);
        float best = 1e30f;
        for (int q = 0; q < nc; q++) {
            const dim3 bk = cand[q], gr = ch_grid(L.g, bk);
            float ms = time_it([&]() {
                k_nd_cheb<T><<<gr, bk, 0, c->stream>>>(A, x, y, d, b, (T)k.cd[1], (T)k.cr[1]);
            });
            if (ms < best) { best = ms; L.ch_blk = bk; }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    EBV_CUDA_TRY(c, cudaGetLastError());
    return EBV_OK;
}

ebv_status autotune_shapes(Ctx *c)
{
    return c->prm.precision != EBV_FP64 ? autotune_shapes_t<float>(c) : autotune_shapes_t<double>(c);
}

ebv_status mac_solve(Ctx *c, const double *b, double *x, int *iters, double *res)
{
    CcProblem P;
    P.H = &c->mac;
    EBV_LAUNCH(c, k_fill, dim3(vblocks(ncell(c->g))), dim3(256), 0, x, ncell(c->g), 0.0);
    return solve(c, P, one<const double>(b), one(x), iters, res, true);
}

ebv_status visc_build(Ctx *c, const double *eta)
{
    const GridD &g = c->g;
    CcLevel &V0 = c->visc.lv[0];
    EBV_LAUNCH(c, k_visc_coeffs, grid3(g.nx + 1, g.ny + 1, g.nz + 1), block3(), 0, g, geomd(c), paramsd(c->prm), eta,
               c->dt_dev, V0.extra_d, V0.bf_d[0], V0.bf_d[1], V0.bf_d[2]);
    return cc_finish_hierarchy(c, c->visc, c->prm.precision != EBV_FP64);
}

namespace {
// The three viscous systems with right-hand sides b (3 x cells): together where
// the other components' vectors and partial sums fit (c->joint), else one
// after another.
ebv_status visc_solve_all(Ctx *c, const double *b, double *x, int *iters, double *res, bool x_zero)
{
    const int N3 = ncell(c->g), slot = c->cur_slot;
    CcProblem P;
    P.H = &c->visc;
    if (c->joint) {
        P.nc = kMaxComp;
        return solve(c, P, V3<const double>(b, b + N3, b + 2 * (size_t)N3), V3<double>(x, x + N3, x + 2 * (size_t)N3),
                     iters, res, x_zero);
    }
    for (int q = 0; q < kMaxComp; q++) {
        select_variant(c->visc, q);
        c->cur_slot = slot + q;
        ebv_status st = solve(c, P, one<const double>(b + q * (size_t)N3), one(x + q * (size_t)N3),
                              iters ? iters + q : nullptr, res ? res + q : nullptr, x_zero);
        if (st != EBV_OK) return st;
    }
    return EBV_OK;
}
}  // namespace

ebv_status visc_solve(Ctx *c, const double *psi, double *x, int *iters, double *res)
{
    const GridD &g = c->g;
    CcLevel &V0 = c->visc.lv[0];
    // (c->DC: scratch of the explicit terms, 3 x cells)
    EBV_LAUNCH(c, k_visc_rhs, cgrid(g), block3(), 0, g, geomd(c), psi, V0.bf_d[0], V0.bf_d[1], V0.bf_d[2], c->DC);
    return visc_solve_all(c, c->DC, x, iters, res, false);
}

ebv_status visc_solve_rhs(Ctx *c, const double *rhs, double *x, int *iters, double *res)
{
    const int n = 3 * ncell(c->g);
    EBV_LAUNCH(c, k_fill, dim3(vblocks(n)), dim3(256), 0, x, n, 0.0);
    return visc_solve_all(c, rhs, x, iters, res, true);
}

ebv_status nodal_solve(Ctx *c, const double *b, double *x, int *iters, double *res)
{
    const int nn = nnode(c->g);
    EBV_LAUNCH(c, k_zero_inactive, dim3(vblocks(nn)), dim3(256), 0, nn, c->nd.lv[0].act, x);
    NdProblem P;
    P.H = &c->nd;
    return solve(c, P, one<const double>(b), one(x), iters, res);
}


// ---- process-wide switches and the TMA encoder --------------------------
namespace {
long long g_spin = kSpinDefault;
int g_fused = 1;
double g_inner_drop = kInnerDropDefault;
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
}  // namespace
long long spin_limit() { return g_spin; }
int fused_sweep_mode() { return g_fused; }
void set_spin_limit(long long cycles) { g_spin = cycles < 0 ? kSpinDefault : cycles; }
void set_fused_sweep(int mode) { g_fused = mode < 0 ? 0 : (mode > 2 ? 2 : mode); }
double refine_inner_drop() { return g_inner_drop; }
void set_inner_drop(double drop) { g_inner_drop = (drop > 0.0 && drop < 1.0) ? drop : kInnerDropDefault; }

bool tma_encode_4d(CUtensorMap *tm, CUtensorMapDataType type, void *base, const uint64_t dims[4],
                   const uint64_t strides[3], const uint32_t box[4])
{
    // (one entry point per process, found by whichever thread comes first; the
    // others wait for it)
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess && f)
            return reinterpret_cast<EncodeTiledFn>(f);
        cudaGetLastError();
        return nullptr;
    }();
    if (!fn || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
    const cuuint64_t d[4] = {dims[0], dims[1], dims[2], dims[3]};
    const cuuint64_t st[3] = {strides[0], strides[1], strides[2]};
    const cuuint32_t bx[4] = {box[0], box[1], box[2], box[3]};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    return fn(tm, type, 4, base, d, st, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace ebv
