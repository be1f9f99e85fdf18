// RBF-FD sub-domain solver (Sec. 3.2 of arXiv:1603.09311): once the
// interface values are known, a sub-domain is solved on its own nodes with
// radial-basis-function finite differences.
//
// At node x_0 with stencil x_1 .. x_n (the node and its n - 1 nearest
// neighbours), the weights of an operator L solve A w = b with
// A_ij = phi(|x_i - x_j|) and b_j = L phi(|x - x_j|) at x_0, for the
// multiquadric phi(r) = sqrt(1 + (eps r)^2).  The operator is the Laplacian
// (the sum of the paper's d^2/dx^2 and d^2/dz^2 matrices; the weights are
// linear in b): Lap phi = (2 eps^2 + eps^4 r^2) / phi^3 in two dimensions.
// Every unknown node i gets the equation
//     sum_{j in stencil(i)} w_ij u_j - i kappa_i u_i = 0,
// the Dirichlet nodes' terms moved to the right-hand side, and the sparse
// complex system is solved by BiCGStab with a Jacobi preconditioner.
//
// Kernels (FP64, this unit compiled without FMA contraction so that the
// squared distances of the neighbour search round as in plain arithmetic):
//   cell_*, knn_kernel  each node's nearest nodes by (squared distance,
//                    index): nodes binned into a cell grid, one thread per
//                    node scanning rings of cells
//   weights_kernel   one thread per node: the n x n multiquadric system,
//                    Gaussian elimination with partial pivoting
//   assemble_kernel  one thread per unknown: the row (ELL, n slots, column
//                    -1 for a Dirichlet neighbour), the diagonal and the
//                    right-hand side
//   bicgstab_kernel  the iterations, a few hundred in one cooperative launch:
//                    element-wise updates, ELL matrix-vector products and dot
//                    products between grid barriers
#include <algorithm>
#include <cmath>
#include <condition_variable>
#include <cstdint>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "sdd.h"
#include "sdd_internal.cuh"

namespace sdd {
namespace {

constexpr int kMaxStencil = 16;
constexpr int kDotThreads = 256;
constexpr int kDotBlocks = 1024;

struct Z {
    double re, im;
};
__device__ __forceinline__ Z zadd(Z a, Z b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Z zsub(Z a, Z b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ Z zmul(Z a, Z b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ Z zdiv(Z a, Z b) {
    const double d = b.re * b.re + b.im * b.im;
    return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
// conj(a) b
__device__ __forceinline__ Z zcdot(Z a, Z b) { return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re}; }

__device__ __forceinline__ double mq(double r2, double eps) { return sqrt(1.0 + eps * eps * r2); }

// Nearest-neighbour search on a grid of square cells of side c over the
// nodes' bounding box: nodes are binned (count, scan, fill), then each node
// scans rings of cells around its own (ring R: Chebyshev cell distance R).
// Every node in ring R + 1 or beyond is at least R c away, so the search
// stops after ring R once the list is full and (R c)^2 exceeds its last
// squared distance (with a relative margin of 1e-9 for the binning's
// rounding).  The order is (squared distance, index), as a scan of all nodes
// gives.
struct CellGrid {
    double x0, z0, c;
    int gx, gz;
};

__device__ __forceinline__ int cell_x(const CellGrid &g, double x) {
    return min(max((int)floor((x - g.x0) / g.c), 0), g.gx - 1);
}
__device__ __forceinline__ int cell_z(const CellGrid &g, double z) {
    return min(max((int)floor((z - g.z0) / g.c), 0), g.gz - 1);
}

__global__ void cell_count_kernel(const double *p, int n, CellGrid g, int32_t *cell, int32_t *count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int id = cell_z(g, p[2 * i + 1]) * g.gx + cell_x(g, p[2 * i]);
    cell[i] = id;
    atomicAdd(&count[id], 1);
}

// start[0 .. m] = exclusive prefix sums of count[0 .. m-1] (one CTA).
__global__ void __launch_bounds__(1024) cell_scan_kernel(const int32_t *count, int m, int32_t *start) {
    __shared__ int32_t part[1024];
    const int t = threadIdx.x;
    const int per = (m + 1023) / 1024;
    const int a = min(t * per, m), b = min(a + per, m);
    int32_t acc = 0;
    for (int k = a; k < b; ++k) acc += count[k];
    part[t] = acc;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const int32_t v = t >= off ? part[t - off] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int32_t run = t > 0 ? part[t - 1] : 0;
    for (int k = a; k < b; ++k) {
        start[k] = run;
        run += count[k];
    }
    if (t == 1023) start[m] = part[1023];
}

__global__ void cell_fill_kernel(const int32_t *cell, int n, int32_t *cursor, int32_t *list) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    list[atomicAdd(&cursor[cell[i]], 1)] = i;
}

__device__ __forceinline__ bool before(double d2, int j, double bd, int bj) {
    return d2 < bd || (d2 == bd && j < bj);
}

__global__ void knn_kernel(const double *p, int n, int ns, CellGrid g, const int32_t *start,
                           const int32_t *list, int32_t *st) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double bd[kMaxStencil];
    int bi[kMaxStencil];
    int cnt = 0;
    const double xi = p[2 * i], zi = p[2 * i + 1];
    const int cx = cell_x(g, xi), cz = cell_z(g, zi);
    const int rmax = max(g.gx, g.gz);
    for (int R = 0; R <= rmax; ++R) {
        for (int dz = -R; dz <= R; ++dz) {
            const int iz = cz + dz;
            if (iz < 0 || iz >= g.gz) continue;
            const int step = (dz == -R || dz == R) ? 1 : 2 * R;
            for (int dx = -R; dx <= R; dx += (step > 0 ? step : 1)) {
                const int ix = cx + dx;
                if (ix < 0 || ix >= g.gx) continue;
                const int id = iz * g.gx + ix;
                for (int q = start[id]; q < start[id + 1]; ++q) {
                    const int j = list[q];
                    const double ddx = p[2 * j] - xi, ddz = p[2 * j + 1] - zi;
                    const double d2 = ddx * ddx + ddz * ddz;
                    if (cnt == ns && !before(d2, j, bd[ns - 1], bi[ns - 1])) continue;
                    int k = cnt < ns ? cnt++ : ns - 1;
                    while (k > 0 && before(d2, j, bd[k - 1], bi[k - 1])) {
                        bd[k] = bd[k - 1];
                        bi[k] = bi[k - 1];
                        --k;
                    }
                    bd[k] = d2;
                    bi[k] = j;
                }
            }
        }
        if (cnt == ns) {
            const double rc = R * g.c;
            if (rc * rc * (1.0 - 1e-9) > bd[ns - 1]) break;
        }
    }
    for (int k = 0; k < ns; ++k) st[(size_t)i * ns + k] = bi[k];
}

// Weights of node i, w[i][k] for stencil entry k.  *err = 1 on a zero pivot
// (coincident nodes).
__global__ void weights_kernel(const double *p, int n, const int32_t *st, int ns, double eps,
                               double *w, int *err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double A[kMaxStencil][kMaxStencil + 1];
    const double self = mq(0.0, eps);
    const double xi = p[2 * i], zi = p[2 * i + 1];
    for (int a = 0; a < ns; ++a) {
        const int ja = st[(size_t)i * ns + a];
        const double xa = p[2 * ja], za = p[2 * ja + 1];
        // the distance is the same both ways
        for (int b = 0; b < a; ++b) {
            const int jb = st[(size_t)i * ns + b];
            const double r = hypot(xa - p[2 * jb], za - p[2 * jb + 1]);
            A[a][b] = A[b][a] = mq(r * r, eps);
        }
        A[a][a] = self;
        const double r = hypot(xa - xi, za - zi);
        const double ph = mq(r * r, eps);
        A[a][ns] = (2.0 * eps * eps + eps * eps * eps * eps * r * r) / (ph * ph * ph);
    }
    for (int c = 0; c < ns; ++c) {
        int piv = c;
        double best = fabs(A[c][c]);
        for (int r = c + 1; r < ns; ++r)
            if (fabs(A[r][c]) > best) {
                best = fabs(A[r][c]);
                piv = r;
            }
        if (!(best > 0.0)) {
            atomicExch(err, 1);
            return;
        }
        if (piv != c)
            for (int k = c; k <= ns; ++k) {
                const double t = A[c][k];
                A[c][k] = A[piv][k];
                A[piv][k] = t;
            }
        for (int r = c + 1; r < ns; ++r) {
            const double f = A[r][c] / A[c][c];
            for (int k = c; k <= ns; ++k) A[r][k] -= f * A[c][k];
        }
    }
    for (int c = ns - 1; c >= 0; --c) {
        double s = A[c][ns];
        for (int k = c + 1; k < ns; ++k) s -= A[c][k] * A[k][ns];
        A[c][ns] = s / A[c][c];
    }
    for (int k = 0; k < ns; ++k) w[(size_t)i * ns + k] = A[k][ns];
}

// Row r (node unk[r]): ELL slots k-major (ew[k nu + r], ecol[k nu + r]),
// the reciprocal of the diagonal d = w_ii - i kappa_i (the Jacobi
// preconditioner), right-hand side -sum_{Dirichlet j} w_ij u_j.
__global__ void assemble_kernel(const int32_t *unk, const int32_t *pos, int nu, const int32_t *st,
                                const double *w, int ns, const double *kappa, const double *vals,
                                double *ew, int32_t *ecol, Z *dinv, Z *rhs) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nu) return;
    const int i = unk[r];
    Z b = {0.0, 0.0};
    double wii = 0.0;
    for (int k = 0; k < ns; ++k) {
        const int j = st[(size_t)i * ns + k];
        const double wij = w[(size_t)i * ns + k];
        const int c = pos[j];
        ew[(size_t)k * nu + r] = wij;
        ecol[(size_t)k * nu + r] = c;
        if (c < 0) {
            b.re -= wij * vals[2 * j];
            b.im -= wij * vals[2 * j + 1];
        }
        if (j == i) wii = wij;
    }
    dinv[r] = zdiv(Z{1.0, 0.0}, Z{wii, -kappa[i]});
    rhs[r] = b;
}

// y = K x: sum over the slots, minus i kappa x on the diagonal
__global__ void spmv_kernel(const double *ew, const int32_t *ecol, int nu, int ns, const int32_t *unk,
                            const double *kappa, const Z *x, Z *y) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nu) return;
    Z acc = {0.0, 0.0};
    for (int k = 0; k < ns; ++k) {
        const int c = ecol[(size_t)k * nu + r];
        if (c >= 0) {
            const double wv = ew[(size_t)k * nu + r];
            acc.re += wv * x[c].re;
            acc.im += wv * x[c].im;
        }
    }
    const double kap = kappa[unk[r]];
    // - i kappa x = kappa (x.im, -x.re)
    acc.re += kap * x[r].im;
    acc.im -= kap * x[r].re;
    y[r] = acc;
}

// Block partials of |a|^2, in the real part.
__global__ void __launch_bounds__(kDotThreads) norm_partial_kernel(const Z *a, int n, Z *part) {
    __shared__ Z sum[kDotThreads];
    Z acc = {0.0, 0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        acc = zadd(acc, zcdot(a[i], a[i]));
    sum[threadIdx.x] = acc;
    __syncthreads();
    for (int off = kDotThreads / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) sum[threadIdx.x] = zadd(sum[threadIdx.x], sum[threadIdx.x + off]);
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sum[0];
}

// Device-side BiCGStab scalars.  stop: 0 running, 1 converged, 2 breakdown,
// 3 a barrier wait ran out, 4 the first one did (nothing was done).
struct Scal {
    Z rho, alpha, omega, beta;
    double rnorm2, bnorm2, tol2;
    int iter, stop;
};

// BiCGStab as one persistent kernel.  Per iteration (dinv = 1 / d)
//   p = r + beta (p - omega v),  y = p / d                     | barrier
//   v = K y,  alpha = rho / <r^, v>                            | barrier
//   s = r - alpha v,  z = s / d                                | barrier
//   t = K z,  omega = <t, s> / <t, t>  (t = 0: s = 0, omega = 0) | barrier
//   x += alpha y + omega z,  r = s - omega t,  |r|^2 and the stop test,
//   rho' = <r^, r>,  beta = (rho' / rho)(alpha / omega)        | barrier
// The rows are cut into blocks of kDotThreads; a dot product is the pairwise
// sum of each block's rows (halving), then of the blocks.
//
// What bounds it: the FP64 pipe (150 operations a row and iteration, a warp
// instruction every 64 cycles on a quarter of an SM: 10 us with two warps on
// each) and five barriers of about 1.2 us with the sums behind three of them.
// Five launches per iteration, replayed as a graph, took 48 us at 32041 rows:
// each launch drains the chip and reads its vectors again.  Here a thread
// keeps its row's vectors in registers and its weights in shared memory; only
// y and z, which the neighbours read, and the block sums go through L2.  What
// a barrier's wait can hide is put there (alpha y, p - omega v, x, alpha /
// omega), and the scalars are formed by one warp, real and imaginary parts in
// its two halves (by every warp they took 60 of 220 operations).
//   SPLIT 2 gives a block of rows to two CTAs (the even and the odd rows, so
//   that the halving sums pair the same rows), one warp on each quarter of an
//   SM: half the FP64 time where there are at most half as many blocks as SMs.
//   KEEP false: more blocks than resident CTAs; each CTA takes several blocks
//   and the vectors stay in global memory.
struct SolveArgs {
    const double *ew;
    const int32_t *ecol, *unk;
    const double *kappa;
    const Z *dinv, *rh;
    Z *r, *p, *v, *x, *y, *z, *s, *t;
    Z *part;         // [5][blocks * SPLIT]: <r^, v>, <t, s>, <t, t>, <r^, r>, <r, r>
    Scal *S;
    unsigned *bar;   // barrier arrivals (zero before the launch)
    int nu, ns, blocks, max_iter;
};

constexpr int kStaticSmem = 256;  // at least what the solver's kernel declares
constexpr long long kBarrierCycles = 4000000000ll;  // about two seconds
constexpr unsigned kBarrierFail = 0x80000000u;
// Launches in a row whose CTAs did not all get onto the GPU (ten minutes)
// before a solve gives up.
constexpr int kTries = 300;

// Barrier of all CTAs of the (cooperative) launch, in two halves.  A wait that
// runs out sets the top bit of the counter while arrivals are missing, by
// compare-and-swap on the count read: once all have arrived nobody can fail the
// barrier any more, and until then nobody has passed it, so every CTA leaves
// this barrier with the same answer.  (Out of line: in the wait's loop it took
// 0.25 us of an iteration's 26.)
__device__ __noinline__ void give_up(unsigned *bar, unsigned v, unsigned epoch) {
    while (!(v & kBarrierFail) && v < epoch) {
        const unsigned seen = atomicCAS(bar, v, v | kBarrierFail);
        if (seen == v) return;
        v = seen;
    }
}
__device__ __forceinline__ void grid_arrive(unsigned *bar, unsigned &epoch) {
    epoch += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}
__device__ __forceinline__ bool grid_wait(unsigned *bar, unsigned epoch, int *ok) {
    if (threadIdx.x == 0) {
        const long long t0 = clock64();
        unsigned v;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((v & kBarrierFail) || v >= epoch) break;
            if (clock64() - t0 > kBarrierCycles) give_up(bar, v, epoch);
        }
        *ok = (v & kBarrierFail) == 0;
    }
    __syncthreads();
    return *ok != 0;
}

// Pairwise sum of n <= 256 complex values by one warp: value i pairs with
// i + 128, then i + 64, ... i + 1 (missing values are zeros); get(i) fetches
// value i < n.  Below 32 values the lower half of the warp adds the real parts
// and the upper half the imaginary ones.  Every lane returns the sum.
template <class F>
__device__ __forceinline__ Z halving_sum(int n, F get) {
    const int lane = threadIdx.x & 31;
    Z a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = 32 * k + lane < n ? get(32 * k + lane) : Z{0.0, 0.0};
    if (n > 128)
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = zadd(a[k], a[k + 4]);
    if (n > 64)
#pragma unroll
        for (int k = 0; k < 2; ++k) a[k] = zadd(a[k], a[k + 2]);
    if (n > 32) a[0] = zadd(a[0], a[1]);
    const bool up = lane >= 16;
    const double give = up ? a[0].re : a[0].im;
    double v = (up ? a[0].im : a[0].re) + __shfl_xor_sync(0xffffffffu, give, 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return {__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 16)};
}

// a / b and a b by a warp that holds both in every lane: the real part in its
// lower half, the imaginary part in its upper half; the operations are those
// of zdiv and zmul.
__device__ __forceinline__ Z halves(double v) {
    return {__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 16)};
}
__device__ __forceinline__ Z zdiv_warp(Z a, Z b) {
    const bool up = (threadIdx.x & 31) >= 16;
    const double d = b.re * b.re + b.im * b.im;
    const double m = (up ? a.im : a.re) * b.re, k = (up ? a.re : a.im) * b.im;
    return halves((m + (up ? -k : k)) / d);
}
__device__ __forceinline__ Z zmul_warp(Z a, Z b) {
    const bool up = (threadIdx.x & 31) >= 16;
    const double m = a.re * (up ? b.im : b.re), k = a.im * (up ? b.re : b.im);
    return halves(m + (up ? k : -k));
}

__device__ __forceinline__ Z ldcg(const Z *p) {
    const double2 v = __ldcg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ void stcg(Z *p, Z v) {
    __stcg(reinterpret_cast<double2 *>(p), make_double2(v.re, v.im));
}

// The sum over all blocks from their partials: up to 1024 blocks, four to a
// value of the halving sum.
template <int SPLIT>
__device__ __forceinline__ Z block_sums(const Z *part, int blocks) {
    auto one = [&](int b) {
        return SPLIT == 1 ? ldcg(part + b) : zadd(ldcg(part + 2 * b), ldcg(part + 2 * b + 1));
    };
    return halving_sum(blocks < 256 ? blocks : 256, [&](int i) {
        Z acc = one(i);
        for (int b = i + 256; b < blocks; b += 256) acc = zadd(acc, one(b));
        return acc;
    });
}

// One row of K times a vector x that other CTAs write (mine: its entry of this
// row): the slots, then - i kappa x on the diagonal.  w, c: the row's weights
// and columns, st apart.  The first slot is the row's own node.
__device__ __forceinline__ Z row_product(const double *w, const int32_t *c, int st, int ns, double kap, const Z *x,
                                         int row, Z mine) {
    Z acc = {0.0, 0.0};
    if (c[0] >= 0) {
        const Z q = c[0] == row ? mine : ldcg(x + c[0]);
        acc = {w[0] * q.re, w[0] * q.im};
    }
#pragma unroll 8
    for (int k = 1; k < ns; ++k) {
        const int j = c[k * st];
        if (j >= 0) {
            const double wv = w[k * st];
            const Z q = ldcg(x + j);
            acc.re += wv * q.re;
            acc.im += wv * q.im;
        }
    }
    acc.re += kap * mine.im;
    acc.im -= kap * mine.re;
    return acc;
}

template <int SPLIT, bool KEEP>
__global__ void __launch_bounds__(kDotThreads / SPLIT, 2) bicgstab_kernel(const SolveArgs A) {
    constexpr int T = kDotThreads / SPLIT;  // rows of a CTA's block (every SPLIT-th of the block)
    constexpr int W = T / 32;
    extern __shared__ __align__(16) unsigned char solve_smem[];
    const int parts = A.blocks * SPLIT, stride = gridDim.x;
    const int nb = (parts - (int)blockIdx.x + stride - 1) / stride;    // this CTA's blocks
    const int nbmax = (parts + stride - 1) / stride;
    Z(*sum)[T] = reinterpret_cast<Z(*)[T]>(solve_smem);                // [2 nbmax][T]
    double *sw = reinterpret_cast<double *>(sum + 2 * nbmax);          // KEEP: [ns][T]
    int32_t *sc = reinterpret_cast<int32_t *>(sw + (KEEP ? A.ns * T : 0));  // KEEP: [ns][T]
    __shared__ struct Shared {
        Z alpha, omega, beta, rho, aw;
        double rnorm2;
        int stop, bar_ok;
    } sh;
    static_assert(sizeof(Shared) <= kStaticSmem, "static shared memory");
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    auto block_of = [&](int i) { return (int)blockIdx.x + i * stride; };
    auto row_of = [&](int i) { return (block_of(i) / SPLIT) * kDotThreads + t * SPLIT + block_of(i) % SPLIT; };
    unsigned epoch = 0;

    const Scal S0 = *A.S;
    if (t == 0) {
        sh.alpha = S0.alpha;
        sh.omega = S0.omega;
        sh.beta = S0.beta;
        sh.rho = S0.rho;
        sh.rnorm2 = S0.rnorm2;
        sh.stop = S0.stop;
    }
    int iter = S0.iter;
    const double goal = S0.tol2 * S0.bnorm2;
    // KEEP: this thread's row; pw = p - omega v, ay = alpha y
    Z r{}, pw{}, v{}, x{}, rh{}, dinv{}, y{}, z{}, s{}, tt{}, ay{};
    double kap = 0.0;
    const int row0 = row_of(0);
    const bool own = row0 < A.nu;
    if (KEEP) {
        for (int k = 0; k < A.ns; ++k) {
            sw[k * T + t] = own ? A.ew[(size_t)k * A.nu + row0] : 0.0;
            sc[k * T + t] = own ? A.ecol[(size_t)k * A.nu + row0] : -1;
        }
        if (own) {
            r = A.r[row0];
            pw = A.p[row0];
            x = A.x[row0];
            rh = A.rh[row0];
            dinv = A.dinv[row0];
            kap = A.kappa[A.unk[row0]];
        }
    }
    // the CTA's partials of one or two dot products (two: values 2 i and
    // 2 i + 1 of sum for its block i), a warp for each
    auto put_partials = [&](bool two, int slot) {
        __syncthreads();
        const int jobs = two ? 2 * nb : nb;
        for (int j = warp; j < jobs; j += W) {
            const int i = two ? j >> 1 : j, w = two ? j & 1 : 0;
            const Z q = halving_sum(T, [&](int k) { return sum[2 * i + w][k]; });
            if (lane == 0) stcg(A.part + (size_t)(slot + w) * parts + block_of(i), q);
        }
    };
    __syncthreads();

    // all CTAs are on the GPU from here on: a wait for one that other kernels
    // keep off it ends here, before anything is changed, and the host tries again
    grid_arrive(A.bar, epoch);
    bool ok = grid_wait(A.bar, epoch, &sh.bar_ok);
    const bool came = ok;
    for (int it = 0; ok && it < A.max_iter && !sh.stop; ++it) {
        const Z beta = sh.beta;
        for (int i = 0; i < nb; ++i) {
            const int row = KEEP ? row0 : row_of(i);
            if (row >= A.nu) continue;
            if (!KEEP) { r = A.r[row]; pw = A.p[row]; dinv = A.dinv[row]; }
            pw = zadd(r, zmul(beta, pw));  // p
            y = zmul(pw, dinv);
            if (!KEEP) A.p[row] = pw;
            stcg(A.y + row, y);
        }
        grid_arrive(A.bar, epoch);
        if (!(ok = grid_wait(A.bar, epoch, &sh.bar_ok))) break;
        for (int i = 0; i < nb; ++i) {
            const int row = KEEP ? row0 : row_of(i);
            Z d = {0.0, 0.0};
            if (row < A.nu) {
                if (KEEP) v = row_product(sw + t, sc + t, T, A.ns, kap, A.y, row, y);
                else {
                    v = row_product(A.ew + row, A.ecol + row, A.nu, A.ns, A.kappa[A.unk[row]], A.y, row,
                                    ldcg(A.y + row));
                    A.v[row] = v;
                    rh = A.rh[row];
                }
                d = zcdot(rh, v);
            }
            sum[2 * i][t] = d;
        }
        put_partials(false, 0);
        grid_arrive(A.bar, epoch);
        if (!(ok = grid_wait(A.bar, epoch, &sh.bar_ok))) break;
        if (warp == 0) {
            const Z rv = block_sums<SPLIT>(A.part, A.blocks);
            const Z al = zdiv_warp(sh.rho, rv);
            if (lane == 0) {
                if (rv.re == 0.0 && rv.im == 0.0) sh.stop = 2;
                else sh.alpha = al;
            }
        }
        __syncthreads();
        if (sh.stop) break;
        const Z alpha = sh.alpha;
        for (int i = 0; i < nb; ++i) {
            const int row = KEEP ? row0 : row_of(i);
            if (row >= A.nu) continue;
            if (!KEEP) { r = A.r[row]; v = A.v[row]; dinv = A.dinv[row]; }
            s = zsub(r, zmul(alpha, v));
            z = zmul(s, dinv);
            if (!KEEP) A.s[row] = s;
            stcg(A.z + row, z);
        }
        grid_arrive(A.bar, epoch);
        if (KEEP) ay = zmul(alpha, y);
        if (!(ok = grid_wait(A.bar, epoch, &sh.bar_ok))) break;
        for (int i = 0; i < nb; ++i) {
            const int row = KEEP ? row0 : row_of(i);
            Z d = {0.0, 0.0}, e = {0.0, 0.0};
            if (row < A.nu) {
                if (KEEP) tt = row_product(sw + t, sc + t, T, A.ns, kap, A.z, row, z);
                else {
                    tt = row_product(A.ew + row, A.ecol + row, A.nu, A.ns, A.kappa[A.unk[row]], A.z, row,
                                     ldcg(A.z + row));
                    A.t[row] = tt;
                    s = A.s[row];
                }
                d = zcdot(tt, s);
                e.re = tt.re * tt.re + tt.im * tt.im;  // <t, t> is real
            }
            sum[2 * i][t] = d;
            sum[2 * i + 1][t] = e;
        }
        put_partials(true, 1);
        grid_arrive(A.bar, epoch);
        if (!(ok = grid_wait(A.bar, epoch, &sh.bar_ok))) break;
        if (warp < 2) {
            const Z q = block_sums<SPLIT>(A.part + (size_t)(1 + warp) * parts, A.blocks);
            if (warp == 1 && lane == 0) sh.aw = q;
            // warp 0 goes on once warp 1 has <t, t>
            asm volatile("bar.sync 1, 64;" ::: "memory");
            if (warp == 0) {
                const Z stt = sh.aw;
                const Z om = zdiv_warp(q, stt);
                if (lane == 0) sh.omega = stt.re == 0.0 ? Z{0.0, 0.0} : om;
            }
        }
        __syncthreads();
        const Z omega = sh.omega;
        for (int i = 0; i < nb; ++i) {
            const int row = KEEP ? row0 : row_of(i);
            Z d = {0.0, 0.0}, e = {0.0, 0.0};
            if (row < A.nu) {
                if (!KEEP) { s = A.s[row]; tt = A.t[row]; rh = A.rh[row]; }
                r = zsub(s, zmul(omega, tt));
                if (!KEEP) A.r[row] = r;
                e.re = r.re * r.re + r.im * r.im;
                d = zcdot(rh, r);
            }
            sum[2 * i][t] = d;
            sum[2 * i + 1][t] = e;
        }
        put_partials(true, 3);
        grid_arrive(A.bar, epoch);
        for (int i = 0; i < nb; ++i) {
            const int row = KEEP ? row0 : row_of(i);
            if (row >= A.nu) continue;
            if (!KEEP) {
                x = A.x[row]; pw = A.p[row]; v = A.v[row];
                ay = zmul(alpha, ldcg(A.y + row));
                z = ldcg(A.z + row);
            }
            x = zadd(x, zadd(ay, zmul(omega, z)));
            pw = zsub(pw, zmul(omega, v));
            if (!KEEP) { A.x[row] = x; A.p[row] = pw; }
        }
        if (warp == 2) {
            const Z aw = zdiv_warp(alpha, omega);
            if (lane == 0) sh.aw = aw;
        }
        if (!(ok = grid_wait(A.bar, epoch, &sh.bar_ok))) break;
        ++iter;
        if (warp < 2) {
            const Z q = block_sums<SPLIT>(A.part + (size_t)(3 + warp) * parts, A.blocks);
            if (warp == 1) {
                if (lane == 0) sh.rnorm2 = q.re;
            } else {
                const Z be = zmul_warp(zdiv_warp(q, sh.rho), sh.aw);
                __syncwarp();
                if (lane == 0) {
                    sh.beta = be;
                    sh.rho = q;
                }
            }
        }
        __syncthreads();
        const double rn = sh.rnorm2;
        const Z rho = sh.rho;
        const int stop = rn <= goal ? 1
                         : (omega.re == 0.0 && omega.im == 0.0) || (rho.re == 0.0 && rho.im == 0.0) ? 2 : 0;
        if (stop) {
            __syncthreads();
            if (t == 0) sh.stop = stop;
            break;
        }
    }
    __syncthreads();
    if (KEEP && own) {
        A.r[row0] = r;
        A.p[row0] = pw;
        A.x[row0] = x;
    }
    if (blockIdx.x == 0 && t == 0) {
        Scal S = S0;
        S.alpha = sh.alpha;
        S.omega = sh.omega;
        S.beta = sh.beta;
        S.rho = sh.rho;
        S.rnorm2 = sh.rnorm2;
        S.iter = iter;
        S.stop = ok ? sh.stop : came ? 3 : 4;
        *A.S = S;
    }
}

__global__ void scatter_u_kernel(const int32_t *unk, int nu, const Z *x, double *u) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nu) return;
    u[2 * unk[r]] = x[r].re;
    u[2 * unk[r] + 1] = x[r].im;
}

__global__ void residual_kernel(const Z *Kx, const Z *b, int n, Z *res) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) res[i] = zsub(b[i], Kx[i]);
}

sdd_status rb_arg(const char *msg) { return (sdd_status)report_error(SDD_E_ARG, msg); }
sdd_status rb_cuda(cudaError_t e, const char *what) {
    return (sdd_status)report_error(SDD_E_CUDA, (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
}
#define RB_CUDA(call)                                                \
    do {                                                             \
        cudaError_t e_ = (call);                                     \
        if (e_ != cudaSuccess) return rb_cuda(e_, #call);            \
    } while (0)

struct RbScratch {
    std::vector<void *> ptrs;
    cudaStream_t st = nullptr;
    cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    // a failed call may return with work in flight on st: the releases are
    // ordered behind it
    ~RbScratch() {
        for (void *p : ptrs) cudaFreeAsync(p, st);
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        if (st) cudaStreamDestroy(st);
    }
    template <class T>
    cudaError_t alloc(T **p, size_t count) {
        cudaError_t e = scratch_alloc((void **)p, count * sizeof(T), st);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
};

// A launch of the solver's kernel: its grid, and how many of its CTAs an SM
// takes.
struct SolveLaunch {
    const void *kernel = nullptr;
    int ctas = 0, per = 0, threads = 0;
    size_t smem = 0;
};

// Iterations of a turn, which another solve waits for at most, and of a launch.
// A turn ends with the host waiting for it (80 us).  A grid of more CTAs than
// SMs leaves no registers for other kernels, so its turns are short and cut
// into short launches, between which those get in.  Two solves of 300 x 300
// nodes (70 ms alone) from two threads: 102 ms so, 115 with 64 iterations a
// launch and 256 a turn, 125 with 256 and 256, 137 one after the other; alone
// the same within 1 %.
constexpr int kTurn = 1024, kFullTurn = 128, kFullRun = 32;

// At most ctas_max CTAs.  KEEP: *L stays empty where the blocks are more.
template <int SPLIT, bool KEEP>
cudaError_t shape_solve(const SolveArgs &A, int n_sm, int ctas_max, SolveLaunch *L) {
    constexpr int T = kDotThreads / SPLIT;
    const int parts = A.blocks * SPLIT;
    auto k = bicgstab_kernel<SPLIT, KEEP>;
    // the same attributes for every solve: others may be launching in other threads
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - kStaticSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    while (e == cudaSuccess && ctas_max > 0 && (!KEEP || parts <= ctas_max)) {
        const int ctas = std::min(parts, ctas_max), nb = (parts + ctas - 1) / ctas;
        const size_t smem = (size_t)nb * 2 * T * sizeof(Z) +
                            (KEEP ? (size_t)A.ns * T * (sizeof(double) + sizeof(int32_t)) : 0);
        int per = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, T, smem);
        if (e != cudaSuccess) return e;
        if (ctas <= per * n_sm) {
            *L = SolveLaunch{(const void *)k, ctas, per, T, smem};
            return cudaSuccess;
        }
        ctas_max = per * n_sm;
    }
    return e != cudaSuccess || KEEP ? e : cudaErrorLaunchOutOfResources;
}

// Two CTAs a block of rows while that leaves at most one CTA an SM (FP64 time
// halves, see bicgstab_kernel); one with the row in registers up to ctas_max
// blocks; else several blocks a CTA.
cudaError_t shape_bicgstab(const SolveArgs &A, int n_sm, int ctas_max, SolveLaunch *L) {
    *L = SolveLaunch{};
    if (2 * A.blocks <= n_sm) return shape_solve<2, true>(A, n_sm, ctas_max, L);
    cudaError_t e = shape_solve<1, true>(A, n_sm, ctas_max, L);
    if (e != cudaSuccess || L->kernel) return e;
    return shape_solve<1, false>(A, n_sm, ctas_max, L);
}

// Solves in flight on one device.  The CTAs of a grid wait for one another, so
// all grids in flight must fit on the GPU together.  With p the smallest number
// of CTAs an SM takes of any of their kernels, no CTA needs more than 1 / p of
// an SM: an SM that cannot take one more has p, and grids of together at most
// p x SMs CTAs all come through.  Launches go in the order of their tickets.
struct SolverQueue {
    std::mutex mu;
    std::condition_variable cv;
    uint64_t next = 0, serving = 0;
    int solves = 0;                             // solves between their first launch and their last
    std::vector<std::pair<int, int>> in_flight; // (CTAs, CTAs an SM takes)

    bool fits(const SolveLaunch &L, int n_sm) const {
        long long sum = L.ctas;
        int p = L.per;
        for (const auto &f : in_flight) {
            sum += f.first;
            p = std::min(p, f.second);
        }
        return in_flight.empty() || sum <= (long long)p * n_sm;
    }
};

SolverQueue &solver_queue(int dev) {
    static std::mutex mu;
    static std::map<int, SolverQueue> queues;
    std::lock_guard<std::mutex> lk(mu);
    return queues[dev];
}

// A solve's place among those of its device, from its first launch to its last.
struct SolverSeat {
    SolverQueue &Q;
    explicit SolverSeat(SolverQueue &q) : Q(q) {
        std::lock_guard<std::mutex> lk(Q.mu);
        ++Q.solves;
    }
    ~SolverSeat() {
        std::lock_guard<std::mutex> lk(Q.mu);
        --Q.solves;
    }
    // Waits for this launch's turn and for room.  alone, shared: the grid of a
    // solve that has the GPU to itself, and of one among others.
    SolveLaunch enter(const SolveLaunch &alone, const SolveLaunch &shared, int n_sm) {
        std::unique_lock<std::mutex> lk(Q.mu);
        const uint64_t me = Q.next++;
        SolveLaunch L;
        Q.cv.wait(lk, [&] {
            L = Q.solves > 1 ? shared : alone;
            return Q.serving == me && Q.fits(L, n_sm);
        });
        Q.in_flight.emplace_back(L.ctas, L.per);
        ++Q.serving;
        Q.cv.notify_all();
        return L;
    }
    void leave(const SolveLaunch &L) {
        std::lock_guard<std::mutex> lk(Q.mu);
        Q.in_flight.erase(std::find(Q.in_flight.begin(), Q.in_flight.end(), std::make_pair(L.ctas, L.per)));
        Q.cv.notify_all();
    }
};

sdd_status check_nodes_eps(const double *nodes_xz, int32_t n, int32_t ns, double eps) {
    if (ns < 2 || ns > kMaxStencil) return rb_arg("n_stencil must be in 2 .. SDD_RBFFD_MAX_STENCIL");
    if (n < ns || n > SDD_RBFFD_MAX_NODES) return rb_arg("n must be in n_stencil .. SDD_RBFFD_MAX_NODES");
    if (!(eps > 0.0) || !std::isfinite(eps)) return rb_arg("eps must be finite and > 0");
    if (!nodes_xz) return rb_arg("nodes_xz must not be NULL");
    for (int i = 0; i < 2 * n; ++i)
        if (!std::isfinite(nodes_xz[i])) return rb_arg("nodes must be finite");
    return SDD_OK;
}

// Stencils and weights on the device (d_p: nodes), timed by ev[0..2].
sdd_status weights_device(const double *h_p, const double *d_p, int n, int ns, double eps, int32_t *d_st,
                          double *d_w, RbScratch &S) {
    // the cell grid: about 2 nodes per cell over the bounding box, at most
    // 4 n + 16 cells
    double x0 = h_p[0], x1 = h_p[0], z0 = h_p[1], z1 = h_p[1];
    for (int i = 1; i < n; ++i) {
        x0 = std::min(x0, h_p[2 * i]);
        x1 = std::max(x1, h_p[2 * i]);
        z0 = std::min(z0, h_p[2 * i + 1]);
        z1 = std::max(z1, h_p[2 * i + 1]);
    }
    const double W = x1 - x0, H = z1 - z0, L = std::max(W, H);
    CellGrid g;
    g.x0 = x0;
    g.z0 = z0;
    g.c = W > 0.0 && H > 0.0 ? std::sqrt(2.0 * W * H / n) : (L > 0.0 ? 2.0 * L / n : 1.0);
    for (;;) {
        const double gx = std::floor(W / g.c) + 1.0, gz = std::floor(H / g.c) + 1.0;
        if (gx * gz <= 4.0 * n + 16.0) {
            g.gx = (int)gx;
            g.gz = (int)gz;
            break;
        }
        g.c *= 1.5;
    }
    const int m = g.gx * g.gz;
    int *d_err;
    int32_t *d_cell, *d_count, *d_start, *d_cursor, *d_list;
    RB_CUDA(S.alloc(&d_err, 1));
    RB_CUDA(S.alloc(&d_cell, (size_t)n));
    RB_CUDA(S.alloc(&d_count, (size_t)m));
    RB_CUDA(S.alloc(&d_start, (size_t)m + 1));
    RB_CUDA(S.alloc(&d_cursor, (size_t)m));
    RB_CUDA(S.alloc(&d_list, (size_t)n));
    RB_CUDA(cudaMemsetAsync(d_err, 0, sizeof(int), S.st));
    RB_CUDA(cudaMemsetAsync(d_count, 0, (size_t)m * sizeof(int32_t), S.st));
    RB_CUDA(cudaEventRecord(S.ev[0], S.st));
    cell_count_kernel<<<(n + 127) / 128, 128, 0, S.st>>>(d_p, n, g, d_cell, d_count);
    cell_scan_kernel<<<1, 1024, 0, S.st>>>(d_count, m, d_start);
    RB_CUDA(cudaMemcpyAsync(d_cursor, d_start, (size_t)m * sizeof(int32_t), cudaMemcpyDeviceToDevice, S.st));
    cell_fill_kernel<<<(n + 127) / 128, 128, 0, S.st>>>(d_cell, n, d_cursor, d_list);
    knn_kernel<<<(n + 127) / 128, 128, 0, S.st>>>(d_p, n, ns, g, d_start, d_list, d_st);
    RB_CUDA(cudaGetLastError());
    RB_CUDA(cudaEventRecord(S.ev[1], S.st));
    weights_kernel<<<(n + 63) / 64, 64, 0, S.st>>>(d_p, n, d_st, ns, eps, d_w, d_err);
    RB_CUDA(cudaGetLastError());
    RB_CUDA(cudaEventRecord(S.ev[2], S.st));
    int h_err = 0;
    RB_CUDA(cudaMemcpyAsync(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, S.st));
    RB_CUDA(cudaStreamSynchronize(S.st));
    if (h_err) return rb_arg("a stencil matrix is singular (coincident nodes)");
    return SDD_OK;
}

}  // namespace
}  // namespace sdd

using namespace sdd;

extern "C" sdd_status sdd_rbffd_weights(const double *nodes_xz, int32_t n, int32_t n_stencil, double eps,
                                        int32_t *stencil, double *weights) {
    sdd_status r = check_nodes_eps(nodes_xz, n, n_stencil, eps);
    if (r != SDD_OK) return r;
    if (!stencil || !weights) return rb_arg("stencil and weights must not be NULL");
    RbScratch S;
    RB_CUDA(cudaStreamCreateWithFlags(&S.st, cudaStreamNonBlocking));
    double *d_p, *d_w;
    int32_t *d_st;
    RB_CUDA(S.alloc(&d_p, 2 * (size_t)n));
    RB_CUDA(S.alloc(&d_st, (size_t)n * n_stencil));
    RB_CUDA(S.alloc(&d_w, (size_t)n * n_stencil));
    for (int k = 0; k < 3; ++k) RB_CUDA(cudaEventCreate(&S.ev[k]));
    RB_CUDA(cudaMemcpyAsync(d_p, nodes_xz, 2 * (size_t)n * sizeof(double), cudaMemcpyHostToDevice, S.st));
    r = weights_device(nodes_xz, d_p, n, n_stencil, eps, d_st, d_w, S);
    if (r != SDD_OK) return r;
    RB_CUDA(cudaMemcpyAsync(stencil, d_st, (size_t)n * n_stencil * sizeof(int32_t), cudaMemcpyDeviceToHost, S.st));
    RB_CUDA(cudaMemcpyAsync(weights, d_w, (size_t)n * n_stencil * sizeof(double), cudaMemcpyDeviceToHost, S.st));
    RB_CUDA(cudaStreamSynchronize(S.st));
    return SDD_OK;
}

extern "C" sdd_status sdd_rbffd_solve(const double *nodes_xz, int32_t n, const uint8_t *dirichlet,
                                      const double *values, const double *kappa, int32_t n_stencil,
                                      double eps, double tol, int32_t max_iter, double *u,
                                      sdd_rbffd_stats *stats) {
    if (stats) *stats = sdd_rbffd_stats{};
    sdd_status r = check_nodes_eps(nodes_xz, n, n_stencil, eps);
    if (r != SDD_OK) return r;
    if (!dirichlet || !values || !kappa || !u) return rb_arg("dirichlet, values, kappa and u must not be NULL");
    if (!(tol > 0.0) || !std::isfinite(tol)) return rb_arg("tol must be finite and > 0");
    if (max_iter < 1) return rb_arg("max_iter must be at least 1");
    std::vector<int32_t> unk, pos(n, -1);
    for (int i = 0; i < n; ++i) {
        if (dirichlet[i] > 1) return rb_arg("dirichlet flags must be 0 or 1");
        if (!std::isfinite(kappa[i])) return rb_arg("kappa must be finite");
        if (dirichlet[i]) {
            if (!std::isfinite(values[2 * i]) || !std::isfinite(values[2 * i + 1]))
                return rb_arg("Dirichlet values must be finite");
        } else {
            pos[i] = (int32_t)unk.size();
            unk.push_back(i);
        }
    }
    const int nu = (int)unk.size();
    for (int i = 0; i < n; ++i) {
        u[2 * i] = dirichlet[i] ? values[2 * i] : 0.0;
        u[2 * i + 1] = dirichlet[i] ? values[2 * i + 1] : 0.0;
    }
    if (stats) stats->unknowns = nu;
    if (nu == 0) return SDD_OK;

    const int ns = n_stencil;
    RbScratch S;
    RB_CUDA(cudaStreamCreateWithFlags(&S.st, cudaStreamNonBlocking));
    double *d_p, *d_w, *d_vals, *d_kap, *d_ew, *d_u;
    int32_t *d_st, *d_unk, *d_pos, *d_ecol;
    Z *d_dinv, *d_b, *x, *rr, *rh, *p, *v, *y, *s, *zz, *t, *part0, *d_part;
    Scal *d_S;
    unsigned *d_bar;
    RB_CUDA(S.alloc(&d_p, 2 * (size_t)n));
    RB_CUDA(S.alloc(&d_st, (size_t)n * ns));
    RB_CUDA(S.alloc(&d_w, (size_t)n * ns));
    RB_CUDA(S.alloc(&d_vals, 2 * (size_t)n));
    RB_CUDA(S.alloc(&d_kap, (size_t)n));
    RB_CUDA(S.alloc(&d_unk, (size_t)nu));
    RB_CUDA(S.alloc(&d_pos, (size_t)n));
    RB_CUDA(S.alloc(&d_ew, (size_t)nu * ns));
    RB_CUDA(S.alloc(&d_ecol, (size_t)nu * ns));
    RB_CUDA(S.alloc(&d_u, 2 * (size_t)n));
    for (Z **q : {&d_dinv, &d_b, &x, &rr, &rh, &p, &v, &y, &s, &zz, &t}) RB_CUDA(S.alloc(q, (size_t)nu));
    RB_CUDA(S.alloc(&part0, (size_t)kDotBlocks));
    RB_CUDA(S.alloc(&d_part, 5 * 2 * (size_t)kDotBlocks));
    RB_CUDA(S.alloc(&d_S, 1));
    RB_CUDA(S.alloc(&d_bar, 1));
    for (int k = 0; k < 5; ++k) RB_CUDA(cudaEventCreate(&S.ev[k]));
    cudaStream_t st = S.st;
    RB_CUDA(cudaMemcpyAsync(d_p, nodes_xz, 2 * (size_t)n * sizeof(double), cudaMemcpyHostToDevice, st));
    RB_CUDA(cudaMemcpyAsync(d_vals, u, 2 * (size_t)n * sizeof(double), cudaMemcpyHostToDevice, st));
    RB_CUDA(cudaMemcpyAsync(d_kap, kappa, (size_t)n * sizeof(double), cudaMemcpyHostToDevice, st));
    RB_CUDA(cudaMemcpyAsync(d_unk, unk.data(), (size_t)nu * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    RB_CUDA(cudaMemcpyAsync(d_pos, pos.data(), (size_t)n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    r = weights_device(nodes_xz, d_p, n, ns, eps, d_st, d_w, S);
    if (r != SDD_OK) return r;

    const int gb = (nu + 127) / 128;
    const int gd = std::min(kDotBlocks, (nu + kDotThreads - 1) / kDotThreads);
    assemble_kernel<<<gb, 128, 0, st>>>(d_unk, d_pos, nu, d_st, d_w, ns, d_kap, d_vals, d_ew, d_ecol, d_dinv, d_b);
    RB_CUDA(cudaGetLastError());
    // x = 0, r = r^ = b, p = v = 0
    RB_CUDA(cudaMemsetAsync(x, 0, (size_t)nu * sizeof(Z), st));
    RB_CUDA(cudaMemsetAsync(p, 0, (size_t)nu * sizeof(Z), st));
    RB_CUDA(cudaMemsetAsync(v, 0, (size_t)nu * sizeof(Z), st));
    RB_CUDA(cudaMemcpyAsync(rr, d_b, (size_t)nu * sizeof(Z), cudaMemcpyDeviceToDevice, st));
    RB_CUDA(cudaMemcpyAsync(rh, d_b, (size_t)nu * sizeof(Z), cudaMemcpyDeviceToDevice, st));
    norm_partial_kernel<<<gd, kDotThreads, 0, st>>>(d_b, nu, part0);
    RB_CUDA(cudaGetLastError());
    std::vector<Z> h_part(gd);
    RB_CUDA(cudaMemcpyAsync(h_part.data(), part0, gd * sizeof(Z), cudaMemcpyDeviceToHost, st));
    RB_CUDA(cudaStreamSynchronize(st));
    double bnorm2 = 0.0;
    for (int k = 0; k < gd; ++k) bnorm2 += h_part[k].re;
    Scal h_S{};
    h_S.alpha = h_S.omega = Z{1.0, 0.0};
    h_S.beta = Z{0.0, 0.0};
    h_S.rho = Z{bnorm2, 0.0};  // <r^, r> with r^ = r = b
    h_S.bnorm2 = bnorm2;
    h_S.rnorm2 = bnorm2;
    h_S.tol2 = tol * tol;
    if (bnorm2 == 0.0) h_S.stop = 1;  // zero right-hand side: x = 0
    RB_CUDA(cudaMemcpyAsync(d_S, &h_S, sizeof(Scal), cudaMemcpyHostToDevice, st));
    RB_CUDA(cudaEventRecord(S.ev[3], st));

    // iterations
    SolveArgs sa{};
    sa.ew = d_ew; sa.ecol = d_ecol; sa.unk = d_unk; sa.kappa = d_kap; sa.dinv = d_dinv; sa.rh = rh;
    sa.r = rr; sa.p = p; sa.v = v; sa.x = x; sa.y = y; sa.z = zz; sa.s = s; sa.t = t;
    sa.part = d_part; sa.S = d_S; sa.bar = d_bar;
    sa.nu = nu; sa.ns = ns;
    sa.blocks = (nu + kDotThreads - 1) / kDotThreads;
    int dev = 0, n_sm = 0;
    RB_CUDA(cudaGetDevice(&dev));
    RB_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    // alone: all the CTAs that fit; beside other solves: half of them
    SolveLaunch alone, shared;
    RB_CUDA(shape_bicgstab(sa, n_sm, 2 * n_sm, &alone));
    if (alone.ctas > n_sm) RB_CUDA(shape_bicgstab(sa, n_sm, n_sm, &shared));
    else shared = alone;
    {
        SolverSeat seat(solver_queue(dev));
        int tries = 0;
        auto turn = [&]() -> cudaError_t {
            const SolveLaunch L = seat.enter(alone, shared, n_sm);
            const bool full = L.ctas > n_sm;
            int left = std::min(max_iter - h_S.iter, full ? kFullTurn : kTurn);
            cudaError_t e = cudaSuccess;
            for (; left > 0 && e == cudaSuccess; left -= sa.max_iter) {
                sa.max_iter = std::min(left, full ? kFullRun : kTurn);
                void *args[] = {&sa};
                e = cudaMemsetAsync(d_bar, 0, sizeof(unsigned), st);
                if (e == cudaSuccess)
                    e = cudaLaunchCooperativeKernel(L.kernel, dim3(L.ctas), dim3(L.threads), args, L.smem, st);
            }
            // waited for before the copy: a copy to pageable memory waits for the
            // grid inside the driver, and other threads' copies wait with it
            const cudaError_t es = cudaStreamSynchronize(st);
            seat.leave(L);
            if (e == cudaSuccess) e = es;
            if (e == cudaSuccess) e = cudaMemcpyAsync(&h_S, d_S, sizeof(Scal), cudaMemcpyDeviceToHost, st);
            return e != cudaSuccess ? e : cudaStreamSynchronize(st);
        };
        while (h_S.iter < max_iter && !h_S.stop) {
            RB_CUDA(turn());
            if (h_S.stop == 4) {  // other kernels held the SMs for two seconds
                if (++tries == kTries)
                    return (sdd_status)report_error(SDD_E_CUDA, "other kernels kept the solver's blocks off the GPU");
                h_S.stop = 0;
                RB_CUDA(cudaMemcpyAsync(d_S, &h_S, sizeof(Scal), cudaMemcpyHostToDevice, st));
                RB_CUDA(cudaStreamSynchronize(st));
                continue;
            }
            tries = 0;
        }
    }
    if (h_S.stop == 3) return (sdd_status)report_error(SDD_E_CUDA, "a wait between the solver's blocks ran out");
    // the true residual |b - K x| / |b|
    spmv_kernel<<<gb, 128, 0, st>>>(d_ew, d_ecol, nu, ns, d_unk, d_kap, x, t);
    residual_kernel<<<gb, 128, 0, st>>>(t, d_b, nu, s);
    norm_partial_kernel<<<gd, kDotThreads, 0, st>>>(s, nu, part0);
    RB_CUDA(cudaGetLastError());
    RB_CUDA(cudaMemcpyAsync(d_u, u, 2 * (size_t)n * sizeof(double), cudaMemcpyHostToDevice, st));
    scatter_u_kernel<<<gb, 128, 0, st>>>(d_unk, nu, x, d_u);
    RB_CUDA(cudaGetLastError());
    RB_CUDA(cudaMemcpyAsync(u, d_u, 2 * (size_t)n * sizeof(double), cudaMemcpyDeviceToHost, st));
    RB_CUDA(cudaMemcpyAsync(h_part.data(), part0, gd * sizeof(Z), cudaMemcpyDeviceToHost, st));
    RB_CUDA(cudaEventRecord(S.ev[4], st));
    RB_CUDA(cudaStreamSynchronize(st));
    double res2 = 0.0;
    for (int k = 0; k < gd; ++k) res2 += h_part[k].re;
    if (stats) {
        float ms = 0.f;
        stats->iterations = h_S.iter;
        stats->rel_residual = bnorm2 > 0.0 ? std::sqrt(res2 / bnorm2) : 0.0;
        RB_CUDA(cudaEventElapsedTime(&ms, S.ev[0], S.ev[1]));
        stats->knn_ms = ms;
        RB_CUDA(cudaEventElapsedTime(&ms, S.ev[1], S.ev[2]));
        stats->weights_ms = ms;
        RB_CUDA(cudaEventElapsedTime(&ms, S.ev[3], S.ev[4]));
        stats->solve_ms = ms;
    }
    if (h_S.stop == 2) return (sdd_status)report_error(SDD_E_TIMEOUT, "BiCGStab broke down before convergence");
    if (h_S.stop != 1) return (sdd_status)report_error(SDD_E_TIMEOUT, "BiCGStab did not reach tol within max_iter");
    return SDD_OK;
}
