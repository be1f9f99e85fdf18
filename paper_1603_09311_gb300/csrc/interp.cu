// Interface values between Monte Carlo nodes (Sec. 5 of arXiv:1603.09311:
// the stochastic solution is computed at some points along an interface and
// the remaining interface values are interpolated).
//
// The paper gives no scheme; the one built here interpolates each real
// component of each evaluation in the arc length s along the interface
// polyline, piecewise linearly or by the natural cubic spline.  Both are
// linear in the knot values, v(s) = sum_j c_j(s) v_j, and the knots'
// estimates are independent, so the standard error carried to s is
// sqrt(sum_j c_j(s)^2 se_j^2).
//
// Kernels (all FP64; chains of dependent FP64 operations, about 70 cycles
// each, are the time, so what can be cut into short ones is):
//   length_kernel         segment lengths of the polyline
//   arc_kernel            their prefix sums, one CTA (chunk sums, a
//                         shared-memory scan, chunk prefixes)
//   spline_factor_kernel  forward coefficients of the natural-spline
//                         equations, one thread a row
//   spline_cols_kernel    G = the spline's second derivatives of every unit
//                         knot vector, one thread a column, as far as they
//                         matter
//   linear_kernel, spline_kernel  values and standard errors
//   scatter_kernel        the knots keep their own estimates
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "sdd.h"
#include "sdd_internal.cuh"

namespace sdd {
namespace {

constexpr int kArcThreads = 1024;

// s[k + 1] = length of segment k
__global__ void length_kernel(const double *p, int n, double *s) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n - 1) s[k + 1] = hypot(p[2 * k + 2] - p[2 * k], p[2 * k + 3] - p[2 * k + 1]);
}

// s[0] = 0, s[k] = sum of the lengths s[1 .. k], in place.  One CTA does only
// the additions: with the square roots in it (twice) it took 60 us for 1025
// nodes, the two kernels take 12.
__global__ void __launch_bounds__(kArcThreads) arc_kernel(int n, double *s) {
    __shared__ double part[kArcThreads];
    const int t = threadIdx.x;
    const int segs = n - 1;
    const int per = (segs + kArcThreads - 1) / kArcThreads;
    const int a = min(t * per, segs), b = min(a + per, segs);
    double acc = 0.0;
    for (int k = a; k < b; ++k) acc += s[k + 1];
    part[t] = acc;
    __syncthreads();
    for (int off = 1; off < kArcThreads; off <<= 1) {
        const double v = t >= off ? part[t - off] : 0.0;
        __syncthreads();
        if (t >= off) part[t] += v;
        __syncthreads();
    }
    double run = t > 0 ? part[t - 1] : 0.0;
    if (t == 0) s[0] = 0.0;
    for (int k = a; k < b; ++k) {
        run += s[k + 1];
        s[k + 1] = run;
    }
}

// The natural spline's second derivatives M solve, for the inner knots
// i = 1 .. n-2 (row r = i - 1), with h_i = s_{i+1} - s_i,
//   h_{i-1} M_{i-1} + 2 (h_{i-1} + h_i) M_i + h_i M_{i+1}
//       = 6 ((v_{i+1} - v_i) / h_i - (v_i - v_{i-1}) / h_{i-1}),
// M_0 = M_{n-1} = 0.  Thomas forward sweep: den_r = 2 (h_{i-1} + h_i) -
// h_{i-1} cp_{r-1}, cp_r = h_i / den_r; rden = 1 / den.
//
// A row's cp depends on the one before through a factor
// h_{i-1} h_i / den^2 <= 1/12 (den >= 3/2 h_{i-1} + 2 h_i), so a sweep that
// starts kWarm rows early from any value in [0, 1/2] has the row's cp to
// 12^-kWarm < 2^-64: every row is a thread's chain of kWarm divisions, not of
// all rows before it (257 knots: 190 us -> 15 us).
constexpr int kWarm = 18;

// What the columns need to know of a call's data: the largest knot spacing (its
// bits; of positive doubles these order as the doubles do), whether the weights
// have to be kept whole, and the columns' farthest reach.
struct SplineScan {
    unsigned long long h_max;
    int whole;   // a component of wide range, or not finite
    int reach;   // largest |i - j| of a kept G[i][j]
    double cut;  // entries of G below it are left out
};

// Columns keep the entries above 2^-100 / h_max^2: a weight is at most 0.13
// h^2 max |G| besides its a or b, h the target's spacing, so what is left out
// changes a weight by less than 2^-100, whatever the spacings.  (A cut against
// the column's own largest entry is not enough: the weights carry h^2, and on
// knots whose spacing grows by 2.6 or more a row they do not fall off at all.)
// The weights add up to one, so where a component's largest modulus is at most
// 2^40 times its smallest a sum loses less than 2^-60 a knot of the moduli of
// its terms.  Other components (zeros, outliers, values that are not finite:
// these count with any weight) keep every weight, and so do spacings whose
// square leaves the double range.
constexpr double kRange = 1099511627776.0;  // 2^40
__device__ __forceinline__ double column_cut(const SplineScan &q) {
    const double h = __longlong_as_double((long long)q.h_max), h2 = h * h;
    return q.whole || !(h2 > 1e-290) || isinf(h2) ? 0.0 : 7.888609052210118e-31 / h2;
}

__global__ void spline_factor_kernel(const double *s, int n, double *cp, double *rden, SplineScan *scan) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row == 0) scan->cut = column_cut(*scan);
    if (row >= n - 2) return;
    double prev = 0.0, d = 0.0;
    for (int r = max(row - kWarm, 0); r <= row; ++r) {
        const int i = r + 1;
        const double hl = s[i] - s[i - 1], hr = s[i + 1] - s[i];
        d = 2.0 * (hl + hr) - (r > 0 ? hl * prev : 0.0);
        prev = hr / d;
    }
    rden[row] = 1.0 / d;
    cp[row] = prev;
}

// Knot spacings must be positive (arc lengths of distinct nodes can still
// round to equal values).  scan (spline, else nullptr): the largest spacing; a
// warp for each component of v and of se (from CTA `from` on) its range.
__global__ void __launch_bounds__(32)
    knots_check_kernel(const double *s, int n, int *err, int from, const double *v, const double *se, int V,
                       SplineScan *scan) {
    if ((int)blockIdx.x < from) {
        const int i = blockIdx.x * 32 + threadIdx.x + 1;
        if (i >= n) return;
        const double h = s[i] - s[i - 1];
        if (!(s[i] > s[i - 1])) atomicExch(err, 1);
        else if (scan) atomicMax(&scan->h_max, (unsigned long long)__double_as_longlong(h));
        return;
    }
    const int c = (int)blockIdx.x - from;
    const double *u = c < V ? v + c : se + (c - V);
    double big = 0.0, small = HUGE_VAL;
    bool bad = false;
    for (int j = threadIdx.x; j < n; j += 32) {
        const double x = fabs(u[(size_t)j * V]);
        bad = bad || !isfinite(x);
        big = fmax(big, x);
        small = fmin(small, x);
    }
    for (int off = 16; off > 0; off >>= 1) {
        big = fmax(big, __shfl_xor_sync(0xffffffffu, big, off));
        small = fmin(small, __shfl_xor_sync(0xffffffffu, small, off));
    }
    bad = __any_sync(0xffffffffu, bad) || big > kRange * small;
    if (bad && threadIdx.x == 0) scan->whole = 1;
}

// Column j of G [n][n]: M(e_j), the second derivatives of the natural spline
// through the unit vector e_j; zero where not written.  The right-hand side of
// row r (knot i = r + 1) is non-zero for i in {j - 1, j, j + 1} only, and the
// entries fall off on both sides, by at least 2/3 a row (0.27 on even knots): a
// column ends where they are below the cut, after about 53 rows on even knots.
__global__ void __launch_bounds__(32)
    spline_cols_kernel(const double *s, int n, const double *cp, const double *rden, double *G, SplineScan *scan) {
    const int j = blockIdx.x * 32 + threadIdx.x;
    int reach = 0;
    if (j < n) {
        const int m = n - 2;
        auto at = [&](int r) -> double & { return G[(size_t)(r + 1) * n + j]; };
        const double cut = scan->cut;
        const int r0 = max(j - 2, 0);  // first row with a right-hand side
        double dprev = 0.0;
        int r1 = r0 - 1;
        for (int r = r0; r < m; ++r) {
            const int i = r + 1;
            const double hl = s[i] - s[i - 1];
            double rhs = 0.0;
            if (j >= i - 1 && j <= i + 1) {
                const double hr = s[i + 1] - s[i];
                if (j == i - 1) rhs = 6.0 / hl;
                else if (j == i) rhs = -(6.0 / hl + 6.0 / hr);
                else rhs = 6.0 / hr;
            }
            const double d = (rhs - hl * dprev) * rden[r];
            at(r) = d;
            dprev = d;
            r1 = r;
            if (r > j && fabs(d) < cut) break;
        }
        double xnext = 0.0;
        int low = r0;
        for (int r = r1; r >= 0; --r) {
            const double x = (r >= r0 ? at(r) : 0.0) - (r < m - 1 ? cp[r] * xnext : 0.0);
            at(r) = x;
            xnext = x;
            low = r;
            if (r < r0 && fabs(x) < cut) break;
        }
        reach = max(r1 + 1 - j, j - (low + 1));
    }
    reach = __reduce_max_sync(0xffffffffu, reach);
    if (threadIdx.x == 0) atomicMax(&scan->reach, reach);
}

// The target's segment: the largest i <= nk - 2 with s_i <= x.
__device__ __forceinline__ int segment(const double *sk, int nk, double x) {
    int lo = 0, hi = nk - 2;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sk[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Thread (target q, component c): with a = (s_{i+1} - t) / h and
// b = (t - s_i) / h the weights are c_i = a, c_{i+1} = b.
__global__ void linear_kernel(const double *sk, int nk, const double *v, const double *se, int V, const double *t,
                              int nt, double *ov, double *ose) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)nt * V) return;
    const int q = (int)(idx / V), c = (int)(idx % V);
    const double x = t[q];
    const int i = segment(sk, nk, x);
    const double h = sk[i + 1] - sk[i];
    const double a = (sk[i + 1] - x) / h, b = (x - sk[i]) / h;
    const double v0 = v[(size_t)i * V + c], v1 = v[(size_t)(i + 1) * V + c];
    ov[idx] = a * v0 + b * v1;
    if (ose) {
        double var = 0.0;
        if (se) {
            const double e0 = a * se[(size_t)i * V + c], e1 = b * se[(size_t)(i + 1) * V + c];
            var = e0 * e0 + e1 * e1;
        }
        ose[idx] = sqrt(var);
    }
}

// CTA q: target q.  The weights
//   c_j = a [j = i] + b [j = i + 1]
//         + (a^3 - a) h^2 / 6 G[i][j] + (b^3 - b) h^2 / 6 G[i+1][j]
// of the columns that reach the segment are formed once, a thread each, then
// every thread adds up a component.  With a thread for each target and
// component and all knots in each sum, 1025 targets x 32 components x 257 knots
// took 0.35 ms; 0.03 ms so, behind 0.04 ms for the columns.
constexpr int kSplineThreads = 64;
constexpr int kWeights = 512;
__global__ void __launch_bounds__(kSplineThreads)
    spline_kernel(const double *sk, int nk, const double *G, const SplineScan *scan, const double *v, const double *se,
                  int V, const double *t, double *ov, double *ose) {
    __shared__ double w[kWeights];
    const size_t q = blockIdx.x;
    const double x = t[q];
    const int i = segment(sk, nk, x);
    const double h = sk[i + 1] - sk[i];
    const double a = (sk[i + 1] - x) / h, b = (x - sk[i]) / h;
    const double al = (a * a * a - a) * h * h / 6.0, be = (b * b * b - b) * h * h / 6.0;
    const double *gi = G + (size_t)i * nk, *gi1 = gi + nk;
    const int reach = scan->whole ? nk : scan->reach;
    const int j0 = max(i - reach, 0), j1 = min(i + 1 + reach, nk - 1);
    for (int c0 = 0; c0 < V; c0 += kSplineThreads) {
        const int c = c0 + threadIdx.x;
        double val = 0.0, var = 0.0;
        for (int k0 = j0; k0 <= j1; k0 += kWeights) {
            const int n = min(j1 + 1 - k0, kWeights);
            __syncthreads();
            for (int k = threadIdx.x; k < n; k += kSplineThreads) {
                const int j = k0 + k;
                double cj = al * gi[j] + be * gi1[j];
                if (j == i) cj += a;
                if (j == i + 1) cj += b;
                w[k] = cj;
            }
            __syncthreads();
            if (c >= V) continue;
            const double *vc = v + (size_t)k0 * V + c;
            if (se) {
                const double *ec = se + (size_t)k0 * V + c;
#pragma unroll 4
                for (int k = 0; k < n; ++k) {
                    val += w[k] * vc[(size_t)k * V];
                    const double e = w[k] * ec[(size_t)k * V];
                    var += e * e;
                }
            } else {
#pragma unroll 4
                for (int k = 0; k < n; ++k) val += w[k] * vc[(size_t)k * V];
            }
        }
        if (c >= V) continue;
        ov[q * V + c] = val;
        if (ose) ose[q * V + c] = sqrt(var);
    }
}

__global__ void gather_kernel(const double *s, const int32_t *idx, int nk, double *out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < nk) out[j] = s[idx[j]];
}

__global__ void scatter_kernel(const double *kv, const double *kse, const int32_t *idx, int nk,
                               int V, double *ov, double *ose) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)nk * V) return;
    const int j = (int)(e / V), c = (int)(e % V);
    ov[(size_t)idx[j] * V + c] = kv[e];
    ose[(size_t)idx[j] * V + c] = kse[e];
}

// Stream and device allocations of one call, released on every return path.
struct Scratch {
    std::vector<void *> ptrs;
    cudaStream_t st = nullptr;
    ~Scratch() {
        for (void *p : ptrs) cudaFreeAsync(p, st);
        if (st) cudaStreamDestroy(st);
    }
    cudaError_t open() { return cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking); }
    template <class T>
    cudaError_t alloc(T **p, size_t count) {
        *p = nullptr;
        cudaError_t e = scratch_alloc((void **)p, count * sizeof(T), st);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
};

#define INTERP_CUDA(call)                                            \
    do {                                                             \
        cudaError_t e_ = (call);                                     \
        if (e_ != cudaSuccess) return cuda_error(e_, #call);         \
    } while (0)

sdd_status cuda_error(cudaError_t e, const char *what) {
    return (sdd_status)report_error(SDD_E_CUDA, (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
}

sdd_status arg_error(const char *msg) { return (sdd_status)report_error(SDD_E_ARG, msg); }

// Interpolation of device knot data to device targets on stream st.  The
// knot check's flag is copied to *h_err, valid once st has been
// synchronised.
sdd_status run_interp(const double *d_sk, int nk, const double *d_v, const double *d_se, int V,
                      const double *d_t, int nt, int kind, double *d_ov, double *d_ose,
                      Scratch &S, cudaStream_t st, int *h_err) {
    const bool spline = kind == SDD_INTERP_SPLINE && nk > 2;
    struct Flags {
        int err;
        SplineScan scan;
    } *flags;
    INTERP_CUDA(S.alloc(&flags, 1));
    INTERP_CUDA(cudaMemsetAsync(flags, 0, sizeof(Flags), st));
    int *err = &flags->err;
    SplineScan *scan = spline ? &flags->scan : nullptr;
    const int pairs = (nk - 1 + 31) / 32, jobs = !spline ? 0 : d_se ? 2 * V : V;
    knots_check_kernel<<<(unsigned)pairs + jobs, 32, 0, st>>>(d_sk, nk, err, pairs, d_v, d_se, V, scan);
    INTERP_CUDA(cudaGetLastError());
    const long long total = (long long)nt * V;
    if (spline) {
        double *G, *cp, *rden;
        INTERP_CUDA(S.alloc(&G, (size_t)nk * nk));
        INTERP_CUDA(S.alloc(&cp, (size_t)nk));
        INTERP_CUDA(S.alloc(&rden, (size_t)nk));
        INTERP_CUDA(cudaMemsetAsync(G, 0, (size_t)nk * nk * sizeof(double), st));
        spline_factor_kernel<<<(nk + 63) / 64, 64, 0, st>>>(d_sk, nk, cp, rden, scan);
        INTERP_CUDA(cudaGetLastError());
        spline_cols_kernel<<<(nk + 31) / 32, 32, 0, st>>>(d_sk, nk, cp, rden, G, scan);
        INTERP_CUDA(cudaGetLastError());
        if (total > 0) {
            spline_kernel<<<(unsigned)nt, kSplineThreads, 0, st>>>(d_sk, nk, G, scan, d_v, d_se, V, d_t, d_ov, d_ose);
            INTERP_CUDA(cudaGetLastError());
        }
    } else if (total > 0) {
        const int threads = 128;
        linear_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, st>>>(d_sk, nk, d_v, d_se, V, d_t, nt,
                                                                                      d_ov, d_ose);
        INTERP_CUDA(cudaGetLastError());
    }
    INTERP_CUDA(cudaMemcpyAsync(h_err, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    return SDD_OK;
}

}  // namespace
}  // namespace sdd

using namespace sdd;

extern "C" sdd_status sdd_interpolate(const double *knots_s, int32_t n_knots, const double *values,
                                      const double *se, int32_t n_vals, const double *targets_s,
                                      int32_t n_targets, int32_t kind, double *out_values,
                                      double *out_se) {
    if (kind != SDD_INTERP_LINEAR && kind != SDD_INTERP_SPLINE)
        return arg_error("kind must be SDD_INTERP_LINEAR or SDD_INTERP_SPLINE");
    if (n_knots < 2) return arg_error("n_knots must be at least 2");
    if (kind == SDD_INTERP_SPLINE && n_knots > SDD_INTERP_MAX_SPLINE_KNOTS)
        return arg_error("n_knots exceeds SDD_INTERP_MAX_SPLINE_KNOTS for the spline");
    if (n_vals < 1) return arg_error("n_vals must be at least 1");
    if (n_targets < 0) return arg_error("n_targets must not be negative");
    if (!knots_s || !values || (n_targets > 0 && (!targets_s || !out_values)))
        return arg_error("knots_s, values, targets_s and out_values must not be NULL");
    for (int i = 0; i < n_knots; ++i) {
        if (!std::isfinite(knots_s[i])) return arg_error("knots must be finite");
        if (i > 0 && !(knots_s[i] > knots_s[i - 1])) return arg_error("knots must be strictly increasing");
    }
    for (int q = 0; q < n_targets; ++q)
        if (!(targets_s[q] >= knots_s[0] && targets_s[q] <= knots_s[n_knots - 1]))
            return arg_error("targets must lie within [knots_s[0], knots_s[n_knots - 1]]");
    if (n_targets == 0) return SDD_OK;
    const bool with_se = se != nullptr && out_se != nullptr;
    const size_t kb = (size_t)n_knots * n_vals, tb = (size_t)n_targets * n_vals;
    Scratch S;
    INTERP_CUDA(S.open());
    const cudaStream_t st = S.st;
    double *sk, *v, *e = nullptr, *t, *ov, *oe = nullptr;
    INTERP_CUDA(S.alloc(&sk, n_knots));
    INTERP_CUDA(S.alloc(&v, kb));
    INTERP_CUDA(S.alloc(&t, n_targets));
    INTERP_CUDA(S.alloc(&ov, tb));
    if (with_se) {
        INTERP_CUDA(S.alloc(&e, kb));
        INTERP_CUDA(S.alloc(&oe, tb));
    }
    INTERP_CUDA(cudaMemcpyAsync(sk, knots_s, n_knots * sizeof(double), cudaMemcpyHostToDevice, st));
    INTERP_CUDA(cudaMemcpyAsync(v, values, kb * sizeof(double), cudaMemcpyHostToDevice, st));
    INTERP_CUDA(cudaMemcpyAsync(t, targets_s, n_targets * sizeof(double), cudaMemcpyHostToDevice, st));
    if (with_se) INTERP_CUDA(cudaMemcpyAsync(e, se, kb * sizeof(double), cudaMemcpyHostToDevice, st));
    int h_err = 0;
    sdd_status r = run_interp(sk, n_knots, v, e, n_vals, t, n_targets, kind, ov, oe, S, st, &h_err);
    if (r != SDD_OK) return r;
    INTERP_CUDA(cudaMemcpyAsync(out_values, ov, tb * sizeof(double), cudaMemcpyDeviceToHost, st));
    if (with_se) INTERP_CUDA(cudaMemcpyAsync(out_se, oe, tb * sizeof(double), cudaMemcpyDeviceToHost, st));
    INTERP_CUDA(cudaStreamSynchronize(st));
    if (h_err) return arg_error("knots must be strictly increasing");
    return SDD_OK;
}

extern "C" sdd_status sdd_interface_values_interp(sdd_ctx *ctx, const double *nodes_xz,
                                                  int32_t n_nodes, int32_t stride, int64_t n_paths,
                                                  int32_t kind, double dt, uint64_t seed,
                                                  const sdd_config *cfg, double *mean, double *se,
                                                  sdd_stats *stats) {
    if (!ctx) return arg_error("ctx must not be NULL");
    if (kind != SDD_INTERP_LINEAR && kind != SDD_INTERP_SPLINE)
        return arg_error("kind must be SDD_INTERP_LINEAR or SDD_INTERP_SPLINE");
    if (n_nodes < 2 || n_nodes > SDD_INTERP_MAX_NODES)
        return arg_error("n_nodes must be in 2 .. SDD_INTERP_MAX_NODES");
    if (stride < 1) return arg_error("stride must be at least 1");
    if (n_paths < 1 || n_paths > INT32_MAX) return arg_error("n_paths must be in 1 .. 2^31-1");
    if (!nodes_xz || !mean || !se) return arg_error("nodes_xz, mean and se must not be NULL");
    for (int i = 1; i < n_nodes; ++i)
        if (nodes_xz[2 * i] == nodes_xz[2 * i - 2] && nodes_xz[2 * i + 1] == nodes_xz[2 * i - 1])
            return arg_error("consecutive interface nodes must differ");
    std::vector<int32_t> kidx;
    for (int i = 0; i < n_nodes; i += stride) kidx.push_back(i);
    if (kidx.back() != n_nodes - 1) kidx.push_back(n_nodes - 1);
    const int nk = (int)kidx.size();
    if (kind == SDD_INTERP_SPLINE && nk > SDD_INTERP_MAX_SPLINE_KNOTS)
        return arg_error("too many Monte Carlo nodes for the spline (SDD_INTERP_MAX_SPLINE_KNOTS)");
    const int E = sdd_n_eval(ctx), V = 2 * E;

    // Monte Carlo at the knots, each under its index along the polyline as
    // RNG node id (the values sdd_interface_values gives those nodes in a
    // call on the whole polyline)
    std::vector<double> knodes(2 * (size_t)nk), kmean((size_t)nk * V), kse((size_t)nk * V);
    std::vector<uint32_t> kid(nk);
    std::vector<int64_t> kpaths(nk, n_paths);
    for (int j = 0; j < nk; ++j) {
        knodes[2 * j] = nodes_xz[2 * (size_t)kidx[j]];
        knodes[2 * j + 1] = nodes_xz[2 * (size_t)kidx[j] + 1];
        kid[j] = (uint32_t)kidx[j];
    }
    const sdd_status mc = sdd_interface_values(ctx, knodes.data(), kid.data(), nk, kpaths.data(), dt,
                                               seed, cfg, kmean.data(), kse.data(), stats);
    if (mc != SDD_OK && mc != SDD_E_TRUNCATED) return mc;

    Scratch S;
    INTERP_CUDA(S.open());
    const cudaStream_t st = S.st;
    double *p, *s, *sk, *kv, *ke, *ov, *oe;
    int32_t *di;
    const size_t ob = (size_t)n_nodes * V;
    INTERP_CUDA(S.alloc(&p, 2 * (size_t)n_nodes));
    INTERP_CUDA(S.alloc(&s, (size_t)n_nodes));
    INTERP_CUDA(S.alloc(&sk, (size_t)nk));
    INTERP_CUDA(S.alloc(&di, (size_t)nk));
    INTERP_CUDA(S.alloc(&kv, (size_t)nk * V));
    INTERP_CUDA(S.alloc(&ke, (size_t)nk * V));
    INTERP_CUDA(S.alloc(&ov, ob));
    INTERP_CUDA(S.alloc(&oe, ob));
    INTERP_CUDA(cudaMemcpyAsync(p, nodes_xz, 2 * (size_t)n_nodes * sizeof(double), cudaMemcpyHostToDevice, st));
    INTERP_CUDA(cudaMemcpyAsync(di, kidx.data(), nk * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    INTERP_CUDA(cudaMemcpyAsync(kv, kmean.data(), (size_t)nk * V * sizeof(double), cudaMemcpyHostToDevice, st));
    INTERP_CUDA(cudaMemcpyAsync(ke, kse.data(), (size_t)nk * V * sizeof(double), cudaMemcpyHostToDevice, st));
    cudaEvent_t ev[2];
    INTERP_CUDA(cudaEventCreate(&ev[0]));
    struct EventGuard {
        cudaEvent_t *e;
        int n = 0;
        ~EventGuard() {
            for (int i = 0; i < n; ++i) cudaEventDestroy(e[i]);
        }
    } eg{ev, 1};
    INTERP_CUDA(cudaEventCreate(&ev[1]));
    eg.n = 2;
    INTERP_CUDA(cudaEventRecord(ev[0], st));
    length_kernel<<<(n_nodes + 127) / 128, 128, 0, st>>>(p, n_nodes, s);
    INTERP_CUDA(cudaGetLastError());
    arc_kernel<<<1, kArcThreads, 0, st>>>(n_nodes, s);
    INTERP_CUDA(cudaGetLastError());
    gather_kernel<<<(nk + 127) / 128, 128, 0, st>>>(s, di, nk, sk);
    INTERP_CUDA(cudaGetLastError());
    int h_err = 0;
    sdd_status r = run_interp(sk, nk, kv, ke, V, s, n_nodes, kind, ov, oe, S, st, &h_err);
    if (r != SDD_OK) return r;
    const long long kt = (long long)nk * V;
    scatter_kernel<<<(unsigned)((kt + 127) / 128), 128, 0, st>>>(kv, ke, di, nk, V, ov, oe);
    INTERP_CUDA(cudaGetLastError());
    INTERP_CUDA(cudaEventRecord(ev[1], st));
    INTERP_CUDA(cudaMemcpyAsync(mean, ov, ob * sizeof(double), cudaMemcpyDeviceToHost, st));
    INTERP_CUDA(cudaMemcpyAsync(se, oe, ob * sizeof(double), cudaMemcpyDeviceToHost, st));
    INTERP_CUDA(cudaStreamSynchronize(st));
    if (h_err) return arg_error("the arc lengths of the Monte Carlo nodes must be strictly increasing");
    if (stats) {
        float ms = 0.f;
        INTERP_CUDA(cudaEventElapsedTime(&ms, ev[0], ev[1]));
        stats->post_ms = ms;
        // lengths, arc length, knot gather, knot check, [spline factor, spline columns], interpolation, scatter
        stats->launches += (kind == SDD_INTERP_SPLINE && nk > 2) ? 8 : 6;
        stats->h2d_bytes += 2 * (uint64_t)n_nodes * sizeof(double) + (uint64_t)nk * sizeof(int32_t) +
                            2 * (uint64_t)nk * V * sizeof(double);
        stats->d2h_bytes += 2 * (uint64_t)ob * sizeof(double) + sizeof(int);
    }
    return mc;
}
