// Double-precision walk (the parity mode).
//
// Every quantity of the walk is FP64 and every discrete decision (exit on
// overshoot, bridge hit, material of a point, counts) is taken with the
// expressions of their definitions in absolute coordinates, so that on the
// same Philox streams the walks agree path by path with any other FP64
// implementation of the same definitions, up to the last-ulp differences of
// log/sin/cos.  Compiled with -fmad=false: no product is fused into a sum.
//
// Steps (Sec. 3.1): uniforms (w + 1/2) 2^-32; W = sqrt(-2 ln u0)
// (cos 2 pi u1, sin 2 pi u1); beta' = beta + sqrt(dt) W; overshoot ->
// theta = d / (d - d') (first-exit-time estimate, second case); both inside
// -> hit iff min_w 2 d_w d'_w / dt <= -ln U (first case with kappa_i = 1);
// else the step counts for the material of beta'.
//
// What bounds it: the FP64 pipe, which takes a warp instruction every 64
// cycles on a quarter of an SM, however many of its lanes are active.  So the
// common step has no FP64 operation but the normals, the move and the material
// test, and a warp with few walks shares them among its lanes (cooperative
// rounds).
#include "walk_sched.cuh"
#include "walk_tm.cuh"

namespace sdd {

// (w + 1/2) 2^-32, the exact value: w and the half as mantissa bits of a double
// in [1, 2), less one (one FP64 operation; a conversion, a sum and a product
// are three).
__device__ __forceinline__ double uni32(uint32_t w) {
    return __hiloint2double((int)(0x3ff00000u | (w >> 12)), (int)((w << 20) | 0x80000u)) - 1.0;
}

template <int KMAX_, int GEO>
struct WalkerF64 {
    using Real = double;
    static constexpr int KMAX = KMAX_;
    static constexpr bool kCoop = true, kAlone = false, kEvents = false, kTurns = false;  // every walk in cooperative rounds
    static constexpr bool kGrouped = false;  // one queue (a grouped plan's order is one queue too)
    static constexpr int kMinCTAs = 2;       // the FP64 pipe is busy with 16 warps an SM
    using Occ = uint32_t;
    using HistT = uint32_t;
    static constexpr int kStored = KMAX - 1;
    static constexpr int kHist = 1;
    static constexpr int kPend = 6;
    static constexpr int kCnt = KMAX > 1 ? KMAX - 1 : 1;

    double x, z;
    uint32_t n;
    uint32_t cnt[kCnt];
    uint32_t path, nid;
    double *pend;  // the lane's column of the exiting steps that wait for their records

    __device__ static int material(const ModelDev &M, double x, double z) {
        if (GEO == GEO_RASTER) {
            const double fx = floor((x - M.xmin) * M.sx);
            const double fz = floor((z - M.zmin) * M.sz);
            long long ix = (long long)fx, iz = (long long)fz;
            if (ix < 0) ix = 0;
            if (ix > M.nx - 1) ix = M.nx - 1;
            if (iz < 0) iz = 0;
            if (iz > M.nz - 1) iz = M.nz - 1;
            return (int)__ldg(M.raster + iz * (long long)M.nx + ix);
        } else {
            int m = (z >= 0.0) ? M.bg_earth : M.bg_air;
            for (int s = 0; s < M.n_shapes; ++s) {
                const ShapeDev &S = M.shapes[s];
                const double *v = S.d;
                bool in;
                if (S.kind == 0) {
                    in = (x >= v[0] && x < v[1] && z >= v[2] && z < v[3]);
                } else {
                    const double sg = S.dsign;
                    const double e0 = sg * ((v[2] - v[0]) * (z - v[1]) - (v[3] - v[1]) * (x - v[0]));
                    const double e1 = sg * ((v[4] - v[2]) * (z - v[3]) - (v[5] - v[3]) * (x - v[2]));
                    const double e2 = sg * ((v[0] - v[4]) * (z - v[5]) - (v[1] - v[5]) * (x - v[4]));
                    in = (e0 >= 0.0 && e1 >= 0.0 && e2 >= 0.0);
                }
                if (in) m = S.mat;
            }
            return m;
        }
    }

    __device__ __forceinline__ void bind(HistT *, double *p) { pend = p; }

    __device__ __forceinline__ void counts(const ModelDev &, uint32_t, uint32_t *c) const {
#pragma unroll
        for (int j = 0; j < kCnt; ++j) c[j] = cnt[j];
    }

    __device__ __forceinline__ static void count(uint32_t (&c)[kCnt], int m) {
#pragma unroll
        for (int j = 1; j < KMAX; ++j) c[j - 1] += (m == j) ? 1u : 0u;
    }

    __device__ __forceinline__ void start(const ModelDev &, const WalkArgs &, const WarpState &S, uint32_t path_, int) {
        x = S.nx0;
        z = S.nz0;
        n = 0;
#pragma unroll
        for (int j = 0; j < kCnt; ++j) cnt[j] = 0;
        path = path_;
        nid = S.nid;
    }

    __device__ static void place(const ModelDev &M, double x, double z, double xn, double zn,
                                 double th, int w, ExitInfo<double> &ei) {
        ei.th = th;
        ei.wall = w;
        ei.x = x + th * (xn - x);
        ei.z = z + th * (zn - z);
        if (w == 0) ei.x = M.xmin;
        if (w == 1) ei.x = M.xmax;
        if (w == 2) ei.z = M.zmin;
        if (w == 3) ei.z = M.zmax;
    }

    // The Euler increment sqrt(dt) W of a step from its Philox words.
    __device__ __forceinline__ static double2 increment(const WalkArgs &A, uint32_t wa, uint32_t wb) {
        const double u0 = uni32(wa), u1 = uni32(wb);
        const double rho = sqrt(-2.0 * log(u0));
        const double ang = 6.283185307179586 * u1;
        double sn, cs;
        sincos(ang, &sn, &cs);
        return make_double2(A.sdt * (rho * cs), A.sdt * (rho * sn));
    }

    // Whether x is certainly further than the reach T of the bridge test from
    // both walls (WalkArgs::clear): the high word of a double, with its sign
    // folded in, orders like the double, so integer compares of high words
    // decide, on the safe side.
    __device__ __forceinline__ static int order_hi(double v) {
        const int h = __double2hiint(v);
        return h ^ ((h >> 31) & 0x7fffffff);
    }
    __device__ __forceinline__ static bool clear_of_walls(const WalkArgs &A, double x, double z) {
        const int hx = order_hi(x), hz = order_hi(z);
        return hx > A.clear[0] && hx < A.clear[1] && hz > A.clear[2] && hz < A.clear[3];
    }

    // Whether step k, (x0, z0) -> (xn, zn), ends the walk; u: its bridge
    // uniform, negative on an overshoot.  All walls' products are compared
    // before the one division: min_w fl(q_w / dt) = fl(min_w q_w / dt).
    __device__ static bool reaches_wall(const ModelDev &M, const WalkArgs &A, uint32_t path, uint32_t nid, uint32_t k,
                                        double x0, double z0, double xn, double zn, double &u) {
        const double d[4] = {x0 - M.xmin, M.xmax - x0, z0 - M.zmin, M.zmax - z0};
        const double dn[4] = {xn - M.xmin, M.xmax - xn, zn - M.zmin, M.zmax - zn};
        u = -1.0;
        if (dn[0] <= 0.0 || dn[1] <= 0.0 || dn[2] <= 0.0 || dn[3] <= 0.0) return true;
        double q = 2.0 * d[0] * dn[0];
#pragma unroll
        for (int w = 1; w < 4; ++w) {
            const double e = 2.0 * d[w] * dn[w];
            if (e < q) q = e;
        }
        // -ln U <= 33 ln 2 < 23 for U >= 2^-33: no uniform can hit above 23
        if (q > 23.000001 * A.dt) return false;
        const double best = q / A.dt;
        if (!(best <= 23.0)) return false;
        const uint4 b = philox4x32_10(make_uint4(k, path, nid, 1u), A.key0, A.key1);
        u = uni32(b.x);
        return best <= -log(u);
    }

    __device__ __forceinline__ static void put_exit(double *p, double x0, double z0, double xn, double zn, double u,
                                                    uint32_t k) {
        p[0] = x0;
        p[32] = z0;
        p[64] = xn;
        p[96] = zn;
        p[128] = u;
        p[160] = __hiloint2double(0, (int)k);
    }

    // The exiting step as put_exit() left it.
    __device__ __forceinline__ void get_exit(double &x0, double &z0, double &xn, double &zn, double &u,
                                             uint32_t &k) const {
        x0 = pend[0];
        z0 = pend[32];
        xn = pend[64];
        zn = pend[96];
        u = pend[128];
        k = (uint32_t)__double2loint(pend[160]);
    }

    // The exit record of an ended walk (tr: it was truncated), with the
    // expressions of the definitions.  For 32 walks at once: a walk alone held
    // the FP64 pipe as long.
    static constexpr bool kLate = true;
    __device__ __forceinline__ static void finish(const ModelDev &M, const WalkArgs &A, int, bool tr, double x0,
                                                  double z0, double xn, double zn, double u, ExitInfo<double> &ei) {
        ei.mlast = material(M, x0, z0);
        if (tr) {
            ei.x = x0; ei.z = z0; ei.th = 0.0; ei.wall = 0;
            return;
        }
        const double d[4] = {x0 - M.xmin, M.xmax - x0, z0 - M.zmin, M.zmax - z0};
        const double dn[4] = {xn - M.xmin, M.xmax - xn, zn - M.zmin, M.zmax - zn};
        double best = 2.0;
        int bw = 0;
        if (u < 0.0) {
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                if (dn[w] <= 0.0) {
                    const double t = d[w] / (d[w] - dn[w]);
                    if (t < best) { best = t; bw = w; }
                }
            }
        } else {
            best = 2.0 * d[0] * dn[0] / A.dt;
#pragma unroll
            for (int w = 1; w < 4; ++w) {
                const double e = 2.0 * d[w] * dn[w] / A.dt;
                if (e < best) { best = e; bw = w; }
            }
            best = best / -log(u);
        }
        place(M, x0, z0, xn, zn, best, bw, ei);
    }

    // Cooperative rounds (scheduler): as in the single-precision walk; the
    // moves are one addition a step and coordinate, and two steps cost about
    // 110 FP64 operations a lane.  7 nodes x 2001 walks at dt 1e-3: 21.2 ms
    // with one walk a lane (280 FP64 operations a step, a warp as long as its
    // longest walk), 1.8 ms so.
    using CoopInc = double2;
    struct Coop {
        double X, Z;
        uint32_t n, path, nid, owner;
        uint32_t cnt[kCnt];
        double X0, Z0, X1, Z1, X2, Z2, U;
    };

    __device__ __forceinline__ void coop_begin(Coop &c, int owner, int) const {
        c.X = __shfl_sync(kFull, x, owner);
        c.Z = __shfl_sync(kFull, z, owner);
        c.n = __shfl_sync(kFull, n, owner);
        c.path = __shfl_sync(kFull, path, owner);
        c.nid = __shfl_sync(kFull, nid, owner);
        c.owner = (uint32_t)owner;
#pragma unroll
        for (int j = 0; j < kCnt; ++j) c.cnt[j] = 0;
    }

    __device__ __forceinline__ static int coop_round(const ModelDev &M, const WalkArgs &A, Coop &c, CoopInc *buf,
                                                     uint32_t q, int per, bool in) {
        const uint4 w = philox_rk(make_uint4((c.n >> 1) + q, c.path, c.nid, 0u), A.rk0, A.rk1);
        double2 a, b;
        // one copy of the normals' code, run twice: it is most of the round
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const double2 d = increment(A, h ? w.z : w.x, h ? w.w : w.y);
            if (in) buf[2 * q + h] = d;
            a = h ? a : d;
            b = d;
        }
        __syncwarp();
        double X = c.X, Z = c.Z;
#pragma unroll 4
        for (int p = 0; p < per - 1; ++p) {
            const double2 u = buf[2 * p], v = buf[2 * p + 1];
            if (p < (int)q) {
                X = X + u.x;
                Z = Z + u.y;
                X = X + v.x;
                Z = Z + v.y;
            }
        }
        c.X0 = X;
        c.Z0 = Z;
        c.X1 = X + a.x;
        c.Z1 = Z + a.y;
        c.X2 = c.X1 + b.x;
        c.Z2 = c.Z1 + b.y;
        const uint32_t k = c.n + 2u * q;
        if (!in || k >= A.max_steps) return 0;
        const bool f0 = clear_of_walls(A, c.X0, c.Z0), f1 = clear_of_walls(A, c.X1, c.Z1);
        const bool f2 = clear_of_walls(A, c.X2, c.Z2);
        if (!(f0 && f1 && f2)) {
#pragma unroll 1
            for (int h = 0; h < 2; ++h)
                if (reaches_wall(M, A, c.path, c.nid, k + h, h ? c.X1 : c.X0, h ? c.Z1 : c.Z0, h ? c.X2 : c.X1,
                                 h ? c.Z2 : c.Z1, c.U))
                    return 1 + h;
        }
        return k + 2u >= A.max_steps ? 3 : 0;
    }

    __device__ __forceinline__ static void coop_count(const ModelDev &M, Coop &c, int k) {
        if (k > 0) count(c.cnt, material(M, c.X1, c.Z1));
        if (k > 1) count(c.cnt, material(M, c.X2, c.Z2));
    }

    __device__ __forceinline__ void coop_next(Coop &c, int per, int last) {
        c.X = __shfl_sync(kFull, c.X2, last);
        c.Z = __shfl_sync(kFull, c.Z2, last);
        c.n += 2u * (uint32_t)per;
    }

    __device__ __forceinline__ void coop_put(const Coop &c, int code, uint32_t q, int lane) const {
        double *p = pend + ((int)c.owner - lane);
        const uint32_t k = c.n + 2u * q;
        if (code == 1) put_exit(p, c.X0, c.Z0, c.X1, c.Z1, c.U, k);
        if (code == 2) put_exit(p, c.X1, c.Z1, c.X2, c.Z2, c.U, k + 1u);
        if (code == 3) put_exit(p, c.X2, c.Z2, c.X2, c.Z2, 0.0, k + 2u);
    }

    __device__ __forceinline__ void coop_end(const Coop &c, unsigned seg, int per, int base, bool mine) {
        const double ex = __shfl_sync(kFull, c.X2, base + per - 1), ez = __shfl_sync(kFull, c.Z2, base + per - 1);
        const uint32_t m = __shfl_sync(kFull, c.n, base) + 2u * (uint32_t)per;
        if (mine) {
            x = ex;
            z = ez;
            n = m;
        }
#pragma unroll
        for (int j = 0; j < kCnt; ++j) {
            const uint32_t v = seg ? __reduce_add_sync(seg, c.cnt[j]) : 0u;
            const uint32_t g = __shfl_sync(kFull, v, base);
            if (mine) cnt[j] += g;
        }
    }

    __device__ static void to_abs(const ModelDev &, double X, double Z, double &ox, double &oz) {
        ox = X;
        oz = Z;
    }

    __device__ static double2 column(double kr, double ki, double z) {
        if (z >= 0.0) {
            const double a = exp(-kr * z);
            double s, c;
            sincos(ki * z, &s, &c);
            return make_double2(a * c, -a * s);
        }
        return make_double2(1.0 - kr * z, -(ki * z));
    }

    __device__ static double2 sample(const ModelDev &M, const SharedTables &T, const WalkArgs &A,
                                     int, int e, double x, double z, double th, int wall, int mlast,
                                     const uint32_t *c) {
        const double dt = A.dt;
        const double *kap = T.kappa + e * M.K;
        double ph = 0.0;
#pragma unroll
        for (int k = 0; k < KMAX; ++k)
            if (k < M.K) ph += kap[k] * ((double)c[k] * dt);
        ph += kap[mlast] * (th * dt);
        ph *= 0.5;
        double sw, cw;
        sincos(ph, &sw, &cw);
        double2 g;
        if (M.g_kind == 1) {
            const double *a = M.g_coef;
            g = make_double2(a[0] + a[2] * x + a[4] * z, a[1] + a[3] * x + a[5] * z);
        } else if (M.g_kind == 2) {
            g = make_double2(x * x - z * z, 0.0);
        } else {
            const EvalDev &E = T.ev[e];
            if (wall == 0) {
                g = column(E.kl_re, E.kl_im, z);
            } else if (wall == 1) {
                g = column(E.kr_re, E.kr_im, z);
            } else {
                const double t = (x - M.xmin) / (M.xmax - M.xmin);
                const double lr = wall == 2 ? E.tl_re : E.bl_re, li = wall == 2 ? E.tl_im : E.bl_im;
                const double rr = wall == 2 ? E.tr_re : E.br_re, ri = wall == 2 ? E.tr_im : E.br_im;
                g = make_double2((1.0 - t) * lr + t * rr, (1.0 - t) * li + t * ri);
            }
        }
        // (cw - i sw)(g.x + i g.y)
        return make_double2(cw * g.x + sw * g.y, cw * g.y - sw * g.x);
    }
};

template <int KMAX, int GEO>
static cudaError_t launch_one(const ModelDev &M, const WalkArgs &A, int grid, int block,
                              cudaStream_t s) {
    const size_t sm = shared_bytes<WalkerF64<KMAX, GEO>>(block / 32, M.E, M.K);
    auto k = walk_kernel<WalkerF64<KMAX, GEO>>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<grid, block, sm, s>>>(M, A);
    return cudaGetLastError();
}

template <int KMAX, int GEO>
static int occ_one(int block, int E, int K) {
    const size_t sm = shared_bytes<WalkerF64<KMAX, GEO>>(block / 32, E, K);
    auto k = walk_kernel<WalkerF64<KMAX, GEO>>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, block, sm) != cudaSuccess) return 0;
    return n;
}

#define SDD_DISPATCH(FN, ...)                                                   \
    switch (kmax * 2 + geo) {                                                   \
    case 4: return FN<2, GEO_SHAPES>(__VA_ARGS__);                              \
    case 5: return FN<2, GEO_RASTER>(__VA_ARGS__);                              \
    case 6: return FN<3, GEO_SHAPES>(__VA_ARGS__);                              \
    case 7: return FN<3, GEO_RASTER>(__VA_ARGS__);                              \
    case 8: return FN<4, GEO_SHAPES>(__VA_ARGS__);                              \
    case 9: return FN<4, GEO_RASTER>(__VA_ARGS__);                              \
    case 16: return FN<8, GEO_SHAPES>(__VA_ARGS__);                             \
    case 17: return FN<8, GEO_RASTER>(__VA_ARGS__);                             \
    default: break;                                                             \
    }

// The TM parity walk (vertical strips).
template <int KMAX>
static cudaError_t launch_tm(const ModelDev &M, const WalkArgs &A, int grid, int block, cudaStream_t s) {
    using W = WalkerTM<double, KMAX>;
    const size_t sm = shared_bytes<W>(block / 32, M.E, M.K);
    auto k = walk_kernel<W>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<grid, block, sm, s>>>(M, A);
    return cudaGetLastError();
}

template <int KMAX>
static int occ_tm(int block, int E, int K) {
    using W = WalkerTM<double, KMAX>;
    const size_t sm = shared_bytes<W>(block / 32, E, K);
    auto k = walk_kernel<W>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, block, sm) != cudaSuccess) return 0;
    return n;
}

#define SDD_TM_DISPATCH(FN, ...)                                                \
    switch (kmax) {                                                             \
    case 2: return FN<2>(__VA_ARGS__);                                          \
    case 3: return FN<3>(__VA_ARGS__);                                          \
    case 4: return FN<4>(__VA_ARGS__);                                          \
    case 8: return FN<8>(__VA_ARGS__);                                          \
    default: break;                                                             \
    }

cudaError_t launch_walk_f64(int kmax, int geo, const ModelDev &M, const WalkArgs &A, int grid,
                            int block, cudaStream_t s) {
    if (geo == GEO_TM) {
        SDD_TM_DISPATCH(launch_tm, M, A, grid, block, s)
        return cudaErrorInvalidValue;
    }
    SDD_DISPATCH(launch_one, M, A, grid, block, s)
    return cudaErrorInvalidValue;
}

int occupancy_f64(int kmax, int geo, int block, int E, int K) {
    if (geo == GEO_TM) {
        SDD_TM_DISPATCH(occ_tm, block, E, K)
        return 0;
    }
    SDD_DISPATCH(occ_one, block, E, K)
    return 0;
}

}  // namespace sdd
