// Single-precision walk (the throughput path).
//
// Position stepping, wall tests, material lookup and the per-walk phase
// factor are FP32; the per-material step counts are integers; the phase sum is
// in 64-bit fractions of a turn and the Monte Carlo sums are FP64.  Compiled
// with -ftz=true -prec-div=false -prec-sqrt=false.
//
// One Euler-Maruyama step of Sec. 3.1 (discretised process, kappa_i = 1):
//   (u0, u1)  two uniforms (w mod 2^23 + 1/2) 2^-23 from one Philox call,
//   r^2 = -2 ln(u0) dt,  beta' = beta + r (cos 2 pi u1, sin 2 pi u1),
// then the boundary rule of the first-exit-time estimate: overshoot ->
// theta = d / (d + |d'|) on the first wall reached; else the Brownian-bridge
// test 2 d d' / dt <= -ln U_gamma with one uniform per step (18 spare bits of
// the step's Philox words); else the step's time goes to the material of
// beta' (Sec. 3.1, no regime change for TE).
//
// The walk runs in centred coordinates X = x - xc, Z = z - zc, so the
// distance to the nearer wall of each pair is h - |X|.  Two steps share one
// Philox call (words 0,1 for the even step, 2,3 for the odd one), and one
// call of iterate() runs 8 steps.
//
// What bounds it: instruction issue.  50 issue slots a step (64 nodes x 1e5
// walks, dt 1e-4; 62 before the signs without flushing, one wall branch for
// two steps and exits recorded apart) at 69 % of the issue rate, 5.5e11
// walk-steps/s; the rest of the rate goes to the wide multiplies of Philox
// (dispatch and math-pipe stalls, with 2.4 of 6 warps eligible on average).
// The kernels take the 80 registers of 3 CTAs an SM and most of them spill
// (64 bytes the one-shape programs, up to 146 the TM walk), in what surrounds
// the steps: local loads and stores are 0.25 % of the instructions with walks
// of 400 steps, 0.06 % with 4000.
// Tried without gain: region counters on the FMA pipe (40.2 -> 40.0 ms), the
// next iteration's words formed between the steps (43.6), 16 steps an
// iteration (39.4 there, but 13.3 -> 16.2 ms at dt 1e-3), 2 or 4 CTAs an SM.
#include <type_traits>

#include "walk_sched.cuh"
#include "walk_tm.cuh"

namespace sdd {

// Uniforms of the single-precision walk: the low 23 bits of a Philox word as
// the mantissa of a float in [1, 2); u = (w mod 2^23 + 1/2) 2^-23 exactly
// (1.m - (1 - 2^-24), an exact difference by Sterbenz' lemma).
__device__ __forceinline__ float one_plus(uint32_t w) { return mant_one(w); }
__device__ __forceinline__ float uni23(uint32_t w) { return one_plus(w) - 0.99999994039535522f; }

// Occupation counters.  KMAX = 2: the step count of material 1.  KMAX = 3, 4:
// power sums s_p = sum over steps of m^p (p = 1 .. KMAX-1), which determine
// the counts of materials 1 .. KMAX-1 (a Vandermonde system, solved once at
// the exit).  KMAX = 8: a per-lane histogram in shared memory, one shared
// atomic add per step.
template <int KMAX>
struct Occupancy {
    uint32_t s[KMAX > 1 ? KMAX - 1 : 1];
    __device__ __forceinline__ void bind(uint32_t) {}
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < (KMAX > 1 ? KMAX - 1 : 1); ++j) s[j] = 0;
    }
    __device__ __forceinline__ void add(int m) {
        const uint32_t u = (uint32_t)m;
        if (KMAX == 2) {
            s[0] += u;
        } else if (KMAX == 3) {
            s[0] += u;
            s[1] += u * u;
        } else if (KMAX == 4) {
            const uint32_t u2 = u * u;
            s[0] += u;
            s[1] += u2;
            s[2] += u2 * u;
        } else {
#pragma unroll
            for (int j = 1; j < KMAX; ++j) s[j - 1] += (m == j) ? 1u : 0u;
        }
    }
    // counts of materials 1 .. KMAX-1
    __device__ __forceinline__ void counts(uint32_t *c) const {
        if (KMAX == 2) {
            c[0] = s[0];
        } else if (KMAX == 3) {
            // s1 = c1 + 2 c2, s2 = c1 + 4 c2
            const uint32_t c2 = (s[1] - s[0]) >> 1;
            c[1] = c2;
            c[0] = s[0] - 2u * c2;
        } else if (KMAX == 4) {
            // s1 = c1 + 2 c2 + 3 c3, s2 = c1 + 4 c2 + 9 c3, s3 = c1 + 8 c2 + 27 c3
            const uint32_t c3 = (s[2] - 3u * s[1] + 2u * s[0]) / 6u;
            const uint32_t c2 = (s[1] - s[0] - 6u * c3) >> 1;
            c[2] = c3;
            c[1] = c2;
            c[0] = s[0] - 2u * c2 - 3u * c3;
        } else {
#pragma unroll
            for (int j = 0; j < KMAX - 1; ++j) c[j] = s[j];
        }
    }
};

template <>
struct Occupancy<8> {
    uint32_t base;  // shared address of hist[0][lane]; material m at base + 128 m
    __device__ __forceinline__ void bind(uint32_t a) { base = a; }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < 8; ++j) asm volatile("st.shared.u32 [%0], %1;" ::"r"(base + 128u * j), "r"(0u));
    }
    __device__ __forceinline__ void add(int m) {
        asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(base + ((uint32_t)m << 7)), "r"(1u));
    }
    __device__ __forceinline__ void counts(uint32_t *c) const {
#pragma unroll
        for (int j = 1; j < 8; ++j) {
            uint32_t v;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(base + 128u * j));
            c[j - 1] = v;
        }
    }
};

// Region counters of the one-shape programs (GC_CONTACT, GC_RECT1, GC_TRI1): ce steps
// on the earth side of the surface, cs steps inside the shape.  The shape
// lies wholly on one side of the surface, so these two give every
// material's count at the exit (WalkerF32::counts).
struct Regions {
    uint32_t ce, cs;
    __device__ __forceinline__ void bind(uint32_t) {}
    __device__ __forceinline__ void clear() { ce = 0u; cs = 0u; }
};

// GC: the material-lookup program (GeoCode).  Up to four shapes' parameters are
// read with compile-time indices, so every one is an immediate constant operand.
template <int KMAX_, int GC>
struct WalkerF32 {
    using Real = float;
    static constexpr int KMAX = KMAX_;
    // records: step counts of materials 1..K-1 (material 0 from the total)
    using Occ = uint32_t;
    using HistT = uint32_t;
    static constexpr int kStored = KMAX - 1;
    static constexpr int kHist = KMAX == 8 ? 8 : 1;
    static constexpr bool kGrouped = GC == GC_RASTER_MULTI;
    // 24 resident warps whose iterations carry four independent Philox
    // chains keep the issue slots fuller than 32 warps in 64 registers
    static constexpr int kMinCTAs = 3;

    // one-shape programs count regions (two predicated adds per step in
    // place of the material selects and the power sums)
    static constexpr bool kRegions = GC == GC_CONTACT || GC == GC_RECT1 || GC == GC_TRI1;

    float X, Z, dmin;  // centred position, distance to the nearest wall
    uint32_t n;        // Euler steps accepted (even at the start of iterate)
    typename std::conditional<kRegions, Regions, Occupancy<KMAX>>::type occ;
    uint32_t pre_x, pre_y;
    const uint32_t *tco;  // GC_RASTER_MULTI: the tile map of this walk's model

    // Shared address of the lane's column of WarpSmem::pend: the step that
    // ends a walk puts there the point before it, its proposed point, its
    // bridge uniform (negative: it overshot a wall) and its number.
    // They go into the warp's ring as they are, and finish() turns them into
    // the exit record when 32 have gathered.  Through shared memory, not
    // registers: the eight exits of
    // an unrolled iteration then leave nothing but the lane's state to merge
    // (in registers it cost 4.6 issue slots a step in moves).
    uint32_t pend;

    __device__ __forceinline__ static bool in_rect(const ShapeDev &S, float X, float Z) {
        return X >= S.f[0] && X < S.f[1] && Z >= S.f[2] && Z < S.f[3];
    }
    __device__ __forceinline__ static bool in_tri(const ShapeDev &S, float X, float Z) {
        return fmaf(S.f[0], X, fmaf(S.f[1], Z, S.f[2])) >= 0.f &&
               fmaf(S.f[3], X, fmaf(S.f[4], Z, S.f[5])) >= 0.f &&
               fmaf(S.f[6], X, fmaf(S.f[7], Z, S.f[8])) >= 0.f;
    }

    __device__ __forceinline__ int material(const ModelDev &M, float X, float Z) const {
        if (GC == GC_RASTER || GC == GC_RASTER_MULTI) {
            // round(v - 1/2) = floor(v) for v = (X + hw) sx >= 0 (magic-number
            // rounding), plus kTile: the index into the tile map, which starts
            // one tile before the raster.  A point inside the domain gives a cell
            // index in -1 .. n (rounding can reach one past an edge), and the
            // map's margin tiles repeat the edge cells, so no clamp is needed.
            // Two-level lookup: the coarse entry (L1-resident) is the material
            // of a uniform tile, else the tile's cells in the pool.
            //
            // The magic number's own bits stay in the indices (its low four
            // are zero) and leave the tile index as one constant, tbias.  The
            // second load is predicated, not branched around: a tenth of the
            // points lie in mixed tiles, so most warps have one, and a branch
            // was taken on nearly every step.  With this, and the lookups of
            // two steps side by side, 57 nodes x 2e5 walks at dt 1e-3: K = 3
            // 14.9 -> 13.9 ms, K = 4 12.8 -> 11.9 ms, K = 5 12.7 -> 9.9 ms (8
            // materials no longer look an iteration's steps up together after
            // it); 12 models 4.63 -> 3.84 ms.
            const uint32_t bx = __float_as_uint(fmaf(X, M.fsx, M.fox) + 12582912.0f);
            const uint32_t bz = __float_as_uint(fmaf(Z, M.fsz, M.foz) + 12582912.0f);
            const char *co = reinterpret_cast<const char *>(GC == GC_RASTER_MULTI ? tco : M.tcoarse);
            const uint32_t tile = (bz >> kTileShift) * (uint32_t)M.ntx + (bx >> kTileShift) - M.tbias;
            const uint32_t c = __ldg(reinterpret_cast<const uint32_t *>(co) + tile);
            const uint32_t cell = (c << (2 * kTileShift)) | ((bz & (kTile - 1)) << kTileShift) | (bx & (kTile - 1));
            uint32_t m = c & 0xffu;
            asm("{\n\t.reg .pred mixed;\n\tsetp.ge.s32 mixed, %1, 0;\n\t@mixed ld.global.nc.u8 %0, [%2];\n\t}"
                : "+r"(m) : "r"(c), "l"(co + M.tpool_off + (uint64_t)cell));
            return (int)m;
        }
        const int m = (Z >= M.fzs) ? M.bg_earth : M.bg_air;
        if (GC == GC_LAYER) return m;
        if (GC == GC_RECT1) return in_rect(M.shapes[0], X, Z) ? M.shapes[0].mat : m;
        if (GC == GC_CONTACT) return (Z >= M.fzs && X >= M.shapes[0].f[0]) ? M.shapes[0].mat : m;
        if (GC == GC_TRI1) return in_tri(M.shapes[0], X, Z) ? M.shapes[0].mat : m;
        // up to 4 shapes unrolled (immediate constants), more in a loop: 16
        // unrolled tests in each of the iteration's 8 steps overflow the
        // instruction cache (64 nodes x 5e4 walks through 6 shapes, dt 1e-3:
        // 90.7 ms with 4 materials and 43.4 with 8, 15.3 and 15.2 in the loop)
        int r = m;
        auto test = [&](const ShapeDev &S) {
            const bool in = S.kind == 0 ? in_rect(S, X, Z) : in_tri(S, X, Z);
            r = in ? S.mat : r;
        };
        if (GC == GC_SHAPES4) {
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (s < M.n_shapes) test(M.shapes[s]);
        } else {
#pragma unroll 1
            for (int s = 0; s < M.n_shapes; ++s) test(M.shapes[s]);
        }
        return r;
    }

    // The step at (X, Z) into the region counters: the earth test and the
    // shape test of material() as predicates, each adding one to its counter
    // (compares with .ftz, as the unit's float compares).
    __device__ __forceinline__ void count_regions(const ModelDev &M, float X, float Z) {
        if (GC == GC_CONTACT) {
            asm("{\n\t.reg .pred pe, ps;\n\t"
                "setp.ge.ftz.f32 pe, %3, %4;\n\t"
                "setp.ge.and.ftz.f32 ps, %2, %5, pe;\n\t"
                "@pe add.u32 %0, %0, 1;\n\t"
                "@ps add.u32 %1, %1, 1;\n\t}"
                : "+r"(occ.ce), "+r"(occ.cs)
                : "f"(X), "f"(Z), "f"(M.fzs), "f"(M.shapes[0].f[0]));
        } else if (GC == GC_TRI1) {
            // the three edge functions as in in_tri(), the compares chained
            const ShapeDev &S = M.shapes[0];
            const float e0 = fmaf(S.f[0], X, fmaf(S.f[1], Z, S.f[2]));
            const float e1 = fmaf(S.f[3], X, fmaf(S.f[4], Z, S.f[5]));
            const float e2 = fmaf(S.f[6], X, fmaf(S.f[7], Z, S.f[8]));
            asm("{\n\t.reg .pred pe, ps;\n\t"
                "setp.ge.ftz.f32 pe, %2, %3;\n\t"
                "setp.ge.ftz.f32 ps, %4, 0f00000000;\n\t"
                "setp.ge.and.ftz.f32 ps, %5, 0f00000000, ps;\n\t"
                "setp.ge.and.ftz.f32 ps, %6, 0f00000000, ps;\n\t"
                "@pe add.u32 %0, %0, 1;\n\t"
                "@ps add.u32 %1, %1, 1;\n\t}"
                : "+r"(occ.ce), "+r"(occ.cs)
                : "f"(Z), "f"(M.fzs), "f"(e0), "f"(e1), "f"(e2));
        } else {
            asm("{\n\t.reg .pred pe, ps;\n\t"
                "setp.ge.ftz.f32 pe, %3, %4;\n\t"
                "setp.ge.ftz.f32 ps, %2, %5;\n\t"
                "setp.lt.and.ftz.f32 ps, %2, %6, ps;\n\t"
                "setp.ge.and.ftz.f32 ps, %3, %7, ps;\n\t"
                "setp.lt.and.ftz.f32 ps, %3, %8, ps;\n\t"
                "@pe add.u32 %0, %0, 1;\n\t"
                "@ps add.u32 %1, %1, 1;\n\t}"
                : "+r"(occ.ce), "+r"(occ.cs)
                : "f"(X), "f"(Z), "f"(M.fzs), "f"(M.shapes[0].f[0]), "f"(M.shapes[0].f[1]),
                  "f"(M.shapes[0].f[2]), "f"(M.shapes[0].f[3]));
        }
    }

    // The accepted step at (x, z) into the occupation counters.
    __device__ __forceinline__ void count_step(const ModelDev &M, float x, float z) {
        if constexpr (kRegions) count_regions(M, x, z);
        else occ.add(material(M, x, z));
    }

    // Counts of materials 1 .. KMAX-1 after nocc counted steps.  Region
    // counters: the shape has cs; with the shape in the earth the earth
    // background has ce - cs and the air nocc - ce, with the shape in the air
    // the earth has ce and the air nocc - ce - cs.
    __device__ __forceinline__ void counts(const ModelDev &M, uint32_t nocc, uint32_t *c) const {
        if constexpr (kRegions) {
            const uint32_t ce = occ.ce, cs = occ.cs;
            const uint32_t ear = M.shape_air ? ce : ce - cs;
            const uint32_t air = nocc - ce - (M.shape_air ? cs : 0u);
            const int ma = M.bg_air, me = M.bg_earth, msh = M.shapes[0].mat;
#pragma unroll
            for (int j = 1; j < KMAX; ++j)
                c[j - 1] = (ma == j ? air : 0u) + (me == j ? ear : 0u) + (msh == j ? cs : 0u);
        } else {
            occ.counts(c);
        }
    }
    __device__ __forceinline__ void bind(HistT *h, float *p) {
        occ.bind((uint32_t)__cvta_generic_to_shared(h));
        pend = (uint32_t)__cvta_generic_to_shared(p);
    }
    static constexpr int kPend = 6;

    __device__ __forceinline__ void start(const ModelDev &M, const WalkArgs &A, const WarpState &S, uint32_t path,
                                          int model) {
        const uint32_t node_id = S.nid;
        if (GC == GC_RASTER_MULTI) tco = A.models[model].tcoarse;
        X = S.fx0;
        Z = S.fz0;
        dmin = fminf(M.fhw - fabsf(X), M.fhh - fabsf(Z));
        n = 0;
        occ.clear();
        pre_x = __umulhi(0xCD9E8D57u, node_id) ^ path ^ A.rk0[0];
        pre_y = 0xCD9E8D57u * node_id;
    }

    __device__ __forceinline__ void put_exit(float X0, float Z0, float Xn, float Zn, float U, uint32_t k) const {
        asm volatile("st.shared.f32 [%0], %1;\n\tst.shared.f32 [%0+128], %2;\n\tst.shared.f32 [%0+256], %3;\n\t"
                     "st.shared.f32 [%0+384], %4;\n\tst.shared.f32 [%0+512], %5;\n\tst.shared.u32 [%0+640], %6;"
                     ::"r"(pend), "f"(X0), "f"(Z0), "f"(Xn), "f"(Zn), "f"(U), "r"(k) : "memory");
    }
    __device__ __forceinline__ void get_exit(float &X0, float &Z0, float &Xn, float &Zn, float &U, uint32_t &k) const {
        asm volatile("ld.shared.f32 %0, [%6];\n\tld.shared.f32 %1, [%6+128];\n\tld.shared.f32 %2, [%6+256];\n\t"
                     "ld.shared.f32 %3, [%6+384];\n\tld.shared.f32 %4, [%6+512];\n\tld.shared.u32 %5, [%6+640];"
                     : "=f"(X0), "=f"(Z0), "=f"(Xn), "=f"(Zn), "=f"(U), "=r"(k) : "r"(pend) : "memory");
    }

    __device__ __forceinline__ static void place(const ModelDev &M, float X, float Z, float Xn, float Zn, float th,
                                                 int w, ExitInfo<float> &ei) {
        ei.th = th;
        ei.wall = w;
        ei.x = fmaf(th, Xn - X, X);
        ei.z = fmaf(th, Zn - Z, Z);
        if (w == 0) ei.x = -M.fhw;
        if (w == 1) ei.x = M.fhw;
        if (w == 2) ei.z = -M.fhh;
        if (w == 3) ei.z = M.fhh;
    }

    // Whether the step (X, Z) -> (Xn, Zn), which came within reach of a wall,
    // ends the walk.  Overshoot (dn <= 0): yes.  Both ends inside: the
    // Brownian-bridge test with one uniform for all walls: the walk touched a
    // wall iff 2 d_w d'_w / dt <= -ln U for the smallest product, tested as
    // U <= exp(-2 d_w d'_w / dt).  U is made of the 18 bits of the step's two
    // Philox words that the normals leave unused:
    // U = (high 9 bits of wa : high 9 bits of wb + 1/2) 2^-18, here as the
    // mantissa of a float in [1, 2) less 1 - 2^-19 (exact).  Every product
    // d_w d'_w is at least pn = dmin dn (the nearest distances before and
    // after the step), so U > exp(-2 pn / dt) rules out a hit without forming
    // the distances; most near-wall steps end there.
    //
    // A warp takes this branch on about every second step (one lane of 32 is
    // enough), and the code stands once per unrolled step: it holds the
    // decision alone.  What follows a hit (the wall, theta, the exit point,
    // the last material) waits for finish().
    __device__ __forceinline__ static bool reaches_wall(const ModelDev &M, const WalkArgs &A, float X0,
                                                        float Z0, float Xn, float Zn, float dn, float pn,
                                                        uint32_t wa, uint32_t wb, float &U) {
        U = __uint_as_float(0x3f800000u | ((wa >> 9) & 0x7fc000u) | ((wb >> 18) & 0x3fe0u)) - 0.99999809265136719f;
        if (dn > 0.f && U > __expf(-pn * A.f_c2dt)) return false;
        const float p0 = (X0 + M.fhw) * (Xn + M.fhw), p1 = (M.fhw - X0) * (M.fhw - Xn);
        const float p2 = (Z0 + M.fhh) * (Zn + M.fhh), p3 = (M.fhh - Z0) * (M.fhh - Zn);
        const float pmin = fminf(fminf(p0, p1), fminf(p2, p3));
        const bool hit = dn <= 0.f || !(U > __expf(-(pmin * A.f_c2dt)));
        U = dn <= 0.f ? -1.f : U;
        return hit;
    }

    // The exit record of an ended walk from what put_exit() left (tr: it was
    // truncated).  Overshoot: theta_w = d_w / (d_w - d'_w) over the walls
    // with d'_w <= 0, smallest first, ties to the first of left, right, top,
    // bottom.  Bridge hit: the wall of the smallest product (first in wall
    // order) and theta = (2 d d' / dt) / (-ln U).
    static constexpr bool kLate = true;
    __device__ __forceinline__ static void finish(const ModelDev &M, const WalkArgs &A, int model, bool tr, float X,
                                                  float Z, float pXn, float pZn, float pU, ExitInfo<float> &ei) {
        if (tr) {
            ei.x = X; ei.z = Z; ei.th = 0.f; ei.wall = 0;
        } else {
            const float d[4] = {X + M.fhw, M.fhw - X, Z + M.fhh, M.fhh - Z};
            const float e[4] = {pXn + M.fhw, M.fhw - pXn, pZn + M.fhh, M.fhh - pZn};
            float best = 2.0f;
            int bw = 0;
            if (pU < 0.f) {
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    if (e[w] <= 0.f) {
                        const float t = d[w] / (d[w] - e[w]);
                        if (t < best) { best = t; bw = w; }
                    }
                }
            } else {
                const float p0 = d[0] * e[0], p1 = d[1] * e[1], p2 = d[2] * e[2], p3 = d[3] * e[3];
                const float pmin = fminf(fminf(p0, p1), fminf(p2, p3));
                const float es = pmin * A.f_c2dt;
                bw = p0 == pmin ? 0 : (p1 == pmin ? 1 : (p2 == pmin ? 2 : 3));
                best = es / -logf(pU);
            }
            place(M, X, Z, pXn, pZn, best, bw, ei);
        }
        WalkerF32 t;
        if (GC == GC_RASTER_MULTI) t.tco = A.models[model].tcoarse;
        ei.mlast = t.material(M, X, Z);
    }

    // The part of an Euler step that does not depend on the position: the
    // step length r = sqrt(-2 ln(u0) dt) and direction of the normal pair
    // (angle 2 pi (u1 - 1/2), so cos(2 pi u1) = -cs and sin(2 pi u1) = -sn)
    // from the step's Philox words (wa, wb).
    struct Incr {
        float r, sn, cs;
    };
    __device__ __forceinline__ static Incr increment(const WalkArgs &A, uint32_t wa, uint32_t wb) {
        Incr d;
        // |.| only guards the last-ulp sign of lg2 near u0 = 1
        d.r = sqrtf(abs_bits(A.f_cdt * __log2f(uni23(wa))));
        __sincosf(fmaf(one_plus(wb), 6.28318530718f, -9.42477796077f), &d.sn, &d.cs);
        return d;
    }

    // The rest of two steps (Philox words w): the moves, one branch for both
    // wall tests, the occupation.  k: steps of this walk since n.  Returns
    // true when the walk reached the boundary.  The branch and its
    // reconvergence cost three issue slots; one for two steps took 64 nodes x
    // 1e5 walks, dt 1e-4, from 41.4 to 40.3 ms (one for four or for eight:
    // 42.8 and 42.3 ms, more live positions).
    __device__ __forceinline__ bool advance2(const ModelDev &M, const WalkArgs &A, const uint4 &w, uint32_t k) {
        const Incr a = increment(A, w.x, w.y), b = increment(A, w.z, w.w);
        const float ra = neg_bits(a.r), rb = neg_bits(b.r);
        const float X1 = fmaf(ra, a.cs, X), Z1 = fmaf(ra, a.sn, Z);
        const float d1 = fminf(M.fhw - abs_bits(X1), M.fhh - abs_bits(Z1));
        const float p1 = dmin * d1;
        const float X2 = fmaf(rb, b.cs, X1), Z2 = fmaf(rb, b.sn, Z1);
        const float d2 = fminf(M.fhw - abs_bits(X2), M.fhh - abs_bits(Z2));
        const float p2 = d1 * d2;
        if (fminf(p1, p2) <= A.f_bthr) {
            float U;
            if (p1 <= A.f_bthr && reaches_wall(M, A, X, Z, X1, Z1, d1, p1, w.x, w.y, U)) {
                put_exit(X, Z, X1, Z1, U, n + k);
                return true;
            }
            if (p2 <= A.f_bthr && reaches_wall(M, A, X1, Z1, X2, Z2, d2, p2, w.z, w.w, U)) {
                put_exit(X1, Z1, X2, Z2, U, n + k + 1u);
                count_step(M, X1, Z1);
                return true;
            }
        }
        count_step(M, X1, Z1);
        count_step(M, X2, Z2);
        X = X2;
        Z = Z2;
        dmin = d2;
        return false;
    }

    // PAIRS Philox calls, two Euler steps each, per call of iterate: the
    // per-iteration work of the scheduler loop (constants, vote, branch) is
    // shared by 2 PAIRS steps.  The calls depend only on the step counter, so
    // all of them are issued first, as independent chains the SM can overlap
    // (a walk that exits early discards the rest).  0 running, 1 exited,
    // 2 truncated (max_steps is a multiple of 8, so a walk is only truncated
    // at the end of an iteration).
    static constexpr int PAIRS = 4;

    __device__ __forceinline__ int iterate(const ModelDev &M, const WalkArgs &A, uint32_t, ExitInfo<float> &) {
        uint4 w[PAIRS];
#pragma unroll
        for (int q = 0; q < PAIRS; ++q) w[q] = philox_rk_pre((n >> 1) + q, 0u, pre_x, pre_y, A.rk0, A.rk1);
#pragma unroll
        for (int q = 0; q < PAIRS; ++q) {
            if (advance2(M, A, w[q], 2u * q)) return 1;
        }
        n += 2 * PAIRS;
        if (n >= A.max_steps) {
            put_exit(X, Z, X, Z, 0.f, n);
            return 2;
        }
        return 0;
    }

    // Cooperative rounds (scheduler): the lanes of a segment of the warp share
    // one walk.  Lane q of the segment forms the increments of pair q of the
    // round (two steps), the ones increment() gives in iterate(); every lane
    // then runs the moves of the pairs before its own, one fused multiply-add
    // a step and coordinate, and tests its own two steps.  The walk is the
    // one iterate() makes, bit for bit.
    static constexpr bool kCoop = true, kAlone = true, kEvents = false;
    using CoopInc = float4;
    struct Coop {
        float X, Z;            // the walk's position at the start of the round
        uint32_t n, kx, ky;    // its step counter and keys
        uint32_t owner;        // the lane that holds the walk
        const uint32_t *tco;
        decltype(WalkerF32::occ) occ;  // this lane's share of the occupation
        float X0, Z0, X1, Z1, X2, Z2, U;  // before, between and after the lane's two steps
    };

    __device__ __forceinline__ void coop_begin(Coop &c, int owner, int lane) const {
        c.X = __shfl_sync(kFull, X, owner);
        c.Z = __shfl_sync(kFull, Z, owner);
        c.n = __shfl_sync(kFull, n, owner);
        c.kx = __shfl_sync(kFull, pre_x, owner);
        c.ky = __shfl_sync(kFull, pre_y, owner);
        c.owner = (uint32_t)owner;
        if (GC == GC_RASTER_MULTI)
            c.tco = reinterpret_cast<const uint32_t *>(
                __shfl_sync(kFull, reinterpret_cast<unsigned long long>(tco), owner));
        if constexpr (KMAX == 8 && !kRegions) c.occ.base = occ.base + 4u * (uint32_t)(owner - lane);
        else c.occ.clear();
    }

    // One round of per pairs.  in: this lane takes part (q < per); buf: the
    // segment's increments.  0, or this lane's first event: 1 and 2, the first
    // and the second of its steps ends the walk; 3, max_steps is reached after
    // both.
    __device__ __forceinline__ static int coop_round(const ModelDev &M, const WalkArgs &A, Coop &c, CoopInc *buf,
                                                     uint32_t q, int per, bool in) {
        const uint4 w = philox_rk_pre((c.n >> 1) + q, 0u, c.kx, c.ky, A.rk0, A.rk1);
        const Incr a = increment(A, w.x, w.y), b = increment(A, w.z, w.w);
        const float ra = neg_bits(a.r), rb = neg_bits(b.r);
        if (in) {
            buf[2 * q] = make_float4(ra, a.sn, a.cs, 0.f);
            buf[2 * q + 1] = make_float4(rb, b.sn, b.cs, 0.f);
        }
        __syncwarp();
        float X = c.X, Z = c.Z;
#pragma unroll 4
        for (int p = 0; p < per - 1; ++p) {
            const float4 u = buf[2 * p], v = buf[2 * p + 1];
            if (p < (int)q) {
                X = fmaf(u.x, u.z, X);
                Z = fmaf(u.x, u.y, Z);
                X = fmaf(v.x, v.z, X);
                Z = fmaf(v.x, v.y, Z);
            }
        }
        c.X0 = X;
        c.Z0 = Z;
        c.X1 = fmaf(ra, a.cs, X);
        c.Z1 = fmaf(ra, a.sn, Z);
        c.X2 = fmaf(rb, b.cs, c.X1);
        c.Z2 = fmaf(rb, b.sn, c.Z1);
        const float d0 = fminf(M.fhw - abs_bits(c.X0), M.fhh - abs_bits(c.Z0));
        const float d1 = fminf(M.fhw - abs_bits(c.X1), M.fhh - abs_bits(c.Z1));
        const float d2 = fminf(M.fhw - abs_bits(c.X2), M.fhh - abs_bits(c.Z2));
        const float p1 = d0 * d1, p2 = d1 * d2;
        const uint32_t k = c.n + 2u * q;
        if (!in || k >= A.max_steps) return 0;
        if (p1 <= A.f_bthr && reaches_wall(M, A, c.X0, c.Z0, c.X1, c.Z1, d1, p1, w.x, w.y, c.U)) return 1;
        if (p2 <= A.f_bthr && reaches_wall(M, A, c.X1, c.Z1, c.X2, c.Z2, d2, p2, w.z, w.w, c.U)) return 2;
        return k + 2u >= A.max_steps ? 3 : 0;
    }

    // The occupation of this lane's first cnt (0 .. 2) steps of the round.
    __device__ __forceinline__ static void coop_count(const ModelDev &M, Coop &c, int cnt) {
        WalkerF32 t;
        t.occ = c.occ;
        t.tco = c.tco;
        if (cnt > 0) t.count_step(M, c.X1, c.Z1);
        if (cnt > 1) t.count_step(M, c.X2, c.Z2);
        c.occ = t.occ;
    }

    // No walk ended in the round: on to the next one (last: the lane of the
    // segment's last pair).
    __device__ __forceinline__ void coop_next(Coop &c, int per, int last) {
        c.X = __shfl_sync(kFull, c.X2, last);
        c.Z = __shfl_sync(kFull, c.Z2, last);
        c.n += 2u * (uint32_t)per;
    }

    // The lane whose step ended the walk leaves it in the owner's column.
    __device__ __forceinline__ void coop_put(const Coop &c, int code, uint32_t q, int lane) const {
        WalkerF32 t;
        t.pend = pend + 4u * (c.owner - (uint32_t)lane);
        const uint32_t k = c.n + 2u * q;
        if (code == 1) t.put_exit(c.X0, c.Z0, c.X1, c.Z1, c.U, k);
        if (code == 2) t.put_exit(c.X1, c.Z1, c.X2, c.Z2, c.U, k + 1u);
        if (code == 3) t.put_exit(c.X2, c.Z2, c.X2, c.Z2, 0.f, k + 2u);
    }

    // The owner takes its walk back: base is the first lane of the walk's
    // segment (seg: this lane's own segment), last the lane of its last pair.
    __device__ __forceinline__ void coop_end(const Coop &c, unsigned seg, int per, int base, bool mine) {
        const float x = __shfl_sync(kFull, c.X2, base + per - 1), z = __shfl_sync(kFull, c.Z2, base + per - 1);
        const uint32_t m = __shfl_sync(kFull, c.n, base) + 2u * (uint32_t)per;
        if (mine) {
            X = x;
            Z = z;
            n = m;
        }
        if constexpr (kRegions) {
            const uint32_t e = seg_sum(c.occ.ce, seg), s = seg_sum(c.occ.cs, seg);
            const uint32_t ge = __shfl_sync(kFull, e, base), gs = __shfl_sync(kFull, s, base);
            if (mine) {
                occ.ce += ge;
                occ.cs += gs;
            }
        } else if constexpr (KMAX < 8) {
#pragma unroll
            for (int j = 0; j < KMAX - 1; ++j) {
                const uint32_t e = seg_sum(c.occ.s[j], seg);
                const uint32_t g = __shfl_sync(kFull, e, base);
                if (mine) occ.s[j] += g;
            }
        }
    }
    __device__ __forceinline__ static uint32_t seg_sum(uint32_t v, unsigned seg) {
        return seg ? __reduce_add_sync(seg, v) : 0u;
    }

    __device__ static void to_abs(const ModelDev &M, float X, float Z, double &x, double &z) {
        x = (double)X + M.xc;
        z = (double)Z + M.zc;
    }

    // 1D column solution at depth z: exp(-k z) in the earth, 1 - k z in air.
    __device__ static void column(float kr, float ki, float z, float &gr, float &gi) {
        if (z >= 0.f) {
            const float a = expf(-kr * z);
            float s, c;
            sincosf(ki * z, &s, &c);
            gr = a * c;
            gi = -a * s;
        } else {
            gr = fmaf(-kr, z, 1.f);
            gi = -ki * z;
        }
    }

    // Sample of one walk for evaluation e: g(exit) exp(-i (1/2) sum_m kappa_{e,m} T_m).
    // The phase in turns, by integer products modulo one turn (exact; see
    // PhaseTurn), then one conversion to radians: with sum and reduction in
    // FP64 a sample took 21 operations of the FP64 pipe (64 cycles a warp
    // each), and 3 so; 2.6e6 walks x 16 evaluations at dt 1e-3 spent 40 % of
    // the pipe on samples and their sums.
    static constexpr bool kTurns = true;
    __device__ static double2 sample(const ModelDev &M, const SharedTables &T, const WalkArgs &A,
                                     int model, int e, float X, float Z, float th, int wall,
                                     int mlast, const uint32_t *c) {
        const bool multi = GC == GC_RASTER_MULTI;
        const int K = multi ? A.models[model].K : M.K;
        float pr;
        // a batched model's own flag: its samples are those it has alone,
        // whatever the launch's other models are
        if (multi ? A.models[model].turns : A.turns) {
            const uint64_t *f = (multi ? A.models[model].turn_frac : T.turn_frac) + e * K;
            const uint32_t whole = (multi ? A.models[model].turn_whole : T.turn_whole)[e * K + mlast];
            uint64_t turn = 0;
#pragma unroll
            for (int k = 0; k < KMAX; ++k)
                if (k < K) turn += f[k] * c[k];
            // theta as a whole step (it can round to one, or past it) and a
            // 64-bit fraction, exact down to 2^-63 (through a signed
            // conversion: the unsigned one takes 1.3 % of a call with 16
            // evaluations)
            const uint32_t step = (uint32_t)th;
            const uint64_t t64 = (uint64_t)(long long)((th - (float)step) * 9223372036854775808.f) << 1;
            turn += step * f[mlast] + __umul64hi(f[mlast], t64) + whole * t64;
            pr = (float)((double)(int64_t)turn * 0x1.921fb54442d18p-62);  // 2 pi 2^-64
        } else {
            const double *kap = (multi ? A.models[model].kappa : M.kappa) + e * K;
            double ph = 0.0;
#pragma unroll
            for (int k = 0; k < KMAX; ++k)
                if (k < K) ph = fma(kap[k], (double)c[k], ph);
            ph = fma(kap[mlast], (double)th, ph);
            ph *= 0.5 * A.dt;
            const double q = rint(ph * 0.15915494309189535);
            pr = (float)fma(-q, 6.283185307179586, ph);
        }
        float sw, cw;
        sincosf(pr, &sw, &cw);
        float gr, gi;
        const float x = X + M.fxc, z = Z + M.fzc;
        if (M.g_kind == 1) {
            const double *a = M.g_coef;
            gr = (float)(a[0] + a[2] * (double)x + a[4] * (double)z);
            gi = (float)(a[1] + a[3] * (double)x + a[5] * (double)z);
        } else if (M.g_kind == 2) {
            gr = x * x - z * z;
            gi = 0.f;
        } else {
            const EvalF &E = multi ? A.models[model].ev[e] : T.evf[e];
            if (wall == 0) {
                column(E.kl_re, E.kl_im, z, gr, gi);
            } else if (wall == 1) {
                column(E.kr_re, E.kr_im, z, gr, gi);
            } else {
                const float t = (X + M.fhw) / (2.f * M.fhw);
                gr = fmaf(t, wall == 2 ? E.td_re : E.bd_re, wall == 2 ? E.tl_re : E.bl_re);
                gi = fmaf(t, wall == 2 ? E.td_im : E.bd_im, wall == 2 ? E.tl_im : E.bl_im);
            }
        }
        // (cw - i sw)(gr + i gi)
        return make_double2((double)fmaf(cw, gr, sw * gi), (double)fmaf(cw, gi, -sw * gr));
    }
};

template <int KMAX, int GC>
static cudaError_t launch_one(const ModelDev &M, const WalkArgs &A, int grid, int block,
                              cudaStream_t s) {
    const size_t sm = shared_bytes<WalkerF32<KMAX, GC>>(block / 32, M.E, M.K);
    auto k = walk_kernel<WalkerF32<KMAX, GC>>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<grid, block, sm, s>>>(M, A);
    return cudaGetLastError();
}

template <int KMAX, int GC>
static int occ_one(int block, int E, int K) {
    const size_t sm = shared_bytes<WalkerF32<KMAX, GC>>(block / 32, E, K);
    auto k = walk_kernel<WalkerF32<KMAX, GC>>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, block, sm) != cudaSuccess) return 0;
    return n;
}

// Kernel variants: materials K <= KMAX in {2, 3, 4, 8} x the six lookup programs.
#define SDD_GC_CASES(FN, KM, ...)                                               \
    switch (gcode) {                                                            \
    case GC_LAYER: return FN<KM, GC_LAYER>(__VA_ARGS__);                        \
    case GC_RECT1: return FN<KM, GC_RECT1>(__VA_ARGS__);                        \
    case GC_TRI1: return FN<KM, GC_TRI1>(__VA_ARGS__);                          \
    case GC_SHAPES4: return FN<KM, GC_SHAPES4>(__VA_ARGS__);                    \
    case GC_SHAPES16: return FN<KM, GC_SHAPES16>(__VA_ARGS__);                  \
    case GC_RASTER: return FN<KM, GC_RASTER>(__VA_ARGS__);                      \
    case GC_CONTACT: return FN<KM, GC_CONTACT>(__VA_ARGS__);                    \
    case GC_RASTER_MULTI: return FN<KM, GC_RASTER_MULTI>(__VA_ARGS__);          \
    default: break;                                                             \
    }

#define SDD_DISPATCH(FN, ...)                                                   \
    switch (kmax) {                                                             \
    case 2: SDD_GC_CASES(FN, 2, __VA_ARGS__) break;                             \
    case 3: SDD_GC_CASES(FN, 3, __VA_ARGS__) break;                             \
    case 4: SDD_GC_CASES(FN, 4, __VA_ARGS__) break;                             \
    case 8: SDD_GC_CASES(FN, 8, __VA_ARGS__) break;                             \
    default: break;                                                             \
    }

// The TM walk (vertical strips, K <= KMAX in {2, 3, 4, 8}).
template <int KMAX>
static cudaError_t launch_tm(const ModelDev &M, const WalkArgs &A, int grid, int block, cudaStream_t s) {
    using W = WalkerTM32<KMAX>;
    const size_t sm = shared_bytes<W>(block / 32, M.E, M.K);
    auto k = walk_kernel<W>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<grid, block, sm, s>>>(M, A);
    return cudaGetLastError();
}

template <int KMAX>
static int occ_tm(int block, int E, int K) {
    using W = WalkerTM32<KMAX>;
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

cudaError_t launch_walk_f32(int kmax, int /*geo*/, const ModelDev &M, const WalkArgs &A, int grid,
                            int block, cudaStream_t s) {
    const int gcode = M.gcode;
    if (gcode == GC_TM) {
        SDD_TM_DISPATCH(launch_tm, M, A, grid, block, s)
        return cudaErrorInvalidValue;
    }
    SDD_DISPATCH(launch_one, M, A, grid, block, s)
    return cudaErrorInvalidValue;
}

int occupancy_f32(int kmax, int gcode, int block, int E, int K) {
    if (gcode == GC_TM) {
        SDD_TM_DISPATCH(occ_tm, block, E, K)
        return 0;
    }
    SDD_DISPATCH(occ_one, block, E, K)
    return 0;
}

}  // namespace sdd
