// Persistent walk scheduler shared by the single- and double-precision walks.
//
// Work model.  The estimator of Sec. 3.1 averages independent walks per
// interface node; the node values are independent of one another (Sec. 5).
// The host cuts every node's paths into work items (node, path range) and
// orders them so that item sizes shrink toward the end of the queue (guided
// self-scheduling, down to one walk per lane): when the queue runs dry, every
// warp holds little unfinished work.  Each warp of a persistent grid takes
// items from a global atomic counter and keeps its 32 lanes busy: a lane
// whose walk has reached the boundary takes the next path of the warp's
// current item at once, and the warp opens the next item as soon as the
// current one is fully handed out, however many earlier items still have
// walks in flight.  Uneven exit times therefore idle no lane until the queue
// is empty; then, and in calls of few walks from the start, the lanes of a
// warp share the walks that are left (cooperative rounds).
//
// Exit records.  A finished walk writes a small record (item, exit point,
// hit fraction theta, wall, last material, per-material step counts) into a
// per-warp ring in shared memory.  Once 32 records are waiting, the whole
// warp turns them into samples g(exit) exp(-i (1/2) sum_m kappa_{e,m} T_m)
// for every evaluation e, lane l handling evaluation l mod Epad.  The samples
// of each item are summed across the lanes with warp shuffles (fixed order)
// and added to the item's slot in global memory (sum re, sum im, sum re^2,
// sum im^2; a few MB, L2-resident).  An item belongs to the one
// warp that opened it, so its slot needs no atomics.  A second kernel adds
// the slots of each node, a warp per node and evaluation, in an order that
// the item table alone fixes.
#pragma once

#include "sdd_internal.cuh"

namespace sdd {

constexpr unsigned kFull = 0xffffffffu;

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32 -> 64-bit products with multipliers 0xD2511F53 and 0xCD9E8D57, the
// key bumped by 0x9E3779B9 / 0xBB67AE85 between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// The same generator when counter words 1..3 are fixed for the whole walk:
// the first round's product of word 2 is precomputed (pre_x = hi1 ^ c1 ^ k0,
// pre_y = lo1), leaving one product in round one.
__device__ __forceinline__ uint4 philox4x32_10_pre(uint32_t c0, uint32_t c3, uint32_t pre_x,
                                                   uint32_t pre_y, uint32_t k0, uint32_t k1) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    uint4 c = make_uint4(pre_x, pre_y, hi0 ^ c3 ^ k1, lo0);
#pragma unroll
    for (int r = 1; r < 10; ++r) {
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
        const uint32_t h0 = __umulhi(0xD2511F53u, c.x), l0 = 0xD2511F53u * c.x;
        const uint32_t h1 = __umulhi(0xCD9E8D57u, c.z), l1 = 0xCD9E8D57u * c.z;
        c = make_uint4(h1 ^ c.y ^ k0, l1, h0 ^ c.w ^ k1, l0);
    }
    return c;
}

// The float 1.m whose mantissa m is the low 23 bits of w:
// (w & 0x007fffff) | 0x3f800000 as one three-input logic operation, the
// exponent bits held in a register (two immediates would take two).
__device__ __forceinline__ float mant_one(uint32_t w) {
    uint32_t r;
    asm("lop3.b32 %0, %1, 0x007fffff, %2, 0xEA;" : "=r"(r) : "r"(w), "r"(0x3f800000u));
    return __uint_as_float(r);
}

// |x| and -x as sign bits alone.  Under -ftz=true fabsf() and unary minus
// flush denormals, which the compiler forms as an addition of their own; the
// float operations that take these flush their inputs anyway, so the plain
// forms give the same results as operand modifiers, without an instruction.
// There were four such additions a step (of about 62 issue slots): the squared
// radius, its negated root and the two coordinates of the wall distance.
__device__ __forceinline__ float abs_bits(float x) {
    float r;
    asm("abs.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float neg_bits(float x) {
    float r;
    asm("neg.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 32 x 32 -> 64-bit product as one wide multiply.
__device__ __forceinline__ void mul_wide(uint32_t a, uint32_t b, uint32_t &lo, uint32_t &hi) {
    uint64_t p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
    lo = (uint32_t)p;
    hi = (uint32_t)(p >> 32);
}

// Philox4x32-10 with the ten round keys given (rk0[r] = k0 + r 0x9E3779B9,
// rk1[r] = k1 + r 0xBB67AE85); with counter words 1..3 fixed for a walk the
// first round's product of word 2 is precomputed (pre_x = hi ^ c1 ^ rk0[0],
// pre_y = lo of 0xCD9E8D57 * c2).
__device__ __forceinline__ uint4 philox_rk_pre(uint32_t c0, uint32_t c3, uint32_t pre_x,
                                               uint32_t pre_y, const uint32_t (&rk0)[10],
                                               const uint32_t (&rk1)[10]) {
    uint32_t lo0, hi0;
    mul_wide(0xD2511F53u, c0, lo0, hi0);
    uint4 c = make_uint4(pre_x, pre_y, hi0 ^ c3 ^ rk1[0], lo0);
#pragma unroll
    for (int r = 1; r < 10; ++r) {
        uint32_t l0, h0, l1, h1;
        mul_wide(0xD2511F53u, c.x, l0, h0);
        mul_wide(0xCD9E8D57u, c.z, l1, h1);
        c = make_uint4(h1 ^ c.y ^ rk0[r], l1, h0 ^ c.w ^ rk1[r], l0);
    }
    return c;
}

__device__ __forceinline__ uint4 philox_rk(uint4 c, const uint32_t (&rk0)[10],
                                           const uint32_t (&rk1)[10]) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t l0, h0, l1, h1;
        mul_wide(0xD2511F53u, c.x, l0, h0);
        mul_wide(0xCD9E8D57u, c.z, l1, h1);
        c = make_uint4(h1 ^ c.y ^ rk0[r], l1, h0 ^ c.w ^ rk1[r], l0);
    }
    return c;
}

// Shared-memory layout of one CTA: model tables, then for each warp its
// exit-record ring and its scheduler state.  A walker W states what it
// records per material: W::Occ (step counts, or occupation times when they
// can be fractional) for W::kStored materials (all but material 0 when that
// one is derived from the step total, else all K), and W::kHist words per
// lane of shared-memory occupation histogram (W::HistT).
template <class W>
struct Ring {
    using Real = typename W::Real;
    Real x[kRing], z[kRing], th[kRing];  // W::kLate: the point before the exiting step and its
    Real xn[W::kLate ? kRing : 1], zn[W::kLate ? kRing : 1];  // uniform, and its end, until the record is made
    uint32_t meta[kRing];  // wall | m_last << 2 | truncated << 6 | model << 8
    int32_t item[kRing];
    uint32_t n[kRing];     // occupation steps (all steps but the exiting one)
    uint32_t path[kRing];
    uint32_t aux[kRing];   // interface randomisations (TM walks)
    typename W::Occ cnt[W::kStored][kRing];
};

// Scheduler state of one warp (every field is the same for all its lanes,
// each lane reads back what it wrote), kept out of registers because only
// the exit handler touches it.
struct WarpState {
    unsigned long long steps[32];
    unsigned long long trunc;
    double nx0, nz0;  // the current item's node,
    float fx0, fz0;   // and in single-precision centred coordinates
    int32_t disp_item, disp_rem, disp_model;
    uint32_t disp_next, nid;
    uint32_t head, tail;
    int32_t queue_empty;
    int32_t home;  // grouped launches: the queue this warp takes items from
};

// The model's rates [E][K] and boundary constants [E], staged in shared
// memory ahead of the warps' areas; sized by the model's E and K.
// The TE walk in single precision keeps its phases as turns and its boundary
// constants as floats there instead, in the same space.
struct SharedTables {
    double *kappa;
    EvalDev *ev;
    uint64_t *turn_frac;   // [E][K]
    EvalF *evf;            // [E]
    uint32_t *turn_whole;  // [E][K]
};
static_assert(sizeof(EvalF) + kMaxK * sizeof(uint32_t) <= sizeof(EvalDev), "turn tables exceed the boundary table");

__host__ __device__ constexpr size_t tables_bytes(int E, int K) {
    return ((size_t)E * K * sizeof(double) + 15) / 16 * 16 + (size_t)E * sizeof(EvalDev);
}

template <class W>
struct WarpSmem {
    Ring<W> ring;
    WarpState st;
    typename W::HistT hist[W::kHist][32];     // per-lane occupation histogram
    typename W::Real pend[W::kPend > 0 ? W::kPend : 1][32];  // exiting steps that wait for their records
    typename W::CoopInc coop[W::kCoop ? 64 : 1];  // step increments of the cooperative rounds
};

template <class W>
__host__ __device__ constexpr size_t shared_bytes(int warps, int E, int K) {
    return (tables_bytes(E, K) + 15) / 16 * 16 + (size_t)warps * sizeof(WarpSmem<W>);
}

// Exit information handed from a walker to the scheduler.
template <class Real>
struct ExitInfo {
    Real x, z, th;  // exit point (walker coordinates) and hit fraction
    int wall;       // 0..3
    int mlast;      // material of the last point inside
    uint32_t nocc;  // occupation steps (all steps but the exiting one)
    uint32_t aux;   // interface randomisations (TM walks)
};

// Scheduler kernel.  W is a walker type providing
//   using Real; static constexpr int KMAX;
//   start(M, A, S, path, model)  -- begin a walk at the warp's current node
//   iterate(M, A, path, ExitInfo&) -> 0 running, 1 exited, 2 truncated
//     (a few Euler steps per call; max_steps is a multiple of them)
//   finalize(M, A, st, ExitInfo&): the exit record of a walk that has ended;
//     kLate: get_exit() the exiting step instead, and finish() makes its record
//   counts(M, nocc, c): steps spent in materials 1..KMAX-1 (at the exit,
//     after nocc occupation steps)
//   bind(h, p): the lane's columns of the occupancy histogram and of the
//     exiting steps that wait for their records (kPend words)
//   kAlone: has iterate(), one walk a lane; kCoop, CoopInc, Coop, coop_*: has
//     cooperative rounds (kEvents: a round can end without ending a walk)
//   static sample(M, T, A, model, e, x, z, th, wall, mlast, counts) -> double2
//   static to_abs(M, x, z, ax, az)
//   kGrouped: takes items from per-model queues (multi-model launches)
//   kMinCTAs: CTAs of 256 threads that must fit on an SM (the register bound)
// Launch bounds: at most 256 threads, and at least W::kMinCTAs such CTAs per
// SM: 3 leaves up to 85 registers a thread, 4 leaves 64.
template <class W>
__global__ void __launch_bounds__(256, W::kMinCTAs) walk_kernel(const __grid_constant__ ModelDev M,
                                                   const WalkArgs A) {
    using Real = typename W::Real;
    constexpr int KMAX = W::KMAX;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SharedTables T;
    T.kappa = reinterpret_cast<double *>(smem_raw);
    T.ev = reinterpret_cast<EvalDev *>(smem_raw + ((size_t)M.E * M.K * sizeof(double) + 15) / 16 * 16);
    WarpSmem<W> &WS = reinterpret_cast<WarpSmem<W> *>(
        smem_raw + (tables_bytes(M.E, M.K) + 15) / 16 * 16)[threadIdx.x >> 5];
    Ring<W> &R = WS.ring;
    WarpState &S = WS.st;

    T.turn_frac = reinterpret_cast<uint64_t *>(T.kappa);
    T.evf = reinterpret_cast<EvalF *>(T.ev);
    T.turn_whole = reinterpret_cast<uint32_t *>(T.evf + M.E);
    if constexpr (W::kTurns) {
        if (A.turns)
            for (int i = threadIdx.x; i < M.E * M.K; i += blockDim.x) {
                const PhaseTurn p = phase_turn(M.kappa[i], A.dt);
                T.turn_frac[i] = p.frac;
                T.turn_whole[i] = p.whole;
            }
        for (int i = threadIdx.x; i < M.E; i += blockDim.x) T.evf[i] = eval_f(M.ev[i]);
    } else {
        for (int i = threadIdx.x; i < M.E * M.K; i += blockDim.x) T.kappa[i] = M.kappa[i];
        for (int i = threadIdx.x; i < M.E; i += blockDim.x) T.ev[i] = M.ev[i];
    }

    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const bool dump = A.rec_steps != nullptr;
    S.steps[lane] = 0ull;
    if (lane == 0) {
        S.trunc = 0ull;
        S.disp_item = -1; S.disp_rem = 0; S.disp_model = 0; S.disp_next = 0; S.nid = 0;
        S.head = S.tail = 0;
        S.queue_empty = 0;
        S.nx0 = S.nz0 = 0.0;
        S.fx0 = S.fz0 = 0.f;
        S.home = 0;
        if (W::kGrouped && A.qbase) {
            const float x = ((float)blockIdx.x + 0.5f) / (float)gridDim.x;
            int m = 0;
            while (m + 1 < A.n_queues && A.home_cut[m + 1] <= x) ++m;
            S.home = m;
        }
    }
    __syncthreads();

    // per-lane walk state
    W w;
    w.bind(&WS.hist[0][lane], &WS.pend[0][lane]);
    bool active = false;
    int item = 0;
    int model = 0;
    uint32_t path = 0;

    // The record of ring entry s as its sample for evaluation e (zero for a
    // truncated walk, or when the records are dumped: then written out).
    auto take = [&](int s, int e) {
        const uint32_t meta = R.meta[s];
        const bool tr = (meta >> 6) & 1u;
        typename W::Occ c[KMAX];
        if constexpr (W::kStored == KMAX) {
#pragma unroll
            for (int j = 0; j < KMAX; ++j) c[j] = R.cnt[j][s];
        } else {
            uint32_t rest = R.n[s];
#pragma unroll
            for (int j = 1; j < KMAX; ++j) {
                c[j] = R.cnt[j - 1][s];
                rest -= c[j];
            }
            c[0] = rest;
        }
        if (dump) {
            if (e == 0) {
                const int64_t o = (int64_t)(R.path[s] - A.items[0].path0);
                double ex, ez;
                W::to_abs(M, R.x[s], R.z[s], ex, ez);
                A.rec_steps[o] = (int64_t)R.n[s] + (tr ? 0 : 1);
#pragma unroll
                for (int j = 0; j < KMAX; ++j)
                    if (j < M.K) {
                        if (A.rec_counts) A.rec_counts[o * M.K + j] = (int64_t)c[j];
                        if (A.rec_occ) A.rec_occ[o * M.K + j] = (double)c[j];
                    }
                if (A.rec_hits) A.rec_hits[o] = (int64_t)R.aux[s];
                A.rec_exit[3 * o + 0] = ex;
                A.rec_exit[3 * o + 1] = ez;
                A.rec_exit[3 * o + 2] = (double)R.th[s];
                A.rec_wall[o] = tr ? -1 : (int)(meta & 3u);
                A.rec_mlast[o] = (int)((meta >> 2) & 7u);
            }
            return make_double2(0.0, 0.0);
        }
        if (tr) return make_double2(0.0, 0.0);
        return W::sample(M, T, A, (int)(meta >> 8), e, R.x[s], R.z[s], R.th[s], (int)(meta & 3u),
                         (int)((meta >> 2) & 7u), c);
    };

    // Add the sums q (re, im, re^2, im^2) of the lanes of each evaluation to
    // item it's slots, in a fixed order.  Lanes e, e + Epad, ... hold
    // evaluation e; a level of the sum halves the values a lane carries while
    // it can, so 32 lanes of one evaluation take 6 additions, not 20.
    auto add_slots = [&](int it, double q0, double q1, double q2, double q3) {
        const int Epad = M.Epad, my_e = lane & (Epad - 1);
        double *o = A.slots + ((size_t)it * M.E + my_e) * 4;
        if (Epad <= 16) {
            const bool up = lane & 16;
            const double g0 = __shfl_xor_sync(kFull, up ? q0 : q2, 16), g1 = __shfl_xor_sync(kFull, up ? q1 : q3, 16);
            q0 = (up ? q2 : q0) + g0;
            q1 = (up ? q3 : q1) + g1;
            if (up) o += 2;
        }
        if (Epad <= 8) {
            const bool up = lane & 8;
            const double g = __shfl_xor_sync(kFull, up ? q0 : q1, 8);
            q0 = (up ? q1 : q0) + g;
            if (up) o += 1;
        }
        for (int off = 4; off >= Epad; off >>= 1) q0 += __shfl_xor_sync(kFull, q0, off);
        if (my_e >= M.E || (lane & 7 & ~(Epad - 1)) != 0) return;
        o[0] += q0;
        if (Epad > 8) o[1] += q1;
        if (Epad > 16) {
            o[2] += q2;
            o[3] += q3;
        }
    };

    // Turn records [head, head + cnt) of the ring (cnt <= 32) into samples,
    // 32 / Epad records a round; lane l handles evaluation l mod Epad.  Up to 4
    // evaluations: all records in ring order, then the sums of each item in
    // the round.  More: item by item, a lane adding up its samples over the
    // item's rounds first, so that the item's slots are touched once.
    auto process = [&](int cnt) {
        const uint32_t head = S.head;
        const int Epad = M.Epad, my_e = lane & (Epad - 1);
        const int per_round = 32 / Epad, my_ro = lane / Epad;
        const int mine_s = (head + lane) & (kRing - 1);
        const int rec_it = lane < cnt ? R.item[mine_s] : -1;
        if (lane < cnt) {
            const uint32_t meta = R.meta[mine_s];
            const bool tr = (meta >> 6) & 1u;
            S.steps[lane] += (unsigned long long)R.n[mine_s] + (tr ? 0ull : 1ull);
            if constexpr (W::kLate) {
                // the exit records of all 32 at once (made by the few lanes of an
                // exit batch they took 120 of its 350 instructions)
                ExitInfo<Real> ex;
                W::finish(M, A, (int)(meta >> 8), tr, R.x[mine_s], R.z[mine_s], R.xn[mine_s], R.zn[mine_s],
                          R.th[mine_s], ex);
                R.x[mine_s] = ex.x;
                R.z[mine_s] = ex.z;
                R.th[mine_s] = ex.th;
                R.meta[mine_s] = meta | (uint32_t)ex.wall | ((uint32_t)ex.mlast << 2);
            }
        }
        __syncwarp();
        unsigned pend = kFull >> (32 - cnt);
        while (pend) {
            const int it = __shfl_sync(kFull, rec_it, __ffs(pend) - 1);
            const unsigned sel = Epad <= 4 ? pend : __ballot_sync(kFull, rec_it == it);
            double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
            for (unsigned left = sel; left;) {
                // this round's records: the lowest per_round bits of left
                unsigned m = left;
                for (int j = 0; j < my_ro; ++j) m &= m - 1u;
                double2 v = make_double2(0.0, 0.0);
                const int at = __ffs(m) - 1;
                if (m && my_e < M.E) v = take((head + at) & (kRing - 1), my_e);
                if (Epad <= 4) {
                    const int my_it = __shfl_sync(kFull, rec_it, at & 31);
                    unsigned todo = dump ? 0u : __ballot_sync(kFull, m != 0u);
                    while (todo) {
                        const int one = __shfl_sync(kFull, my_it, __ffs(todo) - 1);
                        const bool mine = m != 0u && my_it == one;
                        const double b0 = mine ? v.x : 0.0, b1 = mine ? v.y : 0.0;
                        add_slots(one, b0, b1, b0 * b0, b1 * b1);
                        todo &= ~__ballot_sync(kFull, mine);
                    }
                } else {
                    a0 += v.x;
                    a1 += v.y;
                    a2 = fma(v.x, v.x, a2);
                    a3 = fma(v.y, v.y, a3);
                }
                for (int j = 0; j < per_round; ++j) left &= left - 1u;
            }
            if (Epad > 4 && !dump) add_slots(it, a0, a1, a2, a3);
            pend &= ~sel;
        }
        __syncwarp();
        S.head = head + (uint32_t)cnt;
        __syncwarp();
    };

    // Hand paths to idle lanes, opening the next queued item whenever the
    // current one is fully handed out.
    auto refill = [&]() {
        unsigned need = __ballot_sync(kFull, !active && lane < A.max_lanes);
        if (A.cancel && need) {
            // a cancelled request: no more paths; the walks in flight end
            int c = 0;
            if (lane == 0) c = *reinterpret_cast<const volatile int32_t *>(A.cancel);
            if (__shfl_sync(kFull, c, 0)) {
                if (lane == 0) {
                    S.queue_empty = 1;
                    S.disp_rem = 0;
                }
                __syncwarp();
                return;
            }
        }
        while (need) {
            if (S.disp_rem == 0) {
                if (S.queue_empty) break;
                int it = -1;
                if (lane == 0) {
                    if (W::kGrouped && A.qbase) {
                        // the home queue first, then the next ones in turn
                        int m = S.home;
                        for (int t = 0; t < A.n_queues; ++t) {
                            const int q = atomicAdd(A.queue + m, 1);
                            if (q < A.qbase[m + 1] - A.qbase[m]) {
                                it = A.order[A.qbase[m] + q];
                                break;
                            }
                            m = m + 1 == A.n_queues ? 0 : m + 1;
                        }
                        S.home = m;
                    } else {
                        const int q = atomicAdd(A.queue, 1);
                        if (q < A.n_items) it = A.order ? A.order[q] : q;
                    }
                }
                it = __shfl_sync(kFull, it, 0);
                if (it < 0) {
                    if (lane == 0) S.queue_empty = 1;
                    __syncwarp();
                    break;
                }
                const Item I = A.items[it];
                if (!dump) {
                    if (lane < M.E) {
                        double *o = A.slots + ((size_t)it * M.E + lane) * 4;
                        o[0] = 0.0; o[1] = 0.0; o[2] = 0.0; o[3] = 0.0;
                    }
                    if (lane == 0) A.item_trunc[it] = 0;
                }
                if (lane == 0) {
                    S.disp_item = it;
                    S.disp_model = I.model;
                    S.disp_next = I.path0;
                    S.disp_rem = I.count;
                    const double x0 = A.nodes[2 * I.node], z0 = A.nodes[2 * I.node + 1];
                    S.nx0 = x0;
                    S.nz0 = z0;
                    S.fx0 = (float)(x0 - M.xc);
                    S.fz0 = (float)(z0 - M.zc);
                    S.nid = A.node_ids ? A.node_ids[I.node] : (uint32_t)I.node;
                }
                __syncwarp();
                if (I.count == 0) continue;
            }
            const int rem = S.disp_rem;
            const int navail = __popc(need);
            const int k = navail < rem ? navail : rem;
            const int rank = __popc(need & lt_mask);
            const bool mine = ((need >> lane) & 1u) && rank < k;
            if (mine) {
                path = S.disp_next + (uint32_t)rank;
                item = S.disp_item;
                model = S.disp_model;
                active = true;
                w.start(M, A, S, path, model);
            }
            const unsigned got = __ballot_sync(kFull, mine);
            need &= ~got;
            if (lane == 0) {
                S.disp_next += (uint32_t)k;
                S.disp_rem = rem - k;
            }
            __syncwarp();
        }
    };

    // Records of the walks that have ended (st: 1 exited, 2 truncated).
    ExitInfo<Real> ei{};
    auto on_exits = [&](int st) {
        const unsigned em = __ballot_sync(kFull, st != 0);
        const int nex = __popc(em);
        const uint32_t tail = S.tail;
        if (st != 0) {
            const int slot = (tail + __popc(em & lt_mask)) & (kRing - 1);
            const bool tr = st == 2;
            uint32_t meta = ((uint32_t)tr << 6) | ((uint32_t)model << 8);
            if constexpr (W::kLate) {
                Real x0, z0, xn, zn, u;
                w.get_exit(x0, z0, xn, zn, u, ei.nocc);
                R.x[slot] = x0;
                R.z[slot] = z0;
                R.xn[slot] = xn;
                R.zn[slot] = zn;
                R.th[slot] = u;
            } else {
                w.finalize(M, A, st, ei);
                R.x[slot] = ei.x;
                R.z[slot] = ei.z;
                R.th[slot] = ei.th;
                meta |= (uint32_t)ei.wall | ((uint32_t)ei.mlast << 2);
                R.aux[slot] = ei.aux;
            }
            R.meta[slot] = meta;
            R.item[slot] = item;
            R.n[slot] = ei.nocc;
            if (dump) {
                R.path[slot] = path;
                if constexpr (W::kLate) R.aux[slot] = 0;
            }
            typename W::Occ c[W::kStored];
            w.counts(M, ei.nocc, c);
#pragma unroll
            for (int j = 0; j < W::kStored; ++j) R.cnt[j][slot] = c[j];
            if (tr && !dump) atomicAdd(&A.item_trunc[item], 1);
        }
        const unsigned trm = __ballot_sync(kFull, st == 2);
        if (lane == 0) {
            S.tail = tail + (uint32_t)nex;
            if (trm) S.trunc += (unsigned long long)__popc(trm);
        }
        __syncwarp();
    };

    // The rest of an exit: records, refill, and samples once 32 records are
    // waiting, or at the end.
    int n_live = 0;
    auto settle = [&](int ended) {
        on_exits(ended);
        refill();
        n_live = __popc(__ballot_sync(kFull, active));
        while (S.tail - S.head >= 32 || (n_live == 0 && S.tail != S.head)) process((int)min(S.tail - S.head, 32u));
    };
    refill();
    n_live = __popc(__ballot_sync(kFull, active));

    // One walk a lane.  A lane whose walk has ended waits until exit_batch
    // lanes of the warp have, or all of them: the records and the refill cost
    // a warp the same for one ended walk as for several.
    if constexpr (W::kAlone) {
        while (n_live > 0) {
            if (W::kCoop && n_live <= kCoopWalks &&
                (A.max_lanes <= kCoopWalks || (S.queue_empty && S.disp_rem == 0)))
                break;
            const int n_batch = min(n_live, A.exit_batch);
            int st = active ? 0 : -1;
            do {
                if (st == 0) st = w.iterate(M, A, path, ei);
            } while (__popc(__ballot_sync(kFull, st > 0)) < n_batch);
            active = st == 0;
            settle(max(st, 0));
        }
    }

    // Cooperative rounds: the warp has a <= kCoopWalks walks.  Alone in its
    // lane a walk is one dependent chain of about 250 cycles a step (the
    // random words, the normals, the move, the tests).  Here each walk gets
    // 32 / a lanes, two steps a lane and round: the words, the normals and the
    // tests of all its steps are formed side by side, and only the moves
    // remain one after the other.  The lanes work for the same walks until one
    // of them ends.
    if constexpr (W::kCoop) {
        while (n_live > 0) {
            int ended = 0;  // the lane's walk: 1 exited, 2 truncated
            do {
                const unsigned act = __ballot_sync(kFull, active);
                const int per = 32 / n_live;
                const int j = lane / per;
                const uint32_t q = (uint32_t)(lane % per);
                const bool in = j < n_live;
                unsigned m = act;
                for (int t = 0; t < j && in; ++t) m &= m - 1u;
                const int owner = __ffs(m) - 1;
                const unsigned seg = in ? (kFull >> (32 - per)) << (j * per) : 0u;
                const int last = in ? j * per + per - 1 : lane;
                typename W::CoopInc *buf = WS.coop + (in ? j * 2 * per : 0);
                typename W::Coop c;
                w.coop_begin(c, owner, lane);
                int code;
                unsigned events;
                for (;;) {
                    code = W::coop_round(M, A, c, buf, q, per, in);
                    events = __ballot_sync(kFull, code != 0);
                    if (events) break;
                    W::coop_count(M, c, in ? 2 : 0);
                    w.coop_next(c, per, last);
                    __syncwarp();
                }
                // the steps before the segment's first event count (of the
                // event's lane: those before it)
                const int first = (events & seg) ? __ffs(events & seg) - 1 : 32;
                const int base = __popc(act & lt_mask) * per & 31;  // this lane's walk, if it owns one
                if constexpr (W::kEvents) {
                    ended = w.coop_events(M, A, c, code, first, per, active ? base : 0, active, ei);
                } else {
                    W::coop_count(M, c, !in || lane > first ? 0 : (lane < first ? 2 : (code == 3 ? 2 : code - 1)));
                    if (lane == first) w.coop_put(c, code, q, lane);
                    const int fcode = __shfl_sync(kFull, code, first & 31);
                    const int my_st = first == 32 ? 0 : (fcode == 3 ? 2 : 1);
                    const int st_own = __shfl_sync(kFull, my_st, base);
                    w.coop_end(c, seg, per, active ? base : 0, active);
                    ended = active ? st_own : 0;
                }
                __syncwarp();
            } while (__ballot_sync(kFull, ended != 0) == 0);
            if (ended) active = false;
            settle(ended);
        }
    }
    // every item handed to this warp has been flushed (its walks all ended)

    unsigned long long my_steps = S.steps[lane];
    for (int off = 16; off > 0; off >>= 1) my_steps += __shfl_xor_sync(kFull, my_steps, off);
    if (lane == 0 && !dump) {
        atomicAdd(&A.counters[0], my_steps);
        atomicAdd(&A.counters[1], (unsigned long long)S.tail);  // every record was a walk
        atomicAdd(&A.counters[2], S.trunc);
    }
}

}  // namespace sdd
