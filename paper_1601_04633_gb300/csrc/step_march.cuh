// T fused double-MRT time steps per launch (T = 2 or 3), each warp marching up
// its own strip of columns with the states between the steps in registers.
//
// One step moves every population through memory once (112 B per node in
// float32), so a launch per step is bound by HBM. This kernel reads a state
// once and writes the state T steps later: a T-th of the traffic per step.
//
// A warp owns 64 columns, two per lane, of which kCols are written (one or two
// pairs of columns on each side are recomputed by the neighbouring strip), and
// a chunk of rows [j0, j1). It goes up the rows. Whole rows (all planes of the
// strip and its halo) come by one tensor copy per plane block into the warp's
// own ring of kMarchStages shared-memory stages; iteration r has rows r - 1, r,
// r + 1 there and the next ones in flight. It pulls and collides row r (the
// first step), then row r - 1 for the second step, whose pull needs the first
// step's P group (e_y = +1) of row r - 2, kept in registers for two iterations,
// its Z group of row r - 1, kept for one, and its N group of row r, just
// computed; then row r - 2 for the third step from the second's in the same
// way. Columns shift between lanes by shuffles. The last step's row leaves by
// one tensor store per plane block from the warp's output tile. So a warp waits
// for no other warp; a chunk recomputes T - 1 rows on each side.
//
// The arithmetic of a node is collide_pair (the bits of collide_node), walls
// and Nusselt numbers are those of the other step kernels, and between the
// steps the state takes the values it would have after a store (16-bit
// storage: rounded, with the same random bits), so a launch gives the bits of
// T single steps.
//
// Every mbarrier wait is bounded, as in step_tma.cuh: on expiry the warp
// records kErrTimeout, waits (bounded) for the copies it issued and returns.
//
// Measured on one GB300 (2048^2 float32, three steps per launch): 103 us per launch,
// 62.2 M warp instructions (the one-step kernel issues 138 M for the same three steps),
// DRAM 56 % and the float32 pipe 54 % busy over the launch, three warps per scheduler held
// by shared memory (the ring and the output tile) and registers. At 4096^2 it moves the
// state at 0.8 of the copy rate. The times against the one-step kernels stand at the launch
// rule in dmrt.cu.

#pragma once
#include "collide_pair.cuh"
#include "step_tma.cuh"

namespace dmrt {

constexpr int kMarchThreads = 128;  // four warps, four neighbouring items
constexpr int kMarchStages = 4;     // rows in a warp's ring (a power of two)
constexpr int kMarchMax = 3;        // most steps per launch: a strip's side columns allow no more

// Strip geometry. A warp's lane l holds columns x0 = strip * kCols - kLead + 2 l
// and x0 + 1; rows are copied from column strip * kCols - kHalo (a 16-byte
// boundary), kBox columns wide, and kCols columns are stored (a 16-byte multiple).
template <typename L>
struct MarchGeo {
    static constexpr bool k16 = sizeof(typename L::Ef) == 2;
    static constexpr int kCols = k16 ? 56 : 60;
    static constexpr int kLead = k16 ? 4 : 2;
    static constexpr int kHalo = k16 ? 8 : 4;
    static constexpr int kBox = k16 ? 72 : 68;
    static constexpr int kFirst = kLead / 2;  // the first lane that stores
    // Bytes of a row's plane blocks in a stage / of the output tile: the flow
    // (one-type layouts: all 14) planes, then the thermal block (ThetaSplit:
    // theta, then the deviations), each 128-byte aligned.
    __host__ __device__ static constexpr unsigned up(unsigned x) { return (x + 127) & ~127u; }
    __host__ __device__ static constexpr unsigned f_bytes(int w) {
        return (L::kSplit ? 9 : 14) * w * (unsigned)sizeof(typename L::Ef);
    }
    __host__ __device__ static constexpr unsigned g_bytes(int w) {
        return L::kTheta ? w * 4u : L::kSplit ? 5 * w * (unsigned)sizeof(typename L::Eg) : 0;
    }
    __host__ __device__ static constexpr unsigned d_bytes(int w) { return L::kTheta ? 4 * w * 2u : 0; }
    __host__ __device__ static constexpr unsigned g_at(int w) { return L::kSplit ? up(f_bytes(w)) : 0; }
    __host__ __device__ static constexpr unsigned d_at(int w) { return g_at(w) + up(g_bytes(w)); }
    __host__ __device__ static constexpr unsigned size(int w) {
        return L::kSplit ? d_at(w) + up(d_bytes(w)) : up(f_bytes(w));
    }
    static constexpr unsigned kStage = size(kBox);
    static constexpr unsigned kTile = size(kCols);
    static constexpr unsigned kRowBytes = f_bytes(kBox) + g_bytes(kBox) + d_bytes(kBox);  // one row's copies
    static constexpr unsigned kWarp = kMarchStages * kStage + kTile;  // shared memory of a warp
    static constexpr unsigned kSmem = (kMarchThreads / 32) * (kWarp + kMarchStages * 8);
};

// Tensor maps of a launch: whole-row loads from the source (one-type: 14
// planes; split: 9 flow planes, the thermal planes; ThetaSplit: flow, theta,
// deviations) and the stores to the destination (nx columns).
struct MarchMaps {
    CUtensorMap ld[3];
    CUtensorMap st[3];
};

struct MarchArgs {
    StepArgs A;           // src/dst buffers, walls, counters (step_out = step_in + T)
    // Nusselt rows of this launch's steps and of those of the launch before: the
    // last step's, the step's before it, the one's before that. A march launch leaves (theta(0, j), theta(1, j)) as two
    // floats in a row's slot; the next launch's extra block, or the finalize
    // launch, puts the local Nusselt number there and sums the rows (float64 is
    // a slow pipe on this GPU: two of these per row on the marching warps'
    // path kept it half busy).
    double* nu_rows[kMarchMax];
    double* prev_rows[kMarchMax];
    int n_strips, n_chunks, chunk;  // items: strip + n_strips * chunk index; rows per chunk
    float sign_l, sign_r;  // -1: fixed-temperature wall (anti-bounce-back), +1: adiabatic
    float gsh0, gsh1, w0, w1, abb_l, abb_r;  // thermal shifts, rest weights, abb where the wall is fixed, else 0
    const float *wall_l, *wall_r;            // the walls' temperatures; zeros at an adiabatic wall (its profile is not read)
    double nu_scale;
    double (*nu_part)[8][32];  // [kMarchMax] partial sums of rows, when nu_blocks > 1
    unsigned* nu_arrivals;     // blocks of this launch that have written theirs (0 between launches)
    int nu_blocks;             // blocks that sum the rows of the launch before
};

// ---- storage forms --------------------------------------------------------------
// A stored pair of nodes of one plane: 8 bytes (float32) or 4 (16-bit types).
template <typename E>
struct PairElem {
    using T = unsigned;
};
template <>
struct PairElem<float> {
    using T = F2;
};
__device__ __forceinline__ F2 pair_load(F2 r, float) { return r; }
__device__ __forceinline__ F2 pair_load(unsigned r, __half) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&r));
    return f2_pack(v.x, v.y);
}
__device__ __forceinline__ F2 pair_load(unsigned r, __nv_bfloat16) {
    return f2_pack(__uint_as_float(r << 16), __uint_as_float(r & 0xffff0000u));
}
// The stored form of a pair; r0, r1: the nodes' random states (SR).
template <typename E, bool SR>
__device__ __forceinline__ typename PairElem<E>::T pair_store(F2 v, unsigned& r0, unsigned& r1) {
    if constexpr (std::is_same<E, float>::value) {
        return v;
    } else if constexpr (SR) {
        const unsigned a = lcg(r0), b = lcg(r1);
        return pack2_rs<E>(f2_lo(v), f2_hi(v), a, b);
    } else {
        return pack2_rn<E>(f2_lo(v), f2_hi(v));
    }
}

// The stored planes of a pair of nodes. Flow planes in direction order;
// thermal planes in direction order, or (ThetaSplit) theta and the deviations
// of directions 1..4.
template <typename L>
struct PairStored {
    typename PairElem<typename L::Ef>::T f[9];
    typename PairElem<typename L::Eg>::T g[5];  // ThetaSplit: g[1..4] deviations
    F2 theta;                                   // ThetaSplit only
};

template <typename L, bool SR>
__device__ __forceinline__ PairStored<L> pair_encode(const F2 (&f)[9], const F2 (&g)[5], F2 theta,
                                                     const MarchArgs& M, unsigned r0, unsigned r1) {
    using Ef = typename L::Ef;
    using Eg = typename L::Eg;
    PairStored<L> s;
#pragma unroll
    for (int k = 0; k < 9; ++k) s.f[k] = pair_store<Ef, SR>(f[k], r0, r1);
    if constexpr (L::kTheta) {
        s.theta = theta;
#pragma unroll
        for (int k = 1; k < 5; ++k) s.g[k] = pair_store<Eg, SR>(f2_fma(f2_all(-M.w1), theta, g[k]), r0, r1);
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const F2 v = kShifted<Eg> ? f2_sub(g[k], f2_all(k == 0 ? M.gsh0 : M.gsh1)) : g[k];
            s.g[k] = pair_store<Eg, SR>(v, r0, r1);
        }
    }
    return s;
}

// The populations a later step reads from a stored pair.
template <typename L>
__device__ __forceinline__ F2 pair_g(typename PairElem<typename L::Eg>::T r, int k, const MarchArgs& M) {
    const F2 v = pair_load(r, typename L::Eg());
    return kShifted<typename L::Eg> ? f2_add(v, f2_all(k == 0 ? M.gsh0 : M.gsh1)) : v;
}
__device__ __forceinline__ F2 theta_g(F2 theta, unsigned d, const MarchArgs& M) {
    return f2_fma(f2_all(M.w1), theta, pair_load(d, __half()));
}
__device__ __forceinline__ F2 theta_g0(F2 theta, unsigned d1, unsigned d2, unsigned d3, unsigned d4,
                                       const MarchArgs& M) {
    const F2 s = f2_add(f2_add(pair_load(d1, __half()), pair_load(d3, __half())),
                        f2_add(pair_load(d2, __half()), pair_load(d4, __half())));
    return f2_fma(f2_all(M.w0), theta, f2_sub(f2_all(-0.f), s));
}
template <typename L>
__device__ __forceinline__ void pair_decode(const PairStored<L>& s, const MarchArgs& M, F2 (&f)[9], F2 (&g)[5]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) f[k] = pair_load(s.f[k], typename L::Ef());
    if constexpr (L::kTheta) {
        g[0] = theta_g0(s.theta, s.g[1], s.g[2], s.g[3], s.g[4], M);
#pragma unroll
        for (int k = 1; k < 5; ++k) g[k] = theta_g(s.theta, s.g[k], M);
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) g[k] = pair_g<L>(s.g[k], k, M);
    }
}

// ---- a row in shared memory -------------------------------------------------------
// Lane geometry of an item.
struct MarchLane {
    int x0;            // the pair's columns x0, x0 + 1
    int c;             // column x0 in a stage's rows
    bool out;          // a pair this lane writes (x0 inside the cavity)
    bool two;          // both columns inside
    bool left, right;  // holds x = 0 (low half) / x = nx - 1
    bool rhi;          // right: nx - 1 is the high half
    bool wall;         // the warp holds a side wall (uniform): the left one, the right one
    bool wall_l, wall_r;
};

// The pair of direction k (flow: f, thermal: g) at columns x - EX, x + 1 - EX
// of the row in stage s.
template <int EX, int WB, typename E>
__device__ __forceinline__ F2 row_pair(const E* p) {
    if constexpr (EX != 0) {
        return f2_pack(to_f(p[-EX]), to_f(p[1 - EX]));
    } else {
        return pair_load(*reinterpret_cast<const typename PairElem<E>::T*>(p), E());
    }
}
template <typename L, int EX>
__device__ __forceinline__ F2 row_f(const unsigned char* s, int k, int c) {
    using G = MarchGeo<L>;
    return row_pair<EX, G::kBox>(reinterpret_cast<const typename L::Ef*>(s) + L::pf(k) * G::kBox + c);
}
template <typename L, int EX>
__device__ __forceinline__ F2 row_theta(const unsigned char* s, int c) {
    using G = MarchGeo<L>;
    return row_pair<EX, G::kBox>(reinterpret_cast<const float*>(s + G::g_at(G::kBox)) + c);
}
template <typename L, int EX>
__device__ __forceinline__ F2 row_dev(const unsigned char* s, int k, int c) {
    using G = MarchGeo<L>;
    return row_pair<EX, G::kBox>(reinterpret_cast<const __half*>(s + G::d_at(G::kBox)) + (k - 1) * G::kBox + c);
}
template <typename L, int EX>
__device__ __forceinline__ F2 row_g(const unsigned char* s, int k, int c, const MarchArgs& M) {
    using G = MarchGeo<L>;
    using Eg = typename L::Eg;
    if constexpr (L::kTheta) {
        const F2 th = row_theta<L, EX>(s, c);
        if (k == 0) {
            const F2 d = f2_add(f2_add(row_dev<L, 0>(s, 1, c), row_dev<L, 0>(s, 3, c)),
                                f2_add(row_dev<L, 0>(s, 2, c), row_dev<L, 0>(s, 4, c)));
            return f2_fma(f2_all(M.w0), th, f2_sub(f2_all(-0.f), d));
        }
        return f2_fma(f2_all(M.w1), th, row_dev<L, EX>(s, k, c));
    } else {
        const F2 v = row_pair<EX, G::kBox>(reinterpret_cast<const Eg*>(s + G::g_at(G::kBox)) + L::pg(k) * G::kBox + c);
        return kShifted<Eg> ? f2_add(v, f2_all(k == 0 ? M.gsh0 : M.gsh1)) : v;
    }
}

// Values pulled along +x (from the column to the left) / -x.
__device__ __forceinline__ F2 pull_px(F2 v) { return f2_pack(__shfl_up_sync(kFull, f2_hi(v), 1), f2_lo(v)); }
__device__ __forceinline__ F2 pull_mx(F2 v) { return f2_pack(f2_hi(v), __shfl_down_sync(kFull, f2_lo(v), 1)); }

// A temperature wall's value: the node's own opposite, negated across a fixed-
// temperature wall (sign), plus the wall term, which is a product rounded on
// its own (as in the other step kernels).
__device__ __forceinline__ float wall_value(float sign, float og, float add) { return __fmaf_rn(sign, og, add); }

// Side walls at a pulled pair: links from outside x = 0 (directions 1, 5, 8 and
// g 1) and x = nx - 1 (3, 6, 7 and g 3) from the node's own opposites: own f 3,
// f 7, f 6, g 3 (left) or f 1, f 8, f 5, g 1 (right), and the wall's temperature term.
template <bool FLAT>
__device__ __forceinline__ void side_walls(F2 (&f)[9], F2 (&g)[5], const MarchLane& n, const MarchArgs& M, float of,
                                           float oa, float ob, float og, float add) {
    // Selects, not an assignment to one half of a packed pair in a divergent branch (see
    // step_band.cuh). FLAT: both sides' without a branch (float32, 1 % faster; in 16-bit
    // storage the registers it takes cost 2 %).
    const bool rl = n.right && !n.rhi, rh = n.right && n.rhi;
    auto left = [&](F2 v, float w) { return f2_pack(n.left ? w : f2_lo(v), f2_hi(v)); };
    auto right = [&](F2 v, float w) { return f2_pack(rl ? w : f2_lo(v), rh ? w : f2_hi(v)); };
    if (FLAT || n.wall_l) {
        f[1] = left(f[1], of);
        f[5] = left(f[5], oa);
        f[8] = left(f[8], ob);
        g[1] = left(g[1], wall_value(M.sign_l, og, add));
    }
    if (FLAT || n.wall_r) {
        f[3] = right(f[3], of);
        f[6] = right(f[6], oa);
        f[7] = right(f[7], ob);
        g[3] = right(g[3], wall_value(M.sign_r, og, add));
    }
}

// Largest |value| seen, a NaN kept (three-input maximum of sm_100+).
__device__ __forceinline__ float peak_of(float acc, float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(acc), "f"(fabsf(a)), "f"(fabsf(b)));
    return d;
}

// Random states of a pair (stochastic rounding), as in process_item.
__device__ __forceinline__ void pair_random(unsigned salt, int j, const MarchLane& n, const StepArgs& A, unsigned& r0,
                                            unsigned& r1) {
    const unsigned i = (unsigned)(j + A.jglob0) * (unsigned)A.pitch + (unsigned)n.x0;
    r0 = hash32(i ^ salt);
    r1 = hash32((i + 1u) ^ salt);
}

// A pair's stored planes into the warp's output tile (c: the lane's column there).
template <typename L>
__device__ __forceinline__ void pair_tile(const PairStored<L>& s, unsigned char* tile, int c) {
    using G = MarchGeo<L>;
    using Ef = typename L::Ef;
    using Eg = typename L::Eg;
    constexpr int W = G::kCols;
    auto put = [&](unsigned char* p, auto v) { *reinterpret_cast<decltype(v)*>(p) = v; };
#pragma unroll
    for (int k = 0; k < 9; ++k) put(tile + (L::pf(k) * W + c) * (int)sizeof(Ef), s.f[k]);
    if constexpr (L::kTheta) {
        put(tile + G::g_at(W) + c * 4, s.theta);
#pragma unroll
        for (int k = 1; k < 5; ++k) put(tile + G::d_at(W) + ((k - 1) * W + c) * 2, s.g[k]);
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) put(tile + G::g_at(W) + (L::pg(k) * W + c) * (int)sizeof(Eg), s.g[k]);
    }
}

// Sums the rows of steps not yet in the ring (pending = 1: the last step's, local
// Nusselt numbers; T: those of the T steps of a march launch, as temperatures, each
// turned into its local number on the way), in the order of nu_finish_prev; taken:
// the steps this launch takes (0: the finalize launch). Called by all of block
// `block` of the M.nu_blocks that share the partial streams; the last of them to
// arrive adds these up.
//
// A row's number takes five float64 operations, and float64 is a slow pipe here, so for
// tall cavities one block would be longer than the launch around it (200 x 20000 mixed,
// 192 steps: 17.1 ms with one block, 9.1 with eight; 27.2 with one block, a pass of its
// own for the numbers and then one warp per step): one block per 512 rows, up to eight
// (march_args). U: rows of a stream in flight per lane, two in the single-cavity
// launches (four cost 2048^2 in float32, whose registers are at their limit, 4 %), one in
// the batched ones (two cost 64 cavities 2 %), four in the finalize launches.
constexpr int kMarchSumThreads = 256 * kMarchMax;  // of the finalize launch
constexpr int kMarchSumBlocks = 8;
using MarchPart = double[8][32];                   // [kMarchMax] in shared memory
template <int U>
__device__ __forceinline__ void march_nu_finish(const MarchArgs& M, int taken, MarchPart* shared_part, int block) {
    const StepArgs& A = M.A;
    const long long t = __ldcg(A.step_in);
    const int pend = min((int)__ldcg(A.pending), kMarchMax);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int nq = nu_partials(A.ny);
    MarchPart* const part = M.nu_blocks > 1 ? M.nu_part : shared_part;
    for (int task = warp * M.nu_blocks + block; task < nq * pend; task += M.nu_blocks * warps) {
        const int set = task / nq, q = task - set * nq;
        double* rows = M.prev_rows[set];
        auto local = [&](int r) {
            if (pend == 1) return __ldcg(rows + r);
            const float2 th = __ldcg(reinterpret_cast<const float2*>(rows) + r);
            const double tw = (double)__ldg(A.hot + r);
            return M.nu_scale * (8.0 * tw - 9.0 * (double)th.x + (double)th.y);
        };
        auto keep = [&](int r, double v) {  // (a row's slot holds both forms)
            if (pend > 1 && DMRT_IN(r, 0, A.ny, A.err)) rows[r] = v;
        };
        double acc = 0.0;
        int r = lane + 32 * q;
        if (r < A.ny) {  // the partial starts from its first row
            acc = local(r);
            keep(r, acc);
            r += 256;
        }
#pragma unroll U
        for (; r < A.ny; r += 256) {
            const double v = local(r);
            acc += v;
            keep(r, v);
        }
        part[set][q][lane] = acc;
    }
    // (every thread has read the counters before the last block rewrites them)
    if (M.nu_blocks > 1) {
        __threadfence();
        __syncthreads();
        const bool more = threadIdx.x == 0 && atomicInc(M.nu_arrivals, M.nu_blocks - 1) != M.nu_blocks - 1u;
        if (__syncthreads_or(more)) return;
        __threadfence();
    } else {
        __syncthreads();
    }
    if (warp < pend) {
        double p8[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) p8[q] = *(volatile double*)&part[warp][q][lane];  // (those past nq are left out)
        double s = nu_combine(p8, nq);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (lane == 0) {
            const double mean = s * A.nu_inv;
            const long long slot = (t - 1 - warp) % A.cap;
            // (a ring of fewer slots keeps the latest steps)
            if (warp < A.cap && DMRT_IN(slot, 0, A.cap, A.err)) A.nu_ring[slot] = mean;
            if (warp == 0) *A.nu_last = mean;
        }
    }
    if (threadIdx.x == 0) {
        if (taken > 0) *A.step_out = t + taken;
        *A.pending = (unsigned)taken;
    }
}

// The last launch's sums alone, after a run: M.nu_blocks blocks. (Three steps of 1024^2 in
// float32 with their sums: 45.9 us; 54.5 by one block of four warps.)
static __global__ void __launch_bounds__(kMarchSumThreads) march_finalize_kernel(MarchArgs M) {
    __shared__ MarchPart part[kMarchMax];
    grid_dep_wait();  // (launched while the last step finishes)
    march_nu_finish<4>(M, 0, part, blockIdx.x);
}

// What a step needs of the step before it (see the top), the next pull being
// at row q: the P group of row q - 1, shifted for the pull, the P and Z groups
// of row q as they are, and in wall lanes row q's own f 7 (left) or f 8 (right)
// and wall term.
struct MarchCarry {
    F2 of2, of5, of6, og2;  // row q - 1
    F2 pf2, pf5, pf6, pg2;  // row q
    F2 zf0, zf1, zf3, zg0, zg1, zg3;
    float wa, wadd;
};

// One item (strip, chunk) of a cavity by one warp: ring and bars are the warp's,
// the barriers freshly initialised. FIRST: the rows that the first iteration needs are
// waited for before the loop, as the batched launches have it (64 cavities in float32
// 36.2 us per step, 36.4 with that wait in the loop); the single-cavity launches wait in the
// loop (2048^2 in float32 33.0 us, 34.0 with it before).
template <typename L, bool SR, int T, bool FIRST>
__device__ __forceinline__ void march_item(const CUtensorMap* ld, const CUtensorMap* st, const MarchArgs& M,
                                           const PairRates& K, const PairNumbers& C9, int item, int lane,
                                           unsigned char* ring, uint64_t* bars,
                                           unsigned long long limit_ns = kWaitLimitNs) {
    using G = MarchGeo<L>;
    static_assert(T >= 2 && T <= kMarchMax && T - 1 <= G::kLead, "a strip's side columns");
    const StepArgs& A = M.A;
    unsigned char* const tile = ring + kMarchStages * G::kStage;
    const int cidx = item / M.n_strips, strip = item - cidx * M.n_strips;
    const int j0 = cidx * M.chunk, j1 = min(j0 + M.chunk, A.ny);
    MarchLane n;
    n.x0 = strip * G::kCols - G::kLead + 2 * lane;
    n.c = 2 * lane + G::kHalo - G::kLead;
    const bool stores = lane >= G::kFirst && lane < G::kFirst + G::kCols / 2;
    n.out = stores && n.x0 < A.nx;
    n.two = n.x0 + 1 < A.nx;
    n.left = n.x0 == 0;
    n.right = n.x0 >= 0 && (n.x0 == A.nx - 1 || n.x0 + 1 == A.nx - 1);
    n.rhi = n.x0 + 1 == A.nx - 1;
    n.wall_l = strip == 0;
    n.wall_r = (strip + 1) * G::kCols + G::kLead >= A.nx;
    n.wall = n.wall_l || n.wall_r;
    unsigned salt[T];
#pragma unroll
    for (int s = 0; s < T; ++s)
        salt[s] = SR ? hash32(((unsigned)*A.step_in + (unsigned)s) * 0x9e3779b9u + 0x632be5abu) : 0u;
    float peak0 = 0.f, peak1 = 0.f;  // largest |rho|, |theta| of the lane's two columns
    // Step s takes rows max(j0 - (T - 1 - s), 0) .. min(j1 - 1 + (T - 1 - s), ny - 1).
    const int rs = max(j0 - (T - 1), 0), rend = j1 - 1 + (T - 1);
    const int lb = max(rs - 1, 0), ub = min(min(rend, A.ny - 1) + 1, A.ny - 1);  // rows loaded
    auto stage = [&](int row) { return ring + ((row - lb) & (kMarchStages - 1)) * G::kStage; };
    auto bar = [&](int row) { return &bars[(row - lb) & (kMarchStages - 1)]; };
    auto issue = [&](int row) {  // lane 0: the copies of a row into its stage
        unsigned char* s = stage(row);
        uint64_t* b = bar(row);
        const int x = strip * G::kCols - G::kHalo;
        mbar_expect_tx(b, G::kRowBytes);
        tma_load_3d(s, &ld[0], x, row, 0, b);
        if constexpr (L::kSplit) tma_load_3d(s + G::g_at(G::kBox), &ld[1], x, row, 0, b);
        if constexpr (L::kTheta) tma_load_3d(s + G::d_at(G::kBox), &ld[2], x, row, 0, b);
    };
    auto arrived = [&](int row) {
        return __all_sync(kFull, mbar_wait_bounded(bar(row), (unsigned)((row - lb) / kMarchStages) & 1u, limit_ns));
    };
    int issued = min(ub + 1, lb + kMarchStages);  // rows below this one have been issued
    if (lane == 0)
        for (int row = lb; row < issued; ++row) issue(row);
    bool ok = true;
    int waited = lb;  // rows below this one have arrived (!ok: those below waited - 1)
    // On expiry: record it, and wait (bounded) for the copies from the row that failed on.
    auto give_up = [&]() {
        if (lane != 0) return;
        atomicOr(A.err, kErrTimeout);
        for (int row = waited - 1; row < issued; ++row)
            mbar_wait_bounded(bar(row), (unsigned)((row - lb) / kMarchStages) & 1u, limit_ns);
    };
    if constexpr (FIRST) {
        for (; waited <= rs && ok; ++waited) ok = arrived(waited);
        if (!ok) return give_up();
    }

    MarchCarry C[T - 1];
#pragma unroll
    for (int s = 0; s < T - 1; ++s) {
        MarchCarry& X = C[s];
        X.of2 = X.of5 = X.of6 = X.og2 = X.pf2 = X.pf5 = X.pf6 = X.pg2 = 0;
        X.zf0 = X.zf1 = X.zf3 = X.zg0 = X.zg1 = X.zg3 = 0;
        X.wa = X.wadd = 0.f;
    }
    auto wall_term = [&](int r) {
        return n.left ? __fmul_rn(M.abb_l, __ldg(M.wall_l + r)) : n.right ? __fmul_rn(M.abb_r, __ldg(M.wall_r + r)) : 0.f;
    };
    float nadd = n.wall ? wall_term(rs) : 0.f;  // the next row's wall term
    auto own = [&](F2 v) { return n.right && n.rhi ? f2_hi(v) : f2_lo(v); };
    auto nusselt = [&](int s, int j, F2 theta) {  // row j of step s
        if (n.left && j >= j0 && j < j1 && DMRT_IN(j, 0, A.ny, A.err))
            reinterpret_cast<F2*>(M.nu_rows[T - 1 - s])[j] = theta;
    };
    auto watch = [&](F2 rho, F2 theta) {
        peak0 = peak_of(peak0, f2_lo(rho), f2_lo(theta));
        peak1 = peak_of(peak1, f2_hi(rho), f2_hi(theta));
    };
    // Iteration r: step s at row r - s. Every step runs in every iteration: the
    // rows below a chunk's first (in its first iterations) and above the cavity
    // (in a topmost chunk's last) are computed from whatever the stages and the
    // carried state hold, and used by nothing. (Branches around the steps cost
    // more in register moves than the T (T - 1) / 2 extra rows per chunk; so did
    // unrolling the loop, in instruction fetches.)
    const int last = min(rend, A.ny - 1);
#pragma unroll 1
    for (int r = rs; r <= rend; ++r) {
        // Rows up to r + 1 have arrived (without FIRST, the first iteration waits for all from lb on).
        if constexpr (FIRST) {
            if (waited <= ub) {
                ok = arrived(waited);
                ++waited;
                if (!ok) break;
            }
        } else {
            for (; ok && waited <= min(r + 1, ub); ++waited) ok = arrived(waited);
            if (!ok) break;
        }
        F2 f[9], g[5], rho, theta;
        float add = nadd;
        // Step 0 from the stages.
        const unsigned char* Z = stage(r);
        const unsigned char* P = stage(r - 1);
        const unsigned char* N = stage(r + 1);
        const int c = n.c;
        f[0] = row_f<L, 0>(Z, 0, c);
        f[1] = row_f<L, 1>(Z, 1, c);
        f[3] = row_f<L, -1>(Z, 3, c);
        g[0] = row_g<L, 0>(Z, 0, c, M);
        g[1] = row_g<L, 1>(Z, 1, c, M);
        g[3] = row_g<L, -1>(Z, 3, c, M);
        if (r > 0) {
            f[2] = row_f<L, 0>(P, 2, c);
            f[5] = row_f<L, 1>(P, 5, c);
            f[6] = row_f<L, -1>(P, 6, c);
            g[2] = row_g<L, 0>(P, 2, c, M);
        } else {  // bottom wall: the node's own opposites
            f[2] = row_f<L, 0>(Z, 4, c);
            f[5] = row_f<L, 0>(Z, 7, c);
            f[6] = row_f<L, 0>(Z, 8, c);
            g[2] = row_g<L, 0>(Z, 4, c, M);
        }
        if (r < A.ny - 1) {
            f[4] = row_f<L, 0>(N, 4, c);
            f[7] = row_f<L, -1>(N, 7, c);
            f[8] = row_f<L, 1>(N, 8, c);
            g[4] = row_g<L, 0>(N, 4, c, M);
        } else {
            f[4] = row_f<L, 0>(Z, 2, c);
            f[7] = row_f<L, 0>(Z, 5, c);
            f[8] = row_f<L, 0>(Z, 6, c);
            g[4] = row_g<L, 0>(Z, 2, c, M);
        }
        if (n.wall) {
            const bool lf = n.left;
            const float of = own(lf ? row_f<L, 0>(Z, 3, c) : row_f<L, 0>(Z, 1, c));
            const float oa = own(lf ? row_f<L, 0>(Z, 7, c) : row_f<L, 0>(Z, 8, c));
            const float ob = own(lf ? row_f<L, 0>(Z, 6, c) : row_f<L, 0>(Z, 5, c));
            const float og = own(lf ? row_g<L, 0>(Z, 3, c, M) : row_g<L, 0>(Z, 1, c, M));
            side_walls<!G::k16>(f, g, n, M, of, oa, ob, og, add);
            if (r < last) nadd = wall_term(r + 1);  // in flight during this row
        }
        __syncwarp();  // every lane has read row r - 1: its stage takes the next row to load
        if (issued <= ub && issued <= r - 1 + kMarchStages) {
            if (lane == 0) issue(issued);
            ++issued;
        }
        collide_pair(f, g, K, C9, rho, theta);
        if (r < A.ny) watch(rho, theta);
        if (strip == 0) nusselt(0, r, theta);
#pragma unroll
        for (int s = 1; s < T; ++s) {
            const int q = r - s;  // the row of step s; f, g hold step s - 1 at row q + 1
            if constexpr (kShifted<typename L::Ef>) {
                unsigned r0 = 0, r1 = 0;
                if constexpr (SR) pair_random(salt[s - 1], q + 1, n, A, r0, r1);
                const PairStored<L> e = pair_encode<L, SR>(f, g, theta, M, r0, r1);
                pair_decode<L>(e, M, f, g);
            }
            MarchCarry& X = C[s - 1];
            F2 F[9], H[5];
            F[0] = X.zf0;
            F[1] = pull_px(X.zf1);
            F[3] = pull_mx(X.zf3);
            H[0] = X.zg0;
            H[1] = pull_px(X.zg1);
            H[3] = pull_mx(X.zg3);
            F[2] = X.of2;
            F[5] = X.of5;
            F[6] = X.of6;
            H[2] = X.og2;
            F[4] = f[4];
            F[7] = pull_mx(f[7]);
            F[8] = pull_px(f[8]);
            H[4] = g[4];
            if (q == A.ny - 1) F[4] = X.pf2, F[7] = X.pf5, F[8] = X.pf6, H[4] = X.pg2;  // top wall: own opposites
            const float padd = X.wadd;
            if (n.wall) {
                const bool lf = n.left;
                side_walls<!G::k16>(F, H, n, M, own(lf ? X.zf3 : X.zf1), X.wa, own(lf ? X.pf6 : X.pf5),
                           own(lf ? X.zg3 : X.zg1), padd);
                X.wa = n.left ? f2_lo(f[7]) : own(f[8]);
                X.wadd = add;
                add = padd;
            }
            X.of2 = X.pf2;
            X.of5 = pull_px(X.pf5);
            X.of6 = pull_mx(X.pf6);
            X.og2 = X.pg2;
            if (q + 1 == 0) X.of2 = f[4], X.of5 = f[7], X.of6 = f[8], X.og2 = g[4];  // bottom wall: own opposites
            X.pf2 = f[2], X.pf5 = f[5], X.pf6 = f[6], X.pg2 = g[2];
            X.zf0 = f[0], X.zf1 = f[1], X.zf3 = f[3], X.zg0 = g[0], X.zg1 = g[1], X.zg3 = g[3];
#pragma unroll
            for (int k = 0; k < 9; ++k) f[k] = F[k];
#pragma unroll
            for (int k = 0; k < 5; ++k) g[k] = H[k];
            collide_pair(f, g, K, C9, rho, theta);
            if (q < A.ny && q >= max(j0 - (T - 1 - s), 0)) watch(rho, theta);
            if (strip == 0) nusselt(s, q, theta);
        }
        const int q = r - (T - 1);
        if (q >= j0) {
            unsigned r0 = 0, r1 = 0;
            if constexpr (SR) pair_random(salt[T - 1], q, n, A, r0, r1);
            const PairStored<L> e = pair_encode<L, SR>(f, g, theta, M, r0, r1);
            if (lane == 0) bulk_wait_read_all();  // the last row's store has read the tile
            __syncwarp();
            if (stores) pair_tile<L>(e, tile, 2 * (lane - G::kFirst));
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                const int x = strip * G::kCols;
                tma_store_3d(&st[0], tile, x, q, 0);
                if constexpr (L::kSplit) tma_store_3d(&st[1], tile + G::g_at(G::kCols), x, q, 0);
                if constexpr (L::kTheta) tma_store_3d(&st[2], tile + G::d_at(G::kCols), x, q, 0);
                bulk_commit();
            }
        }
    }
    if (lane == 0) bulk_wait_all();  // the stores have read the tile and written global memory
    if (!ok) give_up();
    if (n.out && (!(peak0 < 1e30f) || (n.two && !(peak1 < 1e30f)))) atomicOr(A.err, kErrNonFinite);
}

// A warp's ring and barriers.
template <typename L>
__device__ __forceinline__ void march_warp(unsigned char* smem, int warp, int lane, unsigned char*& ring, uint64_t*& bars) {
    using G = MarchGeo<L>;
    ring = smem + warp * G::kWarp;
    bars = reinterpret_cast<uint64_t*>(smem + (kMarchThreads / 32) * G::kWarp) + warp * kMarchStages;
    if (lane == 0) {
        for (int s = 0; s < kMarchStages; ++s) mbar_init(&bars[s], 1);
        mbar_fence_init();
    }
}

template <typename L, bool SR, int T, int MINB>
__global__ void __launch_bounds__(kMarchThreads, MINB)
    step_march_kernel(const __grid_constant__ MarchMaps maps, const __grid_constant__ MarchArgs M,
                      const __grid_constant__ PairConsts K) {
    extern __shared__ __align__(1024) unsigned char smem_m[];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(kFull, (int)threadIdx.x >> 5, 0);  // (uniform, as the compiler sees it)
    unsigned char* ring;
    uint64_t* bars;
    march_warp<L>(smem_m, warp, lane, ring, bars);
    grid_dep_wait();
    grid_dep_launch();
    // After an expired wait in an earlier launch the state is invalid: return at once.
    if (__syncthreads_or(threadIdx.x == 0 && (*reinterpret_cast<volatile unsigned*>(M.A.err) & kErrTimeout))) return;
    const int extra = (int)blockIdx.x - ((int)gridDim.x - M.nu_blocks);
    if (extra >= 0) {  // the last blocks: the previous launch's Nusselt sums (they have no rows)
        march_nu_finish<2>(M, T, reinterpret_cast<MarchPart*>(smem_m), extra);
        return;
    }
    const int item = blockIdx.x * (kMarchThreads / 32) + warp;
    if (item >= M.n_strips * M.n_chunks) return;
    march_item<L, SR, T, false>(maps.ld, maps.st, M, K.r, K.n, item, lane, ring, bars);
}

// ---- batched sweep ----------------------------------------------------------------
// The same launch over the items of up to kMarchBatch cavities, cavity after
// cavity. The cavities' arguments and rates are kernel parameters, so that a
// warp takes them from the constant bank at its cavity's (uniform) index, as
// the single-cavity kernel does; the tensor maps lie in global memory. The last
// n_cav nu_blocks blocks take the cavities' Nusselt sums.
constexpr int kMarchBatch = 80;  // (parameters of at most 32764 bytes)
struct MarchBatchArgs {
    const CUtensorMap* maps;  // [n_cav][6]: loads, stores of this launch's source buffer
    unsigned* err;            // the batch's error word (an expired wait)
    PairNumbers n;
    int n_cav, items;
    int nu_blocks;            // of each cavity
    unsigned* ctr;            // the single-step launches' two work-pool counters, cleared here (they
                              // alternate by source buffer, which march launches in between do not
                              // keep up); nullptr: another launch clears them
    int first[kMarchBatch];   // first item of each cavity
    MarchArgs M[kMarchBatch];
    PairRates r[kMarchBatch];
};

template <typename L, bool SR, int T, int MINB>
__global__ void __launch_bounds__(kMarchThreads, MINB) batch_march_kernel(const __grid_constant__ MarchBatchArgs B) {
    extern __shared__ __align__(1024) unsigned char smem_m[];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(kFull, (int)threadIdx.x >> 5, 0);
    unsigned char* ring;
    uint64_t* bars;
    march_warp<L>(smem_m, warp, lane, ring, bars);
    grid_dep_wait();
    grid_dep_launch();
    if (__syncthreads_or(threadIdx.x == 0 && (*reinterpret_cast<volatile unsigned*>(B.err) & kErrTimeout))) return;
    const int extra = (int)blockIdx.x - ((int)gridDim.x - B.n_cav * B.nu_blocks);
    if (extra >= 0) {
        if (extra == 0 && B.ctr && threadIdx.x < 2) B.ctr[threadIdx.x] = 0u;
        const int cav = extra / B.nu_blocks;
        march_nu_finish<1>(B.M[cav], T, reinterpret_cast<MarchPart*>(smem_m), extra - cav * B.nu_blocks);
        return;
    }
    const int item = blockIdx.x * (kMarchThreads / 32) + warp;
    if (item >= B.items) return;
    int lo = 0, hi = B.n_cav - 1;  // the cavity whose items hold this one
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (B.first[mid] <= item) lo = mid;
        else hi = mid - 1;
    }
    const CUtensorMap* maps = B.maps + (size_t)lo * 6;
    march_item<L, SR, T, true>(maps, maps + 3, B.M[lo], B.r[lo], B.n, item - B.first[lo], lane, ring, bars);
    if (lane == 0 && (*reinterpret_cast<volatile unsigned*>(B.M[lo].A.err) & kErrTimeout)) atomicOr(B.err, kErrTimeout);
}

// The last launch's Nusselt sums of every cavity, nu_blocks blocks each.
static __global__ void __launch_bounds__(kMarchSumThreads)
    batch_march_finalize_kernel(const __grid_constant__ MarchBatchArgs B) {
    __shared__ MarchPart part[kMarchMax];
    grid_dep_wait();  // (launched while the last step, or another group's sums, finish)
    const int cav = blockIdx.x / B.nu_blocks;
    march_nu_finish<4>(B.M[cav], 0, part, blockIdx.x - cav * B.nu_blocks);
}

// The compiled form for a storage, rounding and steps per launch, its shared memory, and the
// columns of a strip, of a load box and left of the strip (nullptr: none).
struct MarchForm {
    const void* func;
    unsigned smem;
    int cols, box;
};
static_assert(sizeof(MarchBatchArgs) <= 32764, "kernel parameters");
MarchForm march_form(int storage, int rounding, int steps);
MarchForm batch_march_form(int storage, int rounding, int steps);  // float32 and mixed storage

// One float32 item by one warp (first: in the batched launches' form), the copy of the
// chunk's row `row` (from its first one loaded) never complete: the barrier waits for an
// arrival that nobody makes.
cudaError_t launch_march_wait_probe(const MarchMaps& maps, const MarchArgs& M, const PairConsts& K, int item, int row,
                                    bool first, unsigned long long limit_ns, cudaStream_t stream);

}  // namespace dmrt
