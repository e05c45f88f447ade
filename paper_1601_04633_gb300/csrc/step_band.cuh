// Many time steps per launch with the whole cavity on chip, spread over the GPU:
// block b (one per SM, a cooperative launch) keeps rows [b h, (b + 1) h) of the
// cavity in its shared memory, both buffers, and each step exchanges one row
// of crossing populations with the blocks below and above.
//
// For cavities too large for one thread-block cluster (step_cluster.cuh) and
// too small to fill the GPU from HBM or L2, a launch per step (or per three,
// step_march.cuh) costs mostly launch and pipeline latency. Here a step costs
// the exchange (0.8 to 1.1 us measured alone, for rows of 128 and 256 columns) and
// the block's own rows.
//
// Exchange. A row's message is, per plane, the nx values, each in an 8-byte
// word with the step's tag in its high half, written with relaxed 16-byte
// stores of two words and polled by the thread that needs them: a word holds
// its value exactly when the tag is right (a word is written at once), so no
// fence, flag or counter is needed, and the message's latency is one store
// and one load through L2. The upward message holds f 2, f 5, f 6, g 2 of the
// block's last row, the downward one f 4, f 7, f 8, g 4 of its first row. Two
// message slots alternate by step: a thread sends its columns after it has
// read the neighbour's words of the step before, and the neighbour overwrites a
// word two steps later, after it has read this thread's and its neighbours'
// words of the step between, so every reader of the old word is done. Tags
// come from a device counter that the launch's last kernel advances, so no
// word of an earlier launch, or of a replayed one, carries a live tag.
//
// Each thread owns fixed pairs of nodes (collide_pair, the bits of the other
// kernels). 16-bit storage is rounded every step as a store would round it
// (pair_encode / pair_decode); the last step stores its rounded values straight
// to the global buffer. The temperatures at x = 0, 1 of every row and step go to
// a record that the launch's last kernel turns into Nusselt numbers.
//
// What bounds it: up to 192^2 the exchange and the serial chain of a pair's
// collision, above it the blocks' float32 pipes as well (512^2: 1.2 us of its
// 3.5 us per step). Measured at the rule in dmrt.cu (setup_band).
//
// Every poll is bounded: on expiry the block records kErrTimeout and returns,
// and its neighbours' polls expire in turn.
#pragma once
#include <cooperative_groups.h>

#include "step_march.cuh"

namespace dmrt {

constexpr int kBandThreads = 512;  // most threads of a block (128 registers each)
constexpr int kBandWide = 576;     // ... of the form for 513 to 576 pairs (96 registers each)
constexpr int kBandSteps = 512;    // most steps per launch (the Nusselt record's length)
constexpr int kBandMinSteps = 6;   // shorter runs take the other kernels

struct BandArgs {
    MarchArgs M;        // M.A: source buffer and cavity (A.dst unused); constants
    unsigned char* out; // the buffer that takes the final state
    F2* record;         // [kBandSteps][ny] theta at x = 0, 1
    ulonglong2* mail;   // [2 slots][blocks][2 sides][4 planes][words / 2]
    unsigned* epoch;    // tags of this launch start at *epoch + 1
    long long* t_base;  // steps taken before this launch (block 0 leaves it for band_nu_kernel)
    double* last_rows;  // local Nu of the last step
    long long* step_end;  // the counter slot of the final buffer
    int steps, rows;    // steps of the launch; rows per block (h)
    int pairs, words;   // pairs per row; words per message plane (two more on each side of the row)
    unsigned magic;     // ceil(2^32 / row_threads)
    int row_threads;    // pairs of a row rounded up to whole warps
    float* states;      // not null (float32): the state after step s to states + s * stride too
    long long stride;   // floats between recorded states
};

// Item i of a block of nr rows: its row, the rows next to the block's edges
// last, so that a thread with several items starts with those that wait for
// no message, and its first column (past the row: no pair). A row's items fill
// whole warps, so that a warp waits for the messages of one side only.
__device__ __forceinline__ void band_item(const BandArgs& B, int i, int nr, int& r, int& x0) {
    const int k = (int)__umulhi((unsigned)i, B.magic);
    x0 = 2 * (i - k * B.row_threads);
    r = nr <= 2 ? k : k < nr - 2 ? k + 1 : k == nr - 2 ? 0 : nr - 1;
}

// Shared-memory row stride in floats: the row's pairs with two columns on each side.
__host__ __device__ constexpr int band_stride(int nx) { return (nx + 1) / 2 * 2 + 4; }
__host__ __device__ constexpr size_t band_smem(int rows, int nx) { return (size_t)2 * 14 * rows * band_stride(nx) * 4; }

// In one cluster: with the message slots and their barriers.
constexpr int kBandCluster = 16;
__host__ __device__ constexpr size_t band_cluster_smem(int rows, int nx) {
    return band_smem(rows, nx) + (size_t)16 * band_stride(nx) * 4 + 4 * 8;
}

__device__ __forceinline__ void mail_put(ulonglong2* p, F2 v, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"((v & 0xffffffffull) | t),
                 "l"((v >> 32) | t)
                 : "memory");
}
__device__ __forceinline__ void mail_get2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long mail_get(const unsigned long long* p) {
    unsigned long long a;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    return a;
}

// The pulled pairs of a message at columns x0, x0 + 1: planes 0 and 3 unshifted,
// plane 1 from x - EX, plane 2 from x + EX (EX = 1 for the upward message: f 2,
// f 5, f 6, g 2; -1 for the downward one: f 4, f 7, f 8, g 4). box: the words of
// column 0, plane 0. false: the poll expired.
template <int EX>
__device__ __forceinline__ bool mail_read(const unsigned long long* box, int words, int x0, bool first, bool last,
                                          unsigned tag, F2 (&v)[4], unsigned long long limit_ns = kWaitLimitNs) {
    const unsigned long long* p = box + x0;
    const unsigned long long* pl = p + (EX > 0 ? 1 : 2) * words;  // the plane pulled from the left
    const unsigned long long* pr = p + (EX > 0 ? 2 : 1) * words;  // and from the right
    unsigned long long t0 = 0;
    for (int tries = 0;; ++tries) {
        unsigned long long a0, a1, d0, d1;
        mail_get2(p, a0, a1);
        mail_get2(p + 3 * words, d0, d1);
        const unsigned long long l0 = first ? (unsigned long long)tag << 32 : mail_get(pl - 1), l1 = mail_get(pl);
        const unsigned long long r0 = mail_get(pr + 1), r1 = last ? (unsigned long long)tag << 32 : mail_get(pr + 2);
        const unsigned miss = ((unsigned)(a0 >> 32) ^ tag) | ((unsigned)(a1 >> 32) ^ tag) | ((unsigned)(d0 >> 32) ^ tag) |
                              ((unsigned)(d1 >> 32) ^ tag) | ((unsigned)(l0 >> 32) ^ tag) | ((unsigned)(l1 >> 32) ^ tag) |
                              ((unsigned)(r0 >> 32) ^ tag) | ((unsigned)(r1 >> 32) ^ tag);
        if (miss == 0) {
            v[0] = (a0 & 0xffffffffull) | (a1 << 32);
            v[3] = (d0 & 0xffffffffull) | (d1 << 32);
            const F2 l = (l0 & 0xffffffffull) | (l1 << 32), r = (r0 & 0xffffffffull) | (r1 << 32);
            v[1] = EX > 0 ? l : r;
            v[2] = EX > 0 ? r : l;
            return true;
        }
        if ((tries & 255) == 255) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit_ns) return false;
        }
    }
}

// One cluster of up to 16 blocks (small cavities): the same steps, the messages
// going straight into the neighbour's shared memory (st.async, which counts its
// bytes on an mbarrier there) instead of through L2: a message then takes about a
// quarter of a microsecond. A barrier per slot and side is armed with the
// message's bytes one step ahead; a thread that needs the message waits for it.
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_put(unsigned addr, F2 v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(v), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool cluster_wait(uint64_t* bar, unsigned parity, unsigned long long limit_ns = kWaitLimitNs) {
    unsigned long long t0 = 0;
    for (;;) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > limit_ns) return false;
    }
}

// CL: one cluster, messages through shared memory; else a cooperative launch of
// blocks, messages through L2.
// ONE: a thread has at most one pair (its place, walls and addresses then are
// fixed before the steps); else it loops over its pairs in every step.
// MAXT: the most threads: a block of 513 to 576 pairs takes them in one pass with
// fewer registers (383 x 389: 2.67 -> 2.09 us per step; blocks of two passes lose
// 5 % with so few: 512^2 3.49 -> 3.68).
template <typename L, bool SR, bool CL, bool ONE, int MAXT>
__global__ void __launch_bounds__(MAXT) step_band_kernel(const __grid_constant__ BandArgs B,
                                                                 const __grid_constant__ PairConsts K) {
    using Ef = typename L::Ef;
    using Eg = typename L::Eg;
    const MarchArgs& M = B.M;
    const StepArgs& A = M.A;
    extern __shared__ __align__(16) float smem_b[];
    const int nx = A.nx, ny = A.ny, h = B.rows, WS = band_stride(nx);
    const int blk = blockIdx.x, nblk = gridDim.x;
    const int r0 = blk * h, nr = min(h, ny - r0);
    const int plane = h * WS;  // floats per plane
    const int buffer = 14 * plane;
    const int items = nr * B.row_threads;
    // Messages in shared memory (CL): [2 slots][2 sides][4 planes][WS], then a barrier per slot and side.
    float* const inbox = smem_b + 2 * buffer;
    uint64_t* const bars = reinterpret_cast<uint64_t*>(inbox + 16 * WS);
    const unsigned message = 4u * 8u * (unsigned)B.pairs;
    if constexpr (CL) {
        if (threadIdx.x == 0) {
            for (int b = 0; b < 4; ++b) mbar_init(&bars[b], 1);
            mbar_fence_init();
            if (blk > 0) mbar_expect_tx(&bars[2], message);  // the messages the first step reads (slot 1)
            if (blk + 1 < nblk) mbar_expect_tx(&bars[3], message);
        }
        cooperative_groups::this_cluster().sync();
    } else if (*reinterpret_cast<volatile unsigned*>(A.err) & kErrTimeout) {
        return;  // an earlier launch's wait expired
    }
    const unsigned tag0 = *B.epoch + 1u;
    const unsigned t_in = (unsigned)*A.step_in;
    if (blk == 0 && threadIdx.x == 0) *B.t_base = *A.step_in;
    // Message slots: what this block sends and reads, by side (0: below, 1: above).
    const size_t slot_words = (size_t)nblk * 2 * 4 * B.words;
    unsigned long long* const mail = reinterpret_cast<unsigned long long*>(B.mail);
    auto box = [&](int slot, int b, int side) { return mail + slot * slot_words + ((size_t)(b * 2 + side) * 4) * B.words + 2; };
    // A pair's messages after a step (post-collision populations f, g of row r).
    auto send = [&](int s, int r, int x0, const F2 (&f)[9], const F2 (&g)[5], unsigned tag) {
        if constexpr (CL) {
            const int slot = s & 1;
            if (r == 0 && blk > 0) {
                const unsigned d = cluster_addr(inbox + (slot * 2 + 1) * 4 * WS + 2 + x0, blk - 1);
                const unsigned b = cluster_addr(&bars[slot * 2 + 1], blk - 1);
                cluster_put(d, f[4], b);
                cluster_put(d + 4 * WS, f[7], b);
                cluster_put(d + 8 * WS, f[8], b);
                cluster_put(d + 12 * WS, g[4], b);
            }
            if (r == nr - 1 && blk + 1 < nblk) {
                const unsigned d = cluster_addr(inbox + (slot * 2) * 4 * WS + 2 + x0, blk + 1);
                const unsigned b = cluster_addr(&bars[slot * 2], blk + 1);
                cluster_put(d, f[2], b);
                cluster_put(d + 4 * WS, f[5], b);
                cluster_put(d + 8 * WS, f[6], b);
                cluster_put(d + 12 * WS, g[2], b);
            }
            return;
        }
        if (r == 0 && blk > 0) {  // downward, into the previous block's box from above
            ulonglong2* p = reinterpret_cast<ulonglong2*>(box(s & 1, blk - 1, 1) + x0);
            const int w = B.words / 2;
            mail_put(p, f[4], tag);
            mail_put(p + w, f[7], tag);
            mail_put(p + 2 * w, f[8], tag);
            mail_put(p + 3 * w, g[4], tag);
        }
        if (r == nr - 1 && blk + 1 < nblk) {
            ulonglong2* p = reinterpret_cast<ulonglong2*>(box(s & 1, blk + 1, 0) + x0);
            const int w = B.words / 2;
            mail_put(p, f[2], tag);
            mail_put(p + w, f[5], tag);
            mail_put(p + 2 * w, f[6], tag);
            mail_put(p + 3 * w, g[2], tag);
        }
    };
    // The state of this block's rows, and the messages that the first step reads.
    {
        const unsigned char* sf = reinterpret_cast<const unsigned char*>(A.src);
        const unsigned char* sg = L::kSplit ? sf + 9 * A.plane * (long long)sizeof(Ef) : sf;
        const unsigned char* sd = sg + A.plane * 4;  // ThetaSplit: the deviations
        for (int i = threadIdx.x; i < items; i += blockDim.x) {
            int r, x0;
            band_item(B, i, nr, r, x0);
            if (x0 >= nx) continue;
            const long long o = (long long)(r0 + r) * A.pitch + x0;
            if (!DMRT_IN(o + 1, 1, A.plane, A.err) || !DMRT_IN(13 * plane + r * WS + 2 + x0 + 1, 0, buffer, A.err)) continue;
            PairStored<L> e;
            using TF = typename PairElem<Ef>::T;
            using TG = typename PairElem<Eg>::T;
#pragma unroll
            for (int k = 0; k < 9; ++k) e.f[k] = *reinterpret_cast<const TF*>(sf + (L::pf(k) * A.plane + o) * (long long)sizeof(Ef));
            if constexpr (L::kTheta) {
                e.theta = *reinterpret_cast<const F2*>(sg + o * 4);
#pragma unroll
                for (int k = 1; k < 5; ++k) e.g[k] = *reinterpret_cast<const unsigned*>(sd + ((k - 1) * A.plane + o) * 2);
            } else {
#pragma unroll
                for (int k = 0; k < 5; ++k) e.g[k] = *reinterpret_cast<const TG*>(sg + (L::pg(k) * A.plane + o) * (long long)sizeof(Eg));
            }
            F2 f[9], g[5];
            pair_decode<L>(e, M, f, g);
            float* q = smem_b + r * WS + 2 + x0;
#pragma unroll
            for (int k = 0; k < 9; ++k) *reinterpret_cast<F2*>(q + k * plane) = f[k];
#pragma unroll
            for (int k = 0; k < 5; ++k) *reinterpret_cast<F2*>(q + (9 + k) * plane) = g[k];
            send(1, r, x0, f, g, tag0);  // (slot of step -1)
        }
    }
    float peak0 = 0.f, peak1 = 0.f;
    bool dead = false;
    auto lane_of = [&](int x0) {
        MarchLane n;
        n.x0 = x0;
        n.two = x0 + 1 < nx;
        n.left = x0 == 0;
        n.right = x0 + 2 >= nx;
        n.rhi = x0 + 1 == nx - 1;
        return n;
    };
    // The pair at row r, column x0 in step s, from buffer S to buffer D.
    auto pair_step = [&](int s, const float* S, float* D, unsigned tag, unsigned salt, int r, int x0, const MarchLane& n) {
        const int j = r0 + r;
        if (!DMRT_IN(13 * plane + r * WS + 2 + x0 + 1, 0, buffer, A.err) || !DMRT_IN(j, 0, ny, A.err)) return;
        const float* q = S + r * WS + 2 + x0;
        auto at = [&](int k, int dr) { return *reinterpret_cast<const F2*>(q + k * plane + dr * WS); };
        // The pulls shifted in x (directions 1, 5, 8, g 1 from the left, 3, 6, 7,
        // g 3 from the right) stay single values until the side walls have
        // replaced theirs. (An earlier form of this code that changed one half of a packed
        // pair in a divergent branch gave a wrong other half; no small case of it was found.)
        auto px = [&](int k, int dr, float (&v)[2]) {
            const float* p = q + k * plane + dr * WS;
            v[0] = p[-1], v[1] = p[0];
        };
        auto mx = [&](int k, int dr, float (&v)[2]) {
            const float* p = q + k * plane + dr * WS;
            v[0] = p[1], v[1] = p[2];
        };
        auto un = [&](F2 a, float (&v)[2]) { v[0] = f2_lo(a), v[1] = f2_hi(a); };
        F2 f[9], g[5];
        float v1[2], v3[2], v5[2], v6[2], v7[2], v8[2], w1[2], w3[2];
        f[0] = at(0, 0);
        g[0] = at(9, 0);
        px(1, 0, v1);
        mx(3, 0, v3);
        px(10, 0, w1);
        mx(12, 0, w3);
        if (r > 0) {
            f[2] = at(2, -1);
            px(5, -1, v5);
            mx(6, -1, v6);
            g[2] = at(11, -1);
        } else if (j == 0) {  // bottom wall: the node's own opposites
            f[2] = at(4, 0);
            un(at(7, 0), v5);
            un(at(8, 0), v6);
            g[2] = at(13, 0);
        } else if constexpr (CL) {
            const int slot = (s & 1) ^ 1;
            dead |= !cluster_wait(&bars[slot * 2], (unsigned)(s >> 1) & 1u);
            const float* m = inbox + slot * 2 * 4 * WS + 2 + x0;
            f[2] = *reinterpret_cast<const F2*>(m);
            v5[0] = m[WS - 1], v5[1] = m[WS];
            v6[0] = m[2 * WS + 1], v6[1] = m[2 * WS + 2];
            g[2] = *reinterpret_cast<const F2*>(m + 3 * WS);
        } else {
            F2 v[4];
            dead |= !mail_read<1>(box((s & 1) ^ 1, blk, 0), B.words, x0, n.left, n.right, tag, v);
            f[2] = v[0], g[2] = v[3];
            un(v[1], v5);
            un(v[2], v6);
        }
        if (r + 1 < nr) {
            f[4] = at(4, 1);
            mx(7, 1, v7);
            px(8, 1, v8);
            g[4] = at(13, 1);
        } else if (j == ny - 1) {
            f[4] = at(2, 0);
            un(at(5, 0), v7);
            un(at(6, 0), v8);
            g[4] = at(11, 0);
        } else if constexpr (CL) {
            const int slot = (s & 1) ^ 1;
            dead |= !cluster_wait(&bars[slot * 2 + 1], (unsigned)(s >> 1) & 1u);
            const float* m = inbox + (slot * 2 + 1) * 4 * WS + 2 + x0;
            f[4] = *reinterpret_cast<const F2*>(m);
            v7[0] = m[WS + 1], v7[1] = m[WS + 2];
            v8[0] = m[2 * WS - 1], v8[1] = m[2 * WS];
            g[4] = *reinterpret_cast<const F2*>(m + 3 * WS);
        } else {
            F2 v[4];
            dead |= !mail_read<-1>(box((s & 1) ^ 1, blk, 1), B.words, x0, n.left, n.right, tag, v);
            f[4] = v[0], g[4] = v[3];
            un(v[1], v7);
            un(v[2], v8);
        }
        // Side walls: links from outside x = 0 and x = nx - 1 from the node's own opposites.
        auto own = [&](int k, int hi) { return q[k * plane + hi]; };
        if (n.left) {
            v1[0] = own(3, 0);
            v5[0] = own(7, 0);
            v8[0] = own(6, 0);
            w1[0] = wall_value(M.sign_l, own(12, 0), __fmul_rn(M.abb_l, __ldg(M.wall_l + j)));
        }
        if (n.right) {
            const int e = n.rhi ? 1 : 0;
            const float wall = wall_value(M.sign_r, own(10, e), __fmul_rn(M.abb_r, __ldg(M.wall_r + j)));
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (i == e) v3[i] = own(1, e), v6[i] = own(8, e), v7[i] = own(5, e), w3[i] = wall;
            }
        }
        f[1] = f2_pack(v1[0], v1[1]);
        f[3] = f2_pack(v3[0], v3[1]);
        f[5] = f2_pack(v5[0], v5[1]);
        f[6] = f2_pack(v6[0], v6[1]);
        f[7] = f2_pack(v7[0], v7[1]);
        f[8] = f2_pack(v8[0], v8[1]);
        g[1] = f2_pack(w1[0], w1[1]);
        g[3] = f2_pack(w3[0], w3[1]);
        F2 rho, theta;
        collide_pair(f, g, K.r, K.n, rho, theta);
        peak0 = peak_of(peak0, f2_lo(rho), f2_lo(theta));
        if (n.two) peak1 = peak_of(peak1, f2_hi(rho), f2_hi(theta));
        if (n.left) B.record[(size_t)s * ny + j] = theta;
        if constexpr (!kShifted<Ef>) {
            if (B.states) {
                float* d = B.states + (size_t)s * B.stride + (size_t)j * A.pitch + x0;
                if (n.two) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) *reinterpret_cast<F2*>(d + plane_f(k) * A.plane) = f[k];
#pragma unroll
                    for (int k = 0; k < 5; ++k) *reinterpret_cast<F2*>(d + plane_g(k) * A.plane) = g[k];
                } else {
#pragma unroll
                    for (int k = 0; k < 9; ++k) d[plane_f(k) * A.plane] = f2_lo(f[k]);
#pragma unroll
                    for (int k = 0; k < 5; ++k) d[plane_g(k) * A.plane] = f2_lo(g[k]);
                }
            }
        }
        const bool final_step = s == B.steps - 1;
        if (kShifted<Ef> || final_step) {
            unsigned h0 = 0, h1 = 0;
            if constexpr (SR) pair_random(salt, j, n, A, h0, h1);
            const PairStored<L> e = pair_encode<L, SR>(f, g, theta, M, h0, h1);
            if (final_step) {
                unsigned char* df = B.out;
                unsigned char* dg = L::kSplit ? df + 9 * A.plane * (long long)sizeof(Ef) : df;
                const long long o = (long long)j * A.pitch + x0;
                if (!DMRT_IN(o + 1, 1, A.plane, A.err)) return;
                auto put = [&](unsigned char* p, auto v) {
                    using T = decltype(v);
                    if (n.two) *reinterpret_cast<T*>(p) = v;
                    else if constexpr (sizeof(T) == 8) *reinterpret_cast<unsigned*>(p) = (unsigned)v;
                    else *reinterpret_cast<unsigned short*>(p) = (unsigned short)v;
                };
#pragma unroll
                for (int k = 0; k < 9; ++k) put(df + (L::pf(k) * A.plane + o) * (long long)sizeof(Ef), e.f[k]);
                if constexpr (L::kTheta) {
                    put(dg + o * 4, e.theta);
#pragma unroll
                    for (int k = 1; k < 5; ++k) put(dg + A.plane * 4 + ((k - 1) * A.plane + o) * 2, e.g[k]);
                } else {
#pragma unroll
                    for (int k = 0; k < 5; ++k) put(dg + (L::pg(k) * A.plane + o) * (long long)sizeof(Eg), e.g[k]);
                }
                return;
            }
            pair_decode<L>(e, M, f, g);
        }
        send(s, r, x0, f, g, tag + 1u);
        float* d = D + r * WS + 2 + x0;
#pragma unroll
        for (int k = 0; k < 9; ++k) *reinterpret_cast<F2*>(d + k * plane) = f[k];
#pragma unroll
        for (int k = 0; k < 5; ++k) *reinterpret_cast<F2*>(d + (9 + k) * plane) = g[k];
    };
    int r1 = 0, x1 = 0;
    band_item(B, min((int)threadIdx.x, items - 1), nr, r1, x1);
    const bool has1 = (int)threadIdx.x < items && x1 < nx;
    const MarchLane n1 = lane_of(x1);
    __syncthreads();
#pragma unroll 1
    for (int s = 0; s < B.steps; ++s) {
        const float* S = smem_b + (s & 1) * buffer;
        float* D = smem_b + ((s & 1) ^ 1) * buffer;
        const unsigned tag = tag0 + (unsigned)s;  // of the messages this step reads
        if constexpr (CL) {
            // This step's messages come into slot s & 1, whose last ones were read in
            // the step before.
            if (threadIdx.x == 0 && s + 1 < B.steps) {
                if (blk > 0) mbar_expect_tx(&bars[(s & 1) * 2], message);
                if (blk + 1 < nblk) mbar_expect_tx(&bars[(s & 1) * 2 + 1], message);
            }
        }
        const unsigned salt = SR ? hash32((t_in + (unsigned)s) * 0x9e3779b9u + 0x632be5abu) : 0u;
        if constexpr (ONE) {
            if (has1) pair_step(s, S, D, tag, salt, r1, x1, n1);
        } else {
#pragma unroll 1
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                int r, x0;
                band_item(B, i, nr, r, x0);
                if (x0 < nx) pair_step(s, S, D, tag, salt, r, x0, lane_of(x0));
            }
        }
        if (__syncthreads_or(dead)) break;
    }
    if constexpr (CL) cooperative_groups::this_cluster().sync();  // no message still on its way to a block that is gone
    if (dead) atomicOr(A.err, kErrTimeout);
    if (!(peak0 < 1e30f) || !(peak1 < 1e30f)) atomicOr(A.err, kErrNonFinite);
}

// After a band launch: the mean Nusselt number of each of its steps into the
// ring, in the order of nu_finish_prev; the last step's local numbers; the step
// counter; nothing pending; the next launch's tags. One warp per step while a lane
// has at most one row of each partial stream (ny <= 256), else one block per step, a
// warp per stream: short runs of tall cavities waited for the one warp's serial sums
// (6 steps of 8 x 8000 in float32: 176 us with it, 61 with a block).
constexpr int kBandNuWarps = 8;
template <bool BLOCK>
__global__ void __launch_bounds__(32 * kBandNuWarps) band_nu_kernel(const __grid_constant__ BandArgs B) {
    const MarchArgs& M = B.M;
    const StepArgs& A = M.A;
    __shared__ double part[BLOCK ? 8 : 1][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = BLOCK ? (int)blockIdx.x : (int)blockIdx.x * kBandNuWarps + warp;
    grid_dep_wait();           // (launched while the steps finish)
    if (s >= B.steps) return;  // (BLOCK: the whole block)
    const long long t = *B.t_base;
    const F2* rec = B.record + (size_t)s * A.ny;
    const bool last = s == B.steps - 1;
    auto nu_of = [&](int r) {
        const double tw = (double)__ldg(A.hot + r);
        const F2 th = rec[r];
        return M.nu_scale * (8.0 * tw - 9.0 * (double)f2_lo(th) + (double)f2_hi(th));
    };
    if (last || B.steps - s <= A.cap) {
        const int nq = nu_partials(A.ny);
        auto stream = [&](int q) {
            double acc = 0.0;
            int r = lane + 32 * q;
            if (r < A.ny) {
                acc = nu_of(r);
                if (last) B.last_rows[r] = acc;
                r += 256;
            }
            if constexpr (BLOCK) {
#pragma unroll 4
                for (; r < A.ny; r += 256) {
                    const double v = nu_of(r);
                    acc += v;
                    if (last) B.last_rows[r] = v;
                }
            }
            return acc;
        };
        double p8[8];
        if constexpr (BLOCK) {
            part[warp][lane] = stream(warp);
            __syncthreads();
            if (warp > 0) return;
#pragma unroll
            for (int q = 0; q < 8; ++q) p8[q] = part[q][lane];
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) p8[q] = q < nq ? stream(q) : 0.0;
        }
        double sum = nu_combine(p8, nq);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
        if (lane == 0) {
            const double mean = sum * A.nu_inv;
            const long long slot = (t + s) % A.cap;
            if (DMRT_IN(slot, 0, A.cap, A.err)) A.nu_ring[slot] = mean;
            if (last) *A.nu_last = mean;
        }
    }
    if (last && lane == 0) {
        *B.step_end = t + B.steps;
        *A.pending = 0u;
        *B.epoch += (unsigned)B.steps + 1u;
    }
}

// The compiled band kernel of a storage and rounding, across the GPU or in one cluster.
// (items: pairs of a block; a cluster's blocks have at most one per thread)
const void* band_kernel(int storage, int rounding, int items);
const void* band_cluster_kernel(int storage, int rounding);

}  // namespace dmrt
