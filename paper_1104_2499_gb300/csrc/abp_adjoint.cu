// abp_adjoint.cu -- pathwise adjoint of the ensemble mean velocity (abp_backward).
//
// With the noise held fixed, the Euler-Maruyama map s_{n+1} = Phi(s_n, theta, z_n)
// of Eqs. (ereservoir), (velocity), (pot) (Sec. 2) is differentiated in reverse:
//   lambda_n = (dPhi/ds_n)^T lambda_{n+1} + dJ/ds_n,     g += (dPhi/dtheta)^T lambda_{n+1}
// for J_i = sum_{n<N} v_n of each trajectory (the time-averaged velocity times N),
// theta = (D, q, c, d, gamma0, a).  The states are recomputed, not stored:
//   level 0  checkpoints in HBM every K steps, written by the forward integrator;
//   level 1  the K-step segment is re-run from its checkpoint, leaving a
//            sub-checkpoint every kSub steps in context-owned scratch memory;
//   level 2  each kSub-step sub-chunk is re-run from its sub-checkpoint into
//            registers and swept in reverse.
// Every re-run repeats the forward arithmetic bit for bit (same Philox words,
// same Box-Muller, same FMA sequence, same position folds), so the adjoint sees
// exactly the trajectory the forward produced.  Gradient terms are summed in
// FP32 within a segment and in FP64 across segments and trajectories.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <type_traits>

#include "abp.h"
#include "abp_ctx.cuh"
#include "abp_device.cuh"
#include "abp_internal.cuh"

namespace abp {
namespace {

#ifndef ABP_ADJ_SUB
#define ABP_ADJ_SUB 8
#endif
// Block size and minimum resident blocks of the paired reverse kernel.
// Measured on the full differentiation workload (1M x 1e5, K = 1,000),
// backward time: one trajectory per thread 318 ms; paired, 210 registers (two
// 128-thread blocks per SM) 313 ms; paired, capped at 168 registers for three
// blocks per SM (no spills) 304 ms; paired with 4-step sub-chunks 324 ms.
#ifndef ABP_ADJ_REV_PAIR_THREADS
#define ABP_ADJ_REV_PAIR_THREADS 128
#endif
#ifndef ABP_ADJ_REV_PAIR_MIN_BLOCKS
#define ABP_ADJ_REV_PAIR_MIN_BLOCKS 3
#endif
constexpr int kRevPairThreads = ABP_ADJ_REV_PAIR_THREADS;
// Aligned whole chunks of the paired level 1 stepped in groups of this many per
// loop iteration (1: one chunk per iteration).
#ifndef ABP_ADJ_L1_GROUP
#define ABP_ADJ_L1_GROUP 4
#endif
// Threads per block of the level-1 kernel: small blocks, so that one fits on
// an SM beside the reverse kernel's blocks and fills the issue slots they
// leave idle.
constexpr int kL1Threads = 128;
constexpr int kSub = ABP_ADJ_SUB;  // steps per register-resident sub-chunk (a multiple of 4)
static_assert(kSub % 4 == 0 && (kBlockSteps % kSub) == 0, "sub-chunks hold whole Philox blocks");

// Sub-chunks lie on absolute multiples of kSub steps (not on offsets from the segment's
// start, where a checkpoint interval that is no multiple of kSub sent every chunk of most
// segments down the one-step-at-a-time path, without the hand-off: backward of 262,144
// trajectories x 4,000 steps, K = 500 5.2 ms then and 2.66 now, K = 333 6.7 and 2.83, K =
// 1,000 2.82 and 2.59), so that a whole chunk holds whole Philox blocks and no position
// fold falls inside it whatever the segment's start: the segment [s0, s1) has chunks c0 = s0 / kSub .. (s1 - 1) / kSub, the first and the last
// of them possibly partial (when checkpoint_every or the run's length is not a multiple
// of kSub).
struct SegChunks {
    int64_t s0, s1, c0;  // the segment's steps and its first chunk
    int n;               // its chunks
    __device__ __forceinline__ SegChunks(int64_t a, int64_t b) : s0(a), s1(b), c0(a / kSub), n((int)((b + kSub - 1) / kSub - a / kSub)) {}
    __device__ __forceinline__ int64_t begin(int j) const { return j == 0 ? s0 : (c0 + j) * kSub; }
    __device__ __forceinline__ int64_t end(int j) const { return j == n - 1 ? s1 : (c0 + j + 1) * kSub; }
    // chunks [first_whole, last_whole) are whole
    __device__ __forceinline__ int first_whole() const { return s0 % kSub ? 1 : 0; }
    __device__ __forceinline__ int last_whole() const { return max(s1 % kSub ? n - 1 : n, first_whole()); }
};

struct AdjArgs {
    Batch b;
    Ckpt ck;
    Noise nz;
    RoundKeys K;        // Philox round keys of the seed (constant bank)
    float4 *sub;        // [per][n_sub][total_traj] sub-checkpoints (scratch)
    int64_t n_sub;      // sub-checkpoint slots per segment (sub_slots)
    int per;            // segments per launch (segments_per_launch)
    uint4 *words;       // [block][per][n_blk][2][threads] noise hand-off of the launch (scratch), WORDS kernels only
    int64_t n_blk;      // Philox blocks per segment (kSub / 4 per sub-checkpoint slot)
    int tile0;          // first tile of the launch (its group of tiles)
    const double *w;    // [n_sets] dJ/dmean_v, NULL = 1
    double *partials;   // [n_tiles][6]
};

// Noise hand-off from level 1 to the reverse sweep.  Level 1 draws every
// Philox block of its segment anyway; with WORDS it also stores, per block, the
// scaled radii of its two Box-Muller pairs and their two angle words (16 B per
// four steps of a trajectory), and the reverse sweep's level-2 re-run takes them
// from there instead of drawing the block and forming the radii a second time
// (it still forms the angles' sine and cosine).  The reverse kernel holds all the
// registers its three blocks per SM can have, so the blocks are not loaded into
// registers ahead of use: each thread copies its own chunk's blocks into shared
// memory with cp.async, kStages - 1 chunks ahead, and reads them when the chunk
// runs.  The radii are the bits box_muller_f32x2 returned in level 1, and the
// angles are formed by the same code, so every state and gradient is the same
// bit for bit with or without the hand-off.
#ifndef ABP_ADJ_STAGES
#define ABP_ADJ_STAGES 3
#endif
constexpr int kStages = ABP_ADJ_STAGES;

__device__ __forceinline__ void cp_async16(void *dst_smem, const void *src_gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst_smem)), "l"(src_gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Noise of the four steps 4m .. 4m+3 as the forward integrator consumes it:
// the pair (nrs, trig) of each step is exactly what it feeds its fused
// multiply-add, so re-runs reproduce the forward states bit for bit.
__device__ __forceinline__ void block_noise(const Coef<float> &k, const StepStream &ss, const RoundKeys &K,
                                            uint32_t m, float (&nrs)[4], float (&tr)[4]) {
    const uint4 w = step_block(m, ss, K);
    float a, c, s;
    box_muller_f32(w.x, w.y, k.bm, a, c, s);
    nrs[0] = a;
    tr[0] = c;
    nrs[1] = a;
    tr[1] = s;
    box_muller_f32(w.z, w.w, k.bm, a, c, s);
    nrs[2] = a;
    tr[2] = c;
    nrs[3] = a;
    tr[3] = s;
}

// The same noise one step at a time, for partial chunks (one Philox block kept for its
// four steps).
struct NoiseCursor {
    uint32_t m;
    bool valid;
    float nrs[4], tr[4];

    __device__ void at(const Coef<float> &k, const StepStream &ss, const RoundKeys &K, int64_t n, float &nrs_n,
                       float &tr_n) {
        const uint32_t mm = (uint32_t)(n >> 2);
        if (!valid || mm != m) {
            block_noise(k, ss, K, mm, nrs, tr);
            m = mm;
            valid = true;
        }
        const int j = (int)(n & 3);
        nrs_n = j == 0 ? nrs[0] : j == 1 ? nrs[1] : j == 2 ? nrs[2] : nrs[3];
        tr_n = j == 0 ? tr[0] : j == 1 ? tr[1] : j == 2 ? tr[2] : tr[3];
    }
};

// One forward step at absolute index n, including the position fold the
// integrator applies after every kBlockSteps-th step (y depends on y and
// yacc only; the fold's error term and the cell index are not needed here).
__device__ __forceinline__ void fold(float &y, float &yacc, float &pb) {
    float lo = 0.0f;
    int32_t cell = 0;
    fold_position<float>(y, yacc, lo, cell);
    pb = phase_base(y);
}

__device__ __forceinline__ void fwd(const Coef<float> &k, float nrs, float trig, int64_t n, float &y, float &yacc,
                                   float &pb, float &v, float &e) {
    em_step_f32(k, nrs, trig, pb, yacc, v, e);
    if (((n + 1) & (kBlockSteps - 1)) == 0) fold(y, yacc, pb);
}

// One reverse step at the pre-step state (force phase ph, v = vv, e = ee,
// sigma z = sz): parameter terms with lambda_{n+1}, then lambda_n = J^T
// lambda_{n+1} + dJ/ds_n with dJ/dv_n = 1.
__device__ __forceinline__ void reverse_step(const Coef<float> &k, float kx, float dtf, float ph, float vv, float ee,
                                             float sz, float &lx, float &lv, float &le, float (&acc)[6]) {
    float sphi, cphi;
    __sincosf(ph, &sphi, &cphi);
    acc[0] = fmaf(lv, sz, acc[0]);                              // D
    acc[1] += le;                                               // q
    acc[2] = fmaf(le, ee, acc[2]);                              // c
    acc[3] = fmaf(ee * vv, fmaf(-le, vv, lv), acc[3]);          // d
    acc[4] = fmaf(lv, vv, acc[4]);                              // gamma0
    acc[5] = fmaf(lv, fmaf(2.0f * cphi, cphi, -1.0f), acc[5]);  // a
    const float dvdx = kx * sphi * fmaf(2.0f * k.A4, cphi, k.K);
    const float dvdv = fmaf(k.Bd, ee, k.G);
    const float dedv = -2.0f * k.Bd * ee * vv;
    const float dvde = k.Bd * vv;
    const float dede = fmaf(-k.Bd, vv * vv, k.A);
    const float nlx = fmaf(dvdx, lv, lx);
    const float nlv = fmaf(dtf, lx, fmaf(dvdv, lv, fmaf(dedv, le, 1.0f)));
    const float nle = fmaf(dvde, lv, dede * le);
    lx = nlx;
    lv = nlv;
    le = nle;
}

__device__ __forceinline__ void block_sum6(double (&a)[6], double (*red)[6]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < 6; ++j) a[j] += __shfl_down_sync(0xffffffffu, a[j], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < 6; ++j) red[warp][j] = a[j];
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
#pragma unroll
        for (int j = 0; j < 6; ++j) a[j] = lane < nw ? red[lane][j] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < 6; ++j) a[j] += __shfl_down_sync(0xffffffffu, a[j], o);
    }
}

// One Philox block of the hand-off for the thread's two trajectories: the
// scaled Box-Muller radii of its two word pairs (nrA, nrB, as their bits) and
// the two angle words, (nrA, wb_A, nrB, wb_B).  The buffer is laid out by
// kernel block -- [block][block index mrel in the segment][trajectory 0 / 1]
// [thread], the level-1 and reverse kernels mapping blocks and threads to
// trajectories alike -- so that wp (the thread's slot of mrel 0) plus a
// constant reaches every block of a chunk.  Both halves are stored, also where
// the thread's second trajectory repeats its first.
template <bool WORDS>
__device__ __forceinline__ void store_words(const AdjArgs &a, uint4 *wp, int64_t mrel, uint4 w0, uint4 w1, float2 nrA,
                                            float2 nrB) {
    if (WORDS) {
        const int64_t r = dchk(mrel, a.n_blk, a.b.dbg) * (2 * kL1Threads);
        wp[r] = make_uint4(__float_as_uint(nrA.x), w0.y, __float_as_uint(nrB.x), w0.w);
        wp[r + kL1Threads] = make_uint4(__float_as_uint(nrA.y), w1.y, __float_as_uint(nrB.y), w1.w);
    }
}

// Counter block m of the thread's two trajectories.  SHARED: their global ids have one high
// word (all but a pair astride a multiple of 2^32, only for some traj_base), so one head
// serves both.  The loops choose once, outside: asked per block, the branch ends the
// compiler's schedule at every block and a warp alone on its scheduler pays for it (level 1
// of 33,000 trajectories x 1,000 steps 76 us against 65).
template <bool SHARED>
__device__ __forceinline__ void pair_blocks(uint32_t m, const StepStream (&ss)[2], const RoundKeys &K, uint4 &w0,
                                            uint4 &w1) {
    const BlockHead h0 = block_head(m, ss[0].hx);
    w0 = step_block(h0, ss[0], K);
    w1 = step_block(SHARED ? h0 : block_head(m, ss[1].hx), ss[1], K);
}

// Level 1 of segment [s0, s1) of two trajectories (idx[0], idx[1]) of one thread: re-run
// from their checkpoints c0, c1, leaving the state at the start of each chunk in the
// sub-checkpoint scratch.  Whole chunks step the pair with paired FP32 instructions (same
// operations as em_step_f32 / box_muller_f32 on each half, so the sub-checkpoints are the
// scalar ones bit for bit); other chunks step each trajectory on its own.
// store1: whether the second trajectory is real (else it duplicates the first
// one's neighbour and its sub-checkpoints are not written).
template <bool WORDS>
__device__ __forceinline__ void level1_segment2(const AdjArgs &a, float4 *slots, uint4 *wp, const Coef<float> &k,
                                                const StepStream (&ss)[2], const int64_t (&idx)[2], bool store1,
                                                int64_t s0, int64_t s1, float4 c0, float4 c1) {
    const int64_t T = a.b.total_traj;
    const SegChunks seg(s0, s1);
    float y[2] = {c0.x, c1.x};
    float2 Y = make_float2(c0.y, c1.y), V = make_float2(c0.z, c1.z), E = make_float2(c0.w, c1.w);
    float2 PB = make_float2(phase_base(y[0]), phase_base(y[1]));
    const Coef2 k2 = make_coef2(k);
    auto store = [&](int j) {
        const size_t js = (size_t)dchk(j, a.n_sub, a.b.dbg);
        slots[js * T + idx[0]] = make_float4(y[0], Y.x, V.x, E.x);
        if (store1) slots[js * T + idx[1]] = make_float4(y[1], Y.y, V.y, E.y);
    };
    auto whole_chunk = [&](auto shared, int j) {
        const int64_t n0 = (seg.c0 + j) * kSub;
        store(j);
#pragma unroll
        for (int b2 = 0; b2 < kSub / 4; ++b2) {
            uint4 w0, w1;
            pair_blocks<decltype(shared)::value>((uint32_t)(n0 >> 2) + b2, ss, a.K, w0, w1);
            float2 nrA, nrB, cs, sn;
            box_muller_f32x2(make_uint2(w0.x, w1.x), make_uint2(w0.y, w1.y), k2.bm, nrA, cs, sn);
            em_step_f32x2(k2, nrA, cs, PB, Y, V, E);
            em_step_f32x2(k2, nrA, sn, PB, Y, V, E);
            box_muller_f32x2(make_uint2(w0.z, w1.z), make_uint2(w0.w, w1.w), k2.bm, nrB, cs, sn);
            em_step_f32x2(k2, nrB, cs, PB, Y, V, E);
            em_step_f32x2(k2, nrB, sn, PB, Y, V, E);
            store_words<WORDS>(a, wp, (kSub / 4) * (int64_t)j + b2, w0, w1, nrA, nrB);
        }
        if (((n0 + kSub) & (kBlockSteps - 1)) == 0) {
            fold(y[0], Y.x, PB.x);
            fold(y[1], Y.y, PB.y);
        }
    };
    auto partial_chunk = [&](int j) {  // each trajectory on its own
        store(j);
        const int64_t n0 = seg.begin(j), n1 = seg.end(j);
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            const StepStream sq = q ? ss[1] : ss[0];
            float yq = q ? y[1] : y[0], ya = q ? Y.y : Y.x, v = q ? V.y : V.x, e = q ? E.y : E.x, pb = q ? PB.y : PB.x;
            NoiseCursor nc;
            nc.valid = false;
            nc.m = 0;
            for (int64_t n = n0; n < n1; ++n) {
                float nrs, tr;
                nc.at(k, sq, a.K, n, nrs, tr);
                fwd(k, nrs, tr, n, yq, ya, pb, v, e);
            }
            if (q) {
                y[1] = yq, Y.y = ya, V.y = v, E.y = e, PB.y = pb;
            } else {
                y[0] = yq, Y.x = ya, V.x = v, E.x = e, PB.x = pb;
            }
        }
    };
    const int j1 = seg.last_whole();
    int j = 0;
    if (j < seg.first_whole()) partial_chunk(j++);
    if (ss[0].hx == ss[1].hx) {
        // whole chunks in groups of ABP_ADJ_L1_GROUP: one loop iteration per group
        for (; j + ABP_ADJ_L1_GROUP <= j1; j += ABP_ADJ_L1_GROUP) {
#pragma unroll
            for (int c = 0; c < ABP_ADJ_L1_GROUP; ++c) whole_chunk(std::true_type{}, j + c);
        }
#pragma unroll 1
        for (; j < j1; ++j) whole_chunk(std::true_type{}, j);
    } else {
#pragma unroll 1
        for (; j < j1; ++j) whole_chunk(std::false_type{}, j);
    }
    if (j < seg.n) partial_chunk(j);
}

// reverse_step of two trajectories in the halves of FP32 pairs, same
// operations in the same order as the scalar function (each half rounded as
// the scalar operation), so the gradient sums are the scalar kernel's bits.
struct RevCoef2 {
    float2 kx, dtf, twoA4, K, Bd, G, m2Bd, nBd, A, one, mone, two, neg;
};

__device__ __forceinline__ RevCoef2 make_rev_coef2(const Coef<float> &k, float kx, float dtf) {
    RevCoef2 c;
    c.kx = dup2(kx);
    c.dtf = dup2(dtf);
    c.twoA4 = dup2(2.0f * k.A4);
    c.K = dup2(k.K);
    c.Bd = dup2(k.Bd);
    c.G = dup2(k.G);
    c.m2Bd = dup2(-2.0f * k.Bd);
    c.nBd = dup2(-k.Bd);
    c.A = dup2(k.A);
    c.one = dup2(1.0f);
    c.mone = dup2(-1.0f);
    c.two = dup2(2.0f);
    c.neg = dup2(-1.0f);
    return c;
}

__device__ __forceinline__ void reverse_step_x2(const RevCoef2 &c, float2 ph, float2 vv, float2 ee, float2 sz,
                                                float2 &lx, float2 &lv, float2 &le, float2 (&acc)[6]) {
    float2 sphi, cphi;
    __sincosf(ph.x, &sphi.x, &cphi.x);
    __sincosf(ph.y, &sphi.y, &cphi.y);
    acc[0] = __ffma2_rn(lv, sz, acc[0]);
    acc[1] = __fadd2_rn(acc[1], le);
    acc[2] = __ffma2_rn(le, ee, acc[2]);
    acc[3] = __ffma2_rn(__fmul2_rn(ee, vv), __ffma2_rn(__fmul2_rn(le, c.neg), vv, lv), acc[3]);
    acc[4] = __ffma2_rn(lv, vv, acc[4]);
    acc[5] = __ffma2_rn(lv, __ffma2_rn(__fmul2_rn(c.two, cphi), cphi, c.mone), acc[5]);
    const float2 dvdx = __fmul2_rn(__fmul2_rn(c.kx, sphi), __ffma2_rn(c.twoA4, cphi, c.K));
    const float2 dvdv = __ffma2_rn(c.Bd, ee, c.G);
    const float2 dedv = __fmul2_rn(__fmul2_rn(c.m2Bd, ee), vv);
    const float2 dvde = __fmul2_rn(c.Bd, vv);
    const float2 dede = __ffma2_rn(c.nBd, __fmul2_rn(vv, vv), c.A);
    const float2 nlx = __ffma2_rn(dvdx, lv, lx);
    const float2 nlv = __ffma2_rn(c.dtf, lx, __ffma2_rn(dvdv, lv, __ffma2_rn(dedv, le, c.one)));
    const float2 nle = __ffma2_rn(dvde, lv, __fmul2_rn(dede, le));
    lx = nlx;
    lv = nlv;
    le = nle;
}

// Level 2 and the reverse sweep of segment [s0, s1) for two trajectories of one thread
// (idx[0], idx[1]): its kSub-step chunks in reverse order, each re-run from its
// sub-checkpoint into registers and swept backwards, each sub-checkpoint loaded one chunk
// ahead, so that its memory latency overlaps the previous chunk's arithmetic.  Whole
// chunks run the level-2 re-run and the reverse sweep on FP32 pairs;
// other chunks run each trajectory on its own with the scalar functions.
// Shared-memory stage of the hand-off: [kStages][kSub / 4 blocks][2 trajectories][thread].
typedef uint4 WordStage[kSub / 4][2][kRevPairThreads];

template <bool WORDS>
__device__ __forceinline__ void reverse_chunks2(const AdjArgs &a, const float4 *slots, const uint4 *wr,
                                                const Coef<float> &k, const StepStream (&ss)[2], float kx, float dtf,
                                                const int64_t (&idx)[2], int64_t s0, int64_t s1, float2 &lx,
                                                float2 &lv, float2 &le, float2 (&acc)[6], WordStage *stage) {
    const int64_t T = a.b.total_traj;
    const SegChunks seg(s0, s1);
    const int j0w = seg.first_whole(), j1w = seg.last_whole();  // chunks [j0w, j1w) are whole
    const Coef2 k2 = make_coef2(k);
    const RevCoef2 rc = make_rev_coef2(k, kx, dtf);
    // WORDS: copy whole chunk jj's blocks into stage[jj % kStages]; one commit group per
    // call, empty for chunks that are not whole, so that groups and chunks stay in step
    auto fetch = [&](int jj) {
        if (jj >= j0w && jj < j1w) {
            WordStage &st = stage[jj % kStages];
#pragma unroll
            for (int b2 = 0; b2 < kSub / 4; ++b2) {
                const int64_t r = dchk((kSub / 4) * (int64_t)jj + b2, a.n_blk, a.b.dbg) * (2 * kRevPairThreads);
                cp_async16(&st[b2][0][threadIdx.x], wr + r);
                cp_async16(&st[b2][1][threadIdx.x], wr + r + kRevPairThreads);
            }
        }
        cp_async_commit();
    };
    if (WORDS)
#pragma unroll
        for (int i = 0; i < kStages - 1; ++i) fetch(seg.n - 1 - i);
    const size_t jl = (size_t)dchk(seg.n - 1, a.n_sub, a.b.dbg);
    float4 n0c = slots[jl * T + idx[0]], n1c = slots[jl * T + idx[1]];
    for (int j = seg.n - 1; j >= 0; --j) {
        const float4 c0 = n0c, c1 = n1c;
        if (j > 0) {
            const size_t jp = (size_t)dchk(j - 1, a.n_sub, a.b.dbg);
            n0c = slots[jp * T + idx[0]];
            n1c = slots[jp * T + idx[1]];
        }
        if (WORDS) {
            fetch(j - (kStages - 1));
            cp_async_wait<kStages - 1>();  // this thread's copies of chunk j have landed
        }
        if (j >= j0w && j < j1w) {
            const int64_t n0 = (seg.c0 + j) * kSub;
            float2 Y = make_float2(c0.y, c1.y), V = make_float2(c0.z, c1.z), E = make_float2(c0.w, c1.w);
            const float2 PB = make_float2(phase_base(c0.x), phase_base(c1.x));
            float2 ys[kSub], vs[kSub], es[kSub], szs[kSub];
#pragma unroll
            for (int b2 = 0; b2 < kSub / 4; ++b2) {
                float2 nr[2], tr[4];
                float2 cs, sn;
                if (WORDS) {
                    // the radii come as level 1 formed them; the angles are formed here
                    const uint4 w0 = stage[j % kStages][b2][0][threadIdx.x];
                    const uint4 w1 = stage[j % kStages][b2][1][threadIdx.x];
                    nr[0] = make_float2(__uint_as_float(w0.x), __uint_as_float(w1.x));
                    nr[1] = make_float2(__uint_as_float(w0.z), __uint_as_float(w1.z));
                    bm_angle_f32x2(make_uint2(w0.y, w1.y), cs, sn);
                    tr[0] = cs;
                    tr[1] = sn;
                    bm_angle_f32x2(make_uint2(w0.w, w1.w), cs, sn);
                    tr[2] = cs;
                    tr[3] = sn;
                } else {
                    const uint32_t m = (uint32_t)(n0 >> 2) + b2;
                    uint4 w0, w1;
                    pair_blocks<false>(m, ss, a.K, w0, w1);
                    box_muller_f32x2(make_uint2(w0.x, w1.x), make_uint2(w0.y, w1.y), k2.bm, nr[0], cs, sn);
                    tr[0] = cs;
                    tr[1] = sn;
                    box_muller_f32x2(make_uint2(w0.z, w1.z), make_uint2(w0.w, w1.w), k2.bm, nr[1], cs, sn);
                    tr[2] = cs;
                    tr[3] = sn;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = 4 * b2 + i;
                    ys[q] = __ffma2_rn(Y, dup2(kTwoPiF), PB);
                    vs[q] = V;
                    es[q] = E;
                    szs[q] = __fmul2_rn(nr[i >> 1], tr[i]);
                    em_step_f32x2(k2, nr[i >> 1], tr[i], PB, Y, V, E);
                }
            }
#pragma unroll
            for (int i = kSub - 1; i >= 0; --i) reverse_step_x2(rc, ys[i], vs[i], es[i], szs[i], lx, lv, le, acc);
        } else {
            // a partial chunk: scalar path, one trajectory after the other
            const int64_t n0 = seg.begin(j);
            const int len = (int)(seg.end(j) - n0);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 cq = q ? c1 : c0;
                float y = cq.x, yacc = cq.y, v = cq.z, e = cq.w;
                float pb = phase_base(y);
                float lxq = q ? lx.y : lx.x, lvq = q ? lv.y : lv.x, leq = q ? le.y : le.x;
                float accq[6];
#pragma unroll
                for (int r = 0; r < 6; ++r) accq[r] = q ? acc[r].y : acc[r].x;
                NoiseCursor nc;
                nc.valid = false;
                nc.m = 0;
                float ysq[kSub], vsq[kSub], esq[kSub], szq[kSub];
#pragma unroll
                for (int i = 0; i < kSub; ++i) {
                    if (i < len) {
                        float nrs, tr;
                        nc.at(k, ss[q], a.K, n0 + i, nrs, tr);
                        ysq[i] = phase_arg(pb, yacc);
                        vsq[i] = v;
                        esq[i] = e;
                        szq[i] = nrs * tr;
                        fwd(k, nrs, tr, n0 + i, y, yacc, pb, v, e);
                    }
                }
#pragma unroll
                for (int i = kSub - 1; i >= 0; --i)
                    if (i < len) reverse_step(k, kx, dtf, ysq[i], vsq[i], esq[i], szq[i], lxq, lvq, leq, accq);
                if (q) {
                    lx.y = lxq;
                    lv.y = lvq;
                    le.y = leq;
#pragma unroll
                    for (int r = 0; r < 6; ++r) acc[r].y = accq[r];
                } else {
                    lx.x = lxq;
                    lv.x = lvq;
                    le.x = leq;
#pragma unroll
                    for (int r = 0; r < 6; ++r) acc[r].x = accq[r];
                }
            }
        }
    }
}

// One launch per run of consecutive segments, level and group of tiles, runs in reverse
// order: level 1 (a plain forward re-run, light on registers) for the run's segments
// of the group's trajectories, every segment in blocks of its own (blockIdx.y; each
// starts from its own checkpoint), then level 2 and the reverse sweep
// (register-heavy), the run's segments one after the other.  The level-1 launch of the
// run before goes on a second stream while the reverse sweep of a run goes, into the
// other of two sub-checkpoint buffers.  Between segments each trajectory keeps its adjoint
// state lambda = (x, v, e) and its six gradient sums in global memory.
// Trajectories of sets shorter than a segment's start skip it.
constexpr int kAdjGroups = abp_ctx::kAdjGroups;

struct SegView {
    float4 *lam;  // [total_traj] (lambda_x, lambda_v, lambda_e, -)
    double *G;    // [6][total_traj] gradient sums
};

// The sub-checkpoint slots and the thread's hand-off blocks of segment i of a launch.
__device__ __forceinline__ float4 *segment_slots(const AdjArgs &a, int i) {
    return a.sub + (size_t)i * (size_t)a.n_sub * (size_t)a.b.total_traj;
}

template <bool WORDS>
__device__ __forceinline__ uint4 *segment_words(const AdjArgs &a, int block, int i) {
    if (!WORDS) return nullptr;
    return a.words + ((size_t)block * (size_t)a.per + (size_t)i) * (size_t)a.n_blk * (2 * kL1Threads) + threadIdx.x;
}

// Level 1 with two trajectories per thread (trajectories li and li +
// blockDim.x of the block's 2 blockDim.x), `sub` blocks per tile.
template <bool WORDS>
__global__ void __launch_bounds__(kL1Threads) adjoint_level1_pair_kernel(AdjArgs a, int64_t seg0, int sub) {
    const Batch &b = a.b;
    const int64_t seg = seg0 + blockIdx.y;
    float4 *const slots = segment_slots(a, (int)blockIdx.y);
    const int tile = a.tile0 + (int)blockIdx.x / sub;
    const int li = ((int)blockIdx.x % sub) * 2 * (int)blockDim.x + (int)threadIdx.x;
    const int set = b.tile_set[tile];
    const int64_t N = b.set_steps[set], K = a.ck.every, T = b.total_traj;
    const int64_t s0 = seg * K;
    if (s0 >= N) return;  // uniform over the block
    const int64_t s1 = min(s0 + K, N);
    const int count = b.tile_count[tile];
    if (li >= count) return;
    const Coef<float> k = load_coef<float>(b.coef_f, b.params, set, a.nz.dt);  // the forward's own coefficients
    const bool second = li + (int)blockDim.x < count;
    const int64_t idx[2] = {dchk(b.tile_first[tile] + li, T, b.dbg),
                            dchk(b.tile_first[tile] + (second ? li + (int)blockDim.x : li), T, b.dbg)};
    const StepStream ss[2] = {step_stream((uint64_t)idx[0] + a.nz.traj_base, a.K),
                              step_stream((uint64_t)idx[1] + a.nz.traj_base, a.K)};
    const int64_t slot = dchk(seg, a.ck.n_slots, b.dbg);
    level1_segment2<WORDS>(a, slots, segment_words<WORDS>(a, a.tile0 * sub + (int)blockIdx.x, (int)blockIdx.y), k, ss,
                           idx, second, s0, s1, a.ck.ck[(size_t)slot * T + idx[0]],
                           a.ck.ck[(size_t)slot * T + idx[1]]);
}

// The reverse kernel with two trajectories per thread (trajectories li and
// li + blockDim.x of the block's 2 blockDim.x), `sub` blocks per tile.
// MULTI: the launch covers n segments (without it the loop below costs the kernel at its
// register cap a spill, 1% of the sweep).
template <bool WORDS, bool MULTI>
__global__ void __launch_bounds__(kRevPairThreads, ABP_ADJ_REV_PAIR_MIN_BLOCKS) adjoint_reverse_pair_kernel(AdjArgs a, SegView sv, int64_t seg0,
                                                                               int n, int sub, int64_t window) {
    __shared__ WordStage stage[WORDS ? kStages : 1];
    const Batch &b = a.b;
    const int tile = a.tile0 + (int)blockIdx.x / sub;
    const int li = ((int)blockIdx.x % sub) * 2 * (int)blockDim.x + (int)threadIdx.x;
    const int set = b.tile_set[tile];
    const int64_t N = b.set_steps[set], K = a.ck.every, T = b.total_traj;
    if (seg0 * K >= N) return;  // uniform over the block
    const int count = b.tile_count[tile];
    if (li >= count) return;
    const abp_params p = b.params[set];
    const Coef<float> k = load_coef<float>(b.coef_f, b.params, set, a.nz.dt);  // the forward's own coefficients
    const float dtf = (float)a.nz.dt;
    const float kx = (float)(-2.0 * kPi / p.L);
    const bool second = li + (int)blockDim.x < count;
    const int64_t idx[2] = {dchk(b.tile_first[tile] + li, T, b.dbg),
                            dchk(b.tile_first[tile] + (second ? li + (int)blockDim.x : li), T, b.dbg)};
    const StepStream ss[2] = {step_stream((uint64_t)idx[0] + a.nz.traj_base, a.K),
                              step_stream((uint64_t)idx[1] + a.nz.traj_base, a.K)};
    for (int i = MULTI ? n - 1 : 0; i >= 0; --i) {
        const int64_t seg = seg0 + i, s0 = seg * K;
        if (s0 >= N) continue;
        float4 l0 = sv.lam[idx[0]], l1 = sv.lam[idx[1]];
        if (window > 0 && ((seg + 1) * K) % window == 0) l0 = l1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float2 lx = make_float2(l0.x, l1.x), lv = make_float2(l0.y, l1.y), le = make_float2(l0.z, l1.z);
        float2 acc[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) acc[q] = make_float2(0.0f, 0.0f);
        reverse_chunks2<WORDS>(a, segment_slots(a, i), segment_words<WORDS>(a, a.tile0 * sub + (int)blockIdx.x, i), k,
                               ss, kx, dtf, idx, s0, min(s0 + K, N), lx, lv, le, acc, stage);
        sv.lam[idx[0]] = make_float4(lx.x, lv.x, le.x, 0.0f);
#pragma unroll
        for (int q = 0; q < 6; ++q) sv.G[(size_t)q * T + idx[0]] += (double)acc[q].x;
        if (second) {
            sv.lam[idx[1]] = make_float4(lx.y, lv.y, le.y, 0.0f);
#pragma unroll
            for (int q = 0; q < 6; ++q) sv.G[(size_t)q * T + idx[1]] += (double)acc[q].y;
        }
    }
}

// Small batches: level 1 leaves every step's state, (force phase, v, e, sigma z) in one
// 16-byte row, and the sweep only reads them.  There a warp has its scheduler to itself
// and a launch's time is the length of one trajectory's sweep: the pair kernel's thread
// re-runs and sweeps two trajectories, some 62 instructions a step, the one here sweeps
// one, about 26, while level 1 runs all segments of the launch side by side.
__global__ void __launch_bounds__(kL1Threads) adjoint_states_kernel(AdjArgs a, int64_t seg0, int sub) {
    const Batch &b = a.b;
    const int64_t seg = seg0 + blockIdx.y;
    const int tile = a.tile0 + (int)blockIdx.x / sub;
    const int li = ((int)blockIdx.x % sub) * (int)blockDim.x + (int)threadIdx.x;
    const int set = b.tile_set[tile];
    const int64_t N = b.set_steps[set], K = a.ck.every, T = b.total_traj;
    const int64_t s0 = seg * K;
    if (s0 >= N) return;  // uniform over the block
    const int64_t s1 = min(s0 + K, N);
    const Coef<float> k = load_coef<float>(b.coef_f, b.params, set, a.nz.dt);  // the forward's own coefficients
    if (li >= b.tile_count[tile]) return;
    const int64_t idx = dchk(b.tile_first[tile] + li, T, b.dbg);
    const StepStream ss = step_stream((uint64_t)idx + a.nz.traj_base, a.K);
    const float4 c0 = a.ck.ck[(size_t)dchk(seg, a.ck.n_slots, b.dbg) * T + idx];
    float y = c0.x, yacc = c0.y, v = c0.z, e = c0.w;
    float pb = phase_base(y);
    float4 *const rows = segment_slots(a, (int)blockIdx.y) + idx;  // K rows per segment
    int64_t n = s0;
    auto row = [&](int64_t m, float sz) {
        rows[(size_t)dchk(m - s0, a.n_sub, b.dbg) * T] = make_float4(phase_arg(pb, yacc), v, e, sz);
    };
    while (n < s1) {
        float nrs[4], tr[4];
        block_noise(k, ss, a.K, (uint32_t)(n >> 2), nrs, tr);
        if ((n & 3) == 0 && n + 4 <= s1) {  // no fold falls inside a block of four steps
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                row(n + i, nrs[i] * tr[i]);
                em_step_f32(k, nrs[i], tr[i], pb, yacc, v, e);
            }
            n += 4;
            if ((n & (kBlockSteps - 1)) == 0) fold(y, yacc, pb);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i == (int)(n & 3) && n < s1) {
                    row(n, nrs[i] * tr[i]);
                    fwd(k, nrs[i], tr[i], n, y, yacc, pb, v, e);
                    ++n;
                }
        }
    }
}

// The sweep over the rows of a launch's n segments, one trajectory per thread in blocks of
// one warp.  The rows of consecutive segments follow one another, so the copies into the
// thread's own ring (cp.async, kRowGroups - 1 groups of kRowGroup rows ahead, no barrier:
// a thread reads only what it copied) run on across segments.  A group's first reads and
// their sines wait for shared memory, so longer groups are faster as long as the ring leaves
// room for six warps on an SM (32 KB each): backward of 256 trajectories x 4,000 steps, K =
// 64, 262 us with eight groups of 8, 235 with four of 16, 237 with three; of 16,384 x 4,000,
// K = 200, 480, 468 and 516 us (each some 20 us less since the calls ask for no free memory).
constexpr int kRowGroup = 16, kRowGroups = 4, kSweepThreads = 32;

__global__ void __launch_bounds__(kSweepThreads) adjoint_sweep_kernel(AdjArgs a, SegView sv, int64_t seg0, int n,
                                                                      int sub, int64_t window) {
    __shared__ float4 ring[kRowGroup * kRowGroups][kSweepThreads];
    const Batch &b = a.b;
    const int tile = a.tile0 + (int)blockIdx.x / sub;
    const int li = ((int)blockIdx.x % sub) * kSweepThreads + (int)threadIdx.x;
    const int set = b.tile_set[tile];
    const int64_t N = b.set_steps[set], K = a.ck.every, T = b.total_traj;
    const int64_t first = seg0 * K;
    if (first >= N) return;  // uniform over the block
    if (li >= b.tile_count[tile]) return;
    const abp_params p = b.params[set];
    const Coef<float> k = load_coef<float>(b.coef_f, b.params, set, a.nz.dt);  // the forward's own coefficients
    const float dtf = (float)a.nz.dt;
    const float kx = (float)(-2.0 * kPi / p.L);
    const int64_t idx = dchk(b.tile_first[tile] + li, T, b.dbg);
    const int rows = (int)(min(first + n * K, N) - first);
    const float4 *const src = a.sub + idx;
    auto fetch = [&](int g) {
        if (g >= 0)
#pragma unroll
            for (int i = 0; i < kRowGroup; ++i) {
                const int r = g * kRowGroup + i;
                if (r < rows)
                    cp_async16(&ring[(g % kRowGroups) * kRowGroup + i][threadIdx.x],
                               src + (size_t)dchk((int64_t)r, a.n_sub * a.per, b.dbg) * T);
            }
        cp_async_commit();
    };
    const int top = (rows - 1) / kRowGroup;
#pragma unroll 1
    for (int i = 0; i < kRowGroups - 1; ++i) fetch(top - i);
    float4 l0 = sv.lam[idx];
    float lx = l0.x, lv = l0.y, le = l0.z;
    float acc[6] = {0, 0, 0, 0, 0, 0};
    double G[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) G[q] = sv.G[(size_t)q * T + idx];
    int seg = (int)((rows - 1) / K);   // the segment of the launch being swept
    int begin = (int)(seg * K);        // its first row
    auto enter = [&]() {               // windowed adjoint: the window ending at step (seg0 + seg + 1) K starts from zero
        if (window > 0 && ((seg0 + seg + 1) * K) % window == 0) lx = lv = le = 0.0f;
    };
    auto leave = [&]() {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            G[q] += (double)acc[q];
            acc[q] = 0.0f;
        }
        --seg;
        begin -= (int)K;
        if (seg >= 0) enter();
    };
    enter();
    for (int g = top; g >= 0; --g) {
        fetch(g - (kRowGroups - 1));
        cp_async_wait<kRowGroups - 1>();  // this thread's copies of group g have landed
        const int r0 = g * kRowGroup;
        const float4(*const rg)[kSweepThreads] = ring + (g % kRowGroups) * kRowGroup;
        if (r0 >= begin && r0 + kRowGroup <= rows) {
#pragma unroll
            for (int i = kRowGroup - 1; i >= 0; --i) {
                const float4 c = rg[i][threadIdx.x];
                reverse_step(k, kx, dtf, c.x, c.y, c.z, c.w, lx, lv, le, acc);
            }
            if (r0 == begin) leave();
        } else {
#pragma unroll 1
            for (int i = kRowGroup - 1; i >= 0; --i) {
                if (r0 + i >= rows) continue;
                const float4 c = rg[i][threadIdx.x];
                reverse_step(k, kx, dtf, c.x, c.y, c.z, c.w, lx, lv, le, acc);
                if (r0 + i == begin) leave();
            }
        }
    }
    sv.lam[idx] = make_float4(lx, lv, le, 0.0f);
#pragma unroll
    for (int q = 0; q < 6; ++q) sv.G[(size_t)q * T + idx] = G[q];
}

// Per tile: the initial-condition term, the parameter scales and the caller's
// weights, summed in FP64 over the tile's trajectories.
__global__ void __launch_bounds__(kThreads) adjoint_final_kernel(AdjArgs a, SegView sv) {
    __shared__ double red[kThreads / 32][6];
    const Batch &b = a.b;
    const int tile = blockIdx.x;
    const int set = b.tile_set[tile];
    const int64_t N = b.set_steps[set], T = b.total_traj;
    const abp_params p = b.params[set];
    const double dt = a.nz.dt;
    const int64_t first = b.tile_first[tile];
    const int count = b.tile_count[tile];
    int64_t M = 0;
    for (int t = b.set_tile_begin[set]; t < b.set_tile_begin[set + 1]; ++t) M += b.tile_count[t];
    double gsum[6] = {0, 0, 0, 0, 0, 0};
    if (N > 0) {
        // dmean_v/dtheta = (1 / (M N)) dJ_i/dtheta, scaled by the caller's weight
        const double wgt = (a.w ? a.w[set] : 1.0) / ((double)M * (double)N);
        const double Kd = dt * p.h * 0.453 * (2.0 * kPi / p.L);
        for (int li = threadIdx.x; li < count; li += blockDim.x) {
            const int64_t idx = first + li;
            double G[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) G[q] = sv.G[(size_t)q * T + idx];
            // initial condition: v0 = sqrt(D) z depends on D
            if (a.nz.v0_mode == 1) G[0] += (double)sv.lam[idx].y * (double)a.ck.ck[idx].z;
            gsum[0] += wgt * (p.D > 0.0 ? G[0] / (2.0 * p.D) : NAN);
            gsum[1] += wgt * dt * G[1];
            gsum[2] += wgt * (-dt) * G[2];
            gsum[3] += wgt * dt * G[3];
            gsum[4] += wgt * (-dt) * G[4];
            gsum[5] += wgt * 2.0 * Kd * G[5];
        }
    }
    block_sum6(gsum, red);
    if (threadIdx.x == 0)
#pragma unroll
        for (int j = 0; j < 6; ++j) a.partials[(size_t)tile * 6 + j] = gsum[j];
}

// Per trajectory: d vbar_i / d theta (no caller weight, not averaged), from the same
// sums as adjoint_final_kernel -- the initial-condition term and the parameter scales
// applied, divided by the set's step count.  out: [total_traj][6].
__global__ void __launch_bounds__(kThreads) adjoint_traj_kernel(AdjArgs a, SegView sv, double *out) {
    const Batch &b = a.b;
    const int tile = blockIdx.x;
    const int set = b.tile_set[tile];
    const int64_t N = b.set_steps[set], T = b.total_traj;
    const abp_params p = b.params[set];
    const double dt = a.nz.dt;
    const double Kd = dt * p.h * 0.453 * (2.0 * kPi / p.L);
    const double inv_N = N > 0 ? 1.0 / (double)N : 0.0;
    const int64_t first = b.tile_first[tile];
    const int count = b.tile_count[tile];
    for (int li = threadIdx.x; li < count; li += blockDim.x) {
        const int64_t idx = dchk(first + li, T, b.dbg);
        double G[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) G[q] = sv.G[(size_t)q * T + idx];
        if (a.nz.v0_mode == 1) G[0] += (double)sv.lam[idx].y * (double)a.ck.ck[idx].z;
        double *o = out + (size_t)idx * 6;
        if (N == 0) {
#pragma unroll
            for (int q = 0; q < 6; ++q) o[q] = 0.0;
            continue;
        }
        o[0] = (p.D > 0.0 ? G[0] / (2.0 * p.D) : NAN) * inv_N;
        o[1] = dt * G[1] * inv_N;
        o[2] = -dt * G[2] * inv_N;
        o[3] = dt * G[3] * inv_N;
        o[4] = -dt * G[4] * inv_N;
        o[5] = 2.0 * Kd * G[5] * inv_N;
    }
}

__global__ void __launch_bounds__(kThreads) adjoint_set_kernel(Batch b, const double *partials, double *grad) {
    __shared__ double red[kThreads / 32][6];
    const int set = blockIdx.x;
    const int t0 = b.set_tile_begin[set], t1 = b.set_tile_begin[set + 1];
    double a[6] = {0, 0, 0, 0, 0, 0};
    for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x)
#pragma unroll
        for (int j = 0; j < 6; ++j) a[j] += partials[(size_t)t * 6 + j];
    block_sum6(a, red);
    if (threadIdx.x == 0)
#pragma unroll
        for (int j = 0; j < 6; ++j) grad[(size_t)set * 6 + j] = a[j];
}

abp_status set_err(abp_ctx *ctx, abp_status st, const char *msg, cudaError_t e = cudaSuccess) {
    ctx->err = msg;
    if (e != cudaSuccess) {
        ctx->err += ": ";
        ctx->err += cudaGetErrorString(e);
        cudaGetLastError();  // reported here: the next call's launch check must not find it again
    }
    return st;
}

// Scratch of abp_backward, one allocation: the tile partials, the set gradients, the
// weights, lambda, the per-trajectory sums, then the sub-checkpoint buffers and,
// last, the Philox-block buffers of the hand-off (0 bytes without it), each for
// `per` segments: two, alternating by launch, or one where a launch covers every
// segment.  abp_backward_traj reads lambda and the sums of the last call at the
// same offsets, which depend on neither.
struct AdjLayout {
    size_t sub1, sub, part, grad, w, lam, g, words1, words, need;
    size_t off_part, off_grad, off_w, off_lam, off_g, off_sub, off_words;
};

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Sub-checkpoint slots of a segment of K steps: the chunks it can touch (SegChunks), one
// more than K / kSub rounded up when segments start anywhere on the chunk grid.
int64_t sub_slots(int64_t K) { return (K + kSub - 1) / kSub + (K % kSub ? 1 : 0); }

// Kernel blocks per tile of the paired level-1 and reverse kernels (tiles hold up
// to kThreads * ppt trajectories, a block two per thread).
int pair_blocks_per_tile(const abp_ctx *ctx, int threads) {
    const int cap = kThreads * std::max(ctx->ppt, 1);
    return (cap + 2 * threads - 1) / (2 * threads);
}

AdjLayout adj_layout(const abp_ctx *ctx, bool words, int64_t per = 1, bool states = false, int buffers = 2) {
    AdjLayout L;
    const int64_t T = ctx->total_traj, Kc = ctx->cfg.checkpoint_every;
    const int64_t n_sub = states ? Kc : sub_slots(Kc);
    L.sub1 = sizeof(float4) * (size_t)(per * n_sub) * (size_t)T;
    L.sub = buffers * align256(L.sub1);
    L.part = sizeof(double) * 6 * (size_t)std::max(ctx->n_tiles, 1);
    L.grad = sizeof(double) * 6 * (size_t)std::max(ctx->n_sets, 1);
    L.w = sizeof(double) * (size_t)std::max(ctx->n_sets, 1);
    L.lam = sizeof(float4) * (size_t)std::max<int64_t>(T, 1);
    L.g = sizeof(double) * 6 * (size_t)std::max<int64_t>(T, 1);
    const size_t blocks = (size_t)ctx->n_tiles * (size_t)pair_blocks_per_tile(ctx, kL1Threads);
    L.words1 = words ? sizeof(uint4) * blocks * (size_t)(per * n_sub * (kSub / 4)) * 2 * kL1Threads : 0;
    L.words = buffers * align256(L.words1);
    L.off_part = 0;
    L.off_grad = L.off_part + align256(L.part);
    L.off_w = L.off_grad + align256(L.grad);
    L.off_lam = L.off_w + align256(L.w);
    L.off_g = L.off_lam + align256(L.lam);
    L.off_sub = L.off_g + align256(L.g);
    L.off_words = L.off_sub + L.sub;
    L.need = L.off_words + L.words;
    return L;
}

// both kernels must map blocks and threads to trajectories alike for the hand-off
static_assert(kL1Threads == kRevPairThreads, "level 1 and the reverse sweep share a block's trajectories");

// Bytes abp_backward may take for what level 1 hands to the reverse sweep (no hand-off where one
// segment's buffers do not fit): ABP_ADJ_HANDOFF_BYTES (0: never) ...
bool handoff_env(double *budget) {
    const char *env = getenv("ABP_ADJ_HANDOFF_BYTES");
    if (!env || !*env) return false;
    *budget = std::min(strtod(env, nullptr), 1e15);  // segment counts stay in 64 bits
    return true;
}

// ... else half the free device memory, the scratch's own counted as free.
double handoff_memory(const abp_ctx *ctx) {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        return -1.0;
    }
    return (double)((free_b + ctx->d_adj.cap) / 2);
}

// Whether level 1 hands every step's state to the sweep (adjoint_states_kernel): batches of
// at most kStateTraj trajectories whose segments fit ABP_ADJ_STATE_BYTES (0: never) and
// the hand-off's budget.  One backward, the hand-off against this: 300 trajectories x 4,000
// steps, K = 64, 458 -> 205 us; 8,000 x 2,000, K = 64, 341 -> 170, K = 333, 281 -> 174; 8,000
// x 4,000, K = 1,000, 446 -> 275; 16,384 x 4,000, K = 200, 521 -> 440; 24,576 x 4,000, K = 64,
// 966 -> 636 (K = 500, one segment per launch, 647 and 706); 32,768 x 2,000, K = 64, 475 ->
// 465: beyond that the SMs hold more warps than the ring leaves room for and the rows' 32
// bytes a step come from HBM.  Fewer bytes mean more launches (256 MB: 8,000 x 2,000 182 and
// 211 us, 16,384 x 4,000 508; 128 MB: 209, 215 and 647), more cost an allocation and its
// release: up to 0.1 ms of a context's first call and 0.2 of its end at 512 MB.
#ifndef ABP_ADJ_STATE_TRAJ
#define ABP_ADJ_STATE_TRAJ 32768
#endif
constexpr int64_t kStateTraj = ABP_ADJ_STATE_TRAJ;
// A run of one segment has no other to step beside it in level 1, so there the rows' traffic
// counts earlier: one backward of 500 steps, K = 500, 16,384 trajectories 106 us against 127
// with the hand-off, 20,000 119 against 127, 24,576 129 against 128, 32,768 153 against 135.
constexpr int64_t kStateTrajOne = 24576;
double state_bytes() {
    const char *env = getenv("ABP_ADJ_STATE_BYTES");
    return env && *env ? std::min(strtod(env, nullptr), 4e9) : 512.0 * (1 << 20);  // row numbers stay in 32 bits
}
bool use_states(const abp_ctx *ctx, int64_t n_seg, double budget) {
    return ctx->total_traj <= (n_seg > 1 ? kStateTraj : kStateTrajOne) &&
           (double)adj_layout(ctx, false, 1, true).sub <= std::min(budget, state_bytes());
}

// Segments per launch: as many as this many bytes of buffers hold (one where a segment's
// own buffers are larger, or the noise is drawn again), shared evenly over the launches.  A
// launch and its events cost the host some 5 us and the device the start and the drain of
// its blocks, and level 1 of several segments runs side by side: with short segments of
// small batches that is most of the time.  Backward with the hand-off over 4,000 steps, one
// segment per launch against as many as fit: 256 trajectories, K = 64, 892 -> 455 us, K = 200,
// 515 -> 400; 40,000, K = 64, 1,137 -> 884; 60,000 1,315 -> 1,114.  A segment of 262,144
// trajectories and K = 333 to 1,000 fills the GPU and the buffers by itself.
// Level 1 of the next launch runs beside the sweep: while the batch is small enough for both
// to have their warps (of 64 trajectories) on schedulers of their own, no more segments than
// leave them that.  Past it a sweep that shares its scheduler holds up the launch: 4,000
// trajectories, K = 64, eight segments 519 us, twelve 768; 8,000, K = 200, three 458, five
// 660; 12,000 two 481, four 730; 16,384 one 522, two 777; 24,576 one 699, two 929.  At 32,768
// and more the schedulers are shared either way (K = 64, one 1,227, four 775).
#ifndef ABP_ADJ_LAUNCH_BYTES
#define ABP_ADJ_LAUNCH_BYTES (128 << 20)
#endif
int64_t segments_per_launch(const abp_ctx *ctx, bool words, bool states, double budget, int64_t n_seg) {
    if (!words && !states) return 1;
    const AdjLayout L = adj_layout(ctx, words, 1, states);
    int64_t per = (int64_t)((states ? state_bytes() : (double)ABP_ADJ_LAUNCH_BYTES) /
                            (double)std::max<size_t>(L.sub + L.words, 1));
    if (words) per = std::min(per, (int64_t)(budget / (double)std::max<size_t>(L.words, 1)));
    if (states) per = std::min(per, (int64_t)(budget / (double)std::max<size_t>(L.sub, 1)));
    const int64_t lone = (int64_t)4 * 64 * ctx->sm_count;  // trajectories of one warp per scheduler
    if (words && 3 * ctx->total_traj <= 2 * lone)
        per = std::min(per, lone / std::max<int64_t>(ctx->total_traj, 1) - 1);
    per = std::max<int64_t>(1, std::min({per, n_seg, (int64_t)65535}));
    const int64_t launches = (n_seg + per - 1) / per;
    return launches > 0 ? (n_seg + launches - 1) / launches : 1;
}

// The form of a backward call and its scratch: every step's state, the noise hand-off or
// (neither) the noise drawn again, and the segments of a launch.
struct AdjForm {
    bool states, words;
    int64_t per;
    AdjLayout L;
};

AdjForm form_within(const abp_ctx *ctx, int64_t n_seg, double budget) {
    AdjForm f;
    f.states = use_states(ctx, n_seg, budget);
    f.words = !f.states && (double)adj_layout(ctx, true).words <= budget;
    f.per = segments_per_launch(ctx, f.words, f.states, budget, n_seg);
    f.L = adj_layout(ctx, f.words, f.per, f.states, f.per < n_seg ? 2 : 1);
    return f;
}

// Without a budget from the environment the free memory is asked for only where the
// scratch has to grow: the query takes the host some 18 us, a tenth of a short backward
// (33,000 trajectories x 500 steps, K = 500: 155 us with it on every call, 137 without;
// 300 x 1,000, K = 64: 114 and 94).
AdjForm choose_form(const abp_ctx *ctx, int64_t n_seg) {
    double budget = 1e15;
    const bool env = handoff_env(&budget);
    const AdjForm f = form_within(ctx, n_seg, budget);
    return env || (ctx->d_adj.p && f.L.need <= ctx->d_adj.cap) ? f : form_within(ctx, n_seg, handoff_memory(ctx));
}

}  // namespace
}  // namespace abp

using namespace abp;

extern "C" abp_status abp_backward(abp_ctx *ctx, const double *dJ_dmean_v, double *grad) {
    return abp_backward_windowed(ctx, dJ_dmean_v, grad, 0);
}

extern "C" abp_status abp_backward_windowed(abp_ctx *ctx, const double *dJ_dmean_v, double *grad, int64_t window) {
    const NvtxRange nvtx("abp_backward");
    if (!ctx) return ABP_EINVAL;
    if (window < 0 || (window > 0 && (ctx->cfg.checkpoint_every <= 0 || window % ctx->cfg.checkpoint_every != 0)))
        return set_err(ctx, ABP_EINVAL, "abp_backward_windowed: window must be a multiple of checkpoint_every");
    if (!grad) return set_err(ctx, ABP_EINVAL, "abp_backward: grad is NULL");
    const PtrKind kg = ptr_kind(grad, ctx->device);
    if (kg == PtrKind::OtherDevice) return set_err(ctx, ABP_EINVAL, "abp_backward: grad on another GPU");
    if (!ctx->have_batch) return set_err(ctx, ABP_ESTATE, "abp_backward before abp_set_params");
    if (ctx->cfg.checkpoint_every <= 0)
        return set_err(ctx, ABP_ESTATE, "abp_backward needs checkpoint_every > 0 during abp_integrate");
    if (ctx->g < ctx->max_steps) return set_err(ctx, ABP_ESTATE, "abp_backward before the integration completed");
    if (!ctx->ckpt_complete)
        return set_err(ctx, ABP_ESTATE, "abp_backward after abp_load: the checkpoints do not cover the run from step 0");
    const PtrKind kw = dJ_dmean_v ? ptr_kind(dJ_dmean_v, ctx->device) : PtrKind::Host;
    if (kw == PtrKind::OtherDevice) return set_err(ctx, ABP_EINVAL, "abp_backward: weights on another GPU");
    ctx->adj_valid = false;  // until this call has enqueued all of its work: the scratch changes from here on
    const int64_t n_sub = sub_slots(ctx->cfg.checkpoint_every);
    const int64_t Kc = ctx->cfg.checkpoint_every, n_seg = (ctx->max_steps + Kc - 1) / Kc;
    AdjForm form = choose_form(ctx, n_seg);
    bool &states = form.states, &words = form.words;
    int64_t &per = form.per;
    AdjLayout &L = form.L;
    DevBuf &sc = ctx->d_adj;
    if (!sc.p || sc.cap < L.need) {
        sc.release();
        cudaError_t e = cudaMalloc(&sc.p, L.need);
        if (e != cudaSuccess && (per > 1 || states)) {  // no room for several segments: one per launch
            cudaGetLastError();
            per = 1;
            states = false;
            L = adj_layout(ctx, words, per, states, n_seg > 1 ? 2 : 1);
            e = cudaMalloc(&sc.p, L.need);
        }
        if (e != cudaSuccess && words) {  // no room for the hand-off: draw the blocks twice instead
            cudaGetLastError();
            words = false;
            L = adj_layout(ctx, words, per, states, n_seg > 1 ? 2 : 1);
            e = cudaMalloc(&sc.p, L.need);
        }
        if (e != cudaSuccess) {
            sc.p = nullptr;
            cudaGetLastError();
            return set_err(ctx, ABP_ENOMEM, "abp_backward: scratch allocation failed", e);
        }
        sc.cap = L.need;
    }
    sc.bytes = L.need;
    char *base = (char *)sc.p;
    float4 *sub[2] = {(float4 *)(base + L.off_sub), (float4 *)(base + L.off_sub + align256(L.sub1))};
    uint4 *wbuf[2] = {(uint4 *)(base + L.off_words), (uint4 *)(base + L.off_words + align256(L.words1))};
    double *partials = (double *)(base + L.off_part);
    double *gdev = (double *)(base + L.off_grad);
    double *wdev = (double *)(base + L.off_w);
    const size_t lam_bytes = L.lam, g_bytes = L.g;
    SegView sv;
    sv.lam = (float4 *)(base + L.off_lam);
    sv.G = (double *)(base + L.off_g);
    cudaStream_t s = ctx->stream;
    cudaError_t e = cudaSuccess;
    const double *w = nullptr;
    if (dJ_dmean_v) {
        if (kw == PtrKind::Device) {
            w = dJ_dmean_v;
        } else {
            e = cudaMemcpyAsync(wdev, dJ_dmean_v, sizeof(double) * ctx->n_sets, cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward: weight upload", e);
            w = wdev;
        }
    }
    if (ctx->n_sets == 0) return ABP_OK;
    if (ctx->n_tiles > 0) {
        AdjArgs a;
        a.b = ctx->batch();
        a.ck = ctx->ckpt();
        a.nz = ctx->noise();
        a.sub = sub[0];
        a.n_sub = states ? Kc : n_sub;
        a.per = (int)per;
        a.words = nullptr;
        a.tile0 = 0;
        a.n_blk = n_sub * (kSub / 4);
        a.w = w;
        a.partials = partials;
        for (int r = 0; r < 10; ++r) {
            a.K.rk[2 * r] = a.nz.k0 + (uint32_t)r * kPhiloxW0;
            a.K.rk[2 * r + 1] = a.nz.k1 + (uint32_t)r * kPhiloxW1;
        }
        e = cudaMemsetAsync(sv.lam, 0, lam_bytes, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(sv.G, 0, g_bytes, s);
        if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward: clear", e);
        const int64_t n_run = (n_seg + per - 1) / per;  // launches of each kernel
        // blocks per tile: tiles hold up to kThreads * ppt trajectories
        const int cap = kThreads * std::max(ctx->ppt, 1);
        const int sub1 = pair_blocks_per_tile(ctx, kL1Threads);
        const int sub2 = pair_blocks_per_tile(ctx, kRevPairThreads);
        const int sub_st = (cap + kL1Threads - 1) / kL1Threads, sub_sw = (cap + kSweepThreads - 1) / kSweepThreads;
        // The tiles in two halves, each with its own pair of streams: a trajectory's sweep
        // depends on no other's, so while one half's launch of a segment drains (its last
        // blocks fill the SMs partly, and its next launch waits for them) the other half's
        // blocks take the free SMs.  Backward of one set, K = 1,000, against one group:
        // 262,144 trajectories 2.67 -> 2.48 ps per particle-step, 175,104 2.91 -> 2.56,
        // 131,072 3.09 -> 2.71, 1,048,576 2.40 -> 2.38 (three, four and six groups: within 2%
        // of two).  A batch with fewer blocks than SMs runs in one group: it leaves SMs
        // free anyway, and each launch costs host time.  With one or two launches there is
        // little to fill in, so one group too unless it has three blocks per SM (K = 1,000, 2,000
        // steps, two groups against one: 50,000 trajectories 495 us and 430, 100,000 702 and
        // 662, 131,072 793 and 858, 262,144 1,377 and 1,418).
        const int64_t blocks = (int64_t)ctx->n_tiles * sub2;
        const int n_grp = !states && ctx->n_tiles >= 2 && blocks >= (n_run > 2 ? 1 : 3) * (int64_t)ctx->sm_count ? kAdjGroups : 1;
        // the groups' streams and events, kept for the next call
        for (int i = 0; e == cudaSuccess && i < 2 * n_grp - 1; ++i)
            if (!ctx->adj_stream[i]) e = cudaStreamCreateWithFlags(&ctx->adj_stream[i], cudaStreamNonBlocking);
        for (int i = 0; e == cudaSuccess && i < 2 + 4 * n_grp; ++i)
            if (!ctx->adj_ev[i]) e = cudaEventCreateWithFlags(&ctx->adj_ev[i], cudaEventDisableTiming);
        if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward: stream set-up", e);
        struct Group {
            cudaStream_t rev, l1;
            cudaEvent_t *l1_done, *rev_done;  // [2] by launch parity
            int t0, t1;
        } grp[kAdjGroups];
        for (int g = 0; g < n_grp; ++g) {
            grp[g].rev = g == 0 ? s : ctx->adj_stream[2 * g];
            grp[g].l1 = ctx->adj_stream[g == 0 ? 0 : 2 * g - 1];
            grp[g].l1_done = ctx->adj_ev + 2 + 4 * g;
            grp[g].rev_done = ctx->adj_ev + 4 + 4 * g;
            grp[g].t0 = (int)((int64_t)ctx->n_tiles * g / n_grp);
            grp[g].t1 = (int)((int64_t)ctx->n_tiles * (g + 1) / n_grp);
        }
        const cudaEvent_t start = ctx->adj_ev[0], end = ctx->adj_ev[1];
        auto wait = [&](cudaStream_t st, cudaEvent_t ev) {
            if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev, 0);
        };
        auto record = [&](cudaEvent_t ev, cudaStream_t st) {
            if (e == cudaSuccess) e = cudaEventRecord(ev, st);
        };
        // launch j covers the segments [j per, (j + 1) per); level 1 of launch j writes
        // buffer j % 2 and may start once the reverse sweep of launch j + 2, the last
        // reader of that buffer, has finished
        auto segments = [&](int64_t j) { return (unsigned)std::min(per, n_seg - j * per); };
        auto level1 = [&](const Group &g, int64_t j) {
            if (e != cudaSuccess) return;  // nothing is launched whose order is not established
            AdjArgs aj = a;
            aj.sub = sub[j & 1];
            aj.tile0 = g.t0;
            const dim3 g1((unsigned)((int64_t)(g.t1 - g.t0) * sub1), segments(j));
            if (states)
                adjoint_states_kernel<<<dim3((unsigned)((g.t1 - g.t0) * sub_st), segments(j)), kL1Threads, 0, g.l1>>>(
                    aj, j * per, sub_st);
            else if (words) {
                aj.words = wbuf[j & 1];
                adjoint_level1_pair_kernel<true><<<g1, kL1Threads, 0, g.l1>>>(aj, j * per, sub1);
            } else
                adjoint_level1_pair_kernel<false><<<g1, kL1Threads, 0, g.l1>>>(aj, j * per, sub1);
            record(g.l1_done[j & 1], g.l1);
        };
        auto reverse = [&](const Group &g, int64_t j) {
            wait(g.rev, g.l1_done[j & 1]);
            if (e != cudaSuccess) return;
            AdjArgs as = a;
            as.sub = sub[j & 1];
            as.tile0 = g.t0;
            const unsigned g2 = (unsigned)((int64_t)(g.t1 - g.t0) * sub2);
            if (states) {
                adjoint_sweep_kernel<<<(unsigned)((g.t1 - g.t0) * sub_sw), kSweepThreads, 0, g.rev>>>(
                    as, sv, j * per, (int)segments(j), sub_sw, window);
            } else {
                if (words) as.words = wbuf[j & 1];
                const auto kernel = !words    ? adjoint_reverse_pair_kernel<false, false>
                                    : per > 1 ? adjoint_reverse_pair_kernel<true, true>
                                              : adjoint_reverse_pair_kernel<true, false>;
                kernel<<<g2, kRevPairThreads, 0, g.rev>>>(as, sv, j * per, (int)segments(j), sub2, window);
            }
            record(g.rev_done[j & 1], g.rev);
            ctx->launches += 2;
        };
        record(start, s);  // the checkpoints of the forward and the cleared sums are complete
        for (int g = 0; g < n_grp; ++g) {
            wait(grp[g].l1, start);
            if (g > 0) wait(grp[g].rev, start);
            if (n_run > 0) level1(grp[g], n_run - 1);
        }
        for (int64_t j = n_run - 1; e == cudaSuccess && j >= 0; --j)
            for (int g = 0; g < n_grp; ++g) {
                if (j > 0) {
                    if (j + 1 < n_run) wait(grp[g].l1, grp[g].rev_done[(j + 1) & 1]);
                    level1(grp[g], j - 1);
                }
                reverse(grp[g], j);
            }
        // The caller's stream follows all launches: it waits for the sweeps' streams, which have
        // waited for their level-1 streams, and after an error for those as well (on the host
        // where an event cannot be used).
        auto join = [&](cudaStream_t st) {
            cudaError_t je = cudaEventRecord(end, st);
            if (je == cudaSuccess) je = cudaStreamWaitEvent(s, end, 0);
            if (je != cudaSuccess) cudaStreamSynchronize(st);
            if (e == cudaSuccess) e = je;
        };
        for (int g = 1; g < n_grp; ++g) join(grp[g].rev);
        if (e != cudaSuccess)
            for (int g = 0; g < n_grp; ++g) join(grp[g].l1);
        if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward: launch", e);
        adjoint_final_kernel<<<ctx->n_tiles, kThreads, 0, s>>>(a, sv);
        ctx->launches += 1;
    }
    adjoint_set_kernel<<<ctx->n_sets, kThreads, 0, s>>>(ctx->batch(), partials, gdev);
    ctx->launches += 1;
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward: launch", e);
    const size_t out_bytes = sizeof(double) * 6 * (size_t)ctx->n_sets;
    if (kg == PtrKind::Device) {
        e = cudaMemcpyAsync(grad, gdev, out_bytes, cudaMemcpyDeviceToDevice, s);
    } else {
        e = cudaMemcpyAsync(grad, gdev, out_bytes, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward: gradient copy", e);
    ctx->adj_valid = true;
    return ABP_OK;
}

extern "C" abp_status abp_backward_traj(abp_ctx *ctx, double *dvbar) {
    const NvtxRange nvtx("abp_backward_traj");
    if (!ctx) return ABP_EINVAL;
    if (!dvbar) return set_err(ctx, ABP_EINVAL, "abp_backward_traj: dvbar is NULL");
    if (!ctx->have_batch || !ctx->adj_valid)
        return set_err(ctx, ABP_ESTATE, "abp_backward_traj: no abp_backward since the batch was last (re)started");
    const PtrKind k = ptr_kind(dvbar, ctx->device);
    if (k == PtrKind::OtherDevice) return set_err(ctx, ABP_EINVAL, "abp_backward_traj: output on another GPU");
    const int64_t T = ctx->total_traj;
    if (T == 0 || ctx->n_tiles == 0) return ABP_OK;
    // the per-trajectory sums of the last backward call: the same scratch layout as there
    const int64_t n_sub = sub_slots(ctx->cfg.checkpoint_every);
    const AdjLayout L = adj_layout(ctx, false);  // the hand-off buffers come after the sums
    char *base = (char *)ctx->d_adj.p;
    SegView sv;
    sv.lam = (float4 *)(base + L.off_lam);
    sv.G = (double *)(base + L.off_g);
    AdjArgs a;
    a.b = ctx->batch();
    a.ck = ctx->ckpt();
    a.nz = ctx->noise();
    a.sub = nullptr;
    a.n_sub = n_sub;
    a.words = nullptr;
    a.per = 1;
    a.tile0 = 0;
    a.n_blk = 0;
    a.w = nullptr;
    a.partials = nullptr;
    cudaStream_t s = ctx->stream;
    const size_t bytes = sizeof(double) * 6 * (size_t)T;
    DevBuf tmp;
    double *dst = dvbar;
    if (k != PtrKind::Device) {
        const cudaError_t ea = cudaMalloc(&tmp.p, bytes);
        if (ea != cudaSuccess) {
            tmp.p = nullptr;
            cudaGetLastError();
            return set_err(ctx, ABP_ENOMEM, "abp_backward_traj: staging buffer", ea);
        }
        dst = (double *)tmp.p;
    }
    adjoint_traj_kernel<<<ctx->n_tiles, kThreads, 0, s>>>(a, sv, dst);
    ctx->launches += 1;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && k != PtrKind::Device) {
        e = cudaMemcpyAsync(dvbar, dst, bytes, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    tmp.release();
    if (e != cudaSuccess) return set_err(ctx, ABP_ECUDA, "abp_backward_traj", e);
    return ABP_OK;
}
