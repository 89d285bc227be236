// BigBird block-sparse attention forward on Blackwell tensor cores (sm_100a).
//
// What is computed: Eq. (AT) of arXiv 2007.14062 (softmax attention restricted to the out-neighbours of each
// query) over the block graph of App. D.  How, on B200:
//
//   * Two query blocks are stacked into one 128-row tile so that every tcgen05.mma runs at M = 128.  The tile
//     walks a list of key blocks prepared on the host; each is attended by both halves of the tile or by one.
//     The MMAs always cover all 128 rows; rows that do not attend a key block get probability zero for it.
//   * One CTA per SM runs two independent tile streams side by side.  Each stream owns half of tensor memory
//     (scores 128 | probabilities 64 | output accumulator 64 columns), a Q double buffer and a ring of K / V
//     tiles in shared memory, an MMA-issuing thread and a softmax warpgroup.  Two issuing threads keep the
//     tensor pipe full where one thread's issue rate would not (a 64-wide P V instruction takes the pipe less
//     time than one thread needs to issue the next), and the two softmax warpgroups fill each other's gaps on
//     the special-function unit.
//   * Four lanes of a producer warp (per stream one for Q and K, one for V) fetch Q once per tile and the K and V
//     blocks with TMA (128-byte swizzle) straight from the [B, H, N, D] tensors into the stream's ring: nothing is
//     gathered or packed in HBM.
//   * Key blocks are processed two at a time (one "step").  Their K tiles land in adjacent ring slots, so that
//     S = Q K^T of a step is one N = 128 tcgen05.mma per 16 head dimensions.  O += P V follows with P read
//     from tensor memory.
//   * Softmax warpgroup, one thread per row of the tile: the thread pulls its (up to) 128 scores into registers
//     with tcgen05.ld and hands the score columns back at once, so that the next step's Q K^T runs under this
//     step's exponentials; it applies the key-padding mask, takes the row maximum, exponentiates (base 2, fp32),
//     sums, and writes bf16 probabilities with tcgen05.st (zeros for key blocks its half of the tile does not
//     attend).  The accumulator is rescaled only when the running maximum grows by more than 2^8.
//   * An epilogue warpgroup shared by the two streams takes a finished tile's accumulator out of tensor memory,
//     scales it by 1/l and writes the output rows, while the stream's softmax threads are already on the next tile.
//   * A global-row tile of a long sequence is cut along the keys into parts that are separate work items; each
//     writes its unnormalised accumulator and (max, sum) per row to scratch, and a small merge kernel combines
//     the parts in a fixed order.
//   * CTAs are persistent; a scheduler warp draws work for both streams from a global counter: global-row tiles
//     first, then the sparse tiles in (batch, head)-major order.
//
// Every wait on an mbarrier is bounded: on expiry the kernel records BIGBIRD_ETIMEOUT and returns.
#include <algorithm>
#include <mutex>

#include "sm100.cuh"

namespace bigbird {
namespace {

// ------------------------------------------------------------------------------------------------ constants
constexpr int kStepChunks = 2;             // key blocks per step
constexpr int kRingGroups = 4;             // ring of groups of kStepChunks adjacent tiles (the K or the V blocks of one step)
constexpr int kGroupBytes = kStepChunks * kTileBytes;
constexpr int kStreams = 2;                // tile streams per CTA
// warps 0..3 / 4..7: softmax of stream 0 / 1; warps 8..11: epilogue; warp 12: TMA producer; warps 13, 14: MMA issuers
// of stream 0 / 1; warp 15: scheduler
constexpr int kThreads = 512;
constexpr int kWarpEpilogue = 8, kWarpProducer = 12, kWarpMma = 13, kWarpScheduler = 15;
constexpr int kSoftmaxThreads = 128;
// 512 threads start with 128 registers each; the roles then trade.  A sub-partition's registers are shared out
// among its own four warps only (setmaxnreg can hand out no more than those warps gave back): two softmax warps x 200
// (a step's 128 scores plus the loop's temporaries) + an epilogue warp x 56 + a light warp x 56 = 4 x 128 exactly.
// Nothing may spill: a spill here costs a trip to L2, since nearly all of the SM's L1 is configured as shared memory.
#ifndef BB_REGS_SOFTMAX
#define BB_REGS_SOFTMAX 200
#define BB_REGS_EPILOGUE 56
#define BB_REGS_LIGHT 56
#endif
constexpr int kRegsSoftmax = BB_REGS_SOFTMAX, kRegsEpilogue = BB_REGS_EPILOGUE, kRegsLight = BB_REGS_LIGHT;
static_assert(2 * kRegsSoftmax + kRegsEpilogue + kRegsLight <= 4 * 128 && kThreads == 512, "register trade between the four warps of a sub-partition");
constexpr int kTmemCols = 512;
constexpr int kStreamCols = kTmemCols / kStreams;
constexpr int kColS = 0;                   // scores: kStepChunks x 64 fp32 columns
constexpr int kColP = kStepChunks * 64;    // probabilities: kStepChunks x 32 columns of packed bf16 pairs
constexpr int kColO = kColP + kStepChunks * 32;   // output accumulator: 64 fp32 columns
constexpr float kRescaleThreshold = 8.0f;  // in log2 units
constexpr int kSchedSlots = 3;
constexpr int kPartialFloats = 128 * 64 + 2 * 128;   // one part of a split tile: O[128][64], max[128], sum[128]
constexpr int kSegChunks = 96;             // live key blocks per posted segment of a tile (a multiple of kStepChunks)
static_assert(kColO + 64 <= kStreamCols && kSegChunks % kStepChunks == 0, "tensor-memory and segment layout");

// A key block of a tile after the key-padding mask has been applied.
struct __align__(16) ChunkEntry {
    int c;                         // key block
    int who;                       // bits 0..1: kBothHalves, kUpperHalf or kLowerHalf (the halves of the tile that attend it);
                                   // bit 2 (kHasPadding): some of its keys are padding
    unsigned long long kb;         // valid-key bits (never 0: blocks that are entirely padding are dropped)
};
enum { kSegFirst = 1, kSegLast = 2 };
enum { kWhoMask = 3, kHasPadding = 4, kNoChunk = 3 };
struct __align__(16) WorkSlot {
    int w;                         // work index, -1 = no more work
    int bh, batch, qa, qb;
    int n_chunks;
    int flags;
    int part_slot;                 // >= 0: the tile is one part of a split tile and writes partial results there
    unsigned long long qbits_a, qbits_b;
    ChunkEntry chunks[kSegChunks];         // step s of the segment covers chunks [kStepChunks s, kStepChunks (s + 1))
};
// What the softmax threads of a stream hand to the epilogue warpgroup at the end of a tile.
enum { kEpiTile = 0, kEpiDone = 1 };
struct __align__(16) EpiMsg {
    int kind;                      // kEpiTile, or kEpiDone: the stream has no more tiles
    int bh, qa, qb;
    int part_slot;
    int pad_[3];
    float inv[kSoftmaxThreads];    // per row: 1 / l, 0 if there is no such thing, -1 for a padded row, which comes out as zeros
};

struct __align__(16) StreamCtl {
    unsigned long long full[kRingGroups];
    unsigned long long empty[kRingGroups];
    unsigned long long q_full[2], q_empty[2];
    unsigned long long s_full, s_free, p_full, pv_done;
    unsigned long long o_done, o_free;     // a tile's last P V has completed / the epilogue has taken the accumulator
    unsigned long long epi_full[2];
    unsigned long long sched_full[kSchedSlots], sched_empty[kSchedSlots];
    WorkSlot slot[kSchedSlots];
    EpiMsg epi[2];
};
struct __align__(16) SmemCtl {
    StreamCtl st[kStreams];
    unsigned tmem_base;
    int abort_flag;
};
// per stream: two Q buffers of two tiles each, then the ring
constexpr int kStreamSmemQ = 0;
constexpr int kStreamSmemRing = 4 * kTileBytes;
constexpr int kStreamSmemBytes = kStreamSmemRing + kRingGroups * kGroupBytes;
constexpr int kSmemCtl = kStreams * kStreamSmemBytes;
constexpr int kSmemBytes = kSmemCtl + (int)sizeof(SmemCtl) + 1024;   // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 227 * 1024, "shared memory per CTA");

struct KernelParams {
    __nv_bfloat16* out;
    float* lse;
    const unsigned long long* kbits;   // [B * nb] or nullptr
    const Item* items;
    const Step* steps;
    int* counter;                      // [2]: next work index, finished CTAs
    int* status;                       // [2]: code, detail
    int items_per_head, global_tiles;  // of the layout's schedule, the global tiles first
    int parts, part_steps;             // how this launch cuts them (part_steps: key blocks)
    int BH, H, nb;
    int total_work;
    int ahead;                         // tiles that a stream has in hand at most, 2 .. kSchedSlots
    float scale_log2;
    float* partials;                   // [BH * global_tiles * parts][kPartialFloats], if parts > 1
};

// ------------------------------------------------------------------------------------------------ helpers
__device__ __forceinline__ unsigned long long key_bits(const KernelParams& p, int batch, int c) {
    if (c < 0) return 0ull;
    return p.kbits ? p.kbits[(size_t)batch * p.nb + c] : ~0ull;
}
__device__ __forceinline__ float row_max64(const float* s) {
    float mx0 = max3(s[0], s[1], s[2]), mx1 = max3(s[3], s[4], s[5]), mx2 = max3(s[6], s[7], s[8]), mx3 = max3(s[9], s[10], s[11]);
#pragma unroll
    for (int j = 12; j < 60; j += 8) {
        mx0 = max3(mx0, s[j], s[j + 1]);
        mx1 = max3(mx1, s[j + 2], s[j + 3]);
        mx2 = max3(mx2, s[j + 4], s[j + 5]);
        mx3 = max3(mx3, s[j + 6], s[j + 7]);
    }
    return fmaxf(max3(mx0, mx1, fmaxf(s[60], s[61])), max3(mx2, mx3, fmaxf(s[62], s[63])));
}

// Rare paths of the softmax threads.
// -inf over the scores of the padded keys of one key block, in tensor memory.
__device__ __forceinline__ void mask_scores(unsigned taddr, unsigned long long kb) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {                   // 32 keys at a time (rolled: a rare path should not take up code space)
        float s[32];
        const unsigned bits = (unsigned)(kb >> (32 * h));
        tmem_ld32(taddr + 32 * h, s);
        tmem_wait_ld();
#pragma unroll
        for (int t = 0; t < 32; ++t) s[t] = ((bits >> t) & 1u) ? s[t] : -INFINITY;
        tmem_st32(taddr + 32 * h, reinterpret_cast<unsigned*>(s));
    }
    tmem_wait_st();
}
// This thread's row of the output accumulator times alpha (the running maximum moved by more than the threshold).
__device__ __forceinline__ void rescale_accumulator(unsigned taddr, float alpha) {
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        float o[16];
        tmem_ld16(taddr + c * 16, o);
        tmem_wait_ld();
#pragma unroll
        for (int t = 0; t < 16; t += 2) fmul2(o[t], o[t + 1], alpha);
        tmem_st16(taddr + c * 16, reinterpret_cast<unsigned*>(o));
    }
}

// What every role needs to know about its stream.
struct StreamRef {
    StreamCtl* sc;
    unsigned char* smem;           // the stream's Q buffers and ring
    unsigned tmem;                 // tensor-memory address of the stream's first column (lane 0)
};

// ------------------------------------------------------------------------------------------------ scheduler (one warp, both streams)
// Zeros and -inf to the rows of a tile that holds no token.  (By the scheduler itself, with nothing in its way but its own stores: such a
// tile takes no slot and none of its stream's time: [16, 16, 4096] with 1024 to 4096 tokens 213 -> 196 us.  Two stores a round and no
// address arithmetic beside them: with an address made for each store a tile took two microseconds, and a batch without any token,
// [16, 16, 4096], 108 us instead of 81.  Unrolled further it is 73 us, but the 300 bytes more of code cost full sequences 0.5 %.)
// row_a, row_b: blocks of the B H N / 64 ones; row_b < 0: none.
__device__ __forceinline__ void clear_tile(__nv_bfloat16* out, float* lse, int row_a, int row_b, int lane) {
#pragma unroll 1
    for (int h = 0; h < (row_b >= 0 ? 2 : 1); ++h) {
        const size_t tok = (size_t)(h ? row_b : row_a) * kBlock;
        uint4* dst = reinterpret_cast<uint4*>(out + tok * kBlock) + lane;
#pragma unroll 1
        for (int i = 0; i < 8; ++i, dst += 64) dst[0] = dst[32] = make_uint4(0u, 0u, 0u, 0u);
        if (lse) lse[tok + lane] = lse[tok + 32 + lane] = -INFINITY;
    }
}

// Fetches the next work item for a stream that has a token among its rows, drops the key blocks that are entirely padding and posts the
// live list.  Returns the work index (-1: the stream has been told that there is no more work), or -2 after an expired wait.
__device__ __forceinline__ int schedule_one(const KernelParams& p, SmemCtl* ctl, StreamCtl* sc, int stream, unsigned& sched_n, bool& drawn, int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    int w, bh, batch, part_slot;
    bool heavy;
    Item item;
    unsigned long long qbits_a, qbits_b;
#pragma unroll 1
    for (;;) {                                      // up to a tile with a token
        // A stream's first item is its own, which spreads the global tiles over the SMs (the second streams in the opposite order, so
        // that with little work a CTA with a global tile has nothing else); after that they are drawn.
        w = stream == 0 ? (int)blockIdx.x : (int)(2 * gridDim.x - 1 - blockIdx.x);
        static_assert(kStreams == 2, "first items");
        if (drawn) {
            if (lane == 0) w = (int)gridDim.x * kStreams + atomicAdd(&p.counter[0], 1);
            w = __shfl_sync(0xffffffffu, w, 0);
        }
        drawn = true;
        if (w >= p.total_work) w = -1;
        // decode the work index: the parts of the global-row tiles of every (batch, head) first, then the sparse tiles
        bh = 0; batch = 0; part_slot = -1;
        heavy = false;
        item = Item{};
        if (w >= 0) {
            const unsigned heavy_total = (unsigned)(p.BH * p.global_tiles * p.parts);
            heavy = (unsigned)w < heavy_total;
            const unsigned per_head = heavy ? p.global_tiles * p.parts : p.items_per_head - p.global_tiles;
            const unsigned x = heavy ? w : w - heavy_total;
            bh = (int)(x / per_head);                   // (one division for either kind of item: this code is kept small)
            int it = (int)(x - bh * per_head), part = 0;
            batch = (int)((unsigned)bh / (unsigned)p.H);
            if (heavy) {
                part = it % p.parts;
                it = it / p.parts;
                if (p.parts > 1) part_slot = (int)x;
            } else it += p.global_tiles;
            if (BB_CHECK(bh >= 0 && bh < p.BH && it >= 0 && it < p.items_per_head, 71)) item = p.items[(size_t)(bh - batch * p.H) * p.items_per_head + it];
            else w = -1;
            if (heavy) {                                // its list is every block of the sequence
                item.step_begin = part * p.part_steps;
                item.step_count = min(p.part_steps, p.nb - item.step_begin);
            }
            if (!BB_CHECK(item.step_count >= 0 && item.step_begin >= 0 && item.qa >= 0 && item.qa < p.nb && item.qb < p.nb, 72)) w = -1;
        }
        qbits_a = w >= 0 ? key_bits(p, batch, item.qa) : 0ull;
        qbits_b = w >= 0 ? key_bits(p, batch, item.qb) : 0ull;
        if (__builtin_expect(w < 0 || (qbits_a | qbits_b) != 0ull, 1)) break;
        // (nothing for a part of a split tile: the merge zeroes padded rows whatever stands in their parts)
        if (part_slot < 0) clear_tile(p.out, p.lse, bh * p.nb + item.qa, item.qb >= 0 ? bh * p.nb + item.qb : -1, lane);
    }
    const int n_raw = w >= 0 ? item.step_count : 0;
    int i0 = 0;
    bool first = true;
    do {
        const unsigned ss = sched_n % kSchedSlots, sp = (sched_n / kSchedSlots) & 1u;
        // the first slot of an item is known to be free (the caller tested it); later segments of a long tile wait here
        if (!mbar_wait(&sc->sched_empty[ss], sp ^ 1u, &ctl->abort_flag)) { give_up(&ctl->abort_flag, p.status, 11); return -2; }
        WorkSlot* slot = &sc->slot[ss];
        int count = 0;
#pragma unroll 1
        while (i0 < n_raw && count <= kSegChunks - 32) {
            const int i = i0 + lane;
            ChunkEntry e{-1, 0, 0ull};
            bool alive = false;
            if (i < n_raw) {
                const Step s = heavy ? Step{item.step_begin + i, kBothHalves} : p.steps[item.step_begin + i];
                // halves whose query rows are all padding do not attend anything
                const bool ua = s.who != kLowerHalf && qbits_a != 0ull;
                const bool ub = s.who != kUpperHalf && qbits_b != 0ull;
                e.c = s.c;
                e.kb = key_bits(p, batch, s.c);
                e.who = ((ua && ub) ? kBothHalves : (ua ? kUpperHalf : kLowerHalf)) | (e.kb != ~0ull ? kHasPadding : 0);
                alive = e.kb != 0ull && (ua || ub);
                if (!BB_CHECK(s.c >= 0 && s.c < p.nb && (unsigned)s.who <= (unsigned)kLowerHalf, 70)) alive = false;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, alive);
            if (alive) slot->chunks[count + __popc(bal & lt_mask)] = e;
            count += __popc(bal);
            i0 += 32;
        }
        if (lane == 0) {
            slot->w = w;
            slot->bh = bh;
            slot->batch = batch;
            slot->qa = item.qa;
            slot->qb = item.qb;
            slot->n_chunks = count;
            slot->flags = (first ? kSegFirst : 0) | (i0 >= n_raw ? kSegLast : 0);
            slot->qbits_a = qbits_a;
            slot->qbits_b = qbits_b;
            slot->part_slot = w >= 0 ? part_slot : -1;
        }
        __threadfence_block();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sc->sched_full[ss]);
        ++sched_n;
        first = false;
    } while (i0 < n_raw);
    return w;
}

__device__ __forceinline__ void scheduler_role(const KernelParams& p, SmemCtl* ctl, int lane) {
    unsigned sched_n0 = 0, sched_n1 = 0;            // slots posted per stream (scalars: an indexed array would live in local memory)
    unsigned done = 0, drawn = 0;                   // bit s: stream s has been told that there is no more work; has had an item
    IdleClock idle;
    while (done != (1u << kStreams) - 1u) {
        bool progress = false;
#pragma unroll 1
        for (int s = 0; s < kStreams; ++s) {        // (not unrolled: one copy of the code)
            if ((done >> s) & 1u) continue;
            StreamCtl* sc = &ctl->st[s];
            unsigned n = s == 0 ? sched_n0 : sched_n1;
            // (the slot posted `ahead` slots ago must have been given back)
            const unsigned m = n - (unsigned)p.ahead;
            if (n >= (unsigned)p.ahead && !__all_sync(0xffffffffu, mbar_test(&sc->sched_empty[m % kSchedSlots], (m / kSchedSlots) & 1u))) continue;
            bool d = (drawn >> s) & 1u;
            const int w = schedule_one(p, ctl, sc, s, n, d, lane);
            drawn |= 1u << s;
            if (s == 0) sched_n0 = n; else sched_n1 = n;
            if (w == -2) return;
            if (w < 0) done |= 1u << s;
            progress = true;
        }
        if (progress) idle.reset();
        else if (!__all_sync(0xffffffffu, idle.tick(&ctl->abort_flag, p.status, 12, 400))) return;
    }
}

// ------------------------------------------------------------------------------------------------ TMA producer (two lanes per stream)
// Four lanes of the producer warp: per stream one fetches Q and the K blocks, the other the V blocks.  The ring
// order of a stream is the order in which its MMA thread consumes groups, K0 K1 V0 K2 V1 K3 ...: the K blocks of
// step t go to ring entry 2t - 1 (0 for t = 0), its V blocks to entry 2t + 2, so the two lanes never need to talk.
// A lane cannot block (it shares its warp with the others): it polls, backing off briefly between rounds.
__device__ __forceinline__ bool poll_wait(unsigned long long* bar, unsigned parity, IdleClock& idle, int* abort_flag, int* status, int code) {
    while (!mbar_test(bar, parity))
        if (!idle.tick(abort_flag, status, code, 20)) return false;
    idle.reset();
    return true;
}

__device__ __forceinline__ void producer_role(const KernelParams& p, SmemCtl* ctl, const StreamRef& sr, bool v_lane,
                                              const CUtensorMap* tm_q, const CUtensorMap* tm_k, const CUtensorMap* tm_v) {
    StreamCtl* sc = sr.sc;
    int* abort_flag = &ctl->abort_flag;
    const CUtensorMap* tm = v_lane ? tm_v : tm_k;
    unsigned sched_n = 0, q_n = 0, step_n = 0;      // step_n: steps of this stream seen so far
    IdleClock idle;
    for (;;) {
        const unsigned ss = sched_n % kSchedSlots, sp = (sched_n / kSchedSlots) & 1u;
        if (!poll_wait(&sc->sched_full[ss], sp, idle, abort_flag, p.status, 13)) return;
        const WorkSlot* slot = &sc->slot[ss];
        const int w = slot->w, flags = slot->flags, bh = slot->bh, n = slot->n_chunks;
        if (w >= 0) {
            if (!v_lane && (flags & kSegFirst)) {
                const int qa = slot->qa, qb = slot->qb;
                const unsigned qs = q_n & 1u;
                if (!poll_wait(&sc->q_empty[qs], ((q_n >> 1) & 1u) ^ 1u, idle, abort_flag, p.status, 12)) return;
                mbar_expect_tx(&sc->q_full[qs], qb >= 0 ? 2 * kTileBytes : kTileBytes);
                tma_load_tile(sr.smem + kStreamSmemQ + qs * 2 * kTileBytes, tm_q, (bh * p.nb + qa) * kBlock, &sc->q_full[qs]);
                if (qb >= 0) tma_load_tile(sr.smem + kStreamSmemQ + qs * 2 * kTileBytes + kTileBytes, tm_q, (bh * p.nb + qb) * kBlock, &sc->q_full[qs]);
                ++q_n;
            }
            for (int i = 0; i < n; i += kStepChunks) {
                const int cnt = min(kStepChunks, n - i);
                const unsigned ring_i = v_lane ? 2u * step_n + 2u : (step_n == 0u ? 0u : 2u * step_n - 1u);
                const unsigned g = ring_i % kRingGroups, ph = (ring_i / kRingGroups) & 1u;
                const int c0 = slot->chunks[i].c, c1 = cnt > 1 ? slot->chunks[i + 1].c : 0;
                if (!BB_CHECK(bh >= 0 && bh < p.BH && c0 >= 0 && c0 < p.nb && c1 >= 0 && c1 < p.nb && n <= kSegChunks, 73)) return;
                if (!poll_wait(&sc->empty[g], ph ^ 1u, idle, abort_flag, p.status, 10)) return;
                mbar_expect_tx(&sc->full[g], cnt * kTileBytes);
                tma_load_tile(sr.smem + kStreamSmemRing + g * kGroupBytes, tm, (bh * p.nb + c0) * kBlock, &sc->full[g]);
                if (cnt > 1) tma_load_tile(sr.smem + kStreamSmemRing + g * kGroupBytes + kTileBytes, tm, (bh * p.nb + c1) * kBlock, &sc->full[g]);
                ++step_n;
            }
        }
        mbar_arrive(&sc->sched_empty[ss]);
        ++sched_n;
        if (w < 0) return;
    }
}

// ------------------------------------------------------------------------------------------------ MMA issuer (one thread per stream)
// One thread per stream walks the posted slots; a round issues S = Q K^T of a step and, behind it, O += P V of the
// step before (whose probabilities the softmax threads were writing meanwhile).  The thread is alone in its warp, so
// nothing hides its latencies: every branch stalls it until the target is known and every barrier test is a round
// trip to shared memory.  Hence the shape of the loop: the two barriers a product needs are tested back to back and
// one branch takes the combined result; a second key block and the end of a tile are predicated instructions.
// Ring entries (see the producer): the K blocks of step t sit in entry 2t - 1 (0 for t = 0), its V blocks in 2t + 2.
__device__ __forceinline__ void mma_role(const KernelParams& p, SmemCtl* ctl, const StreamRef& sr) {
    StreamCtl* sc = sr.sc;
    int* abort_flag = &ctl->abort_flag;
    unsigned q_n = 0, sched_n = 0, grp_n = 0, pv_n = 0, tile_n = 0;   // grp_n: steps whose Q K^T was issued; tile_n: tiles handed to the epilogue
    int fail = 0;                               // code of the wait that was abandoned, if any
    unsigned pend_cnt = 0;                      // key blocks of the step whose P V is still to be issued (0: none)
    bool pend_fresh = false;                    // ... it is the first of its tile: it overwrites O
    bool pend_last = false;                     // ... the last of its tile: the accumulator is complete after it
    bool tile_steps = false;                    // the current tile has had a step
    const unsigned q_base = smem_u32(sr.smem + kStreamSmemQ), ring_base = smem_u32(sr.smem + kStreamSmemRing);
    // both barriers at once; the blocking waits only if one of them is not there yet
    auto wait2 = [&](unsigned long long* b1, unsigned par1, bool need1, int code1, unsigned long long* b2, unsigned par2, int code2) -> bool {
        const bool t1 = mbar_test(b1, par1), t2 = mbar_test(b2, par2);
        if (__builtin_expect((t1 || !need1) && t2, 1)) return true;
        if (need1 && !mbar_wait(b1, par1, abort_flag)) { fail = code1; return false; }
        if (!mbar_wait(b2, par2, abort_flag)) { fail = code2; return false; }
        return true;
    };
    for (;;) {
        const unsigned ss = sched_n % kSchedSlots, sp = (sched_n / kSchedSlots) & 1u;
        if (!mbar_wait(&sc->sched_full[ss], sp, abort_flag)) { fail = 23; break; }
        const WorkSlot* slot = &sc->slot[ss];
        const int w = slot->w, flags = slot->flags, n = slot->n_chunks;
        const bool work = w >= 0;
        const bool first = work && (flags & kSegFirst), last = work && (flags & kSegLast);
        if (first) {
            tile_steps = false;
            ++q_n;                              // this tile's Q sits in buffer (q_n - 1) & 1
            if (!mbar_wait(&sc->q_full[(q_n - 1) & 1u], ((q_n - 1) >> 1) & 1u, abort_flag)) { fail = 24; break; }
        }
        const unsigned qs = (q_n - 1) & 1u;
        const unsigned long long q_desc = smem_desc_sw128(q_base + qs * 2 * kTileBytes);
        // one round per step of the slot; the slot that says "no more work" gets one round without a Q K^T, which
        // issues the very last P V
        const int n_rounds = work ? (n + kStepChunks - 1) / kStepChunks : (w < 0 ? 1 : 0);
        bool tile_fresh = first;
#pragma unroll 1
        for (int r = 0; r < n_rounds; ++r) {
            const unsigned cnt = work ? (unsigned)min(kStepChunks, n - r * kStepChunks) : 0u;
            if (cnt) {
                // S[:, 0 .. 64 cnt) = Q K^T: the softmax threads must have pulled the previous scores out of tensor
                // memory, and the K blocks must have landed
                const unsigned ring_i = grp_n == 0u ? 0u : 2u * grp_n - 1u;
                const unsigned g = ring_i % kRingGroups, ph = (ring_i / kRingGroups) & 1u;
                // the blocks of a group are adjacent: their 64 cnt rows form one K-major operand
                const unsigned long long k_desc = smem_desc_sw128(ring_base + g * kGroupBytes);
                const unsigned idesc = kIdescQK64 + ((cnt - 1u) << 20);                    // N = 64 cnt
                if (!wait2(&sc->s_free, (grp_n - 1u) & 1u, grp_n > 0u, 25, &sc->full[g], ph, 20)) break;
                tc_fence_after();
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)  // 16 head dims (32 bytes inside the swizzled row) per MMA
                    mma_ss(sr.tmem + kColS, q_desc + (unsigned long long)(kk * 2), k_desc + (unsigned long long)(kk * 2), idesc, kk > 0);
                tc_commit(&sc->s_full);
                tc_commit(&sc->empty[g]);
                ++grp_n;
            }
            if (pend_cnt) {
                // O (+)= sum_j P_j V_j with the V blocks of the pending step
                const unsigned ring_i = 2u * pv_n + 2u;
                const unsigned g = ring_i % kRingGroups, ph = (ring_i / kRingGroups) & 1u;
                const unsigned long long v_desc = smem_desc_sw128(ring_base + g * kGroupBytes);
                const unsigned acc0 = pend_fresh ? 0u : 1u, two = pend_cnt > 1u ? 1u : 0u;
                // the epilogue must have taken the previous tile's accumulator before this tile's first P V overwrites it
                if (pend_fresh && tile_n > 0 && !mbar_wait(&sc->o_free, (tile_n - 1) & 1u, abort_flag)) { fail = 27; break; }
                if (!wait2(&sc->p_full, pv_n & 1u, true, 22, &sc->full[g], ph, 21)) break;
                tc_fence_after();
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)  // 16 keys per MMA: 8 packed columns of P_j, two 8-row groups of V_j
                    mma_ts(sr.tmem + kColO, sr.tmem + kColP + kk * 8, v_desc + (unsigned long long)((kk * 2048) >> 4), kIdescPV, kk > 0 ? 1u : acc0);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    mma_ts_if(sr.tmem + kColO, sr.tmem + kColP + 32 + kk * 8, v_desc + (unsigned long long)((kTileBytes + kk * 2048) >> 4), kIdescPV, 1u, two);
                tc_commit(&sc->pv_done);
                tc_commit_if(&sc->o_done, pend_last ? 1u : 0u);
                tc_commit(&sc->empty[g]);
                tile_n += pend_last ? 1u : 0u;
                ++pv_n;
            }
            pend_cnt = cnt;
            pend_fresh = tile_fresh;
            pend_last = false;
            tile_fresh = tile_fresh && cnt == 0u;
            tile_steps = tile_steps || cnt != 0u;
        }
        if (fail) break;
        if (last) {
            tc_commit(&sc->q_empty[qs]);        // every Q K^T of the tile has been issued
            // the tile's last P V is the pending one (the tile's last segment may be empty); a tile without any step (a part
            // of a split tile whose keys are all padding) leaves the mark of the tile before it alone
            pend_last = pend_last || tile_steps;
        }
        mbar_arrive(&sc->sched_empty[ss]);
        ++sched_n;
        if (w < 0) break;
    }
    if (fail) give_up(abort_flag, p.status, fail);
}

// ------------------------------------------------------------------------------------------------ softmax (one warpgroup per stream, one thread per row)
__device__ __forceinline__ void softmax_role(const KernelParams& p, SmemCtl* ctl, const StreamRef& sr, int warp, int lane) {
    StreamCtl* sc = sr.sc;
    int* abort_flag = &ctl->abort_flag;
    const int quad = warp & 3;                      // tensor-memory lanes this warp may touch: 32*quad .. +31
    const int row = quad * 32 + lane;               // row of the 128-row tile
    const bool lower = row >= kBlock;
    const int my_who = lower ? kLowerHalf : kUpperHalf;
    const unsigned lane_addr = sr.tmem + ((unsigned)(quad * 32) << 16);
    const float sl2 = p.scale_log2;
    unsigned sched_n = 0, grp_n = 0, msg_n = 0;
    bool ok = true;
    int fail = 0;                                   // code of the wait that was abandoned, if any
    float m_ref = -INFINITY, l_sum = 0.f;
    bool o_dirty = false;                           // has any P V been issued for this tile yet
    // exponentials of the 64 scores of one key block, packed in place: afterwards s[0..31] hold the bit
    // patterns of the 32 words of bf16 probability pairs (four partial sums, so that the adds do not form one chain)
    auto exp_pack = [&](float* s, float neg_m, float& sum0, float& sum1) {
        float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            float x0, x1, p0, p1;
            ffma2(x0, x1, s[2 * j], s[2 * j + 1], sl2, neg_m);
            p0 = ex2(x0);
            p1 = ex2(x1);
            if (j & 1) fadd2(b0, b1, p0, p1);
            else fadd2(a0, a1, p0, p1);
            s[j] = __uint_as_float(pack_bf16(p0, p1));
        }
        fadd2(a0, a1, b0, b1);
        fadd2(sum0, sum1, a0, a1);
    };
    while (ok) {
        const unsigned ss = sched_n % kSchedSlots, sp = (sched_n / kSchedSlots) & 1u;
        if (!mbar_wait(&sc->sched_full[ss], sp, abort_flag)) { fail = 30; break; }
        __syncwarp();
        const WorkSlot* slot = &sc->slot[ss];
        const int w = slot->w, flags = slot->flags, n = slot->n_chunks;
        if (w < 0) {                                // tell the epilogue that this stream is finished
            // (The entry reused here holds the message of the last tile but one.  That one has been read once the last tile's P V has
            // been issued, since its first product waits for the accumulator before.  Waiting for the epilogue to take the last tile
            // would not do: if that tile has one step, the last but one may still be in the accumulator, and its phase of o_free has the
            // other parity, so that the wait passes at once.)
            if (msg_n > 0 && !mbar_wait(&sc->pv_done, (grp_n - 1) & 1u, abort_flag)) { fail = 36; break; }
            EpiMsg* msg = &sc->epi[msg_n & 1u];
            if (row == 0) msg->kind = kEpiDone;
            mbar_arrive(&sc->epi_full[msg_n & 1u]);
            break;
        }
        if (flags & kSegFirst) {
            m_ref = -INFINITY;
            l_sum = 0.f;
            o_dirty = false;
        }
        for (int i = 0; i < n && ok; i += kStepChunks) {
            const ChunkEntry* e = &slot->chunks[i];
            const int cnt = min(kStepChunks, n - i);
            // which of the step's key blocks my half of the tile attends (warp-uniform)
            const int who0 = e[0].who, who1 = cnt > 1 ? e[1].who : kNoChunk;
            const bool mine0 = (who0 & kWhoMask) == kBothHalves || (who0 & kWhoMask) == my_who;
            const bool mine1 = (who1 & kWhoMask) == kBothHalves || (who1 & kWhoMask) == my_who;
            ok = mbar_wait(&sc->s_full, grp_n & 1u, abort_flag);
            if (!ok) { fail = 31; break; }
            __syncwarp();                           // lanes leave the wait one by one: back in step before the warp-wide loads
            tc_fence_after();
            // A key block with padded keys (rare: the one holding a sequence's end) gets -inf written over their
            // scores in tensor memory first, so that the common path below carries no masking code at all.
            if (__builtin_expect(((who0 | who1) & kHasPadding) != 0, 0)) {
#pragma unroll 1
                for (int c = 0; c < cnt; ++c)
                    if ((c == 0 ? mine0 : mine1) && (e[c].who & kHasPadding)) mask_scores(lane_addr + kColS + 64 * c, e[c].kb);
            }
            float s[128];
            if (mine0) tmem_ld64(lane_addr + kColS, s);
            if (mine1) tmem_ld64(lane_addr + kColS + 64, s + 64);
            tmem_wait_ld();
            // the score columns are free again: the next step's Q K^T may overwrite them
            tc_fence_before();
            mbar_arrive(&sc->s_free);
            float alpha = 1.f;
            bool rescale = false;
            if (mine0 || mine1) {
                float m_loc = -INFINITY;
                if (mine0) m_loc = row_max64(s);
                if (mine1) m_loc = fmaxf(m_loc, row_max64(s + 64));
                const float m_cand = m_loc * sl2;
                const bool need = m_cand > m_ref + kRescaleThreshold;        // true on the first step (m_ref = -inf)
                rescale = __any_sync(0xffffffffu, need);
                if (need) {
                    alpha = ex2(m_ref - m_cand);
                    m_ref = m_cand;
                }
            }
            // probabilities into registers first: the previous step's P V has this long to finish
            float sum0 = 0.f, sum1 = 0.f;
            const float neg_m = -m_ref;
            if (mine0) exp_pack(s, neg_m, sum0, sum1);
            if (mine1) exp_pack(s + 64, neg_m, sum0, sum1);
            // the previous step's P V must be complete before its probabilities are overwritten or O is touched
            if (grp_n > 0) {
                ok = mbar_wait(&sc->pv_done, (grp_n - 1) & 1u, abort_flag);
                if (!ok) { fail = 32; break; }
                __syncwarp();
                tc_fence_after();
            }
            if (__builtin_expect(rescale && o_dirty, 0)) rescale_accumulator(lane_addr + kColO, alpha);
            if (mine0) tmem_st32(lane_addr + kColP, reinterpret_cast<unsigned*>(s));
            else tmem_st32_zero(lane_addr + kColP);
            if (cnt > 1) {
                if (mine1) tmem_st32(lane_addr + kColP + 32, reinterpret_cast<unsigned*>(s + 64));
                else tmem_st32_zero(lane_addr + kColP + 32);
            }
            if (!ok) break;
            l_sum = l_sum * alpha + (sum0 + sum1);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(&sc->p_full);
            ++grp_n;
            o_dirty = true;
        }
        if (!ok) break;
        if (flags & kSegLast) {
            // -------------------------------------------------------- end of the tile: lse now, the output rows via the epilogue
            const int my_q = lower ? slot->qb : slot->qa;
            const unsigned long long qbits = lower ? slot->qbits_b : slot->qbits_a;
            const bool have = o_dirty;
            const int part_slot = slot->part_slot;
            const int r64 = row & (kBlock - 1);
            float inv = 0.f;
            if (part_slot >= 0) {
                // one part of a split tile: (max, sum) from here, the raw accumulator from the epilogue
                float* part = p.partials + (size_t)part_slot * kPartialFloats;
                part[128 * 64 + row] = have ? m_ref : -INFINITY;
                part[128 * 64 + 128 + row] = have ? l_sum : 0.f;
            } else if (my_q >= 0) {                 // warp-uniform
                const bool token = (qbits >> r64) & 1ull, good = have && token && l_sum > 0.f;
                const size_t tok = ((size_t)slot->bh * p.nb + my_q) * kBlock + r64;
                if (p.lse) p.lse[tok] = good ? (m_ref + __log2f(l_sum)) * 0.6931471805599453f : -INFINITY;
                inv = good ? __frcp_rn(l_sum) : (token ? 0.f : -1.f);
                // (a tile that is no part has a step: one of its rows is a token, and a block is in its own window)
            }
            if (have) {                             // CTA-uniform per stream: every thread of the warpgroup posts
                EpiMsg* msg = &sc->epi[msg_n & 1u];
                msg->inv[row] = inv;
                if (row == 0) {
                    msg->kind = kEpiTile;
                    msg->bh = slot->bh;
                    msg->qa = slot->qa;
                    msg->qb = slot->qb;
                    msg->part_slot = part_slot;
                }
                mbar_arrive(&sc->epi_full[msg_n & 1u]);      // (release: the message is visible to whoever sees the phase complete)
                ++msg_n;
            }
        }
        tc_fence_before();
        mbar_arrive(&sc->sched_empty[ss]);
        ++sched_n;
    }
    if (fail) give_up(abort_flag, p.status, fail);
}

// ------------------------------------------------------------------------------------------------ epilogue (one warpgroup, both streams)
// Each warp serves its 32 rows of whichever stream has a finished tile: accumulator out of tensor memory,
// scaled by 1/l, to the output rows (or raw, to the scratch of a split tile's part).
__device__ __forceinline__ void epilogue_role(const KernelParams& p, SmemCtl* ctl, unsigned char* smem, unsigned tmem, int warp, int lane) {
    int* abort_flag = &ctl->abort_flag;
    const int quad = warp & 3;
    const int row = quad * 32 + lane;
    const int r64 = row & (kBlock - 1);
    const bool lower = row >= kBlock;
    // per stream, packed so that the loop below is one copy of the code: bits 0..15 messages taken, 16..30 tiles
    // taken (only parities are used), bit 31 the stream is finished
    unsigned state0 = 0u, state1 = 0u;              // (scalars: an indexed array would live in local memory)
    IdleClock idle;
    while (!((state0 & state1) >> 31)) {
        bool progress = false;
#pragma unroll 1
        for (int s = 0; s < kStreams; ++s) {
            const unsigned st = s == 0 ? state0 : state1;
            if (st >> 31) continue;
            StreamCtl* sc = &ctl->st[s];
            const unsigned msg_n = st & 0xffffu, tile_n = (st >> 16) & 0x7fffu;
            const unsigned e = msg_n & 1u, eph = (msg_n >> 1) & 1u;
            if (!__all_sync(0xffffffffu, mbar_test(&sc->epi_full[e], eph))) continue;
            const EpiMsg* msg = &sc->epi[e];
            // (The accumulator is waited for by one suspended try, which ends with it or after a microsecond or two, and not until it is
            // there: a tile's last P V is issued when the stream's next item is there, and for that the scheduler may have to wait until
            // this warp has served the other stream.  With a test and the sleep below instead of the try the last tile was late:
            // [3, 16, 512] 15.9 us against 15.4.)
            if (msg->kind != kEpiDone && !__all_sync(0xffffffffu, mbar_test(&sc->o_done, tile_n & 1u) || mbar_try(&sc->o_done, tile_n & 1u))) continue;
            progress = true;
            const unsigned st_next = msg->kind == kEpiDone ? (st | 0x80000000u) : (((msg_n + 1u) & 0xffffu) | (((tile_n + 1u) & 0x7fffu) << 16));
            if (s == 0) state0 = st_next; else state1 = st_next;
            if (st_next >> 31) continue;
            const int bh = msg->bh, my_q = lower ? msg->qb : msg->qa, part_slot = msg->part_slot;
            const float inv = msg->inv[row];
            __syncwarp();
            tc_fence_after();
            const unsigned lane_addr = tmem + s * kStreamCols + ((unsigned)(quad * 32) << 16);
            // the row's destination: the output tensor, or (raw fp32) the scratch of a split tile's part
            const bool partial = part_slot >= 0;
            unsigned char* dst = partial ? reinterpret_cast<unsigned char*>(p.partials + (size_t)part_slot * kPartialFloats + row * 64)
                                         : reinterpret_cast<unsigned char*>(p.out + (((size_t)bh * p.nb + (my_q >= 0 ? my_q : 0)) * kBlock + r64) * kBlock);
            bool write = partial || my_q >= 0;              // warp-uniform
            if (!BB_CHECK(bh >= 0 && bh < p.BH && my_q < p.nb && part_slot < p.BH * max(p.global_tiles, 1) * p.parts, 74)) write = false;
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                float o[32];
                tmem_ld32(lane_addr + kColO + c * 32, o);
                tmem_wait_ld();
                if (c == 1) { tc_fence_before(); mbar_arrive(&sc->o_free); }       // the accumulator has been taken
                if (!write) continue;
                if (partial) {
                    float4* d4 = reinterpret_cast<float4*>(dst) + 8 * c;
#pragma unroll
                    for (int j = 0; j < 8; ++j) d4[j] = make_float4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
                } else {
                    // (a select for padded rows: what stands in them may be anything, and with it their sums)
                    const bool token = inv >= 0.f;
                    uint4* d4 = reinterpret_cast<uint4*>(dst) + 4 * c;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint4 v;
                        v.x = token ? pack_bf16(o[8 * j + 0] * inv, o[8 * j + 1] * inv) : 0u;
                        v.y = token ? pack_bf16(o[8 * j + 2] * inv, o[8 * j + 3] * inv) : 0u;
                        v.z = token ? pack_bf16(o[8 * j + 4] * inv, o[8 * j + 5] * inv) : 0u;
                        v.w = token ? pack_bf16(o[8 * j + 6] * inv, o[8 * j + 7] * inv) : 0u;
                        d4[j] = v;
                    }
                }
            }
        }
        if (progress) idle.reset();
        else {
            // (a short sleep, not a suspended wait on one stream's barrier: that would not see the other stream's
            // message for up to 4 us, and the stream's next tile cannot overwrite the accumulator before it is taken)
            __nanosleep(400);
            if (!__all_sync(0xffffffffu, idle.tick(abort_flag, p.status, 41, 0))) return;
        }
    }
}

// ------------------------------------------------------------------------------------------------ the kernel
__global__ void __launch_bounds__(kThreads, 1)
attn_fwd_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                      const __grid_constant__ CUtensorMap tm_v, const KernelParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + kSmemCtl);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;      // (uniform, and known to be)

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStreams; ++s) {
            StreamCtl* sc = &ctl->st[s];
            for (int i = 0; i < kRingGroups; ++i) { mbar_init(&sc->full[i], 1); mbar_init(&sc->empty[i], 1); }
            for (int i = 0; i < 2; ++i) { mbar_init(&sc->q_full[i], 1); mbar_init(&sc->q_empty[i], 1); mbar_init(&sc->epi_full[i], kSoftmaxThreads); }
            mbar_init(&sc->s_full, 1);
            mbar_init(&sc->s_free, kSoftmaxThreads);    // every softmax thread arrives itself: converging the warp and
            mbar_init(&sc->p_full, kSoftmaxThreads);    // electing a lane was measured 10% slower on the whole kernel
            mbar_init(&sc->pv_done, 1);
            mbar_init(&sc->o_done, 1);
            mbar_init(&sc->o_free, kSoftmaxThreads);    // the 128 epilogue threads
            for (int i = 0; i < kSchedSlots; ++i) { mbar_init(&sc->sched_full[i], 1); mbar_init(&sc->sched_empty[i], 3 + kSoftmaxThreads); }    // two producer lanes, the MMA thread, the softmax threads
        }
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kWarpProducer) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_release();
    grid_dependency_wait();
    const unsigned tmem = *(volatile unsigned*)&ctl->tmem_base;
    const StreamRef s0{&ctl->st[0], smem, tmem};
    const StreamRef s1{&ctl->st[1], smem + kStreamSmemBytes, tmem + kStreamCols};

    if (warp < kWarpEpilogue) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
        softmax_role(p, ctl, warp < 4 ? s0 : s1, warp, lane);
    } else if (warp < kWarpProducer) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsEpilogue));
        epilogue_role(p, ctl, smem, tmem, warp, lane);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLight));
        if (warp == kWarpScheduler) scheduler_role(p, ctl, lane);
        else if (warp == kWarpProducer) { if (lane < 2 * kStreams) producer_role(p, ctl, (lane & 1) ? s1 : s0, lane >= kStreams, &tm_q, &tm_k, &tm_v); }
        else if (elect_one()) mma_role(p, ctl, warp == kWarpMma ? s0 : s1);
    }

    // ------------------------------------------------------------------------------------------------ teardown
    __syncthreads();
    if (*(volatile int*)&ctl->abort_flag) {
        // a wait expired: give copies and MMAs still in flight time to land before shared and tensor memory go away
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    tc_fence_after();
    if (warp == kWarpProducer) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0) {
        // the last CTA to finish re-arms the work counter for the next launch
        __threadfence();
        const int done = atomicAdd(&p.counter[1], 1);
        if (done == (int)gridDim.x - 1) {
            p.counter[0] = 0;
            p.counter[1] = 0;
            __threadfence();
        }
    }
}

// Adds up the parts of the split tiles, in a fixed order: results do not depend on scheduling.  One CTA per (batch*head, split
// tile, group of 16 rows); 16 threads share a row, each owning 4 of its 64 output columns.
__global__ void __launch_bounds__(256)
merge_split_tiles_kernel(const float* __restrict__ partials, const Item* __restrict__ items, const unsigned long long* __restrict__ kbits,
                         __nv_bfloat16* __restrict__ out, float* __restrict__ lse, int H, int nb, int items_per_head, int tiles_per_head,
                         int nparts) {
    grid_dependency_release();
    const int rgrp = blockIdx.x & 7, tile = (blockIdx.x >> 3) % tiles_per_head, bh = (blockIdx.x >> 3) / tiles_per_head;
    const int row = rgrp * 16 + (threadIdx.x >> 4), c4 = threadIdx.x & 15, r64 = row & (kBlock - 1);
    const Item& item = items[(size_t)(bh % H) * items_per_head + tile];
    const int q = row >= kBlock ? item.qb : item.qa;
    grid_dependency_wait();
    if (q < 0) return;
    const unsigned long long qb = kbits ? kbits[(size_t)(bh / H) * nb + q] : ~0ull;
    const float* base = partials + (size_t)(bh * tiles_per_head + tile) * nparts * kPartialFloats;
    const float* stats = base + 128 * 64 + row;
    float m = -INFINITY, l = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p0 = 0; p0 < nparts; p0 += 8) {         // eight parts at a time, all of their loads in flight together
        float mp[8], lp[8], mx = m;
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const size_t off = (size_t)min(p0 + u, nparts - 1) * kPartialFloats;
            mp[u] = stats[off];
            lp[u] = p0 + u < nparts ? stats[off + 128] : 0.f;
            v[u] = reinterpret_cast<const float4*>(base + off)[row * 16 + c4];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = fmaxf(mx, lp[u] > 0.f ? mp[u] : -INFINITY);
        if (mx == -INFINITY) continue;
        const float scale = exp2f(m - mx);           // 0 on the first parts that have anything
        m = mx;
        l *= scale;
        acc.x *= scale; acc.y *= scale; acc.z *= scale; acc.w *= scale;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (!(lp[u] > 0.f)) continue;            // (such a part has left no accumulator)
            const float wgt = exp2f(mp[u] - mx);
            l += wgt * lp[u];
            acc.x += wgt * v[u].x; acc.y += wgt * v[u].y; acc.z += wgt * v[u].z; acc.w += wgt * v[u].w;
        }
    }
    const bool token = (qb >> r64) & 1ull, good = token && l > 0.f;
    const float inv = good ? 1.f / l : 0.f;
    const size_t tok = ((size_t)bh * nb + q) * kBlock + r64;
    reinterpret_cast<uint2*>(out + tok * kBlock)[c4] = token ? make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv))
                                                             : make_uint2(0u, 0u);
    if (lse && c4 == 0) lse[tok] = good ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
}

// Self-test of the bounded wait: one thread waits on an mbarrier that nothing ever arrives on, with the same
// helper and the same limit as the attention kernel; the wait gives up, records BIGBIRD_ETIMEOUT and the kernel
// returns normally.
__global__ void wait_expiry_selftest_kernel(int* status) {
    __shared__ unsigned long long bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!mbar_wait(&bar, 0u, &abort_flag)) give_up(&abort_flag, status, 99);
    }
}

// One 64-bit word per (batch, key block): bit t = key_padding_mask[batch, block*64 + t] != 0; and n_zero words to be cleared.
__global__ void __launch_bounds__(256) pack_mask_kernel(const uint8_t* __restrict__ kpm, unsigned long long* __restrict__ kbits, int n_words, int* __restrict__ zero,
                                                        int n_zero) {
    grid_dependency_release();
    grid_dependency_wait();
    if (blockIdx.x == 0 && (int)threadIdx.x < n_zero) zero[threadIdx.x] = 0;
    const int word = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (word >= n_words) return;
    const uint8_t* src = kpm + (size_t)word * kBlock;
    const unsigned lo = __ballot_sync(0xffffffffu, src[lane] != 0);
    const unsigned hi = __ballot_sync(0xffffffffu, src[lane + 32] != 0);
    if (lane == 0) kbits[word] = ((unsigned long long)hi << 32) | lo;
}

// ------------------------------------------------------------------------------------------------ host side
}  // namespace

cudaError_t launch_wait_expiry_selftest(DeviceScratch& sc, cudaStream_t stream) {
    wait_expiry_selftest_kernel<<<1, 32, 0, stream>>>(sc.status);
    return cudaGetLastError();
}

namespace {

// Per device, once, with that device current: the kernel's shared-memory attribute (a per-device property of the
// function) and the device's SM count.
struct KernelDevice {
    bool ready = false;
    int sm_count = 0;
};
constexpr int kMaxKernelDevices = 64;
std::mutex g_kernel_mu, g_launch_mu;
KernelDevice g_kernel_dev[kMaxKernelDevices];

cudaError_t kernel_setup(int device, int* sm_count) {
    if (device < 0 || device >= kMaxKernelDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_kernel_mu);
    KernelDevice& d = g_kernel_dev[device];
    if (!d.ready) {
        cudaError_t e = cudaFuncSetAttribute(attn_fwd_sm100_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return e;
        d.ready = true;
    }
    *sm_count = d.sm_count;
    return cudaSuccess;
}

// How a launch cuts the tiles of global blocks: their lists are as long as the sequence, the other tiles' a dozen blocks, so that
// they outlast everything else unless the GPU has a lot to do.  As many parts as there are three quarters of what each stream gets
// altogether in a list, or lengths of another tile if that is longer, rounded up: a part is at least two thirds as long.  Measured, uncut (or in parts of 32) -> cut like this: one sequence of 3001 tokens in 4096,
// 12 heads 60 -> 42 us (the chain of a global tile was 50 of them); [2, 12, 1024] stays uncut.
struct Cut {
    int parts, part_steps;
};
Cut cut_global_tiles(const bigbird_layout& L, int B, int sms, int max_parts) {
    if (L.global_tiles == 0) return Cut{1, L.nb};
    const int64_t per_stream = (int64_t)B * (int64_t)L.steps.size() / (kStreams * sms);
    const int64_t sparse = L.sparse_tiles_per_head
        ? ((int64_t)L.steps.size() - (int64_t)L.H * L.global_tiles * L.nb) / ((int64_t)L.H * L.sparse_tiles_per_head) : 0;
    const int64_t want = std::max<int64_t>({8, sparse, per_stream * 3 / 4});
    if (L.nb < 2 * want) return Cut{1, L.nb};           // (adding up the parts costs as much as what is left to gain)
    int parts = (int)std::min<int64_t>((L.nb + want - 1) / want, std::max(1, max_parts));
    const int part_steps = ((L.nb + parts - 1) / parts + kStepChunks - 1) / kStepChunks * kStepChunks;
    parts = (L.nb + part_steps - 1) / part_steps;
    return Cut{parts, part_steps};
}

void set_shape(KernelParams& p, const bigbird_layout& L, int B, Cut cut, float scale, int sm_count) {
    p.items_per_head = L.items_per_head;
    p.global_tiles = L.global_tiles;
    p.parts = cut.parts;
    p.part_steps = cut.part_steps;
    p.BH = B * L.H;
    p.H = L.H;
    p.nb = L.nb;
    p.total_work = p.BH * (L.global_tiles * cut.parts + L.sparse_tiles_per_head);
    // Tiles that a stream has in hand are not drawn by another one that runs dry, so with few tiles in all it should have few: [1, 12,
    // 16384] with 13000 tokens (5 tiles per stream) 75 us with three, 69 with two; [16, 16, 4096] ragged (28, many of them without a
    // token) 204 and 210; [8, 12, 4096] (10) 125 with either.  A tile with a list of five key blocks or less, though, is over before the
    // scheduler has another, so there only fewer than four count as few: [4, 12, 4096] (5.2 tiles per stream) with lists of three 43.9
    // us with three, 45.8 with two, but with lists of eight 71.8 and 67.0; [4, 16, 2048] (3.5) with lists of five 44.1 and 40.5.
    const int64_t lists = (int64_t)L.steps.size() - (int64_t)L.H * L.global_tiles * L.nb, tiles = (int64_t)L.H * L.sparse_tiles_per_head;
    p.ahead = p.total_work < (2 * lists > 11 * tiles ? 8 : 4) * kStreams * sm_count ? 2 : kSchedSlots;
    p.scale_log2 = scale * 1.4426950408889634f;
}

// One CTA per SM, each running kStreams tile streams; every SM gets work before any stream gets its second tile.
int grid_size(int sm_count, int total_work) { return std::max(1, std::min(sm_count, total_work)); }

// The work counter of the calls on one stream, or null.  Calls on one stream take turns and the last CTA of each leaves the pair at
// zero, so they can share one that the library keeps; calls on different streams cannot, and neither can a captured call, which
// runs on whatever stream its graph is launched on: those count in their own workspace, and a kernel has to zero it first.  (A call
// with a mask always does: the kernel that packs the mask is there anyway.)  No stream gets an id that another one has had.  Under
// the lock.
int* stream_counter(DeviceScratch& sc, cudaStream_t stream) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) return nullptr;
    if (cudaStreamGetId(stream, &id) != cudaSuccess) return nullptr;
    int i = 0;
    while (i < sc.streams && sc.stream_ids[i] != id) ++i;
    if (i == kCounterSlots) return nullptr;
    if (i == sc.streams) sc.stream_ids[sc.streams++] = id;
    return sc.counters + 2 * i;
}

// The kernels of a call, in the order of the stream, each allowed to begin before the one in front of it has drained: they wait for
// it (grid_dependency_wait) before they touch memory that it may use.
cudaError_t enqueue(const KernelParams& p, const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                    const uint8_t* kpm, unsigned long long* kbits, int n_words, int* zero, int n_zero, int sm_count, cudaStream_t stream, int* launches) {
    cudaError_t e = cudaSuccess;
    if (n_words || n_zero) {
        e = launch_chained(pack_mask_kernel, (unsigned)std::max(1, (n_words * 32 + 255) / 256), 256, 0, stream, kpm, kbits, n_words, zero, n_zero);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    e = launch_chained(attn_fwd_sm100_kernel, (unsigned)grid_size(sm_count, p.total_work), kThreads, kSmemBytes, stream, tm_q, tm_k, tm_v, p);
    if (e != cudaSuccess) return e;
    ++*launches;
    if (p.parts > 1) {
        e = launch_chained(merge_split_tiles_kernel, (unsigned)(p.BH * p.global_tiles * 8), 256, 0, stream, (const float*)p.partials, p.items, p.kbits, p.out, p.lse,
                           p.H, p.nb, p.items_per_head, p.global_tiles, p.parts);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

}  // namespace

int launch_attn_fwd_sm100(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, DeviceScratch& sc, cudaMemPool_t pool,
                          int* launches, cudaError_t* cuda_err) {
    *cuda_err = cudaSuccess;
    if (!(a.scale > 0.f) || !(a.scale < INFINITY)) return BIGBIRD_EINVAL;
    const int64_t rows = (int64_t)a.B * a.H * a.N;
    if (rows >= (1ll << 31) || (int64_t)a.B * a.H * L.items_per_head >= (1ll << 31)) return BIGBIRD_EUNSUPPORTED;

    int device = 0, sm_count = 0;
    cudaError_t de = cudaGetDevice(&device);
    if (de == cudaSuccess) de = kernel_setup(device, &sm_count);
    if (de != cudaSuccess) { *cuda_err = de; return BIGBIRD_ECUDA; }

    CUtensorMap tm_q, tm_k, tm_v;
    if (!make_map(&tm_q, a.q, (uint64_t)rows) || !make_map(&tm_k, a.k, (uint64_t)rows) || !make_map(&tm_v, a.v, (uint64_t)rows)) {
        *cuda_err = cudaErrorInvalidValue;
        return BIGBIRD_ECUDA;
    }

    // scratch of this call, on the caller's stream: parts of split tiles, packed mask bits, work counter (where the kernel that packs
    // the mask can zero it)
    int* counter = nullptr;
    if (!a.kpm) {
        std::lock_guard<std::mutex> lock(g_launch_mu);
        counter = stream_counter(sc, a.stream);
    }
    const int own_counter = counter ? 0 : 2;
    const Cut cut = cut_global_tiles(L, a.B, sm_count, 1 << 20);
    const size_t words = a.kpm ? (size_t)a.B * a.nb : 0;
    const size_t off_bits = cut.parts > 1 ? (size_t)a.B * a.H * L.global_tiles * cut.parts * kPartialFloats * sizeof(float) : 0;
    unsigned char* ws = nullptr;
    const size_t off_counter = off_bits + words * sizeof(unsigned long long), bytes = off_counter + own_counter * sizeof(int);
    if (bytes) {
        cudaError_t e = cudaMallocFromPoolAsync((void**)&ws, bytes, pool, a.stream);
        if (e != cudaSuccess) { *cuda_err = e; return BIGBIRD_ECUDA; }
    }

    KernelParams p{};
    p.out = (__nv_bfloat16*)a.out;
    p.lse = a.lse;
    p.kbits = words ? (const unsigned long long*)(ws + off_bits) : nullptr;
    p.partials = (float*)ws;
    p.items = dl.items;
    p.steps = dl.steps;
    p.counter = counter ? counter : (int*)(ws + off_counter);
    p.status = sc.status;
    set_shape(p, L, a.B, cut, a.scale, sm_count);

    cudaError_t e = enqueue(p, tm_q, tm_k, tm_v, a.kpm, (unsigned long long*)(ws + off_bits), (int)words, p.counter, own_counter, sm_count, a.stream, launches);
    if (ws) {
        const cudaError_t ef = cudaFreeAsync(ws, a.stream);
        if (e == cudaSuccess) e = ef;
    }
    *cuda_err = e;
    return e == cudaSuccess ? BIGBIRD_OK : BIGBIRD_ECUDA;
}

}  // namespace bigbird

// ------------------------------------------------------------------------------------------------ no-allocation entry point
// bigbird_attn_fwd_static: the tensor-core forward for callers that must not allocate device memory (see
// include/bigbird.h).  Everything bigbird_attn_fwd keeps in cudaMalloc'ed library scratch lives here in one
// fixed array that is part of the loaded module: status and work-counter words, the packed key-padding bits,
// and the device copy of the layout's tile schedule, which is sent again whenever another layout is used.
namespace bigbird {
namespace {

constexpr size_t kStaticMaskWords = 16384;      // B * N/b
constexpr size_t kStaticItems = 8192;           // H * tiles per head
constexpr size_t kStaticSteps = 131072;         // (key block, halves) entries summed over heads
constexpr size_t kStaticParts = 128;            // parts of split global tiles (more tiles than fit stay whole)
// N/b: the tiles of global blocks of longer sequences outlast everything else if they are not cut, however little room is left for
// parts, and the allocating entry point cuts them as finely as it pays.
constexpr int kStaticBlocks = 96;
constexpr size_t kStaticOffMask = 256;          // bytes 0..15: status[2], counter[2]
constexpr size_t kStaticOffItems = kStaticOffMask + kStaticMaskWords * sizeof(unsigned long long);
constexpr size_t kStaticOffSteps = kStaticOffItems + kStaticItems * sizeof(Item);
constexpr size_t kStaticOffParts = kStaticOffSteps + kStaticSteps * sizeof(Step);
constexpr size_t kStaticBytes = kStaticOffParts + kStaticParts * kPartialFloats * sizeof(float);     // about 5.8 MB per GPU

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

struct StaticDevice {
    unsigned char* base = nullptr;              // device address of g_static_scratch on this device
    int sm_count = 0;
    uint64_t schedule_uid = 0;                  // layout whose schedule the array holds (0: none)
    bool graphs_send = false;                   // a captured call sends a schedule: the array may hold that one at any time from then on
};
std::mutex g_static_mu;
StaticDevice g_static_dev[64];

// Once per device, with that device current: the device address of the array (its name is only a host-side
// stand-in in host code) and the kernel's shared-memory attribute.
cudaError_t static_setup(int device, StaticDevice* out) {
    std::lock_guard<std::mutex> lock(g_static_mu);
    StaticDevice& d = g_static_dev[device];
    if (!d.base) {
        void* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess) return e;
        int sms = 0;
        e = kernel_setup(device, &sms);
        if (e != cudaSuccess) return e;
        d.sm_count = sms;
        d.base = (unsigned char*)ptr;
    }
    *out = d;
    return cudaSuccess;
}

void static_remember_schedule(int device, uint64_t uid, bool captured = false) {
    std::lock_guard<std::mutex> lock(g_static_mu);
    g_static_dev[device].schedule_uid = uid;
    if (captured) g_static_dev[device].graphs_send = true;
}

}  // namespace
}  // namespace bigbird

extern "C" int bigbird_attn_fwd_static(const void* q, const void* k, const void* v, const bigbird_layout* L,
                                       const uint8_t* key_padding_mask, void* out, float* lse, int B, int H, int64_t N,
                                       int D, int b, float scale, int dtype, void* stream_) {
    using namespace bigbird;
    if (!q || !k || !v || !L || !out) return BIGBIRD_EINVAL;
    if (B < 1 || H < 1 || N < 1 || D < 1 || b < 1) return BIGBIRD_EINVAL;
    if (L->N != N || L->b != b || L->H != H) return BIGBIRD_EINVAL;
    if (dtype != BIGBIRD_BF16 || D != 64 || b != 64) return BIGBIRD_EUNSUPPORTED;
    if ((((uintptr_t)q) | ((uintptr_t)k) | ((uintptr_t)v) | ((uintptr_t)out)) & 15) return BIGBIRD_EINVAL;
    if (!(scale > 0.f) || !(scale < INFINITY)) return BIGBIRD_EINVAL;
    const int64_t rows = (int64_t)B * H * N;
    if (rows >= (1ll << 31) || (int64_t)B * H * L->items_per_head >= (1ll << 31)) return BIGBIRD_EUNSUPPORTED;
    // the fixed scratch bounds the problem
    const size_t words = (size_t)B * L->nb, n_items = L->items.size(), n_steps = L->steps.size();
    if (words > kStaticMaskWords || n_items > kStaticItems || n_steps > kStaticSteps) return BIGBIRD_ELIMIT;
    if (L->nb > kStaticBlocks) return BIGBIRD_ELIMIT;

    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return BIGBIRD_ECUDA;
    if (device < 0 || device >= 64) return BIGBIRD_EUNSUPPORTED;
    StaticDevice sd;
    if (static_setup(device, &sd) != cudaSuccess) return BIGBIRD_ECUDA;
    cudaStream_t stream = (cudaStream_t)stream_;
    int* words4 = reinterpret_cast<int*>(sd.base);
    unsigned long long* kbits_dev = reinterpret_cast<unsigned long long*>(sd.base + kStaticOffMask);
    Item* items_dev = reinterpret_cast<Item*>(sd.base + kStaticOffItems);
    Step* steps_dev = reinterpret_cast<Step*>(sd.base + kStaticOffSteps);

    CUtensorMap tm_q, tm_k, tm_v;
    if (!make_map(&tm_q, q, (uint64_t)rows) || !make_map(&tm_k, k, (uint64_t)rows) || !make_map(&tm_v, v, (uint64_t)rows))
        return BIGBIRD_ECUDA;

    // The array keeps what the last call left: status and work counter must start at zero, and the schedule of
    // this call's layout replaces the previous one (step offsets made absolute, as the kernel expects).
    if (!key_padding_mask) {                    // (else the kernel that packs the mask does it)
        e = cudaMemsetAsync(words4, 0, 16, stream);
        if (e != cudaSuccess) return BIGBIRD_ECUDA;
    }
    // The schedule is sent only when the array does not hold this layout's already (copies from the handle's own
    // host arrays, which live as long as the handle).  Copies that are captured have not been made, and are made whenever the
    // graph runs.
    if (sd.schedule_uid != L->uid || sd.graphs_send) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(stream, &capture);
        const bool captured = capture != cudaStreamCaptureStatusNone;
        if (e == cudaSuccess) e = cudaMemcpyAsync(items_dev, L->items_abs.data(), n_items * sizeof(Item), cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess && n_steps) e = cudaMemcpyAsync(steps_dev, L->steps.data(), n_steps * sizeof(Step), cudaMemcpyHostToDevice, stream);
        static_remember_schedule(device, e == cudaSuccess && !captured ? L->uid : 0, captured);
        if (e != cudaSuccess) return BIGBIRD_ECUDA;
    }

    const size_t tiles = (size_t)B * H * L->global_tiles;
    const Cut cut = cut_global_tiles(*L, B, sd.sm_count, tiles ? (int)std::min<size_t>(kStaticParts / tiles, 1 << 20) : 1);

    KernelParams p{};
    p.out = (__nv_bfloat16*)out;
    p.lse = lse;
    p.kbits = key_padding_mask ? kbits_dev : nullptr;
    p.partials = reinterpret_cast<float*>(sd.base + kStaticOffParts);
    p.items = items_dev;
    p.steps = steps_dev;
    p.status = words4;
    p.counter = words4 + 2;
    set_shape(p, *L, B, cut, scale, sd.sm_count);
    int launches = 0;
    if (enqueue(p, tm_q, tm_k, tm_v, key_padding_mask, kbits_dev, key_padding_mask ? (int)words : 0, words4, key_padding_mask ? 4 : 0, sd.sm_count, stream, &launches) != cudaSuccess)
        return BIGBIRD_ECUDA;
    return BIGBIRD_OK;
}

extern "C" int bigbird_last_status_static(void* stream, int* status, int* detail) {
    using namespace bigbird;
    if (!status) return BIGBIRD_EINVAL;
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return BIGBIRD_ECUDA;
    if (device < 0 || device >= 64) return BIGBIRD_EUNSUPPORTED;
    StaticDevice sd;
    if (static_setup(device, &sd) != cudaSuccess) return BIGBIRD_ECUDA;
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return BIGBIRD_ECUDA;
    int host[2] = {0, 0};                       // a stack buffer: nothing is allocated
    if (cudaMemcpy(host, sd.base, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return BIGBIRD_ECUDA;
    *status = host[0];
    if (detail) *detail = host[1];
    return BIGBIRD_OK;
}
