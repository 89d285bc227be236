// Gradients of BigBird block-sparse attention on Blackwell tensor cores (sm_100a): bf16 tensors, b = D = 64.
//
// The derivatives of Eq. (AT) of arXiv 2007.14062 (the paper trains through the operation, Sec. 4 and App. E.1, and leaves
// them to autodiff).  With P = exp(scale q k^T - lse) recomputed from the saved lse and delta_i = sum_d dout[i, d] out[i, d]:
//     dv = P^T dout,   dS = P o (dout v^T - delta),   dq = scale dS k,   dk = scale dS^T q.
//
// Both gradients by query (dq) and by key (dk, dv) have the same shape, so one kernel makes them:
//     rows   X1 | X2:  two query blocks (Q | dO), or two key blocks (K | V), stacked into a 128-row tile
//     steps  Y1 | Y2:  a key block (K | V) of the rows' lists, or a query block (Q | dO) of the transposed lists
//     S = X1 Y1^T, dP = X2 Y2^T;   acc0 += dS Y1  (dq, or dk);   acc1 += P Y2  (dv; key tiles only)
// Every operand is the 64 x 64 tile that TMA brings in: Y1 and Y2 serve once with their head dimension as the contraction
// (S, dP) and once with their token dimension (acc).  P and dS go back to tensor memory as the A operand, each as the sum of
// two bf16 numbers (16 significant bits): the products keep the precision of the fp32 path to below the rounding of the
// results, at twice the number of the accumulating MMAs.
//
// In the kernel's form for layouts with many of them (kShare), a block of the column side that only the upper rows of a tile attend shares
// a step with one that only the lower rows attend: each has its products with all 128 rows, the second ones leaving the lanes of the upper
// half alone (the instruction's vector of disabled lanes).  The products are as many as if the two had a step of their own, but the way of
// a step through the hands of four warps is gone once and not twice: 6312 steps instead of 8740 for the sparse tiles of the base layout,
// 12 heads, both kinds.
//
// Nothing carries over from step to step but the accumulators, so the steps of a tile are dealt in turn to three warpgroups
// with a 128-column score buffer each.  One thread issues the scores of a step as soon as its buffer is free, another the
// accumulation of the steps in turn.  An epilogue warpgroup takes a finished tile's accumulators while the next tile's scores
// are being computed.
// CTAs are persistent; a scheduler warp draws work from a counter: the tiles of global blocks first, cut along their (full)
// lists into parts where they would outlast the rest, then per (batch, head) the key tiles and the query tiles.  A part
// leaves its fp32 accumulators in scratch; whichever part is done last sums all of them in a fixed order.  No float atomics:
// results are bit-reproducible.
//
// Measured (gradients of the base workload [8, 12, 4096, 64]): CUDA-core kernels 16.3 ms; one thread issuing all MMAs 857 us,
// the same from one elected thread 557, columns 16 at a time with the next 16 on their way 527, two issuing threads 505, all
// roles on the ring, tests ahead of the commits and rows written by TMA 497 us ([1, 12, 16384, 64] with 13000 valid tokens
// 338 -> 193 us from the second of these to the last), and 189 with the parts of a cut tile fetched together ([2, 12, 1024]
// 54 -> 39.5 us, there no longer cut, 40.1 now); 430 us at full clocks.  A step took 1400 cycles then; its MMAs need 640 of the tensor pipe
// (51% of the launch by its counter then, 52% now; 555 steps per SM), without any elementwise work it takes 1100, without any MMAs 1150: what is
// left is the way of a step through the hands of four warps with three steps in flight, which is all that tensor memory holds.  Two
// threads per row (24 warps) were no faster.
//
// With shared steps [8, 12, 4096] takes 417.5 us at full clocks (430 with a step for each block) and forward and gradients together 628
// instead of 646 under the power cap; the launch says which layouts gain.  A shared step takes two of the seven places in the ring of Y.  (Nine of them, for which a tile's
// results left through its own row buffer, were no faster there, and the tile after next waited for that buffer: [8, 12, 4224] ETC 359 us
// against 345 under the power cap, [1, 2, 384] 13.5 against 13.35.)
//
// A first kernel makes, per query row, -lse * log2 e (-inf for rows without probabilities) and -delta, packs the key-padding
// mask and zeroes the counters.
#include <algorithm>

#include "sm100.cuh"

namespace bigbird {
namespace {

constexpr int kBufs = 3;                   // score buffers, each served by one warpgroup
constexpr int kRing = 2 * kBufs;           // ring of steps
constexpr int kStages = 7;                 // ring of Y1 | Y2 pairs: one for a step, two if the halves of the tile share it (kShare; else step entry e has place e)
static_assert(kRing <= kStages, "a place for each step");
constexpr int kSlots = 3;                  // tiles (or segments of long ones) posted by the scheduler (two: [3, 16, 4096] ragged, forward and
                                           // gradients, 212.5 us against 209.2)
constexpr int kSegSteps = 64;              // steps per posted segment, at least 33
// warps 0..11: the three elementwise warpgroups; 12..15: epilogue; 16: scheduler; 17: TMA producer; 18, 19: MMA issuers (scores,
// accumulations)
constexpr int kThreads = 640;
constexpr int kWarpEpilogue = 12, kWarpScheduler = 16, kWarpProducer = 17, kWarpScore = 18;
// 640 threads start with 96 registers each; a sub-partition's five warps share 480: three elementwise warps x 120 (32 columns
// of S and of dP and what becomes of them), an epilogue warp x 64 and a light warp x 56.
constexpr int kRegsElem = 120, kRegsEpilogue = 64, kRegsLight = 56;
static_assert(kBufs * kRegsElem + kRegsEpilogue + kRegsLight <= 5 * 96, "register trade between the five warps of a sub-partition");
constexpr int kTmemCols = 512;
constexpr int kBufCols = 128;              // S 64 | dP 64; dS (query tiles) or P and dS (key tiles) take their places
constexpr int kColAcc = kBufs * kBufCols;  // acc0 64 | acc1 64
static_assert(kColAcc + 128 <= kTmemCols, "tensor memory");
constexpr int kStatFloats = 2 * kBlock;    // per block of query rows: 64 x (-lse log2 e), 64 x (-delta)
constexpr int kPartialFloats = 2 * 128 * kBlock;   // one part of a split tile: acc0, acc1
enum { kDkv = 0, kDq = 1 };
enum { kSegFirst = 1, kSegLast = 2 };
// A step: one block that both halves of the tile attend or only one of them, or (kShare, kSecond) one for the upper half and another for the
// lower, whose rows are computed with 128-row products that leave the lanes of the other half alone.
enum { kAttends = 1, kPadded = 2, kSecond = 4 };        // of a half: it attends the step; some of its block's tokens are padding; its block is c1
// what there is to know about a ring entry: the halves (kLower times the lower one's bits), kind, first and last step of its tile, the
// tile's row buffer and the parity of that buffer's phase; kInfoEnd: no more steps; from bit kInfoStage the places of Y, 4 bits each
enum { kLower = 8, kInfoShared = kSecond * kLower, kInfoDkv = 64, kInfoFirst = 128, kInfoLast = 256, kInfoX = 512, kInfoXPar = 1024, kInfoEnd = 2048 };
constexpr int kInfoStage = 12;
static_assert(kStages <= 16, "bits of a place");

struct __align__(16) StepPart {
    int c;                         // block of the column side
    int halves;                    // kAttends, kPadded, kSecond of the upper half, and kLower times those of the lower
    unsigned long long kb;         // valid-token bits of the block (never 0)
};
struct StepEntry {
    StepPart part[2];              // kShare: part[1].c < 0 if there is one block only; else part[0] alone is used
};
struct __align__(16) TileSlot {
    int w;                         // work index, -1 = no more work
    int kind, bh, ra, rb;          // rb == kNoBlock: no lower half
    int n;                         // steps of this segment
    int flags;
    int split;                     // index of the split tile, -1 if it is not split
    int part;
    int pad_[3];
    unsigned long long rbits_a, rbits_b;
    StepEntry steps[kSegSteps];
};
struct __align__(16) SmemCtl {
    unsigned long long full[kRing], empty[kRing];
    unsigned long long x_full[2], x_empty[2];
    unsigned long long sdp_full[kBufs], p_full[kBufs];
    unsigned long long acc_full, acc_free, epi_sync;
    unsigned long long slot_full[kSlots], slot_empty[kSlots], slot_loaded[kSlots];
    TileSlot slot[kSlots];
    float x_stats[2][2][kStatFloats];      // query tiles: statistics of the rows
    float y_stats[kStages][kStatFloats];   // key tiles: of the step's query block
    unsigned info[kRing];
    unsigned long long bits[kRing][2];     // the valid-token bits of the step's blocks
    unsigned tmem_base;
    int abort_flag;
    int merge_last;
};
constexpr int kSmemX = 0;                                      // two buffers of X1a X1b X2a X2b
constexpr int kSmemRing = 2 * 4 * kTileBytes;
constexpr int kSmemOut = kSmemRing + kStages * 2 * kTileBytes;    // four tiles on their way out
constexpr int kSmemCtl = kSmemOut + 4 * kTileBytes;
constexpr int kSmemBytes = kSmemCtl + (int)sizeof(SmemCtl) + 1024;   // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 227 * 1024, "shared memory per CTA");

struct KernelParams {
    __nv_bfloat16 *dq, *dk, *dv;
    const float* stats;                    // [BH * nb][kStatFloats]
    const unsigned long long* kbits;       // [B * nb] or nullptr
    const Item *items_q, *items_k;         // sparse tiles, [H] x stride
    const Step *steps_q, *steps_k;
    const int* global_pairs;
    int* counter;                          // next work index
    int* arrived;                          // [2 * BH * global_tiles] parts of each split tile that are done
    int* status;                           // [2]: code, detail
    float* partials;
    int q_stride, sparse_tiles, global_tiles;
    int parts, part_steps;                 // how the tiles of global blocks are cut
    int BH, H, nb, total_work;
    int ahead;                             // posted slots that may wait for their loads when the next tile is drawn, 1 .. kSlots
    float scale, scale_log2;
};

__device__ __forceinline__ unsigned long long token_bits(const KernelParams& p, int batch, int c) {
    if (c < 0) return 0ull;
    return p.kbits ? p.kbits[(size_t)batch * p.nb + c] : ~0ull;
}

// ------------------------------------------------------------------------------------------------ scheduler (one warp)
// Zeros to a block of 64 gradient rows, for tiles that hold no token.  (By the scheduler itself: such a tile takes no slot and nobody
// else's time.  Gradients of [2, 12, 1024] with 333 and 1024 tokens 40.1 -> 38.0 us.  Stores without address arithmetic between them:
// [8, 12, 4224] ETC with one full sequence out of eight 151 -> 127 us.  Inline: the share of registers that this warp has left is
// known here, and a function of its own need not keep to it.)
__device__ __forceinline__ void clear_block(__nv_bfloat16* g, size_t block, int lane) {
    uint4* dst = reinterpret_cast<uint4*>(g) + block * (8 * kBlock) + lane;
#pragma unroll
    for (int i = 0; i < 16; ++i) dst[32 * i] = make_uint4(0u, 0u, 0u, 0u);
}

template <bool kShare>
__device__ __forceinline__ void scheduler_role(const KernelParams& p, SmemCtl* ctl, int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    unsigned slot_n = 0;
    bool first_item = true;
    for (;;) {
        int w = (int)blockIdx.x;                    // the first item is the CTA's own, the others are drawn
        if (!first_item) {
            if (slot_n >= (unsigned)p.ahead) {      // once what was posted `ahead` slots ago has been loaded (not before: see the launch)
                const unsigned m = slot_n - (unsigned)p.ahead;
                if (!mbar_wait(&ctl->slot_loaded[m % kSlots], (m / kSlots) & 1u, &ctl->abort_flag)) { give_up(&ctl->abort_flag, p.status, 114); return; }
                __syncwarp();
            }
            if (lane == 0) w = (int)gridDim.x + atomicAdd(p.counter, 1);
            w = __shfl_sync(0xffffffffu, w, 0);
        }
        first_item = false;
        if (w >= p.total_work) w = -1;
        int kind = 0, bh = 0, ra = kNoBlock, rb = kNoBlock, begin = 0, n_raw = 0, split = -1, part = 0;
        const Step* steps = nullptr;               // nullptr: blocks begin, begin + 1, ... attended by both halves
        if (w >= 0) {
            const int heavy = p.BH * p.global_tiles * p.parts;
            if (w < 2 * heavy) {
                kind = w < heavy ? kDkv : kDq;
                const int x = kind == kDkv ? w : w - heavy;
                const int tile = x / p.parts;      // (batch, head) major
                part = x - tile * p.parts;
                bh = tile / p.global_tiles;
                const int t = tile - bh * p.global_tiles;
                ra = p.global_pairs[2 * t];
                rb = p.global_pairs[2 * t + 1];
                begin = part * p.part_steps;
                n_raw = min(p.part_steps, p.nb - begin);
                if (p.parts > 1) split = kind * p.BH * p.global_tiles + tile;
            } else {
                const int x = w - 2 * heavy;
                bh = x / (2 * p.sparse_tiles);
                int it = x - bh * 2 * p.sparse_tiles;
                kind = it < p.sparse_tiles ? kDkv : kDq;
                if (kind == kDq) it -= p.sparse_tiles;
                const Item item = kind == kDkv ? p.items_k[(size_t)(bh % p.H) * p.sparse_tiles + it] : p.items_q[(size_t)(bh % p.H) * p.q_stride + it];
                ra = item.qa;
                rb = item.qb;
                begin = item.step_begin;
                n_raw = item.step_count;
                steps = kind == kDkv ? p.steps_k : p.steps_q;
            }
            if (!BB_CHECK(bh >= 0 && bh < p.BH && ra >= 0 && ra < p.nb && rb < p.nb && n_raw >= 0 && begin >= 0, 171)) w = -1;
        }
        const int batch = bh / p.H;
        const unsigned long long rbits_a = w >= 0 ? token_bits(p, batch, ra) : 0ull, rbits_b = w >= 0 ? token_bits(p, batch, rb) : 0ull;
        if (__builtin_expect(w >= 0 && (rbits_a | rbits_b) == 0ull, 0)) {        // no row is a token (then no part of a split tile arrives, and nobody merges)
            if (split < 0 || part == 0)
#pragma unroll 1
                for (int i = 0; i < (rb >= 0 ? 4 : 2); ++i)
                    if (kind == kDkv || !(i & 1)) clear_block(kind == kDq ? p.dq : (i & 1) ? p.dv : p.dk, (size_t)bh * p.nb + (i < 2 ? ra : rb), lane);
            continue;
        }
        int i0 = 0;
        bool first = true;
        StepEntry held{};                          // last step of a full segment: kept for the next one, so that no tile's last
        bool holding = false;                      // segment turns out to be empty
        do {
            const unsigned ss = slot_n % kSlots;
            if (!mbar_wait(&ctl->slot_empty[ss], ((slot_n / kSlots) & 1u) ^ 1u, &ctl->abort_flag)) { give_up(&ctl->abort_flag, p.status, 111); return; }
            __syncwarp();
            TileSlot* slot = &ctl->slot[ss];
            int count = 0;
            if (holding) {
                if (lane == 0) slot->steps[0] = held;
                count = 1;
            }
#pragma unroll 1
            while (i0 < n_raw && count <= kSegSteps - 32) {
                const int i = i0 + lane;
                int c = -1;
                unsigned long long kb = 0ull;
                bool ua = false, ub = false;
                if (i < n_raw) {
                    const Step s = steps ? steps[begin + i] : Step{begin + i, kBothHalves};
                    c = s.c;
                    if (BB_CHECK(c >= 0 && c < p.nb, 170)) kb = token_bits(p, batch, c);
                    ua = s.who != kLowerHalf && rbits_a != 0ull && kb != 0ull;
                    ub = s.who != kUpperHalf && rbits_b != 0ull && kb != 0ull;
                }
                const int flags = kAttends | (kb != ~0ull ? kPadded : 0), halves = (ua ? flags : 0) | (ub ? flags * kLower : 0);
                if constexpr (kShare) {
                    // In turn a block of both halves and one of the upper half together with one of the lower (what is left of either
                    // by itself): steps of one and of two blocks alternate, so that the ring holds the same number of steps at any time.
                    const unsigned b_both = __ballot_sync(0xffffffffu, ua && ub), b_up = __ballot_sync(0xffffffffu, ua && !ub),
                                   b_lo = __ballot_sync(0xffffffffu, ub && !ua);
                    const int n_both = __popc(b_both), n_up = __popc(b_up), n_lo = __popc(b_lo), n_one = max(n_up, n_lo);
                    if (ua || ub) {
                        const int rank = __popc((ua ? (ub ? b_both : b_up) : b_lo) & lt_mask);
                        const int at = rank + (ua && ub ? min(rank, n_one) : min(rank + 1, n_both));
                        const bool second = !ua && rank < n_up, alone = !second && (ub || rank >= n_lo);
                        StepPart* part = slot->steps[count + at].part;
                        part[second ? 1 : 0] = StepPart{c, halves | (second ? kSecond * kLower : 0), kb};
                        if (alone) part[1] = StepPart{-1, 0, 0ull};
                    }
                    count += n_both + n_one;
                } else {
                    const unsigned bal = __ballot_sync(0xffffffffu, ua || ub);
                    if (ua || ub) slot->steps[count + __popc(bal & lt_mask)].part[0] = StepPart{c, halves, kb};
                    count += __popc(bal);
                }
                i0 += 32;
            }
            __syncwarp();
            holding = i0 < n_raw && count > 0;
            if (holding) held = slot->steps[--count];
            if (lane == 0) {
                slot->w = w;
                slot->kind = kind;
                slot->bh = bh;
                slot->ra = ra;
                slot->rb = rb;
                slot->n = count;
                slot->flags = (first ? kSegFirst : 0) | (i0 >= n_raw ? kSegLast : 0);
                slot->split = split;
                slot->part = part;
                slot->rbits_a = rbits_a;
                slot->rbits_b = rbits_b;
            }
            __threadfence_block();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->slot_full[ss]);
            ++slot_n;
            first = false;
        } while (i0 < n_raw);
        if (w < 0) return;
    }
}

// ------------------------------------------------------------------------------------------------ TMA producer (one thread)
template <bool kShare>
__device__ __forceinline__ void producer_role(const KernelParams& p, SmemCtl* ctl, unsigned char* smem, const CUtensorMap* tm_q,
                                              const CUtensorMap* tm_k, const CUtensorMap* tm_v, const CUtensorMap* tm_do) {
    int* abort_flag = &ctl->abort_flag;
    unsigned slot_n = 0, tile_n = 0, step_n = 0, done_n = 0;      // done_n: steps known to be accumulated
    unsigned stage = 0, free_stages = kStages, shared_steps = 0;  // bit n mod 32 of shared_steps: step n has two blocks
    bool fresh = false;                             // no step of the tile has been loaded yet
    int fail = 0;
    // room for a step of `blocks` blocks
    auto room = [&](unsigned blocks) -> bool {
        if constexpr (kShare) {
            while (free_stages < blocks || step_n - done_n == (unsigned)kRing) {
                if (!mbar_wait(&ctl->empty[done_n % kRing], (done_n / kRing) & 1u, abort_flag)) return false;
                free_stages += 1u + ((shared_steps >> (done_n & 31u)) & 1u);
                ++done_n;
            }
            return true;
        } else {
            return mbar_wait(&ctl->empty[step_n % kRing], ((step_n / kRing) & 1u) ^ 1u, abort_flag);
        }
    };
    for (;;) {
        const unsigned ss = slot_n % kSlots;
        if (!mbar_wait(&ctl->slot_full[ss], (slot_n / kSlots) & 1u, abort_flag)) { fail = 113; break; }
        const TileSlot* slot = &ctl->slot[ss];
        const int w = slot->w, flags = slot->flags, n = slot->n, bh = slot->bh;
        const bool dkv = slot->kind == kDkv;
        if (w < 0) {                                // the last entries of the ring, one for each score buffer's warps
            for (int i = 0; i < kBufs; ++i, ++step_n) {
                if (!room(0)) { fail = 110; break; }
                const unsigned g = step_n % kRing;
                ctl->info[g] = kInfoEnd;
                __threadfence_block();              // (nothing is loaded into this entry: its word is on its own ahead of the arrival)
                mbar_arrive(&ctl->full[g]);
            }
            break;
        }
        if (flags & kSegFirst) fresh = true;
        const CUtensorMap *tm1 = dkv ? tm_q : tm_k, *tm2 = dkv ? tm_do : tm_v;
        for (int i = 0; i < n; ++i) {
            const StepPart e0 = slot->steps[i].part[0];
            StepPart e1{-1, 0, 0ull};
            if constexpr (kShare) e1 = slot->steps[i].part[1];
            const int c0 = e0.c, c1 = e1.c;
            unsigned info = (unsigned)(e0.halves | e1.halves) | (dkv ? kInfoDkv : 0) | (i == n - 1 && (flags & kSegLast) ? kInfoLast : 0);
            if (fresh) {
                const int ra = slot->ra, rb = slot->rb;
                const unsigned xs = tile_n & 1u;
                if (!mbar_wait(&ctl->x_empty[xs], ((tile_n >> 1) & 1u) ^ 1u, abort_flag)) { fail = 112; break; }
                unsigned char* x = smem + kSmemX + xs * 4 * kTileBytes;
                unsigned long long* bar = &ctl->x_full[xs];
                const CUtensorMap *xm1 = dkv ? tm_k : tm_q, *xm2 = dkv ? tm_v : tm_do;
                const int blocks = rb >= 0 ? 2 : 1;
                if (!BB_CHECK(bh >= 0 && bh < p.BH && ra >= 0 && ra < p.nb && rb < p.nb && rb >= kNoBlock, 172)) return;
                mbar_expect_tx(bar, blocks * (2 * kTileBytes + (dkv ? 0 : kStatFloats * 4)));
                for (int j = 0; j < blocks; ++j) {
                    const int row = bh * p.nb + (j ? rb : ra);
                    tma_load_tile(x + j * kTileBytes, xm1, row * kBlock, bar);
                    tma_load_tile(x + (2 + j) * kTileBytes, xm2, row * kBlock, bar);
                    if (!dkv) bulk_load(ctl->x_stats[xs][j], p.stats + (size_t)row * kStatFloats, kStatFloats * 4, bar);
                }
                ++tile_n;
                fresh = false;
                info |= kInfoFirst;
            }
            info |= (((tile_n - 1) & 1u) ? kInfoX : 0) | ((((tile_n - 1) >> 1) & 1u) ? kInfoXPar : 0);
            if (!BB_CHECK(n <= kSegSteps && c0 >= 0 && c0 < p.nb && c1 < p.nb && (c1 >= 0) == ((info & kInfoShared) != 0), 173)) return;
            const unsigned blocks = c1 >= 0 ? 2u : 1u, g = step_n % kRing;
            if (!room(blocks)) { fail = 110; break; }
            if constexpr (kShare) {
                free_stages -= blocks;
                const unsigned bit = 1u << (step_n & 31u);
                shared_steps = c1 >= 0 ? shared_steps | bit : shared_steps & ~bit;
                const unsigned next = stage + 1 == kStages ? 0u : stage + 1;
                ctl->info[g] = info | (stage << kInfoStage) | (next << (kInfoStage + 4));
                ctl->bits[g][1] = e1.kb;
            } else {
                ctl->info[g] = info;
                stage = g;                          // a place for each entry
            }
            ctl->bits[g][0] = e0.kb;
            mbar_expect_tx(&ctl->full[g], blocks * (2 * kTileBytes + (dkv ? kStatFloats * 4 : 0)));
#pragma unroll 1
            for (unsigned j = 0; j < blocks; ++j) {
                const int row = bh * p.nb + (j ? c1 : c0);
                unsigned char* y = smem + kSmemRing + stage * 2 * kTileBytes;
                tma_load_tile(y, tm1, row * kBlock, &ctl->full[g]);
                tma_load_tile(y + kTileBytes, tm2, row * kBlock, &ctl->full[g]);
                if (dkv) bulk_load(ctl->y_stats[stage], p.stats + (size_t)row * kStatFloats, kStatFloats * 4, &ctl->full[g]);
                if (kShare && ++stage == kStages) stage = 0;
            }
            ++step_n;
        }
        if (fail) break;
        mbar_arrive(&ctl->slot_loaded[ss]);
        mbar_arrive(&ctl->slot_empty[ss]);
        ++slot_n;
    }
    if (fail) give_up(abort_flag, p.status, fail);
}

// ------------------------------------------------------------------------------------------------ MMA issuers (two threads)
// Each is alone in its warp, so nothing hides the latency of its instructions: an MMA takes some 30 cycles to issue, a barrier
// test 45, a test behind a commit 200.  One thread that issued everything and walked the posted tiles needed 1740 cycles a step.
// So one issues the scores (S and dP) and one the accumulations, and both see the ring only, where each entry comes with a word
// that says what there is to know about the step.  full[] tells both of a loaded entry, empty[] (committed behind a step's
// accumulation) frees the ring entry and its Y for the producer and, three steps on, the score buffer for the first thread.  The tests for
// the next step come before a step's commit: behind it they cost four times as much.
template <bool kShare>
__device__ __forceinline__ void score_role(const KernelParams& p, SmemCtl* ctl, unsigned char* smem, unsigned tmem) {
    int* abort_flag = &ctl->abort_flag;
    constexpr unsigned kStageDesc = (2 * kTileBytes) >> 4, kTileDesc = kTileBytes >> 4;
    const unsigned ring0 = smem_desc_lo(smem_u32(smem + kSmemRing)), x0 = smem_desc_lo(smem_u32(smem + kSmemX));
    unsigned stg = 0, ph = 0, buf = 0;              // this step's ring entry (and its phase) and score buffer
    unsigned old = 0, old_ph = 0, n = 0;            // ring entry and phase of the step three back; steps issued, up to kBufs
    unsigned x1 = x0;                               // row buffer of the tile
    bool have_f = false, have_e = false;            // the tests made ahead
    unsigned info = 0;
    int fail = 0;
    for (;;) {
        if (!have_f) {
            if (!mbar_wait(&ctl->full[stg], ph, abort_flag)) { fail = 120; break; }
            info = ld_shared(&ctl->info[stg]);
        }
        if (info & kInfoEnd) break;
        if (n == (unsigned)kBufs) {                 // the buffer's last user must have been accumulated
            if (!have_e && !mbar_wait(&ctl->empty[old], old_ph, abort_flag)) { fail = 121; break; }
            if (++old == kRing) { old = 0; old_ph ^= 1u; }
        } else ++n;
        if (info & kInfoFirst) {
            const unsigned xs = (info & kInfoX) ? 1u : 0u;
            if (!mbar_wait(&ctl->x_full[xs], (info & kInfoXPar) ? 1u : 0u, abort_flag)) { fail = 124; break; }
            x1 = x0 + xs * 4 * kTileDesc;
        }
        tc_fence_after();
        const unsigned y1 = ring0 + (kShare ? (info >> kInfoStage) & 15u : stg) * kStageDesc, d = tmem + buf * kBufCols;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) mma_ss_lo(d, x1 + kk * 2, y1 + kk * 2, kIdescQK64, kk > 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) mma_ss_lo(d + 64, x1 + 2 * kTileDesc + kk * 2, y1 + kTileDesc + kk * 2, kIdescQK64, kk > 0);
        if (kShare && (info & kInfoShared)) {       // over the lanes of the lower half: with its own block
            const unsigned z1 = ring0 + ((info >> (kInfoStage + 4)) & 15u) * kStageDesc;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma_ss_half(d, x1 + kk * 2, z1 + kk * 2, kIdescQK64, kk > 0, ~0u, 0u);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma_ss_half(d + 64, x1 + 2 * kTileDesc + kk * 2, z1 + kTileDesc + kk * 2, kIdescQK64, kk > 0, ~0u, 0u);
        }
        unsigned long long* const done = &ctl->sdp_full[buf];
        if (++buf == kBufs) buf = 0;
        if (++stg == kRing) { stg = 0; ph ^= 1u; }
        have_f = mbar_test(&ctl->full[stg], ph);
        have_e = mbar_test(&ctl->empty[old], old_ph);
        info = ld_shared(&ctl->info[stg]);                      // (read again if the entry is not there yet)
        tc_commit(done);
    }
    if (fail) give_up(abort_flag, p.status, fail);
}

template <bool kShare>
__device__ __forceinline__ void accumulate_role(const KernelParams& p, SmemCtl* ctl, unsigned char* smem, unsigned tmem) {
    int* abort_flag = &ctl->abort_flag;
    constexpr unsigned kStageDesc = (2 * kTileBytes) >> 4, kTileDesc = kTileBytes >> 4;
    const unsigned ring0 = smem_desc_lo(smem_u32(smem + kSmemRing)), acc = tmem + kColAcc;
    unsigned stg = 0, ph = 0, buf = 0, par = 0;     // ring entry and its phase, score buffer and the parity of its p_full
    unsigned acc_n = 0;                             // tiles handed to the epilogue
    bool have_f = false, have_p = false;            // the tests made ahead
    unsigned info = 0;
    int fail = 0;
    for (;;) {
        if (!have_f) {
            if (!mbar_wait(&ctl->full[stg], ph, abort_flag)) { fail = 125; break; }
            info = ld_shared(&ctl->info[stg]);
        }
        if (info & kInfoEnd) break;
        // the epilogue must have taken the previous tile's accumulators before this tile's first product overwrites them
        if ((info & kInfoFirst) && acc_n > 0 && !mbar_wait(&ctl->acc_free, (acc_n - 1) & 1u, abort_flag)) { fail = 127; break; }
        if (!have_p && !mbar_wait(&ctl->p_full[buf], par, abort_flag)) { fail = 122; break; }
        tc_fence_after();
        const unsigned keep = (info & kInfoFirst) ? 0u : 1u;
        // 16 tokens per MMA: 8 packed columns of A (the high halves, then the low halves), two 8-row groups of Y
        if constexpr (kShare) {
            unsigned y1 = ring0 + ((info >> kInfoStage) & 15u) * kStageDesc, skip_upper = 0u, skip_lower = (info & kInfoShared) ? ~0u : 0u;
#pragma unroll 1
            for (;;) {                                  // a shared step: the upper half's block, then the lower half's, each for its lanes
                unsigned a = tmem + buf * kBufCols;
                if (info & kInfoDkv) {
                    const unsigned y2 = y1 + kTileDesc;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        mma_ts_half(acc + 64, a + kk * 16, y2 + ((kk * 2048) >> 4), kIdescPV, kk > 0 ? 1u : keep, skip_upper, skip_lower);
                        mma_ts_half(acc + 64, a + kk * 16 + 8, y2 + ((kk * 2048) >> 4), kIdescPV, 1u, skip_upper, skip_lower);
                    }
                    a += 64;
                }
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    mma_ts_half(acc, a + kk * 16, y1 + ((kk * 2048) >> 4), kIdescPV, kk > 0 ? 1u : keep, skip_upper, skip_lower);
                    mma_ts_half(acc, a + kk * 16 + 8, y1 + ((kk * 2048) >> 4), kIdescPV, 1u, skip_upper, skip_lower);
                }
                if (!skip_lower) break;
                y1 = ring0 + ((info >> (kInfoStage + 4)) & 15u) * kStageDesc;
                skip_upper = ~0u;
                skip_lower = 0u;
            }
        } else {
            const unsigned y1 = ring0 + stg * kStageDesc;
            unsigned a = tmem + buf * kBufCols;
            if (info & kInfoDkv) {
                const unsigned y2 = y1 + kTileDesc;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    mma_ts_lo(acc + 64, a + kk * 16, y2 + ((kk * 2048) >> 4), kIdescPV, kk > 0 ? 1u : keep);
                    mma_ts_lo(acc + 64, a + kk * 16 + 8, y2 + ((kk * 2048) >> 4), kIdescPV, 1u);
                }
                a += 64;
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                mma_ts_lo(acc, a + kk * 16, y1 + ((kk * 2048) >> 4), kIdescPV, kk > 0 ? 1u : keep);
                mma_ts_lo(acc, a + kk * 16 + 8, y1 + ((kk * 2048) >> 4), kIdescPV, 1u);
            }
        }
        const unsigned now = info;
        unsigned long long* const done = &ctl->empty[stg];
        if (++buf == kBufs) { buf = 0; par ^= 1u; }
        if (++stg == kRing) { stg = 0; ph ^= 1u; }
        have_f = mbar_test(&ctl->full[stg], ph);
        have_p = mbar_test(&ctl->p_full[buf], par);
        info = ld_shared(&ctl->info[stg]);                      // (read again if the entry is not there yet)
        tc_commit(done);
        if (now & kInfoLast) {                      // (the tile's scores and elementwise work are done as well: its rows may go)
            tc_commit(&ctl->acc_full);
            tc_commit(&ctl->x_empty[(now & kInfoX) ? 1 : 0]);
            ++acc_n;
        }
    }
    if (fail) give_up(abort_flag, p.status, fail);
}

// ------------------------------------------------------------------------------------------------ elementwise (three warpgroups, one thread per row)
// The 64 columns of a step, 16 at a time, the next 16 on their way out of tensor memory meanwhile.  What takes the place of 16
// columns of fp32 is 8 columns of packed high halves and 8 of low halves.
// -inf over S and zero over dP of a step's padded tokens, in tensor memory: either may have overflowed.  (Rare: the blocks that hold a
// sequence's end.  Key tiles need it although their padded queries have -inf for their statistics: that makes P zero only where S is
// below infinity.  A test per 16 columns in dq_columns and dkv_columns cost training 5%.)
__device__ __forceinline__ void mask_scores(unsigned buf, unsigned long long bits64) {
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        float s[16], d[16];
        const unsigned bits = (unsigned)(bits64 >> (16 * c));
        tmem_ld16(buf + 16 * c, s);
        tmem_ld16(buf + 64 + 16 * c, d);
        tmem_wait_ld();
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const bool token = (bits >> t) & 1u;
            s[t] = token ? s[t] : -INFINITY;
            d[t] = token ? d[t] : 0.f;
        }
        tmem_st16(buf + 16 * c, reinterpret_cast<unsigned*>(s));
        tmem_st16(buf + 64 + 16 * c, reinterpret_cast<unsigned*>(d));
    }
    tmem_wait_st();
}
// Query tiles: dS = exp2(S sl2 + nl) (dP + nd) over S.
__device__ __forceinline__ void dq_columns(unsigned buf, float sl2, float nl, float nd) {
    float s[2][16], d[2][16];
    tmem_ld16(buf, s[0]);
    tmem_ld16(buf + 64, d[0]);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float *sc = s[c & 1], *dc = d[c & 1];
        tmem_wait_ld();
        if (c < 3) {
            tmem_ld16(buf + 16 * (c + 1), s[(c + 1) & 1]);
            tmem_ld16(buf + 64 + 16 * (c + 1), d[(c + 1) & 1]);
        }
        unsigned o[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float x0, x1;
            ffma2(x0, x1, sc[2 * j], sc[2 * j + 1], sl2, nl);
            add_mul2(x0, x1, dc[2 * j], dc[2 * j + 1], nd, nd, ex2(x0), ex2(x1));
            split_bf16(x0, x1, o[j], o[8 + j]);
        }
        tmem_st16(buf + 16 * c, o);
    }
}
// Key tiles: P over S and dS over dP; the statistics belong to the columns.
__device__ __forceinline__ void dkv_columns(unsigned buf, float sl2, const float2* nl, const float2* nd) {
    float s[2][16], d[2][16];
    tmem_ld16(buf, s[0]);
    tmem_ld16(buf + 64, d[0]);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float *sc = s[c & 1], *dc = d[c & 1];
        tmem_wait_ld();
        if (c < 3) {
            tmem_ld16(buf + 16 * (c + 1), s[(c + 1) & 1]);
            tmem_ld16(buf + 64 + 16 * (c + 1), d[(c + 1) & 1]);
        }
        unsigned o[16], u[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 n2 = nl[8 * c + j], d2 = nd[8 * c + j];
            float x0, x1;
            ffma2v(x0, x1, sc[2 * j], sc[2 * j + 1], sl2, n2.x, n2.y);
            x0 = ex2(x0);
            x1 = ex2(x1);
            split_bf16(x0, x1, o[j], o[8 + j]);
            add_mul2(x0, x1, dc[2 * j], dc[2 * j + 1], d2.x, d2.y, x0, x1);
            split_bf16(x0, x1, u[j], u[8 + j]);
        }
        tmem_st16(buf + 16 * c, o);
        tmem_st16(buf + 64 + 16 * c, u);
    }
}

// Like the issuing threads they walk the ring only: every third entry is theirs.
template <bool kShare>
__device__ __forceinline__ void elementwise_role(const KernelParams& p, SmemCtl* ctl, unsigned tmem, int warp, int lane) {
    int* abort_flag = &ctl->abort_flag;
    const unsigned g = (unsigned)warp >> 2;         // warpgroup = score buffer
    const int row = (warp & 3) * 32 + lane;
    const unsigned half_shift = row >= kBlock ? 3 : 0;
    static_assert(kLower == 8, "");
    const unsigned buf = tmem + ((unsigned)((warp & 3) * 32) << 16) + g * kBufCols;
    const float* x_stats = &ctl->x_stats[0][row >= kBlock][row & (kBlock - 1)];
    unsigned stage = g, par = 0, full_par = 0;      // par: of this buffer's use; the ring has twice as many entries as there are buffers
    int fail = 0;
    for (;;) {
        if (!mbar_wait(&ctl->full[stage], full_par, abort_flag)) { fail = 132; break; }
        const unsigned info = ld_shared(&ctl->info[stage]);
        if (info & kInfoEnd) break;
        const bool dkv = info & kInfoDkv;
        const unsigned half = (info >> half_shift) & 7u;        // warp-uniform
        const bool mine = half & kAttends, second = kShare && (half & kSecond);
        float nl = 0.f, nd = 0.f;
        if (!dkv) {
            const unsigned xs = (info & kInfoX) ? 1u : 0u;
            if (!mbar_wait(&ctl->x_full[xs], (info & kInfoXPar) ? 1u : 0u, abort_flag)) { fail = 134; break; }
            nl = x_stats[xs * 2 * kStatFloats];
            nd = x_stats[xs * 2 * kStatFloats + kBlock];
        }
        if (!mbar_wait(&ctl->sdp_full[g], par, abort_flag)) { fail = 131; break; }
        __syncwarp();                               // lanes leave the wait one by one
        tc_fence_after();
        if (__builtin_expect((half & kPadded) != 0, 0)) mask_scores(buf, ctl->bits[stage][second]);
        if (!mine) {
            tmem_st32_zero(buf);
            tmem_st32_zero(buf + 32);
            if (dkv) {
                tmem_st32_zero(buf + 64);
                tmem_st32_zero(buf + 96);
            }
        } else if (dkv) {
            const float2* st = reinterpret_cast<const float2*>(ctl->y_stats[kShare ? (info >> (kInfoStage + (second ? 4 : 0))) & 15u : stage]);
            dkv_columns(buf, p.scale_log2, st, st + 32);
        } else {
            dq_columns(buf, p.scale_log2, nl, nd);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&ctl->p_full[g]);
        par ^= 1u;
        if (stage == g) stage = g + kBufs;
        else { stage = g; full_par ^= 1u; }
    }
    if (fail) give_up(abort_flag, p.status, fail);
}

// ------------------------------------------------------------------------------------------------ epilogue (one warpgroup)
// All epilogue threads (a bounded wait like every other: a warp that has given up must not leave the others in a hardware barrier).
__device__ __forceinline__ bool epilogue_sync(SmemCtl* ctl, unsigned& n) {
    mbar_arrive(&ctl->epi_sync);
    const bool ok = mbar_wait(&ctl->epi_sync, n & 1u, &ctl->abort_flag);
    ++n;
    __syncwarp();
    return ok;
}

// Sums the parts of a split tile (the last one to arrive does) and writes the rows.
__device__ __forceinline__ void merge_parts(const KernelParams& p, const TileSlot* slot, int tid) {
    const bool dkv = slot->kind == kDkv;
    const float* base = p.partials + (size_t)slot->split * p.parts * kPartialFloats;
    // four columns of four rows at a time, so that their loads are in flight together
#pragma unroll 1
    for (int i0 = tid; i0 < (dkv ? 2 : 1) * 128 * 16; i0 += 4 * 128) {
        const float4* src = reinterpret_cast<const float4*>(base) + i0;       // rows of 16 float4, the accumulators one behind the other
        float4 acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int pt = 0; pt < p.parts; ++pt, src += kPartialFloats / 4) {     // fixed order: results do not depend on scheduling
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldcg(src + 128 * u);
#pragma unroll
            for (int u = 0; u < 4; ++u) { acc[u].x += v[u].x; acc[u].y += v[u].y; acc[u].z += v[u].z; acc[u].w += v[u].w; }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + 128 * u, m = idx >> 11, row = (idx >> 4) & 127, c4 = idx & 15;
            const int blk = row >= kBlock ? slot->rb : slot->ra;
            if (blk < 0) continue;
            const unsigned long long bits = row >= kBlock ? slot->rbits_b : slot->rbits_a;
            const bool row_ok = (bits >> (row & 63)) & 1ull;     // (a select: see the epilogue)
            const float f = m ? 1.f : p.scale;
            __nv_bfloat16* dst = (dkv ? (m ? p.dv : p.dk) : p.dq) + (((size_t)slot->bh * p.nb + blk) * kBlock + (row & 63)) * kBlock;
            reinterpret_cast<uint2*>(dst)[c4] = row_ok ? make_uint2(pack_bf16(acc[u].x * f, acc[u].y * f), pack_bf16(acc[u].z * f, acc[u].w * f))
                                                       : make_uint2(0u, 0u);
        }
    }
}

__device__ __forceinline__ void epilogue_role(const KernelParams& p, SmemCtl* ctl, unsigned char* smem, unsigned tmem, int warp, int lane,
                                              const CUtensorMap* tm_dq, const CUtensorMap* tm_dk, const CUtensorMap* tm_dv) {
    int* abort_flag = &ctl->abort_flag;
    const int quad = warp & 3, row = quad * 32 + lane, r64 = row & (kBlock - 1);
    const bool lower = row >= kBlock;
    const unsigned acc = tmem + ((unsigned)(quad * 32) << 16) + kColAcc;
    unsigned char* const stage = smem + kSmemOut;   // [accumulator][half of the tile]: 64 x 64 bf16, swizzled
    const unsigned my_row = smem_u32(stage) + (lower ? kTileBytes : 0) + r64 * 128;
    unsigned slot_n = 0, acc_n = 0, sync_n = 0;
    bool have = false;                              // has the tile had any step
    int fail = 0;
    for (;;) {
        const unsigned ss = slot_n % kSlots;
        if (!mbar_wait(&ctl->slot_full[ss], (slot_n / kSlots) & 1u, abort_flag)) { fail = 140; break; }
        __syncwarp();
        const TileSlot* slot = &ctl->slot[ss];
        const int flags = slot->flags;
        if (slot->w < 0) break;
        if (flags & kSegFirst) have = false;
        have = have || slot->n > 0;
        if (flags & kSegLast) {
            const bool dkv = slot->kind == kDkv;
            const int split = slot->split, n_chunks = dkv ? 8 : 4;     // of 16 columns
            if (!BB_CHECK(slot->bh >= 0 && slot->bh < p.BH && slot->ra >= 0 && slot->ra < p.nb && slot->rb < p.nb &&
                          split < 2 * p.BH * p.global_tiles && slot->part >= 0 && slot->part < p.parts, 174)) break;
            const bool row_ok = ((lower ? slot->rbits_b : slot->rbits_a) >> r64) & 1ull;
            // (a tile without a step is a part of a split one: one of its rows is a token, and a block is in its own list)
            if (row == 0) bulk_wait_read();         // the previous tile has left the staging tiles
            if (!epilogue_sync(ctl, sync_n)) { fail = 142; break; }
            if (have) {
                if (!mbar_wait(&ctl->acc_full, acc_n & 1u, abort_flag)) { fail = 141; break; }
                __syncwarp();
                tc_fence_after();
                ++acc_n;
            }
            float* part = p.partials + ((size_t)max(split, 0) * p.parts + slot->part) * kPartialFloats + row * kBlock;
#pragma unroll 1
            for (int c = 0; c < n_chunks; ++c) {
                float o[16];
                if (have) {
                    tmem_ld16(acc + 16 * c, o);
                    tmem_wait_ld();
                    if (c == n_chunks - 1) { tc_fence_before(); mbar_arrive(&ctl->acc_free); }
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) o[j] = 0.f;
                }
                const int m = c >> 2;
                if (split >= 0) {
                    float4* d4 = reinterpret_cast<float4*>(part + m * 128 * kBlock) + 4 * (c & 3);
#pragma unroll
                    for (int j = 0; j < 4; ++j) d4[j] = make_float4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
                } else {
                    // A padded row is zeroed by a select and not by a factor: a padded key takes part like any other up to here, and
                    // since its scores are not in lse, its sums may be infinite or NaN.
                    const float f = m ? 1.f : p.scale;
                    const unsigned base = my_row + m * 2 * kTileBytes;
                    unsigned w[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) w[j] = row_ok ? pack_bf16(o[2 * j] * f, o[2 * j + 1] * f) : 0u;
#pragma unroll
                    for (int j = 0; j < 2; ++j)     // 16 bytes of a row; the swizzle keeps the rows of a store in different banks
                        st_shared16(base + (((2 * (c & 3) + j) ^ (r64 & 7)) << 4), w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
                }
            }
            if (split < 0) {
                proxy_fence();
                if (!epilogue_sync(ctl, sync_n)) { fail = 142; break; }
                if (row == 0) {
                    const int first = slot->bh * p.nb, ra = (first + slot->ra) * kBlock, rb = (first + slot->rb) * kBlock;
                    const bool two = slot->rb >= 0;
                    const CUtensorMap* tm0 = dkv ? tm_dk : tm_dq;
                    tma_store_tile(tm0, ra, stage);
                    if (two) tma_store_tile(tm0, rb, stage + kTileBytes);
                    if (dkv) {
                        tma_store_tile(tm_dv, ra, stage + 2 * kTileBytes);
                        if (two) tma_store_tile(tm_dv, rb, stage + 3 * kTileBytes);
                    }
                    bulk_commit();
                }
            } else {
                __threadfence();
                if (!epilogue_sync(ctl, sync_n)) { fail = 142; break; }
                if (row == 0) ctl->merge_last = atomicAdd(&p.arrived[split], 1) == p.parts - 1;
                if (!epilogue_sync(ctl, sync_n)) { fail = 142; break; }
                if (ctl->merge_last) {
                    __threadfence();
                    merge_parts(p, slot, row);
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->slot_empty[ss]);
        ++slot_n;
    }
    if (row == 0) bulk_wait_all();
    if (fail) give_up(abort_flag, p.status, fail);
}

// ------------------------------------------------------------------------------------------------ the kernel
template <bool kShare>
__global__ void __launch_bounds__(kThreads, 1)
attn_bwd_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                      const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                      const __grid_constant__ CUtensorMap tm_dq, const __grid_constant__ CUtensorMap tm_dk,
                      const __grid_constant__ CUtensorMap tm_dv, const KernelParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(smem + kSmemCtl);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;      // (uniform, and known to be)

    if (threadIdx.x == 0) {
        for (int i = 0; i < kRing; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&ctl->x_full[i], 1); mbar_init(&ctl->x_empty[i], 1); }
        for (int i = 0; i < kBufs; ++i) { mbar_init(&ctl->sdp_full[i], 1); mbar_init(&ctl->p_full[i], 128); }
        mbar_init(&ctl->acc_full, 1);
        mbar_init(&ctl->acc_free, 128);
        mbar_init(&ctl->epi_sync, 128);
        for (int i = 0; i < kSlots; ++i) { mbar_init(&ctl->slot_full[i], 1); mbar_init(&ctl->slot_empty[i], 1 + 4); mbar_init(&ctl->slot_loaded[i], 1); }   // producer, epilogue warps
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

    if (warp < kWarpEpilogue) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsElem));
        elementwise_role<kShare>(p, ctl, tmem, warp, lane);
    } else if (warp < kWarpScheduler) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsEpilogue));
        epilogue_role(p, ctl, smem, tmem, warp, lane, &tm_dq, &tm_dk, &tm_dv);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLight));
        if (warp == kWarpScheduler) scheduler_role<kShare>(p, ctl, lane);
        else if (warp == kWarpProducer) { if (elect_one()) producer_role<kShare>(p, ctl, smem, &tm_q, &tm_k, &tm_v, &tm_do); }
        else if (warp == kWarpScore) { if (elect_one()) score_role<kShare>(p, ctl, smem, tmem); }
        else if (elect_one()) accumulate_role<kShare>(p, ctl, smem, tmem);
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
}

// Per query row: -lse log2 e (-inf: padded, or nothing attended) and -delta; the key-padding mask as one 64-bit word per
// block; zeroed counters.  Eight threads share a row.  Reads out and dout once: memory bound.
constexpr int kPrepThreads = 256, kPrepRows = kPrepThreads / 8;
__global__ void __launch_bounds__(kPrepThreads)
attn_bwd_prepare_kernel(const uint4* __restrict__ out, const uint4* __restrict__ dout, const float* __restrict__ lse,
                        const uint8_t* __restrict__ kpm, float* __restrict__ stats, unsigned long long* __restrict__ kbits,
                        int* __restrict__ counters, int n_counters, long long rows, int N, int H, int row_ctas, int n_words) {
    grid_dependency_release();
    grid_dependency_wait();
    if ((int)blockIdx.x >= row_ctas) {             // the last CTAs: mask words and counters
        const int part = blockIdx.x - row_ctas, stride = gridDim.x - row_ctas;
        for (int i = part * kPrepThreads + threadIdx.x; i < n_counters; i += stride * kPrepThreads) counters[i] = 0;
        const int lane = threadIdx.x & 31;
        for (int word = (part * kPrepThreads + threadIdx.x) >> 5; word < n_words; word += stride * (kPrepThreads >> 5)) {
            const uint8_t* src = kpm + (size_t)word * kBlock;
            const unsigned lo = __ballot_sync(0xffffffffu, src[lane] != 0), hi = __ballot_sync(0xffffffffu, src[lane + 32] != 0);
            if (lane == 0) kbits[word] = ((unsigned long long)hi << 32) | lo;
        }
        return;
    }
    const int sub = threadIdx.x & 7;
    const long long r0 = (long long)blockIdx.x * (2 * kPrepRows) + (threadIdx.x >> 3);
    uint4 a[2], b[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const long long r = r0 + u * kPrepRows;
        if (r < rows) { a[u] = out[r * 8 + sub]; b[u] = dout[r * 8 + sub]; }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const long long r = r0 + u * kPrepRows;
        if (r >= rows) continue;                   // (whole groups of eight threads)
        const unsigned* x = reinterpret_cast<const unsigned*>(&a[u]);
        const unsigned* y = reinterpret_cast<const unsigned*>(&b[u]);
        float d = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            d = fmaf(__uint_as_float(x[j] << 16), __uint_as_float(y[j] << 16), d);
            d = fmaf(__uint_as_float(x[j] & 0xffff0000u), __uint_as_float(y[j] & 0xffff0000u), d);
        }
        const unsigned group = 0xffu << (threadIdx.x & 24);
        d += __shfl_xor_sync(group, d, 1);
        d += __shfl_xor_sync(group, d, 2);
        d += __shfl_xor_sync(group, d, 4);
        if (sub == 0) {
            const long long bh = r / N;
            const int tok = (int)(r - bh * N);
            const float l = lse[r];
            const bool alive = l > -INFINITY && (!kpm || kpm[(size_t)(bh / H) * N + tok] != 0);
            float* st = stats + (r / kBlock) * kStatFloats + (r & (kBlock - 1));
            st[0] = alive ? -l * 1.4426950408889634f : -INFINITY;
            st[kBlock] = alive ? -d : 0.f;
        }
    }
}

struct KernelDevice {
    bool ready = false;
    int sm_count = 0;
};
std::mutex g_bwd_mu;
KernelDevice g_bwd_dev[64];

cudaError_t kernel_setup(int device, int* sm_count) {
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_bwd_mu);
    KernelDevice& d = g_bwd_dev[device];
    if (!d.ready) {
        cudaError_t e = cudaFuncSetAttribute(attn_bwd_sm100_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_bwd_sm100_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return e;
        d.ready = true;
    }
    *sm_count = d.sm_count;
    return cudaSuccess;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

bool attn_bwd_sm100_takes(const BwdArgs& a) {
    const int64_t rows = (int64_t)a.B * a.H * a.N;
    return a.dtype == BIGBIRD_BF16 && a.D == kBlock && a.b == kBlock && rows < (1ll << 31) && (int64_t)a.B * a.H * a.nb * 2 < (1ll << 28);
}

int launch_attn_bwd_sm100(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, cudaMemPool_t pool, int* status, int* launches,
                          cudaError_t* cuda_err) {
    auto fail = [&](cudaError_t e) { *cuda_err = e; return BIGBIRD_ECUDA; };
    int device = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = kernel_setup(device, &sms);
    if (e != cudaSuccess) return fail(e);
    const int BH = a.B * a.H;
    const int64_t rows = (int64_t)BH * a.N;
    CUtensorMap tm_q, tm_k, tm_v, tm_do, tm_dq, tm_dk, tm_dv;
    if (!make_map(&tm_q, a.q, (uint64_t)rows) || !make_map(&tm_k, a.k, (uint64_t)rows) || !make_map(&tm_v, a.v, (uint64_t)rows) ||
        !make_map(&tm_do, a.dout, (uint64_t)rows) || !make_map(&tm_dq, a.dq, (uint64_t)rows) || !make_map(&tm_dk, a.dk, (uint64_t)rows) ||
        !make_map(&tm_dv, a.dv, (uint64_t)rows))
        return fail(cudaErrorInvalidValue);

    // Tiles of global blocks have nb steps where the others have about ten: cut them into parts of about a third of what each
    // SM gets altogether, so that none of them is still running when the rest is done, but no more than one for every 16 steps
    // (rounded up: parts of 11 steps or more), and not at all up to 32 steps: adding the parts up takes about 5 us on the path of
    // the last one (it was 24 when a thread fetched one value after the other), and up to 32 steps that is more than a cut gains.
    // Measured, gradients of B, 12 heads, nb blocks in us: [2, nb 16] 39.7 uncut, 48.2 in two, 52.5 in four; [1, 32] 41.5 uncut, 45.6 in
    // two; four heads [1, 32] 33.6, 34.7; [1, 64] 68.0 uncut, 70.0 in two, 69.6 in three, 70.4 in four, 73.2 in eight; [1, 256] 255 uncut,
    // 232 in two, 231 in three; [3, 16 heads, 96] 345 uncut, 356 in two (the last two under the power cap).  (With three tiles drawn ahead
    // whatever the launch [1, 64] was 93.7 uncut and 74.6 in three, since a CTA with a whole global tile had two more tiles to do.)
    const int64_t steps = (int64_t)a.B * ((int64_t)L.steps.size() + (int64_t)L.steps_t.size() + (int64_t)a.H * L.global_tiles * a.nb);
    const int64_t want = std::max<int64_t>(16, steps / (3 * sms));
    const int want_parts = a.nb <= 32 ? 1 : (int)((a.nb + want - 1) / want);
    const int part_steps = (a.nb + want_parts - 1) / want_parts, parts = (a.nb + part_steps - 1) / part_steps;

    // workspace of this call, on the caller's stream
    const int n_split = parts > 1 ? 2 * BH * L.global_tiles : 0;
    const size_t n_words = a.kpm ? (size_t)a.B * a.nb : 0, n_counters = 1 + (size_t)n_split;
    const size_t off_bits = align256((size_t)BH * a.nb * kStatFloats * sizeof(float));
    const size_t off_cnt = off_bits + align256(n_words * sizeof(unsigned long long));
    const size_t off_part = off_cnt + align256(n_counters * sizeof(int));
    const size_t bytes = off_part + (size_t)n_split * parts * kPartialFloats * sizeof(float);
    unsigned char* ws = nullptr;
    e = cudaMallocFromPoolAsync((void**)&ws, bytes, pool, a.stream);
    if (e != cudaSuccess) return fail(e);

    KernelParams p{};
    p.dq = (__nv_bfloat16*)a.dq;
    p.dk = (__nv_bfloat16*)a.dk;
    p.dv = (__nv_bfloat16*)a.dv;
    p.stats = (const float*)ws;
    p.kbits = a.kpm ? (const unsigned long long*)(ws + off_bits) : nullptr;
    p.counter = (int*)(ws + off_cnt);
    p.arrived = p.counter + 1;
    p.partials = (float*)(ws + off_part);
    p.status = status;
    p.items_q = dl.items + L.global_tiles;
    p.q_stride = L.items_per_head;
    p.items_k = dl.items_t;
    p.steps_q = dl.steps;
    p.steps_k = dl.steps_t;
    p.global_pairs = dl.global_pairs;
    p.sparse_tiles = L.sparse_tiles_per_head;
    p.global_tiles = L.global_tiles;
    p.parts = parts;
    p.part_steps = part_steps;
    p.BH = BH;
    p.H = a.H;
    p.nb = a.nb;
    p.total_work = 2 * BH * (L.global_tiles * parts + L.sparse_tiles_per_head);
    // A tile that is drawn is nobody else's.  CTAs that have drawn three before the others have looked at their first (tiles without a
    // token are through at once, those of global blocks take the longest) decide the end of a launch with few tiles, so there the next
    // one is drawn when the loads of the last are under way, which is in time: six steps of them are in the ring.  Unless that is all
    // the tile has.  Gradients, three ahead / one, us: [2, 12, 1024] (2.6 tiles per CTA) with 341 and 1004 tokens 44.9 / 34.8, full 44.8 / 40.1,
    // [1, 12, 2048] (2.6) 58.5 / 42.0, [4, 12, 1536] (7.8) 92.1 / 90.7; [4, 12, 2048] (10.4) 118.8 / 118.2 and without random blocks
    // 84.1 / 85.9; [4, 12, 384] (1.9 tiles of six steps) 22.7 / 23.6.
    p.ahead = p.total_work < 8 * sms && a.nb > kRing ? 1 : kSlots;
    p.scale = a.scale;
    p.scale_log2 = a.scale * 1.4426950408889634f;

    const int row_ctas = (int)((rows + 2 * kPrepRows - 1) / (2 * kPrepRows));
    const int extra = (int)std::min<size_t>(64, 1 + n_words / 64 + n_counters / 2048);
    e = launch_chained(attn_bwd_prepare_kernel, (unsigned)(row_ctas + extra), kPrepThreads, 0, a.stream, (const uint4*)a.out, (const uint4*)a.dout, a.lse, a.kpm,
                       (float*)ws, (unsigned long long*)(ws + off_bits), p.counter, (int)n_counters, (long long)rows, (int)a.N, a.H, row_ctas, (int)n_words);
    if (e == cudaSuccess) {
        ++*launches;
        // Shared steps where they make the sparse tiles' steps fewer by more than a fifth: what they cost every step (the places of Y are
        // counted, three more ballots a list, more code) is more than they gain below.  Measured, a step for each block / shared, us:
        // [8, 12, 4096] (28 % fewer) 483 / 474 under the power cap, [2, 12, 4096] 128.4 / 124.3, [4, 12, 4096] without random blocks, w = 1
        // (25 %) 140 / 137, [3, 16, 1024] (21 %) 65.8 / 64.7; [8, 12, 4224] ETC (16 %) 334 / 346, [3, 16, 512] (none) 34.9 / 36.0.
        const bool share = 5 * (L.tile_blocks - L.tile_steps_shared) > L.tile_blocks;
        e = launch_chained(share ? attn_bwd_sm100_kernel<true> : attn_bwd_sm100_kernel<false>, (unsigned)std::min(sms, p.total_work), kThreads, kSmemBytes, a.stream, tm_q, tm_k, tm_v, tm_do, tm_dq, tm_dk, tm_dv, p);
        if (e == cudaSuccess) ++*launches;
    }
    const cudaError_t ef = cudaFreeAsync(ws, a.stream);
    if (e == cudaSuccess) e = ef;
    return e == cudaSuccess ? BIGBIRD_OK : fail(e);
}

}  // namespace bigbird
