// Attention-graph layout of BigBird (arXiv 2007.14062, Sec. 2 and App. D) and the tile schedule the
// tensor-core kernel walks.  Host code only.
#include "layout.h"

#include <algorithm>
#include <atomic>
#include <new>
#include <utility>

#include "../../include/bigbird.h"

namespace bigbird {
namespace {

// SplitMix64 (Steele, Lea, Flood 2014): the generator named by the layout spec in bigbird.h.
struct SplitMix64 {
    uint64_t s;
    explicit SplitMix64(uint64_t key) : s(key) {}
    uint64_t next() {
        s += 0x9E3779B97F4A7C15ull;
        uint64_t z = s;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    }
    // uniform integer in [0, m): floor(z * m / 2^64)
    uint64_t below(uint64_t m) { return (uint64_t)(((unsigned __int128)next() * m) >> 64); }
};

void global_flags(const bigbird_layout& L, std::vector<uint8_t>& is_global) {
    is_global.assign(L.nb, 0);
    if (L.mode == BIGBIRD_ETC) {
        for (int c = 0; c < L.g; ++c) is_global[c] = 1;             // Sec. 2, ETC: the g prepended tokens
    } else {
        const int first = (L.g + 1) / 2, last = L.g / 2;            // Sec. 2, ITC: a subset G of existing tokens
        for (int c = 0; c < first; ++c) is_global[c] = 1;
        for (int c = L.nb - last; c < L.nb; ++c) is_global[c] = 1;
    }
}

// Key blocks of one non-global query block: window (App. D item 2), global columns (item 3), random (item 1).
// Works on the few blocks of the row and not on all nb of them: position i of the ascending candidate list (the blocks that
// are neither in the window nor global) is i plus the excluded blocks before it, and of the shuffled list only the entries
// that a swap has moved are kept.
// (Rows with many random blocks write the list out: finding an entry among the moved ones is a search.)
struct RowScratch {
    std::vector<int32_t> taken;                            // window and global blocks, ascending
    std::vector<int32_t> all;                              // the candidate list, if written out
    std::vector<std::pair<uint64_t, int32_t>> moved;       // (position, block) of the entries that differ from the ascending list
};
void sparse_row(const bigbird_layout& L, const std::vector<int32_t>& globals, int h, int j, RowScratch& s, std::vector<int32_t>& out) {
    const int nb = L.nb, hw = (L.w - 1) / 2;
    const int lo = std::max(0, j - hw), hi = std::min(nb - 1, j + hw);
    std::vector<int32_t>& taken = s.taken;
    taken.clear();
    for (size_t i = 0;; ++i) {                             // merge of the window with the ascending global blocks
        if (i == globals.size() || globals[i] >= lo) {
            for (int c = lo; c <= hi; ++c) taken.push_back(c);
            for (; i < globals.size(); ++i)
                if (globals[i] > hi) taken.push_back(globals[i]);
            break;
        }
        taken.push_back(globals[i]);
    }
    const size_t row_begin = out.size();
    out.insert(out.end(), taken.begin(), taken.end());
    const uint64_t m = (uint64_t)nb - taken.size(), take = std::min<uint64_t>((uint64_t)L.r, m);
    if (take == 0) return;
    auto ascending = [&](uint64_t i) {
        int32_t c = (int32_t)i;
        for (int32_t e : taken) {
            if (e > c) break;
            ++c;
        }
        return c;
    };
    SplitMix64 gen((L.seed << 40) ^ ((uint64_t)h << 20) ^ (uint64_t)j);
    if (take > 32) {
        s.all.clear();
        size_t i = 0;
        for (int32_t c = 0; c < nb; ++c) {
            if (i < taken.size() && taken[i] == c) ++i;
            else s.all.push_back(c);
        }
        for (uint64_t t = 0; t < take; ++t) std::swap(s.all[t], s.all[t + gen.below(m - t)]);
        out.insert(out.end(), s.all.begin(), s.all.begin() + take);
        std::sort(out.begin() + row_begin, out.end());
        return;
    }
    s.moved.clear();
    auto entry = [&](uint64_t i) -> std::pair<uint64_t, int32_t>* {
        for (auto& e : s.moved)
            if (e.first == i) return &e;
        return nullptr;
    };
    for (uint64_t t = 0; t < take; ++t) {                  // swap entries t and p; entry t is final afterwards
        const uint64_t p = t + gen.below(m - t);
        auto *et = entry(t), *ep = entry(p);
        const int32_t ct = et ? et->second : ascending(t), cp = ep ? ep->second : ascending(p);
        out.push_back(cp);
        if (p != t) {
            if (ep) ep->second = ct;
            else s.moved.emplace_back(p, ct);
        }
    }
    std::sort(out.begin() + row_begin, out.end());
}

// Steps of a tile that stacks rows qa (upper half) and qb (lower half, or kNoBlock) of one head's lists: the merge of the
// two ascending lists.
struct TileScratch {
    std::vector<int32_t> both, pa, pb;
};
void sparse_tile(const std::vector<int32_t>& ptr, const std::vector<int32_t>& idx, size_t row0, int qa, int qb, TileScratch& t,
                 std::vector<Step>& steps) {
    const int32_t ea = ptr[row0 + qa + 1];
    int32_t ia = ptr[row0 + qa];
    if (qb == kNoBlock) {
        for (; ia < ea; ++ia) steps.push_back(Step{idx[ia], kBothHalves});
        return;
    }
    const int32_t eb = ptr[row0 + qb + 1];
    int32_t ib = ptr[row0 + qb];
    t.both.clear();
    t.pa.clear();
    t.pb.clear();
    while (ia < ea || ib < eb) {
        if (ib == eb || (ia < ea && idx[ia] < idx[ib])) t.pa.push_back(idx[ia++]);
        else if (ia == ea || idx[ib] < idx[ia]) t.pb.push_back(idx[ib++]);
        else { t.both.push_back(idx[ia]); ++ia; ++ib; }
    }
    // shared, upper-only and lower-only key blocks take turns, so that any run of three entries gives both halves of the tile
    // about the same amount of work.  (The forward kernel takes two entries at a time: an upper-only and a lower-only block are in
    // one such pair in 658 of the 2221 pairs of a base layout's sparse tiles, 12 heads.)
    const size_t ns = std::max(t.both.size(), std::max(t.pa.size(), t.pb.size()));
    for (size_t s = 0; s < ns; ++s) {
        if (s < t.both.size()) steps.push_back(Step{t.both[s], kBothHalves});
        if (s < t.pa.size()) steps.push_back(Step{t.pa[s], kUpperHalf});
        if (s < t.pb.size()) steps.push_back(Step{t.pb[s], kLowerHalf});
    }
}

}  // namespace

int build_layout_host(bigbird_layout* L) {
    const int nb = L->nb, H = L->H;
    std::vector<uint8_t> is_global;
    std::vector<int32_t> globals;
    RowScratch row_scratch;
    global_flags(*L, is_global);
    for (int c = 0; c < nb; ++c)
        if (is_global[c]) globals.push_back(c);

    // ---- CSR ------------------------------------------------------------------------------------
    L->row_ptr.assign(1, 0);
    L->col_idx.clear();
    for (int h = 0; h < H; ++h) {
        for (int j = 0; j < nb; ++j) {
            if (is_global[j]) {
                for (int c = 0; c < nb; ++c) L->col_idx.push_back(c);       // global rows attend everything
            } else {
                sparse_row(*L, globals, h, j, row_scratch, L->col_idx);
            }
            if (L->col_idx.size() > (size_t)INT32_MAX) return BIGBIRD_EUNSUPPORTED;
            L->row_ptr.push_back((int32_t)L->col_idx.size());
        }
    }

    // ---- the graph by key block (what the gradients of K and V walk) ----------------------------
    L->col_ptr.assign((size_t)H * nb + 1, 0);
    L->row_idx.assign(L->col_idx.size(), 0);
    for (int h = 0; h < H; ++h)
        for (int j = 0; j < nb; ++j)
            for (int32_t e = L->row_ptr[(size_t)h * nb + j]; e < L->row_ptr[(size_t)h * nb + j + 1]; ++e)
                ++L->col_ptr[(size_t)h * nb + L->col_idx[e] + 1];
    for (size_t i = 0; i < (size_t)H * nb; ++i) L->col_ptr[i + 1] += L->col_ptr[i];
    {
        std::vector<int32_t> fill(L->col_ptr.begin(), L->col_ptr.end() - 1);
        for (int h = 0; h < H; ++h)
            for (int j = 0; j < nb; ++j)                                     // ascending j: each list comes out sorted
                for (int32_t e = L->row_ptr[(size_t)h * nb + j]; e < L->row_ptr[(size_t)h * nb + j + 1]; ++e)
                    L->row_idx[fill[(size_t)h * nb + L->col_idx[e]]++] = j;
    }

    // ---- tile schedule ----------------------------------------------------------------------------
    // Query blocks are stacked two by two into 2b-row tiles: the global blocks among themselves (every key
    // block is attended by both halves), the others in ascending order.  A step is one key block together
    // with the halves of the tile that attend it.
    std::vector<int> gq, sq;
    for (int j = 0; j < nb; ++j) (is_global[j] ? gq : sq).push_back(j);
    const int n_gtiles = ((int)gq.size() + 1) / 2, n_stiles = ((int)sq.size() + 1) / 2;
    L->global_tiles = n_gtiles;
    L->items_per_head = n_gtiles + n_stiles;
    L->items.clear();
    L->steps.clear();
    L->step_base.clear();
    TileScratch tmp;
    for (int h = 0; h < H; ++h) {
        const int32_t base = (int32_t)L->steps.size();
        L->step_base.push_back(base);
        auto rel = [&]() { return (int32_t)L->steps.size() - base; };
        for (int t = 0; t < n_gtiles; ++t) {                   // (exported; the kernels know the list of a global block)
            Item it{};
            it.qa = gq[2 * t];
            it.qb = 2 * t + 1 < (int)gq.size() ? gq[2 * t + 1] : kNoBlock;
            it.step_begin = rel();
            it.step_count = nb;
            it.part = -1;
            it.nparts = 1;
            it.tile = t;
            for (int c = 0; c < nb; ++c) L->steps.push_back(Step{c, kBothHalves});
            L->items.push_back(it);
        }
        for (int t = 0; t < n_stiles; ++t) {
            Item it{};
            it.qa = sq[2 * t];
            it.qb = 2 * t + 1 < (int)sq.size() ? sq[2 * t + 1] : kNoBlock;
            it.step_begin = rel();
            it.part = -1;
            it.nparts = 1;
            sparse_tile(L->row_ptr, L->col_idx, (size_t)h * nb, it.qa, it.qb, tmp, L->steps);
            it.step_count = rel() - it.step_begin;
            L->items.push_back(it);
        }
    }
    L->items_abs = L->items;
    for (int h = 0; h < H; ++h)
        for (int i = 0; i < L->items_per_head; ++i) L->items_abs[(size_t)h * L->items_per_head + i].step_begin += L->step_base[h];

    // ---- what the tensor-core gradients walk besides: pairs of key blocks with the query blocks that attend them ----
    // (the global key blocks are attended by every query block, so their tiles need no list)
    L->sparse_tiles_per_head = n_stiles;
    L->n_globals = (int)gq.size();
    L->block_order = gq;
    L->block_order.insert(L->block_order.end(), sq.begin(), sq.end());
    L->global_pairs.assign(2 * (size_t)n_gtiles, kNoBlock);
    for (size_t i = 0; i < gq.size(); ++i) L->global_pairs[i] = gq[i];
    L->items_t.clear();
    L->steps_t.clear();
    if (L->b == 64) {
        for (int h = 0; h < H; ++h)
            for (int t = 0; t < n_stiles; ++t) {
                Item it{};
                it.qa = sq[2 * t];
                it.qb = 2 * t + 1 < (int)sq.size() ? sq[2 * t + 1] : kNoBlock;
                it.step_begin = (int32_t)L->steps_t.size();
                it.part = -1;
                it.nparts = 1;
                sparse_tile(L->col_ptr, L->row_idx, (size_t)h * nb, it.qa, it.qb, tmp, L->steps_t);
                it.step_count = (int32_t)L->steps_t.size() - it.step_begin;
                L->items_t.push_back(it);
            }
        auto count = [&](const Item& it, const std::vector<Step>& steps) {
            int64_t n[3] = {0, 0, 0};
            for (int i = 0; i < it.step_count; ++i) ++n[steps[(size_t)it.step_begin + i].who];
            L->tile_blocks += it.step_count;
            L->tile_steps_shared += n[kBothHalves] + std::max(n[kUpperHalf], n[kLowerHalf]);
        };
        for (size_t i = 0; i < L->items_abs.size(); ++i)
            if ((int)(i % L->items_per_head) >= n_gtiles) count(L->items_abs[i], L->steps);
        for (const Item& it : L->items_t) count(it, L->steps_t);
    }
    return BIGBIRD_OK;
}

}  // namespace bigbird

extern "C" {

int bigbird_build_layout(int64_t N, int b, int w, int g, int r, uint64_t seed, int H, int mode,
                         bigbird_layout** out_layout) {
    if (!out_layout) return BIGBIRD_EINVAL;
    *out_layout = nullptr;
    if (N <= 0 || b <= 0 || N % b != 0) return BIGBIRD_EINVAL;
    const int64_t nb64 = N / b;
    if (nb64 >= (1 << 20) || H < 1 || H >= (1 << 20)) return BIGBIRD_EINVAL;     // stream-key field widths
    if (w < 1 || (w % 2) == 0 || g < 0 || g > nb64 || r < 0) return BIGBIRD_EINVAL;
    if (mode != BIGBIRD_ITC && mode != BIGBIRD_ETC) return BIGBIRD_EINVAL;
    if (seed >= (1ull << 24)) return BIGBIRD_EINVAL;                              // seed << 40 must not overflow
    bigbird_layout* L = new (std::nothrow) bigbird_layout();
    if (!L) return BIGBIRD_ENOMEM;
    L->N = N; L->b = b; L->w = w; L->g = g; L->r = r; L->H = H; L->mode = mode; L->seed = seed;
    L->nb = (int)nb64;
    static std::atomic<uint64_t> next_uid{1};
    L->uid = next_uid.fetch_add(1);
    int rc;
    try {
        rc = bigbird::build_layout_host(L);
    } catch (const std::bad_alloc&) {
        rc = BIGBIRD_ENOMEM;
    }
    if (rc != BIGBIRD_OK) { delete L; return rc; }
    *out_layout = L;
    return BIGBIRD_OK;
}

int bigbird_layout_nnz(const bigbird_layout* L, int64_t* nnz) {
    if (!L || !nnz) return BIGBIRD_EINVAL;
    *nnz = (int64_t)L->col_idx.size();
    return BIGBIRD_OK;
}

int bigbird_layout_export(const bigbird_layout* L, int32_t* row_ptr, int32_t* col_idx) {
    if (!L || !row_ptr || !col_idx) return BIGBIRD_EINVAL;
    std::copy(L->row_ptr.begin(), L->row_ptr.end(), row_ptr);
    std::copy(L->col_idx.begin(), L->col_idx.end(), col_idx);
    return BIGBIRD_OK;
}

int bigbird_layout_export_transposed(const bigbird_layout* L, int32_t* col_ptr, int32_t* row_idx) {
    if (!L || !col_ptr || !row_idx) return BIGBIRD_EINVAL;
    std::copy(L->col_ptr.begin(), L->col_ptr.end(), col_ptr);
    std::copy(L->row_idx.begin(), L->row_idx.end(), row_idx);
    return BIGBIRD_OK;
}

const char* bigbird_strerror(int code) {
    switch (code) {
        case BIGBIRD_OK: return "ok";
        case BIGBIRD_EINVAL: return "invalid argument";
        case BIGBIRD_EUNSUPPORTED: return "unsupported shape or dtype";
        case BIGBIRD_ECUDA: return "CUDA call failed";
        case BIGBIRD_ETIMEOUT: return "bounded device wait expired";
        case BIGBIRD_ENOMEM: return "out of memory";
        case BIGBIRD_ELIMIT: return "problem exceeds the fixed scratch of the no-allocation entry point";
        case BIGBIRD_EINTERNAL: return "index check failed inside a kernel (checked build)";
        default: return "unknown error";
    }
}

}  // extern "C"

extern "C" int bigbird_layout_schedule(const bigbird_layout* L, int32_t* sizes, int32_t* items, int32_t* step_base,
                                       int32_t* steps) {
    if (!L || !sizes) return BIGBIRD_EINVAL;
    static_assert(sizeof(bigbird::Item) == 8 * sizeof(int32_t), "Item is exported as 8 int32");
    static_assert(sizeof(bigbird::Step) == 2 * sizeof(int32_t), "Step is exported as 2 int32");
    sizes[0] = L->items_per_head;
    sizes[1] = L->global_tiles;
    sizes[2] = (int32_t)L->steps.size();
    sizes[3] = L->H;
    if (items) std::copy((const int32_t*)L->items.data(), (const int32_t*)(L->items.data() + L->items.size()), items);
    if (step_base) std::copy(L->step_base.begin(), L->step_base.end(), step_base);
    if (steps) std::copy((const int32_t*)L->steps.data(), (const int32_t*)(L->steps.data() + L->steps.size()), steps);
    return BIGBIRD_OK;
}
