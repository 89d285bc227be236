// Host-side attention-graph layout and the tile schedule derived from it.
#pragma once
#include <cstdint>
#include <mutex>
#include <vector>

namespace bigbird {

// One step of a tile's key sweep.  A tile stacks two query blocks (upper half = rows 0..b-1, lower half =
// rows b..2b-1).  A step names one key block and which halves of the tile attend it.
struct Step {
    int32_t c;      // key block
    int32_t who;    // kBothHalves, kUpperHalf or kLowerHalf
};
constexpr int32_t kBothHalves = 0;
constexpr int32_t kUpperHalf = 1;
constexpr int32_t kLowerHalf = 2;
constexpr int32_t kNoBlock = -1;

// A tile of two query blocks and a contiguous range of steps, in the form in which bigbird_layout_schedule exports it.  (Launches may
// cut the tiles of global blocks into parts, by what else there is to do; the layout keeps them whole.)
struct Item {
    int32_t qa;          // query block of the upper half
    int32_t qb;          // query block of the lower half, or kNoBlock
    int32_t step_begin;  // index into the head's step array
    int32_t step_count;
    int32_t part;        // -1
    int32_t nparts;      // 1
    int32_t tile;        // index among the head's global tiles (0 for the others)
    int32_t pad_;
};

struct DeviceLayout {
    int device = -1;
    int32_t* row_ptr = nullptr;
    int32_t* col_idx = nullptr;
    int32_t* col_ptr = nullptr;
    int32_t* row_idx = nullptr;
    Item* items = nullptr;
    Step* steps = nullptr;
    Item* items_t = nullptr;           // tiles of key blocks over the transposed lists
    Step* steps_t = nullptr;
    int32_t* global_pairs = nullptr;   // [global_tiles * 2]
    int32_t* block_order = nullptr;    // [nb]
    void* block = nullptr;             // the one allocation that holds the arrays above
};

}  // namespace bigbird

struct bigbird_layout {
    int64_t N;
    int b, w, g, r, H, mode;
    uint64_t seed;
    uint64_t uid;                              // unique per handle for the life of the process, never 0
    int nb;
    // CSR over rows h*nb + j (the exported product)
    std::vector<int32_t> row_ptr;
    std::vector<int32_t> col_idx;
    // the same graph by key block: rows h*nb + c list, ascending, the query blocks that attend key block c
    std::vector<int32_t> col_ptr;
    std::vector<int32_t> row_idx;
    // tile schedule: per head the same number of items, the tiles of global blocks first
    int items_per_head = 0;
    int global_tiles = 0;                      // of two global blocks each
    std::vector<bigbird::Item> items;          // [H * items_per_head], step_begin relative to the head's first step
    std::vector<bigbird::Item> items_abs;      // the same with step_begin made absolute (what the kernel reads)
    std::vector<int32_t> step_base;            // [H] offset of the head's steps in `steps`
    std::vector<bigbird::Step> steps;
    // the same for tiles that stack two key blocks and walk the query blocks that attend them (b == 64 only); global
    // key blocks have no list, every query block attends them
    int sparse_tiles_per_head = 0;
    std::vector<int32_t> global_pairs;         // [global_tiles * 2], the last entry kNoBlock if their number is odd
    int n_globals = 0;                         // global blocks, and all blocks with the global ones first
    std::vector<int32_t> block_order;
    std::vector<bigbird::Item> items_t;        // [H * sparse_tiles_per_head], step_begin absolute
    std::vector<bigbird::Step> steps_t;
    // blocks in the lists of the sparse tiles of both kinds, and how many steps they are where a block of the upper half only and one of
    // the lower half only share one (b == 64 only)
    int64_t tile_blocks = 0, tile_steps_shared = 0;
    // device copies, made on first use
    mutable std::mutex mu;
    mutable bigbird::DeviceLayout dev;
};

namespace bigbird {
// Builds CSR and schedule; returns 0 or a negative BIGBIRD_* code.
int build_layout_host(bigbird_layout* L);
}
