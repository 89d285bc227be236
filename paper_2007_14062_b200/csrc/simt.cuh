// Shared pieces of the CUDA-core kernels: tile shapes, staging of rows in shared memory, the two register-tiled products, and
// the division of the work between the CTAs of a cluster.
//
// A CTA owns up to TM * TY rows of one block (TY = threads / 16 rows of threads, TM rows each) and walks the tokens of the
// blocks in the rows' list, kc at a time, as one sequence: a chunk may begin in one block and end in the next, so block sizes
// that are no multiple of the chunk waste nothing.  A thread's micro-tile is TM rows by kc / 16 tokens (scores) or by D / 16
// columns (sums), which reads 12 to 15 shared-memory wavefronts per 64 to 112 FMAs of a warp.
//
// The tiles of global blocks have a list as long as the sequence.  The CTAs of a cluster share one such tile, each taking a
// contiguous share of its chunks, and add up their results through distributed shared memory in the order of their ranks (no
// scratch, no atomics, the same bits every time); the other tiles go to one CTA each.
#pragma once
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math_constants.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"
#include "../../include/bigbird.h"

namespace bigbird {
namespace {
namespace cg = cooperative_groups;

__device__ __forceinline__ void store2(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
__device__ __forceinline__ void store2(__nv_bfloat16* p, float a, float b) { *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b); }
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Four values of a row into shared memory: asynchronously if no conversion is needed; zeros if src is null.
__device__ __forceinline__ void stage4(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (src) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void stage4(float* dst, const __nv_bfloat16* src) {
    *reinterpret_cast<float4*>(dst) = src ? load4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// The part of a list that this CTA walks, as tokens first .. last - 1 of the concatenated blocks.
struct Walk {
    const int32_t* list;
    int b;
    unsigned inv_b;        // floor(2^32 / b), 2^32 - 1 for b = 1
    int first, last;
    // token of the sequence behind position i; only for first <= i < last
    __device__ __forceinline__ int token(int i) const {
        int e = (int)__umulhi((unsigned)i, inv_b), r = i - e * b;      // e is i / b or one less
        if (r >= b) { ++e; r -= b; }
        return list[e] * b + r;
    }
};

// Rows i0 .. i0 + kc - 1 of the walk into shared memory, ld floats apart; rows past its end become zeros.
template <int D, typename T>
__device__ __forceinline__ void stage_chunk(float* dst, int ld, const T* src, const Walk& w, int i0, int kc) {
    constexpr int Q = D / 4;
    for (int idx = threadIdx.x; idx < kc * Q; idx += blockDim.x) {
        const int r = idx / Q, c = idx % Q, i = i0 + r;
        stage4(dst + r * ld + 4 * c, i < w.last ? src + (size_t)w.token(i) * D + 4 * c : (const T*)nullptr);
    }
}
// `rows` consecutive rows, of which `have` exist.
template <int D, typename T>
__device__ __forceinline__ void stage_rows(float* dst, int ld, const T* src, int rows, int have) {
    constexpr int Q = D / 4;
    for (int idx = threadIdx.x; idx < rows * Q; idx += blockDim.x) {
        const int r = idx / Q, c = idx % Q;
        stage4(dst + r * ld + 4 * c, r < have ? src + (size_t)r * D + 4 * c : (const T*)nullptr);
    }
}

// Pairs of floats on the packed fp32 pipe: half the instructions for the same FMAs.  (A plain FFMA of three registers runs at
// 59 TFLOP/s on this part, as the packed one does, but takes every issue slot that the shared-memory loads need.)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair(float a, float b) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ float2 unpair(f32x2 x) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x)); return r; }
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ void mul2(f32x2& x, f32x2 a) { asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(x) : "l"(a)); }

// acc[i][j] = sum_d a[i][d] b[16 j][d] over rows lda and ldb floats apart.  Even and odd d are summed apart and added at the end.
// The loops of both products are bound by the latency of shared memory, so they are unrolled as far as it helps: [2, 12, 52 x 84, 64]
// forward and gradients 2814 us with 4 rounds here and 2 in sum_tile, 2702 with 8 and 4, 2673 with 16 and 4, 2684 with 16 and 8;
// [2, 8, 2560, 128] 308 with 4 and 2, 304.7 with 4 and 4, 301.5 with 8 and 8.  That some instances spill a few registers outside of these
// loops then (up to 200 bytes) costs less than it gains.  [2, 12, about 4096 tokens], 4 and 2 / as it is, forward and gradients: blocks
// of 64 with D = 32 325 / 313 and 1040 / 1022, with D = 64 521 / 501 and 1713 / 1660, with D = 128 901 / 872 and 3465 / 3416; with D = 32
// blocks of 16 111 / 107 and 353 / 342, of 96 428 / 420 and 1442 / 1420, of 169 787 / 772 and 2513 / 2468.
template <int TM, int TN, int D>
__device__ __forceinline__ void dot_tile(float (&acc)[TM][TN], const float* a, int lda, const float* b, int ldb) {
    f32x2 s[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) s[i][j] = 0;
#pragma unroll (D <= 64 ? 16 : 8)
    for (int d = 0; d < D; d += 4) {
        ulonglong2 x[TM], y[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) x[i] = *reinterpret_cast<const ulonglong2*>(a + i * lda + d);
#pragma unroll
        for (int j = 0; j < TN; ++j) y[j] = *reinterpret_cast<const ulonglong2*>(b + 16 * j * ldb + d);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                fma2(s[i][j], x[i].x, y[j].x);
                fma2(s[i][j], x[i].y, y[j].y);
            }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const float2 r = unpair(s[i][j]);
            acc[i][j] = r.x + r.y;
        }
}

// A thread's columns of a D-wide row: D / 16 of them, in groups of 4 (2 for D = 32), kept as pairs of adjacent ones.
template <int D>
struct Cols {
    static constexpr int G = D == 32 ? 2 : 4;      // columns per group, adjacent
    static constexpr int NG = D / 16 / G;          // groups, 16 G apart
    static constexpr int N = G * NG / 2;           // pairs
    __device__ static __forceinline__ int at(int tx, int c) { return G * tx + (2 * c / G) * 16 * G + 2 * c % G; }     // first column of pair c
};

// acc[i][c] += sum_t p[i][t] v[t][columns c] over kc tokens; v points at row 0.
template <int TM, int D>
__device__ __forceinline__ void sum_tile(f32x2 (&acc)[TM][Cols<D>::N], const float* p, int ldp, const float* v, int ldv, int kc, int tx) {
    using C = Cols<D>;
#pragma unroll (D <= 64 ? 4 : 8)
    for (int t = 0; t < kc; t += 4) {
        float4 w[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) w[i] = *reinterpret_cast<const float4*>(p + i * ldp + t);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            f32x2 x[C::N];
#pragma unroll
            for (int g = 0; g < C::NG; ++g) {
                const float* src = v + (t + u) * ldv + C::at(tx, g * C::G / 2);
                if constexpr (C::G == 4) {
                    const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(src);
                    x[2 * g] = y.x; x[2 * g + 1] = y.y;
                } else {
                    x[0] = *reinterpret_cast<const f32x2*>(src);
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const float f = u == 0 ? w[i].x : u == 1 ? w[i].y : u == 2 ? w[i].z : w[i].w;
                const f32x2 ff = pair(f, f);
#pragma unroll
                for (int c = 0; c < C::N; ++c) fma2(acc[i][c], ff, x[c]);
            }
        }
    }
}
// The sums times f, or zeros: a select, since what stands in padded rows may be anything, and with it their sums.
template <int D, typename T>
__device__ __forceinline__ void store_cols(T* row, const f32x2* acc, float f, int tx, bool zero = false) {
    using C = Cols<D>;
#pragma unroll
    for (int c = 0; c < C::N; ++c) {
        const float2 x = unpair(acc[c]);
        store2(row + C::at(tx, c), zero ? 0.f : x.x * f, zero ? 0.f : x.y * f);
    }
}

// Over the 16 threads that share a row.
__device__ __forceinline__ float row_max16(float x) {
#pragma unroll
    for (int s = 1; s < 16; s <<= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, s));
    return x;
}
__device__ __forceinline__ float row_sum16(float x) {
#pragma unroll
    for (int s = 1; s < 16; s <<= 1) x += __shfl_xor_sync(0xffffffffu, x, s);
    return x;
}

// ------------------------------------------------------------------------------------------------ work division
// Tiles of global blocks first (they are the longest): one cluster each.  Then the others: one CTA each, unless there are so
// few tiles that they are shared as well.
struct Tiling {
    int rows;              // rows of a tile (the last one of a block may have fewer)
    int tiles;             // per block
    int split_blocks;      // leading entries of `order` whose tiles are shared by a cluster
    int cluster;
    int BH, H, nb, b;
    unsigned inv_b;        // see Walk
    const int32_t* order;  // [nb] global blocks first
};
struct Tile {
    int bh, blk, row0, rank, shares;
};
__device__ __forceinline__ bool find_tile(const Tiling& t, Tile& out) {
    const unsigned cl = (unsigned)t.cluster, cluster_id = blockIdx.x / cl, rank = blockIdx.x % cl;
    const unsigned per_block = (unsigned)t.BH * t.tiles, shared = t.split_blocks * per_block;
    unsigned x;
    if (cluster_id < shared) {
        x = cluster_id;
        out.rank = (int)rank;
        out.shares = (int)cl;
    } else {
        x = shared + (cluster_id - shared) * cl + rank;
        out.rank = 0;
        out.shares = 1;
        if (x >= (unsigned)t.nb * per_block) return false;
    }
    const unsigned o = x / per_block, y = x - o * per_block;
    out.bh = (int)(y / t.tiles);
    out.row0 = (int)(y % t.tiles) * t.rows;
    out.blk = t.order[o];
    return true;
}
// What a CTA walks of a list: whole chunks of kc tokens, shared out evenly.
__device__ __forceinline__ Walk share_walk(const Tiling& t, const int32_t* ptr, const int32_t* idx, const Tile& tile, int kc) {
    const int64_t at = (int64_t)(tile.bh % t.H) * t.nb + tile.blk;
    const int begin = ptr[at], tokens = (ptr[at + 1] - begin) * t.b, chunks = (tokens + kc - 1) / kc;
    return Walk{idx + begin, t.b, t.inv_b, min(tokens, chunks * tile.rank / tile.shares * kc), min(tokens, chunks * (tile.rank + 1) / tile.shares * kc)};
}

struct Shape {
    Tiling t;
    int threads, grid;
};
// Two rows per thread where four would leave half of the GPU idle; else six where that covers a block with no more padding than four would
// (the larger micro-tile reads less shared memory per FMA).  Seven where that pads no more than six and gives a CTA all of its twelve
// rows of threads: at most 192 threads have 168 registers each, and two CTAs of six warps fill the four sub-partitions evenly (84 rows:
// six warps instead of seven).  With fewer warps it is the slower one: [2, 12, about 4096 tokens, 64], six / seven rows per thread,
// forward and gradients in us: blocks of 84 688 / 679 and 2320 / 2297, of 160 1202 / 1180 and 3926 / 3850, of 70 (five warps) 595 / 674 and 2028 /
// 2269, of 140 1080 / 1219 and 3593 / 3992, of 200 1505 / 1662 and 5095 / 5697, of 42 (three) 424 / 420 and 1395 / 1584.  Four for D = 128,
// whose sums take twice the registers.
constexpr int max_threads(int tm) { return tm == 7 ? 192 : 256; }
inline int row_tiles(int tm, int b) { return (b + max_threads(tm) / 16 * tm - 1) / (max_threads(tm) / 16 * tm); }
// Rows of threads of a CTA: an even number, so that a warp has two.
inline int thread_rows(int tm, int b) {
    const int tiles = row_tiles(tm, b), rows = (b + tiles - 1) / tiles;
    return std::max(2, ((rows + tm - 1) / tm + 1) / 2 * 2);
}
inline int padded_rows(int tm, int b) { return row_tiles(tm, b) * thread_rows(tm, b) * tm; }
inline int rows_per_thread(const bigbird_layout& L, int BH, int D, int slots) {
    if (2 * (int64_t)BH * L.nb * ((L.b + 63) / 64) <= slots) return 2;
    if (D > 64 || padded_rows(6, L.b) > padded_rows(4, L.b)) return 4;
    return padded_rows(7, L.b) <= padded_rows(6, L.b) && thread_rows(7, L.b) == max_threads(7) / 16 ? 7 : 6;
}

// tm: rows per thread; kc: tokens per chunk; slots: CTAs that fit the GPU at a time.
inline Shape make_shape(int tm, const bigbird_layout& L, const DeviceLayout& dl, int BH, int slots, int kc) {
    Shape s{};
    const int b = L.b, nb = L.nb;
    s.t.tiles = row_tiles(tm, b);
    s.t.rows = (b + s.t.tiles - 1) / s.t.tiles;
    s.threads = 16 * thread_rows(tm, b);
    s.t.BH = BH;
    s.t.H = L.H;
    s.t.nb = nb;
    s.t.b = b;
    s.t.inv_b = b == 1 ? 0xffffffffu : (unsigned)((1ull << 32) / (unsigned)b);
    s.t.order = dl.block_order;
    const int64_t tiles = (int64_t)BH * nb * s.t.tiles;
    const int64_t entries = (int64_t)L.col_idx.size();
    const int64_t longest = ((int64_t)nb * b + kc - 1) / kc;                             // chunks of a global tile
    const int64_t mean = entries * b / ((int64_t)L.H * nb * kc);                         // of all tiles
    const int64_t even = entries / L.H * BH * s.t.tiles * b / kc / slots;                // of a slot if the work is spread evenly
    int cl = 1;
    if (2 * tiles <= slots) {
        // the GPU is half empty or worse: all tiles are shared, down to one chunk per CTA (a short fp32 sequence, 16 tiles of 8
        // chunks: a chunk takes an SM at least 2 us)
        while (cl < 8 && 2 * cl * tiles <= slots && 2 * cl <= mean + 1) cl *= 2;
        while (cl < 8 && L.n_globals && longest / cl > std::max<int64_t>(4, 2 * mean)) cl *= 2;
        s.t.split_blocks = nb;
    } else if (L.n_globals > 0) {
        // shares of half an even load, so that a global tile does not outlast the rest
        while (cl < 8 && longest / cl > std::max<int64_t>(4, even / 2)) cl *= 2;
        s.t.split_blocks = L.n_globals;
    }
    if (cl == 1) s.t.split_blocks = 0;
    s.t.cluster = cl;
    const int64_t shared = (int64_t)s.t.split_blocks * BH * s.t.tiles;
    s.grid = (int)((shared + (tiles - shared + cl - 1) / cl) * cl);
    return s;
}
// Once per kernel and device, with that device current.
inline cudaError_t allow_smem(const void* kernel, size_t bytes, std::once_flag (&once)[64]) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[device], [&] { e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); });
    return e;
}
template <typename... Ps, typename... As>
cudaError_t launch_clusters(void (*kernel)(Ps...), const Shape& s, size_t smem, cudaStream_t stream, As... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)s.grid);
    cfg.blockDim = dim3((unsigned)s.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)s.t.cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = s.t.cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace
}  // namespace bigbird
