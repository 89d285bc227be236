// CUDA-core gradients of BigBird attention (arXiv 2007.14062, Eq. (AT) over the block lists of App. D; the paper
// trains through this op, Sec. 4 and App. E.1, and leaves the derivatives to autodiff).  fp32 arithmetic throughout.
//
// With P = softmax(scale q k^T) over the attended valid keys (recomputed here from the saved lse), out = P v and
// delta_i = sum_d dout[i, d] out[i, d]:
//     dv = P^T dout,   dS = P o (dout v^T - delta),   dq = scale dS k,   dk = scale dS^T q.
// One kernel in two forms, launched one after the other:
//     by query block    rows q | dout, chunks k | v of the rows' list:              dq = sum dS k  (and delta of its rows, to scratch)
//     by key block      rows k | v,    chunks q | dout of the transposed list:      dv = sum P dout, dk = sum dS q
// Both kinds of scores are register-tiled products over shared memory, and so are the sums, with P or dS passing through shared
// memory between the 16 threads that share a row.  See simt.cuh for the tile shapes and for how clusters share the long tiles.
// Padded query rows get dq = 0 and give nothing to dk, dv; padded keys get dk = dv = 0.
// Bound by shared-memory latency and the FMA pipes (three products per pair of tokens by query, four by key).  Measured (four lanes per
// row with two exchanges per score before): [2, 12, 52 x 84, 64] with three global blocks 12.16 -> 2.04 ms.
#include "simt.cuh"

namespace bigbird {
namespace {

template <int D>
struct BwdShape {
    static constexpr int KC = D == 128 ? 32 : 64;  // tokens per chunk: two CTAs fit an SM
    static constexpr int LD = D + 4, LDP = KC + 4; // padded rows: 16-byte aligned, and what a warp reads at once falls into different banks
    static size_t smem(int rows_pad) { return sizeof(float) * (2 * (size_t)rows_pad * LD + 2 * (size_t)KC * LD + (size_t)rows_pad * LDP + 2 * (size_t)rows_pad); }
};

// dynamic shared memory: X1, X2 [rows][LD] | Y1, Y2 [KC][LD] | P [rows][LDP] | bias, -delta of the rows
template <typename T, int D, int TM, bool kDkv>
__global__ void __launch_bounds__(max_threads(TM), 2)
attn_bwd_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, const T* __restrict__ out,
                     const float* __restrict__ lse, const T* __restrict__ dout, const int32_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                     const uint8_t* __restrict__ kpm, T* __restrict__ g0, T* __restrict__ g1, float* __restrict__ minus_delta, Tiling tiling,
                     int64_t N, float scale) {
    using S = BwdShape<D>;
    using C = Cols<D>;
    constexpr int KC = S::KC, LD = S::LD, LDP = S::LDP, TN = KC / 16, NA = kDkv ? 2 : 1;
    __shared__ float sbias[KC], sdelta[KC];        // of the chunk's tokens
    extern __shared__ __align__(16) float smem[];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, rows_pad = (blockDim.x >> 4) * TM;
    float* const x1 = smem;
    float* const x2 = x1 + rows_pad * LD;
    float* const y1 = x2 + rows_pad * LD;
    float* const y2 = y1 + KC * LD;
    float* const sp = y2 + KC * LD;
    float* const row_bias = sp + rows_pad * LDP;
    float* const row_delta = row_bias + rows_pad;

    grid_dependency_release();
    grid_dependency_wait();
    Tile tile;
    if (!find_tile(tiling, tile)) return;          // (a CTA without a tile belongs to a cluster that shares none)
    const int b = tiling.b, batch = tile.bh / tiling.H;
    const int64_t base = (int64_t)tile.bh * N * D, base_row = (int64_t)tile.bh * N;
    const int have = min(tiling.rows, b - tile.row0);
    const int tok0 = tile.blk * b + tile.row0;     // first row
    const uint8_t* mask = kpm ? kpm + (int64_t)batch * N : nullptr;
    const Walk w = share_walk(tiling, ptr, idx, tile, KC);
    const T *rows1 = (kDkv ? k : q) + base, *rows2 = (kDkv ? v : dout) + base, *cols1 = (kDkv ? q : k) + base, *cols2 = (kDkv ? dout : v) + base;

    // P = exp(scale s + bias of the row + bias of the token): -lse on the query side, -inf for what takes no part
    auto query_bias = [&](int tok) -> float {
        const float l = lse[base_row + tok];
        return l > -CUDART_INF_F && (!mask || mask[tok] != 0) ? -l : -CUDART_INF_F;
    };
    auto key_bias = [&](int tok) -> float { return !mask || mask[tok] != 0 ? 0.f : -CUDART_INF_F; };
    bool live = false;
    if ((int)threadIdx.x < rows_pad) {             // (a thread per row: there are at least as many)
        const int r = threadIdx.x;
        const float x = r < have ? (kDkv ? key_bias(tok0 + r) : query_bias(tok0 + r)) : -CUDART_INF_F;
        row_bias[r] = x;
        live = x > -CUDART_INF_F;
    }
    live = __syncthreads_or(live);                 // a tile without any live row is zeros
    if (live) {
        stage_rows<D>(x1, LD, rows1 + (int64_t)tok0 * D, rows_pad, have);
        stage_rows<D>(x2, LD, rows2 + (int64_t)tok0 * D, rows_pad, have);
        stage_chunk<D>(y1, LD, cols1, w, w.first, KC);
        stage_chunk<D>(y2, LD, cols2, w, w.first, KC);
    }
    if (!kDkv) {
#pragma unroll 2
        for (int i = 0; i < TM; ++i) {             // -delta of the rows, for this kernel and (once) for the other one
            const int r = ty * TM + i;
            float d = 0.f;
            if (r < have) {
                const int64_t at = base + (int64_t)(tok0 + r) * D;
                for (int c = 4 * tx; c < D; c += 64) {
                    const float4 a = load4(dout + at + c), o = load4(out + at + c);
                    d = fmaf(a.x, o.x, fmaf(a.y, o.y, fmaf(a.z, o.z, fmaf(a.w, o.w, d))));
                }
            }
            __syncwarp();
            d = -row_sum16(d);
            if (tx == 0) {
                row_delta[r] = d;
                if (r < have && tile.rank == 0) minus_delta[base_row + tok0 + r] = d;
            }
        }
    }
    // bias and -delta of a chunk's tokens: threads 0 .. KC - 1 (a CTA of one warp: two each) look one chunk ahead
    float next_bias[2] = {-CUDART_INF_F, -CUDART_INF_F}, next_delta[2] = {0.f, 0.f};
    auto look = [&](int i0, int u) {
        const int i = i0 + 32 * u + (int)threadIdx.x;
        next_bias[u] = -CUDART_INF_F;
        if (i >= w.last) return;
        const int tok = w.token(i);
        next_bias[u] = kDkv ? query_bias(tok) : key_bias(tok);
        if (kDkv) next_delta[u] = minus_delta[base_row + tok];
    };
    auto look_ahead = [&](int i0) {
        if ((int)threadIdx.x < KC) look(i0, 0);
        if (blockDim.x < KC) look(i0, 1);
    };
    if (live) look_ahead(w.first);

    const float *r1 = x1 + ty * TM * LD, *r2 = x2 + ty * TM * LD;
    float* const prow = sp + ty * TM * LDP;
    f32x2 acc[NA][TM][C::N];
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int c = 0; c < C::N; ++c) acc[a][i][c] = 0;
    for (int i0 = w.first; i0 < w.last && live; i0 += KC) {
        if ((int)threadIdx.x < KC) { sbias[threadIdx.x] = next_bias[0]; sdelta[threadIdx.x] = next_delta[0]; }
        if (blockDim.x < KC) { sbias[32 + threadIdx.x] = next_bias[1]; sdelta[32 + threadIdx.x] = next_delta[1]; }
        copy_wait();
        const bool any = __syncthreads_or(fmaxf(next_bias[0], next_bias[1]) > -CUDART_INF_F);
        if (i0 + KC < w.last) look_ahead(i0 + KC);
        if (any) {
            float s[TM][TN];
            dot_tile<TM, TN, D>(s, r1, LD, y1 + tx * LD, LD);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float x = row_bias[ty * TM + i] + sbias[tx + 16 * j];
                    prow[i * LDP + tx + 16 * j] = x > -CUDART_INF_F ? expf(fmaf(s[i][j], scale, x)) : 0.f;
                }
            __syncwarp();                          // a row is read by the half-warp that wrote it
            if (kDkv) {
                sum_tile<TM, D>(acc[NA - 1], prow, LDP, y2, LD, KC, tx);
                __syncwarp();
            }
            dot_tile<TM, TN, D>(s, r2, LD, y2 + tx * LD, LD);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j)       // (this thread's own P)
                    prow[i * LDP + tx + 16 * j] *= s[i][j] + (kDkv ? sdelta[tx + 16 * j] : row_delta[ty * TM + i]);
            __syncwarp();
            sum_tile<TM, D>(acc[0], prow, LDP, y1, LD, KC, tx);
        }
        __syncthreads();                           // the chunk has been read
        if (i0 + KC < w.last) {
            stage_chunk<D>(y1, LD, cols1, w, i0 + KC, KC);
            stage_chunk<D>(y2, LD, cols2, w, i0 + KC, KC);
        }
    }
    copy_wait();

    if (tile.shares > 1) {
        // every CTA of the cluster leaves its sums in its shared memory; each then adds up its share of the rows
        cg::cluster_group cluster = cg::this_cluster();
        __syncthreads();
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int i = 0; i < TM; ++i) store_cols<D>(smem + (a * rows_pad + ty * TM + i) * LD, acc[a][i], 1.f, tx);
        cluster.sync();
        const int per = (have + tile.shares - 1) / tile.shares, r_end = min(have, per * (tile.rank + 1));
        for (int r = per * tile.rank + ty; r < r_end; r += blockDim.x >> 4)
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                f32x2 sum[C::N];
#pragma unroll
                for (int c = 0; c < C::N; ++c) sum[c] = 0;
#pragma unroll
                for (int s = 0; s < 8; ++s) {      // (at most eight shares; their loads are in flight together)
                    if (s >= tile.shares) continue;
                    const float* part = cluster.map_shared_rank(smem, s) + (a * rows_pad + r) * LD;
#pragma unroll
                    for (int c = 0; c < C::N; ++c) fma2(sum[c], pair(1.f, 1.f), *reinterpret_cast<const f32x2*>(part + C::at(tx, c)));
                }
                store_cols<D>((a ? g1 : g0) + base + (int64_t)(tok0 + r) * D, sum, a ? 1.f : scale, tx);
            }
        cluster.sync();                            // nobody leaves while its shared memory is being read
        return;
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = ty * TM + i;
        if (r >= have) continue;
        const int64_t at = base + (int64_t)(tok0 + r) * D;
        store_cols<D>(g0 + at, acc[0][i], scale, tx);
        if (kDkv) store_cols<D>(g1 + at, acc[NA - 1][i], 1.f, tx);
    }
}

template <typename T, int D, int TM, bool kDkv>
cudaError_t launch_one(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms, float* minus_delta) {
    static std::once_flag once[64];
    const cudaError_t e = allow_smem((const void*)attn_bwd_simt_kernel<T, D, TM, kDkv>, BwdShape<D>::smem(max_threads(TM) / 16 * TM), once);
    if (e != cudaSuccess) return e;
    const Shape s = make_shape(TM, L, dl, a.B * a.H, 2 * sms, BwdShape<D>::KC);
    return launch_clusters(attn_bwd_simt_kernel<T, D, TM, kDkv>, s, BwdShape<D>::smem(s.threads / 16 * TM), a.stream, (const T*)a.q, (const T*)a.k,
                           (const T*)a.v, (const T*)a.out, a.lse, (const T*)a.dout, (const int32_t*)(kDkv ? dl.col_ptr : dl.row_ptr),
                           (const int32_t*)(kDkv ? dl.row_idx : dl.col_idx), a.kpm, (T*)(kDkv ? a.dk : a.dq), (T*)a.dv, minus_delta, s.t, a.N, a.scale);
}
template <typename T, int D, int TM>
cudaError_t launch_tm(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms, float* ws) {
    const cudaError_t e = launch_one<T, D, TM, false>(a, L, dl, sms, ws);
    return e == cudaSuccess ? launch_one<T, D, TM, true>(a, L, dl, sms, ws) : e;
}
template <typename T, int D>
cudaError_t launch_d(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms, float* ws) {
    const int tm = rows_per_thread(L, a.B * a.H, D, 2 * sms);
    if (tm == 2) return launch_tm<T, D, 2>(a, L, dl, sms, ws);
    if constexpr (D <= 64) {
        if (tm == 6) return launch_tm<T, D, 6>(a, L, dl, sms, ws);
        if (tm == 7) return launch_tm<T, D, 7>(a, L, dl, sms, ws);
    }
    return launch_tm<T, D, 4>(a, L, dl, sms, ws);
}
template <typename T>
cudaError_t launch_t(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms, float* ws) {
    switch (a.D) {
        case 32: return launch_d<T, 32>(a, L, dl, sms, ws);
        case 64: return launch_d<T, 64>(a, L, dl, sms, ws);
        case 128: return launch_d<T, 128>(a, L, dl, sms, ws);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_attn_bwd_simt(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, cudaMemPool_t pool, int sms, int* launches) {
    // workspace of this call, on the caller's stream: -delta of every query row
    float* ws = nullptr;
    cudaError_t e = cudaMallocFromPoolAsync((void**)&ws, sizeof(float) * (size_t)a.B * a.H * a.N, pool, a.stream);
    if (e != cudaSuccess) return e;
    e = a.dtype == BIGBIRD_BF16 ? launch_t<__nv_bfloat16>(a, L, dl, sms, ws) : launch_t<float>(a, L, dl, sms, ws);
    const cudaError_t ef = cudaFreeAsync(ws, a.stream);
    if (e == cudaSuccess) e = ef;
    if (e == cudaSuccess) *launches += 2;
    return e;
}

}  // namespace bigbird
