// CUDA-core BigBird attention forward (arXiv 2007.14062, Eq. (AT) over the block lists of App. D).
// fp32 arithmetic throughout; the path for fp32 tensors and an independent check for the tensor-core kernel.
//
// A CTA keeps its rows of q in shared memory and walks the rows' key blocks in chunks: scores in registers, online softmax over
// the 16 threads that share a row, probabilities to shared memory (read back by the same 16 threads), output sums in registers.
// The next chunk's K is on its way while the probabilities and sums are made; its V is requested when the sums are done, and both
// are waited for at the top of the chunk.  See simt.cuh for the tile shapes and for how clusters share the long tiles.
// Bound by shared-memory latency and the FMA pipes.  Measured (a warp per row before, no reuse of K and V in registers): [2, 12, 52 x 84,
// 64] with three global blocks 3740 -> 640 us, [2, 8, 2560, 128] padded 1547 -> 300 us, [1, 2, 512, 64] 22.6 -> 13.8 us (18.5 with four rows per
// thread and launches that wait for the kernel in front to drain).
#include "simt.cuh"

namespace bigbird {
namespace {

template <int D>
struct FwdShape {
    static constexpr int KC = 64;                  // tokens per chunk
    static constexpr int LD = D + 4, LDP = KC + 4; // padded rows: 16-byte aligned, and what a warp reads at once falls into different banks
    static constexpr bool kAlias = D == 128;       // P takes the place of K (which then cannot be fetched ahead): two CTAs fit an SM
    static size_t smem(int rows_pad) {
        const size_t k = (size_t)KC * LD, p = (size_t)rows_pad * LDP;
        return sizeof(float) * ((size_t)rows_pad * LD + (kAlias ? std::max(k, p) : k + p) + (size_t)KC * D);
    }
};

// V of padded keys becomes zero: a chunk may hold the end of one block and the beginning of another that is all padding, uninitialised
// perhaps, and 0 * NaN is not 0.  Rare, and not inline: it shares no registers with the loop then.  ([2, 8, 2560, 128] padded 305.8 us
// without it, 307.5 like this, 313.5 inline.)
template <int D, int KC>
__device__ __noinline__ void zero_padded(float* sv, const uint8_t* svalid) {
#pragma unroll 1
    for (int r = threadIdx.x >> 5; r < KC; r += blockDim.x >> 5)
        if (!svalid[r])
            for (int c = threadIdx.x & 31; c < D / 4; c += 32) *reinterpret_cast<float4*>(sv + r * D + 4 * c) = make_float4(0.f, 0.f, 0.f, 0.f);
}

// dynamic shared memory: Q [rows][LD] | K [KC][LD] | P [rows][LDP] (in K's place for D = 128) | V [KC][D]
template <typename T, int D, int TM>
__global__ void __launch_bounds__(max_threads(TM), 2)
attn_fwd_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, const int32_t* __restrict__ row_ptr,
                     const int32_t* __restrict__ col_idx, const uint8_t* __restrict__ kpm, T* __restrict__ out, float* __restrict__ lse,
                     Tiling tiling, int64_t N, float scale) {
    using S = FwdShape<D>;
    using C = Cols<D>;
    constexpr int KC = S::KC, LD = S::LD, LDP = S::LDP, TN = KC / 16;
    __shared__ uint8_t svalid[KC];
    extern __shared__ __align__(16) float smem[];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, rows_pad = (blockDim.x >> 4) * TM;
    float* const sq = smem;
    float* const sk = sq + rows_pad * LD;
    float* const sp = S::kAlias ? sk : sk + KC * LD;
    float* const sv = S::kAlias ? sk + max(KC * LD, rows_pad * LDP) : sp + rows_pad * LDP;

    grid_dependency_release();
    grid_dependency_wait();
    Tile tile;
    if (!find_tile(tiling, tile)) return;          // (a CTA without a tile belongs to a cluster that shares none)
    const int b = tiling.b, batch = tile.bh / tiling.H;
    const int64_t base = (int64_t)tile.bh * N * D;
    const int have = min(tiling.rows, b - tile.row0);
    const int tok0 = tile.blk * b + tile.row0;     // first row
    const uint8_t* mask = kpm ? kpm + (int64_t)batch * N : nullptr;
    const Walk w = share_walk(tiling, row_ptr, col_idx, tile, KC);
    const T *kb = k + base, *vb = v + base;
    // whether a chunk's tokens are keys: threads 0 .. 63 (a CTA of one warp: two each) look one chunk ahead
    auto key_valid = [&](int i) -> unsigned { return i < w.last && (!mask || mask[w.token(i)] != 0) ? 1u : 0u; };
    auto chunk_valid = [&](int i0) -> unsigned {
        unsigned f = threadIdx.x < KC ? key_valid(i0 + threadIdx.x) : 0u;
        if (blockDim.x < KC) f |= key_valid(i0 + 32 + threadIdx.x) << 1;
        return f;
    };
    // is any row of the tile a token (a thread per row: there are at least as many)
    const bool row_live = __syncthreads_or((int)threadIdx.x < have && (!mask || mask[tok0 + threadIdx.x] != 0));
    if (row_live) {
        stage_rows<D>(sq, LD, q + base + (int64_t)tok0 * D, rows_pad, have);
        stage_chunk<D>(sk, LD, kb, w, w.first, KC);
        stage_chunk<D>(sv, D, vb, w, w.first, KC);
    }
    unsigned vf = row_live ? chunk_valid(w.first) : 0u;

    const float* qrow = sq + ty * TM * LD;
    float* prow = sp + ty * TM * LDP;
    f32x2 o[TM][C::N];
    float m[TM], l[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = 0.f;                                // this thread's keys only
#pragma unroll
        for (int c = 0; c < C::N; ++c) o[i][c] = 0;
    }
    for (int i0 = w.first; i0 < w.last && row_live; i0 += KC) {
        if (threadIdx.x < KC) svalid[threadIdx.x] = (uint8_t)(vf & 1u);
        if (blockDim.x < KC) svalid[32 + threadIdx.x] = (uint8_t)(vf >> 1);
        copy_wait();
        const int with_keys = __syncthreads_count(vf != 0u);       // threads, of those that look, that have seen a key
        const bool any = with_keys != 0;
        if (i0 + KC < w.last) vf = chunk_valid(i0 + KC);
        if (any) {
            if (mask && with_keys < KC) zero_padded<D, KC>(sv, svalid);       // (every thread of a one-warp CTA looks at two keys: always)
            float s[TM][TN];
            dot_tile<TM, TN, D>(s, qrow, LD, sk + tx * LD, LD);
            bool valid[TN];
#pragma unroll
            for (int j = 0; j < TN; ++j) valid[j] = svalid[tx + 16 * j] != 0;
            __syncthreads();                       // K has been read
            if (!S::kAlias && i0 + KC < w.last) stage_chunk<D>(sk, LD, kb, w, i0 + KC, KC);
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                float mx = -CUDART_INF_F;
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    s[i][j] = valid[j] ? s[i][j] * scale : -CUDART_INF_F;
                    mx = fmaxf(mx, s[i][j]);
                }
                const float m_old = m[i];
                m[i] = mx = fmaxf(m_old, row_max16(mx));
                if (mx == -CUDART_INF_F) mx = 0.f;          // nothing so far but scores that overflowed to -inf: probabilities of zero
                const float alpha = expf(m_old - mx);       // 0 on the first chunk
                l[i] *= alpha;
#pragma unroll
                for (int c = 0; c < C::N; ++c) mul2(o[i][c], pair(alpha, alpha));
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float p = expf(s[i][j] - mx);
                    l[i] += p;
                    prow[i * LDP + tx + 16 * j] = p;
                }
            }
            __syncwarp();                          // a row's probabilities are read by the half-warp that wrote them
            sum_tile<TM, D>(o, prow, LDP, sv, D, KC, tx);
        }
        __syncthreads();                           // V (and K, or P in its place) has been read
        if (i0 + KC < w.last) {
            if (S::kAlias || !any) stage_chunk<D>(sk, LD, kb, w, i0 + KC, KC);
            stage_chunk<D>(sv, D, vb, w, i0 + KC, KC);
        }
    }
    copy_wait();
#pragma unroll
    for (int i = 0; i < TM; ++i) l[i] = row_sum16(l[i]);

    if (tile.shares > 1) {
        // every CTA of the cluster leaves its (O, m, l) in its shared memory; each then adds up its share of the rows
        constexpr int LDO = D + 4;
        cg::cluster_group cluster = cg::this_cluster();
        __syncthreads();
        float* const so = smem;                    // [rows][LDO], columns D, D + 1: m, l
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            float* row = so + (ty * TM + i) * LDO;
            store_cols<D>(row, o[i], 1.f, tx);
            if (tx == 0) { row[D] = m[i]; row[D + 1] = l[i]; }
        }
        cluster.sync();
        const int per = (have + tile.shares - 1) / tile.shares, r_end = min(have, per * (tile.rank + 1));
        for (int r = per * tile.rank + ty; r < r_end; r += blockDim.x >> 4) {
            // (at most eight shares; all remote loads of a row are in flight together)
            float ms[8], mx = -CUDART_INF_F, sum = 0.f;
            f32x2 acc[C::N];
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                ms[s] = s < tile.shares ? cluster.map_shared_rank(so, s)[r * LDO + D] : -CUDART_INF_F;
                mx = fmaxf(mx, ms[s]);
            }
#pragma unroll
            for (int c = 0; c < C::N; ++c) acc[c] = 0;
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                if (ms[s] == -CUDART_INF_F) continue;
                const float* row = cluster.map_shared_rank(so, s) + r * LDO;
                const float f = expf(ms[s] - mx);
                sum = fmaf(f, row[D + 1], sum);
#pragma unroll
                for (int c = 0; c < C::N; ++c) fma2(acc[c], pair(f, f), *reinterpret_cast<const f32x2*>(row + C::at(tx, c)));
            }
            const int tok = tok0 + r;
            const bool token = !mask || mask[tok] != 0, good = token && sum > 0.f;
            store_cols<D>(out + base + (int64_t)tok * D, acc, good ? 1.f / sum : 0.f, tx, !token);
            if (lse && tx == 0) lse[(int64_t)tile.bh * N + tok] = good ? mx + logf(sum) : -CUDART_INF_F;
        }
        cluster.sync();                            // nobody leaves while its shared memory is being read
        return;
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = ty * TM + i, tok = tok0 + r;
        if (r >= have) continue;
        const bool token = !mask || mask[tok] != 0, good = token && l[i] > 0.f;
        store_cols<D>(out + base + (int64_t)tok * D, o[i], good ? 1.f / l[i] : 0.f, tx, !token);
        if (lse && tx == 0) lse[(int64_t)tile.bh * N + tok] = good ? m[i] + logf(l[i]) : -CUDART_INF_F;
    }
}

template <typename T, int D, int TM>
cudaError_t launch_tm(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms) {
    static std::once_flag once[64];
    const cudaError_t e = allow_smem((const void*)attn_fwd_simt_kernel<T, D, TM>, FwdShape<D>::smem(max_threads(TM) / 16 * TM), once);
    if (e != cudaSuccess) return e;
    const Shape s = make_shape(TM, L, dl, a.B * a.H, 2 * sms, FwdShape<D>::KC);
    return launch_clusters(attn_fwd_simt_kernel<T, D, TM>, s, FwdShape<D>::smem(s.threads / 16 * TM), a.stream, (const T*)a.q, (const T*)a.k, (const T*)a.v,
                           (const int32_t*)dl.row_ptr, (const int32_t*)dl.col_idx, a.kpm, (T*)a.out, a.lse, s.t, a.N, a.scale);
}
template <typename T, int D>
cudaError_t launch_d(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms) {
    const int tm = rows_per_thread(L, a.B * a.H, D, 2 * sms);
    if (tm == 2) return launch_tm<T, D, 2>(a, L, dl, sms);
    if constexpr (D <= 64) {
        if (tm == 6) return launch_tm<T, D, 6>(a, L, dl, sms);
        if (tm == 7) return launch_tm<T, D, 7>(a, L, dl, sms);
    }
    return launch_tm<T, D, 4>(a, L, dl, sms);
}
template <typename T>
cudaError_t launch_t(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms) {
    switch (a.D) {
        case 32: return launch_d<T, 32>(a, L, dl, sms);
        case 64: return launch_d<T, 64>(a, L, dl, sms);
        case 128: return launch_d<T, 128>(a, L, dl, sms);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_attn_fwd_simt(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms, int* launches) {
    const cudaError_t e = a.dtype == BIGBIRD_BF16 ? launch_t<__nv_bfloat16>(a, L, dl, sms) : launch_t<float>(a, L, dl, sms);
    if (e == cudaSuccess) ++*launches;
    return e;
}

}  // namespace bigbird
