// Training-time context construction (Sec. 3.4, Algorithm 1) and its quality measure (Eq. 6).
//
// The label co-occurrence matrix is counted on the GPU from per-frame label bit sets (the format
// pm_select writes); the greedy construction itself is sequential over labels, works on a K x K
// matrix of at most a few hundred labels, and runs on the host.
#include <algorithm>
#include <numeric>
#include <vector>

#include "common.cuh"

namespace {

constexpr int COOC_MAX_LABELS_PER_FRAME = 64;

// Two forms; counts stay exact in fp32 up to 2^24 frames.
//
// Direct: a warp per frame.  The lanes list the set bits of its label words in shared memory, then every ordered pair
// (the diagonal included) adds 1 to co[i, j].  Bound by the atomics of pairs that many frames share.
constexpr int COOC_THREADS = 256;

__global__ void __launch_bounds__(COOC_THREADS)
cooccurrence_direct_kernel(const uint32_t* __restrict__ labels, int n_frames, int n_labels, float* __restrict__ co, int* __restrict__ status) {
    __shared__ int ids[COOC_THREADS / 32][COOC_MAX_LABELS_PER_FRAME];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (n_labels + 31) / 32;
    const uint32_t tail = (n_labels & 31) ? (1u << (n_labels & 31)) - 1u : 0xFFFFFFFFu;      // bits of the last word
    int* mine = ids[warp];
    for (int f = blockIdx.x * (COOC_THREADS / 32) + warp; f < n_frames; f += gridDim.x * (COOC_THREADS / 32)) {
        int n = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const int w = w0 + lane;
            uint32_t bits = w < nw ? __ldg(labels + (size_t)f * nw + w) & (w == nw - 1 ? tail : 0xFFFFFFFFu) : 0u;
            int incl = __popc(bits);
            int at = n - incl;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += v;
            }
            for (at += incl; bits && at < COOC_MAX_LABELS_PER_FRAME; bits &= bits - 1, ++at) mine[at] = w * 32 + __ffs((int)bits) - 1;
            n += __shfl_sync(0xFFFFFFFFu, incl, 31);
        }
        if (n > COOC_MAX_LABELS_PER_FRAME) {             // more labels than a frame may carry here
            if (lane == 0 && status) atomicCAS(status, 0, (int)PM_ERR_CAPACITY);
            n = COOC_MAX_LABELS_PER_FRAME;
        }
        __syncwarp();
        for (int p = lane; p < n * n; p += 32) atomicAdd(co + (size_t)mine[p / n] * n_labels + mine[p % n], 1.0f);
        __syncwarp();
    }
}

// Histogram: counts go to a triangular histogram of the block in shared memory and from there, zeros skipped, to both
// halves of co.  A tile of frames' label words is brought to shared memory in order (an odd word stride keeps the threads
// on different banks) and a thread takes a frame.  While a tile's frames keep only some of the warps busy, frames of more than
// COOC_FEW labels are left to all warps in turn, a lane per pair (135 frames per block, 64 labels each: 98 us against 131; 405
// frames per block: 226 against 150).
//
// The histogram pays once the block's counts outnumber its entries; the line is at as many frames as the triangle has entries.  us,
// direct / histogram, 5 labels drawn per frame and the same 5 in every frame: 80 labels (3240 entries) 2000 frames 7.9 / 9.5 and
// 11.6 / 9.5, 7000 frames 9.5 / 11.4 and 22 / 9.5, 118287 frames 77 / 25 and 269 / 11; 320 labels (51360 entries)
// 20000 frames 10 / 18 and 39 / 16, 60000 frames 18 / 25 and 98 / 20.
constexpr int COOC_HIST_LABELS = 320;
constexpr int COOC_HIST_THREADS = 1024;
constexpr int COOC_FEW = 8, COOC_BUSY = 384;
constexpr int COOC_LIST_BYTES = (COOC_HIST_THREADS / 32 * COOC_MAX_LABELS_PER_FRAME + COOC_HIST_THREADS) * 2;
constexpr int COOC_SMEM = 220 * 1024;

__device__ __forceinline__ void hist_add(uint32_t* hist, int i, int j) { atomicAdd(hist + j * (j + 1) / 2 + i, 1u); }      // i <= j

template <bool BUSY>
__global__ void __launch_bounds__(COOC_HIST_THREADS)
cooccurrence_hist_kernel(const uint32_t* __restrict__ labels, int n_frames, int n_labels, int tile_frames,
                         float* __restrict__ co, int* __restrict__ status) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int nw = (n_labels + 31) / 32, stride = nw | 1, lane = threadIdx.x & 31;
    const uint32_t tail = (n_labels & 31) ? (1u << (n_labels & 31)) - 1u : 0xFFFFFFFFu;
    const int n_hist = n_labels * (n_labels + 1) / 2, hist_words = (n_hist + 3) & ~3;
    uint32_t* hist = smem;                               // entry j (j + 1) / 2 + i, i <= j
    uint16_t* lists = reinterpret_cast<uint16_t*>(smem + hist_words);
    uint16_t* list = lists + (threadIdx.x >> 5) * COOC_MAX_LABELS_PER_FRAME;                   // labels of the warp's frame
    uint16_t* many = lists + COOC_HIST_THREADS / 32 * COOC_MAX_LABELS_PER_FRAME;               // frames of the tile with more than COOC_FEW labels
    uint32_t* words = smem + hist_words + COOC_LIST_BYTES / 4;
    __shared__ int n_many;
    for (int i = threadIdx.x; i < hist_words / 4; i += COOC_HIST_THREADS) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0, 0, 0, 0);
    for (long long f0 = (long long)blockIdx.x * tile_frames; f0 < n_frames; f0 += (long long)gridDim.x * tile_frames) {
        const int nf = (int)min((long long)tile_frames, n_frames - f0);
        __syncthreads();
        if (threadIdx.x == 0) n_many = 0;
        for (int i = threadIdx.x; i < nf * nw; i += COOC_HIST_THREADS) {
            const int w = i % nw;
            words[(i / nw) * stride + w] = __ldg(labels + (size_t)f0 * nw + i) & (w == nw - 1 ? tail : 0xFFFFFFFFu);
        }
        __syncthreads();
        if ((int)threadIdx.x < nf) {
            uint32_t* mine = words + (size_t)threadIdx.x * stride;
            int n = 0;
            for (int w = 0; w < nw; ++w) n += __popc(mine[w]);
            if constexpr (BUSY) {
                if (n > COOC_MAX_LABELS_PER_FRAME) {     // more labels than a frame may carry here: drop the last ones
                    if (status) atomicCAS(status, 0, (int)PM_ERR_CAPACITY);
                    for (int w = nw - 1; n > COOC_MAX_LABELS_PER_FRAME; --w)
                        for (; n > COOC_MAX_LABELS_PER_FRAME && mine[w]; --n) mine[w] &= ~(1u << (31 - __clz(mine[w])));
                }
                for (int wi = 0; wi < nw; ++wi)
                    for (uint32_t bi = mine[wi]; bi; bi &= bi - 1) {
                        const int i = wi * 32 + __ffs((int)bi) - 1;
                        uint32_t bj = bi;                // j from i on
                        for (int wj = wi;;) {
                            for (; bj; bj &= bj - 1) hist_add(hist, i, wj * 32 + __ffs((int)bj) - 1);
                            if (++wj >= nw) break;
                            bj = mine[wj];
                        }
                    }
            } else if (n > COOC_FEW) {
                many[atomicAdd(&n_many, 1)] = (uint16_t)threadIdx.x;
            } else if (n > 0) {
                uint64_t ids[2] = {0, 0};                // 16 bits each, the last label found lowest
                for (int w = 0; w < nw; ++w)
                    for (uint32_t b = mine[w]; b; b &= b - 1) {
                        ids[1] = ids[1] << 16 | ids[0] >> 48;
                        ids[0] = ids[0] << 16 | (uint64_t)(w * 32 + __ffs((int)b) - 1);
                    }
                for (int q = 0; q < n; ++q) {
                    const int j = (int)(ids[0] & 0xFFFFu);         // the highest label left
                    for (int r = 0; r < n - q; ++r) hist_add(hist, (int)((r < 4 ? ids[0] : ids[1]) >> (16 * (r & 3)) & 0xFFFFu), j);
                    ids[0] = ids[0] >> 16 | ids[1] << 48;
                    ids[1] >>= 16;
                }
            }
        }
        if constexpr (BUSY) continue;
        __syncthreads();
        for (int q = threadIdx.x >> 5; q < n_many; q += COOC_HIST_THREADS / 32) {
            const uint32_t* row = words + (size_t)many[q] * stride;
            int m = 0;
            for (int w = 0; w < nw; ++w) {
                const uint32_t b = row[w];
                const int at = m + __popc(b & ((1u << lane) - 1u));
                if ((b >> lane & 1u) && at < COOC_MAX_LABELS_PER_FRAME) list[at] = (uint16_t)(w * 32 + lane);
                m += __popc(b);
            }
            if (m > COOC_MAX_LABELS_PER_FRAME) {
                if (lane == 0 && status) atomicCAS(status, 0, (int)PM_ERR_CAPACITY);
                m = COOC_MAX_LABELS_PER_FRAME;
            }
            __syncwarp();
            for (int p = lane; p < m * (m + 1) / 2; p += 32) {            // pair p = j (j + 1) / 2 + i of the list, i <= j
                int j = (int)(0.5f * (sqrtf((float)(8 * p + 1)) - 1.f));
                j += (j + 1) * (j + 2) / 2 <= p ? 1 : j * (j + 1) / 2 > p ? -1 : 0;
                hist_add(hist, list[p - j * (j + 1) / 2], list[j]);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int j = threadIdx.x >> 5; j < n_labels; j += COOC_HIST_THREADS / 32)
        for (int i = lane; i <= j; i += 32) {
            const uint32_t v = hist[j * (j + 1) / 2 + i];
            if (!v) continue;
            atomicAdd(co + (size_t)j * n_labels + i, (float)v);
            if (i != j) atomicAdd(co + (size_t)i * n_labels + j, (float)v);
        }
}

}  // namespace

extern "C" {

int pm_cooccurrence(const uint32_t* labels, int n_frames, int n_labels, float* co, int32_t* status_out,
                    void* cuda_stream) {
    if (n_frames < 0 || n_labels <= 0 || !co || (n_frames > 0 && !labels)) return PM_ERR_ARG;
    if (n_frames > (1 << 24)) return PM_ERR_CAPACITY;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (cudaMemsetAsync(co, 0, sizeof(float) * (size_t)n_labels * n_labels, st) != cudaSuccess) return PM_ERR_CUDA;
    if (status_out && cudaMemsetAsync(status_out, 0, sizeof(int32_t), st) != cudaSuccess) return PM_ERR_CUDA;
    if (n_frames == 0) return PM_OK;
    int dev = 0, n_sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PM_ERR_CUDA;
    const long long entries = (long long)n_labels * (n_labels + 1) / 2;
    if (n_labels <= COOC_HIST_LABELS && n_frames >= entries) {
        const size_t stride = (size_t)(((n_labels + 31) / 32) | 1) * sizeof(uint32_t);
        const size_t fixed = (size_t)((entries + 3) & ~3ll) * sizeof(uint32_t) + COOC_LIST_BYTES;
        // frames of a tile: one per thread, fewer where their label words would not fit
        const int fit = (int)std::min<size_t>(COOC_HIST_THREADS, (COOC_SMEM - fixed) / stride);
        const int tile = std::min(fit, (n_frames + n_sms - 1) / n_sms);
        const size_t bytes = tile * stride + fixed;
        static SmemGrant grant[2];
        const bool busy = tile >= COOC_BUSY;
        const auto kernel = busy ? cooccurrence_hist_kernel<true> : cooccurrence_hist_kernel<false>;
        if (grant[busy].ensure(kernel, (int)bytes) != cudaSuccess) return PM_ERR_CUDA;
        kernel<<<std::min((n_frames + tile - 1) / tile, n_sms), COOC_HIST_THREADS, bytes, st>>>(labels, n_frames, n_labels, tile, co, status_out);
    } else {
        cooccurrence_direct_kernel<<<std::min((n_frames + 7) / 8, 16 * n_sms), COOC_THREADS, 0, st>>>(labels, n_frames, n_labels, co, status_out);
    }
    return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}

int pm_build_contexts(const float* co, int n_labels, int max_size, int max_contexts, int allow_overlap,
                      int32_t* ctx_offsets, int32_t* ctx_ids, int* n_contexts) {
    if (!co || n_labels <= 0 || max_size <= 0 || max_contexts <= 0 || !ctx_offsets || !ctx_ids || !n_contexts)
        return PM_ERR_ARG;
    const int K = n_labels;
    auto C = [&](int i, int j) { return co[(size_t)i * K + j]; };
    std::vector<int> valid;
    for (int l = 0; l < K; ++l) if (C(l, l) > 0.f) valid.push_back(l);
    std::vector<int> order = valid;                   // most frequent first, ties by label
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return C(a, a) > C(b, b); });
    std::vector<std::vector<int>> ctx;
    std::vector<char> assigned(K, 0);
    std::vector<int> cand;
    for (int l : order) {
        if (!allow_overlap && assigned[l]) continue;
        if ((int)ctx.size() >= max_contexts) break;   // full: no later cluster can be kept
        // the up to B-1 strongest neighbours: a row usually has many more candidates than are kept, so only
        // those are put in order (a total order: the labels break ties)
        cand.clear();
        const float* row = co + (size_t)l * K;
        for (int j : valid)
            if (j != l && row[j] > 0.f && (allow_overlap || !assigned[j])) cand.push_back(j);
        const size_t keep = std::min(cand.size(), (size_t)max_size - 1);
        std::partial_sort(cand.begin(), cand.begin() + keep, cand.end(),
                          [&](int a, int b) { return row[a] > row[b] || (row[a] == row[b] && a < b); });
        cand.resize(keep);
        cand.push_back(l);
        std::sort(cand.begin(), cand.end());
        if (std::find(ctx.begin(), ctx.end(), cand) == ctx.end()) {
            ctx.push_back(cand);
            if (!allow_overlap) for (int j : cand) assigned[j] = 1;
        }
    }
    std::vector<char> covered(K, 0);
    for (auto& c : ctx) for (int j : c) covered[j] = 1;
    for (int l : valid) {                             // leftovers go where they co-occur most, if there is room
        if (covered[l]) continue;
        int best = -1;
        double best_fit = -1.0;
        for (size_t c = 0; c < ctx.size(); ++c) {
            if ((int)ctx[c].size() >= max_size) continue;
            double fit = 0.0;
            for (int j : ctx[c]) fit += C(l, j);
            if (fit > best_fit) { best = (int)c; best_fit = fit; }
        }
        if (best >= 0) {
            ctx[best].insert(std::upper_bound(ctx[best].begin(), ctx[best].end(), l), l);
            covered[l] = 1;
        }
    }
    ctx_offsets[0] = 0;
    for (size_t c = 0; c < ctx.size(); ++c) {
        std::copy(ctx[c].begin(), ctx[c].end(), ctx_ids + ctx_offsets[c]);
        ctx_offsets[c + 1] = ctx_offsets[c] + (int)ctx[c].size();
    }
    *n_contexts = (int)ctx.size();
    return PM_OK;
}

int pm_intra_coherence(const float* co_norm, int n_labels, const int32_t* ctx_offsets, const int32_t* ctx_ids,
                       int n_contexts, double* out) {
    if (!co_norm || n_labels <= 0 || n_contexts < 0 || !out || (n_contexts > 0 && (!ctx_offsets || !ctx_ids)))
        return PM_ERR_ARG;
    double total = 0.0;
    for (int c = 0; c < n_contexts; ++c) {
        const int lo = ctx_offsets[c], hi = ctx_offsets[c + 1], n = hi - lo;
        if (n < 0) return PM_ERR_ARG;
        double s = 0.0;
        for (int a = lo; a < hi; ++a)
            for (int b = lo; b < hi; ++b) {
                const int i = ctx_ids[a], j = ctx_ids[b];
                if (i < 0 || i >= n_labels || j < 0 || j >= n_labels) return PM_ERR_ARG;
                if (a != b) s += co_norm[(size_t)i * n_labels + j];
            }
        if (n >= 2) total += s / ((double)n * (n - 1));
    }
    *out = n_contexts > 0 ? total / n_contexts : 0.0;
    return PM_OK;
}

}  // extern "C"
