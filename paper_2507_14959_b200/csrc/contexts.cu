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

// One thread per frame: a tile of frames' label words is brought to shared memory in order, then every thread
// walks the set bits of its frame (an odd word stride keeps the threads on different banks) and counts each
// unordered pair, the diagonal included.
// HIST: counts go to a triangular histogram of the block in shared memory and from there, zeros skipped, to
// both halves of co; up to COOC_HIST_LABELS labels, so that it fits.  With more labels the pairs are
// spread thinly enough for direct adds.  118287 frames, 80 labels: 30.2 us with a warp per frame and a global
// atomic per ordered pair (118287 warps of work and the hot pairs' atomics in one queue), 12.5 us now.
// Counts stay exact in fp32 up to 2^24 frames.
constexpr int COOC_HIST_LABELS = 320;
constexpr int COOC_HIST_THREADS = 1024, COOC_THREADS = 256;
constexpr int COOC_SMEM = 220 * 1024;

template <bool HIST>
__global__ void __launch_bounds__(HIST ? COOC_HIST_THREADS : COOC_THREADS)
cooccurrence_kernel(const uint32_t* __restrict__ labels, int n_frames, int n_labels, int tile_frames,
                    float* __restrict__ co, int* __restrict__ status) {
    extern __shared__ uint32_t smem[];
    const int nw = (n_labels + 31) / 32, stride = nw | 1;
    const uint32_t tail = (n_labels & 31) ? (1u << (n_labels & 31)) - 1u : 0xFFFFFFFFu;      // bits of the last word
    uint32_t* hist = smem + (size_t)tile_frames * stride;            // entry j (j + 1) / 2 + i, i <= j
    const int n_hist = HIST ? n_labels * (n_labels + 1) / 2 : 0;
    for (int i = threadIdx.x; i < n_hist; i += blockDim.x) hist[i] = 0u;
    for (long long f0 = (long long)blockIdx.x * tile_frames; f0 < n_frames; f0 += (long long)gridDim.x * tile_frames) {
        const int nf = (int)min((long long)tile_frames, n_frames - f0);
        __syncthreads();
        for (int i = threadIdx.x; i < nf * nw; i += blockDim.x) {
            const int w = i % nw;
            smem[(i / nw) * stride + w] = __ldg(labels + (size_t)f0 * nw + i) & (w == nw - 1 ? tail : 0xFFFFFFFFu);
        }
        __syncthreads();
        if ((int)threadIdx.x < nf) {
            uint32_t* mine = smem + (size_t)threadIdx.x * stride;
            int n = 0;
            for (int w = 0; w < nw; ++w) n += __popc(mine[w]);
            if (n > COOC_MAX_LABELS_PER_FRAME) {         // more labels than a frame may carry here: drop the last ones
                if (status) atomicCAS(status, 0, (int)PM_ERR_CAPACITY);
                for (int w = nw - 1; n > COOC_MAX_LABELS_PER_FRAME; --w)
                    for (; n > COOC_MAX_LABELS_PER_FRAME && mine[w]; --n) mine[w] &= ~(1u << (31 - __clz(mine[w])));
            }
            for (int wi = 0; wi < nw; ++wi)
                for (uint32_t bi = mine[wi]; bi; bi &= bi - 1) {
                    const int i = wi * 32 + __ffs((int)bi) - 1;
                    uint32_t bj = bi;                    // j from i on
                    for (int wj = wi;;) {
                        for (; bj; bj &= bj - 1) {
                            const int j = wj * 32 + __ffs((int)bj) - 1;
                            if (HIST) {
                                atomicAdd(hist + j * (j + 1) / 2 + i, 1u);
                            } else {
                                atomicAdd(co + (size_t)j * n_labels + i, 1.0f);
                                if (i != j) atomicAdd(co + (size_t)i * n_labels + j, 1.0f);
                            }
                        }
                        if (++wj >= nw) break;
                        bj = mine[wj];
                    }
                }
        }
    }
    if (HIST) {
        __syncthreads();
        for (int j = threadIdx.x >> 5; j < n_labels; j += COOC_HIST_THREADS / 32)
            for (int i = threadIdx.x & 31; i <= j; i += 32) {
                const uint32_t v = hist[j * (j + 1) / 2 + i];
                if (!v) continue;
                atomicAdd(co + (size_t)j * n_labels + i, (float)v);
                if (i != j) atomicAdd(co + (size_t)i * n_labels + j, (float)v);
            }
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
    const size_t stride = (size_t)(((n_labels + 31) / 32) | 1) * sizeof(uint32_t);
    static SmemGrant grant_hist, grant;
    auto launch = [&](auto kernel, SmemGrant& g, int threads, size_t hist_bytes, int blocks_per_sm) {
        // frames of a tile: one per thread, fewer where their label words would not fit
        const int fit = (int)std::min<size_t>(threads, (COOC_SMEM / blocks_per_sm - hist_bytes) / stride);
        const int per_block = (n_frames + n_sms * blocks_per_sm - 1) / (n_sms * blocks_per_sm);
        const int tile = std::max(1, std::min(fit, per_block));
        const size_t bytes = tile * stride + hist_bytes;
        if (bytes > 227 * 1024) return PM_ERR_CAPACITY;      // one frame's words do not fit: over a million labels
        if (g.ensure(kernel, (int)bytes) != cudaSuccess) return PM_ERR_CUDA;
        const int blocks = std::min((n_frames + tile - 1) / tile, n_sms * blocks_per_sm);
        kernel<<<blocks, threads, bytes, st>>>(labels, n_frames, n_labels, tile, co, status_out);
        return PM_OK;
    };
    const size_t hist_bytes = (size_t)n_labels * (n_labels + 1) / 2 * sizeof(uint32_t);
    const int rc = n_labels <= COOC_HIST_LABELS ? launch(cooccurrence_kernel<true>, grant_hist, COOC_HIST_THREADS, hist_bytes, 1)
                                                : launch(cooccurrence_kernel<false>, grant, COOC_THREADS, 0, 8);
    if (rc != PM_OK) return rc;
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
