// C ABI of the Polymorph library: model upload, adapter arenas, per-batch routing plan
// (bucketing of frames by adapter set, tile -> LoRA slab lists) and the launch sequences.
#include <algorithm>
#include <array>
#include <chrono>
#include <cstdio>
#include <cstring>
#include <new>

#include "common.cuh"

int gemm_tile_n(int n_out);   // gemm_tcgen05.cu

namespace {

#define CK(expr)                                                                        \
    do {                                                                                \
        cudaError_t _e = (expr);                                                        \
        if (_e != cudaSuccess) {                                                        \
            err = std::string(#expr) + ": " + cudaGetErrorString(_e);                   \
            return _e == cudaErrorMemoryAllocation ? PM_ERR_OOM : PM_ERR_CUDA;          \
        }                                                                               \
    } while (0)

template <typename T> T host_cvt(float v);
template <> float host_cvt<float>(float v) { return v; }
template <> bf16 host_cvt<bf16>(float v) { return __float2bfloat16_rn(v); }

struct DevBuf {              // owning device allocation
    void* p = nullptr;
    size_t bytes = 0;
    ~DevBuf() { if (p) cudaFree(p); }
    cudaError_t alloc(size_t n) {
        if (p) { cudaFree(p); p = nullptr; }
        bytes = n;
        if (n == 0) return cudaSuccess;
        return cudaMalloc(&p, n);
    }
    template <typename T> T* as() const { return reinterpret_cast<T*>(p); }
};

template <typename T>
cudaError_t upload(DevBuf& buf, const float* host, size_t n) {
    cudaError_t e = buf.alloc(n * sizeof(T));
    if (e != cudaSuccess) return e;
    std::vector<T> tmp(n);
    for (size_t i = 0; i < n; ++i) tmp[i] = host_cvt<T>(host[i]);
    return cudaMemcpy(buf.p, tmp.data(), n * sizeof(T), cudaMemcpyHostToDevice);
}

// [k_in, n_out] row-major -> [n_out, k_in]
template <typename T>
cudaError_t upload_transposed(DevBuf& buf, const float* w, int k_in, int n_out) {
    cudaError_t e = buf.alloc((size_t)k_in * n_out * sizeof(T));
    if (e != cudaSuccess) return e;
    std::vector<T> tmp((size_t)k_in * n_out);
    for (int k = 0; k < k_in; ++k)
        for (int n = 0; n < n_out; ++n) tmp[(size_t)n * k_in + k] = host_cvt<T>(w[(size_t)k * n_out + n]);
    return cudaMemcpy(buf.p, tmp.data(), tmp.size() * sizeof(T), cudaMemcpyHostToDevice);
}

size_t esize(int dtype) { return dtype == 0 ? 2 : 4; }

// One linear with its LoRA arenas.
struct LinearObj {
    LinearDev dev;
    DevBuf wt, bias, at, bt, lng, lnc1, lnc2;
    int slabs_max = 0, max_adapters = 0, dtype = 0;
    std::vector<float> ln_gamma, ln_beta;      // non-empty: the LayerNorm in front of this linear is folded in

    // ln_g / ln_b (host [k_in], bf16 build only): fold LN(x) = (x - mean) rstd gamma + beta into the linear:
    //   W' = gamma o W (then rounded to bf16), g[n] = sum_k W'[k,n] over the ROUNDED values (what the
    //   tensor cores multiply), b' = b + beta W.
    int init(int k_in, int n_out, const float* w, const float* b, int max_adapters_, int slabs_max_,
             int dtype_, std::string& err, const float* ln_g = nullptr, const float* ln_b = nullptr) {
        dev.k_in = k_in; dev.n_out = n_out;
        slabs_max = slabs_max_; max_adapters = max_adapters_; dtype = dtype_;
        if (dtype == 0 && ln_g && ln_b) {
            ln_gamma.assign(ln_g, ln_g + k_in); ln_beta.assign(ln_b, ln_b + k_in);
            std::vector<float> wf((size_t)k_in * n_out), bf(n_out), gs(n_out);
            std::vector<double> gsum(n_out, 0.0), bsum(n_out, 0.0);
            for (int k = 0; k < k_in; ++k)
                for (int n = 0; n < n_out; ++n) {
                    const float v = __bfloat162float(__float2bfloat16_rn(ln_g[k] * w[(size_t)k * n_out + n]));
                    wf[(size_t)k * n_out + n] = v;
                    gsum[n] += v;
                    bsum[n] += (double)ln_b[k] * w[(size_t)k * n_out + n];
                }
            for (int n = 0; n < n_out; ++n) { gs[n] = (float)gsum[n]; bf[n] = (float)(b[n] + bsum[n]); }
            CK(upload_transposed<bf16>(wt, wf.data(), k_in, n_out));
            CK(upload<float>(bias, bf.data(), n_out));
            CK(upload<float>(lng, gs.data(), n_out));
            dev.ln_g = lng.as<float>();
        } else {
            if (dtype == 0) CK(upload_transposed<bf16>(wt, w, k_in, n_out));
            else CK(upload_transposed<float>(wt, w, k_in, n_out));
            CK(upload<float>(bias, b, n_out));
        }
        dev.Wt = wt.p; dev.bias = bias.as<float>();
        if (max_adapters > 0 && slabs_max > 0) {
            const size_t RS = (size_t)slabs_max * PM_SLAB;
            CK(at.alloc((size_t)max_adapters * RS * k_in * esize(dtype)));
            CK(bt.alloc((size_t)max_adapters * RS * n_out * esize(dtype)));
            CK(cudaMemset(at.p, 0, at.bytes));
            CK(cudaMemset(bt.p, 0, bt.bytes));
            dev.lora.At = at.p; dev.lora.Bt = bt.p;
            if (dev.ln_g) {
                CK(lnc1.alloc((size_t)max_adapters * RS * sizeof(float)));
                CK(lnc2.alloc((size_t)max_adapters * RS * sizeof(float)));
                CK(cudaMemset(lnc1.p, 0, lnc1.bytes));
                CK(cudaMemset(lnc2.p, 0, lnc2.bytes));
                dev.ln_c1 = lnc1.as<float>(); dev.ln_c2 = lnc2.as<float>();
            }
        }
        if (dtype == 0) {
            const int bn = gemm_tile_n(n_out);
            bool ok = tm_encode_2d(&dev.tm_w, wt.p, k_in, n_out, (uint64_t)k_in * 2, 64, bn, 128);
            if (ok && dev.lora.At) {
                ok = tm_encode_2d(&dev.tm_bt, bt.p, PM_SLAB, (uint64_t)max_adapters * slabs_max * n_out,
                                  PM_SLAB * 2, PM_SLAB, bn, 32);
            }
            if (!ok) { err = "cuTensorMapEncodeTiled failed (static operands)"; return PM_ERR_CUDA; }
            dev.has_tm = true;
            if (!gemm_encode_pair_maps(dev, max_adapters, slabs_max)) { err = "cuTensorMapEncodeTiled failed (half-tile operands)"; return PM_ERR_CUDA; }
            if (!small_linear_encode(dev, max_adapters, slabs_max)) { err = "cuTensorMapEncodeTiled failed (few-row operands)"; return PM_ERR_CUDA; }
        }
        return PM_OK;
    }

    template <typename T>
    int set_adapter_t(int a, int rank, const float* A, const float* B, std::string& err) {
        const int k_in = dev.k_in, n_out = dev.n_out;
        const size_t RS = (size_t)slabs_max * PM_SLAB;
        std::vector<T> ha(RS * k_in, host_cvt<T>(0.f)), hb(RS * n_out, host_cvt<T>(0.f));
        std::vector<float> c1(RS, 0.f), c2(RS, 0.f);
        if (A && B) {
            const bool fold = dev.ln_g != nullptr;
            std::vector<double> s1(rank, 0.0), s2(rank, 0.0);
            for (int k = 0; k < k_in; ++k)
                for (int j = 0; j < rank; ++j) {
                    const float a0 = A[(size_t)k * rank + j];
                    const T av = host_cvt<T>(fold ? ln_gamma[k] * a0 : a0);
                    ha[(size_t)j * k_in + k] = av;
                    if (fold) { s1[j] += (double)(float)av; s2[j] += (double)ln_beta[k] * a0; }
                }
            for (int j = 0; j < rank && fold; ++j) { c1[j] = (float)s1[j]; c2[j] = (float)s2[j]; }
            for (int j = 0; j < rank; ++j)
                for (int n = 0; n < n_out; ++n)
                    hb[((size_t)(j / PM_SLAB) * n_out + n) * PM_SLAB + (j % PM_SLAB)] =
                        host_cvt<T>(B[(size_t)j * n_out + n]);
        }
        CK(cudaMemcpy(at.as<T>() + (size_t)a * RS * k_in, ha.data(), ha.size() * sizeof(T), cudaMemcpyHostToDevice));
        CK(cudaMemcpy(bt.as<T>() + (size_t)a * RS * n_out, hb.data(), hb.size() * sizeof(T), cudaMemcpyHostToDevice));
        if (dev.ln_g) {
            CK(cudaMemcpy(lnc1.as<float>() + (size_t)a * RS, c1.data(), RS * sizeof(float), cudaMemcpyHostToDevice));
            CK(cudaMemcpy(lnc2.as<float>() + (size_t)a * RS, c2.data(), RS * sizeof(float), cudaMemcpyHostToDevice));
        }
        return PM_OK;
    }
    int set_adapter(int a, int rank, const float* A, const float* B, std::string& err) {
        if ((int)adapted.size() < max_adapters) adapted.assign(max_adapters, 0);
        adapted[a] = (A && B) ? 1 : 0;
        n_adapted = 0;
        for (char c : adapted) n_adapted += c;
        return dtype == 0 ? set_adapter_t<bf16>(a, rank, A, B, err) : set_adapter_t<float>(a, rank, A, B, err);
    }
    // adapters that really touch this linear (a NULL A/B pair leaves it un-adapted); with none, the
    // forward skips the shrink and the LoRA steps here altogether -- the paper's cheap variant, LoRA in
    // the last blocks only (Sec. 3.1), then costs nothing in the other blocks
    std::vector<char> adapted;
    int n_adapted = 0;
};

// Per-batch routing: validation, bucketing, tile plan, upload.
struct Router {
    int max_frames = 0, max_set = 0, max_adapters = 0, slabs_max = 0, tokens = 0;
    int slab_cap = 0, max_tiles = 0;
    DevBuf blob;
    // pinned host copies of the blob, used in turn: the host may plan a few steps ahead of the GPU
    // without waiting for an earlier upload to have left its staging buffer
    static constexpr int N_STAGE = 4;
    void* stage[N_STAGE] = {nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t uploaded[N_STAGE] = {nullptr, nullptr, nullptr, nullptr};
    bool upload_pending[N_STAGE] = {false, false, false, false};
    int stage_next = 0;
    size_t blob_bytes = 0;
    size_t off_perm = 0, off_soff = 0, off_sids = 0, off_src = 0, off_tn = 0, off_ts = 0, off_tsc = 0, off_tm = 0;
    RouteDev dev;
    std::vector<int32_t> last_off, last_ids;
    std::vector<int> last_fixed;     // frame_of_slot then src_of_slot of the cached plan (branched forward)
    // changes whenever the launch sequence that follows from the plan may change (a new host plan; a
    // device plan for another frame count): recorded CUDA graphs are keyed by it
    unsigned long long version = 0;
    int device_plan_frames = -1;
    int last_frames = -1;
    bool last_sorted = false;
    std::vector<int> perm_host, sorted_ids;
    uint64_t row_mask[256][4];       // scratch of build(): the rows of the pair at hand that use an adapter
    long long plans_built = 0;       // host plans built (cache misses) and the host time they took
    double plan_host_ms = 0.0;

    ~Router() {
        for (int i = 0; i < N_STAGE; ++i) {
            if (stage[i]) cudaFreeHost(stage[i]);
            if (uploaded[i]) cudaEventDestroy(uploaded[i]);
        }
    }

    int init(int max_frames_, int max_set_, int max_adapters_, int slabs_max_, int tokens_, std::string& err) {
        max_frames = max_frames_; max_set = max_set_; max_adapters = max_adapters_;
        slabs_max = slabs_max_; tokens = tokens_;
        const int frames_per_pair = (2 * PM_TILE_M - 1) / tokens + 2;      // frames a 256-row pair can touch
        slab_cap = std::min(frames_per_pair * max_set, max_adapters) * slabs_max;
        dev.tile_slab_cap = std::min(((PM_TILE_M - 1) / tokens + 2) * max_set, max_adapters) * slabs_max;
        max_tiles = (int)(((size_t)max_frames * tokens + 2 * PM_TILE_M - 1) / (2 * PM_TILE_M)) * 2;   // even
        auto take = [&](size_t& off, size_t bytes) { off = blob_bytes; blob_bytes += (bytes + 255) & ~(size_t)255; };
        take(off_perm, sizeof(int) * max_frames);
        take(off_soff, sizeof(int) * (max_frames + 1));
        take(off_sids, sizeof(int) * std::max(1, max_frames * max_set));
        take(off_src, sizeof(int) * max_frames);
        take(off_tn, sizeof(int) * max_tiles);
        take(off_ts, sizeof(int) * std::max(1, max_tiles * slab_cap));
        take(off_tsc, sizeof(float) * std::max(1, max_tiles * slab_cap));
        take(off_tm, sizeof(uint32_t) * 4 * std::max(1, max_tiles * slab_cap));
        CK(blob.alloc(blob_bytes));
        CK(cudaMemset(blob.p, 0, blob_bytes));
        for (int i = 0; i < N_STAGE; ++i) {
            CK(cudaMallocHost(&stage[i], blob_bytes));
            memset(stage[i], 0, blob_bytes);
            CK(cudaEventCreateWithFlags(&uploaded[i], cudaEventDisableTiming));
        }
        uint8_t* b = blob.as<uint8_t>();
        dev.perm = (int*)(b + off_perm); dev.slot_off = (int*)(b + off_soff); dev.slot_ids = (int*)(b + off_sids);
        dev.src_slot = (int*)(b + off_src);
        dev.tile_nslabs = (int*)(b + off_tn); dev.tile_slab = (int*)(b + off_ts);
        dev.tile_scale = (float*)(b + off_tsc); dev.tile_mask = (uint32_t*)(b + off_tm);
        dev.tokens = tokens; dev.slab_cap = slab_cap;
        return PM_OK;
    }

    // offsets/ids: host CSR.  ranks[a] == 0 means "not registered".
    // frame_of_slot / src_of_slot (both or neither, n_frames entries, sort_frames false): the CSR is
    // already in slot order; slot i reports to output row frame_of_slot[i] and starts from the trunk
    // rows of slot src_of_slot[i] (the branched forward's plan).
    int build(int n_frames, const int32_t* offsets, const int32_t* ids, const std::vector<int>& ranks,
              const std::vector<float>& scales, bool sort_frames, const Launch& L, std::string& err,
              const int* frame_of_slot = nullptr, const int* src_of_slot = nullptr) {
        if (n_frames < 0 || (n_frames > 0 && (!offsets))) { err = "bad frame count or NULL set_offsets"; return PM_ERR_ARG; }
        if (n_frames > max_frames) { err = "n_frames exceeds max_frames"; return PM_ERR_CAPACITY; }
        if (n_frames > 0 && offsets[0] != 0) { err = "set_offsets[0] must be 0"; return PM_ERR_ARG; }
        for (int f = 0; f < n_frames; ++f) {
            if (offsets[f + 1] < offsets[f]) { err = "set_offsets not monotone"; return PM_ERR_ARG; }
            if (offsets[f + 1] - offsets[f] > max_set) { err = "a frame has more adapters than max_set"; return PM_ERR_CAPACITY; }
        }
        const int nnz = n_frames > 0 ? offsets[n_frames] : 0;
        if (nnz > 0 && !ids) { err = "NULL set_ids"; return PM_ERR_ARG; }
        // unchanged sets (the common case: temporal continuity) reuse the uploaded plan
        const bool fixed = frame_of_slot != nullptr;
        if (fixed && (!src_of_slot || sort_frames)) { err = "inconsistent slot plan"; return PM_ERR_ARG; }
        if (n_frames == last_frames && sort_frames == last_sorted && (int)last_ids.size() == nnz &&
            std::equal(offsets, offsets + n_frames + 1, last_off.begin()) &&
            std::equal(ids, ids + nnz, last_ids.begin()) &&
            last_fixed.size() == (fixed ? (size_t)2 * n_frames : 0) &&
            (!fixed || (std::equal(frame_of_slot, frame_of_slot + n_frames, last_fixed.begin()) &&
                        std::equal(src_of_slot, src_of_slot + n_frames, last_fixed.begin() + n_frames))))
            return PM_OK;
        const int si = stage_next;
        stage_next = (stage_next + 1) % N_STAGE;
        if (upload_pending[si]) { CK(cudaEventSynchronize(uploaded[si])); upload_pending[si] = false; }
        const auto t_start = std::chrono::steady_clock::now();
        // per frame: sorted ids, validated
        sorted_ids.resize(nnz);
        int widest = 0;
        for (int f = 0; f < n_frames; ++f) {
            int* b = sorted_ids.data() + offsets[f];
            const int n = offsets[f + 1] - offsets[f];
            std::copy(ids + offsets[f], ids + offsets[f + 1], b);
            std::sort(b, b + n);
            for (int i = 0; i < n; ++i) {
                const int a = b[i];
                if (a < 0 || a >= max_adapters) { err = "adapter id out of range"; return PM_ERR_ARG; }
                if (i > 0 && b[i - 1] == a) { err = "duplicate adapter id in a frame's set"; return PM_ERR_ARG; }
                if (ranks[a] == 0) { err = "adapter id not registered"; return PM_ERR_STATE; }
            }
            widest = std::max(widest, n);
        }
        auto set_of = [&](int f) { return std::make_pair(sorted_ids.data() + offsets[f], sorted_ids.data() + offsets[f + 1]); };
        perm_host.resize(n_frames);
        for (int f = 0; f < n_frames; ++f) perm_host[f] = f;
        if (sort_frames)
            std::stable_sort(perm_host.begin(), perm_host.end(), [&](int a, int b) {
                const auto sa = set_of(a), sb = set_of(b);
                return std::lexicographical_compare(sa.first, sa.second, sb.first, sb.second);
            });
        uint8_t* s = (uint8_t*)stage[si];
        int* h_perm = (int*)(s + off_perm); int* h_soff = (int*)(s + off_soff); int* h_sids = (int*)(s + off_sids);
        int* h_src = (int*)(s + off_src);
        int* h_tn = (int*)(s + off_tn); int* h_ts = (int*)(s + off_ts);
        float* h_tsc = (float*)(s + off_tsc); uint32_t* h_tm = (uint32_t*)(s + off_tm);
        h_soff[0] = 0;
        for (int i = 0; i < n_frames; ++i) {
            const auto st_ = set_of(perm_host[i]);
            h_perm[i] = fixed ? frame_of_slot[i] : perm_host[i];
            h_src[i] = fixed ? src_of_slot[i] : i;
            std::copy(st_.first, st_.second, h_sids + h_soff[i]);
            h_soff[i + 1] = h_soff[i] + (int)(st_.second - st_.first);
        }
        const long long rows = (long long)n_frames * tokens;
        const int n_pairs = (int)((rows + 2 * PM_TILE_M - 1) / (2 * PM_TILE_M));
        const int n_tiles = 2 * n_pairs;
        for (int p = 0; p < n_pairs; ++p) {
            const long long r0 = (long long)p * 2 * PM_TILE_M, r1 = std::min(rows, r0 + 2 * PM_TILE_M);
            uint64_t used[4] = {0, 0, 0, 0};                // adapters of the pair's frames, and how many slabs they have
            int n_ps = 0;
            for (int slot = (int)(r0 / tokens); slot <= (int)((r1 - 1) / tokens); ++slot) {
                const int b0 = (int)(std::max(r0, (long long)slot * tokens) - r0);
                const int b1 = (int)(std::min(r1, (long long)(slot + 1) * tokens) - r0);     // bits [b0, b1)
                uint64_t m[4];
                for (int q = 0; q < 4; ++q) {
                    const int lo = std::max(b0, 64 * q) - 64 * q, hi = std::min(b1, 64 * q + 64) - 64 * q;
                    m[q] = hi <= lo ? 0ull : (hi - lo == 64 ? ~0ull : ((1ull << (hi - lo)) - 1ull) << lo);
                }
                const auto st_ = set_of(perm_host[slot]);
                for (const int* ap = st_.first; ap != st_.second; ++ap) {
                    uint64_t* rm = row_mask[*ap];
                    const uint64_t bit = 1ull << (*ap & 63);
                    if (!(used[*ap >> 6] & bit)) {
                        used[*ap >> 6] |= bit;
                        n_ps += (ranks[*ap] + PM_SLAB - 1) / PM_SLAB;
                        for (int q = 0; q < 4; ++q) rm[q] = m[q];
                    } else {
                        for (int q = 0; q < 4; ++q) rm[q] |= m[q];
                    }
                }
            }
            if (n_ps > slab_cap) { err = "tile needs more LoRA slabs than the plan capacity"; return PM_ERR_CAPACITY; }
            h_tn[2 * p] = h_tn[2 * p + 1] = n_ps;
            size_t at0 = (size_t)(2 * p) * slab_cap, at1 = at0 + slab_cap;
            for (int w = 0; w < 4; ++w)
                for (uint64_t bits = used[w]; bits; bits &= bits - 1) {
                    const int a = w * 64 + __builtin_ctzll(bits);
                    const int nsl = (ranks[a] + PM_SLAB - 1) / PM_SLAB;
                    for (int j = 0; j < nsl; ++j, ++at0, ++at1) {
                        h_ts[at0] = h_ts[at1] = a * slabs_max + j;
                        h_tsc[at0] = h_tsc[at1] = scales[a];
                        std::memcpy(h_tm + at0 * 4, row_mask[a], 16);          // rows 0..127 (little-endian words)
                        std::memcpy(h_tm + at1 * 4, row_mask[a] + 2, 16);      // rows 128..255
                    }
                }
        }
        plan_host_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
        ++plans_built;
        PlanSegments seg;
        seg.n = 0;
        auto used_part = [&](size_t off, size_t bytes) {
            if (bytes == 0) return;
            seg.at[seg.n] = (uint32_t)(off / 16);
            seg.units[seg.n++] = (uint32_t)((bytes + 15) / 16);
        };
        const size_t entries = (size_t)n_tiles * slab_cap;
        used_part(off_perm, sizeof(int) * n_frames);
        used_part(off_soff, sizeof(int) * (n_frames + 1));
        used_part(off_sids, sizeof(int) * nnz);
        used_part(off_src, sizeof(int) * n_frames);
        used_part(off_tn, sizeof(int) * n_tiles);
        used_part(off_ts, sizeof(int) * entries);
        used_part(off_tsc, sizeof(float) * entries);
        used_part(off_tm, sizeof(uint32_t) * 4 * entries);
        CK(launch_plan_upload(L, stage[si], blob.p, seg));
        CK(cudaEventRecord(uploaded[si], L.st));
        upload_pending[si] = true;
        ++version; device_plan_frames = -1;
        dev.n_frames = n_frames; dev.n_tiles = n_tiles; dev.max_set = widest;
        last_off.assign(offsets, offsets + n_frames + 1);
        last_ids.assign(ids, ids + nnz);
        last_fixed.clear();
        if (fixed) {
            last_fixed.assign(frame_of_slot, frame_of_slot + n_frames);
            last_fixed.insert(last_fixed.end(), src_of_slot, src_of_slot + n_frames);
        }
        last_frames = n_frames; last_sorted = sort_frames;
        return PM_OK;
    }
    void invalidate() { last_frames = -1; }

    // The same tables built by kernels from a CSR on the device; the host never sees the sets, so
    // max_set is the handle's upper bound and the cached host plan is forgotten.
    int build_on_device(const Launch& L, int n_frames, const int32_t* d_off, const int32_t* d_ids,
                        const AdapterMeta& meta, std::string& err) {
        if (n_frames > max_frames || n_frames > PM_DEVICE_PLAN_MAX_FRAMES) { err = "n_frames exceeds the device planner's limit"; return PM_ERR_CAPACITY; }
        invalidate();
        if (device_plan_frames != n_frames) { ++version; device_plan_frames = n_frames; }
        dev.n_frames = n_frames;
        dev.n_tiles = (int)(((long long)n_frames * tokens + 2 * PM_TILE_M - 1) / (2 * PM_TILE_M)) * 2;
        dev.max_set = max_set;
        CK(launch_device_plan(L, dev, n_frames, max_set, max_adapters, slabs_max, d_off, d_ids, meta));
        return PM_OK;
    }
};

// Copies a CSR that may live on the device to the host (synchronising the stream if it does).
int fetch_csr(const int32_t* offsets, const int32_t* ids, int n_frames, cudaStream_t st,
              std::vector<int32_t>& hoff, std::vector<int32_t>& hids, const int32_t** o, const int32_t** i,
              std::string& err) {
    *o = offsets; *i = ids;
    if (!offsets || n_frames <= 0) return PM_OK;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, offsets) != cudaSuccess) { cudaGetLastError(); return PM_OK; }
    if (at.type != cudaMemoryTypeDevice) return PM_OK;
    hoff.resize(n_frames + 1);
    CK(cudaMemcpyAsync(hoff.data(), offsets, sizeof(int32_t) * (n_frames + 1), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const int nnz = hoff[n_frames];
    if (nnz < 0) { err = "negative set_offsets"; return PM_ERR_ARG; }
    hids.resize(std::max(nnz, 1));
    if (nnz > 0) {
        if (!ids) { err = "NULL set_ids"; return PM_ERR_ARG; }
        CK(cudaMemcpyAsync(hids.data(), ids, sizeof(int32_t) * nnz, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    *o = hoff.data(); *i = hids.data();
    return PM_OK;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// handles
// ---------------------------------------------------------------------------------------
struct pm_linear_s {
    int k_in = 0, n_out = 0, max_adapters = 0, max_rank = 0, slabs_max = 0, max_set = 0, max_frames = 0;
    int tokens = 0, epilogue = 0, dtype = 0, n_sms = 148;
    LinearObj lin;
    Router router;
    std::vector<int> ranks;
    std::vector<float> scales;
    DevBuf scale_dev, rank_dev, t32, tbuf, status;
    AdapterMeta meta;
    CUtensorMap tm_t;
    long long launches = 0;
    std::string err;
};

struct pm_handle_s {
    pm_config cfg;
    int tokens = 0, g2 = 0, patch_dim = 0, slabs_max = 0, n_sms = 148;
    LinearObj patch;                         // no LoRA
    std::vector<LinearObj> lin;              // [layers*4]
    DevBuf cls, pos, ln1_g, ln1_b, ln2_g, ln2_b, lnf_g, lnf_b, head_wt, head_b;
    // activations
    DevBuf X, U, QKV, ATT, H, PATCH, Z, t32, tbuf, status, ln_stats;
    CUtensorMap tm_patch, tm_att, tm_h, tm_t, tm_x_in;
    CUtensorMap tm_y_qkv, tm_y_x, tm_y_h;      // outputs, for the TMA-store epilogue
    CUtensorMap tm_att_q, tm_att_kv;           // attention operands over QKV
    ActMaps sm_patch, sm_att, sm_h, sm_x;  // x operands of the few-row linear kernel and the shrink
    int tm_rows = -1;
    Router router;
    // adapters
    std::vector<int> ranks;
    std::vector<float> scales;
    std::vector<std::vector<int32_t>> cls_ids;
    std::vector<std::vector<float>> head_w, head_b_host, acc;
    DevBuf scale_dev, rank_dev, hcat, hbias, hcls, hoff;
    AdapterMeta meta;
    bool heads_dirty = true;
    int most_cls = 0;                // longest class list of an adapter
    // cover tables
    DevBuf first, provider, mask_scratch, metrics;
    bool cover_ready = false;
    long long launches = 0;
    Profiler prof;
    std::string err;
    // whole-network kernel for a handful of frames (latency_kernel.cu)
    DevBuf lat_lin, lat_kv, lat_bar;
    CUtensorMap lat_tm_kv;
    bool lat_dirty = true, lat_on = true;
    // recorded launch sequences of the forward entry points (see run_graphed)
    struct GraphEntry {
        const void* key_ptr[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
        int key_int[4] = {0, 0, 0, 0};
        unsigned long long plan_version = 0;
        cudaStream_t st = nullptr;
        bool small_batch = true;            // pm_set_small_batch_kernel at the time: chooses kernels linear by linear
        cudaGraphExec_t exec = nullptr;     // null: seen once, not recorded yet
        long long launches = 0;
        unsigned long long last_use = 0;
        bool same_key(const GraphEntry& o) const {
            return std::equal(key_ptr, key_ptr + 5, o.key_ptr) && std::equal(key_int, key_int + 4, o.key_int) &&
                   plan_version == o.plan_version && st == o.st && small_batch == o.small_batch;
        }
    };
    std::vector<GraphEntry> graphs;
    bool graphs_on = true;
    unsigned long long graph_clock = 0;
    void drop_graphs() {
        for (GraphEntry& g : graphs) if (g.exec) cudaGraphExecDestroy(g.exec);
        graphs.clear();
    }
    ~pm_handle_s() { drop_graphs(); }
};

namespace {

// Runs `enqueue` (which puts one forward's kernels on `key.st`), recording it as a CUDA graph the
// second time the same call is seen -- same buffers, sizes, stream and routing plan -- and replaying
// the graph from then on: back-to-back kernels of a replay start about 2 us closer to each other than
// individually launched ones.  Falls back to plain launches on the legacy default stream (it cannot
// be captured), while the caller is itself capturing, and while per-launch profiling is on.
template <typename F>
int run_graphed(pm_handle_s* h, pm_handle_s::GraphEntry key, F&& enqueue) {
    constexpr size_t MAX_GRAPHS = 8;
    std::string& err = h->err;
    cudaStream_t st = key.st;
    key.small_batch = h->lat_on;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (!h->graphs_on || h->prof.on || st == nullptr || st == cudaStreamLegacy ||
        cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return enqueue();
    }
    pm_handle_s::GraphEntry* e = nullptr;
    for (auto& g : h->graphs) if (g.same_key(key)) e = &g;
    if (!e) {                                    // first sighting: remember it, launch plainly
        if (h->graphs.size() >= MAX_GRAPHS) {
            size_t old = 0;
            for (size_t i = 1; i < h->graphs.size(); ++i) if (h->graphs[i].last_use < h->graphs[old].last_use) old = i;
            if (h->graphs[old].exec) cudaGraphExecDestroy(h->graphs[old].exec);
            h->graphs.erase(h->graphs.begin() + old);
        }
        key.last_use = ++h->graph_clock;
        h->graphs.push_back(key);
        return enqueue();
    }
    e->last_use = ++h->graph_clock;
    if (!e->exec) {                              // second sighting: record
        const long long l0 = h->launches;
        if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            cudaGetLastError();
            h->graphs_on = false;
            return enqueue();
        }
        const int rc = enqueue();
        cudaGraph_t g = nullptr;
        const cudaError_t ce = cudaStreamEndCapture(st, &g);
        const long long recorded = h->launches - l0;
        h->launches = l0;                        // nothing has run yet
        cudaGraphExec_t exec = nullptr;
        if (rc == PM_OK && ce == cudaSuccess && g && cudaGraphInstantiate(&exec, g, 0) == cudaSuccess) {
            e->exec = exec;
            e->launches = recorded;
        }
        if (g) cudaGraphDestroy(g);
        if (!e->exec) {                          // could not record: never try again on this handle
            cudaGetLastError();
            h->graphs_on = false;
            if (rc != PM_OK) return rc;
            return enqueue();
        }
    }
    CK(cudaGraphLaunch(e->exec, st));
    h->launches += e->launches;
    return PM_OK;
}

int slabs_for(int max_rank) { return (max_rank + PM_SLAB - 1) / PM_SLAB; }

int sync_meta(DevBuf& scale_dev, DevBuf& rank_dev, const std::vector<float>& scales,
              const std::vector<int>& ranks, std::string& err) {
    CK(cudaMemcpy(scale_dev.p, scales.data(), scales.size() * sizeof(float), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(rank_dev.p, ranks.data(), ranks.size() * sizeof(int), cudaMemcpyHostToDevice));
    return PM_OK;
}

template <typename T>
int rebuild_heads(pm_handle_s* h) {
    std::string& err = h->err;
    const int d = h->cfg.d, na = h->cfg.max_adapters;
    std::vector<int> hoff(na + 1, 0);
    for (int a = 0; a < na; ++a) hoff[a + 1] = hoff[a] + (h->ranks[a] ? (int)h->cls_ids[a].size() : 0);
    h->most_cls = 0;
    for (int a = 0; a < na; ++a) h->most_cls = std::max(h->most_cls, hoff[a + 1] - hoff[a]);
    const int total = hoff[na];
    std::vector<T> hc((size_t)std::max(total, 1) * d);
    std::vector<float> hb(std::max(total, 1));
    std::vector<int> hk(std::max(total, 1));
    for (int a = 0; a < na; ++a) {
        if (!h->ranks[a]) continue;
        const int n = (int)h->cls_ids[a].size();
        for (int j = 0; j < n; ++j) {
            const int r = hoff[a] + j;
            for (int c = 0; c < d; ++c) hc[(size_t)r * d + c] = host_cvt<T>(h->head_w[a][(size_t)c * n + j]);
            hb[r] = h->head_b_host[a][j];
            hk[r] = h->cls_ids[a][j];
        }
    }
    CK(h->hcat.alloc(hc.size() * sizeof(T)));
    CK(h->hbias.alloc(hb.size() * sizeof(float)));
    CK(h->hcls.alloc(hk.size() * sizeof(int)));
    CK(h->hoff.alloc(hoff.size() * sizeof(int)));
    CK(cudaMemcpy(h->hcat.p, hc.data(), hc.size() * sizeof(T), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(h->hbias.p, hb.data(), hb.size() * sizeof(float), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(h->hcls.p, hk.data(), hk.size() * sizeof(int), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(h->hoff.p, hoff.data(), hoff.size() * sizeof(int), cudaMemcpyHostToDevice));
    h->heads_dirty = false;
    return PM_OK;
}

int encode_activation_maps(pm_handle_s* h, int rows) {
    if (h->tm_rows == rows) return PM_OK;
    const int d = h->cfg.d;
    const int prow = rows / h->tokens * h->g2;
    bool ok = tm_encode_2d(&h->tm_patch, h->PATCH.p, h->patch_dim, prow, (uint64_t)h->patch_dim * 2, 64, PM_TILE_M, 128)
           && tm_encode_2d(&h->tm_x_in, h->X.p, d, rows, (uint64_t)d * 2, 64, PM_TILE_M, 128)
           && tm_encode_2d(&h->tm_att, h->ATT.p, d, rows, (uint64_t)d * 2, 64, PM_TILE_M, 128)
           && tm_encode_2d(&h->tm_h, h->H.p, h->cfg.mlp, rows, (uint64_t)h->cfg.mlp * 2, 64, PM_TILE_M, 128)
           && tm_encode_2d(&h->tm_y_qkv, h->QKV.p, 3 * d, rows, (uint64_t)3 * d * 2, 32, 32, 64)
           && tm_encode_2d(&h->tm_y_x, h->X.p, d, rows, (uint64_t)d * 2, 32, 32, 64)
           && tm_encode_2d(&h->tm_y_h, h->H.p, h->cfg.mlp, rows, (uint64_t)h->cfg.mlp * 2, 32, 32, 64)
           && attention_encode_maps(h->QKV.as<bf16>(), rows / h->tokens, h->tokens, h->cfg.heads, &h->tm_att_q,
                                    &h->tm_att_kv)
           && act_encode(&h->sm_patch, h->PATCH.p, h->patch_dim, prow) && act_encode(&h->sm_x, h->X.p, d, rows)
           && act_encode(&h->sm_att, h->ATT.p, d, rows) && act_encode(&h->sm_h, h->H.p, h->cfg.mlp, rows);
    if (!ok) { h->err = "cuTensorMapEncodeTiled failed (activations)"; return PM_ERR_CUDA; }
    h->tm_rows = rows;
    return PM_OK;
}

// n_frames frames enter; the first trunk_layers blocks run on them without adapters; then every
// frame's rows are copied to its further slots (n_slots >= n_frames in all; slot i < n_frames is
// frame perm[i] itself) and the remaining blocks and the heads run on all slots with the plan's
// per-slot adapter sets.  The one-stream forward is trunk_layers = 0, n_slots = n_frames.
template <typename T>
int forward_t(pm_handle_s* h, const void* frames, int n_frames, int n_slots, int trunk_layers,
              float* scores_out, float* base_out, cudaStream_t st) {
    std::string& err = h->err;
    const pm_config& c = h->cfg;
    const int T_ = h->tokens, d = c.d;
    int rows = n_frames * T_;
    Launch L; L.st = st; L.launches = &h->launches; L.status = h->status.as<int>(); L.prof = &h->prof;
    const RouteDev& R = h->router.dev;
    constexpr bool TC = sizeof(T) == 2;
    if (TC) { int rc = encode_activation_maps(h, rows); if (rc) return rc; }
    PatchEpi pe; pe.g2 = h->g2; pe.tokens = T_; pe.pos = h->pos.as<float>();
    PatchEpi none;
    T* X = h->X.as<T>(); T* U = h->U.as<T>(); T* QKV = h->QKV.as<T>(); T* ATT = h->ATT.as<T>();
    T* Hb = h->H.as<T>(); T* P = h->PATCH.as<T>();

    // st: per-row LayerNorm statistics of x when the linear has its LayerNorm folded in, else null
    auto linear = [&](LinearObj& lo, const T* x, const CUtensorMap* tmx, int nrows, int tokens_pf, bool lora,
                      int epi, const T* residual, const PatchEpi& pep, T* y, const float2* st = nullptr) -> cudaError_t {
        if constexpr (TC) {
            const bool use_lora = lora && R.max_set > 0 && lo.n_adapted > 0;
            // few rows: the whole linear in one kernel, with tiles for one wave of the SMs
            const ActMaps& sx = tmx == &h->tm_patch ? h->sm_patch : tmx == &h->tm_att ? h->sm_att : tmx == &h->tm_h ? h->sm_h : h->sm_x;
            if (h->lat_on && small_linear_fits(lo.dev, use_lora ? &R : nullptr, nrows, epi, h->n_sms))
                return launch_small_linear(L, lo.dev, use_lora ? &R : nullptr, sx, nrows, epi, (const bf16*)residual, pep, (bf16*)y,
                                           h->n_sms, c.ln_eps);
            if (use_lora) {
                // with LayerNorm folded in, the shrink computes the row statistics on its way through x
                cudaError_t e = launch_shrink(L, lo.dev, R, sx, nrows, h->tbuf.as<bf16>(), h->n_sms, const_cast<float2*>(st), c.ln_eps);
                if (e != cudaSuccess) return e;
            } else if (st) {
                cudaError_t e = launch_row_stats(L, (const bf16*)x, const_cast<float2*>(st), nrows, lo.dev.k_in, c.ln_eps);
                if (e != cudaSuccess) return e;
            }
            const CUtensorMap* tmy = (void*)y == h->QKV.p ? &h->tm_y_qkv
                                   : (void*)y == h->H.p ? &h->tm_y_h
                                   : (void*)y == h->X.p ? &h->tm_y_x : nullptr;
            return launch_lora_gemm(L, lo.dev, use_lora ? &R : nullptr, *tmx, &h->tm_t, tmy, nrows, epi,
                                    (const bf16*)residual, pep, (bf16*)y, h->n_sms, st, use_lora);
        } else {
            return launch_naive_linear<T>(L, lo.dev, R, h->meta, h->slabs_max, x, nrows, tokens_pf,
                                          lora ? h->t32.as<float>() : nullptr, epi, residual, pep, y);
        }
    };

    CK(launch_im2col<T>(L, (const T*)frames, R.perm, P, n_frames, c.img, c.patch, h->cls.as<float>(), h->pos.as<float>(), X, d, h->n_sms));
    CK(linear(h->patch, P, &h->tm_patch, n_frames * h->g2, h->g2, false, EPI_PATCH, nullptr, pe, X));
    int n_cur = n_frames;                     // slots the blocks currently run on
    for (int l = 0; l <= c.layers; ++l) {
        if (l == trunk_layers && n_slots != n_cur) {
            // end of the shared trunk: every further slot starts from its frame's rows
            CK(launch_fanout_rows<T>(L, X, R.src_slot, n_frames, n_slots, T_, d));
            n_cur = n_slots;
            rows = n_slots * T_;
            if (TC) { int rc = encode_activation_maps(h, rows); if (rc) return rc; }
        }
        if (l == c.layers) break;
        const bool lora = l >= trunk_layers;
        if constexpr (TC) {
            // LayerNorm 1 is folded into the qkv weights: only the row statistics are computed (by the
            // shrink when there is one, else by a pass of their own)
            CK(linear(h->lin[l * 4 + 0], X, &h->tm_x_in, rows, T_, lora, EPI_NONE, nullptr, none, QKV, h->ln_stats.as<float2>()));
        } else {
            CK(launch_layernorm<T>(L, X, h->ln1_g.as<float>() + (size_t)l * d, h->ln1_b.as<float>() + (size_t)l * d, U, rows, d, c.ln_eps));
            CK(linear(h->lin[l * 4 + 0], U, nullptr, rows, T_, lora, EPI_NONE, nullptr, none, QKV));
        }
        if constexpr (TC) {
            if (attention_tc_supported(T_))
                CK(launch_attention_tc(L, h->tm_att_q, h->tm_att_kv, (const bf16*)QKV, (bf16*)ATT, n_cur, T_, c.heads, h->n_sms));
            else
                CK(launch_attention_mma(L, (const bf16*)QKV, (bf16*)ATT, n_cur, T_, c.heads));
        }
        else CK(launch_attention_simple<T>(L, QKV, ATT, n_cur, T_, c.heads));
        CK(linear(h->lin[l * 4 + 1], ATT, &h->tm_att, rows, T_, lora, EPI_RESIDUAL, X, none, X));
        if constexpr (TC) {
            CK(linear(h->lin[l * 4 + 2], X, &h->tm_x_in, rows, T_, lora, EPI_GELU, nullptr, none, Hb, h->ln_stats.as<float2>()));
        } else {
            CK(launch_layernorm<T>(L, X, h->ln2_g.as<float>() + (size_t)l * d, h->ln2_b.as<float>() + (size_t)l * d, U, rows, d, c.ln_eps));
            CK(linear(h->lin[l * 4 + 2], U, nullptr, rows, T_, lora, EPI_GELU, nullptr, none, Hb));
        }
        CK(linear(h->lin[l * 4 + 3], Hb, &h->tm_h, rows, T_, lora, EPI_RESIDUAL, X, none, X));
    }
    CK(launch_heads<T>(L, X, n_slots, n_frames, n_frames, T_, d, c.ln_eps, h->lnf_g.as<float>(), h->lnf_b.as<float>(),
                       h->Z.as<float>(), h->head_wt.as<T>(), h->head_b.as<float>(), c.n_classes,
                       h->hcat.as<T>(), h->hbias.as<float>(), h->hcls.as<int>(), h->hoff.as<int>(), h->most_cls, R,
                       scores_out, base_out, h->n_sms));
    return PM_OK;
}

// ---- the whole-network kernel: small batches of small models in one launch --------------------------
constexpr int LAT_ROWS = 16;
int lat_tiles_per_frame(const pm_handle_s* h) { return (h->tokens + LAT_ROWS - 1) / LAT_ROWS; }

bool latency_eligible(const pm_handle_s* h, int n_frames) {
    const pm_config& c = h->cfg;
    if (!h->lat_on || c.dtype != 0 || c.d > 384 || c.mlp > 1536 || h->patch_dim > 1536 || c.max_set > 8) return false;
    if (c.d % 64 || c.mlp % 64 || h->patch_dim % 64 || c.d / c.heads != 64 || c.patch != 16) return false;
    if (h->tokens > 256) return false;               // a head's keys are one TMA box
    if (h->slabs_max * c.max_set > 8 || c.layers > 64) return false;                  // LoRA slabs of one linear: one ring step
    if ((long long)n_frames * lat_tiles_per_frame(h) > h->n_sms) return false;       // one CTA per SM, all resident
    return latency_smem_bytes(c.d, c.mlp, h->patch_dim, h->tokens, c.layers) <= 227 * 1024;
}

// slots: perm (slot -> frame) or null; set lists: device CSR over slots
int forward_latency(pm_handle_s* h, const void* frames, int n_frames, const int* perm, const int* d_off, const int* d_ids,
                    float* scores_out, float* base_out, cudaStream_t st) {
    std::string& err = h->err;
    const pm_config& c = h->cfg;
    bool maps_ok = true;
    auto view = [&](const LinearObj& lo) {
        LatLinear v;
        std::memset(&v, 0, sizeof(v));
        v.Wt = (const bf16*)lo.dev.Wt; v.bias = lo.dev.bias; v.ln_g = lo.dev.ln_g;
        v.At = (const bf16*)lo.dev.lora.At; v.Bt = (const bf16*)lo.dev.lora.Bt; v.c1 = lo.dev.ln_c1; v.c2 = lo.dev.ln_c2;
        for (size_t a = 0; a < lo.adapted.size() && a < 256; ++a) if (lo.adapted[a]) v.adapted[a >> 5] |= 1u << (a & 31);
        if (lo.n_adapted == 0) { v.At = nullptr; v.Bt = nullptr; }
        v.k_in = lo.dev.k_in; v.n_out = lo.dev.n_out;
        // the kernel's own boxes: half a chunk of outputs, one slab of A^T, a chunk's rows of one slab of B^T
        maps_ok = maps_ok && tm_encode_2d(&v.tm_w, lo.dev.Wt, v.k_in, v.n_out, (uint64_t)v.k_in * 2, 64, 64, 128);
        if (v.At) {
            const uint64_t arena_slabs = (uint64_t)c.max_adapters * h->slabs_max;
            maps_ok = maps_ok && tm_encode_2d(&v.tm_at, lo.dev.lora.At, v.k_in, arena_slabs * PM_SLAB, (uint64_t)v.k_in * 2, 64, PM_SLAB, 128);
            maps_ok = maps_ok && tm_encode_2d(&v.tm_bt, lo.dev.lora.Bt, PM_SLAB, arena_slabs * v.n_out, PM_SLAB * 2, PM_SLAB, 128, 32);
        }
        return v;
    };
    if (h->lat_dirty) {
        std::vector<LatLinear> lv;
        for (const LinearObj& lo : h->lin) lv.push_back(view(lo));
        lv.push_back(view(h->patch));
        lv.back().At = nullptr; lv.back().Bt = nullptr;         // the patch projection carries no adapter
        if (!maps_ok) { err = "cuTensorMapEncodeTiled failed (whole-network kernel)"; return PM_ERR_CUDA; }
        CK(h->lat_lin.alloc(lv.size() * sizeof(LatLinear)));
        CK(cudaMemcpy(h->lat_lin.p, lv.data(), lv.size() * sizeof(LatLinear), cudaMemcpyHostToDevice));
        if (!h->lat_kv.p) {
            const int max_f = h->n_sms / lat_tiles_per_frame(h);
            const size_t kv_rows = (size_t)2 * std::max(1, max_f) * h->tokens;
            CK(h->lat_kv.alloc(kv_rows * 2 * c.d * sizeof(bf16)));
            CK(cudaMemset(h->lat_kv.p, 0, h->lat_kv.bytes));
            CK(h->lat_bar.alloc(sizeof(unsigned int) * std::max(1, max_f) * c.heads));     // a frame's counters: one, or one per head
            const int tpad = (h->tokens + 15) / 16 * 16;
            if (tpad > 256 || !tm_encode_2d(&h->lat_tm_kv, h->lat_kv.p, (uint64_t)2 * c.d, kv_rows, (uint64_t)2 * c.d * 2, 64, tpad, 128)) {
                err = "cuTensorMapEncodeTiled failed (key/value exchange buffer)"; return PM_ERR_CUDA;
            }
        }
        h->lat_dirty = false;
    }
    LatArgs a;
    a.frames = (const bf16*)frames; a.n_frames = n_frames; a.img = c.img; a.grid = c.img / c.patch; a.tokens = h->tokens;
    a.tiles_pf = lat_tiles_per_frame(h); a.d = c.d; a.heads = c.heads; a.mlp = c.mlp; a.layers = c.layers;
    a.n_classes = c.n_classes; a.patch_dim = h->patch_dim; a.eps = c.ln_eps;
    a.lin = h->lat_lin.as<LatLinear>(); a.tm_kv = h->lat_tm_kv;
    a.cls = h->cls.as<float>(); a.pos = h->pos.as<float>(); a.lnf_g = h->lnf_g.as<float>(); a.lnf_b = h->lnf_b.as<float>();
    a.head_wt = h->head_wt.as<bf16>(); a.head_b = h->head_b.as<float>();
    a.hcat = h->hcat.as<bf16>(); a.hbias = h->hbias.as<float>(); a.hcls = h->hcls.as<int>(); a.hoff = h->hoff.as<int>();
    a.set_off = d_off; a.set_ids = d_ids; a.perm = perm;
    a.max_set = c.max_set; a.max_adapters = c.max_adapters; a.slabs_max = h->slabs_max;
    a.rank = h->meta.rank; a.scale = h->meta.scale;
    a.kv = h->lat_kv.as<bf16>(); a.bar = h->lat_bar.as<unsigned int>();
    a.scores_out = scores_out; a.base_out = base_out; a.status = nullptr;
    Launch L; L.st = st; L.launches = &h->launches; L.status = h->status.as<int>(); L.prof = &h->prof;
    CK(launch_latency_forward(L, a));
    return PM_OK;
}

template <typename T>
int create_t(pm_handle_s* h, const pm_backbone* w) {
    std::string& err = h->err;
    const pm_config& c = h->cfg;
    const int d = c.d, L = c.layers, m = c.mlp, K = c.n_classes, T_ = h->tokens;
    int rc = h->patch.init(h->patch_dim, d, w->patch_w, w->patch_b, 0, 0, c.dtype, err);
    if (rc) return rc;
    h->lin.resize((size_t)L * 4);
    for (int l = 0; l < L; ++l) {
        const float* ws[4] = {w->qkv_w + (size_t)l * d * 3 * d, w->proj_w + (size_t)l * d * d,
                              w->fc1_w + (size_t)l * d * m, w->fc2_w + (size_t)l * m * d};
        const float* bs[4] = {w->qkv_b + (size_t)l * 3 * d, w->proj_b + (size_t)l * d,
                              w->fc1_b + (size_t)l * m, w->fc2_b + (size_t)l * d};
        const int kin[4] = {d, d, d, m}, nout[4] = {3 * d, d, m, d};
        for (int p = 0; p < 4; ++p) {
            // qkv follows LayerNorm 1 and fc1 follows LayerNorm 2: folded into their weights (bf16 build)
            const float* lg = p == 0 ? w->ln1_g + (size_t)l * d : p == 2 ? w->ln2_g + (size_t)l * d : nullptr;
            const float* lb = p == 0 ? w->ln1_b + (size_t)l * d : p == 2 ? w->ln2_b + (size_t)l * d : nullptr;
            rc = h->lin[l * 4 + p].init(kin[p], nout[p], ws[p], bs[p], c.max_adapters, h->slabs_max, c.dtype, err, lg, lb);
            if (rc) return rc;
        }
    }
    CK(upload<float>(h->cls, w->cls, d));
    CK(upload<float>(h->pos, w->pos, (size_t)T_ * d));
    CK(upload<float>(h->ln1_g, w->ln1_g, (size_t)L * d)); CK(upload<float>(h->ln1_b, w->ln1_b, (size_t)L * d));
    CK(upload<float>(h->ln2_g, w->ln2_g, (size_t)L * d)); CK(upload<float>(h->ln2_b, w->ln2_b, (size_t)L * d));
    CK(upload<float>(h->lnf_g, w->lnf_g, d)); CK(upload<float>(h->lnf_b, w->lnf_b, d));
    CK(upload_transposed<T>(h->head_wt, w->head_w, d, K));
    CK(upload<float>(h->head_b, w->head_b, K));
    const size_t rows = (size_t)c.max_frames * T_;
    const size_t rows_pad = (rows + PM_TILE_M - 1) / PM_TILE_M * PM_TILE_M;
    // U holds the normalised rows of the fp32 build only (the bf16 build folds LayerNorm into the weights)
    CK(h->X.alloc(rows_pad * d * sizeof(T))); CK(h->U.alloc(sizeof(T) == 2 ? 0 : rows_pad * d * sizeof(T)));
    CK(h->QKV.alloc(rows_pad * 3 * d * sizeof(T))); CK(h->ATT.alloc(rows_pad * d * sizeof(T)));
    CK(h->H.alloc(rows_pad * m * sizeof(T)));
    CK(h->PATCH.alloc(rows_pad * h->patch_dim * sizeof(T)));
    CK(h->Z.alloc(sizeof(T) == 2 ? 0 : (size_t)c.max_frames * d * sizeof(float)));      // the bf16 build's heads normalise their rows themselves
    CK(h->ln_stats.alloc(rows_pad * sizeof(float2)));
    CK(cudaMemset(h->X.p, 0, h->X.bytes)); if (h->U.p) CK(cudaMemset(h->U.p, 0, h->U.bytes));
    CK(cudaMemset(h->QKV.p, 0, h->QKV.bytes)); CK(cudaMemset(h->ATT.p, 0, h->ATT.bytes));
    CK(cudaMemset(h->H.p, 0, h->H.bytes)); CK(cudaMemset(h->PATCH.p, 0, h->PATCH.bytes));
    rc = h->router.init(c.max_frames, c.max_set, c.max_adapters, h->slabs_max, T_, err);
    if (rc) return rc;
    if (c.dtype == 0) {
        const size_t tb = (size_t)h->router.max_tiles * std::max(1, h->router.slab_cap) * PM_TILE_M * PM_SLAB;
        CK(h->tbuf.alloc(tb * sizeof(bf16)));
        CK(cudaMemset(h->tbuf.p, 0, h->tbuf.bytes));
        if (!tm_encode_2d(&h->tm_t, h->tbuf.p, PM_SLAB, tb / PM_SLAB, PM_SLAB * 2, PM_SLAB, PM_TILE_M, 32)) {
            err = "cuTensorMapEncodeTiled failed (slab buffer)"; return PM_ERR_CUDA;
        }
    } else {
        CK(h->t32.alloc(rows * std::max(1, c.max_set) * h->slabs_max * PM_SLAB * sizeof(float)));
    }
    return PM_OK;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// exported functions
// ---------------------------------------------------------------------------------------
extern "C" {

int pm_create(const pm_config* cfg, const pm_backbone* w, pm_handle* out) {
    if (!cfg || !w || !out) return PM_ERR_ARG;
    *out = nullptr;
    const pm_config& c = *cfg;
    if (c.patch != 16 || c.img <= 0 || c.img % c.patch || c.d <= 0 || c.d % 64 || c.heads <= 0 ||
        c.d != c.heads * 64 || c.mlp <= 0 || c.mlp % 64 || c.layers <= 0 || c.n_classes <= 0 ||
        c.d > 1024 || c.max_adapters < 0 || c.max_adapters > 256 || c.max_rank < 0 || c.max_set < 0 ||
        c.max_frames <= 0 || (c.dtype != 0 && c.dtype != 1))
        return PM_ERR_ARG;
    const float* const* fields = reinterpret_cast<const float* const*>(w);
    for (size_t i = 0; i < sizeof(pm_backbone) / sizeof(const float*); ++i)
        if (!fields[i]) return PM_ERR_ARG;
    pm_handle_s* h = new (std::nothrow) pm_handle_s();
    if (!h) return PM_ERR_OOM;
    h->cfg = c;
    const int g = c.img / c.patch;
    h->g2 = g * g; h->tokens = g * g + 1; h->patch_dim = 3 * c.patch * c.patch;
    h->slabs_max = slabs_for(c.max_rank);
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&h->n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        delete h; return PM_ERR_CUDA;
    }
    h->ranks.assign(std::max(1, c.max_adapters), 0);
    h->scales.assign(std::max(1, c.max_adapters), 0.f);
    h->cls_ids.resize(c.max_adapters); h->head_w.resize(c.max_adapters);
    h->head_b_host.resize(c.max_adapters); h->acc.resize(c.max_adapters);
    int rc = c.dtype == 0 ? create_t<bf16>(h, w) : create_t<float>(h, w);
    std::string& err = h->err;
    auto fail = [&](int code) { fprintf(stderr, "pm_create: %s\n", h->err.c_str()); delete h; return code; };
    if (rc) return fail(rc);
    if (h->scale_dev.alloc(h->scales.size() * sizeof(float)) != cudaSuccess ||
        h->rank_dev.alloc(h->ranks.size() * sizeof(int)) != cudaSuccess ||
        h->status.alloc(sizeof(int)) != cudaSuccess ||
        cudaMemset(h->status.p, 0, sizeof(int)) != cudaSuccess) { err = "allocation failed"; return fail(PM_ERR_OOM); }
    rc = sync_meta(h->scale_dev, h->rank_dev, h->scales, h->ranks, err);
    if (rc) return fail(rc);
    h->meta.scale = h->scale_dev.as<float>(); h->meta.rank = h->rank_dev.as<int>();
    if (cudaDeviceSynchronize() != cudaSuccess) { err = "device synchronize failed"; return fail(PM_ERR_CUDA); }
    *out = h;
    return PM_OK;
}

int pm_register_adapter(pm_handle h, int id, const pm_adapter* a) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    const pm_config& c = h->cfg;
    if (!a || id < 0 || id >= c.max_adapters) { err = "adapter id out of range"; return PM_ERR_ARG; }
    if (a->rank <= 0 || a->rank > c.max_rank) { err = "adapter rank exceeds max_rank"; return PM_ERR_CAPACITY; }
    if (!a->A || !a->B || a->n_cls < 0 || (a->n_cls > 0 && (!a->class_ids || !a->head_w || !a->head_b))) {
        err = "NULL adapter field"; return PM_ERR_ARG;
    }
    std::vector<char> seen(c.n_classes, 0);
    for (int j = 0; j < a->n_cls; ++j) {
        const int k = a->class_ids[j];
        if (k < 0 || k >= c.n_classes || seen[k]) { err = "class ids must be distinct and in range"; return PM_ERR_ARG; }
        seen[k] = 1;
    }
    for (int i = 0; i < c.layers * 4; ++i)
        if ((a->A[i] == nullptr) != (a->B[i] == nullptr)) { err = "A and B must both be given or both NULL"; return PM_ERR_ARG; }
    for (int i = 0; i < c.layers * 4; ++i) {
        int rc = h->lin[i].set_adapter(id, a->rank, a->A[i], a->B[i], err);
        if (rc) return rc;
    }
    h->ranks[id] = a->rank; h->scales[id] = a->scale;
    h->cls_ids[id].assign(a->class_ids, a->class_ids + a->n_cls);
    h->head_w[id].assign(a->head_w, a->head_w + (size_t)c.d * a->n_cls);
    h->head_b_host[id].assign(a->head_b, a->head_b + a->n_cls);
    if (a->acc) h->acc[id].assign(a->acc, a->acc + a->n_cls);
    else h->acc[id].assign(a->n_cls, 1.f);
    h->heads_dirty = true; h->cover_ready = false; h->lat_dirty = true;
    h->router.invalidate();
    h->drop_graphs();                 // recorded launch sequences refer to the old adapters and heads
    return sync_meta(h->scale_dev, h->rank_dev, h->scales, h->ranks, err);
}

int pm_set_cover(pm_handle h, float tau) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    const int K = h->cfg.n_classes, na = h->cfg.max_adapters;
    const int AW = std::max(1, (na + 63) / 64);
    // Algorithm 2 visits contexts by increasing size |C| (all listed classes), ties by id
    std::vector<int> order;
    for (int a = 0; a < na; ++a) if (h->ranks[a]) order.push_back(a);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        return h->cls_ids[x].size() < h->cls_ids[y].size();
    });
    std::vector<int> first(K, -1);
    std::vector<uint64_t> prov((size_t)K * AW, 0);
    for (int a : order)
        for (size_t j = 0; j < h->cls_ids[a].size(); ++j) {
            if (!(h->acc[a][j] >= tau)) continue;
            const int k = h->cls_ids[a][j];
            if (first[k] < 0) first[k] = a;
            prov[(size_t)k * AW + (a >> 6)] |= 1ull << (a & 63);
        }
    CK(h->first.alloc(first.size() * sizeof(int)));
    CK(h->provider.alloc(prov.size() * sizeof(uint64_t)));
    // the select kernel's block counter (word 0, zero between launches) + per-frame adapter masks
    CK(h->mask_scratch.alloc((1 + (size_t)h->cfg.max_frames * AW) * sizeof(uint64_t)));
    CK(cudaMemset(h->mask_scratch.p, 0, h->mask_scratch.bytes));
    if (!h->metrics.p) {
        CK(h->metrics.alloc(3 * sizeof(unsigned long long)));
        CK(cudaMemset(h->metrics.p, 0, h->metrics.bytes));
    }
    CK(cudaMemcpy(h->first.p, first.data(), first.size() * sizeof(int), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(h->provider.p, prov.data(), prov.size() * sizeof(uint64_t), cudaMemcpyHostToDevice));
    h->cover_ready = true;
    return PM_OK;
}

void pm_destroy(pm_handle h) {
    if (!h) return;
    cudaDeviceSynchronize();
    delete h;
}

int pm_forward(pm_handle h, const void* frames, int n_frames, const int32_t* set_offsets,
               const int32_t* set_ids, float* scores_out, float* base_out, void* cuda_stream) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (n_frames < 0 || (n_frames > 0 && (!frames || !set_offsets || !scores_out))) { err = "NULL argument"; return PM_ERR_ARG; }
    if (n_frames == 0) return PM_OK;
    if (n_frames > h->cfg.max_frames) { err = "n_frames exceeds max_frames"; return PM_ERR_CAPACITY; }
    std::vector<int32_t> hoff, hids;
    const int32_t *o, *i;
    int rc = fetch_csr(set_offsets, set_ids, n_frames, st, hoff, hids, &o, &i, err);
    if (rc) return rc;
    Launch up; up.st = st;
    rc = h->router.build(n_frames, o, i, h->ranks, h->scales, true, up, err);
    if (rc) return rc;
    if (h->heads_dirty) {
        rc = h->cfg.dtype == 0 ? rebuild_heads<bf16>(h) : rebuild_heads<float>(h);
        if (rc) return rc;
    }
    pm_handle_s::GraphEntry key;
    key.key_ptr[0] = frames; key.key_ptr[1] = scores_out; key.key_ptr[2] = base_out;
    key.key_int[0] = n_frames; key.key_int[1] = 0 /* entry point */;
    // the kernels read the plan from device tables at fixed addresses; of its contents only the widest
    // set shapes the launch sequence, so a recorded sequence is replayed for any sets of the same width
    key.key_int[2] = h->router.dev.max_set;
    const bool small = latency_eligible(h, n_frames);
    key.key_int[3] = small ? 1 : 0;
    key.plan_version = 0; key.st = st;
    return run_graphed(h, key, [&]() {
        if (small) {
            const RouteDev& R = h->router.dev;
            return forward_latency(h, frames, n_frames, R.perm, R.slot_off, R.slot_ids, scores_out, base_out, st);
        }
        return h->cfg.dtype == 0 ? forward_t<bf16>(h, frames, n_frames, n_frames, 0, scores_out, base_out, st)
                                 : forward_t<float>(h, frames, n_frames, n_frames, 0, scores_out, base_out, st);
    });
}

int pm_forward_device_sets(pm_handle h, const void* frames, int n_frames, const int32_t* set_offsets,
                           const int32_t* set_ids, float* scores_out, float* base_out, void* cuda_stream) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (n_frames < 0 || (n_frames > 0 && (!frames || !set_offsets || !set_ids || !scores_out))) { err = "NULL argument"; return PM_ERR_ARG; }
    if (n_frames == 0) return PM_OK;
    if (n_frames > h->cfg.max_frames) { err = "n_frames exceeds max_frames"; return PM_ERR_CAPACITY; }
    if (h->heads_dirty) {
        int rc = h->cfg.dtype == 0 ? rebuild_heads<bf16>(h) : rebuild_heads<float>(h);
        if (rc) return rc;
    }
    if (n_frames > PM_DEVICE_PLAN_MAX_FRAMES) { err = "n_frames exceeds the device planner's limit"; return PM_ERR_CAPACITY; }
    // the plan tables on the device are about to be rewritten (by the kernels below or by their replay):
    // whatever host plan was uploaded before is gone
    h->router.invalidate();
    pm_handle_s::GraphEntry key;
    key.key_ptr[0] = frames; key.key_ptr[1] = scores_out; key.key_ptr[2] = base_out;
    key.key_ptr[3] = set_offsets; key.key_ptr[4] = set_ids;
    key.key_int[0] = n_frames; key.key_int[1] = 1 /* entry point */;
    const bool small = latency_eligible(h, n_frames);
    key.key_int[3] = small ? 1 : 0;
    // the launch sequence of a device plan depends on the frame count only, not on the lists
    key.plan_version = 0; key.st = st;
    return run_graphed(h, key, [&]() {
        // a handful of frames of a small model: the whole network in one launch, straight from the lists
        if (small) return forward_latency(h, frames, n_frames, nullptr, set_offsets, set_ids, scores_out, base_out, st);
        Launch L; L.st = st; L.launches = &h->launches; L.status = h->status.as<int>(); L.prof = &h->prof;
        int rc = h->router.build_on_device(L, n_frames, set_offsets, set_ids, h->meta, err);
        if (rc) return rc;
        return h->cfg.dtype == 0 ? forward_t<bf16>(h, frames, n_frames, n_frames, 0, scores_out, base_out, st)
                                 : forward_t<float>(h, frames, n_frames, n_frames, 0, scores_out, base_out, st);
    });
}

int pm_forward_branched(pm_handle h, const void* frames, int n_frames, const int32_t* set_offsets,
                        const int32_t* set_ids, int trunk_layers, float* scores_out, float* base_out,
                        void* cuda_stream) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    const pm_config& c = h->cfg;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (n_frames < 0 || (n_frames > 0 && (!frames || !set_offsets || !scores_out))) { err = "NULL argument"; return PM_ERR_ARG; }
    if (trunk_layers < 0 || trunk_layers > c.layers) { err = "trunk_layers out of range"; return PM_ERR_ARG; }
    if (n_frames == 0) return PM_OK;
    if (n_frames > c.max_frames) { err = "n_frames exceeds max_frames"; return PM_ERR_CAPACITY; }
    for (int i = 0; i < trunk_layers * 4; ++i)
        if (h->lin[i].n_adapted > 0) { err = "a registered adapter touches a block of the shared trunk"; return PM_ERR_STATE; }
    std::vector<int32_t> hoff, hids;
    const int32_t *o, *ids;
    int rc = fetch_csr(set_offsets, set_ids, n_frames, st, hoff, hids, &o, &ids, err);
    if (rc) return rc;
    if (o[0] != 0) { err = "set_offsets[0] must be 0"; return PM_ERR_ARG; }
    for (int f = 0; f < n_frames; ++f) {
        if (o[f + 1] < o[f]) { err = "set_offsets not monotone"; return PM_ERR_ARG; }
        if (o[f + 1] - o[f] > c.max_set) { err = "a frame has more adapters than max_set"; return PM_ERR_CAPACITY; }
    }
    if (o[n_frames] > 0 && !ids) { err = "NULL set_ids"; return PM_ERR_ARG; }
    // slots [0, F): the frames themselves, in caller order (the trunk's rows); they carry the base
    // branch when base scores are wanted, else the frame's lowest adapter.  Every other (frame,
    // adapter) branch gets a slot of its own behind them, grouped by adapter so that neighbouring
    // rows share LoRA slabs.
    std::vector<std::pair<int, int>> extra;          // (adapter, frame)
    std::vector<int32_t> boff(1, 0), bids;
    std::vector<int> fos, src;
    for (int f = 0; f < n_frames; ++f) {
        std::vector<int> s(ids + o[f], ids + o[f + 1]);
        std::sort(s.begin(), s.end());
        for (size_t i = 0; i < s.size(); ++i) {
            if (s[i] < 0 || s[i] >= c.max_adapters) { err = "adapter id out of range"; return PM_ERR_ARG; }
            if (i > 0 && s[i - 1] == s[i]) { err = "duplicate adapter id in a frame's set"; return PM_ERR_ARG; }
            if (h->ranks[s[i]] == 0) { err = "adapter id not registered"; return PM_ERR_STATE; }
        }
        size_t first_extra = 0;
        if (!base_out && !s.empty()) { bids.push_back(s[0]); first_extra = 1; }
        boff.push_back((int32_t)bids.size());
        fos.push_back(f); src.push_back(f);
        for (size_t i = first_extra; i < s.size(); ++i) extra.emplace_back(s[i], f);
    }
    std::sort(extra.begin(), extra.end());
    const long long n_slots = (long long)n_frames + (long long)extra.size();
    if (n_slots > c.max_frames) { err = "frames plus adapter branches exceed max_frames"; return PM_ERR_CAPACITY; }
    if (c.max_set < 1 && !extra.empty()) { err = "max_set is 0"; return PM_ERR_CAPACITY; }
    for (auto& e : extra) {
        bids.push_back(e.first); boff.push_back((int32_t)bids.size());
        fos.push_back(e.second); src.push_back(e.second);
    }
    if (bids.empty()) bids.push_back(0);
    Launch up; up.st = st;
    rc = h->router.build((int)n_slots, boff.data(), bids.data(), h->ranks, h->scales, false, up, err,
                         fos.data(), src.data());
    if (rc) return rc;
    if (h->heads_dirty) {
        rc = c.dtype == 0 ? rebuild_heads<bf16>(h) : rebuild_heads<float>(h);
        if (rc) return rc;
    }
    pm_handle_s::GraphEntry key;
    key.key_ptr[0] = frames; key.key_ptr[1] = scores_out; key.key_ptr[2] = base_out;
    key.key_int[0] = n_frames; key.key_int[1] = 2 /* entry point */; key.key_int[2] = trunk_layers;
    key.key_int[3] = (int)n_slots;
    key.plan_version = (unsigned long long)h->router.dev.max_set; key.st = st;
    return run_graphed(h, key, [&]() {
        return c.dtype == 0 ? forward_t<bf16>(h, frames, n_frames, (int)n_slots, trunk_layers, scores_out, base_out, st)
                            : forward_t<float>(h, frames, n_frames, (int)n_slots, trunk_layers, scores_out, base_out, st);
    });
}

int pm_select(pm_handle h, const float* scores, int n_frames, float score_thr, int context_copy,
              int has_prev, uint32_t* prev_labels, const int32_t* prev_offsets, const int32_t* prev_ids,
              int32_t* next_offsets, int32_t* next_ids, int ids_capacity, void* cuda_stream) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    if (!h->cover_ready) { err = "pm_set_cover has not been called since the last registration"; return PM_ERR_STATE; }
    if (n_frames < 0 || !scores || !next_offsets || (!next_ids && ids_capacity > 0) || ids_capacity < 0) { err = "NULL argument"; return PM_ERR_ARG; }
    if (has_prev && (!prev_labels || !prev_offsets || !prev_ids)) { err = "has_prev needs prev_labels, prev_offsets and prev_ids"; return PM_ERR_ARG; }
    if (n_frames > h->cfg.max_frames) { err = "n_frames exceeds max_frames"; return PM_ERR_CAPACITY; }
    Launch L; L.st = (cudaStream_t)cuda_stream; L.launches = &h->launches; L.status = h->status.as<int>();
    L.prof = &h->prof;
    CK(launch_select(L, scores, n_frames, h->cfg.n_classes, h->cfg.max_adapters, score_thr, context_copy,
                     has_prev, prev_labels, prev_offsets, prev_ids, h->first.as<int>(),
                     h->provider.as<uint64_t>(), h->mask_scratch.as<uint64_t>(), next_offsets, next_ids,
                     ids_capacity, h->metrics.as<unsigned long long>()));
    return PM_OK;
}

int pm_metrics_reset(pm_handle h, void* cuda_stream) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    if (!h->metrics.p) { err = "pm_set_cover has not been called"; return PM_ERR_STATE; }
    CK(cudaMemsetAsync(h->metrics.p, 0, h->metrics.bytes, (cudaStream_t)cuda_stream));
    return PM_OK;
}

int pm_metrics_read(pm_handle h, void* cuda_stream, long long* frames, long long* contexts, long long* switches) {
    if (!h) return PM_ERR_ARG;
    std::string& err = h->err;
    if (!h->metrics.p) { err = "pm_set_cover has not been called"; return PM_ERR_STATE; }
    unsigned long long v[3] = {0, 0, 0};
    CK(cudaStreamSynchronize((cudaStream_t)cuda_stream));
    CK(cudaMemcpy(v, h->metrics.p, sizeof(v), cudaMemcpyDeviceToHost));
    if (frames) *frames = (long long)v[0];
    if (contexts) *contexts = (long long)v[1];
    if (switches) *switches = (long long)v[2];
    return PM_OK;
}

static int read_status(DevBuf& status, cudaStream_t st, std::string& err) {
    int v = 0;
    CK(cudaStreamSynchronize(st));
    CK(cudaMemcpy(&v, status.p, sizeof(int), cudaMemcpyDeviceToHost));
    if (v != 0) {
        CK(cudaMemset(status.p, 0, sizeof(int)));
        err = v == PM_ERR_TIMEOUT ? "a bounded device-side wait expired" : "device status word set";
    }
    return v;
}

int pm_status(pm_handle h, void* cuda_stream) {
    if (!h) return PM_ERR_ARG;
    return read_status(h->status, (cudaStream_t)cuda_stream, h->err);
}

const char* pm_last_error(pm_handle h) { return h ? h->err.c_str() : "NULL handle"; }

int pm_profile_enable(pm_handle h, int on) {
    if (!h) return PM_ERR_ARG;
    h->prof.on = on != 0;
    if (on) h->prof.used = 0;
    return PM_OK;
}

int pm_profile_read(pm_handle h, void* cuda_stream, double* ms_by_class, long long* launches_by_class) {
    if (!h || !ms_by_class || !launches_by_class) return PM_ERR_ARG;
    std::string& err = h->err;
    CK(cudaStreamSynchronize((cudaStream_t)cuda_stream));
    for (int c = 0; c < KC_COUNT; ++c) { ms_by_class[c] = 0.0; launches_by_class[c] = 0; }
    for (size_t i = 0; i < h->prof.used; ++i) {
        float ms = 0.f;
        CK(cudaEventElapsedTime(&ms, h->prof.ev[2 * i], h->prof.ev[2 * i + 1]));
        ms_by_class[h->prof.cls[i]] += ms;
        launches_by_class[h->prof.cls[i]] += 1;
    }
    h->prof.used = 0;
    return PM_OK;
}
long long pm_launch_count(pm_handle h) { return h ? h->launches : 0; }

int pm_plan_stats(pm_handle h, long long* plans_built, double* host_ms) {
    if (!h) return PM_ERR_ARG;
    if (plans_built) *plans_built = h->router.plans_built;
    if (host_ms) *host_ms = h->router.plan_host_ms;
    return PM_OK;
}

int pm_set_small_batch_kernel(pm_handle h, int on) {
    if (!h) return PM_ERR_ARG;
    h->lat_on = on != 0;
    return PM_OK;
}

int pm_set_graphs(pm_handle h, int on) {
    if (!h) return PM_ERR_ARG;
    h->graphs_on = on != 0;
    if (!h->graphs_on) h->drop_graphs();
    return PM_OK;
}

// ---- single operators -------------------------------------------------------------------
int pm_linear_create(int k_in, int n_out, const float* w, const float* bias, int max_adapters,
                     int max_rank, int max_set, int max_frames, int tokens, int epilogue, int dtype,
                     pm_linear* out) {
    if (!out) return PM_ERR_ARG;
    *out = nullptr;
    if (!w || !bias || k_in <= 0 || n_out <= 0 || k_in % 64 || n_out % 64 || max_adapters < 0 ||
        max_adapters > 256 || max_rank < 0 || max_set < 0 || max_frames <= 0 || tokens <= 0 ||
        epilogue < 0 || epilogue > 2 || (dtype != 0 && dtype != 1))
        return PM_ERR_ARG;
    pm_linear_s* l = new (std::nothrow) pm_linear_s();
    if (!l) return PM_ERR_OOM;
    std::string& err = l->err;
    l->k_in = k_in; l->n_out = n_out; l->max_adapters = max_adapters; l->max_rank = max_rank;
    l->slabs_max = slabs_for(max_rank); l->max_set = max_set; l->max_frames = max_frames;
    l->tokens = tokens; l->epilogue = epilogue; l->dtype = dtype;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&l->n_sms, cudaDevAttrMultiProcessorCount, dev);
    auto fail = [&](int code) { fprintf(stderr, "pm_linear_create: %s\n", l->err.c_str()); delete l; return code; };
    int rc = l->lin.init(k_in, n_out, w, bias, max_adapters, l->slabs_max, dtype, err);
    if (rc) return fail(rc);
    rc = l->router.init(max_frames, max_set, std::max(1, max_adapters), l->slabs_max, tokens, err);
    if (rc) return fail(rc);
    l->ranks.assign(std::max(1, max_adapters), 0);
    l->scales.assign(std::max(1, max_adapters), 0.f);
    const size_t rows = (size_t)max_frames * tokens;
    cudaError_t e = l->scale_dev.alloc(l->scales.size() * sizeof(float));
    if (e == cudaSuccess) e = l->rank_dev.alloc(l->ranks.size() * sizeof(int));
    if (e == cudaSuccess) e = l->status.alloc(sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(l->status.p, 0, sizeof(int));
    if (e == cudaSuccess && dtype == 1)
        e = l->t32.alloc(rows * std::max(1, max_set) * std::max(1, l->slabs_max) * PM_SLAB * sizeof(float));
    size_t tb = 0;
    if (e == cudaSuccess && dtype == 0) {
        tb = (size_t)l->router.max_tiles * std::max(1, l->router.slab_cap) * PM_TILE_M * PM_SLAB;
        e = l->tbuf.alloc(tb * sizeof(bf16));
        if (e == cudaSuccess) e = cudaMemset(l->tbuf.p, 0, l->tbuf.bytes);
    }
    if (e != cudaSuccess) { err = cudaGetErrorString(e); return fail(e == cudaErrorMemoryAllocation ? PM_ERR_OOM : PM_ERR_CUDA); }
    if (dtype == 0 && !tm_encode_2d(&l->tm_t, l->tbuf.p, PM_SLAB, tb / PM_SLAB, PM_SLAB * 2, PM_SLAB, PM_TILE_M, 32)) {
        err = "cuTensorMapEncodeTiled failed (slab buffer)"; return fail(PM_ERR_CUDA);
    }
    rc = sync_meta(l->scale_dev, l->rank_dev, l->scales, l->ranks, err);
    if (rc) return fail(rc);
    l->meta.scale = l->scale_dev.as<float>(); l->meta.rank = l->rank_dev.as<int>();
    if (cudaDeviceSynchronize() != cudaSuccess) { err = "device synchronize failed"; return fail(PM_ERR_CUDA); }
    *out = l;
    return PM_OK;
}

int pm_linear_register(pm_linear l, int id, int rank, float scale, const float* A, const float* B) {
    if (!l) return PM_ERR_ARG;
    std::string& err = l->err;
    if (id < 0 || id >= l->max_adapters || !A || !B) { err = "bad adapter id or NULL matrices"; return PM_ERR_ARG; }
    if (rank <= 0 || rank > l->max_rank) { err = "adapter rank exceeds max_rank"; return PM_ERR_CAPACITY; }
    int rc = l->lin.set_adapter(id, rank, A, B, err);
    if (rc) return rc;
    l->ranks[id] = rank; l->scales[id] = scale;
    l->router.invalidate();
    return sync_meta(l->scale_dev, l->rank_dev, l->scales, l->ranks, err);
}

int pm_linear_forward(pm_linear l, const void* x, int n_frames, const int32_t* set_offsets,
                      const int32_t* set_ids, const void* residual, void* y, void* cuda_stream) {
    if (!l) return PM_ERR_ARG;
    std::string& err = l->err;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (n_frames < 0 || (n_frames > 0 && (!x || !y || !set_offsets))) { err = "NULL argument"; return PM_ERR_ARG; }
    if (l->epilogue == EPI_RESIDUAL && n_frames > 0 && !residual) { err = "epilogue 2 needs a residual"; return PM_ERR_ARG; }
    if (n_frames == 0) return PM_OK;
    if (l->dtype == 0 && ((uintptr_t)x | (uintptr_t)y | (l->epilogue == EPI_RESIDUAL ? (uintptr_t)residual : 0)) & 15) {
        err = "x, y and a residual that is added must be 16-byte aligned"; return PM_ERR_CUDA;
    }
    Launch L; L.st = st; L.launches = &l->launches; L.status = l->status.as<int>();
    int rc = l->router.build(n_frames, set_offsets, set_ids, l->ranks, l->scales, false, L, err);
    if (rc) return rc;
    const RouteDev& R = l->router.dev;
    const int rows = n_frames * l->tokens;
    PatchEpi none;
    if (l->dtype == 0 && small_linear_fits(l->lin.dev, &R, rows, l->epilogue, l->n_sms)) {
        ActMaps sx;
        if (!act_encode(&sx, x, l->k_in, rows)) { err = "cuTensorMapEncodeTiled failed (x)"; return PM_ERR_CUDA; }
        CK(launch_small_linear(L, l->lin.dev, &R, sx, rows, l->epilogue, (const bf16*)residual, none, (bf16*)y, l->n_sms, 0.f));
    } else if (l->dtype == 0) {
        CUtensorMap tm_x;
        if (!tm_encode_2d(&tm_x, x, l->k_in, rows, (uint64_t)l->k_in * 2, 64, PM_TILE_M, 128)) {
            err = "cuTensorMapEncodeTiled failed (x); x must be 16-byte aligned"; return PM_ERR_CUDA;
        }
        CUtensorMap tm_y;
        if (!tm_encode_2d(&tm_y, y, l->n_out, rows, (uint64_t)l->n_out * 2, 32, 32, 64)) {
            err = "cuTensorMapEncodeTiled failed (y); y must be 16-byte aligned"; return PM_ERR_CUDA;
        }
        const bool lora = R.max_set > 0 && l->lin.dev.lora.At != nullptr;
        if (lora) {
            ActMaps sx;
            if (!act_encode(&sx, x, l->k_in, rows)) { err = "cuTensorMapEncodeTiled failed (x)"; return PM_ERR_CUDA; }
            CK(launch_shrink(L, l->lin.dev, R, sx, rows, l->tbuf.as<bf16>(), l->n_sms, nullptr, 0.f));
        }
        CK(launch_lora_gemm(L, l->lin.dev, lora ? &R : nullptr, tm_x, &l->tm_t, &tm_y, rows, l->epilogue,
                            (const bf16*)residual, none, (bf16*)y, l->n_sms, nullptr, lora));
    } else {
        CK(launch_naive_linear<float>(L, l->lin.dev, R, l->meta, l->slabs_max, (const float*)x, rows, l->tokens,
                                      l->t32.as<float>(), l->epilogue, (const float*)residual, none, (float*)y));
    }
    return PM_OK;
}

int pm_linear_status(pm_linear l, void* cuda_stream) {
    if (!l) return PM_ERR_ARG;
    return read_status(l->status, (cudaStream_t)cuda_stream, l->err);
}
const char* pm_linear_last_error(pm_linear l) { return l ? l->err.c_str() : "NULL handle"; }
void pm_linear_destroy(pm_linear l) {
    if (!l) return;
    cudaDeviceSynchronize();
    delete l;
}

int pm_linear_kernel(int k_in, int n_out, int rows, int epilogue, int adapters, int n_sms, int32_t* form) {
    if (!form || k_in <= 0 || n_out <= 0 || k_in % 64 || n_out % 64 || rows <= 0 || epilogue < 0 || epilogue > 3 || n_sms < 1) return PM_ERR_ARG;
    LinearForm f;
    if (!small_linear_form(k_in, n_out, adapters != 0, rows, epilogue, n_sms, &f)) f = gemm_form(k_in, n_out, adapters != 0, rows, epilogue, n_sms);
    form[0] = f.kernel; form[1] = f.width; form[2] = f.split; form[3] = f.threads;
    return PM_OK;
}

int pm_layernorm(const void* x, const float* gamma, const float* beta, void* y, int rows, int d,
                 float eps, int dtype, void* cuda_stream) {
    if (!x || !gamma || !beta || !y || rows < 0 || d <= 0 || d % 8 || d > 1024 || (dtype != 0 && dtype != 1))
        return PM_ERR_ARG;
    Launch L; L.st = (cudaStream_t)cuda_stream;
    cudaError_t e = dtype == 0 ? launch_layernorm<bf16>(L, (const bf16*)x, gamma, beta, (bf16*)y, rows, d, eps)
                               : launch_layernorm<float>(L, (const float*)x, gamma, beta, (float*)y, rows, d, eps);
    return e == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}

int pm_attention(const void* qkv, void* out, int n_frames, int tokens, int heads, int dtype,
                 void* cuda_stream) {
    if (!qkv || !out || n_frames < 0 || tokens <= 0 || heads <= 0 || (dtype != 0 && dtype != 1))
        return PM_ERR_ARG;
    Launch L; L.st = (cudaStream_t)cuda_stream;
    if (n_frames == 0) return PM_OK;
    cudaError_t e;
    if (dtype == 1) {
        e = launch_attention_simple<float>(L, (const float*)qkv, (float*)out, n_frames, tokens, heads);
    } else if (attention_tc_supported(tokens)) {
        // the operator has no handle, hence no status word of its own: a bounded wait that expires is
        // reported through the return code of a later call on the same device
        // (one word per device, allocated on first use)
        static std::atomic<int*> status_words[64];
        int dev = 0, n_sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 ||
            cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return PM_ERR_CUDA;
        int* status_word = status_words[dev].load(std::memory_order_acquire);
        if (!status_word) {
            if (cudaMalloc(&status_word, sizeof(int)) != cudaSuccess) return PM_ERR_OOM;
            if (cudaMemset(status_word, 0, sizeof(int)) != cudaSuccess) return PM_ERR_CUDA;
            int* expected = nullptr;
            if (!status_words[dev].compare_exchange_strong(expected, status_word, std::memory_order_acq_rel)) {
                cudaFree(status_word);                    // another thread got there first
                status_word = expected;
            }
        }
        L.status = status_word;
        CUtensorMap tm_q, tm_kv;
        if (!attention_encode_maps((const bf16*)qkv, n_frames, tokens, heads, &tm_q, &tm_kv)) return PM_ERR_CUDA;
        e = launch_attention_tc(L, tm_q, tm_kv, (const bf16*)qkv, (bf16*)out, n_frames, tokens, heads, n_sms);
    } else {
        e = launch_attention_mma(L, (const bf16*)qkv, (bf16*)out, n_frames, tokens, heads);
    }
    return e == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}

}  // extern "C"
