// The fused base + multi-LoRA linear (Sec. 3.1: y = xW + b + sum_a s_a (x A_a) B_a) for few rows: one 128 x BN
// output tile per CTA (or per cluster of S CTAs that share K), everything of the linear in one kernel.
//
// What bounds it is neither bandwidth nor the tensor cores but the chain launch -> first bytes -> K loop -> t ->
// expand -> epilogue, so every link is shortened:
//   - the tile is the narrowest that fits the SMs in one wave: many CTAs, each with little to fetch;
//   - the shrink rides on the K loop's own MMAs (a stage's slab rows lie behind its W rows, the accumulators side by side in
//     tensor memory: one operand of BN + 16 columns per slab) and the epilogue warps take the LayerNorm statistics from the same stages: one pass over x;
//   - t stays in tensor memory: rounded in place of its accumulator columns, it is the expand MMAs' A operand there, and
//     the shared memory is the ring's;
//   - the copies are issued by two threads (x and W; adapter slabs), since issuing is a serial cost;
//   - weights, adapter slabs, plan entries, bias and LayerNorm vectors do not depend on the kernel before: they are
//     requested before the kernel waits for it (programmatic dependent launch);
//   - split K (long K, narrow output): each CTA of the cluster makes a partial tile, its own partial t and
//     expand included (the expand is linear in t); the partials are exchanged through distributed shared memory, as
//     asynchronous stores that count themselves on the receiver's barrier, and every CTA sums and stores BN / S columns.  A partial t enters the expand as two bf16 parts (16 significant
//     bits, two MMAs per slab): rounded to one, shares that cancel would leave their rounding in the sum.
// One 197-token frame of width 768, rank-16 adapters, replayed back to back: qkv 5.0 us, proj 4.9, fc1 5.6, fc2 6.9; four frames
// 7.4, 5.7, 9.5 and 11.6; eight frames 12.3, 9.4, 14.4 and 16.3.  (Issued behind a lane test, the shrink in MMAs of its own and partial sums
// released by each warp: 7.0, 6.9, 7.3, 9.7; 9.7, 7.4, 11.2, 16.0; 13.1, 10.5, 17.4, 19.0.)
// Warp roles: 0 = x / W copies, 1 = tensor memory + MMA, 2 = adapter copies, 3 = slab list, 4..11 = statistics, t, epilogue.
#include "common.cuh"
#include "f32x2.cuh"
#include "tcgen05_ptx.cuh"

#define BUMP(L) do { if ((L).launches) ++*(L).launches; } while (0)

namespace {

constexpr int BM = PM_TILE_M;
constexpr int BK = 64;
constexpr int EW = 8;                                  // epilogue warps: two per tensor-memory lane quarter
constexpr int FIRST_EW = 4;
constexpr int THREADS = 32 * (FIRST_EW + EW);
constexpr int MAX_STAGES = 8;
constexpr int GROUP = 8;                               // slabs of one pass over x: 128 accumulator columns
constexpr int LIST = 64;                               // slabs a tile may use
constexpr int A_BLOCK = BM * BK * 2;                   // 16 KB: one K block of the tile's rows

constexpr int WIDTHS[PM_SMALL_WIDTHS] = {64, 128, 192, 256};
__host__ __device__ constexpr int kps_of(int bn) { return bn == 64 ? 2 : 1; }       // K blocks per stage: two where the MMAs of one are shorter than its issue

// tail of the shared memory: what the list warp prepares, half-row statistics, vectors, barriers
struct Tail {
    uint4 mask[LIST];
    float c[LIST][2 * PM_SLAB];                        // LayerNorm folded in: c1 then c2 of the slab
    float scale[LIST];
    int slab[LIST];
    float2 half_stats[2][BM];                          // mean, sum of squared deviations of half a row
    float bias[256], ln_g[256];
    uint64_t bars[2 * MAX_STAGES + 5];
    uint32_t tmem_slot;
    int abort_flag, n_active;
};

struct SmallArgs {
    int rows, k_in, n_out, n_tiles;
    const float* bias;
    const bf16* residual;
    bf16* y;
    PatchEpi pe;
    const int* tile_nslabs;                            // null = no LoRA
    const int* tile_slab;
    const float* tile_scale;
    const uint32_t* tile_mask;
    int slab_cap;
    const float *ln_g, *ln_c1, *ln_c2;
    float ln_eps;
    int* status;
    int ring_bytes;
};

template <int BN, int S>
__host__ __device__ constexpr int recv_bytes() { return S > 1 ? (S - 1) * BM * (BN / S) * 4 : 0; }

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* v) {
    if constexpr (N == 8) tmem_ld8(taddr, v);
    else if constexpr (N == 16) tmem_ld16(taddr, v);
    else tmem_ld32(taddr, v);
}

// N accumulator columns of one row, from column c of the tile / n0 of the output on -> bias / LayerNorm / GELU /
// residual (res, already fetched) / patch placement -> global memory
template <int N, int EPI, bool LNF>
__device__ __forceinline__ void finish_columns(const SmallArgs& args, const Tail& tail, const uint32_t* v, const uint4* res,
                                               int row, int c, int n0, float2 st) {
    if (row >= args.rows) return;
    size_t orow = (size_t)row;
    uint64_t f[N / 2];
    const uint64_t rstd2 = pk2(st.y, st.y), nmean2 = pk2(-st.x, -st.x);
#pragma unroll
    for (int j = 0; j < N; j += 4) {
        const float4 b4 = *reinterpret_cast<const float4*>(tail.bias + c + j);
        uint64_t a0 = pk2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
        uint64_t a1 = pk2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        if constexpr (LNF) {
            const float4 g4 = *reinterpret_cast<const float4*>(tail.ln_g + c + j);
            a0 = fma2(rstd2, fma2(nmean2, pk2(g4.x, g4.y), a0), pk2(b4.x, b4.y));
            a1 = fma2(rstd2, fma2(nmean2, pk2(g4.z, g4.w), a1), pk2(b4.z, b4.w));
        } else {
            a0 = add2(a0, pk2(b4.x, b4.y));
            a1 = add2(a1, pk2(b4.z, b4.w));
        }
        if constexpr (EPI == EPI_GELU) { a0 = gelu_erf2(a0); a1 = gelu_erf2(a1); }
        f[j >> 1] = a0;
        f[(j >> 1) + 1] = a1;
    }
    if constexpr (EPI == EPI_RESIDUAL) {
#pragma unroll
        for (int q = 0; q < N / 8; ++q) {
            const uint32_t w[4] = {res[q].x, res[q].y, res[q].z, res[q].w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                f[q * 4 + e] = add2(f[q * 4 + e], pk2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xFFFF0000u)));
        }
    } else if constexpr (EPI == EPI_PATCH) {
        const int p = row % args.pe.g2;
        orow = (size_t)(row / args.pe.g2) * args.pe.tokens + 1 + p;
        const float* pos = args.pe.pos + (size_t)(1 + p) * args.n_out + n0;
#pragma unroll
        for (int j = 0; j < N; j += 4) {
            const float4 p4 = __ldg(reinterpret_cast<const float4*>(pos + j));
            f[j >> 1] = add2(f[j >> 1], pk2(p4.x, p4.y));
            f[(j >> 1) + 1] = add2(f[(j >> 1) + 1], pk2(p4.z, p4.w));
        }
    }
    uint4* o4 = reinterpret_cast<uint4*>(args.y + orow * args.n_out + n0);
#pragma unroll
    for (int q = 0; q < N / 8; ++q) {
        uint4 o;
        float lo, hi;
        upk2(f[q * 4 + 0], lo, hi); o.x = pack_bf16(lo, hi);
        upk2(f[q * 4 + 1], lo, hi); o.y = pack_bf16(lo, hi);
        upk2(f[q * 4 + 2], lo, hi); o.z = pack_bf16(lo, hi);
        upk2(f[q * 4 + 3], lo, hi); o.w = pack_bf16(lo, hi);
        o4[q] = o;
    }
}

template <int N, int EPI>
__device__ __forceinline__ void fetch_residual(const SmallArgs& args, int row, int n0, uint4* res) {
    if constexpr (EPI == EPI_RESIDUAL) {
        const uint4* r4 = reinterpret_cast<const uint4*>(args.residual + (size_t)row * args.n_out + n0);
#pragma unroll
        for (int q = 0; q < N / 8; ++q) res[q] = row < args.rows ? r4[q] : make_uint4(0, 0, 0, 0);
    }
}

template <int BN, int EPI, bool LNF, int S>
__global__ void __launch_bounds__(THREADS, 1)
small_linear_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                    const __grid_constant__ CUtensorMap tm_bt, const __grid_constant__ CUtensorMap tm_at,
                    const SmallArgs args) {
    constexpr int KPS = kps_of(BN);
    constexpr int X_BYTES = KPS * A_BLOCK;
    constexpr int B_BLOCK = BN * BK * 2, W_BYTES = KPS * B_BLOCK;
    constexpr int A_SLAB = KPS * PM_SLAB * BK * 2;     // a slab's rows of a stage
    constexpr int B_SLAB = BN * PM_SLAB * 2;
    constexpr int TMEM_COLS = BN + GROUP * PM_SLAB <= 256 ? 256 : 512;
    constexpr int EMPTY_COUNT = LNF ? 1 + EW : 1;      // MMA commit, and the statistics' readers
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t base = smem_u32(smem);
    const uint32_t recv_s = base + (uint32_t)args.ring_bytes;
    Tail& tail = *reinterpret_cast<Tail*>(smem + args.ring_bytes + recv_bytes<BN, S>());
    const uint32_t bars = smem_u32(tail.bars);
    auto full_bar = [&](int s) { return bars + 8u * s; };              // both copying threads' bytes of a stage
    auto empty_bar = [&](int s) { return bars + 8u * (MAX_STAGES + s); };
    const uint32_t tacc_bar = bars + 8u * (2 * MAX_STAGES);            // shrink accumulator complete
    const uint32_t tready_bar = tacc_bar + 8u;                         // t written over its accumulator columns
    const uint32_t tfull_bar = tacc_bar + 16u;                         // tile complete
    const uint32_t stats_bar = tacc_bar + 24u;                         // half-row statistics exchanged
    const uint32_t recv_bar = tacc_bar + 32u;                          // the other CTAs' partial sums are here
    volatile int* abort_flag = &tail.abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ks = S > 1 ? (int)cluster_ctarank() : 0;
    const int tile = blockIdx.x / S;
    const int m = tile / args.n_tiles, n = tile - m * args.n_tiles;
    // this CTA's K blocks, whole stages; an odd last stage's second block lies past K and reads as zero
    const int all_kb = args.k_in / BK, all_st = (all_kb + KPS - 1) / KPS;
    const int st0 = all_st * ks / S, num_st = all_st * (ks + 1) / S - st0;
    const int kb0 = st0 * KPS, num_kb = min(all_kb, kb0 + num_st * KPS) - kb0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), EMPTY_COUNT); }
        mbar_init(tacc_bar, 1); mbar_init(tready_bar, EW); mbar_init(tfull_bar, 1); mbar_init(stats_bar, EW + 1);
        mbar_init(recv_bar, 1);
        tail.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (S > 1) mbar_expect_tx(recv_bar, (uint32_t)recv_bytes<BN, S>());
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tail.tmem_slot), TMEM_COLS);
        tmem_relinquish();
    } else if (warp == 3) {
        // the slabs that some row of THIS 128-row tile uses (the plan lists those of the 256-row pair)
        int na = 0;
        const int ns = args.tile_nslabs ? __ldg(args.tile_nslabs + m) : 0;
        for (int i0 = 0; i0 < ns; i0 += 32) {
            const size_t at = (size_t)m * args.slab_cap + i0 + lane;
            uint4 mk = make_uint4(0, 0, 0, 0);
            int slab = 0;
            float sc = 0.f;
            if (i0 + lane < ns) {
                mk = __ldg(reinterpret_cast<const uint4*>(args.tile_mask) + at);
                slab = __ldg(args.tile_slab + at);
                sc = __ldg(args.tile_scale + at);
            }
            const bool on = (mk.x | mk.y | mk.z | mk.w) != 0u;
            const uint32_t b = __ballot_sync(0xFFFFFFFFu, on);
            const int to = na + __popc(b & ((1u << lane) - 1u));
            if (on && to < LIST) { tail.mask[to] = mk; tail.slab[to] = slab; tail.scale[to] = sc; }
            na = min(LIST, na + __popc(b));
        }
        if (lane == 0) tail.n_active = na;
    } else if (warp >= FIRST_EW) {
        for (int i = threadIdx.x - 32 * FIRST_EW; i < BN; i += 32 * EW) {
            tail.bias[i] = __ldg(args.bias + n * BN + i);
            if (LNF) tail.ln_g[i] = __ldg(args.ln_g + n * BN + i);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (S > 1) cluster_sync_all();            // the peers' barriers are initialised
    dep_release();
    const uint32_t tmem_base = tail.tmem_slot;
    const uint32_t t_tmem = tmem_base + BN;
    const int na = tail.n_active;
    const int n_groups = na == 0 ? 1 : (na + GROUP - 1) / GROUP;
    const int per_group = min(na, GROUP);
    const int stage_bytes = X_BYTES + W_BYTES + per_group * A_SLAB;
    const int STG = min(MAX_STAGES, args.ring_bytes / stage_bytes);
    const bool usable = (base & 1023u) == 0;       // swizzled operands need a 1024-byte aligned window
    if (!usable && threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);

    if (!usable) {
        // fall through to the teardown
    } else if (warp == 0) {
        if (elect_one()) {
            // -------------------------------------------------------------- x and W copies
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            const int pre = min(STG, num_st);
            for (int st = 0; st < pre; ++st) {
                mbar_expect_tx(full_bar(st), X_BYTES + W_BYTES);
                tma_load_4d(base + st * stage_bytes + X_BYTES, &tm_w, 0, 0, kb0 + st * KPS, n * (BN / 8), full_bar(st));
                if (na == 0) mbar_arrive(full_bar(st));                  // nobody brings slabs
            }
            dep_wait();
            for (int st = 0; st < pre; ++st)
                tma_load_3d(base + st * stage_bytes, &tm_x, 0, m * BM, kb0 + st * KPS, full_bar(st));
            for (int g = 0; g < n_groups && ok; ++g) {
                for (int st = 0; st < num_st; ++st) {
                    if (g > 0 || st >= pre) {
                        ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                        if (!ok) break;
                        const uint32_t sa = base + stage * stage_bytes;
                        if (g == 0) {
                            mbar_expect_tx(full_bar(stage), X_BYTES + W_BYTES);
                            tma_load_3d(sa, &tm_x, 0, m * BM, kb0 + st * KPS, full_bar(stage));
                            tma_load_4d(sa + X_BYTES, &tm_w, 0, 0, kb0 + st * KPS, n * (BN / 8), full_bar(stage));
                            if (na == 0) mbar_arrive(full_bar(stage));
                        } else {                                          // further slabs: another pass over x
                            if (LNF) mbar_arrive_n(empty_bar(stage), EW);
                            mbar_expect_tx(full_bar(stage), X_BYTES);
                            tma_load_3d(sa, &tm_x, 0, m * BM, kb0 + st * KPS, full_bar(stage));
                        }
                    }
                    if (++stage == STG) { stage = 0; phase ^= 1u; }
                }
                // The group's B slabs are the other thread's, but this one waits for their stage too: a parity wait tells
                // only neighbouring uses apart, and in a ring of one stage the next group's wait would be satisfied
                // by the use before the B slabs.
                if (ok && g + 1 < n_groups) ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                if (++stage == STG) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 2) {
        if (na > 0 && elect_one()) {
            // -------------------------------------------------------------- adapter copies
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int g = 0; g < n_groups && ok; ++g) {
                const int g0 = g * GROUP, cnt = min(GROUP, na - g0);
                for (int st = 0; st < num_st; ++st) {
                    ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    mbar_expect_tx(full_bar(stage), cnt * A_SLAB);
                    const uint32_t sa = base + stage * stage_bytes + X_BYTES + W_BYTES;
#pragma unroll 1
                    for (int i = 0; i < cnt; ++i)
                        tma_load_4d(sa + i * A_SLAB, &tm_at, 0, 0, kb0 + st * KPS, tail.slab[g0 + i] * (PM_SLAB / 8), full_bar(stage));
                    if (++stage == STG) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);      // the group's B slabs
                if (!ok) break;
                if (LNF) mbar_arrive_n(empty_bar(stage), EW);
                mbar_expect_tx(full_bar(stage), cnt * B_SLAB);
                mbar_arrive(full_bar(stage));
#pragma unroll 1
                for (int i = 0; i < cnt; ++i)
                    tma_load_2d(base + stage * stage_bytes + i * B_SLAB, &tm_bt, 0, tail.slab[g0 + i] * args.n_out + n * BN, full_bar(stage));
                if (++stage == STG) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // -------------------------------------------------------------- MMA issuer
            const uint32_t idesc = instr_desc(BN);
            const uint64_t da0 = smem_desc(base, 128), db0 = smem_desc_groups(base + X_BYTES, KPS * 1024);
            const uint64_t ds0 = smem_desc_groups(base + X_BYTES + W_BYTES, KPS * 1024);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int g = 0; g < n_groups && ok; ++g) {
                const int cnt = min(GROUP, na - g * GROUP);
                const uint32_t idesc_t = instr_desc(max(cnt, 1) * PM_SLAB);
                // W tile and slabs are adjacent in a stage and their accumulators in tensor memory: one MMA makes both where
                // N allows it.  An MMA of 128 rows takes at least 49 cycles however narrow: 64 and 48 columns apart 845
                // cycles per stage, 112 together 555; 768 -> 2304 on one frame 6.1 -> 4.9 us.
                const bool joint = BN + max(cnt, 0) * PM_SLAB <= 256;
                const uint32_t idesc_j = instr_desc(joint ? BN + max(cnt, 0) * PM_SLAB : BN);
                for (int kb = 0; kb < num_kb; kb += KPS) {
                    ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t so = (uint64_t)((stage * stage_bytes) >> 4);
#pragma unroll
                    for (int j = 0; j < KPS; ++j) {
                        if (j > 0 && kb + j >= num_kb) break;
                        const uint64_t da = da0 + so + (j * A_BLOCK >> 4), db = db0 + so + (j * 1024 >> 4);
                        const uint64_t ds = ds0 + so + (j * 1024 >> 4);
                        if (g == 0) {
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k) umma_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc_j, (kb | j | k) != 0);
                        }
                        if (cnt > 0 && (g > 0 || !joint)) {
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k) umma_bf16(t_tmem, da + 2 * k, ds + 2 * k, idesc_t, (kb | j | k) != 0);
                        }
                    }
                    umma_commit(empty_bar(stage));
                    if (++stage == STG) { stage = 0; phase ^= 1u; }
                }
                if (!ok || cnt <= 0) break;
                umma_commit(tacc_bar);
                ok = mbar_wait(tready_bar, g & 1, abort_flag, args.status);
                if (ok) ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sb = base + stage * stage_bytes;
                for (int i = 0; i < cnt; ++i) {
                    umma_bf16_ts(tmem_base, t_tmem + i * PM_SLAB, smem_desc(sb + i * B_SLAB, 32), idesc, 1u);
                    if constexpr (S > 1) umma_bf16_ts(tmem_base, t_tmem + i * PM_SLAB + PM_SLAB / 2, smem_desc(sb + i * B_SLAB, 32), idesc, 1u);
                }
                umma_commit(empty_bar(stage));
                if (++stage == STG) { stage = 0; phase ^= 1u; }
            }
            if (ok) umma_commit(tfull_bar);
        }
    } else if (warp == 3) {
        if (LNF) {
            // the slabs' LayerNorm terms, for the warps that turn the accumulator into t
            for (int i = lane; i < na * 2 * PM_SLAB; i += 32) {
                const int s = i / (2 * PM_SLAB), j = i % (2 * PM_SLAB);
                tail.c[s][j] = __ldg((j < PM_SLAB ? args.ln_c1 : args.ln_c2) + (size_t)tail.slab[s] * PM_SLAB + (j & (PM_SLAB - 1)));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(stats_bar);
        }
    } else {
        // ------------------------------------------------------------------ statistics, t, epilogue
        const int quarter = warp & 3;                 // TMEM lanes 32*quarter .. +31
        const int half = (warp - FIRST_EW) >> 2;
        const int r = quarter * 32 + lane;
        const int row = m * BM + r;
        constexpr int CPW = BN / 64;                  // 32-column chunks of this warp (S == 1)
        constexpr int CS = BN / S, HC = CS / 2;       // S > 1: columns a CTA finishes, and a thread of it
        constexpr bool RES_AHEAD = S > 1 || BN <= 128;
        bool ok = true;
        float2 st = make_float2(0.f, 1.f);
        dep_wait();
        // residual rows are fetched now where they fit the registers, behind the K loop
        uint4 res[RES_AHEAD ? (S > 1 ? HC / 8 : CPW * 4) : 4];
        if constexpr (RES_AHEAD && EPI == EPI_RESIDUAL) {
            if constexpr (S > 1) fetch_residual<HC, EPI>(args, row, n * BN + ks * CS + half * HC, res);
            else
#pragma unroll
                for (int c = 0; c < CPW; ++c) fetch_residual<32, EPI>(args, row, n * BN + half * (BN / 2) + c * 32, res + c * 4);
        }
        if constexpr (LNF) {
            // follow the ring: this thread sums its half of its row of each x block, relative to its first element
            // (which keeps the sum of squares well conditioned)
            float pivot = 0.f;
            uint64_t np = 0, s1 = pk2(0.f, 0.f), s2 = s1;
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < num_kb && ok; kb += KPS) {
                ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
#pragma unroll
                for (int j = 0; j < KPS; ++j) {
                    if (j > 0 && kb + j >= num_kb) break;
                    const uint32_t row_addr = base + stage * stage_bytes + j * A_BLOCK + r * 128;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint4 q;
                        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                                     : "r"(row_addr + (((half * 4 + c) ^ (r & 7)) << 4)));
                        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
                        if (kb == 0 && j == 0 && c == 0) {
                            pivot = __uint_as_float(w[0] << 16);
                            np = pk2(-pivot, -pivot);
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint64_t a = add2(pk2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xFFFF0000u)), np);
                            s1 = add2(s1, a);
                            s2 = fma2(a, a, s2);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty_bar(stage));
                if (++stage == STG) { stage = 0; phase ^= 1u; }
            }
            if (ok) {
                // the two halves of a row (equal counts) are merged through shared memory
                float a0, a1, b0, b1;
                upk2(s1, a0, a1);
                upk2(s2, b0, b1);
                const float inv_n = 2.f / (float)args.k_in;
                const float m1 = (a0 + a1) * inv_n;
                tail.half_stats[half][r] = make_float2(pivot + m1, fmaxf((b0 + b1) - (a0 + a1) * m1, 0.f));
                __syncwarp();
                if (lane == 0) mbar_arrive(stats_bar);
                ok = mbar_wait(stats_bar, 0, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                const float2 h0 = tail.half_stats[0][r], h1 = tail.half_stats[1][r];
                const float dm = h1.x - h0.x;
                const float var = (h0.y + h1.y) / (float)args.k_in + 0.25f * dm * dm;
                st = make_float2(0.5f * (h0.x + h1.x), rsqrtf(var + args.ln_eps));
            }
        }
        const float inv_rstd = 1.f / st.y;
        const uint32_t t_lane = t_tmem + ((uint32_t)(quarter * 32) << 16);
        for (int g = 0; g < n_groups && na > 0 && ok; ++g) {
            ok = mbar_wait(tacc_bar, g & 1, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            const int g0 = g * GROUP, cnt = min(GROUP, na - g0);
            for (int i = half; i < cnt; i += 2) {               // the two warps of a lane quarter take slabs in turn
                uint32_t v[16];
                tmem_ld16(t_lane + (uint32_t)(i * PM_SLAB), v);
                const uint32_t mk = reinterpret_cast<const uint32_t*>(&tail.mask[g0 + i])[quarter];
                const float sc = (mk >> lane) & 1u ? tail.scale[g0 + i] : 0.f;
                tmem_ld_wait();
                if constexpr (LNF) {
                    // divided by rstd: the epilogue applies rstd to the whole accumulator
                    const float* c = tail.c[g0 + i];
#pragma unroll
                    for (int j = 0; j < PM_SLAB; ++j)
                        v[j] = __float_as_uint(fmaf(-st.x, c[j], __uint_as_float(v[j])) + inv_rstd * c[PM_SLAB + j]);
                }
                // over the slab's own accumulator columns: a row's 16 values as 8 columns of bf16 pairs, then (K split) what the
                // rounding leaves of them as 8 more
                uint32_t o[PM_SLAB];
#pragma unroll
                for (int j = 0; j < PM_SLAB; j += 2) {
                    const float t0 = __uint_as_float(v[j]) * sc, t1 = __uint_as_float(v[j + 1]) * sc;
                    const uint32_t hi = o[j >> 1] = pack_bf16(t0, t1);
                    o[(PM_SLAB + j) >> 1] = pack_bf16(t0 - __uint_as_float(hi << 16), t1 - __uint_as_float(hi & 0xFFFF0000u));
                }
                if constexpr (S > 1) tmem_st16(t_lane + (uint32_t)(i * PM_SLAB), o);
                else tmem_st8(t_lane + (uint32_t)(i * PM_SLAB), o);
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tready_bar);
        }
        if (ok) {
            ok = mbar_wait(tfull_bar, 0, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
        }
        if (ok) {
            tc_fence_after();
            const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
            if constexpr (S == 1) {
#pragma unroll
                for (int c = 0; c < CPW; ++c) {
                    const int col = half * (BN / 2) + c * 32;
                    uint32_t v[32];
                    tmem_ld32(t_row + (uint32_t)col, v);
                    if constexpr (!RES_AHEAD) fetch_residual<32, EPI>(args, row, n * BN + col, res);
                    tmem_ld_wait();
                    finish_columns<32, EPI, LNF>(args, tail, v, res + (RES_AHEAD ? c * 4 : 0), row, col, n * BN + col, st);
                }
            } else {
                // recv[src][16-byte column group][row]: src = the sender's place among the other CTAs
                constexpr int CW = HC % 32 == 0 ? 32 : HC % 16 == 0 ? 16 : 8;      // columns at a time
#pragma unroll
                for (int c = 0; c < HC; c += CW) {
                    uint32_t v[S - 1][CW];
#pragma unroll
                    for (int jj = 1; jj < S; ++jj) tmem_ld<CW>(t_row + (uint32_t)((ks + jj) % S * CS + half * HC + c), v[jj - 1]);
                    tmem_ld_wait();
#pragma unroll
                    for (int jj = 1; jj < S; ++jj) {
                        const int j = (ks + jj) % S, src = ks < j ? ks : ks - 1;
                        const uint32_t dst = mapa_cluster(recv_s, (uint32_t)j) + (uint32_t)(((src * (CS / 4) + (half * HC + c) / 4) * BM + r) * 16);
                        const uint32_t bar = mapa_cluster(recv_bar, (uint32_t)j);
#pragma unroll
                        for (int e = 0; e < CW; e += 4) st_async_v4(dst + (uint32_t)(e / 4 * BM * 16), v[jj - 1] + e, bar);
                    }
                }
                ok = mbar_wait_cluster(recv_bar, 0, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (ok) {
#pragma unroll
                    for (int c = 0; c < HC; c += CW) {
                        uint32_t own[CW], v[CW];
                        tmem_ld<CW>(t_row + (uint32_t)(ks * CS + half * HC + c), own);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < S; ++j) {            // always summed in the order of the K shares
                            const int src = j < ks ? j : j - 1;
                            const uint32_t at = recv_s + (uint32_t)(((src * (CS / 4) + (half * HC + c) / 4) * BM + r) * 16);
#pragma unroll
                            for (int e = 0; e < CW; e += 4) {
                                uint4 q = make_uint4(own[e], own[e + 1], own[e + 2], own[e + 3]);
                                if (j != ks)
                                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                                 : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "r"(at + (uint32_t)(e / 4 * BM * 16)));
                                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                                for (int i = 0; i < 4; ++i)
                                    v[e + i] = j == 0 ? w[i] : __float_as_uint(__uint_as_float(v[e + i]) + __uint_as_float(w[i]));
                            }
                        }
                        const int col = ks * CS + half * HC + c;
                        finish_columns<CW, EPI, LNF>(args, tail, v, res + c / 8, row, col, n * BN + col, st);
                    }
                }
            }
        }
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    dep_wait();               // never finish before the kernel this one was allowed to overtake
    if (*abort_flag) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);    // let copies / MMAs in flight land
    }
    tc_fence_before();
    __syncthreads();
    if (S > 1) cluster_sync_all();            // no CTA leaves while a peer may still write to it
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

struct Maps { CUtensorMap x, w, bt, at; };

template <int BN, int EPI, bool LNF = false, int S = 1>
cudaError_t launch(const Launch& L, const Maps& t, SmallArgs a, int tiles) {
    constexpr int OTHER = recv_bytes<BN, S>() + (int)sizeof(Tail);
    constexpr int RING = (227 * 1024 - OTHER) / 1024 * 1024;
    // a full group of slabs leaves two stages, and its B slabs fit one
    static_assert(RING / (kps_of(BN) * (A_BLOCK + BN * BK * 2 + GROUP * PM_SLAB * BK * 2)) >= 2, "ring");
    static_assert(GROUP * BN * PM_SLAB * 2 <= kps_of(BN) * (A_BLOCK + BN * BK * 2 + GROUP * PM_SLAB * BK * 2), "B slabs");
    static SmemGrant grant;
    if (cudaError_t e = grant.ensure(small_linear_kernel<BN, EPI, LNF, S>, RING + OTHER); e != cudaSuccess) return e;
    a.ring_bytes = RING;
    ProfScope ps(L, KC_GEMM);
    const cudaError_t e = launch_overlapped(L, small_linear_kernel<BN, EPI, LNF, S>, tiles * S, THREADS, RING + OTHER, S,
                                            t.x, t.w, t.bt, t.at, a);
    BUMP(L);
    return e;
}

template <int BN>
cudaError_t launch_epi(const Launch& L, const Maps& t, const SmallArgs& a, int epi, int tiles, int split) {
    if (a.ln_g) {            // LayerNorm folded in: only the epilogues that follow a LayerNorm
        if (epi == EPI_GELU) return launch<BN, EPI_GELU, true>(L, t, a, tiles);
        if (epi == EPI_NONE) return launch<BN, EPI_NONE, true>(L, t, a, tiles);
        return cudaErrorInvalidValue;
    }
    switch (epi) {
        case EPI_GELU: return launch<BN, EPI_GELU>(L, t, a, tiles);
        case EPI_RESIDUAL:
            if constexpr (BN <= 128) if (split == 4) return launch<BN, EPI_RESIDUAL, false, 4>(L, t, a, tiles);
            if (split == 2) return launch<BN, EPI_RESIDUAL, false, 2>(L, t, a, tiles);
            return launch<BN, EPI_RESIDUAL>(L, t, a, tiles);
        case EPI_PATCH: return launch<BN, EPI_PATCH>(L, t, a, tiles);
        default: return launch<BN, EPI_NONE>(L, t, a, tiles);
    }
}

struct Shape { int width = -1, split = 1; };          // width: index into WIDTHS, -1 = not for this kernel

// The split of K and the tile width: as many CTAs as fit the SMs in one wave.  K is split where it is long
// (3072 -> 768 with adapters: 4 ways 7.1 us against 10.3 on 197 rows, 2 ways 15.4 against 20.5 on 1576; at 768
// inputs it costs what it gives, 768 -> 768 in two 5.0 against 5.3 us on 197 rows, 5.9 against 5.3 on 394, 9.5 against 5.8 on 788); the
// four-way split stops at 128 columns, whose partial sums leave the ring room.
// Without adapters the alternative is a GEMM kernel alone, to which wide tiles lose: unsplit 256-wide ones always.  With a
// residual, whose rows this kernel fetches and stores by thread, so do all but the narrow ones (64 columns, K in two 128) while the GEMM
// covers the rows in one round of 128-wide tiles, us here / GEMM, frames of 197 tokens:
//   768 -> 768 64-wide 6 frames 5.3 / 6.4, 128-wide 8: 7.7 / 6.9, 14: 8.1 / 7.6;  384 -> 384 64-wide 14: 4.5 / 5.2, 128-wide 16: 6.7 / 5.0;
//   1024 -> 1024 128-wide 10: 8.2 / 8.1;  3072 -> 768 in two, 128-wide 6: 10.7 / 12.0, 192-wide 8: 13.2 / 12.9, 256-wide 12: 16.9 / 13.3;
//   1536 -> 384 in two, 128-wide 10: 7.8 / 8.0, 192-wide 16: 9.9 / 8.9.
// Where it would take wider tiles or more rounds, unsplit 128-wide tiles win, or 192-wide ones with K in two; unsplit 192-wide ones still lose:
//   512 -> 512 128-wide 24: 6.8 / 8.6;  2048 -> 512 24: 11.6, 256-wide in two 14.2 / 15.8;  256 -> 256 (K too short for pairs) 28: 5.4 / 7.1;
//   3072 -> 576 (pairs are 192-wide) 64-wide 8: 10.7, 192-wide in two 12.5 / 15.7, 12: 13.4 / 15.9;
//   768 -> 768 192-wide 16: 10.3 / 8.9;  192 -> 192 192-wide 32: 7.6 / 4.4.
// With adapters the alternative is two kernels, whose t is rounded to bf16 once where the shares' t here keep 16 bits: K in two at 256
// columns stays here although it is slower (3072 -> 768, 12 frames 22.5 / 19.5, 14: 22.5 / 20.6; 2048 -> 512, 24 frames 18.3 / 21.0).
// Unsplit tiles of long K with adapters, which follow where the split no longer fits, are not always the faster side either: 3072 -> 768
// 192-wide 16 frames 24.2 / 23.4, 28: 30.5 / 29.3; 4096 -> 1024 256-wide 12: 34.8 / 30.0, 24: 39.0 / 41.7; 1536 -> 640 128-wide 12: 12.8 / 14.8.
Shape pick_shape(int k_in, int n_out, bool lora, int rows, int epi, int n_sms) {
    const long long m = (rows + BM - 1) / BM;
    const bool long_k = epi == EPI_RESIDUAL && k_in >= 1536, alone = epi == EPI_RESIDUAL && !lora;
    auto fits = [&](int i, int split) { return n_out % WIDTHS[i] == 0 && m * (n_out / WIDTHS[i]) * split <= n_sms; };
    for (int split = long_k ? 4 : 1; split >= 1; split >>= 1) {
        const int widest = split == 4 ? 128 : alone ? 64 * split : split == 1 && !lora ? 192 : 256;
        for (int i = 0; i < PM_SMALL_WIDTHS && WIDTHS[i] <= widest; ++i)
            if (fits(i, split)) return {i, split};
    }
    if (alone && !gemm_narrow_round(k_in, n_out, rows, n_sms)) {
        if (fits(1, 1)) return {1, 1};
        if (long_k && fits(2, 2)) return {2, 2};       // (256-wide in two takes as many CTAs as 128-wide unsplit)
    }
    return Shape();
}

}  // namespace

bool small_linear_encode(LinearDev& lin, int max_adapters, int slabs_max) {
    const uint64_t arena_rows = (uint64_t)max_adapters * slabs_max * PM_SLAB;
    for (int i = 0; i < PM_SMALL_WIDTHS; ++i) {
        if (!tm_encode_groups(&lin.tm_sw[i], lin.Wt, lin.k_in, lin.n_out, WIDTHS[i], kps_of(WIDTHS[i]))) return false;
        if (lin.lora.At && !tm_encode_2d(&lin.tm_sbt[i], lin.lora.Bt, PM_SLAB, arena_rows / PM_SLAB * lin.n_out, PM_SLAB * 2, PM_SLAB, WIDTHS[i], 32))
            return false;
    }
    for (int k = 0; k < 2; ++k)
        if (lin.lora.At && !tm_encode_groups(&lin.tm_sat[k], lin.lora.At, lin.k_in, arena_rows, PM_SLAB, k + 1)) return false;
    return true;
}

bool act_encode(ActMaps* m, const void* x, int k_in, uint64_t rows) {
    return tm_encode_kblocks(&m->k[0], x, k_in, rows, BM, 1) && tm_encode_kblocks(&m->k[1], x, k_in, rows, BM, 2);
}

static bool has_lora(const LinearDev& lin, const RouteDev* R) {
    return R && R->slab_cap > 0 && R->max_set > 0 && lin.lora.At != nullptr;
}

bool small_linear_form(int k_in, int n_out, bool lora, int rows, int epi, int n_sms, LinearForm* form) {
    const Shape s = pick_shape(k_in, n_out, lora, rows, epi, n_sms);
    if (s.width < 0) return false;
    *form = {LINEAR_FEW_ROWS, WIDTHS[s.width], s.split, THREADS};
    return true;
}

bool small_linear_fits(const LinearDev& lin, const RouteDev* R, int rows, int epi, int n_sms) {
    const bool lora = has_lora(lin, R);
    return pick_shape(lin.k_in, lin.n_out, lora, rows, epi, n_sms).width >= 0 && (!lora || R->tile_slab_cap <= LIST);
}

cudaError_t launch_small_linear(const Launch& L, const LinearDev& lin, const RouteDev* R, const ActMaps& x, int rows,
                                int epi, const bf16* residual, const PatchEpi& pe, bf16* y, int n_sms, float ln_eps) {
    if (rows <= 0) return cudaSuccess;
    const bool lora = has_lora(lin, R);
    const Shape shape = pick_shape(lin.k_in, lin.n_out, lora, rows, epi, n_sms);
    const int w = shape.width;
    if (w < 0) return cudaErrorInvalidValue;
    SmallArgs a = {};
    a.rows = rows; a.k_in = lin.k_in; a.n_out = lin.n_out; a.n_tiles = lin.n_out / WIDTHS[w];
    a.bias = lin.bias; a.residual = residual; a.y = y; a.pe = pe;
    if (lora) {
        a.tile_nslabs = R->tile_nslabs; a.tile_slab = R->tile_slab; a.tile_scale = R->tile_scale; a.tile_mask = R->tile_mask;
        a.slab_cap = R->slab_cap;
    }
    a.ln_g = lin.ln_g; a.ln_c1 = lin.ln_c1; a.ln_c2 = lin.ln_c2; a.ln_eps = ln_eps;
    a.status = L.status;
    const int kps = kps_of(WIDTHS[w]);
    Maps t;
    t.x = x.k[kps - 1]; t.w = lin.tm_sw[w];
    t.bt = lora ? lin.tm_sbt[w] : t.w;           // placeholders are never dereferenced
    t.at = lora ? lin.tm_sat[kps - 1] : t.w;
    const int tiles = (rows + BM - 1) / BM * a.n_tiles;
    switch (WIDTHS[w]) {
        case 64: return launch_epi<64>(L, t, a, epi, tiles, shape.split);
        case 128: return launch_epi<128>(L, t, a, epi, tiles, shape.split);
        case 192: return launch_epi<192>(L, t, a, epi, tiles, shape.split);
        default: return launch_epi<256>(L, t, a, epi, tiles, shape.split);
    }
}
