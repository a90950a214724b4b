// Shrink on the tensor cores: t[tile][s][row][j] = mask(row) * s_a * sum_k x[row,k] A_a[k, 16 s' + j], the first half of
// the LoRA term (Sec. 3.1), scaled and rounded to bf16 as the A operand of the fused GEMM's K = 16 steps; with a
// LayerNorm folded into the linear also the row statistics the GEMM needs.
//
// One CTA per 128-row tile (or a cluster of S CTAs that share K).  The tile's rows stream through shared memory once
// per group of adapter slabs, next to the group's A^T slabs, and one UMMA of N = 16 * slabs per 16 K columns
// accumulates in tensor memory; the epilogue warps scale, mask, round and store each slab as a [128 x 16] block.
//
// Full grids (more tiles than two per SM) are bound by their one read of x; three CTAs per SM keep every tile of a
// batch in flight at once.  Smaller grids are bound by the chain inside a CTA, and what made it long was serial work:
// a thread that re-read the slab list for every copy, one copy per slab and 64 columns, list, masks and LayerNorm
// terms fetched slab by slab in the epilogue.  So: x and adapter copies are issued by two threads, a copy brings two
// blocks of 64 columns where a CTA has shared memory for it, a warp prepares the slab data in shared memory, slabs
// that none of the tile's own rows use (the plan lists those of the 256-row pair) are only zeroed, the list and the
// first adapter slabs are fetched before the kernel waits for the one before it, and long K is split over a cluster
// where the tiles leave half of the SMs idle (partial sums through distributed shared memory, as asynchronous stores that
// count themselves on the receiver's barrier).
// Shrink + GEMM of one linear, replayed back to back, rank 16, 1 to 3 adapters per 197-token frame:
//   16 frames: qkv 16.2, proj 11.7 us; 37: qkv 24.8, fc2 36.9 us (K in two); 64: proj 21.8, fc2 59.8 us; 256: qkv 151, fc2 226 us.
// Warp roles: 0 = x copies, 1 = tensor memory + MMA, 2 = adapter copies, 3 = slab list, 4.. = statistics and t.
#include "common.cuh"
#include "f32x2.cuh"
#include "tcgen05_ptx.cuh"

#define BUMP(L) do { if ((L).launches) ++*(L).launches; } while (0)

namespace {

constexpr int BM = PM_TILE_M;
constexpr int BK = 64;
constexpr int MAX_STAGES = 6;
constexpr int FIRST_EW = 4;
constexpr int X_BLOCK = BM * BK * 2;                   // 16 KB
constexpr int A_BLOCK = PM_SLAB * BK * 2;              // 2 KB: one slab's rows, 64 columns
constexpr int T_F32 = BM * PM_SLAB * 4;                // 8 KB: a slab's partial sums

// The forms: Full for more than two tiles per SM, Mid for up to two, Wide and Split (a cluster per tile) for up to one.
//   KPS: K blocks per stage.  EW: epilogue warps.  GROUP: slabs per pass over x.
//   M_LIST / C_LIST: slabs whose masks and scales / LayerNorm terms fit the prepared list; the rest is read where it is used.
struct Full { static constexpr int KPS = 1, EW = 4, GROUP = 8, M_LIST = 40, C_LIST = 12, CTAS = 3; };
struct Mid { static constexpr int KPS = 1, EW = 8, GROUP = 16, M_LIST = 64, C_LIST = 32, CTAS = 2; };
struct Wide { static constexpr int KPS = 2, EW = 8, GROUP = 16, M_LIST = 64, C_LIST = 64, CTAS = 1; };
struct Split { static constexpr int KPS = 2, EW = 8, GROUP = 8, M_LIST = 64, C_LIST = 1, CTAS = 1; };
// Slabs of a pair that are told apart by use: 24 adapters (three frames of eight) of rank 64.  A pair with more takes every slab
// for both of its tiles.  Lists of 32 (Full) and 64 slabs did that from rank 32 on; 1 to 8 of 128 adapters per 197-token frame,
// shrink + GEMM, before -> now:  256 frames (Full), rank 32: 768 -> 2304 291 -> 270 us, 3072 -> 768 440 -> 375 us; rank 64:
// 475 -> 439 and 729 -> 604 us;  128 frames (Mid), rank 64: 260 -> 233 and 462 -> 390 us.
constexpr int LIST = 96;

template <typename F>
struct Tail {
    uint4 mask[F::M_LIST];
    float c[F::C_LIST][2 * PM_SLAB];                   // LayerNorm folded in: c1 then c2 of the slab
    float scale[F::M_LIST];
    int slab[LIST];                                    // arena slab
    uint8_t place[LIST];                               // place in the tile's list
    float2 half_stats[F::EW == 8 ? 2 : 1][F::EW == 8 ? BM : 1];     // mean, sum of squared deviations of half a row
    uint64_t bars[2 * MAX_STAGES + 4];
    uint32_t tmem_slot;
    int abort_flag, n_active;
};
static_assert(sizeof(Tail<Full>) <= 3 * 1024 && sizeof(Tail<Wide>) <= 15 * 1024, "shared memory");

struct ShrinkArgs {
    int rows, k_in, slab_cap, n_tiles;
    int reverse;                   // visit the tiles from the last row tile down (see launch_shrink)
    const int* tile_nslabs;
    const int* tile_slab;
    const float* tile_scale;
    const uint32_t* tile_mask;
    bf16* tbuf;
    int* status;
    // LayerNorm folded into the adapters (x is the raw residual stream, the arena holds gamma o A):
    //   t = s (rstd (x A' - mean c1) + c2);  stored divided by rstd, because the fused GEMM applies rstd to its
    //   whole accumulator, base and LoRA part alike.  The statistics go to stats_out for the GEMM; every row tile
    //   is then visited, with or without slabs.
    const float* ln_c1;
    const float* ln_c2;
    float2* stats_out;
    float ln_eps;
    int ring_bytes;
};

template <typename F, int S>
__host__ __device__ constexpr int recv_bytes() { return S > 1 ? (S - 1) * ((F::GROUP + S - 1) / S) * T_F32 : 0; }

template <typename F, bool STATS, int S>
__global__ void __launch_bounds__(32 * (FIRST_EW + F::EW), F::CTAS)
shrink_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_at, const ShrinkArgs args) {
    constexpr int KPS = F::KPS, EW = F::EW, GROUP = F::GROUP;
    constexpr int X_BYTES = KPS * X_BLOCK, A_SLAB = KPS * A_BLOCK;
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t base = smem_u32(smem);
    const int recv_off = args.ring_bytes;
    Tail<F>& tail = *reinterpret_cast<Tail<F>*>(smem + recv_off + recv_bytes<F, S>());
    const uint32_t bars = smem_u32(tail.bars);
    auto full_bar = [&](int s) { return bars + 8u * s; };              // both copying threads' bytes of a stage
    auto empty_bar = [&](int s) { return bars + 8u * (MAX_STAGES + s); };
    const uint32_t tfull_bar = bars + 8u * (2 * MAX_STAGES);
    const uint32_t tempty_bar = tfull_bar + 8u;
    const uint32_t stats_bar = tfull_bar + 16u;                        // LayerNorm terms prepared, half-row statistics exchanged
    const uint32_t recv_bar = tfull_bar + 24u;                         // the other CTAs' partial sums are here
    volatile int* abort_flag = &tail.abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ks = S > 1 ? (int)cluster_ctarank() : 0;
    const int tb = (int)blockIdx.x / S;
    const int tile = args.reverse ? args.n_tiles - 1 - tb : tb;
    const int ns = __ldg(args.tile_nslabs + tile);
    if (ns == 0 && !STATS) {                  // nothing to do for this tile (the whole cluster leaves; an exited CTA
        dep_wait();                           // counts as having released the kernel's dependents)
        return;
    }
    const size_t plan0 = (size_t)tile * args.slab_cap;
    const bool listed = ns <= LIST;           // else every slab is taken as active and its data read where it is used
    const int all_kb = args.k_in / BK;

    if (threadIdx.x == 0) {
        // a stage is free again when its MMAs are done and, with statistics, the epilogue warps have read it too
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), STATS ? 1 + EW : 1); }
        mbar_init(tfull_bar, 1);
        mbar_init(tempty_bar, EW);
        mbar_init(stats_bar, EW + 1);
        mbar_init(recv_bar, 1);
        tail.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    uint32_t acc_cols = 32;                   // power of two >= 16 * slabs of a pass
    while ((int)acc_cols < min(ns, GROUP) * PM_SLAB) acc_cols <<= 1;
    if (warp == 1) {
        tmem_alloc(smem_u32(&tail.tmem_slot), acc_cols);
        tmem_relinquish();
    } else if (warp == 3) {
        // the slabs that some row of THIS 128-row tile uses come first in the list, the others last
        int na = 0, nz = 0;
        for (int i0 = 0; listed && i0 < ns; i0 += 32) {
            const int i = i0 + lane;
            uint4 mk = make_uint4(0, 0, 0, 0);
            int slab = 0;
            float sc = 0.f;
            if (i < ns) {
                mk = __ldg(reinterpret_cast<const uint4*>(args.tile_mask) + plan0 + i);
                slab = __ldg(args.tile_slab + plan0 + i);
                sc = __ldg(args.tile_scale + plan0 + i);
            }
            const bool on = (mk.x | mk.y | mk.z | mk.w) != 0u, off = !on && i < ns;
            const uint32_t bon = __ballot_sync(0xFFFFFFFFu, on), boff = __ballot_sync(0xFFFFFFFFu, off);
            const uint32_t below = (1u << lane) - 1u;
            const int to = on ? na + __popc(bon & below) : LIST - 1 - nz - __popc(boff & below);
            if (on || off) { tail.slab[to] = slab; tail.place[to] = (uint8_t)i; }
            if (on && to < F::M_LIST) { tail.mask[to] = mk; tail.scale[to] = sc; }
            na += __popc(bon);
            nz += __popc(boff);
        }
        if (lane == 0) tail.n_active = listed ? na : ns;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (S > 1) cluster_sync_all();            // the peers' barriers are initialised
    const uint32_t tmem_base = tail.tmem_slot;
    const int na = tail.n_active;
    const int per_group = min(na, GROUP);
    // the first group's slabs i = ks mod S arrive from every other CTA
    if (S > 1 && threadIdx.x == 0 && na > 0) mbar_expect_tx(recv_bar, (uint32_t)((S - 1) * ((per_group - ks + S - 1) / S) * T_F32));
    const int stage_bytes = X_BYTES + per_group * A_SLAB;
    const int STG = min(MAX_STAGES, args.ring_bytes / stage_bytes);
    // groups of slabs; for the statistics a tile without slabs still makes one pass over x
    const int n_groups = na == 0 ? (STATS ? 1 : 0) : (na + GROUP - 1) / GROUP;
    // Stages [st0, st1) of group g are this CTA's.  A cluster shares the first group; further ones are its first
    // CTA's alone (their partial sums would need the exchange area again).
    const int all_st = (all_kb + KPS - 1) / KPS;
    auto share = [&](int g, int& st0, int& st1) {
        if (S == 1) { st0 = 0; st1 = all_st; }
        else if (g == 0) { st0 = all_st * ks / S; st1 = all_st * (ks + 1) / S; }
        else { st0 = 0; st1 = ks == 0 ? all_st : 0; }
    };
    auto slab_id = [&](int i) { return listed ? tail.slab[i] : __ldg(args.tile_slab + plan0 + i); };
    const bool usable = (base & 1023u) == 0;       // swizzled operands need a 1024-byte aligned window
    if (!usable && threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);

    if (!usable) {
        // fall through to the teardown
    } else if (warp == 0) {
        if (elect_one()) {
            // -------------------------------------------------------------- x copies
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            dep_wait();
            for (int g = 0; g < n_groups && ok; ++g) {
                int st0, st1;
                share(g, st0, st1);
                for (int st = st0; st < st1; ++st) {
                    ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    if (STATS && g > 0) mbar_arrive_n(empty_bar(stage), EW);      // the statistics' warps read the first pass only
                    mbar_expect_tx(full_bar(stage), X_BYTES);
                    if (na == 0) mbar_arrive(full_bar(stage));                    // nobody brings slabs
                    tma_load_3d(base + stage * stage_bytes, &tm_x, 0, tile * BM, st * KPS, full_bar(stage));
                    if (++stage == STG) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // -------------------------------------------------------------- adapter copies (not the earlier kernel's results)
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int g = 0; g < n_groups && na > 0 && ok; ++g) {
                int st0, st1;
                share(g, st0, st1);
                const int g0 = g * GROUP, cnt = min(GROUP, na - g0);
                for (int st = st0; st < st1; ++st) {
                    ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    mbar_expect_tx(full_bar(stage), cnt * A_SLAB);
                    const uint32_t sa = base + stage * stage_bytes + X_BYTES;
#pragma unroll 1
                    for (int i = 0; i < cnt; ++i)
                        tma_load_4d(sa + i * A_SLAB, &tm_at, 0, 0, st * KPS, slab_id(g0 + i) * (PM_SLAB / 8), full_bar(stage));
                    if (++stage == STG) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // -------------------------------------------------------------- MMA issuer
            const uint64_t da0 = smem_desc(base, 128), db0 = smem_desc_groups(base + X_BYTES, KPS * 1024);
            int stage = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int g = 0; g < n_groups && ok; ++g) {
                int st0, st1;
                share(g, st0, st1);
                if (st0 == st1) break;
                const int cnt = min(GROUP, na - g * GROUP);
                const uint32_t idesc = instr_desc(max(cnt, 1) * PM_SLAB);
                // the one accumulator: the epilogue warps have drained the previous group
                ok = mbar_wait(tempty_bar, acc_phase ^ 1u, abort_flag, args.status);
                if (!ok) break;
                tc_fence_after();
                uint32_t accumulate = 0;
                for (int st = st0; st < st1; ++st) {
                    ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                    if (!ok) break;
                    if (cnt > 0) {
                        tc_fence_after();
                        const uint64_t so = (uint64_t)((stage * stage_bytes) >> 4);
#pragma unroll
                        for (int j = 0; j < KPS; ++j) {
                            if (j > 0 && st * KPS + j >= all_kb) break;
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k) {
                                umma_bf16(tmem_base, da0 + so + (j * X_BLOCK >> 4) + 2 * k, db0 + so + (j * 1024 >> 4) + 2 * k, idesc, accumulate);
                                accumulate = 1;
                            }
                        }
                        umma_commit(empty_bar(stage));
                    } else {
                        mbar_arrive(empty_bar(stage));                   // statistics only
                    }
                    if (++stage == STG) { stage = 0; phase ^= 1u; }
                }
                if (ok && cnt > 0) umma_commit(tfull_bar);
                acc_phase ^= 1u;
            }
        }
    } else if (warp == 3) {
        // The fused GEMM that follows needs t (and the row statistics) only when its first tile's base K loop is
        // over: it may start on every SM this kernel's CTAs have left, while the slowest tiles finish.  It reads x
        // without waiting for this kernel, so it is released only when the kernel that wrote x has finished.
        dep_wait();
        dep_release();
        if (STATS) {
            for (int i = lane; i < min(listed ? na : 0, F::C_LIST) * 2 * PM_SLAB; i += 32) {
                const int s = i / (2 * PM_SLAB), j = i % (2 * PM_SLAB);
                tail.c[s][j] = __ldg((j < PM_SLAB ? args.ln_c1 : args.ln_c2) + (size_t)tail.slab[s] * PM_SLAB + (j & (PM_SLAB - 1)));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(stats_bar);
        }
    } else {
        // ------------------------------------------------------------------ statistics and t (warps 4..)
        const int quarter = warp & 3;
        const int half = (warp - FIRST_EW) >> 2;      // EW == 8: two warps per lane quarter
        constexpr int SHARES = EW / 4;
        const int r = quarter * 32 + lane;
        bool ok = true;
        float2 st = make_float2(0.f, 1.f);
        dep_wait();                                   // the GEMM that last read the t buffer has finished
        if (listed && ks == 0)
            for (int i = LIST - (ns - na) + half; i < LIST; i += SHARES) {           // slabs of the pair's other tile only
                uint4* dst = reinterpret_cast<uint4*>(args.tbuf + ((plan0 + tail.place[i]) * BM + r) * PM_SLAB);
                dst[0] = dst[1] = make_uint4(0, 0, 0, 0);
            }
        if constexpr (STATS) {
            // follow the ring: on the first pass a thread sums its row (EW == 8: half of its row) of each x block,
            // relative to its first element, which keeps the sum of squares well conditioned; packed pairs
            constexpr int CH = 8 / SHARES;             // 16-byte chunks of a block's row
            float pivot = 0.f;
            uint64_t np = 0, s1 = pk2(0.f, 0.f), s2 = s1;
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < all_kb && ok; kb += KPS) {
                ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
#pragma unroll
                for (int j = 0; j < KPS; ++j) {
                    if (j > 0 && kb + j >= all_kb) break;
                    const uint32_t row_addr = base + stage * stage_bytes + j * X_BLOCK + r * 128;
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        uint4 q;
                        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                                     : "r"(row_addr + (((half * CH + c) ^ (r & 7)) << 4)));
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
                float a0, a1, b0, b1;
                upk2(s1, a0, a1);
                upk2(s2, b0, b1);
                const float inv_n = (float)SHARES / (float)args.k_in;
                const float m1 = (a0 + a1) * inv_n;
                const float dev = fmaxf((b0 + b1) - (a0 + a1) * m1, 0.f);          // sum of squared deviations
                if constexpr (SHARES == 2) tail.half_stats[half][r] = make_float2(pivot + m1, dev);
                __syncwarp();
                if (lane == 0) mbar_arrive(stats_bar);
                ok = mbar_wait(stats_bar, 0, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if constexpr (SHARES == 2) {          // the two halves of a row (equal counts) are merged
                    const float2 h0 = tail.half_stats[0][r], h1 = tail.half_stats[1][r];
                    const float dm = h1.x - h0.x;
                    st = make_float2(0.5f * (h0.x + h1.x), rsqrtf((h0.y + h1.y) / (float)args.k_in + 0.25f * dm * dm + args.ln_eps));
                } else {
                    st = make_float2(pivot + m1, rsqrtf(dev / (float)args.k_in + args.ln_eps));
                }
                if (half == 0 && tile * BM + r < args.rows) args.stats_out[tile * BM + r] = st;
            }
        }
        const float inv_rstd = 1.f / st.y;
        const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
        // slab i of the list: accumulator -> scale, mask, folded LayerNorm -> bf16 -> t
        auto finish = [&](uint32_t* v, int i) {
            const int at = listed ? tail.place[i] : i;
            const bool held = listed && i < F::M_LIST;
            const uint32_t mk = held ? reinterpret_cast<const uint32_t*>(&tail.mask[i])[quarter] : __ldg(args.tile_mask + (plan0 + at) * 4 + quarter);
            const float sc = (mk >> lane) & 1u ? (held ? tail.scale[i] : __ldg(args.tile_scale + plan0 + at)) : 0.f;
            if constexpr (STATS) {
                if (listed && i < F::C_LIST) {
                    const float* c = tail.c[i];
#pragma unroll
                    for (int j = 0; j < PM_SLAB; ++j)
                        v[j] = __float_as_uint(fmaf(-st.x, c[j], __uint_as_float(v[j])) + inv_rstd * c[PM_SLAB + j]);
                } else {
                    const size_t slab = (size_t)slab_id(i) * PM_SLAB;
#pragma unroll
                    for (int j = 0; j < PM_SLAB; ++j)
                        v[j] = __float_as_uint(fmaf(-st.x, __ldg(args.ln_c1 + slab + j), __uint_as_float(v[j])) +
                                               inv_rstd * __ldg(args.ln_c2 + slab + j));
                }
            }
            uint4 o[2];
            uint32_t* ow = reinterpret_cast<uint32_t*>(o);
#pragma unroll
            for (int j = 0; j < PM_SLAB; j += 2)
                ow[j >> 1] = pack_bf16(__uint_as_float(v[j]) * sc, __uint_as_float(v[j + 1]) * sc);
            uint4* dst = reinterpret_cast<uint4*>(args.tbuf + ((plan0 + at) * BM + r) * PM_SLAB);
            dst[0] = o[0];
            dst[1] = o[1];
        };
        uint32_t acc_phase = 0;
        for (int g = 0; g < n_groups && na > 0 && ok; ++g) {
            int st0, st1;
            share(g, st0, st1);
            if (st0 == st1) break;
            const int g0 = g * GROUP, cnt = min(GROUP, na - g0);
            ok = mbar_wait(tfull_bar, acc_phase, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t recv_s = base + (uint32_t)recv_off;
            constexpr int PER = (GROUP + S - 1) / S;       // slabs i = j mod S are finished by CTA j
            if (S > 1 && g == 0) {
                // recv[src][i / S][4 columns][row]: src = the sender's place among the other CTAs
                for (int i = half; i < cnt; i += SHARES) {
                    const int j = i % S;
                    if (j == ks) continue;
                    uint32_t v[16];
                    tmem_ld16(t_row + (uint32_t)(i * PM_SLAB), v);
                    tmem_ld_wait();
                    const int src = ks < j ? ks : ks - 1;
                    const uint32_t dst = mapa_cluster(recv_s, (uint32_t)j) + (uint32_t)((src * PER + i / S) * T_F32 + r * 16);
                    const uint32_t bar = mapa_cluster(recv_bar, (uint32_t)j);
#pragma unroll
                    for (int e = 0; e < 16; e += 4) st_async_v4(dst + (uint32_t)(e / 4 * BM * 16), v + e, bar);
                }
                ok = mbar_wait_cluster(recv_bar, 0, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
            }
            for (int i = half; i < cnt; i += SHARES) {
                if (S > 1 && g == 0 && i % S != ks) continue;
                uint32_t v[16];
                tmem_ld16(t_row + (uint32_t)(i * PM_SLAB), v);
                tmem_ld_wait();
                if (S > 1 && g == 0) {
                    float sum[16];
#pragma unroll
                    for (int j = 0; j < S; ++j) {              // always summed in the order of the K shares
                        const int src = j < ks ? j : j - 1;
                        const uint32_t at = recv_s + (uint32_t)((src * PER + i / S) * T_F32 + r * 16);
#pragma unroll
                        for (int e = 0; e < 16; e += 4) {
                            uint4 q = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                            if (j != ks)
                                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                             : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "r"(at + (uint32_t)(e / 4 * BM * 16)));
                            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k) sum[e + k] = j == 0 ? __uint_as_float(w[k]) : sum[e + k] + __uint_as_float(w[k]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(sum[e]);
                }
                finish(v, g0 + i);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty_bar);
            acc_phase ^= 1u;
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
        tmem_dealloc(tmem_base, acc_cols);
    }
}

template <typename F, bool STATS, int S>
cudaError_t launch(const Launch& L, const CUtensorMap& tm_x, const CUtensorMap& tm_at, ShrinkArgs a) {
    constexpr int OTHER = recv_bytes<F, S>() + (int)sizeof(Tail<F>);
    // a multiprocessor has 228 KB, of which every CTA takes one for the system
    a.ring_bytes = (228 * 1024 / F::CTAS - 1024 - OTHER) / 1024 * 1024;
    static SmemGrant grant;
    if (cudaError_t e = grant.ensure(shrink_kernel<F, STATS, S>, a.ring_bytes + OTHER); e != cudaSuccess) return e;
    ProfScope ps(L, KC_SHRINK);
    const cudaError_t e = launch_overlapped(L, shrink_kernel<F, STATS, S>, a.n_tiles * S, 32 * (FIRST_EW + F::EW), a.ring_bytes + OTHER, S, tm_x, tm_at, a);
    BUMP(L);
    return e;
}

}  // namespace

cudaError_t launch_shrink(const Launch& L, const LinearDev& lin, const RouteDev& R, const ActMaps& x, int rows,
                          bf16* tbuf, int n_sms, float2* stats_out, float ln_eps) {
    if (R.n_tiles <= 0) return cudaSuccess;
    if (R.slab_cap <= 0) return stats_out ? cudaErrorInvalidValue : cudaSuccess;   // nothing to shrink
    if ((lin.ln_g != nullptr) != (stats_out != nullptr)) return cudaErrorInvalidValue;
    ShrinkArgs a;
    a.rows = rows; a.k_in = lin.k_in; a.slab_cap = R.slab_cap; a.n_tiles = R.n_tiles;
    a.tile_nslabs = R.tile_nslabs; a.tile_slab = R.tile_slab; a.tile_scale = R.tile_scale;
    a.tile_mask = R.tile_mask; a.tbuf = tbuf; a.status = L.status;
    a.ln_c1 = lin.ln_c1; a.ln_c2 = lin.ln_c2;
    a.stats_out = stats_out; a.ln_eps = ln_eps;
    // x larger than the L2 cache was written front to back by the kernel before this one, so its tail
    // is what the cache still holds: start there, and leave the front in the cache for the GEMM that
    // follows (which walks front to back)
    a.reverse = (size_t)rows * lin.k_in * sizeof(bf16) > ((size_t)96 << 20) ? 1 : 0;
    const int tiles = R.n_tiles;
    if (tiles > 2 * n_sms)
        return stats_out ? launch<Full, true, 1>(L, x.k[0], lin.tm_sat[0], a) : launch<Full, false, 1>(L, x.k[0], lin.tm_sat[0], a);
    if (tiles > n_sms)
        return stats_out ? launch<Mid, true, 1>(L, x.k[0], lin.tm_sat[0], a) : launch<Mid, false, 1>(L, x.k[0], lin.tm_sat[0], a);
    if (stats_out) return launch<Wide, true, 1>(L, x.k[1], lin.tm_sat[1], a);
    if (lin.k_in >= 1536 && tiles * 4 <= n_sms) return launch<Split, false, 4>(L, x.k[1], lin.tm_sat[1], a);
    if (lin.k_in >= 1536 && tiles * 2 <= n_sms) return launch<Split, false, 2>(L, x.k[1], lin.tm_sat[1], a);
    return launch<Wide, false, 1>(L, x.k[1], lin.tm_sat[1], a);
}
