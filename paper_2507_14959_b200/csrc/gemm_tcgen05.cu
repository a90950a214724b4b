// Fused base + multi-LoRA GEMM on the sm_100a tensor cores (Sec. 3.1: y = xW + sum_a s_a (xA_a)B_a).
//
//   y[128 x BN tile] = x_tile W^T_tile                        (K/64 pipeline stages, 4 UMMAs each)
//                    + sum over the tile's LoRA slabs  t_slab B_slab   (one K=16 UMMA per slab,
//                      into the SAME TMEM accumulator)
//                    -> epilogue: bias, GELU / residual / patch-embed placement, bf16 store.
//
// t (the scaled, row-masked shrink x A_cat of the tile) is produced by launch_shrink before the
// GEMM and fetched by TMA like any other operand.  Operands are staged by TMA into 128B- (base)
// and 32B- (LoRA slab) swizzled shared memory; a single thread issues tcgen05.mma; accumulators
// live in TMEM (two buffers, so the epilogue of one tile overlaps the main loop of the next).
// Warp roles: warp 0 = TMA producer, warp 1 = TMEM owner + MMA issuer, warps 2.. = epilogue (a warp per
// 64 columns of a TMEM lane quarter).
// Every mbarrier wait is bounded: on expiry the CTA raises an abort flag, records
// PM_ERR_TIMEOUT in the status word, drains and returns.
// The CTA-pair variant (lora_gemm_pair_kernel, cta_group::2, 256-row tiles of 128, 192 or 256 columns) serves most shapes, the single-CTA
// kernel short K and other widths (pick_pair_width).  Both start while the kernel before them on the stream still runs
// (programmatic dependent launch): 768 -> 768 with shrink on 197 x 256 rows 77.6 us behind its end, 73.4 so; on 197 x 37 rows 21.2, 15.4.
#include "common.cuh"
#include "f32x2.cuh"
#include "tcgen05_ptx.cuh"

#define BUMP(L) do { if ((L).launches) ++*(L).launches; } while (0)

namespace {

constexpr int BM = PM_TILE_M;
constexpr int BK = 64;
constexpr int SLABS_PER_STAGE = 4;

struct GemmArgs {
    int rows, k_in, n_out, m_tiles, n_tiles, epi;
    const float* bias;
    const bf16* residual;
    bf16* y;
    PatchEpi pe;
    // LoRA plan (null tile_nslabs = no LoRA)
    const int* tile_nslabs;
    const int* tile_slab;
    int slab_cap;
    int tma_store;             // 1: the epilogue stores through shared memory + TMA (tm_y valid)
    int wait_x;                // 0: the kernel before on the stream is this linear's shrink, x is complete; 1: await it first
    int* status;
    // LayerNorm folded into the linear (LNF kernels): y = rstd (acc - mean g) + bias, per row / column
    const float* ln_g;
    const float2* ln_stats;
};

constexpr int STAGING_BYTES = 32 * 64;                  // one chunk: [32 rows x 32 bf16]
constexpr int PLAN_BYTES = 2048;
constexpr int P_ACC_COLS = 256;                        // pair kernel: tensor-memory columns of one of the two accumulators

// The single-CTA kernel: an epilogue warp per 64 columns of a lane quarter, as in the pair kernel below.  The short K loops that
// run here are no longer than an epilogue: with eight warps 192 -> 768 took 12.2, 16.0 and 27.8 us on 64, 128 and 256 frames
// of 197 tokens, with sixteen 9.9, 13.1 and 23.7.
// 256-wide tiles leave room for four stages and one staging buffer per warp.
template <int BN>
struct Smem {
    static constexpr int EW = BN / 16;
    static constexpr int BUFFERS = BN == 256 ? 1 : 2;
    static constexpr int STAGES = 4;
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = BN * BK * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int T_SLAB_BYTES = BM * PM_SLAB * 2;      // 4096
    static constexpr int B_SLAB_BYTES = BN * PM_SLAB * 2;
    static constexpr int STAGING_OFFSET = STAGES * STAGE_BYTES;
    static constexpr int PLAN_OFFSET = STAGING_OFFSET + EW * BUFFERS * STAGING_BYTES;
    static constexpr int BAR_OFFSET = PLAN_OFFSET + PLAN_BYTES;
    static constexpr int TOTAL = BAR_OFFSET + 256;             // + barriers (base must be 1024-aligned)
};

// Epilogue of one 128 x BN accumulator by one epilogue warp: its share of the tile's 32-column
// chunks goes TMEM -> registers -> bias / GELU / residual / patch placement -> bf16 -> shared
// memory -> TMA store (or straight to global memory).  Returns false once the CTA is aborting.
// PAIR: the accumulator-free barrier lives in the even CTA of a pair (tempty_addr is a cluster address).
// RES_SMEM: request_residual has asked TMA for the residual rows of this warp's two chunks, into the staging buffers that the
// results will leave from (completion on res_bar); else per-thread global loads.
template <int BN, int EPI, int HALVES, int BUFFERS, bool PAIR, bool LNF, bool RES_SMEM>
__device__ __forceinline__ bool epilogue_tile(const GemmArgs& args, const CUtensorMap& tm_y, uint32_t staging,
                                              uint32_t& chunk_no, uint32_t tmem_base, int acc, uint32_t acc_phase,
                                              uint32_t tfull_addr, uint32_t tempty_addr, volatile int* abort_flag,
                                              int m, int n, int quarter, int half, int lane,
                                              uint32_t res_bar, uint32_t res_phase) {
    constexpr int CPW = BN / 32 / HALVES;         // 32-column chunks per epilogue warp
    static_assert(!RES_SMEM || CPW == 2, "a staging buffer per chunk");
    const int row = m * BM + quarter * 32 + lane;     // m: 128-row tile index
    const bool row_ok = row < args.rows;
    const int n_chunks = min(BN / 32, (args.n_out - n * BN) / 32);      // even: n_out % 64 == 0
    const int my_chunks = n_chunks / HALVES;
    const int c0 = half * my_chunks;
    // Without RES_SMEM a thread fetches its residual rows before the accumulator is ready, so that their latency hides behind the main
    // loop; where sixteen warps share the registers only the first chunk, and the next one as soon as the one before it is added
    // (384 -> 768 on 32, 64 and 256 frames of 197 tokens, no adapters, us with eight warps and all rows held / sixteen and all rows, which spilled /
    // now: 11.2 / 11.8 / 10.5, 16.5 / 17.5 / 15.7, 55.2 / 57.9 / 54.7; 128-wide tiles, eight warps, 384 -> 384 on 20 frames a chunk at a time 5.5, all
    // rows 5.2).  (In-place use, y == residual, is safe: the same thread reads an element here and is the only one to overwrite it
    // below, and a chunk's columns are its own.)
    constexpr bool RES_REGS = EPI == EPI_RESIDUAL && !RES_SMEM;
    constexpr int HELD = RES_REGS && BN <= 128 ? CPW : 1;
    uint4 rr[HELD][4];
    const uint4* rr_from = nullptr;
    if constexpr (RES_REGS) {
        rr_from = reinterpret_cast<const uint4*>(args.residual + (size_t)row * args.n_out + n * BN + c0 * 32);
#pragma unroll
        for (int cc = 0; cc < HELD; ++cc)
#pragma unroll
            for (int q = 0; q < 4; ++q) rr[cc][q] = row_ok && cc < my_chunks ? rr_from[cc * 4 + q] : make_uint4(0, 0, 0, 0);
    }
    bool ok = PAIR ? mbar_wait_cluster(tfull_addr, acc_phase, abort_flag, args.status)
                   : mbar_wait(tfull_addr, acc_phase, abort_flag, args.status);
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (!ok) return false;
    tc_fence_after();
    size_t orow = (size_t)row;
    const float* pos_row = nullptr;
    if (EPI == EPI_PATCH && row_ok) {
        const int p = row % args.pe.g2;
        orow = (size_t)(row / args.pe.g2) * args.pe.tokens + 1 + p;
        pos_row = args.pe.pos + (size_t)(1 + p) * args.n_out;
    }
    const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * (PAIR ? P_ACC_COLS : BN));
    float2 st = make_float2(0.f, 1.f);                 // (mean, rstd) of this thread's row
    if (LNF && row_ok) st = args.ln_stats[row];
#pragma unroll
    for (int cc = 0; cc < CPW; ++cc) {
        if (cc >= my_chunks) break;
        const int c = c0 + cc;
        const int n0 = n * BN + c * 32;
        uint32_t v[32];
        tmem_ld32(t_row + (uint32_t)(c * 32), v);
        tmem_ld_wait();
        if (cc == my_chunks - 1) {
            // every TMEM read of this accumulator is done: hand the buffer back early
            tc_fence_before();
            __syncwarp();
            if (elect_one()) { if (PAIR) mbar_arrive_cluster(tempty_addr); else mbar_arrive(tempty_addr); }
        }
        // bias (and the folded LayerNorm: rstd (acc - mean g) + b) and GELU, two columns per instruction
        uint64_t fp[16];                                 // columns (2i, 2i+1) of this chunk
        const uint64_t rstd2 = pk2(st.y, st.y), nmean2 = pk2(-st.x, -st.x);
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float4 b4 = __ldg(reinterpret_cast<const float4*>(args.bias + n0 + j));
            uint64_t a0 = pk2(__uint_as_float(v[j + 0]), __uint_as_float(v[j + 1]));
            uint64_t a1 = pk2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
            if constexpr (LNF) {
                const float4 g4 = __ldg(reinterpret_cast<const float4*>(args.ln_g + n0 + j));
                a0 = fma2(rstd2, fma2(nmean2, pk2(g4.x, g4.y), a0), pk2(b4.x, b4.y));
                a1 = fma2(rstd2, fma2(nmean2, pk2(g4.z, g4.w), a1), pk2(b4.z, b4.w));
            } else {
                a0 = add2(a0, pk2(b4.x, b4.y));
                a1 = add2(a1, pk2(b4.z, b4.w));
            }
            if constexpr (EPI == EPI_GELU) { a0 = gelu_erf2(a0); a1 = gelu_erf2(a1); }
            fp[j >> 1] = a0;
            fp[(j >> 1) + 1] = a1;
        }
        if constexpr (EPI == EPI_RESIDUAL) {
            if constexpr (RES_SMEM) {
                if (cc == 0) {
                    ok = mbar_wait(res_bar, res_phase, abort_flag, args.status);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) return false;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint4 r4v;
                if constexpr (RES_SMEM) {
                    // where this thread puts its result below: 16-byte chunk q of row `lane`
                    const uint32_t a = staging + chunk_no % BUFFERS * STAGING_BYTES + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4);
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(r4v.x), "=r"(r4v.y), "=r"(r4v.z), "=r"(r4v.w) : "r"(a));
                } else {
                    r4v = rr[cc % HELD][q];
                }
                const uint32_t w[4] = {r4v.x, r4v.y, r4v.z, r4v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    fp[q * 4 + e] = add2(fp[q * 4 + e], pk2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xFFFF0000u)));
            }
            if constexpr (RES_REGS && HELD < CPW) {
                if (row_ok && cc + 1 < my_chunks) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) rr[0][q] = rr_from[(cc + 1) * 4 + q];
                }
            }
        } else if constexpr (EPI == EPI_PATCH) {
            if (row_ok) {
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 p4 = __ldg(reinterpret_cast<const float4*>(pos_row + n0 + j));
                    fp[j >> 1] = add2(fp[j >> 1], pk2(p4.x, p4.y));
                    fp[(j >> 1) + 1] = add2(fp[(j >> 1) + 1], pk2(p4.z, p4.w));
                }
            }
        }
        uint4 o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float lo, hi;
            upk2(fp[q * 4 + 0], lo, hi); o[q].x = pack_bf16(lo, hi);
            upk2(fp[q * 4 + 1], lo, hi); o[q].y = pack_bf16(lo, hi);
            upk2(fp[q * 4 + 2], lo, hi); o[q].z = pack_bf16(lo, hi);
            upk2(fp[q * 4 + 3], lo, hi); o[q].w = pack_bf16(lo, hi);
        }
        if (args.tma_store) {
            // [32 rows x 64 B] block, 16-byte chunks XOR-swizzled by (row >> 1) & 3 (64B
            // swizzle), then one TMA store; rows past the end are clipped by the tensor map
            const uint32_t buf = staging + chunk_no % BUFFERS * STAGING_BYTES;
            if constexpr (!RES_SMEM) {
                if (elect_one()) { if constexpr (BUFFERS == 2) bulk_wait_read1(); else bulk_wait_read0(); }      // the store that last used this buffer has read it
                __syncwarp();
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                st_shared_v4(buf + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4), o[q]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (elect_one()) {
                tma_store_2d(&tm_y, buf, n0, m * BM + quarter * 32);
                bulk_commit();
            }
            ++chunk_no;
        } else if (row_ok) {
            uint4* o4 = reinterpret_cast<uint4*>(args.y + orow * args.n_out + n0);
#pragma unroll
            for (int q = 0; q < 4; ++q) o4[q] = o[q];
        }
    }
    return true;
}

// Asks TMA for the residual rows of an epilogue warp's two chunks (rows past the end read as zero), into the warp's staging
// buffers as soon as the stores of its previous tile have read them: ahead of their use by what is left of the tile's main loop then
// (all of it for a CTA's first tile, little where an epilogue takes as long as a main loop).
template <int BN>
__device__ __forceinline__ void request_residual(const CUtensorMap& tm_res, uint32_t staging, uint32_t res_bar, int m, int n, int quarter, int half) {
    if (elect_one()) {
        bulk_wait_read0();
        mbar_expect_tx(res_bar, 2 * 32 * 64);
        for (int cc = 0; cc < 2; ++cc)
            tma_load_2d(staging + cc * (32 * 64), &tm_res, n * BN + (half * 2 + cc) * 32, m * BM + quarter * 32, res_bar);
    }
    __syncwarp();
}

template <int BN, int EPI, bool LNF>
__global__ void __launch_bounds__(64 + 32 * Smem<BN>::EW, 1)
lora_gemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                 const __grid_constant__ CUtensorMap tm_t, const __grid_constant__ CUtensorMap tm_bt,
                 const __grid_constant__ CUtensorMap tm_y, const GemmArgs args) {
    using S = Smem<BN>;
    constexpr int EW = S::EW, STAGES = S::STAGES;
    constexpr int NTHREADS = 64 + 32 * EW;
    constexpr int HALVES = EW / 4;                // epilogue warps per TMEM lane quarter
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if (base & 1023u) {                       // swizzled operands need a 1024-byte aligned window
        if (threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);
        return;
    }
    uint8_t* smem = smem_raw;
    const uint32_t bars = base + S::BAR_OFFSET;
    // barrier words: full[STAGES], empty[STAGES], tmem_full[2], tmem_empty[2]
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    auto tfull_bar = [&](int s) { return bars + 8u * (2 * STAGES + s); };
    auto tempty_bar = [&](int s) { return bars + 8u * (2 * STAGES + 2 + s); };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + S::BAR_OFFSET + 8 * (2 * STAGES + 4));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + S::BAR_OFFSET + 8 * (2 * STAGES + 4) + 8);
    int* plan = reinterpret_cast<int*>(smem + S::PLAN_OFFSET);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total_tiles = args.m_tiles * args.n_tiles;
    const int num_kb = args.k_in / BK;

    // The LoRA plan of this CTA's tiles (slab count + arena slab ids) is copied to shared memory
    // once, so that the producer and the MMA issuer never wait on a global load between tiles.
    const int plan_stride = 1 + args.slab_cap;
    const int plan_tiles = args.tile_nslabs ? PLAN_BYTES / (4 * plan_stride) : 0;
    if (args.tile_nslabs) {
        for (int i = threadIdx.x / 8; i < plan_tiles; i += NTHREADS / 8) {
            const int tile = blockIdx.x + i * gridDim.x;
            if (tile >= total_tiles) break;
            const int m = tile / args.n_tiles;
            const int ns = args.tile_nslabs[m];
            if ((threadIdx.x & 7) == 0) plan[i * plan_stride] = ns;
            for (int q = threadIdx.x & 7; q < ns; q += 8) plan[i * plan_stride + 1 + q] = args.tile_slab[m * args.slab_cap + q];
        }
    }
    auto tile_ns = [&](int it, int m) -> int {
        if (!args.tile_nslabs) return 0;
        return it < plan_tiles ? plan[it * plan_stride] : args.tile_nslabs[m];
    };
    auto tile_slab_id = [&](int it, int m, int q) -> int {
        return it < plan_tiles ? plan[it * plan_stride + 1 + q] : args.tile_slab[m * args.slab_cap + q];
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(tfull_bar(s), 1); mbar_init(tempty_bar(s), EW); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(smem_u32((const void*)tmem_slot), 2 * BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    dep_release();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true, dep_done = false;
            int it = 0;
            if (args.wait_x) { dep_wait(); dep_done = true; }
            for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, ++it) {
                const int m = tile / args.n_tiles, n = tile % args.n_tiles;
                for (int kb = 0; kb < num_kb && ok; ++kb) {
                    ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    mbar_expect_tx(full_bar(stage), S::STAGE_BYTES);
                    const uint32_t sa = base + stage * S::STAGE_BYTES;
                    tma_load_2d(sa, &tm_x, kb * BK, m * BM, full_bar(stage));
                    tma_load_2d(sa + S::A_BYTES, &tm_w, kb * BK, n * BN, full_bar(stage));
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                const int ns = tile_ns(it, m);
                if (ns > 0 && !dep_done) { dep_wait(); dep_done = true; }     // t comes from the shrink kernel
                for (int g0 = 0; g0 < ns && ok; g0 += SLABS_PER_STAGE) {
                    const int cnt = min(SLABS_PER_STAGE, ns - g0);
                    ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    mbar_expect_tx(full_bar(stage), cnt * (S::T_SLAB_BYTES + S::B_SLAB_BYTES));
                    const uint32_t sa = base + stage * S::STAGE_BYTES;
                    for (int i = 0; i < cnt; ++i) {
                        const int slot = m * args.slab_cap + g0 + i;
                        const int slab = tile_slab_id(it, m, g0 + i);
                        tma_load_2d(sa + i * S::T_SLAB_BYTES, &tm_t, 0, slot * BM, full_bar(stage));
                        tma_load_2d(sa + S::A_BYTES + i * S::B_SLAB_BYTES, &tm_bt, 0,
                                    slab * args.n_out + n * BN, full_bar(stage));
                    }
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idesc = instr_desc(BN);
            // Descriptors of stage 0; a stage adds STAGE_BYTES / 16 and a K step of 16 adds 2 to the
            // address field.  Keeping the issuing thread's work per K block to a handful of
            // instructions matters: the tensor pipe runs dry whenever this thread is late.
            const uint64_t da0 = smem_desc(base, 128), db0 = smem_desc(base + S::A_BYTES, 128);
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            int it = 0;
            for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, ++it) {
                const int m = tile / args.n_tiles;
                const int ns = tile_ns(it, m);
                ok = mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, args.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                uint32_t accumulate = 0;
                for (int kb = 0; kb < num_kb && ok; ++kb) {
                    ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t so = (uint64_t)(stage * (S::STAGE_BYTES >> 4));
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        umma_bf16(d_tmem, da0 + so + 2 * k, db0 + so + 2 * k, idesc, accumulate);
                        accumulate = 1;
                    }
                    umma_commit(empty_bar(stage));
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                for (int g0 = 0; g0 < ns && ok; g0 += SLABS_PER_STAGE) {
                    const int cnt = min(SLABS_PER_STAGE, ns - g0);
                    ok = mbar_wait(full_bar(stage), phase, abort_flag, args.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sa = base + stage * S::STAGE_BYTES;
                    const uint32_t sb = sa + S::A_BYTES;
                    for (int i = 0; i < cnt; ++i) {
                        umma_bf16(d_tmem, smem_desc(sa + i * S::T_SLAB_BYTES, 32),
                                  smem_desc(sb + i * S::B_SLAB_BYTES, 32), idesc, accumulate);
                        accumulate = 1;
                    }
                    umma_commit(empty_bar(stage));
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                if (ok) umma_commit(tfull_bar(acc));
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..)
        const int quarter = warp & 3;                 // TMEM lanes 32*quarter .. +31
        const int half = (warp - 2) >> 2;             // which share of the tile's 32-column chunks
        const uint32_t staging = base + S::STAGING_OFFSET + (uint32_t)(warp - 2) * (S::BUFFERS * STAGING_BYTES);
        dep_wait();                                   // row statistics, residual; rows that the kernel before still reads
        int acc = 0;
        uint32_t acc_phase = 0;
        uint32_t chunk_no = 0;                        // running chunk counter: picks the staging buffer
        bool ok = true;
        for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
            const int m = tile / args.n_tiles, n = tile % args.n_tiles;
            ok = epilogue_tile<BN, EPI, HALVES, S::BUFFERS, false, LNF, false>(args, tm_y, staging, chunk_no, tmem_base, acc,
                                                              acc_phase, tfull_bar(acc), tempty_bar(acc), abort_flag,
                                                              m, n, quarter, half, lane, 0u, 0u);
            if (!ok) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (args.tma_store && elect_one()) bulk_wait_all();
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    dep_wait();               // never finish before the kernel this one was allowed to overtake
    if (*abort_flag) {
        // give copies and MMAs still in flight time to land before shared memory / TMEM go away
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 2 * BN);
    }
}

// ---------------------------------------------------------------------------------------
// The same GEMM on CTA pairs (BN = 128, 192 or 256).  Two CTAs of a cluster share one
// 256 x BN output tile: each stages its own 128 rows of x (and of the t slabs) and HALF of the
// W^T tile (and of the B slabs), so every byte of W^T crosses the L2 -> SM fabric once per 256
// rows instead of once per 128, and one tcgen05.mma.cta_group::2 (M = 256) issued by the even
// CTA drives the tensor cores of both SMs, each accumulating its own 128 rows in its own TMEM.
//   full[s]    (even CTA)   bytes of both CTAs' loads of stage s (the odd CTA's TMA signals it)
//   empty[s]   (both CTAs)  the pair MMAs that read stage s are done (multicast commit)
//   tfull[a]   (both CTAs)  accumulator a is complete (multicast commit)
//   tempty[a]  (even CTA)   both CTAs' epilogue warps have drained accumulator a
// Eight (128 columns), six, or with a 256-wide residual five stages per CTA.  No TMA multicast is used.
// ---------------------------------------------------------------------------------------
constexpr int P_A_BYTES = BM * BK * 2;                 // 16 KB: this CTA's 128 rows of x
constexpr int P_T_SLAB_BYTES = BM * PM_SLAB * 2;       // 4 KB
constexpr int P_MAX_STAGES = 8;
constexpr int P_MAX_EW = 16;
constexpr int P_BAR_BYTES = 512;
// By tile width: an epilogue warp takes 64 columns of one lane quarter (two chunks), so 256 columns take 16 warps.  With a residual
// there is a staging buffer for each chunk (request_residual); else 256-wide tiles have one per warp, which leaves the ring its sixth stage.
// Two per warp and five stages, us, five stages / six, no adapters, frames of 197 tokens: 3072 -> 256, 75 and 256 frames 23.0 / 22.0 and 71.1 / 68.5;
// 3072 -> 768, 256 frames 165 / 159; 768 -> 2304, 128 frames 67.3 / 66.3, with adapters 81.3 / 77.9.
// Patch placement stores rows by thread straight to memory, where more warps only spread the writes: eight at 256 columns too
// (768 -> 768 on 96, 128 and 256 frames of 196 patches 45.8, 57.6 and 104.9 us with sixteen, 44.9, 56.6 and 102.8 with eight).
template <int BN, int EPI>
struct PairCfg {
    static constexpr int BUFFERS = BN < 256 || EPI == EPI_RESIDUAL ? 2 : 1;
    static constexpr int STAGING_PER_WARP = BUFFERS * STAGING_BYTES;
    static constexpr int HALVES = BN == 256 && EPI == EPI_PATCH ? 2 : BN / 64;      // epilogue warps per lane quarter
    static constexpr int EW = 4 * HALVES;
    static constexpr int THREADS = 64 + 32 * EW;
    static constexpr int B_BYTES = (BN / 2) * BK * 2;                      // this CTA's half of the W^T tile
    static constexpr int STAGE_BYTES = P_A_BYTES + B_BYTES;
    static constexpr int B_SLAB_BYTES = (BN / 2) * PM_SLAB * 2;
    static constexpr int REST = EW * STAGING_PER_WARP + PLAN_BYTES + P_BAR_BYTES;
    static constexpr int FIT = (227 * 1024 - REST) / STAGE_BYTES;
    static constexpr int STAGES = FIT < P_MAX_STAGES ? FIT : P_MAX_STAGES;
    static constexpr int STAGING_OFFSET = STAGES * STAGE_BYTES;
    static constexpr int PLAN_OFFSET = STAGING_OFFSET + EW * STAGING_PER_WARP;
    static constexpr int BAR_OFFSET = PLAN_OFFSET + PLAN_BYTES;
    static constexpr int TOTAL = BAR_OFFSET + P_BAR_BYTES;
    static_assert(SLABS_PER_STAGE * B_SLAB_BYTES <= B_BYTES, "LoRA stage");
    static_assert(STAGES >= (EPI == EPI_RESIDUAL ? 5 : 6), "long K needs the depth");
    static_assert(8 * (2 * P_MAX_STAGES + 4) + 24 + 8 * P_MAX_EW <= P_BAR_BYTES, "barriers");
};

template <int BN, int EPI, bool LNF>
__global__ void __launch_bounds__(PairCfg<BN, EPI>::THREADS, 1)
lora_gemm_pair_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                      const __grid_constant__ CUtensorMap tm_t, const __grid_constant__ CUtensorMap tm_bt,
                      const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_res,
                      const GemmArgs args) {
    using C = PairCfg<BN, EPI>;
    constexpr int P_STAGES = C::STAGES, P_EW = C::EW;
    constexpr bool RES = EPI == EPI_RESIDUAL;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    const uint32_t rank = cluster_ctarank();          // 0: issues the MMAs, 1: its peer
    uint8_t* smem = smem_raw;
    const uint32_t bars = base + C::BAR_OFFSET;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (P_MAX_STAGES + s); };
    auto tfull_bar = [&](int s) { return bars + 8u * (2 * P_MAX_STAGES + s); };
    auto tempty_bar = [&](int s) { return bars + 8u * (2 * P_MAX_STAGES + 2 + s); };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + C::BAR_OFFSET + 8 * (2 * P_MAX_STAGES + 4));
    // the peer CTA's TMEM base: written only by the peer (any time before the cluster barrier below),
    // never by this CTA, so there is no ordering to get wrong
    volatile uint32_t* peer_slot = tmem_slot + 1;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::BAR_OFFSET + 8 * (2 * P_MAX_STAGES + 4) + 8);
    // res_bar[w]: the residual rows of epilogue warp w's chunks have landed (residual kernels)
    auto res_bar = [&](int w) { return bars + 8u * (2 * P_MAX_STAGES + 4) + 24u + 8u * w; };
    int* plan = reinterpret_cast<int*>(smem + C::PLAN_OFFSET);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pair_id = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int total_tiles = args.m_tiles * args.n_tiles;      // m_tiles counts 256-row tiles here
    const int num_kb = args.k_in / BK;

    // LoRA plan of this CTA's tiles (both halves of a 256-row tile carry the same slab list)
    const int plan_stride = 1 + args.slab_cap;
    const int plan_tiles = args.tile_nslabs ? PLAN_BYTES / (4 * plan_stride) : 0;
    if (args.tile_nslabs) {
        for (int i = threadIdx.x / 8; i < plan_tiles; i += C::THREADS / 8) {
            const int tile = pair_id + i * n_pairs;
            if (tile >= total_tiles) break;
            const int m = 2 * (tile / args.n_tiles) + (int)rank;
            const int ns = args.tile_nslabs[m];
            if ((threadIdx.x & 7) == 0) plan[i * plan_stride] = ns;
            for (int q = threadIdx.x & 7; q < ns; q += 8) plan[i * plan_stride + 1 + q] = args.tile_slab[m * args.slab_cap + q];
        }
    }
    auto tile_ns = [&](int it, int m) -> int {
        if (!args.tile_nslabs) return 0;
        return it < plan_tiles ? plan[it * plan_stride] : args.tile_nslabs[m];
    };
    auto tile_slab_id = [&](int it, int m, int q) -> int {
        return it < plan_tiles ? plan[it * plan_stride + 1 + q] : args.tile_slab[m * args.slab_cap + q];
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < P_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(tfull_bar(s), 1); mbar_init(tempty_bar(s), 2 * P_EW); }
        for (int w = 0; w < P_EW; ++w) mbar_init(res_bar(w), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(smem_u32((const void*)tmem_slot), 512);     // all of this SM's tensor memory
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // both CTAs must hold the same TMEM columns (the pair MMA uses one address for both); tell the peer
    if (threadIdx.x == 0) st_cluster_u32(mapa_cluster(smem_u32((const void*)peer_slot), rank ^ 1u), tmem_base);
    cluster_sync_all();          // barriers initialised and TMEM bases exchanged in both CTAs
    dep_release();
    const bool usable = ((base & 1023u) == 0) && (*peer_slot == tmem_base);
    if (!usable && threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);

    if (!usable) {
        // fall through to the teardown
    } else if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true, dep_done = false;
            int it = 0;
            // x comes from the kernel before (unless that one is this linear's shrink, which releases this kernel
            // only when x is complete): until it has finished, the first stages' weights are fetched alone
            int pre = 0;
            if (args.wait_x) {
                pre = min(P_STAGES, num_kb);
                const int m = 2 * (pair_id / args.n_tiles) + (int)rank, n = pair_id % args.n_tiles;
                for (int kb = 0; kb < pre; ++kb) {
                    if (rank == 0) mbar_expect_tx(full_bar(kb), 2 * C::STAGE_BYTES);
                    tma_load_2d_pair(base + kb * C::STAGE_BYTES + P_A_BYTES, &tm_w, kb * BK, n * BN + (int)rank * (BN / 2), mapa_cluster(full_bar(kb), 0));
                }
                dep_wait();
                dep_done = true;
                for (int kb = 0; kb < pre; ++kb)
                    tma_load_2d_pair(base + kb * C::STAGE_BYTES, &tm_x, kb * BK, m * BM, mapa_cluster(full_bar(kb), 0));
                if (pre == P_STAGES) phase = 1u; else stage = pre;
            }
            for (int tile = pair_id; tile < total_tiles && ok; tile += n_pairs, ++it) {
                const int m2 = tile / args.n_tiles, n = tile % args.n_tiles;
                const int m = 2 * m2 + (int)rank;                   // this CTA's 128-row tile
                for (int kb = it == 0 ? pre : 0; kb < num_kb && ok; ++kb) {
                    ok = mbar_wait_cluster(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    const uint32_t fb = mapa_cluster(full_bar(stage), 0);
                    if (rank == 0) mbar_expect_tx(full_bar(stage), 2 * C::STAGE_BYTES);
                    const uint32_t sa = base + stage * C::STAGE_BYTES;
                    tma_load_2d_pair(sa, &tm_x, kb * BK, m * BM, fb);
                    tma_load_2d_pair(sa + P_A_BYTES, &tm_w, kb * BK, n * BN + (int)rank * (BN / 2), fb);
                    if (++stage == P_STAGES) { stage = 0; phase ^= 1u; }
                }
                const int ns = tile_ns(it, m);
                if (ns > 0 && !dep_done) { dep_wait(); dep_done = true; }     // t comes from the shrink kernel
                for (int g0 = 0; g0 < ns && ok; g0 += SLABS_PER_STAGE) {
                    const int cnt = min(SLABS_PER_STAGE, ns - g0);
                    ok = mbar_wait_cluster(empty_bar(stage), phase ^ 1u, abort_flag, args.status);
                    if (!ok) break;
                    const uint32_t fb = mapa_cluster(full_bar(stage), 0);
                    if (rank == 0) mbar_expect_tx(full_bar(stage), 2 * cnt * (P_T_SLAB_BYTES + C::B_SLAB_BYTES));
                    const uint32_t sa = base + stage * C::STAGE_BYTES;
                    for (int i = 0; i < cnt; ++i) {
                        const int slot = m * args.slab_cap + g0 + i;
                        const int slab = tile_slab_id(it, m, g0 + i);
                        tma_load_2d_pair(sa + i * P_T_SLAB_BYTES, &tm_t, 0, slot * BM, fb);
                        tma_load_2d_pair(sa + P_A_BYTES + i * C::B_SLAB_BYTES, &tm_bt, 0,
                                         slab * args.n_out + n * BN + (int)rank * (BN / 2), fb);
                    }
                    if (++stage == P_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (even CTA only)
        if (rank == 0 && elect_one()) {
            const uint32_t idesc = instr_desc_pair(BN);
            const uint64_t da0 = smem_desc(base, 128), db0 = smem_desc(base + P_A_BYTES, 128);
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            int it = 0;
            for (int tile = pair_id; tile < total_tiles && ok; tile += n_pairs, ++it) {
                const int m = 2 * (tile / args.n_tiles);
                const int ns = tile_ns(it, m);
                ok = mbar_wait_cluster(tempty_bar(acc), acc_phase ^ 1u, abort_flag, args.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * P_ACC_COLS);
                uint32_t accumulate = 0;
                for (int kb = 0; kb < num_kb && ok; ++kb) {
                    ok = mbar_wait_cluster(full_bar(stage), phase, abort_flag, args.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t so = (uint64_t)(stage * (C::STAGE_BYTES >> 4));
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        umma_bf16_pair(d_tmem, da0 + so + 2 * k, db0 + so + 2 * k, idesc, accumulate);
                        accumulate = 1;
                    }
                    umma_commit_pair(empty_bar(stage));
                    if (++stage == P_STAGES) { stage = 0; phase ^= 1u; }
                }
                for (int g0 = 0; g0 < ns && ok; g0 += SLABS_PER_STAGE) {
                    const int cnt = min(SLABS_PER_STAGE, ns - g0);
                    ok = mbar_wait_cluster(full_bar(stage), phase, abort_flag, args.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sa = base + stage * C::STAGE_BYTES;
                    const uint32_t sb = sa + P_A_BYTES;
                    for (int i = 0; i < cnt; ++i) {
                        umma_bf16_pair(d_tmem, smem_desc(sa + i * P_T_SLAB_BYTES, 32),
                                       smem_desc(sb + i * C::B_SLAB_BYTES, 32), idesc, accumulate);
                        accumulate = 1;
                    }
                    umma_commit_pair(empty_bar(stage));
                    if (++stage == P_STAGES) { stage = 0; phase ^= 1u; }
                }
                if (ok) umma_commit_pair(tfull_bar(acc));
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (both CTAs)
        const int quarter = warp & 3;
        const int half = (warp - 2) >> 2;
        const uint32_t staging = base + C::STAGING_OFFSET + (uint32_t)(warp - 2) * C::STAGING_PER_WARP;
        dep_wait();                                   // row statistics, residual; rows that the kernel before still reads
        int acc = 0;
        uint32_t acc_phase = 0, res_phase = 0;
        uint32_t chunk_no = 0;
        bool ok = true;
        for (int tile = pair_id; tile < total_tiles && ok; tile += n_pairs) {
            const int m = 2 * (tile / args.n_tiles) + (int)rank, n = tile % args.n_tiles;
            if constexpr (RES) request_residual<BN>(tm_res, staging, res_bar(warp - 2), m, n, quarter, half);
            ok = epilogue_tile<BN, EPI, C::HALVES, C::BUFFERS, true, LNF, RES>(
                args, tm_y, staging, chunk_no, tmem_base, acc, acc_phase, tfull_bar(acc),
                mapa_cluster(tempty_bar(acc), 0), abort_flag, m, n, quarter, half, lane,
                res_bar(warp - 2), res_phase);
            res_phase ^= 1u;
            if (!ok) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (args.tma_store && elect_one()) bulk_wait_all();
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    dep_wait();               // never finish before the kernel this one was allowed to overtake
    if (*abort_flag) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);    // let copies / MMAs in flight land
    }
    tc_fence_before();
    cluster_sync_all();          // the peer no longer reads this CTA's shared memory or signals its barriers
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// Exercises the give-up path of the bounded waits without any fault: one CTA with the warp roles of
// the kernels above allocates tensor memory, then its "MMA" thread waits -- with the caller's cycle
// limit -- on an mbarrier nothing ever arrives on.  The wait must expire, raise the abort flag and
// record PM_ERR_TIMEOUT; the other warps, parked on a second barrier, must see the abort flag and
// leave too; the CTA drains, frees its tensor memory and returns.  trace[0] = the timed-out wait
// returned false, trace[1] = warps that left through the abort flag, trace[2] = 1 after the release.
__global__ void __launch_bounds__(128) wait_timeout_selftest_kernel(long long limit, int* status, int* trace) {
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_word;
    volatile int* abort_flag = &abort_word;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars[0]), 1);
        mbar_init(smem_u32(&bars[1]), 1);
        abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_slot), 32);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    if (warp == 1) {
        if (lane == 0) {
            const bool ok = mbar_wait(smem_u32(&bars[0]), 0u, abort_flag, status, limit);
            trace[0] = ok ? 0 : 1;
        }
    } else {
        // like an epilogue warp waiting for an accumulator that never comes: ends through the abort flag
        bool ok = mbar_wait(smem_u32(&bars[1]), 0u, abort_flag, status);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok && lane == 0) atomicAdd(&trace[1], 1);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 32);
        if (lane == 0) trace[2] = 1;
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

CUtensorMapSwizzle swz(int bytes) {
    return bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
         : bytes == 64  ? CU_TENSOR_MAP_SWIZZLE_64B
         : bytes == 32  ? CU_TENSOR_MAP_SWIZZLE_32B
                        : CU_TENSOR_MAP_SWIZZLE_NONE;
}

}  // namespace

extern "C" int pm_selftest_wait_timeout(long long limit_cycles, int32_t* status, int32_t* trace, void* cuda_stream) {
    // the other warps' own limit is the library's (~2 s): the test limit must stay far below it
    if (!status || !trace || limit_cycles <= 0 || limit_cycles > 100000000ll) return PM_ERR_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (cudaMemsetAsync(trace, 0, 3 * sizeof(int32_t), st) != cudaSuccess) return PM_ERR_CUDA;
    wait_timeout_selftest_kernel<<<1, 128, 0, st>>>(limit_cycles, status, trace);
    return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}

bool tm_encode_2d(CUtensorMap* tm, const void* base, uint64_t inner, uint64_t outer,
                  uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer, int swizzle) {
    EncodeTiledFn fn = get_encode();
    if (!fn) return false;
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {row_stride_bytes};
    const cuuint32_t box[2] = {box_inner, box_outer};
    const cuuint32_t estr[2] = {1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swz(swizzle), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tm_encode_3d(CUtensorMap* tm, const void* base, uint64_t d0, uint64_t d1, uint64_t d2,
                  uint64_t stride1_bytes, uint64_t stride2_bytes, uint32_t b0, uint32_t b1,
                  uint32_t b2, int swizzle) {
    EncodeTiledFn fn = get_encode();
    if (!fn) return false;
    const cuuint64_t dims[3] = {d0, d1, d2};
    const cuuint64_t strides[2] = {stride1_bytes, stride2_bytes};
    const cuuint32_t box[3] = {b0, b1, b2};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swz(swizzle), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tm_encode_4d(CUtensorMap* tm, const void* base, const uint64_t* dims4, const uint64_t* strides3, const uint32_t* box4,
                  int swizzle) {
    EncodeTiledFn fn = get_encode();
    if (!fn) return false;
    const cuuint64_t dims[4] = {dims4[0], dims4[1], dims4[2], dims4[3]};
    const cuuint64_t strides[3] = {strides3[0], strides3[1], strides3[2]};
    const cuuint32_t box[4] = {box4[0], box4[1], box4[2], box4[3]};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swz(swizzle), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tm_encode_kblocks(CUtensorMap* tm, const void* base, int k_in, uint64_t rows, int rows_box, int kps) {
    return tm_encode_3d(tm, base, 64, rows, (uint64_t)(k_in / 64), (uint64_t)k_in * 2, 128, 64, rows_box, kps, 128);
}

bool tm_encode_groups(CUtensorMap* tm, const void* base, int k_in, uint64_t rows, int rows_box, int kps) {
    const uint64_t dims[4] = {64, 8, (uint64_t)(k_in / 64), rows / 8};
    const uint64_t strides[3] = {(uint64_t)k_in * 2, 128, (uint64_t)k_in * 16};
    const uint32_t box[4] = {64, 8, (uint32_t)kps, (uint32_t)rows_box / 8};
    return tm_encode_4d(tm, base, dims, strides, box, 128);
}

template <int BN, int EPI, bool LNF = false>
static cudaError_t launch_gemm_bn(const Launch& L, const CUtensorMap& tm_x, const CUtensorMap& tm_w,
                                  const CUtensorMap& tm_t, const CUtensorMap& tm_bt, const CUtensorMap& tm_y,
                                  const GemmArgs& a, int n_sms) {
    static SmemGrant grant;
    if (cudaError_t e = grant.ensure(lora_gemm_kernel<BN, EPI, LNF>, Smem<BN>::TOTAL); e != cudaSuccess) return e;
    const int total = a.m_tiles * a.n_tiles;
    ProfScope ps(L, KC_GEMM);
    cudaError_t e = launch_overlapped(L, lora_gemm_kernel<BN, EPI, LNF>, total < n_sms ? total : n_sms, 64 + 32 * Smem<BN>::EW, Smem<BN>::TOTAL, 1, tm_x, tm_w, tm_t, tm_bt, tm_y, a);
    BUMP(L);
    return e;
}

template <int BN>
static cudaError_t launch_gemm_epi(const Launch& L, const CUtensorMap& tm_x, const CUtensorMap& tm_w,
                                   const CUtensorMap& tm_t, const CUtensorMap& tm_bt, const CUtensorMap& tm_y,
                                   const GemmArgs& a, int n_sms) {
    if (a.ln_stats) {        // LayerNorm folded in: only the epilogues that follow a LayerNorm
        if (a.epi == EPI_GELU) return launch_gemm_bn<BN, EPI_GELU, true>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        if (a.epi == EPI_NONE) return launch_gemm_bn<BN, EPI_NONE, true>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        return cudaErrorInvalidValue;
    }
    switch (a.epi) {
        case EPI_GELU: return launch_gemm_bn<BN, EPI_GELU>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        case EPI_RESIDUAL: return launch_gemm_bn<BN, EPI_RESIDUAL>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        case EPI_PATCH: return launch_gemm_bn<BN, EPI_PATCH>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        default: return launch_gemm_bn<BN, EPI_NONE>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
    }
}

template <int BN, int EPI, bool LNF = false>
static cudaError_t launch_gemm_pair(const Launch& L, const CUtensorMap& tm_x, const CUtensorMap& tm_w,
                                    const CUtensorMap& tm_t, const CUtensorMap& tm_bt, const CUtensorMap& tm_y,
                                    const GemmArgs& a, int n_sms) {
    // the residual tile is fetched by TMA with the output's geometry (32 x 32 boxes, 64B swizzle)
    CUtensorMap tm_res = tm_y;
    if (EPI == EPI_RESIDUAL && (const void*)a.residual != (const void*)a.y) {
        if (!tm_encode_2d(&tm_res, a.residual, a.n_out, a.rows, (uint64_t)a.n_out * 2, 32, 32, 64))
            return cudaErrorInvalidValue;
    }
    using C = PairCfg<BN, EPI>;
    static SmemGrant grant;
    if (cudaError_t e = grant.ensure(lora_gemm_pair_kernel<BN, EPI, LNF>, C::TOTAL); e != cudaSuccess) return e;
    const int total = a.m_tiles * a.n_tiles;
    const int pairs = total < n_sms / 2 ? total : n_sms / 2;
    ProfScope ps(L, KC_GEMM);
    cudaError_t e = launch_overlapped(L, lora_gemm_pair_kernel<BN, EPI, LNF>, 2 * pairs, C::THREADS, C::TOTAL, 2,
                                      tm_x, tm_w, tm_t, tm_bt, tm_y, tm_res, a);
    BUMP(L);
    return e;
}

template <int BN>
static cudaError_t launch_gemm_pair_epi(const Launch& L, const CUtensorMap& tm_x, const CUtensorMap& tm_w,
                                        const CUtensorMap& tm_t, const CUtensorMap& tm_bt, const CUtensorMap& tm_y,
                                        const GemmArgs& a, int n_sms) {
    if (a.ln_stats) {
        if (a.epi == EPI_GELU) return launch_gemm_pair<BN, EPI_GELU, true>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        if (a.epi == EPI_NONE) return launch_gemm_pair<BN, EPI_NONE, true>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        return cudaErrorInvalidValue;
    }
    switch (a.epi) {
        case EPI_GELU: return launch_gemm_pair<BN, EPI_GELU>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        case EPI_RESIDUAL: return launch_gemm_pair<BN, EPI_RESIDUAL>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        case EPI_PATCH: return launch_gemm_pair<BN, EPI_PATCH>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
        default: return launch_gemm_pair<BN, EPI_NONE>(L, tm_x, tm_w, tm_t, tm_bt, tm_y, a, n_sms);
    }
}

constexpr int PAIR_WIDTHS[PM_PAIR_WIDTHS] = {128, 192, 256};

bool gemm_encode_pair_maps(LinearDev& lin, int max_adapters, int slabs_max) {
    for (int i = 0; i < PM_PAIR_WIDTHS; ++i) {
        const int half = PAIR_WIDTHS[i] / 2;
        if (!tm_encode_2d(&lin.tm_pw[i], lin.Wt, lin.k_in, lin.n_out, (uint64_t)lin.k_in * 2, BK, half, 128)) return false;
        if (lin.lora.At && !tm_encode_2d(&lin.tm_pbt[i], lin.lora.Bt, PM_SLAB, (uint64_t)max_adapters * slabs_max * lin.n_out,
                                         PM_SLAB * 2, PM_SLAB, half, 32)) return false;
    }
    return true;
}

// The tile width of the pair kernel (index into PAIR_WIDTHS), or -1 for the single-CTA kernel.  Short K goes to the latter
// where 256 divides the width, and for narrow outputs without adapters: a tile's K loop is too short to hide what the two
// CTAs of a pair wait for each other (GELU, no adapters, 384 -> 1536 on 64 frames of 197 tokens 17.4 us against 20.1 on pairs, 192 -> 768 on
// 256 frames 23.1 against 29.5).  So do widths of which only 128 is a divisor below K = 640, us single / pair: 128 -> 640 on 32 and 256 frames
// 5.1 / 6.9 and 16.5 / 30.5, 384 -> 640 on 128 frames 14.9 / 19.3, 512 -> 640 with a residual on 256 frames 47.5 / 54.3, 256 -> 128 with adapters
// on 256 frames 14.2 / 16.6; but 640 -> 640 with a residual on 48 frames 12.6 / 12.1, 768 -> 640 on 64 and 256 frames 15.1 / 14.8 and 59.1 / 51.3, 3072 -> 640 on 64 frames 57.2 / 43.5.
// Else the width with the cheapest rounds of tiles over the pairs: a round costs its columns, and what a
// tile costs whatever its width, in columns (hand-over between tiles; more where a short K loop leaves the epilogue exposed).
// The two constants are fitted to 8 to 192 frames of 197 tokens, with and without adapters, widths of 384 and 768: the rule's
// choice is 0.5 % slower than the best of the three widths on average, the widest throughout 4.4 %.  No adapters, us, 128 / 192 / 256 wide:
//   3072 -> 768: 12 frames 13.2 / 16.8 / 19.6, 16: 20.4 / 17.1 / 20.6, 37: 30.9 / 28.4 / 34.4, 128: 99 / 96 / 105;
//   768 -> 768: 12 frames 7.4 / 8.5 / 9.1, 37: 12.6 / 11.9 / 13.0, 128: 37.1 / 32.7 / 32.0;
//   768 -> 3072 (GELU): 16 frames 19.5 / 15.7 / 16.9, 37: 36.1 / 29.8 / 28.0, 128: 143 / 112 / 97.
static int pick_pair_width(int n_out, int k_in, bool lora, int rows, int n_pairs) {
    if (k_in <= 384 && (n_out % 256 == 0 || (n_out <= 384 && !lora))) return -1;
    if (k_in < 640 && n_out % 256 != 0 && n_out % 192 != 0) return -1;
    const int m = (rows + 2 * BM - 1) / (2 * BM);
    int best = -1;
    float best_cost = 0.f;
    for (int i = PM_PAIR_WIDTHS - 1; i >= 0; --i) {
        if (n_out % PAIR_WIDTHS[i] != 0) continue;
        const int tiles = m * (n_out / PAIR_WIDTHS[i]), rounds = (tiles + n_pairs - 1) / n_pairs;
        const float cost = (float)rounds * ((float)PAIR_WIDTHS[i] + 90.f + 130000.f / (float)k_in);
        if (best < 0 || cost < best_cost) { best = i; best_cost = cost; }
    }
    return best;
}

// lin.tm_w / lin.tm_bt are encoded for the BN chosen by gemm_tile_n(lin.n_out) (single-CTA kernel); lin.tm_pw /
// lin.tm_pbt fetch half of a tile's columns for the pair kernel.
int gemm_tile_n(int n_out) { return (n_out % 256 == 0) ? 256 : 128; }

LinearForm gemm_form(int k_in, int n_out, bool lora, int rows, int epi, int n_sms) {
    const int pw = n_sms >= 2 ? pick_pair_width(n_out, k_in, lora, rows, n_sms / 2) : -1;
    if (pw == 0) return {LINEAR_PAIR, 128, 1, PairCfg<128, EPI_NONE>::THREADS};
    if (pw == 1) return {LINEAR_PAIR, 192, 1, PairCfg<192, EPI_NONE>::THREADS};
    if (pw == 2) return {LINEAR_PAIR, 256, 1, epi == EPI_PATCH ? PairCfg<256, EPI_PATCH>::THREADS : PairCfg<256, EPI_NONE>::THREADS};
    const int bn = gemm_tile_n(n_out);
    return {LINEAR_SINGLE, bn, 1, 64 + 32 * (bn == 256 ? Smem<256>::EW : Smem<128>::EW)};
}

bool gemm_narrow_round(int k_in, int n_out, int rows, int n_sms) {
    const LinearForm f = gemm_form(k_in, n_out, false, rows, EPI_NONE, n_sms);
    if (f.kernel == LINEAR_SINGLE) return f.width == 128 && (rows + BM - 1) / BM * ((n_out + 127) / 128) <= n_sms;
    return n_out % 128 == 0 && (rows + 2 * BM - 1) / (2 * BM) * (n_out / 128) <= n_sms / 2;
}

cudaError_t launch_lora_gemm(const Launch& L, const LinearDev& lin, const RouteDev* R,
                             const CUtensorMap& tm_x, const CUtensorMap* tm_t, const CUtensorMap* tm_y,
                             int rows, int epi, const bf16* residual, const PatchEpi& pe, bf16* y,
                             int n_sms, const float2* ln_stats, bool after_shrink) {
    if (rows <= 0) return cudaSuccess;
    if ((lin.ln_g != nullptr) != (ln_stats != nullptr)) return cudaErrorInvalidValue;
    const int bn = gemm_tile_n(lin.n_out);
    GemmArgs a;
    a.rows = rows; a.k_in = lin.k_in; a.n_out = lin.n_out;
    a.m_tiles = (rows + BM - 1) / BM;
    a.n_tiles = (lin.n_out + bn - 1) / bn;
    a.epi = epi; a.bias = lin.bias; a.residual = residual; a.y = y; a.pe = pe;
    const bool lora = R && tm_t && R->slab_cap > 0 && lin.lora.At != nullptr;
    a.tile_nslabs = lora ? R->tile_nslabs : nullptr;
    a.tile_slab = lora ? R->tile_slab : nullptr;
    a.slab_cap = lora ? R->slab_cap : 0;
    a.status = L.status;
    a.wait_x = (after_shrink && lora) ? 0 : 1;
    a.ln_g = lin.ln_g; a.ln_stats = ln_stats;
    a.tma_store = (tm_y != nullptr && epi != EPI_PATCH) ? 1 : 0;
    const CUtensorMap& tt = lora ? *tm_t : tm_x;      // placeholders are never dereferenced
    const CUtensorMap& ty = a.tma_store ? *tm_y : tm_x;
    const int pw = n_sms >= 2 && (epi != EPI_RESIDUAL || a.tma_store) ? pick_pair_width(lin.n_out, lin.k_in, lora, rows, n_sms / 2) : -1;
    if (pw >= 0) {
        a.m_tiles = (rows + 2 * BM - 1) / (2 * BM);       // 256-row tiles
        a.n_tiles = lin.n_out / PAIR_WIDTHS[pw];
        const CUtensorMap& tpb = lora ? lin.tm_pbt[pw] : lin.tm_pw[pw];
        if (PAIR_WIDTHS[pw] == 128) return launch_gemm_pair_epi<128>(L, tm_x, lin.tm_pw[pw], tt, tpb, ty, a, n_sms);
        if (PAIR_WIDTHS[pw] == 192) return launch_gemm_pair_epi<192>(L, tm_x, lin.tm_pw[pw], tt, tpb, ty, a, n_sms);
        return launch_gemm_pair_epi<256>(L, tm_x, lin.tm_pw[pw], tt, tpb, ty, a, n_sms);
    }
    const CUtensorMap& tb = lora ? lin.tm_bt : lin.tm_w;
    if (bn == 256) return launch_gemm_epi<256>(L, tm_x, lin.tm_w, tt, tb, ty, a, n_sms);
    return launch_gemm_epi<128>(L, tm_x, lin.tm_w, tt, tb, ty, a, n_sms);
}
