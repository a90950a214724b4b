// Attention of the bf16 build: softmax(q k^T / 8) v per (frame, head), head dim 64.
//
// Four kernels.  The two that serve the model shapes, attention_pipe_kernel (one key block, up to
// 208 tokens: persistent, two query tiles in flight; attention_few_kernel for a few pairs) and attention_tc_kernel (up to 624 tokens, several
// key blocks), run both contractions on the tcgen05 tensor cores with scores and probabilities in
// tensor memory; they are described where they are defined.  attention_mma_kernel is the
// register-level kernel for sequences beyond 624 tokens:
//
// One CTA owns one (frame, head) (or a slice of its query rows when there are more than 256):
// K and V of the head are staged once in shared memory (16-byte chunks XOR-swizzled by row so
// that ldmatrix is conflict-free), each warp owns 16 query rows and walks the keys in blocks of
// 64 with an online softmax in fp32; both contractions run on the tensor cores
// (mma.sync m16n8k16, bf16 in, fp32 accumulate).  Key blocks are trimmed to the 8-key tile, so
// 197 tokens cost 200 key columns, not 256.
#include <algorithm>

#include "common.cuh"
#include "f32x2.cuh"
#include "tcgen05_ptx.cuh"

#define BUMP(L) do { if ((L).launches) ++*(L).launches; } while (0)

namespace {

constexpr int HD = 64;               // head dim
constexpr int KB = 64;               // keys per online-softmax block

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

// grid (q_slices, frames*heads); block = warps*32; dynamic smem = 2 * tpad * 128 bytes
__global__ void __launch_bounds__(512) attention_mma_kernel(const bf16* __restrict__ qkv, bf16* __restrict__ out,
                                                            int tokens, int heads, int tpad, int rows_per_cta) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int f = blockIdx.y / heads, h = blockIdx.y % heads;
    const int d = heads * HD;
    const size_t row0 = (size_t)f * tokens;
    const bf16* base = qkv + row0 * 3 * d + h * HD;
    uint8_t* Ks = smem;
    uint8_t* Vs = smem + (size_t)tpad * 128;
    // ---- stage K and V: chunk c of row r lives at r*128 + ((c ^ (r & 7)) * 16); rows >= tokens are 0
    for (int i = threadIdx.x; i < tpad * 16; i += blockDim.x) {
        const int r = i >> 4, c = i & 7, isv = (i >> 3) & 1;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < tokens) v = *reinterpret_cast<const uint4*>(base + (size_t)r * 3 * d + (1 + isv) * d + c * 8);
        *reinterpret_cast<uint4*>((isv ? Vs : Ks) + r * 128 + ((c ^ (r & 7)) << 4)) = v;
    }
    __syncthreads();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int q0 = blockIdx.x * rows_per_cta + warp * 16;
    if (q0 >= tokens) return;
    // ---- Q fragments (A operand), straight from global memory
    uint32_t qa[4][4];
    {
        const int r_lo = q0 + g, r_hi = q0 + g + 8;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const int c = ks * 16 + 2 * t;
            qa[ks][0] = r_lo < tokens ? *reinterpret_cast<const uint32_t*>(base + (size_t)r_lo * 3 * d + c) : 0u;
            qa[ks][1] = r_hi < tokens ? *reinterpret_cast<const uint32_t*>(base + (size_t)r_hi * 3 * d + c) : 0u;
            qa[ks][2] = r_lo < tokens ? *reinterpret_cast<const uint32_t*>(base + (size_t)r_lo * 3 * d + c + 8) : 0u;
            qa[ks][3] = r_hi < tokens ? *reinterpret_cast<const uint32_t*>(base + (size_t)r_hi * 3 * d + c + 8) : 0u;
        }
    }
    const uint32_t ks_addr = (uint32_t)__cvta_generic_to_shared(Ks);
    const uint32_t vs_addr = (uint32_t)__cvta_generic_to_shared(Vs);
    const float sl2 = 0.125f * 1.4426950408889634f;       // 1/sqrt(64) * log2(e)
    float o[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;

    for (int k0 = 0; k0 < tokens; k0 += KB) {
        const int valid = min(KB, tokens - k0);
        const int nt16 = (valid + 15) >> 4;            // 16-key groups in this block
        float s[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) { s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f; }
        // S = Q K^T
#pragma unroll
        for (int j = 0; j < 4; ++j) {                  // pairs of 8-key tiles
            if (j < nt16) {
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const int mi = lane >> 3;
                    const int r = k0 + j * 16 + (mi >> 1) * 8 + (lane & 7);
                    const int c = ks * 2 + (mi & 1);
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4(ks_addr + r * 128 + ((c ^ (r & 7)) << 4), b0, b1, b2, b3);
                    mma_bf16(s[2 * j], qa[ks], b0, b1);
                    mma_bf16(s[2 * j + 1], qa[ks], b2, b3);
                }
            }
        }
        // scale, mask, online softmax
        float bm_lo = -INFINITY, bm_hi = -INFINITY;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int key = k0 + i * 8 + 2 * t;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool ok = (key + (e & 1)) < tokens && (i >> 1) < nt16;
                s[i][e] = ok ? s[i][e] * sl2 : -INFINITY;
            }
            bm_lo = fmaxf(bm_lo, fmaxf(s[i][0], s[i][1]));
            bm_hi = fmaxf(bm_hi, fmaxf(s[i][2], s[i][3]));
        }
        bm_lo = fmaxf(bm_lo, __shfl_xor_sync(0xFFFFFFFFu, bm_lo, 1));
        bm_lo = fmaxf(bm_lo, __shfl_xor_sync(0xFFFFFFFFu, bm_lo, 2));
        bm_hi = fmaxf(bm_hi, __shfl_xor_sync(0xFFFFFFFFu, bm_hi, 1));
        bm_hi = fmaxf(bm_hi, __shfl_xor_sync(0xFFFFFFFFu, bm_hi, 2));
        const float nm_lo = fmaxf(m_lo, bm_lo), nm_hi = fmaxf(m_hi, bm_hi);   // finite: key k0 is valid
        const float cf_lo = exp2f(m_lo - nm_lo), cf_hi = exp2f(m_hi - nm_hi);
        m_lo = nm_lo; m_hi = nm_hi;
        float rs_lo = 0.f, rs_hi = 0.f;
        uint32_t pa[4][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float p0 = exp2f(s[i][0] - nm_lo), p1 = exp2f(s[i][1] - nm_lo);
            const float p2 = exp2f(s[i][2] - nm_hi), p3 = exp2f(s[i][3] - nm_hi);
            rs_lo += p0 + p1;
            rs_hi += p2 + p3;
            pa[i >> 1][(i & 1) * 2 + 0] = pack2(p0, p1);
            pa[i >> 1][(i & 1) * 2 + 1] = pack2(p2, p3);
        }
        l_lo = l_lo * cf_lo + rs_lo;
        l_hi = l_hi * cf_hi + rs_hi;
#pragma unroll
        for (int i = 0; i < 8; ++i) { o[i][0] *= cf_lo; o[i][1] *= cf_lo; o[i][2] *= cf_hi; o[i][3] *= cf_hi; }
        // O += P V
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {               // 16-key steps
            if (kk < nt16) {
#pragma unroll
                for (int n = 0; n < 4; ++n) {          // pairs of 8-dim tiles
                    const int mi = lane >> 3;
                    const int r = k0 + kk * 16 + (mi & 1) * 8 + (lane & 7);
                    const int c = n * 2 + (mi >> 1);
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4_t(vs_addr + r * 128 + ((c ^ (r & 7)) << 4), b0, b1, b2, b3);
                    mma_bf16(o[2 * n], pa[kk], b0, b1);
                    mma_bf16(o[2 * n + 1], pa[kk], b2, b3);
                }
            }
        }
    }
    // row sums live in the 4 threads of a quad
    l_lo += __shfl_xor_sync(0xFFFFFFFFu, l_lo, 1);
    l_lo += __shfl_xor_sync(0xFFFFFFFFu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xFFFFFFFFu, l_hi, 1);
    l_hi += __shfl_xor_sync(0xFFFFFFFFu, l_hi, 2);
    const float inv_lo = 1.f / l_lo, inv_hi = 1.f / l_hi;
    const int r_lo = q0 + g, r_hi = q0 + g + 8;
    bf16* obase = out + row0 * d + h * HD;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int c = i * 8 + 2 * t;
        if (r_lo < tokens) *reinterpret_cast<uint32_t*>(obase + (size_t)r_lo * d + c) = pack2(o[i][0] * inv_lo, o[i][1] * inv_lo);
        if (r_hi < tokens) *reinterpret_cast<uint32_t*>(obase + (size_t)r_hi * d + c) = pack2(o[i][2] * inv_hi, o[i][3] * inv_hi);
    }
}
// ---------------------------------------------------------------------------------------
// tcgen05 attention.  K and V of a (frame, head) pair are brought in by TMA (128B swizzle), the query rows are taken
// 128 at a time:
//     S = Q K^T            UMMA 128 x nb x 16, four K steps, fp32 scores in tensor memory
//     P = exp2(c (S - m))  one score row per thread (tcgen05.ld), written back over S as packed bf16 (tcgen05.st),
//                          row sums kept in registers; m: see score_reference
//     O = P V              UMMA 128 x 64 x 16 with the A operand read from tensor memory and V as
//                          an MN-major shared-memory operand, one K step per 16 keys
//     out = O / rowsum     tcgen05.ld, bf16, straight to global memory
// Keys come in blocks of up to 208 (13 x 16).  attention_tc_kernel serves several key blocks: every block's scores are
// formed once and taken relative to the row's first 16 scores, so O is never rescaled and no pass for the maxima is
// needed.  One CTA per SM walks a contiguous range of (pair, query tile) units, keeping the pair's keys and values and
// fetching the next query tile ahead.  Tensor memory holds two regions of scores (208 columns each) and O behind
// them; the issuing thread forms the scores of the next step in the other region while the softmax warps sweep this
// one (per region: one mbarrier "scores formed", one "probabilities written"), and issues a block's P V product as
// soon as its probabilities are written.  ATT_SHARES softmax warps per lane quarter split the key columns of a
// block; they exchange row sums through shared memory.
// 16 frames of 577 tokens, 12 heads: 77.3 us with a pass for the maxima and a CTA per tile, 45.6 us now.
// (One key block goes to the pipelined kernel further down.)
// ---------------------------------------------------------------------------------------
constexpr int AQ = 128;                    // query rows per tile
constexpr int AKB = 208;                   // keys per score block
constexpr int ATT_SHARES = 2;              // softmax warps per lane quarter of the multi-block kernel (they split the key columns)
constexpr int ATT_THREADS = 32 + 128 * ATT_SHARES;
constexpr int AQ_BYTES = AQ * 128;
constexpr int AKB_BYTES = AKB * 128;
constexpr int ATT_MAX_BLOCKS = 3;

constexpr uint32_t ATT_O_COL = 2 * AKB;    // tensor-memory columns: two regions of scores, O behind them

struct AttnArgs {
    int tokens, heads, tpad, n_blocks, n_qtiles, n_items, n_units;      // items: (frame, head) pairs; units: their query tiles
    const bf16* qkv;
    bf16* out;
    int* status;
};

// maximum of the first `lim` of 32 score columns (all of them if lim >= 32)
template <int N, bool MASK>
__device__ __forceinline__ float chunk_max(const uint32_t* v, int lim, float m) {
    float t[4] = {m, -INFINITY, -INFINITY, -INFINITY};       // four independent chains
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float sj = __uint_as_float(v[j]);
        t[j & 3] = fmaxf(t[j & 3], (!MASK || j < lim) ? sj : -INFINITY);
    }
    return fmaxf(fmaxf(t[0], t[1]), fmaxf(t[2], t[3]));
}
__device__ __forceinline__ float ex2_approx(float x) {     // one MUFU instruction; flushes denormals
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// p_j = exp2(c s_j - mc) (0 beyond lim), packed to bf16 pairs; adds the p_j to the two halves of sum
template <int N, bool MASK>
__device__ __forceinline__ void chunk_probs(const uint32_t* v, int lim, uint64_t c2, uint64_t nmc2, uint32_t* packed, uint64_t& sum) {
    uint64_t t[2] = {sum, pk2(0.f, 0.f)};                    // independent chains
#pragma unroll
    for (int j = 0; j < N; j += 2) {
        float x0, x1;
        upk2(fma2(pk2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), c2, nmc2), x0, x1);
        float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
        if (MASK) { p0 = j < lim ? p0 : 0.f; p1 = j + 1 < lim ? p1 : 0.f; }
        t[(j >> 1) & 1] = add2(t[(j >> 1) & 1], pk2(p0, p1));
        packed[j >> 1] = pack2(p0, p1);
    }
    sum = add2(t[0], t[1]);
}

// What a row's exponentials are taken relative to: not the row's maximum but the maximum of its first 16 scores.
// Softmax does not depend on the reference as long as nothing overflows (the reference is one of the scores, so the
// largest term is at least 1), and this one needs 16 scores instead of a pass over all of them -- nor an exchange
// between the warps that share a row: each reads those 16.  A row whose sum says that a score lies more than
// about 100 / c = 550 above the reference (or is not a number) is computed again by attention_rows_exact.
__device__ __forceinline__ float score_reference(uint32_t t_s, int valid) {
    uint32_t v[16];
    tmem_ld16(t_s, v);
    tmem_ld_wait();
    return valid >= 16 ? chunk_max<16, false>(v, 16, -INFINITY) : chunk_max<16, true>(v, valid, -INFINITY);
}
constexpr float ROW_SUM_LIMIT = 1.2676506e30f;               // 2^100
// Large terms times large values may overflow O where the quotient is finite.  A row with a sum beyond this looks at its
// accumulators and is computed again if one is not finite (below it, only values beyond 2^112 could overflow).
constexpr float ROW_SUM_CHECK = 65536.f;
template <int N>
__device__ __forceinline__ bool all_finite(const uint32_t (&v)[N]) {
    uint64_t z = pk2(0.f, 0.f);
#pragma unroll
    for (int e = 0; e < N; e += 2) z = fma2(pk2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), pk2(0.f, 0.f), z);
    float lo, hi;
    upk2(z, lo, hi);
    return lo + hi == 0.f;
}

// Sweep over the score columns [0, ncols) that start at tensor-memory address t_s (ncols a multiple of 16, `valid` of
// them real), 16 at a time with the next load in flight: P (packed bf16, 8 columns per 16 scores) goes to t_p onwards
// and the row sum of this range is returned.  P of a piece is stored when the next piece has been loaded, so t_p may
// lie up to 16 columns behind t_s.
__device__ __forceinline__ float score_probs_sweep(uint32_t t_s, uint32_t t_p, int ncols, int valid, float c, float mc) {
    uint32_t va[16], vb[16];
    const uint64_t c2 = pk2(c, c), nmc2 = pk2(-mc, -mc);
    uint64_t sum = pk2(0.f, 0.f);
    auto piece = [&](const uint32_t* v, int c0) {
        const int lim = valid - c0;
        uint32_t pk[8];
        if (lim >= 16) chunk_probs<16, false>(v, 16, c2, nmc2, pk, sum);
        else chunk_probs<16, true>(v, lim, c2, nmc2, pk, sum);
        tmem_ld_wait();
        tmem_st8(t_p + (uint32_t)(c0 >> 1), pk);
    };
    tmem_ld16(t_s, va);
    tmem_ld_wait();
#pragma unroll 1
    for (int c0 = 0; c0 < ncols; c0 += 32) {
        if (c0 + 16 < ncols) tmem_ld16(t_s + (uint32_t)(c0 + 16), vb);
        piece(va, c0);
        if (c0 + 16 < ncols) {
            if (c0 + 32 < ncols) tmem_ld16(t_s + (uint32_t)(c0 + 32), va);
            piece(vb, c0 + 16);
        }
    }
    float lo, hi;
    upk2(sum, lo, hi);
    return lo + hi;
}

// The same sweep over `np` pieces of 16 columns, `valid` of the columns real (only
// the last piece may have others): P (packed bf16, 8 columns per piece) goes to t_p onwards and the row sum of this
// range is returned.  Software pipeline: while the exponentials of a piece go through the special-function unit, the
// next piece is loaded and the one before is summed, packed and stored -- with one piece after the other the warps of
// a scheduler queued for that unit together and idled together.  P of a piece is stored after the next piece has been
// loaded.  For the kernel with two softmax warps per scheduler (47.9 -> 44.7 us); with four, whose threads
// have 96 registers, it spills (86.6 -> 96.9 us).
__device__ __forceinline__ float score_probs_sweep_ahead(uint32_t t_s, uint32_t t_p, int np, int valid, float c, float mc) {
    uint32_t va[16], vb[16];
    float pa[16], pb[16];
    const uint64_t c2 = pk2(c, c), nmc2 = pk2(-mc, -mc);
    uint64_t sum0 = pk2(0.f, 0.f), sum1 = sum0;
    auto load = [&](uint32_t* v, int i) { tmem_ld16(t_s + (uint32_t)(16 * i), v); };
    auto exps = [&](const uint32_t* v, float* p) {
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            float x0, x1;
            upk2(fma2(pk2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), c2, nmc2), x0, x1);
            p[j] = ex2_approx(x0);
            p[j + 1] = ex2_approx(x1);
        }
    };
    auto finish = [&](const float* p, int i) {
        uint32_t pk[8];
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
            sum0 = add2(sum0, pk2(p[j], p[j + 1]));
            sum1 = add2(sum1, pk2(p[j + 2], p[j + 3]));
            pk[j >> 1] = pack2(p[j], p[j + 1]);
            pk[(j >> 1) + 1] = pack2(p[j + 2], p[j + 3]);
        }
        tmem_st8(t_p + (uint32_t)(8 * i), pk);
    };
    auto mask = [&](float* p, int i) {
#pragma unroll
        for (int j = 0; j < 16; ++j) p[j] = 16 * i + j < valid ? p[j] : 0.f;
    };
    auto result = [&]() {
        float a0, a1;
        upk2(add2(sum0, sum1), a0, a1);
        return a0 + a1;
    };
    load(va, 0);
    tmem_ld_wait();
    if (np == 1) {
        exps(va, pa);
        mask(pa, 0);
        finish(pa, 0);
        return result();
    }
    load(vb, 1);
    exps(va, pa);
    tmem_ld_wait();
    int i = 1;
#pragma unroll 1
    while (i + 1 < np) {                     // vb: piece i; pa: piece i - 1, not finished
        load(va, i + 1);
        exps(vb, pb);
        finish(pa, i - 1);
        tmem_ld_wait();
        ++i;
        if (i + 1 >= np) {
            exps(va, pa);
            finish(pb, i - 1);
            mask(pa, i);
            finish(pa, i);
            return result();
        }
        load(vb, i + 1);
        exps(va, pa);
        finish(pb, i - 1);
        tmem_ld_wait();
        ++i;
    }
    exps(vb, pb);
    finish(pa, i - 1);
    mask(pb, i);
    finish(pb, i);
    return result();
}

// The rows described above are computed again when the CTA's tiles are done and the operands' shared memory is free, in groups
// of 16 query rows.  (A call in the sweep's loop costs its registers: 256 frames 87 -> 130 us.)  Until then a thread notes them
// as one bit per tile of its row; the last bit stands for all further tiles.  256 frames of 197 tokens, 12 heads: 86 us
// without such rows, 156 with one row in a hundred out of range, 399 with all (row by row in the loop: 87, 1700, 35000).
__device__ __forceinline__ uint32_t redo_bit(int tile) { return 1u << min(tile, 31); }

// One group by one warp, with the rows' true (running) maxima on mma.sync.  `stage`: REDO_STAGE bytes of shared memory of
// this warp: two buffers in turn, each 16 keys and their values (16-byte chunks XOR-swizzled by row).
constexpr int REDO_STAGE = 2 * 2 * 16 * 128;
__device__ __noinline__ void attention_rows_exact(const bf16* qkv, bf16* out, int tokens, int d, int f, int h, int q0, uint32_t stage) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, mi = lane >> 3, l7 = lane & 7;
    const float c_ = 0.125f * 1.4426950408889634f;
    const bf16* base = qkv + (size_t)f * tokens * 3 * d + h * HD;
    auto fetch = [&](int k0) {                                     // 16 keys and values; keys past the end read as zero
        const uint32_t to = stage + (uint32_t)((k0 >> 4) & 1) * (REDO_STAGE / 2);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = mi + 4 * (i & 3), key = k0 + row;
            const bf16* src = base + (size_t)min(key, tokens - 1) * 3 * d + (1 + (i >> 2)) * d + l7 * 8;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(to + (uint32_t)((i >> 2) * 2048 + row * 128 + ((l7 ^ (row & 7)) << 4))), "l"(src), "r"(key < tokens ? 16 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(0);
    uint32_t qa[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int row = q0 + g + 8 * (e & 1), c = ks * 16 + 2 * t + 8 * (e >> 1);
            qa[ks][e] = row < tokens ? *reinterpret_cast<const uint32_t*>(base + (size_t)row * 3 * d + c) : 0u;
        }
    float o[8][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < tokens; k0 += 16) {
        if (k0 + 16 < tokens) {
            fetch(k0 + 16);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        const uint32_t k_s = stage + (uint32_t)((k0 >> 4) & 1) * (REDO_STAGE / 2), v_s = k_s + 2048u;
        float s[2][4] = {};
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const int r = (mi >> 1) * 8 + l7, c = ks * 2 + (mi & 1);
            uint32_t b0, b1, b2, b3;
            ldsm_x4(k_s + r * 128 + ((c ^ (r & 7)) << 4), b0, b1, b2, b3);
            mma_bf16(s[0], qa[ks], b0, b1);
            mma_bf16(s[1], qa[ks], b2, b3);
        }
        uint32_t pa[4];
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {                           // rows g, g + 8
            float x[4], nm = m[hi];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                x[e] = k0 + (e >> 1) * 8 + 2 * t + (e & 1) < tokens ? s[e >> 1][2 * hi + (e & 1)] * c_ : -INFINITY;
                nm = fmaxf(nm, x[e]);
            }
            nm = fmaxf(nm, __shfl_xor_sync(0xFFFFFFFFu, nm, 1));
            nm = fmaxf(nm, __shfl_xor_sync(0xFFFFFFFFu, nm, 2));
            const float cf = ex2_approx(m[hi] - nm);               // 0 the first time
            m[hi] = nm;
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = ex2_approx(x[e] - nm);
            l[hi] = l[hi] * cf + ((x[0] + x[1]) + (x[2] + x[3]));
            pa[hi] = pack2(x[0], x[1]);
            pa[2 + hi] = pack2(x[2], x[3]);
#pragma unroll
            for (int i = 0; i < 8; ++i) { o[i][2 * hi] *= cf; o[i][2 * hi + 1] *= cf; }
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int r = (mi & 1) * 8 + l7, c = n * 2 + (mi >> 1);
            uint32_t b0, b1, b2, b3;
            ldsm_x4_t(v_s + r * 128 + ((c ^ (r & 7)) << 4), b0, b1, b2, b3);
            mma_bf16(o[2 * n], pa, b0, b1);
            mma_bf16(o[2 * n + 1], pa, b2, b3);
        }
        __syncwarp();                                              // this buffer is fetched into again two steps on
    }
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
        float sum = l[hi];
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 1);
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 2);
        const float inv = 1.f / sum;
        const int row = q0 + g + 8 * hi;
        bf16* orow = out + ((size_t)f * tokens + row) * d + h * HD;
        if (row < tokens)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<uint32_t*>(orow + i * 8 + 2 * t) = pack2(o[i][2 * hi] * inv, o[i][2 * hi + 1] * inv);
    }
}

// Warp `me` of `warps`: every warps'th of the groups that are noted in marks[n_sets][parts][AQ rows], tile by tile (warps at work
// side by side share keys and values).  Tile i of set k is the CTA's tile c = i * n_sets + k of n_tiles, that is query tile
// c % n_qtiles of unit u0 + c / n_qtiles * step.
__device__ __noinline__ void redo_groups(const AttnArgs& args, const uint32_t* marks, int n_sets, int parts, int u0, int step, int n_tiles,
                                         int me, int warps) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const int lane = threadIdx.x & 31;
    uint32_t m = 0;                                              // lane e: 16-row group e % 8 of set e / 8
    if (lane < n_sets * 8)
        for (int i = 0; i < parts * 16; ++i) m |= marks[((lane >> 3) * parts + (i >> 4)) * AQ + (lane & 7) * 16 + (i & 15)];
    int turn = 0;
    for (int i = 0; i * n_sets < n_tiles; ++i)
        for (uint32_t groups = __ballot_sync(0xFFFFFFFFu, (m & redo_bit(i)) != 0u); groups; groups &= groups - 1) {
            const int e = __ffs((int)groups) - 1, c = i * n_sets + (e >> 3);
            if (turn++ % warps != me || c >= n_tiles) continue;
            const int u = u0 + c / args.n_qtiles * step + c % args.n_qtiles, fh = u / args.n_qtiles, q0 = u % args.n_qtiles * AQ + (e & 7) * 16;
            if (q0 < args.tokens)
                attention_rows_exact(args.qkv, args.out, args.tokens, args.heads * HD, fh / args.heads, fh % args.heads, q0,
                                     smem_u32(smem_raw) + (uint32_t)(me * REDO_STAGE));
        }
}

// Share k takes the 16-key pieces [att_first(k), att_first(k + 1)) of a key block (capped to the block's pieces) and
// leaves its P at the start of its own score columns.
__host__ __device__ constexpr int att_first(int k) { return k == 0 ? 0 : k == 1 ? 7 : 13; }

__global__ void __launch_bounds__(ATT_THREADS, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kv,
                    const __grid_constant__ AttnArgs args) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if (base & 1023u) {                       // swizzled operands need a 1024-byte aligned window
        if (threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);
        return;
    }
    // this CTA's query tiles: a contiguous range of all (pair, query tile) units, pair by pair
    const int u0 = (int)((long long)args.n_units * blockIdx.x / gridDim.x), u1 = (int)((long long)args.n_units * (blockIdx.x + 1) / gridDim.x);
    const int d = args.heads * HD;
    const int T = args.tokens;
    const int n_blocks = args.n_blocks;
    auto q_s = [&](int u) { return base + (uint32_t)((u - u0) & 1) * AQ_BYTES; };       // two query tiles in turn
    const uint32_t k_s = base + 2 * AQ_BYTES;
    const uint32_t v_s = k_s + n_blocks * AKB_BYTES;
    const uint32_t bars = v_s + n_blocks * AKB_BYTES;
    // barriers: scores of a step formed, per score region (s_bar[2]); a step's probabilities written by all softmax
    // warps (c_bar[2]); O complete (o_bar); O read out (ofree_bar); the shares' row sums exchanged (sum_bar);
    // operands landed (q_bar[2], k_bar, v_bar)
    auto s_bar = [&](uint32_t r) { return bars + 8u * r; };
    auto c_bar = [&](uint32_t r) { return bars + 16u + 8u * r; };
    const uint32_t o_bar = bars + 32, ofree_bar = bars + 40, sum_bar = bars + 48;
    auto q_bar = [&](int u) { return bars + 56u + 8u * (uint32_t)((u - u0) & 1); };
    auto k_bar = [&](int b) { return bars + 72u + 8u * (uint32_t)b; };       // key block b landed
    auto v_bar = [&](int b) { return bars + 96u + 8u * (uint32_t)b; };       // value block b landed
    uint8_t* bar_ptr = smem_raw + (bars - base);
    float* sums_base = reinterpret_cast<float*>(bar_ptr + 160);  // two tiles in turn: [share][row]
    constexpr int shares = ATT_SHARES;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bar_ptr + 128);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 136);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int b = 0; b < ATT_MAX_BLOCKS; ++b) { mbar_init(k_bar(b), 1); mbar_init(v_bar(b), 1); }
        for (uint32_t r = 0; r < 2; ++r) { mbar_init(s_bar(r), 1); mbar_init(c_bar(r), 4 * shares); mbar_init(q_bar(u0 + (int)r), 1); }
        mbar_init(o_bar, 1); mbar_init(ofree_bar, 4 * shares);
        mbar_init(sum_bar, 4 * shares);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (warp == 0) {
        tmem_alloc(smem_u32((const void*)tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t o_tmem = tmem_base + ATT_O_COL;
    uint32_t redo = 0;                                           // this thread's rows to compute again, see redo_bit
    dep_release();

    if (warp == 0) {
        if (u0 < u1 && elect_one()) {
            // ------------------------------------------------------ TMA + MMA issue
            // Steps run over all tiles: key block g % n_blocks of tile u0 + g / n_blocks.  The scores of step g + 1 are formed
            // in the other region while the softmax warps are at step g; products issued by this thread run in issue
            // order, so a region's P V product is through before the scores issued after it overwrite the region.
            const uint32_t idesc_pv = instr_desc_b_mn(HD);
            // descriptors built once; a K step adds 2 (32 B) for Q / K and 128 (2048 B) for V
            const uint64_t dk0 = smem_desc(k_s, 128), dv0 = smem_desc(v_s, 128);
            bool ok = true;
            int pair = u0 / args.n_qtiles, loads = 0;            // the pair whose keys and values are here; how often they were brought
            auto load_q = [&](int u) {
                const int fh = u / args.n_qtiles, f = fh / args.heads, h = fh % args.heads;
                mbar_expect_tx(q_bar(u), AQ_BYTES);
                tma_load_2d(q_s(u), &tm_q, h * HD, f * T + (u % args.n_qtiles) * AQ, q_bar(u));
            };
            auto load_kv = [&](int which, uint32_t to, auto bar) {             // which: 1 keys, 2 values
                const int f = pair / args.heads, h = pair % args.heads;
                for (int b = 0; b < n_blocks; ++b) {
                    mbar_expect_tx(bar(b), (uint32_t)AKB_BYTES);
                    tma_load_2d(to + b * AKB_BYTES, &tm_kv, which * d + h * HD, f * T + b * AKB, bar(b));
                }
            };
            dep_wait();                                          // everything else follows from what these loads bring
            load_q(u0);
            load_kv(1, k_s, k_bar);
            load_kv(2, v_s, v_bar);
            if (u0 + 1 < u1) load_q(u0 + 1);
            const uint32_t n_steps = (uint32_t)((u1 - u0) * n_blocks);
            auto issue_scores = [&](uint32_t g) {
                const int b = (int)g % n_blocks, u = u0 + (int)g / n_blocks;
                const uint32_t r = g & 1u;
                // the region's previous scores (step g - 2) must have been consumed
                ok = mbar_wait(c_bar(r), ((g >> 1) & 1u) ^ 1u, abort_flag, args.status);
                if (ok && b == 0) ok = mbar_wait(q_bar(u), (uint32_t)((u - u0) >> 1) & 1u, abort_flag, args.status);
                if (ok) ok = mbar_wait(k_bar(b), (uint32_t)loads & 1u, abort_flag, args.status);
                if (!ok) return;
                tc_fence_after();
                const uint32_t idesc_s = instr_desc(min(AKB, args.tpad - b * AKB));
                const uint64_t dq = smem_desc(q_s(u), 128), bo = (uint64_t)((b * AKB_BYTES) >> 4);
#pragma unroll
                for (int k = 0; k < HD / 16; ++k)
                    umma_bf16(tmem_base + r * (uint32_t)AKB, dq + 2 * k, dk0 + bo + 2 * k, idesc_s, k > 0);
                umma_commit(s_bar(r));
            };
            issue_scores(0);
            for (uint32_t g = 0; g < n_steps && ok; ++g) {
                const int b = (int)g % n_blocks, u = u0 + (int)g / n_blocks;
                const uint32_t r = g & 1u;
                const bool last = b == n_blocks - 1;
                const bool new_pair = last && g + 1 < n_steps && (u + 1) / args.n_qtiles != pair;
                if (!new_pair && g + 1 < n_steps) issue_scores(g + 1);
                // the step's probabilities are written (so its scores, the tile's last ones included, exist)
                ok = ok && mbar_wait(c_bar(r), (g >> 1) & 1u, abort_flag, args.status);
                if (ok) ok = mbar_wait(v_bar(b), (uint32_t)loads & 1u, abort_flag, args.status);
                if (!ok) break;
                tc_fence_after();
                if (last && u + 2 < u1) load_q(u + 2);           // this tile's query rows are no longer needed
                if (new_pair) { ++pair; load_kv(1, k_s, k_bar); }            // nor the pair's keys
                if (b == 0 && u > u0) {
                    // the first product of a tile overwrites O: the previous tile's must have been read out
                    ok = mbar_wait(ofree_bar, (uint32_t)(u - u0 - 1) & 1u, abort_flag, args.status);
                    if (!ok) break;
                    tc_fence_after();
                }
                const int pieces = min(AKB, args.tpad - b * AKB) / 16;
                const uint64_t bo = (uint64_t)((b * AKB_BYTES) >> 4);
                // P of piece kk sits where its share left it: the first share's from column 16 on (columns 0..15 of a tile's
                // first block are everybody's reference), the others' at the start of their own columns
                uint32_t p_col = 16;
                for (int kk = 0; kk < pieces; ++kk) {
                    if (kk == att_first(1)) p_col = (uint32_t)(kk * 16);
                    umma_bf16_ts(o_tmem, tmem_base + r * (uint32_t)AKB + p_col, dv0 + bo + 128 * kk, idesc_pv, (b > 0 || kk > 0) ? 1u : 0u);
                    p_col += 8;
                }
                if (last) umma_commit(o_bar);
                if (new_pair) {
                    ++loads;
                    // the values are free once the tile's O is complete
                    ok = mbar_wait(o_bar, (uint32_t)(u - u0) & 1u, abort_flag, args.status);
                    if (!ok) break;
                    load_kv(2, v_s, v_bar);
                    issue_scores(g + 1);
                }
            }
        }
    } else {
        // ---------------------------------------------------------- softmax + output
        const int quarter = warp & 3;                            // TMEM lanes 32*quarter .. +31
        const int share = (warp - 1) >> 2;                       // which share of the key columns
        const int row = quarter * 32 + lane;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const float c = 0.125f * 1.4426950408889634f;            // 1/sqrt(64) * log2(e)
        uint32_t g = 0;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const uint32_t par = (uint32_t)(u - u0) & 1u;
            float* sums = sums_base + par * ATT_SHARES * AQ;
            const int fh = u / args.n_qtiles, qt = u % args.n_qtiles, f = fh / args.heads, h = fh % args.heads;
            const int q_row = qt * AQ + row;
            const bool warp_active = qt * AQ + quarter * 32 < T;      // else: no row of this warp exists
            float mc = 0.f, l = 0.f;
            for (int b = 0; b < n_blocks; ++b, ++g) {
                const uint32_t r = g & 1u;
                ok = mbar_wait(s_bar(r), (g >> 1) & 1u, abort_flag, args.status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_s = t_lane + r * (uint32_t)AKB;
                // this warp's columns of key block b
                const int np = min(AKB, args.tpad - b * AKB) / 16;
                const int p0 = min(att_first(share), np), p1 = min(att_first(share + 1), np);
                if (warp_active) {
                    if (b == 0) mc = score_reference(t_s, T) * c;
                    if (p1 > p0) {
                        const uint32_t at = t_s + (uint32_t)(p0 * 16);
                        l += score_probs_sweep_ahead(at, share == 0 ? at + 16u : at, p1 - p0, T - b * AKB - p0 * 16, c, mc);
                        tmem_st_wait();
                    }
                }
                if (b == n_blocks - 1) {
                    sums[share * AQ + row] = l;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(sum_bar);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(c_bar(r));
            }
            if (!ok) break;
            ok = mbar_wait(sum_bar, par, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            l = 0.f;
#pragma unroll
            for (int k = 0; k < shares; ++k) l += sums[k * AQ + row];
            if (q_row < T && !(l < ROW_SUM_LIMIT)) redo |= redo_bit(u - u0);
            // O = sum over the key blocks of P V is complete: the finished rows are written out
            ok = mbar_wait(o_bar, par, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            // the output columns are split between the shares
            constexpr int OCOLS = HD / shares;
            uint32_t v[OCOLS];
            const bool writes = warp_active;
            if (writes) {
#pragma unroll
                for (int part = 0; part < OCOLS / 32; ++part) tmem_ld32(t_lane + ATT_O_COL + (uint32_t)(share * OCOLS + part * 32), v + part * 32);
                tmem_ld_wait();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(ofree_bar);               // O is in registers: the next tile's products may start
            if (writes) {
                const float inv = 1.f / l;
                bf16* orow = args.out + ((size_t)f * T + q_row) * d + h * HD + share * OCOLS;
                if (q_row < T && l > ROW_SUM_CHECK && !all_finite(v)) redo |= redo_bit(u - u0);
                if (q_row < T && l < ROW_SUM_LIMIT) {
                    // 32-byte stores: one full sector per row per instruction
#pragma unroll
                    for (int q = 0; q < OCOLS / 16; ++q) {
                        uint32_t o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            o[e] = pack2(__uint_as_float(v[q * 16 + 2 * e]) * inv, __uint_as_float(v[q * 16 + 2 * e + 1]) * inv);
                        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                     ::"l"(orow + q * 16), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]),
                                       "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                                     : "memory");
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
    const int any = __syncthreads_or(redo != 0u);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (any && !*abort_flag) {
        uint32_t* marks = reinterpret_cast<uint32_t*>(sums_base);
        if (warp > 0) marks[(warp - 1) / 4 * AQ + (warp & 3) * 32 + lane] = redo;
        __syncthreads();
        if (warp > 0) redo_groups(args, marks, 1, shares, u0, args.n_qtiles, u1 - u0, warp - 1, 4 * shares);
    }
}

// ---------------------------------------------------------------------------------------
// Pipelined variant for sequences of one key block (up to 208 tokens, at most two query tiles):
// one persistent CTA per SM walks (frame, head) items and keeps two query tiles in flight, each in
// its own half of tensor memory with its own group of eight softmax warps:
//     warp 0         TMA: K, V and the query tiles of item j+2 land while items j, j+1 are computed
//     warp 1         MMA issue:  S(c), then P V of tile c-1, then S(c+1), ...
//     warps 2..9     softmax + output of the even tiles (tensor-memory columns 0..255)
//     warps 10..17   the same for the odd tiles (columns 256..511)
// so the tensor pipe, the two softmax groups and the loads of the following items overlap inside one
// CTA.  Two warps share each quarter of the 128 rows (a warp reaches the tensor-memory lanes
// 32 (w mod 4) .. +31 only) and split the key columns: the first seven 16-key pieces and the rest.
// The sweeps are chains of dependent operations, so what bounds them is how many warps a scheduler can switch between
// -- four per scheduler here against two with one warp per quarter -- and how many sweeps a tile needs: one (see
// score_reference; with a sweep for the row maxima and their exchange in front of it, 256 frames of 197 tokens, 12 heads: 99.6 us, now 86.4).
// The halves exchange their row sums through shared memory (mbarriers, bounded waits).
// Column map of a tile's 256-column slot: scores 0..207; P of the first half over 16..71 (the first 16 columns stay:
// both halves read their reference there), P of the second half in 208..255 (so that it never lands on scores the
// first half still reads); O in 128..191 once both halves are done.  Tile c of a CTA is query tile c % nq of its item c / nq.
// ---------------------------------------------------------------------------------------
constexpr int APIPE_GROUP_WARPS = 8;
constexpr int APIPE_THREADS = 64 + 2 * 32 * APIPE_GROUP_WARPS;      // 576
constexpr int APIPE_ITEM_BYTES = 2 * AKB_BYTES + 2 * AQ_BYTES;      // K, V, two query tiles
constexpr int APIPE_SPLIT = 7;                                       // 16-key pieces of the first half
constexpr int APIPE_XCHG_BYTES = 2 * 2 * AQ * 4;                     // row sums [group][half][row]

__device__ __forceinline__ int pipe_items(const AttnArgs& args) {      // of this CTA: blockIdx.x, + gridDim.x, ...
    return (args.n_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
}

__global__ void __launch_bounds__(APIPE_THREADS, 1)
attention_pipe_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kv,
                      const __grid_constant__ AttnArgs args) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if (base & 1023u) {                       // swizzled operands need a 1024-byte aligned window
        if (threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);
        return;
    }
    const int T = args.tokens, nq = args.n_qtiles, d = args.heads * HD;
    const int my_items = pipe_items(args);
    const int my_tiles = my_items * nq;
    const int n_pieces = args.tpad / 16, split = min(APIPE_SPLIT, n_pieces);
    auto k_s = [&](int buf) { return base + buf * APIPE_ITEM_BYTES; };
    auto v_s = [&](int buf) { return base + buf * APIPE_ITEM_BYTES + AKB_BYTES; };
    auto q_s = [&](int buf, int qt) { return base + buf * APIPE_ITEM_BYTES + 2 * AKB_BYTES + qt * AQ_BYTES; };
    float* xchg = reinterpret_cast<float*>(smem_raw + 2 * APIPE_ITEM_BYTES);
    const uint32_t bars = base + 2 * APIPE_ITEM_BYTES + APIPE_XCHG_BYTES;
    auto kv_full = [&](int b) { return bars + 8u * b; };
    auto buf_free = [&](int b) { return bars + 16u + 8u * b; };
    auto s_ready = [&](int sl) { return bars + 32u + 8u * sl; };
    auto p_ready = [&](int sl) { return bars + 48u + 8u * sl; };
    auto o_ready = [&](int sl) { return bars + 64u + 8u * sl; };
    auto slot_free = [&](int sl) { return bars + 80u + 8u * sl; };
    auto sum_bar = [&](int sl) { return bars + 112u + 8u * sl; };
    uint8_t* bar_ptr = smem_raw + (bars - base);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bar_ptr + 128);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 136);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(kv_full(i), 1); mbar_init(buf_free(i), 1);
            mbar_init(s_ready(i), 1); mbar_init(p_ready(i), APIPE_GROUP_WARPS);
            mbar_init(o_ready(i), 1); mbar_init(slot_free(i), APIPE_GROUP_WARPS);
            mbar_init(sum_bar(i), APIPE_GROUP_WARPS);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(smem_u32((const void*)tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    uint32_t redo = 0;                                           // this thread's rows to compute again, see redo_bit
    dep_release();

    if (warp == 0) {
        if (elect_one()) {
            // ---------------------------------------------------------------- TMA producer
            bool ok = true;
            dep_wait();                            // everything else follows from what these loads bring
            for (int j = 0; j < my_items && ok; ++j) {
                const int buf = j & 1;
                // the buffer's previous item (j - 2) must be through its last P V product
                ok = mbar_wait(buf_free(buf), (((uint32_t)j >> 1) & 1u) ^ 1u, abort_flag, args.status);
                if (!ok) break;
                const int item = (int)blockIdx.x + j * (int)gridDim.x;
                const int f = item / args.heads, h = item % args.heads;
                mbar_expect_tx(kv_full(buf), (uint32_t)(2 * AKB_BYTES + nq * AQ_BYTES));
                tma_load_2d(k_s(buf), &tm_kv, d + h * HD, f * T, kv_full(buf));
                for (int qt = 0; qt < nq; ++qt) tma_load_2d(q_s(buf, qt), &tm_q, h * HD, f * T + qt * AQ, kv_full(buf));
                tma_load_2d(v_s(buf), &tm_kv, 2 * d + h * HD, f * T, kv_full(buf));
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ---------------------------------------------------------------- MMA issue
            const uint32_t idesc_s = instr_desc(args.tpad), idesc_pv = instr_desc_b_mn(HD);
            bool ok = true;
            // O(p) = P(p) V: P is the packed bf16 the two halves left in tile p's slot
            auto issue_pv = [&](int p) {
                const int slot = p & 1, buf = (p / nq) & 1;
                ok = mbar_wait(p_ready(slot), ((uint32_t)p >> 1) & 1u, abort_flag, args.status);
                if (!ok) return;
                tc_fence_after();
                const uint32_t s_tmem = tmem_base + (uint32_t)(slot * 256);
                const uint64_t dv0 = smem_desc(v_s(buf), 128);
                for (int kk = 0; kk < n_pieces; ++kk) {
                    const uint32_t p_col = kk < split ? (uint32_t)(16 + kk * 8) : (uint32_t)(208 + (kk - split) * 8);
                    umma_bf16_ts(s_tmem + 128u, s_tmem + p_col, dv0 + 128 * kk, idesc_pv, kk > 0 ? 1u : 0u);
                }
                umma_commit(o_ready(slot));
                if (p % nq == nq - 1) umma_commit(buf_free(buf));     // the item's operands are no longer read
            };
            for (int c = 0; c < my_tiles && ok; ++c) {
                const int j = c / nq, qt = c % nq, buf = j & 1, slot = c & 1;
                if (qt == 0) ok = mbar_wait(kv_full(buf), ((uint32_t)j >> 1) & 1u, abort_flag, args.status);
                // the slot's previous tile (c - 2) must have been read out
                ok = ok && mbar_wait(slot_free(slot), (((uint32_t)c >> 1) & 1u) ^ 1u, abort_flag, args.status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t dq0 = smem_desc(q_s(buf, qt), 128), dk0 = smem_desc(k_s(buf), 128);
#pragma unroll
                for (int k = 0; k < HD / 16; ++k)
                    umma_bf16(tmem_base + (uint32_t)(slot * 256), dq0 + 2 * k, dk0 + 2 * k, idesc_s, k > 0);
                umma_commit(s_ready(slot));
                if (c >= 1) issue_pv(c - 1);
            }
            if (ok && my_tiles > 0) issue_pv(my_tiles - 1);
        }
    } else {
        // -------------------------------------------------------------------- softmax + output
        const int group = (warp - 2) / APIPE_GROUP_WARPS;        // 0: even tiles, 1: odd tiles
        const int half = ((warp - 2) % APIPE_GROUP_WARPS) >> 2;  // which share of the key columns
        const int quarter = warp & 3;                            // TMEM lanes 32*quarter .. +31
        const int row = quarter * 32 + lane;                     // row of the query tile
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(group * 256);
        const int col0 = half == 0 ? 0 : split * 16;             // first key column of this warp
        const int ncols = half == 0 ? split * 16 : (n_pieces - split) * 16;
        const uint32_t t_p = t_lane + (half == 0 ? 16u : 208u);  // where this warp's P goes
        float* my_sum = xchg + (group * 2 + half) * AQ;
        float* other_sum = xchg + (group * 2 + (half ^ 1)) * AQ;
        const float c_ = 0.125f * 1.4426950408889634f;           // 1/sqrt(64) * log2(e)
        bool ok = true;
        for (int c = group; c < my_tiles && ok; c += 2) {
            const uint32_t par = ((uint32_t)c >> 1) & 1u;
            const int j = c / nq, qt = c % nq;
            const int item = (int)blockIdx.x + j * (int)gridDim.x;
            const int f = item / args.heads, h = item % args.heads;
            const int q_row = qt * AQ + row;
            const bool warp_active = qt * AQ + quarter * 32 < T;     // else: no row of this warp exists
            ok = mbar_wait(s_ready(group), par, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            float l = 0.f;
            if (warp_active) {
                const float mc = score_reference(t_lane, T) * c_;    // columns 0..15: no P is written there
                if (ncols > 0) l = score_probs_sweep(t_lane + (uint32_t)col0, t_p, ncols, T - col0, c_, mc);
                tmem_st_wait();
            }
            my_sum[row] = l;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { mbar_arrive(sum_bar(group)); mbar_arrive(p_ready(group)); }
            ok = mbar_wait(sum_bar(group), par, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            l += other_sum[row];
            if (q_row < T && !(l < ROW_SUM_LIMIT)) redo |= redo_bit(c >> 1);
            ok = mbar_wait(o_ready(group), par, abort_flag, args.status);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            if (warp_active) {
                // each half writes 32 of the 64 output columns
                const float inv = 1.f / l;
                bf16* orow = args.out + ((size_t)f * T + q_row) * d + h * HD + half * 32;
                uint32_t v[32];
                tmem_ld32((t_lane + 128u) + (uint32_t)(half * 32), v);
                tmem_ld_wait();
                if (q_row < T && l > ROW_SUM_CHECK && !all_finite(v)) redo |= redo_bit(c >> 1);
                if (q_row < T && l < ROW_SUM_LIMIT) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            o[e] = pack2(__uint_as_float(v[q * 16 + 2 * e]) * inv,
                                         __uint_as_float(v[q * 16 + 2 * e + 1]) * inv);
                        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                     ::"l"(orow + q * 16), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]),
                                       "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                                     : "memory");
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(slot_free(group));
        }
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    dep_wait();               // never finish before the kernel this one was allowed to overtake
    if (*abort_flag) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);    // let copies / MMAs in flight land
    }
    tc_fence_before();
    const int any = __syncthreads_or(redo != 0u);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (any && !*abort_flag) {
        uint32_t* marks = reinterpret_cast<uint32_t*>(xchg);
        if (warp > 1) marks[(warp - 2) / 4 * AQ + (warp & 3) * 32 + lane] = redo;
        __syncthreads();
        if (warp > 1)
            redo_groups(args, marks, 2, 2, (int)blockIdx.x * args.n_qtiles, (int)gridDim.x * args.n_qtiles, pipe_items(args) * args.n_qtiles,
                        warp - 2, 2 * APIPE_GROUP_WARPS);
    }
}

// ---------------------------------------------------------------------------------------
// Few (frame, head) pairs of one key block: one CTA per 16 query rows.  With few pairs the kernels above leave most SMs
// idle and each pair is one long chain (a sweep over the scores through tensor memory between two products); here the pair's rows
// spread over the SMs and four warps split the keys, so a warp has at most four 16-key groups: scores on
// mma.sync, softmax against the warp's own maximum in registers, P V, and the four partial results are merged
// through shared memory.  K and V arrive by TMA (128B swizzle, which is what ldmatrix wants), each on a barrier.
// 12 pairs of 197 tokens, back to back: 7.6 us with the pipelined kernel, 4.4 us; 3 pairs: 7.4 and 3.0 us.
// ---------------------------------------------------------------------------------------
constexpr int AFEW_ROWS = 16;
constexpr int AFEW_WARPS = 4;
constexpr int AFEW_GROUPS = (AKB / 16 + AFEW_WARPS - 1) / AFEW_WARPS;      // 16-key groups of a warp
constexpr int AFEW_OSTRIDE = HD + 4;                                       // floats of a partial output row

struct AttnFewSmem {
    uint8_t k[AKB_BYTES], v[AKB_BYTES];
    float o[AFEW_WARPS][AFEW_ROWS][AFEW_OSTRIDE];
    float m[AFEW_WARPS][AFEW_ROWS], l[AFEW_WARPS][AFEW_ROWS];
    uint64_t bars[2];
    int abort_flag;
};

__global__ void __launch_bounds__(32 * AFEW_WARPS)
attention_few_kernel(const __grid_constant__ CUtensorMap tm_kv, const bf16* qkv, bf16* out,
                     int tokens, int heads, int* status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    AttnFewSmem& sm = *reinterpret_cast<AttnFewSmem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int q0 = (int)blockIdx.x * AFEW_ROWS;
    const int f = blockIdx.y / heads, h = blockIdx.y % heads, d = heads * HD;
    const uint32_t k_bar = smem_u32(&sm.bars[0]), v_bar = smem_u32(&sm.bars[1]);
    const uint32_t k_s = smem_u32(sm.k), v_s = smem_u32(sm.v);
    const bool usable = (smem_u32(smem_raw) & 1023u) == 0;       // the swizzle is a function of the address
    if (threadIdx.x == 0) {
        mbar_init(k_bar, 1);
        mbar_init(v_bar, 1);
        sm.abort_flag = usable ? 0 : 1;
        if (!usable) atomicCAS(status, 0, (int)PM_ERR_CUDA);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    dep_release();
    dep_wait();
    if (threadIdx.x == 0 && usable) {
        mbar_expect_tx(k_bar, AKB_BYTES);
        tma_load_2d(k_s, &tm_kv, d + h * HD, f * tokens, k_bar);
        mbar_expect_tx(v_bar, AKB_BYTES);
        tma_load_2d(v_s, &tm_kv, 2 * d + h * HD, f * tokens, v_bar);
    }
    // Q fragments straight from global memory; rows past the end repeat the last one and are not stored
    uint32_t qa[4][4];
    const int r_lo = min(q0 + g, tokens - 1), r_hi = min(q0 + g + 8, tokens - 1);
    {
        const bf16* lo = qkv + ((size_t)f * tokens + r_lo) * 3 * d + h * HD;
        const bf16* hi = qkv + ((size_t)f * tokens + r_hi) * 3 * d + h * HD;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const int c = ks * 16 + 2 * t;
            qa[ks][0] = *reinterpret_cast<const uint32_t*>(lo + c);
            qa[ks][1] = *reinterpret_cast<const uint32_t*>(hi + c);
            qa[ks][2] = *reinterpret_cast<const uint32_t*>(lo + c + 8);
            qa[ks][3] = *reinterpret_cast<const uint32_t*>(hi + c + 8);
        }
    }
    // this warp's 16-key groups
    const int groups = (tokens + 15) / 16, g0 = groups * warp / AFEW_WARPS, g1 = groups * (warp + 1) / AFEW_WARPS;
    const float c_ = 0.125f * 1.4426950408889634f;               // 1/sqrt(64) * log2(e)
    float s[2 * AFEW_GROUPS][4];
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;
    float o[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    const int mi = lane >> 3;
    if (__all_sync(0xFFFFFFFFu, mbar_wait(k_bar, 0, &sm.abort_flag, status))) {
#pragma unroll
        for (int i = 0; i < AFEW_GROUPS; ++i) {
            float* s0 = s[2 * i];
            float* s1 = s[2 * i + 1];
#pragma unroll
            for (int e = 0; e < 4; ++e) s0[e] = s1[e] = 0.f;
            if (g0 + i < g1) {
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const int r = (g0 + i) * 16 + (mi >> 1) * 8 + (lane & 7), c = ks * 2 + (mi & 1);
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4(k_s + r * 128 + ((c ^ (r & 7)) << 4), b0, b1, b2, b3);
                    mma_bf16(s0, qa[ks], b0, b1);
                    mma_bf16(s1, qa[ks], b2, b3);
                }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int key = (g0 + i) * 16 + (e >> 2) * 8 + 2 * t + (e & 1);
                float& x = e < 4 ? s0[e] : s1[e & 3];
                x = g0 + i < g1 && key < tokens ? x * c_ : -INFINITY;
                if (e & 2) m_hi = fmaxf(m_hi, x);
                else m_lo = fmaxf(m_lo, x);
            }
        }
        m_lo = fmaxf(m_lo, __shfl_xor_sync(0xFFFFFFFFu, m_lo, 1));
        m_lo = fmaxf(m_lo, __shfl_xor_sync(0xFFFFFFFFu, m_lo, 2));
        m_hi = fmaxf(m_hi, __shfl_xor_sync(0xFFFFFFFFu, m_hi, 1));
        m_hi = fmaxf(m_hi, __shfl_xor_sync(0xFFFFFFFFu, m_hi, 2));
        // a warp without a key (fewer groups than warps) keeps -inf and contributes nothing
        const float b_lo = m_lo == -INFINITY ? 0.f : m_lo, b_hi = m_hi == -INFINITY ? 0.f : m_hi;
        uint32_t pa[AFEW_GROUPS][4];
#pragma unroll
        for (int i = 0; i < 2 * AFEW_GROUPS; ++i) {
            const float p0 = ex2_approx(s[i][0] - b_lo), p1 = ex2_approx(s[i][1] - b_lo);
            const float p2 = ex2_approx(s[i][2] - b_hi), p3 = ex2_approx(s[i][3] - b_hi);
            l_lo += p0 + p1;
            l_hi += p2 + p3;
            pa[i >> 1][(i & 1) * 2 + 0] = pack2(p0, p1);
            pa[i >> 1][(i & 1) * 2 + 1] = pack2(p2, p3);
        }
        l_lo += __shfl_xor_sync(0xFFFFFFFFu, l_lo, 1);
        l_lo += __shfl_xor_sync(0xFFFFFFFFu, l_lo, 2);
        l_hi += __shfl_xor_sync(0xFFFFFFFFu, l_hi, 1);
        l_hi += __shfl_xor_sync(0xFFFFFFFFu, l_hi, 2);
        if (__all_sync(0xFFFFFFFFu, mbar_wait(v_bar, 0, &sm.abort_flag, status))) {
#pragma unroll
            for (int i = 0; i < AFEW_GROUPS; ++i) {
                if (g0 + i >= g1) break;
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    const int r = (g0 + i) * 16 + (mi & 1) * 8 + (lane & 7), c = n * 2 + (mi >> 1);
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4_t(v_s + r * 128 + ((c ^ (r & 7)) << 4), b0, b1, b2, b3);
                    mma_bf16(o[2 * n], pa[i], b0, b1);
                    mma_bf16(o[2 * n + 1], pa[i], b2, b3);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        *reinterpret_cast<float2*>(&sm.o[warp][g][i * 8 + 2 * t]) = make_float2(o[i][0], o[i][1]);
        *reinterpret_cast<float2*>(&sm.o[warp][g + 8][i * 8 + 2 * t]) = make_float2(o[i][2], o[i][3]);
    }
    if (t == 0) {
        sm.m[warp][g] = m_lo; sm.l[warp][g] = l_lo;
        sm.m[warp][g + 8] = m_hi; sm.l[warp][g + 8] = l_hi;
    }
    __syncthreads();
    // 128 threads merge 16 rows x 64 columns: 8 columns each
    const int row = threadIdx.x >> 3, c0 = (threadIdx.x & 7) * 8;
    float m = sm.m[0][row];
#pragma unroll
    for (int w = 1; w < AFEW_WARPS; ++w) m = fmaxf(m, sm.m[w][row]);
    float l = 0.f, acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll
    for (int w = 0; w < AFEW_WARPS; ++w) {
        const float a = ex2_approx(sm.m[w][row] - m);            // 0 for a warp without keys
        l = fmaf(sm.l[w][row], a, l);
        const float4 x = *reinterpret_cast<const float4*>(&sm.o[w][row][c0]), y = *reinterpret_cast<const float4*>(&sm.o[w][row][c0 + 4]);
        acc[0] = fmaf(x.x, a, acc[0]); acc[1] = fmaf(x.y, a, acc[1]); acc[2] = fmaf(x.z, a, acc[2]); acc[3] = fmaf(x.w, a, acc[3]);
        acc[4] = fmaf(y.x, a, acc[4]); acc[5] = fmaf(y.y, a, acc[5]); acc[6] = fmaf(y.z, a, acc[6]); acc[7] = fmaf(y.w, a, acc[7]);
    }
    if (q0 + row < tokens && !sm.abort_flag) {
        const float inv = 1.f / l;
        *reinterpret_cast<uint4*>(out + ((size_t)f * tokens + q0 + row) * d + h * HD + c0) =
            make_uint4(pack2(acc[0] * inv, acc[1] * inv), pack2(acc[2] * inv, acc[3] * inv), pack2(acc[4] * inv, acc[5] * inv),
                       pack2(acc[6] * inv, acc[7] * inv));
    }
    if (*(volatile int*)&sm.abort_flag)
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);        // let copies in flight land
}

}  // namespace

bool attention_tc_supported(int tokens) { return (tokens + 15) / 16 * 16 <= ATT_MAX_BLOCKS * AKB; }

bool attention_encode_maps(const bf16* qkv, int n_frames, int tokens, int heads, CUtensorMap* tm_q,
                           CUtensorMap* tm_kv) {
    const uint64_t w = (uint64_t)3 * heads * HD, rows = (uint64_t)n_frames * tokens;
    return tm_encode_2d(tm_q, qkv, w, rows, w * 2, HD, AQ, 128) &&
           tm_encode_2d(tm_kv, qkv, w, rows, w * 2, HD, AKB, 128);
}

cudaError_t launch_attention_tc(const Launch& L, const CUtensorMap& tm_q, const CUtensorMap& tm_kv,
                                const bf16* qkv, bf16* out, int n_frames, int tokens, int heads, int n_sms) {
    if (n_frames <= 0) return cudaSuccess;
    AttnArgs a;
    a.tokens = tokens; a.heads = heads;
    a.tpad = (tokens + 15) / 16 * 16;
    a.n_blocks = (a.tpad + AKB - 1) / AKB;
    a.n_qtiles = (tokens + AQ - 1) / AQ;
    a.n_items = n_frames * heads;
    a.n_units = a.n_items * a.n_qtiles;
    a.qkv = qkv; a.out = out; a.status = L.status;
    // up to a third as many (frame, head) pairs as SMs: 12 pairs of 197 tokens 4.4 against 7.6 us, 48 pairs 7.6 against 7.7, 72
    // pairs 9.8 against 7.8; 65 tokens: 48 pairs 3.9 against 4.6, 96 pairs 5.7 against 4.8
    const int row_tiles = (tokens + AFEW_ROWS - 1) / AFEW_ROWS;
    if (a.n_blocks == 1 && 3 * n_frames * heads <= n_sms) {
        static SmemGrant grant;
        if (cudaError_t e = grant.ensure(attention_few_kernel, (int)sizeof(AttnFewSmem)); e != cudaSuccess) return e;
        ProfScope ps(L, KC_ATTENTION);
        cudaError_t e = launch_overlapped(L, attention_few_kernel, dim3(row_tiles, n_frames * heads), 32 * AFEW_WARPS, sizeof(AttnFewSmem), 1,
                                          tm_kv, qkv, out, tokens, heads, L.status);
        BUMP(L);
        return e;
    }
    if (a.n_blocks == 1 && a.n_qtiles <= 2 && n_sms > 0) {
        // one key block: the pipelined persistent kernel
        const size_t psmem = 2 * (size_t)APIPE_ITEM_BYTES + APIPE_XCHG_BYTES + 192;
        static SmemGrant grant;
        if (cudaError_t e = grant.ensure(attention_pipe_kernel, (int)psmem); e != cudaSuccess) return e;
        ProfScope ps(L, KC_ATTENTION);
        cudaError_t e = launch_overlapped(L, attention_pipe_kernel, std::min(a.n_items, n_sms), APIPE_THREADS, psmem, 1, tm_q, tm_kv, a);
        BUMP(L);
        return e;
    }
    // all of tensor memory and most of the shared memory: one CTA per SM
    const size_t smem = 2 * (size_t)AQ_BYTES + (size_t)a.n_blocks * 2 * AKB_BYTES + 160 + 2 * ATT_SHARES * AQ * sizeof(float);
    static SmemGrant grant;
    if (cudaError_t e = grant.ensure(attention_tc_kernel, (int)smem); e != cudaSuccess) return e;
    ProfScope ps(L, KC_ATTENTION);
    cudaError_t e = launch_overlapped(L, attention_tc_kernel, n_sms > 0 ? std::min(a.n_units, n_sms) : a.n_units, ATT_THREADS,
                                      smem, 1, tm_q, tm_kv, a);
    BUMP(L);
    return e;
}

cudaError_t launch_attention_mma(const Launch& L, const bf16* qkv, bf16* out, int n_frames, int tokens,
                                 int heads) {
    if (n_frames <= 0) return cudaSuccess;
    const int groups = (tokens + 15) / 16;
    const int slices = (groups + 15) / 16;
    const int warps = (groups + slices - 1) / slices;
    const int tpad = groups * 16;
    const size_t smem = (size_t)tpad * 256;
    if (smem > 227 * 1024) return launch_attention_simple<bf16>(L, qkv, out, n_frames, tokens, heads);
    static SmemGrant grant;
    if (cudaError_t e = grant.ensure(attention_mma_kernel, (int)smem); e != cudaSuccess) return e;
    ProfScope ps(L, KC_ATTENTION);
    dim3 grid(slices, n_frames * heads);
    attention_mma_kernel<<<grid, warps * 32, smem, L.st>>>(qkv, out, tokens, heads, tpad, warps * 16);
    BUMP(L);
    return cudaGetLastError();
}
