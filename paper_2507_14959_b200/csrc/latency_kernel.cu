// Whole-network kernel for a handful of frames (the single-stream operating point of Sec. 4): patch
// embedding, all encoder blocks with their unmerged LoRA terms (Sec. 3.1), final LayerNorm, base and
// adapter heads with sigmoid and merge (Fig. 5b) in ONE launch.
//
// Everything in a ViT block except attention is local to a token row, so a CTA owns 16 token rows of one
// frame from the first layer to the last and keeps their residual stream (fp32) and every intermediate in
// shared memory.  What a CTA reads from L2 is static -- weights, LoRA slabs, bias vectors, in an order that
// is known when the kernel starts -- so one producer thread walks that order and keeps a ring of 32 KB
// shared-memory slots full by TMA, across the boundaries of linears and blocks, while the eight consumer
// warps multiply what has landed (full / empty transaction barriers per slot, no CTA-wide barrier in the
// stream).  Every CTA reads every weight, 13 CTAs per frame.
// The one exchange per block is attention: each CTA publishes the keys and values of its rows (two global
// buffers used in turn) as soon as those columns of the qkv product are done, counts itself in at the
// frame's counter and goes on with the query columns; a second producer thread waits for the counter
// (bounded) and fetches the heads' keys and values, the next head's while this one is computed.  Each CTA
// attends from its 16 query rows to all keys of its frame: four warp pairs split the keys, the two warps
// of a pair split the head dimension, partial softmax results are merged through shared memory.
// What bounds a whole tile per CTA is the instruction chain of eight warps, not the weights (a third of what an SM can draw
// from L2), so while the batch leaves SMs idle a cluster with one CTA per head shares each tile: a CTA computes its
// head's queries, keys and values, attends for that head, and computes its part of the outputs of every other linear;
// rows it finishes go, rounded, to the same place in every CTA of the cluster (distributed shared memory), four
// exchanges per block on mbarriers that count the bytes (bounded waits).  DeiT-tiny, one CTA per tile -> one per
// head: one frame 299 -> 172 us (no adapter), 314 -> 185 (three), three frames 316 -> 184; from the fourth frame on
// the clusters do not fit 148 SMs.
// Contractions run on mma.sync m16n8k16 (bf16 in, fp32 accumulate): with 16 rows per CTA there is no
// 128-row tile to give to tcgen05.
// LayerNorm uses the folded form the other kernels use: y = rstd (x W' - mean g) + b'.
#include "common.cuh"

#define BUMP(L) do { if ((L).launches) ++*(L).launches; } while (0)

namespace {

constexpr int LT_ROWS = 16;
constexpr int LT_CWARPS = 8;                 // consumer warps
constexpr int LT_CTHREADS = LT_CWARPS * 32;
constexpr int LT_THREADS = LT_CTHREADS + 64; // + the weight producer's warp + the key/value producer's warp
constexpr int LT_BOX_BYTES = 128 * 128;      // [128 output rows][64 bf16 inputs], 128B swizzle
constexpr int LT_SLOT_BYTES = 2 * LT_BOX_BYTES;  // a ring step: two K boxes of a chunk of outputs
// shared tiles: a ring step is six [64 outputs][64 inputs] boxes, so that a linear is one or two steps: waiting for a slot
// and handing it back costs a warp about 260 cycles even when the data are long there
constexpr int LT_SLOT_SHARED = 6 * 8192;
constexpr int LT_MAX_SLOTS = 8;
constexpr int LT_MAX_SET = 8;
constexpr int LT_MAX_SLABS = 8;              // active LoRA slabs of one linear
constexpr int LT_HD = 64;
constexpr int LT_MAX_SHARE = 6;              // CTAs that share a row tile, one per head (rows of up to 384)
constexpr int LT_KSPLIT = 4;                 // key ranges of the attention warps
constexpr int LT_ST = 8;                     // key tiles (8 keys) of one range, at most (256 tokens)
constexpr int LT_LDX = LT_HD + 8;            // shared tiles: row stride of a CTA's 64 fp32 columns (conflict-free)
constexpr long long LT_WAIT_CYCLES = 4000000000ll;

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float ex2(float x) {            // 2^x, one special-function instruction; 2^-inf = 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pk_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t bar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(bar) : "memory");
}

// untiled copy: both addresses 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, %0;" ::"n"(LT_CTHREADS) : "memory"); }

}  // namespace

namespace {

struct LatSmem {               // offsets (bytes) into dynamic shared memory
    int ring, kbuf, vbuf, xres, abuf, qbuf, hbuf, tbuf, stats, colv, slabs, misc, total;
    int lda, ldh, ldq, ldt;    // row strides in bf16 elements
    int kv_bytes;              // one head's keys (or values): [tpad rows][128 bytes], and a kilobyte behind them
    int cv_floats;             // one vector pack: bias[nmax], g[nmax], c1[128], c2[128]
};

__host__ __device__ inline LatSmem lat_layout(int d, int mlp, int patch_dim, int tokens, int layers, int ring_bytes, bool shared) {
    LatSmem s;
    auto up = [](int v) { return (v + 127) & ~127; };
    const int wide = mlp > patch_dim ? mlp : patch_dim, nmax = 3 * d > mlp ? 3 * d : mlp;
    s.lda = d + 8; s.ldh = wide + 8; s.ldq = d + 8; s.ldt = LT_MAX_SLABS * PM_SLAB + 8;
    const int tpad = (tokens + 15) / 16 * 16;
    s.kv_bytes = ((tpad * 128 + 1023) & ~1023) + 1024;      // + 1 KB that stays zero behind the values (see the P V loop)
    s.cv_floats = 2 * nmax + 2 * LT_MAX_SLABS * PM_SLAB;
    int o = 0;
    s.ring = o; o += ring_bytes;                      // 1024-byte aligned, as the 128B swizzle wants
    s.kbuf = o; o += s.kv_bytes;
    s.vbuf = o; o += s.kv_bytes;
    s.xres = o; o = up(o + (shared ? LT_ROWS * LT_LDX + d : LT_ROWS * d) * 4);       // shared: own columns, then a whole CLS row
    s.abuf = o; o = up(o + LT_ROWS * s.lda * 2);
    s.qbuf = o; o = up(o + LT_ROWS * s.ldq * 2);
    // the MLP's hidden rows (and the gathered patches); between blocks' MLPs: the attention warps' partial results
    const int hb = LT_ROWS * s.ldh * 2, pb = (shared ? LT_CWARPS : LT_KSPLIT) * LT_ROWS * (LT_HD + 2) * 4;
    s.hbuf = o; o = up(o + (hb > pb ? hb : pb));
    s.tbuf = o; o = up(o + LT_ROWS * s.ldt * 2);
    s.stats = o; o = up(o + LT_ROWS * 16);
    s.colv = o; o = up(o + 2 * s.cv_floats * 4);
    s.slabs = o; o = up(o + layers * 4 * 32);
    s.misc = o; o = up(o + 512);     // the adapter set, abort flag, mbarriers
    s.total = o;
    return s;
}

struct ActiveSet { int n; int id[LT_MAX_SET]; int slabs[LT_MAX_SET]; float scale[LT_MAX_SET]; };
// the LoRA slabs one linear applies to this frame: slab i belongs to set member who[i] and is its slab sl[i]
struct SlabTab { int n; uint8_t who[LT_MAX_SLABS]; uint8_t sl[LT_MAX_SLABS]; int per; int pad[2]; };   // per: K boxes of A^T in a step of a shared tile
static_assert(sizeof(SlabTab) == 32, "one table entry is 32 bytes");
static_assert(sizeof(ActiveSet) <= 128, "the adapter set sits in the first 128 bytes of the last region");

struct Ctx {
    uint8_t* sm;
    LatSmem L;
    int warp, lane, g, t, ns;
    uint32_t slot, phase;      // ring position: the same in every consumer thread (and in the producer)
    uint32_t li;               // linears done so far (their vector packs alternate between two buffers)
    int share, rank;           // CTAs on this row tile (a cluster) and this one's place among them
    uint32_t slot_bytes;
    bool ready;                // shared tiles: the next step's slot has been waited for already
    uint32_t xno;              // exchanges of rows between them so far (two barriers used in turn)
    int* status;
    volatile int* abort_flag;
};

__device__ __forceinline__ uint32_t bars(const Ctx& cx) { return s_u32(cx.sm + cx.L.misc + 256); }
__device__ __forceinline__ uint32_t full_bar(const Ctx& cx, uint32_t i) { return bars(cx) + 8u * i; }
__device__ __forceinline__ uint32_t empty_bar(const Ctx& cx, uint32_t i) { return bars(cx) + 64u + 8u * i; }
__device__ __forceinline__ uint32_t kfull_bar(const Ctx& cx) { return bars(cx) + 128u; }
__device__ __forceinline__ uint32_t kempty_bar(const Ctx& cx) { return bars(cx) + 136u; }
__device__ __forceinline__ uint32_t vfull_bar(const Ctx& cx) { return bars(cx) + 144u; }
__device__ __forceinline__ uint32_t vempty_bar(const Ctx& cx) { return bars(cx) + 152u; }
__device__ __forceinline__ uint32_t cfull_bar(const Ctx& cx, uint32_t b) { return bars(cx) + 160u + 8u * b; }
__device__ __forceinline__ uint32_t cempty_bar(const Ctx& cx, uint32_t b) { return bars(cx) + 176u + 8u * b; }
__device__ __forceinline__ uint32_t kvdone_bar(const Ctx& cx, uint32_t part) { return bars(cx) + 192u + 8u * part; }

__device__ __forceinline__ uint32_t xchg_bar(const Ctx& cx) { return bars(cx) + 208u + 8u * (cx.xno & 1u); }

// Shared tiles: the columns of chunk i of this CTA's part of a linear, as two halves of 64 (b < 0: only one).
// qkv: its head's keys and values, then its head's queries; other linears: the rank'th part of the outputs.
struct Halves { int a, b; };
// (part: outputs of the linear per CTA, passed in: a division in front of every chunk cost 2 % of a frame.)
__device__ __forceinline__ int share_chunks(int part, bool qkv) { return qkv ? 2 : (part + 127) >> 7; }
__device__ __forceinline__ Halves share_chunk(const Ctx& cx, int part, int d, bool qkv, int i) {
    Halves hv;
    if (qkv) {
        hv.a = (i == 0 ? d : 0) + cx.rank * LT_HD;
        hv.b = i == 0 ? 2 * d + cx.rank * LT_HD : -1;
        return hv;
    }
    hv.a = cx.rank * part + i * 128;
    hv.b = i * 128 + 64 < part ? hv.a + 64 : -1;
    return hv;
}
// the same shared-memory address in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// A warp's 16 x 16 part of the rows (the accumulator layout of mma: lo[q] / hi[q] = columns n0 + 8 q, + 1 of rows g and
// g + 8, n0 = 16-aligned column + 2 t) goes to the same place in every CTA of the tile: a 4 x 4 transpose in each
// quad makes it one 16-byte store per lane and CTA, and the stores to peers count their bytes on the peers' exchange barrier
// themselves, so nobody waits for stores to be performed before saying so.  (4-byte stores of fp32 rows and a release: 239
// against 182 us per frame.)
__device__ __forceinline__ uint4 quad_transpose(int t, const uint32_t (&lo)[2], const uint32_t (&hi)[2]) {
    const uint32_t r0 = __shfl_xor_sync(0xFFFFFFFFu, t & 1 ? lo[0] : hi[0], 1), r1 = __shfl_xor_sync(0xFFFFFFFFu, t & 1 ? lo[1] : hi[1], 1);
    const uint32_t p0 = t & 1 ? r0 : lo[0], p1 = t & 1 ? hi[0] : r0, q0 = t & 1 ? r1 : lo[1], q1 = t & 1 ? hi[1] : r1;
    const uint32_t e0 = __shfl_xor_sync(0xFFFFFFFFu, t & 2 ? p0 : q0, 2), e1 = __shfl_xor_sync(0xFFFFFFFFu, t & 2 ? p1 : q1, 2);
    return t & 2 ? make_uint4(e0, e1, q0, q1) : make_uint4(p0, p1, e0, e1);
}
// ... for row quad_row(), columns n0 + quad_col() .. + 7
__device__ __forceinline__ int quad_row(const Ctx& cx) { return cx.g + 8 * (cx.t & 1); }
__device__ __forceinline__ int quad_col(const Ctx& cx) { return 8 * (cx.t >> 1) - 2 * cx.t; }
__device__ __forceinline__ void put_rows(const Ctx& cx, bf16* buf, int ld, int n0, const uint32_t (&lo)[2], const uint32_t (&hi)[2]) {
    const uint4 v = quad_transpose(cx.t, lo, hi);
    bf16* dst = buf + quad_row(cx) * ld + n0 + quad_col(cx);
    *reinterpret_cast<uint4*>(dst) = v;
    const uint32_t addr = s_u32(dst), bar = xchg_bar(cx);
    for (int i = 1, r = cx.rank + 1; i < cx.share; ++i, ++r) {
        if (r == cx.share) r = 0;
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                     ::"r"(peer_addr(addr, r)), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(peer_addr(bar, r)) : "memory");
    }
}
// eight bytes of a row
__device__ __forceinline__ void put_piece(const Ctx& cx, bf16* dst, uint2 v) {
    *reinterpret_cast<uint2*>(dst) = v;
    const uint32_t addr = s_u32(dst), bar = xchg_bar(cx);
    for (int i = 1, r = cx.rank + 1; i < cx.share; ++i, ++r) {
        if (r == cx.share) r = 0;
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                     ::"r"(peer_addr(addr, r)), "r"(v.x), "r"(v.y), "r"(peer_addr(bar, r)) : "memory");
    }
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// The order in which a linear's chunks of 128 outputs are taken (producer and consumers alike).  qkv (width d):
// the chunk with the first head's keys, the chunk with its values, the other chunks with key or value
// columns, then the chunks of query columns alone -- the frame's other CTAs can fetch the first head's keys
// and values, and then the others', while this CTA is still multiplying.  Every other linear: as they come.
struct ChunkOrder { int n_chunks, ck, cv, n_kv; bool qkv, reorder; };
__device__ __forceinline__ ChunkOrder chunk_order(int N, int d, bool qkv) {
    ChunkOrder o;
    o.n_chunks = (N + 127) >> 7; o.qkv = qkv; o.reorder = qkv && o.n_chunks > 2;
    o.ck = d >> 7; o.cv = (2 * d) >> 7; o.n_kv = o.n_chunks - o.ck;
    return o;
}
__device__ __forceinline__ int chunk_at(const ChunkOrder& o, int i) {
    if (!o.reorder) return i;
    if (i == 0) return o.ck;
    if (i == 1) return o.cv;
    const int j = i - 2, rest = o.n_kv - 2;              // chunks with key / value columns besides ck and cv
    if (j >= rest) return j - rest;                      // query columns alone: chunks 0 .. ck - 1
    const int c = o.ck + 1 + j;
    return c >= o.cv ? c + 1 : c;
}
// position after which the first head's (part 0) / all heads' (part 1) keys and values of this CTA are stored;
// a qkv of one or two chunks is not reordered and reports once, at its end
__device__ __forceinline__ int publish_pos(const ChunkOrder& o, int part) {
    if (!o.qkv) return -1;
    if (!o.reorder) return part == 0 ? -1 : o.n_chunks - 1;
    return part == 0 ? 1 : o.n_kv - 1;
}

// Bounded wait on a barrier.  Once a wait has run out the CTA is aborting: later waits return at once and
// the results are meaningless (the status word says so).
__device__ __forceinline__ void bar_wait(const Ctx& cx, uint32_t bar, uint32_t parity) {
    if (bar_try(bar, parity)) return;
    const long long t0 = clock64();
    while (!bar_try(bar, parity)) {
        if (*cx.abort_flag) return;
        if (clock64() - t0 > LT_WAIT_CYCLES) {
            *cx.abort_flag = 1;
            atomicCAS(cx.status, 0, (int)PM_ERR_TIMEOUT);
            return;
        }
    }
}
// the vectors and the first step of the next linear
__device__ __forceinline__ void linear_ready(Ctx& cx) {
    bar_wait(cx, cfull_bar(cx, cx.li & 1u), (cx.li >> 1) & 1u);
    bar_wait(cx, full_bar(cx, cx.slot), cx.phase);
    cx.ready = true;
}
// The end of a linear (or of attention) whose `cols` columns per CTA went to all CTAs of the tile: this CTA's warps have
// written theirs and the peers' bytes are here.  One such point lies between any two uses of a buffer that the peers
// write, so a peer never overwrites rows still read here: rows written after exchange e were last read before their
// reader sent its own part of e.  Bytes of exchange e + 1 may land before this CTA's last warp is through with e, hence two
// barriers; those of e + 2 cannot.
// While the bytes are on their way the warps wait for the next linear's vectors and first step (`more`: there is one).
template <bool CL>
__device__ __forceinline__ void rows_sync(Ctx& cx, int cols, bool more) {
    if constexpr (!CL) { consumer_sync(); return; }
    const uint32_t bar = xchg_bar(cx), parity = (cx.xno >> 1) & 1u;
    __syncwarp();
    if (cx.lane == 0) {
        if (cx.warp == 0) bar_expect(bar, (uint32_t)((cx.share - 1) * cols * LT_ROWS * 2));
        else bar_arrive(bar);
    }
    if (more) linear_ready(cx);
    const long long t0 = clock64();
    for (;;) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok || *cx.abort_flag) break;
        if (clock64() - t0 > LT_WAIT_CYCLES) {
            *cx.abort_flag = 1;
            atomicCAS(cx.status, 0, (int)PM_ERR_TIMEOUT);
            break;
        }
    }
    ++cx.xno;
}
__device__ __forceinline__ void ring_advance(Ctx& cx) {
    if (++cx.slot == (uint32_t)cx.ns) { cx.slot = 0; cx.phase ^= 1u; }
}
// consumer side of one ring step: wait until the slot's copies have landed / hand the slot back
__device__ __forceinline__ uint32_t step_acquire(Ctx& cx) {
    if (!cx.ready) bar_wait(cx, full_bar(cx, cx.slot), cx.phase);
    cx.ready = false;
    return s_u32(cx.sm + cx.L.ring) + cx.slot * cx.slot_bytes;
}
__device__ __forceinline__ void step_release(Ctx& cx) {
    __syncwarp();
    if (cx.lane == 0) bar_arrive(empty_bar(cx, cx.slot));
    ring_advance(cx);
}
// producer side: wait until the eight consumer warps have handed the slot back (first lap: at once)
__device__ __forceinline__ uint32_t step_claim(Ctx& cx, uint32_t bytes) {
    bar_wait(cx, empty_bar(cx, cx.slot), cx.phase ^ 1u);
    bar_expect(full_bar(cx, cx.slot), bytes);
    return s_u32(cx.sm + cx.L.ring) + cx.slot * cx.slot_bytes;
}

// What the weight producer sends for one linear, in this order (the consumers take it in the same order):
//   the vector pack (bias, g, c1, c2) into the linear's pack buffer;
//   LoRA shrink, if any slab is active: K/128 steps, each the [16 rows][64] boxes of A^T of all active slabs
//   for two K boxes (the second K box's slabs 16 KB into the slot);
//   for each chunk of 128 outputs, in the order of chunk_at(): K/128 steps of W^T, each two
//   K boxes of the chunk ([64 rows][64] boxes, two per K box of a full chunk), then the chunk's rows of
//   the active slabs' B^T ([128 rows][16] boxes, four per step).
// Shared tiles: this CTA's chunks only, in steps of up to six 8 KB boxes (a K box of a chunk = its one or two halves);
// A^T in steps of up to 24 [16 rows][64] boxes; the B^T rows come as one [128 rows][16] box per slab and half (its second
// 64 rows unused), up to twelve per step.
template <bool CL>
__device__ void produce_linear(Ctx& cx, const LatLinear* lin, const SlabTab& st, const ActiveSet& as, int rs, int slabs_max,
                               int d, bool qkv) {
    const int N = lin->n_out, K = lin->k_in, k_boxes = K >> 6, n_chunks = (N + 127) >> 7, n_sl = st.n;
    const bool folded = lin->ln_g != nullptr;
    {
        const uint32_t b = cx.li & 1u, use = cx.li >> 1;
        bar_wait(cx, cempty_bar(cx, b), (use & 1u) ^ 1u);
        const uint32_t dst = s_u32(cx.sm + cx.L.colv) + b * (uint32_t)cx.L.cv_floats * 4u;
        const uint32_t vb = (uint32_t)N * 4u;
        const uint32_t bytes = vb + (folded ? vb : 0u) + (folded ? (uint32_t)n_sl * 128u : 0u);
        bar_expect(cfull_bar(cx, b), bytes);
        bulk_copy(dst, lin->bias, vb, cfull_bar(cx, b));
        if (folded) {
            bulk_copy(dst + vb, lin->ln_g, vb, cfull_bar(cx, b));
            for (int i = 0; i < n_sl; ++i) {
                const int arow = as.id[st.who[i]] * rs + st.sl[i] * PM_SLAB;
                bulk_copy(dst + 2u * vb + i * 64u, lin->c1 + arow, 64u, cfull_bar(cx, b));
                bulk_copy(dst + 2u * vb + LT_MAX_SLABS * 64u + i * 64u, lin->c2 + arow, 64u, cfull_bar(cx, b));
            }
        }
        ++cx.li;
    }
    if (CL && n_sl) {
        const int per = st.per;
        for (int kb0 = 0; kb0 < k_boxes && !*cx.abort_flag; kb0 += per) {
            const int nb = min(per, k_boxes - kb0);
            const uint32_t dst = step_claim(cx, (uint32_t)(nb * n_sl) * 2048u);
            for (int b = 0; b < nb; ++b)
                for (int i = 0; i < n_sl; ++i)
                    tma_box(dst + (uint32_t)(b * n_sl + i) * 2048u, &lin->tm_at, (kb0 + b) * 64, as.id[st.who[i]] * rs + st.sl[i] * PM_SLAB,
                            full_bar(cx, cx.slot));
            ring_advance(cx);
        }
    } else if (n_sl) {
        for (int kb0 = 0; kb0 < k_boxes && !*cx.abort_flag; kb0 += 2) {
            const int nb = min(2, k_boxes - kb0);
            const uint32_t dst = step_claim(cx, (uint32_t)(nb * n_sl) * 2048u);
            for (int b = 0; b < nb; ++b)
                for (int i = 0; i < n_sl; ++i)
                    tma_box(dst + b * LT_BOX_BYTES + i * 2048u, &lin->tm_at, (kb0 + b) * 64, as.id[st.who[i]] * rs + st.sl[i] * PM_SLAB,
                            full_bar(cx, cx.slot));
            ring_advance(cx);
        }
    }
    if (CL) {
        const int part = N / cx.share, mine = share_chunks(part, qkv);
        for (int ci = 0; ci < mine; ++ci) {
            const Halves hv = share_chunk(cx, part, d, qkv, ci);
            const int halves = hv.b < 0 ? 1 : 2, per = halves == 2 ? 3 : 6, slabs = halves == 2 ? 6 : 12;
            for (int kb0 = 0; kb0 < k_boxes && !*cx.abort_flag; kb0 += per) {
                const int nb = min(per, k_boxes - kb0);
                const uint32_t dst = step_claim(cx, (uint32_t)(nb * halves) * 8192u);
                for (int b = 0; b < nb; ++b) {
                    tma_box(dst + (uint32_t)(b * halves) * 8192u, &lin->tm_w, (kb0 + b) * 64, hv.a, full_bar(cx, cx.slot));
                    if (halves == 2) tma_box(dst + b * 16384u + 8192u, &lin->tm_w, (kb0 + b) * 64, hv.b, full_bar(cx, cx.slot));
                }
                ring_advance(cx);
            }
            for (int s0 = 0; s0 < n_sl && !*cx.abort_flag; s0 += slabs) {
                const int cnt = min(slabs, n_sl - s0);
                const uint32_t dst = step_claim(cx, (uint32_t)(cnt * halves) * 4096u);
                for (int j = 0; j < cnt; ++j) {
                    const int row = (as.id[st.who[s0 + j]] * slabs_max + st.sl[s0 + j]) * N;
                    tma_box(dst + (uint32_t)(j * halves) * 4096u, &lin->tm_bt, 0, row + hv.a, full_bar(cx, cx.slot));
                    if (halves == 2) tma_box(dst + j * 8192u + 4096u, &lin->tm_bt, 0, row + hv.b, full_bar(cx, cx.slot));
                }
                ring_advance(cx);
            }
        }
        return;
    }
    const ChunkOrder order = chunk_order(N, d, qkv);
    for (int ci = 0; ci < n_chunks; ++ci) {
        const int nc = chunk_at(order, ci);
        const int rows = min(128, N - nc * 128);
        for (int kb0 = 0; kb0 < k_boxes && !*cx.abort_flag; kb0 += 2) {
            const int nb = min(2, k_boxes - kb0);
            const uint32_t dst = step_claim(cx, (uint32_t)(nb * rows) * 128u);
            for (int b = 0; b < nb; ++b)
                for (int hf = 0; hf * 64 < rows; ++hf)
                    tma_box(dst + b * LT_BOX_BYTES + hf * 8192u, &lin->tm_w, (kb0 + b) * 64, nc * 128 + hf * 64, full_bar(cx, cx.slot));
            ring_advance(cx);
        }
        for (int s0 = 0; s0 < n_sl && !*cx.abort_flag; s0 += 4) {
            const int cnt = min(4, n_sl - s0);
            const uint32_t dst = step_claim(cx, (uint32_t)cnt * 4096u);
            for (int j = 0; j < cnt; ++j) {
                const int i = s0 + j;
                tma_box(dst + j * 4096u, &lin->tm_bt, 0, (as.id[st.who[i]] * slabs_max + st.sl[i]) * N + nc * 128, full_bar(cx, cx.slot));
            }
            ring_advance(cx);
        }
    }
}

// one K box of weights (row r of it per lane) against 64 columns of A
__device__ __forceinline__ void mma_box(const Ctx& cx, uint32_t a_row, uint32_t box, int r, float (&acc)[2][2][4]) {
    const int mi = cx.lane >> 3;
    // all eight fetches first, then the eight multiplications (four independent accumulators in turn)
    uint32_t a[4][4], b[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        ldsm4(a_row + ks * 32, a[ks][0], a[ks][1], a[ks][2], a[ks][3]);
        const int c = ks * 2 + (mi & 1);
        ldsm4(box + r * 128 + ((c ^ (r & 7)) << 4), b[ks][0], b[ks][1], b[ks][2], b[ks][3]);
    }
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        mma16816(acc[0][ks & 1], a[ks], b[ks][0], b[ks][1]);
        mma16816(acc[1][ks & 1], a[ks], b[ks][2], b[ks][3]);
    }
}
// one ring step of weights ([rows][64 inputs], this warp's 16 rows) against 64 columns of A (bf16, shared memory)
__device__ __forceinline__ void mma_step(Ctx& cx, uint32_t a_row0, int nb, bool active, float (&acc)[2][2][4]) {
    const uint32_t box0 = step_acquire(cx);
    if (active) {
        const int mi = cx.lane >> 3;
        const int r = cx.warp * 16 + (mi >> 1) * 8 + (cx.lane & 7);
        for (int bx = 0; bx < nb; ++bx) mma_box(cx, a_row0 + bx * 128, box0 + bx * LT_BOX_BYTES, r, acc);
    }
    step_release(cx);
}
__device__ __forceinline__ void acc_zero(float (&acc)[2][2][4]) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[q][h][0] = acc[q][h][1] = acc[q][h][2] = acc[q][h][3] = 0.f;
}

// The consumers' side of a linear's chunks: y[16, N] = A[16, K] W + t B.  A thread's eight values of a chunk
// go to epi(n0, y) in one call -- y[q][0..1] = columns n0 + 8 q, n0 + 8 q + 1 of row g, y[q][2..3] the same
// columns of row g + 8 -- so that the epilogue can fetch everything it needs before its first store.
// qkv: after the chunks at the two publish positions each warp reports at the barrier on which the key/value
// producer waits before it counts the CTA in at the frame's counter.
template <typename Epi>
__device__ void linear16(Ctx& cx, const bf16* A, int lda, int K, int N, int n_sl, int d, bool qkv,
                         Epi epi) {
    const int k_boxes = K >> 6, n_chunks = (N + 127) >> 7;
    const uint32_t a_base = s_u32(A) + ((cx.lane & 15) * lda + (cx.lane >> 4) * 8) * 2;
    const uint32_t t_row = s_u32(cx.sm + cx.L.tbuf) + ((cx.lane & 15) * cx.L.ldt + (cx.lane >> 4) * 8) * 2;
    const ChunkOrder order = chunk_order(N, d, qkv);
    for (int ci = 0; ci < n_chunks; ++ci) {
        const int nc = chunk_at(order, ci);
        const int rows = min(128, N - nc * 128);
        const bool active = cx.warp * 16 < rows;
        float acc[2][2][4];
        acc_zero(acc);
        for (int kb0 = 0; kb0 < k_boxes; kb0 += 2) mma_step(cx, a_base + kb0 * 128, min(2, k_boxes - kb0), active, acc);
        for (int s0 = 0; s0 < n_sl; s0 += 4) {
            const uint32_t box = step_acquire(cx);
            if (active) {
                // B^T rows are 32 bytes (16 ranks), 32B swizzle: the 16-byte half c of row n sits at c ^ ((n >> 2) & 1)
                const int n = cx.warp * 16 + ((cx.lane >> 4) & 1) * 8 + (cx.lane & 7), c = (cx.lane >> 3) & 1;
                const uint32_t b_row = box + n * 32 + ((c ^ ((n >> 2) & 1)) << 4);
                const int cnt = min(4, n_sl - s0);
                for (int j = 0; j < cnt; ++j) {
                    uint32_t a[4], b0, b1, b2, b3;
                    ldsm4(t_row + (s0 + j) * 32, a[0], a[1], a[2], a[3]);
                    ldsm4(b_row + j * 4096, b0, b1, b2, b3);
                    mma16816(acc[0][j & 1], a, b0, b1);
                    mma16816(acc[1][j & 1], a, b2, b3);
                }
            }
            step_release(cx);
        }
        if (active) {
            float y[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e) y[q][e] = acc[q][0][e] + acc[q][1][e];
            epi(nc * 128 + cx.warp * 16 + 2 * cx.t, y);
        }
        // this warp's keys and values of the block (the first head's / all) are stored: tell the key/value producer
        if (ci == publish_pos(order, 0) || ci == publish_pos(order, 1)) {
            __syncwarp();
            if (cx.lane == 0) {
                if (ci == publish_pos(order, 0)) bar_arrive(kvdone_bar(cx, 0));
                if (ci == publish_pos(order, 1)) bar_arrive(kvdone_bar(cx, 1));
            }
        }
    }
}

// n K steps of 16 from K step k0 of a ring step: boxes of [64 inputs] `box_bytes` apart, row r of them per lane
__device__ __forceinline__ void mma_run(const Ctx& cx, uint32_t a_row, uint32_t slot, uint32_t box_bytes, int r, int k0, int n, float (&acc)[2][2][4]) {
    const int mi = cx.lane >> 3;
    const uint32_t row = slot + r * 128;
#pragma unroll 2
    for (int i = 0; i < n; i += 2) {
        uint32_t a[2][4], b[2][4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = k0 + i + q, c = (k & 3) * 2 + (mi & 1);
            ldsm4(a_row + k * 32, a[q][0], a[q][1], a[q][2], a[q][3]);
            ldsm4(row + (k >> 2) * box_bytes + ((c ^ (r & 7)) << 4), b[q][0], b[q][1], b[q][2], b[q][3]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            mma16816(acc[0][q], a[q], b[q][0], b[q][1]);
            mma16816(acc[1][q], a[q], b[q][2], b[q][3]);
        }
    }
}

// The same for the chunks of a shared tile.  A chunk of 128 columns: a warp per 16 of them, as above.  A chunk of 64:
// four warps for each half of a step's K, the second four's sums added through `red` (4 KB that nothing else uses
// meanwhile).
template <typename Epi>
__device__ void linear16_shared(Ctx& cx, const bf16* A, int lda, int K, int part, int n_sl, int d, bool qkv, void* red, Epi epi) {
    const int k_boxes = K >> 6, mine = share_chunks(part, qkv), half = cx.warp >> 2, wq = cx.warp & 3, mi = cx.lane >> 3;
    const uint32_t a_base = s_u32(A) + ((cx.lane & 15) * lda + (cx.lane >> 4) * 8) * 2;
    const uint32_t t_row = s_u32(cx.sm + cx.L.tbuf) + ((cx.lane & 15) * cx.L.ldt + (cx.lane >> 4) * 8) * 2;
#pragma unroll 1
    for (int ci = 0; ci < mine; ++ci) {
        const Halves hv = share_chunk(cx, part, d, qkv, ci);
        const bool two = hv.b >= 0;
        const int halves = two ? 2 : 1, per = two ? 3 : 6, slabs = two ? 6 : 12;
        float acc[2][2][4];
        acc_zero(acc);
        const int r = (two ? cx.warp : wq) * 16 + (mi >> 1) * 8 + (cx.lane & 7);
        for (int kb0 = 0; kb0 < k_boxes; kb0 += per) {
            const int nb = min(per, k_boxes - kb0);
            const uint32_t slot = step_acquire(cx);
            mma_run(cx, a_base + kb0 * 128, slot, (uint32_t)halves * 8192u, r, two ? 0 : half * 2 * nb, two ? 4 * nb : 2 * nb, acc);
            step_release(cx);
        }
        for (int s0 = 0; s0 < n_sl; s0 += slabs) {
            const uint32_t box = step_acquire(cx);
            if (two || half == 0) {
                const int n = wq * 16 + ((cx.lane >> 4) & 1) * 8 + (cx.lane & 7), c = (cx.lane >> 3) & 1;
                const uint32_t b_row = box + half * 4096 + n * 32 + ((c ^ ((n >> 2) & 1)) << 4);
                const int cnt = min(slabs, n_sl - s0);
                for (int j = 0; j < cnt; ++j) {
                    uint32_t a[4], b0, b1, b2, b3;
                    ldsm4(t_row + (s0 + j) * 32, a[0], a[1], a[2], a[3]);
                    ldsm4(b_row + j * halves * 4096, b0, b1, b2, b3);
                    mma16816(acc[0][j & 1], a, b0, b1);
                    mma16816(acc[1][j & 1], a, b2, b3);
                }
            }
            step_release(cx);
        }
        float y[2][4];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) y[q][e] = acc[q][0][e] + acc[q][1][e];
        if (!two) {
            float4* rd = reinterpret_cast<float4*>(red) + wq * 64 + cx.lane;
            if (half) {
                rd[0] = make_float4(y[0][0], y[0][1], y[0][2], y[0][3]);
                rd[32] = make_float4(y[1][0], y[1][1], y[1][2], y[1][3]);
            }
            asm volatile("bar.sync %0, 64;" ::"r"(2 + wq) : "memory");
            if (!half) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float4 v = rd[q * 32];
                    y[q][0] += v.x; y[q][1] += v.y; y[q][2] += v.z; y[q][3] += v.w;
                }
            }
        }
        if (two || half == 0) epi((half ? hv.b : hv.a) + wq * 16 + 2 * cx.t, y);
        if (qkv && ci == 0) {                       // this warp's keys and values of the block are stored
            __syncwarp();
            if (cx.lane == 0) bar_arrive(kvdone_bar(cx, 0));
        }
    }
}
template <bool CL, typename Epi>
__device__ __forceinline__ void linear_rows(Ctx& cx, const bf16* A, int lda, int K, int N, int part, int n_sl, int d, bool qkv, void* red, Epi epi) {
    if constexpr (CL) linear16_shared(cx, A, lda, K, part, n_sl, d, qkv, red, epi);
    else linear16(cx, A, lda, K, N, n_sl, d, qkv, epi);
}

// The consumers' side of a linear's shrink steps: warp i < n_sl multiplies the rows by slab i of A^T and
// hands epi(row, i, j, v[j], v[j + 1]) its 16 x 16 result (even j).
template <bool CL, typename Epi>
__device__ void shrink16(Ctx& cx, const bf16* A, int lda, int K, int n_sl, int per, Epi epi) {
    const int k_boxes = K >> 6;
    const uint32_t a_base = s_u32(A) + ((cx.lane & 15) * lda + (cx.lane >> 4) * 8) * 2;
    const bool active = cx.warp < n_sl;
    float acc[2][2][4];
    acc_zero(acc);
    if (CL) {
        const int mi = cx.lane >> 3, r = cx.warp * 16 + (mi >> 1) * 8 + (cx.lane & 7);
        for (int kb0 = 0; kb0 < k_boxes; kb0 += per) {
            const uint32_t slot = step_acquire(cx);
            if (active) mma_run(cx, a_base + kb0 * 128, slot, (uint32_t)n_sl * 2048u, r, 0, 4 * min(per, k_boxes - kb0), acc);
            step_release(cx);
        }
    } else {
        for (int kb0 = 0; kb0 < k_boxes; kb0 += 2) mma_step(cx, a_base + kb0 * 128, min(2, k_boxes - kb0), active, acc);
    }
    if (active) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int j = q * 8 + 2 * cx.t;
            epi(cx.g, cx.warp, j, acc[q][0][0] + acc[q][1][0], acc[q][0][1] + acc[q][1][1]);
            epi(cx.g + 8, cx.warp, j, acc[q][0][2] + acc[q][1][2], acc[q][0][3] + acc[q][1][3]);
        }
    }
}

// GELU as the layer-by-layer GEMM epilogue computes it: x (1/2 + 1/2 tanh(x q(x^2))), q a quadratic fitted so that
// the result stays within 3e-5 of x Phi(x); one special-function instruction per element
__device__ __forceinline__ float gelu_fit(float v) {
    const float t = fminf(v * v, 50.f);                     // Phi has long saturated where the fitted q would turn over
    float q = fmaf(t, -3.5151945e-04f, 3.7005664e-02f);
    q = fmaf(q, t, 0.79750784f);
    float h;
    asm("tanh.approx.f32 %0, %1;" : "=f"(h) : "f"(v * q));
    return v * fmaf(h, 0.5f, 0.5f);
}

// abuf <- bf16(xres); stats[r] = (mean, rstd, 1/rstd) of the rounded row (what the tensor cores multiply).
// A warp takes two rows at once (two independent reduction chains); d is a multiple of 64, at most 384.
__device__ void round_rows_and_stats(Ctx& cx, int d, float eps) {
    const float* x = reinterpret_cast<const float*>(cx.sm + cx.L.xres);
    bf16* a = reinterpret_cast<bf16*>(cx.sm + cx.L.abuf);
    float4* st = reinterpret_cast<float4*>(cx.sm + cx.L.stats);
    const int n2 = d >> 6;                                  // float2 per lane and row
    for (int r = 2 * cx.warp; r < LT_ROWS; r += 2 * LT_CWARPS) {
        float2 v[2][6];
        float sum[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                v[q][i] = make_float2(0.f, 0.f);
                if (i < n2) {
                    const int c = 2 * cx.lane + 64 * i;
                    const float2 f = *reinterpret_cast<const float2*>(x + (r + q) * d + c);
                    const __nv_bfloat162 h = __floats2bfloat162_rn(f.x, f.y);
                    *reinterpret_cast<__nv_bfloat162*>(a + (r + q) * cx.L.lda + c) = h;
                    v[q][i] = __bfloat1622float2(h);
                    sum[q] += v[q][i].x + v[q][i].y;
                }
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sum[0] += __shfl_xor_sync(0xFFFFFFFFu, sum[0], o);
            sum[1] += __shfl_xor_sync(0xFFFFFFFFu, sum[1], o);
        }
        const float inv_d = 1.f / (float)d;
        const float mean[2] = {sum[0] * inv_d, sum[1] * inv_d};
        float sq[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < 6; ++i)
                if (i < n2) { const float t0 = v[q][i].x - mean[q], t1 = v[q][i].y - mean[q]; sq[q] += t0 * t0 + t1 * t1; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sq[0] += __shfl_xor_sync(0xFFFFFFFFu, sq[0], o);
            sq[1] += __shfl_xor_sync(0xFFFFFFFFu, sq[1], o);
        }
        if (cx.lane < 2) {
            const float rstd = rsqrtf((cx.lane ? sq[1] : sq[0]) * inv_d + eps);
            st[r + cx.lane] = make_float4(cx.lane ? mean[1] : mean[0], rstd, 1.f / rstd, 0.f);
        }
    }
}

// stats[r] of the rounded rows in abuf (shared tiles: they arrive there rounded).  Half a warp per row.
__device__ void stats_of_rows(Ctx& cx, int d, float eps) {
    const bf16* a = reinterpret_cast<const bf16*>(cx.sm + cx.L.abuf);
    float4* st = reinterpret_cast<float4*>(cx.sm + cx.L.stats);
    const int n2 = d >> 6, r = 2 * cx.warp + (cx.lane >> 4), l = cx.lane & 15;
    float2 v[12];
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        v[2 * i] = v[2 * i + 1] = make_float2(0.f, 0.f);
        if (i < n2) {
            const uint2 u = *reinterpret_cast<const uint2*>(a + r * cx.L.lda + 4 * l + 64 * i);
            v[2 * i] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
            v[2 * i + 1] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
            sum += (v[2 * i].x + v[2 * i].y) + (v[2 * i + 1].x + v[2 * i + 1].y);
        }
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    const float inv_d = 1.f / (float)d, mean = sum * inv_d;
    float sq = 0.f;
#pragma unroll
    for (int i = 0; i < 12; ++i)
        if (i < 2 * n2) { const float t0 = v[i].x - mean, t1 = v[i].y - mean; sq += t0 * t0 + t1 * t1; }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
    if (l == 0) {
        const float rstd = rsqrtf(sq * inv_d + eps);
        st[r] = make_float4(mean, rstd, 1.f / rstd, 0.f);
    }
}

// CL: the cluster's CTAs (as many as heads) share one tile of 16 rows.
template <bool CL>
__global__ void __launch_bounds__(LT_THREADS, 1) latency_forward_kernel(const __grid_constant__ LatArgs args) {
    extern __shared__ __align__(1024) uint8_t smem[];
    if (s_u32(smem) & 1023u) {                 // swizzled boxes need a 1024-byte aligned window
        if (threadIdx.x == 0) atomicCAS(args.status, 0, (int)PM_ERR_CUDA);
        return;
    }
    Ctx cx;
    cx.sm = smem;
    cx.slot_bytes = CL ? LT_SLOT_SHARED : LT_SLOT_BYTES; cx.ready = false;
    cx.L = lat_layout(args.d, args.mlp, args.patch_dim, args.tokens, args.layers, args.ring_slots * (int)cx.slot_bytes, CL);
    cx.ns = args.ring_slots;
    cx.warp = threadIdx.x >> 5; cx.lane = threadIdx.x & 31; cx.g = cx.lane >> 2; cx.t = cx.lane & 3;
    cx.share = CL ? args.heads : 1;
    cx.rank = CL ? (int)(blockIdx.x % (unsigned)cx.share) : 0;
    cx.xno = 0;
    const int tile = CL ? (int)(blockIdx.x / (unsigned)cx.share) : (int)blockIdx.x;
    const int f = tile / args.tiles_pf, rt = tile % args.tiles_pf;     // slot, row tile
    const int frame = args.perm ? args.perm[f] : f;                                  // input / output row
    const int T = args.tokens, d = args.d, r0 = rt * LT_ROWS;
    const int tpad = (T + 15) / 16 * 16;
    const int rs = args.slabs_max * PM_SLAB;
    float* xres = reinterpret_cast<float*>(smem + cx.L.xres);    // element (r, n) at r * ldx + n - x0
    const int ldx = CL ? LT_LDX : args.d, x0 = CL ? cx.rank * LT_HD : 0;
    bf16* abuf = reinterpret_cast<bf16*>(smem + cx.L.abuf);
    bf16* hbuf = reinterpret_cast<bf16*>(smem + cx.L.hbuf);
    bf16* qbuf = reinterpret_cast<bf16*>(smem + cx.L.qbuf);
    bf16* tbuf = reinterpret_cast<bf16*>(smem + cx.L.tbuf);
    const float4* stats = reinterpret_cast<const float4*>(smem + cx.L.stats);
    ActiveSet* as = reinterpret_cast<ActiveSet*>(smem + cx.L.misc);
    SlabTab* slabtab = reinterpret_cast<SlabTab*>(smem + cx.L.slabs);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + cx.L.misc + 192);
    cx.slot = 0; cx.phase = 0; cx.li = 0; cx.status = args.status; cx.abort_flag = abort_flag;
    if (threadIdx.x == 0) {
        for (int i = 0; i < LT_MAX_SLOTS; ++i) { bar_init(full_bar(cx, i), 1); bar_init(empty_bar(cx, i), LT_CWARPS); }
        bar_init(kfull_bar(cx), 1); bar_init(kempty_bar(cx), LT_CWARPS);
        bar_init(vfull_bar(cx), 1); bar_init(vempty_bar(cx), LT_CWARPS);
        for (int b = 0; b < 2; ++b) { bar_init(cfull_bar(cx, b), 1); bar_init(cempty_bar(cx, b), LT_CWARPS); }
        bar_init(kvdone_bar(cx, 0), LT_CWARPS); bar_init(kvdone_bar(cx, 1), LT_CWARPS);
        if (CL) { bar_init(xchg_bar(cx), LT_CWARPS); ++cx.xno; bar_init(xchg_bar(cx), LT_CWARPS); cx.xno = 0; }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }

    // ---- the frame's adapter set: valid, registered, distinct ids in ascending order
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        as->n = 0;
        const int o0 = args.set_off[f], cnt = args.set_off[f + 1] - o0;
        bool bad = cnt < 0 || o0 < 0;
        for (int i = 0; i < cnt && !bad; ++i) {
            const int a = args.set_ids[o0 + i];
            if (a < 0 || a >= args.max_adapters || args.rank[a] <= 0) { atomicCAS(args.status, 0, (int)PM_ERR_ARG); continue; }
            int at = 0;
            bool dup = false;
            while (at < as->n && as->id[at] <= a) { dup |= as->id[at] == a; ++at; }
            if (dup) { atomicCAS(args.status, 0, (int)PM_ERR_ARG); continue; }
            if (as->n == args.max_set) {                    // keep the lowest max_set ids
                atomicCAS(args.status, 0, (int)PM_ERR_CAPACITY);
                if (at == as->n) continue;
                --as->n;
            }
            for (int j = as->n; j > at; --j) as->id[j] = as->id[j - 1];
            as->id[at] = a;
            ++as->n;
        }
        if (bad) atomicCAS(args.status, 0, (int)PM_ERR_ARG);
        for (int i = 0; i < as->n; ++i) {
            as->slabs[i] = (args.rank[as->id[i]] + PM_SLAB - 1) / PM_SLAB;
            as->scale[i] = args.scale[as->id[i]];
        }
    }
    __syncthreads();
    // ---- per linear: the slabs of the set's adapters that touch it (adapters in ascending id; at most
    // LT_MAX_SLABS slabs, which the host checks against max_set * slabs_max)
    if ((int)threadIdx.x < args.layers * 4) {
        const LatLinear& lin = args.lin[threadIdx.x];
        SlabTab st;
        st.n = 0;
        if (lin.At) {
            for (int i = 0; i < as->n; ++i) {
                const int a = as->id[i];
                if (!((lin.adapted[a >> 5] >> (a & 31)) & 1u)) continue;
                for (int s = 0; s < as->slabs[i] && st.n < LT_MAX_SLABS; ++s) { st.who[st.n] = (uint8_t)i; st.sl[st.n] = (uint8_t)s; ++st.n; }
            }
        }
        st.per = st.n ? 24 / st.n : 24;
        slabtab[threadIdx.x] = st;
    }
    __syncthreads();
    if (CL) cluster_barrier();                    // every peer runs and has set its barriers up
    // ---- the weight producer: one thread, the whole network's static operands in consumption order
    if (cx.warp == LT_CWARPS) {
        if (elect_one()) {
            SlabTab none;
            none.n = 0;
            produce_linear<CL>(cx, args.lin + (size_t)args.layers * 4, none, *as, rs, args.slabs_max, d, false);
            for (int l = 0; l < args.layers && !*abort_flag; ++l)
                for (int j = 0; j < 4; ++j)
                    produce_linear<CL>(cx, args.lin + (size_t)l * 4 + j, slabtab[l * 4 + j], *as, rs, args.slabs_max, d, j == 0);
        }
        if (CL) { __syncwarp(); cluster_barrier(); }
        return;
    }
    // ---- the key/value producer: per block, wait for the frame's CTAs, then one head after the other
    if (cx.warp == LT_CWARPS + 1) {
        unsigned int* counter = args.bar + (CL ? f * cx.share + cx.rank : f);       // shared tiles: one per frame and head
        uint32_t idx = 0;
        if (elect_one()) for (int l = 0; l < args.layers && !*abort_flag; ++l) {
            // Twice per block -- for the first head, then for the others -- : the consumer warps have stored this
            // CTA's keys and values (ordinary stores, fetched by TMA on the other side: order the two proxies as
            // well as the scopes), so the CTA counts itself in: everything its threads stored up to there is
            // visible to whoever sees the count.  Then the heads' keys and values, one after the other.
            const int kv_row0 = ((l & 1) * args.n_frames + f) * T;
            const bool two = !CL && chunk_order(3 * d, d, true).reorder;   // else: one count-in per block
            for (int part = 0; part < (two ? 2 : 1) && !*abort_flag; ++part) {
                bar_wait(cx, kvdone_bar(cx, CL ? 0 : two ? part : 1), (uint32_t)l & 1u);
                if (*abort_flag) break;
                asm volatile("fence.proxy.async.global;" ::: "memory");
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
                const unsigned int per = two ? 2u : 1u;
                const unsigned int want = (unsigned int)args.tiles_pf * (per * (unsigned int)l + (unsigned int)part + 1u);
                const long long t0 = clock64();
                unsigned int seen;
                do {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
                    if (seen < want && (*abort_flag || clock64() - t0 > LT_WAIT_CYCLES)) {
                        if (!*abort_flag) { *abort_flag = 1; atomicCAS(args.status, 0, (int)PM_ERR_TIMEOUT); }
                        break;
                    }
                } while (seen < want);
                if (*abort_flag) break;
                asm volatile("fence.proxy.async.global;" ::: "memory");
                const int h0 = CL ? cx.rank : !two ? 0 : part == 0 ? 0 : 1;
                const int h1 = CL ? cx.rank + 1 : !two ? args.heads : part == 0 ? 1 : args.heads;
                for (int h = h0; h < h1; ++h, ++idx) {
                    bar_wait(cx, kempty_bar(cx), (idx & 1u) ^ 1u);
                    bar_expect(kfull_bar(cx), (uint32_t)tpad * 128u);
                    tma_box(s_u32(smem + cx.L.kbuf), &args.tm_kv, h * LT_HD, kv_row0, kfull_bar(cx));
                    bar_wait(cx, vempty_bar(cx), (idx & 1u) ^ 1u);
                    bar_expect(vfull_bar(cx), (uint32_t)tpad * 128u);
                    tma_box(s_u32(smem + cx.L.vbuf), &args.tm_kv, d + h * LT_HD, kv_row0, vfull_bar(cx));
                }
            }
        }
        if (CL) { __syncwarp(); cluster_barrier(); }
        return;
    }

    // ================================ consumers (256 threads) ================================
    // ---- patch gather: hbuf[r][c*P*P + py*P + px] = frame[c][gy*P + py][gx*P + px] of token r0 + r (token 0 = CLS)
    {
        const int P = 16, per_row = args.patch_dim / 8;
        const bf16* fr = args.frames + (size_t)frame * 3 * args.img * args.img;
        for (int i = threadIdx.x; i < LT_ROWS * per_row; i += LT_CTHREADS) {
            const int r = i / per_row, ch = i % per_row, tok = r0 + r;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (tok >= 1 && tok < T) {
                const int p = tok - 1, gy = p / args.grid, gx = p % args.grid;
                const int col = ch * 8, c = col / (P * P), py = (col / P) % P, px = col % P;
                v = *reinterpret_cast<const uint4*>(fr + ((size_t)c * args.img + gy * P + py) * args.img + gx * P + px);
            }
            *reinterpret_cast<uint4*>(hbuf + r * cx.L.ldh + ch * 8) = v;
        }
    }
    // the kilobyte behind the values is read as keys whose probabilities are zero: it has to hold finite numbers
    for (int i = threadIdx.x; i < 256; i += LT_CTHREADS)
        reinterpret_cast<uint32_t*>(smem + cx.L.vbuf + cx.L.kv_bytes - 1024)[i] = 0u;
    consumer_sync();
    if (CL) linear_ready(cx);

    // the vector pack of the linear the consumers are at: wait for it / hand its buffer back
    auto pack_acquire = [&]() -> const float* {
        if (!CL) bar_wait(cx, cfull_bar(cx, cx.li & 1u), (cx.li >> 1) & 1u);      // shared tiles: linear_ready() has
        return reinterpret_cast<const float*>(smem + cx.L.colv) + (cx.li & 1u) * cx.L.cv_floats;
    };
    auto pack_release = [&]() {
        __syncwarp();
        if (cx.lane == 0) bar_arrive(cempty_bar(cx, cx.li & 1u));
        ++cx.li;
    };
    // ---- patch projection + positions; the CLS row
    {
        const float* cv = pack_acquire();
        linear_rows<CL>(cx, hbuf, cx.L.ldh, args.patch_dim, d, LT_HD, 0, d, false, qbuf, [&](int n0, float (&y)[2][4]) {
            uint32_t row[2][2];                             // [hi][q], rounded
#pragma unroll
            for (int hi = 0; hi < 2; ++hi) {
                const int r = cx.g + 8 * hi, tok = r0 + r;
                float2 p[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if (tok < T) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) p[q] = *reinterpret_cast<const float2*>(args.pos + (size_t)tok * d + n0 + 8 * q);
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int n = n0 + 8 * q;
                    float2 out = make_float2(0.f, 0.f);             // rows past the frame stay zero
                    if (tok == 0) out = make_float2(args.cls[n] + p[q].x, args.cls[n + 1] + p[q].y);
                    else if (tok < T) out = make_float2(y[q][2 * hi] + cv[n] + p[q].x, y[q][2 * hi + 1] + cv[n + 1] + p[q].y);
                    *reinterpret_cast<float2*>(xres + r * ldx + n - x0) = out;
                    row[hi][q] = pk_bf16(out.x, out.y);
                }
            }
            if constexpr (CL) put_rows(cx, abuf, cx.L.lda, n0, row[0], row[1]);
        });
        pack_release();
    }
    rows_sync<CL>(cx, LT_HD, true);

    // LoRA shrink of a linear with slab table `st` on the rows A: t[r][16 i + j] (bf16) = s_a (x A_a)
    // (folded linears: s_a ((x A' - mean c1) + c2 / rstd), the fused accumulator being scaled by rstd afterwards)
    auto shrink = [&](const SlabTab& st, const bf16* A, int lda, int K, int N, bool folded, const float* cv) {
        if (!st.n) return;
        shrink16<CL>(cx, A, lda, K, st.n, st.per, [&](int r, int i, int j, float v0, float v1) {
            if (folded) {
                const float* c1 = cv + 2 * N + i * PM_SLAB + j;
                const float* c2 = c1 + LT_MAX_SLABS * PM_SLAB;
                v0 = (v0 - stats[r].x * c1[0]) + c2[0] * stats[r].z;
                v1 = (v1 - stats[r].x * c1[1]) + c2[1] * stats[r].z;
            }
            const float sc = as->scale[st.who[i]];
            *reinterpret_cast<uint32_t*>(tbuf + r * cx.L.ldt + i * PM_SLAB + j) = pk_bf16(v0 * sc, v1 * sc);
        });
        consumer_sync();
    };
    // x += y + b.  Shared tiles: the fp32 rows stay with the CTA that owns their columns, the others get them rounded; the
    // first CTA of the frame's first tile also gets the CLS row behind the last block, for the heads.
    auto residual = [&](const float* cv, bool last) {
        return [=, &cx](int n0, float (&y)[2][4]) {
            float2 x[2][2], b[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                b[q] = *reinterpret_cast<const float2*>(cv + n0 + 8 * q);
                x[q][0] = *reinterpret_cast<const float2*>(xres + cx.g * ldx + n0 - x0 + 8 * q);
                x[q][1] = *reinterpret_cast<const float2*>(xres + (cx.g + 8) * ldx + n0 - x0 + 8 * q);
            }
            uint32_t row[2][2];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int hi = 0; hi < 2; ++hi) {
                    float2 v = x[q][hi];
                    if (r0 + cx.g + 8 * hi < T) {
                        v = make_float2(v.x + y[q][2 * hi] + b[q].x, v.y + y[q][2 * hi + 1] + b[q].y);
                        *reinterpret_cast<float2*>(xres + (cx.g + 8 * hi) * ldx + n0 - x0 + 8 * q) = v;
                    }
                    row[hi][q] = pk_bf16(v.x, v.y);
                    if (CL && last && hi == 0 && cx.g == 0)
                        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};"
                                     ::"r"(peer_addr(s_u32(xres + LT_ROWS * LT_LDX + n0 + 8 * q), 0)), "f"(v.x), "f"(v.y) : "memory");
                }
            if constexpr (CL) put_rows(cx, abuf, cx.L.lda, n0, row[0], row[1]);
        };
    };

    const float att_scale = 0.125f * 1.4426950408889634f;  // 1/sqrt(64) * log2(e)
    const int mlp_part = CL ? args.mlp / cx.share : args.mlp;    // a CTA's columns of the hidden layer
    uint32_t head_no = 0;                                    // heads attended so far (all blocks)
    // the attended rows; shared tiles: beside this head's queries, since a peer may be done while qkv still reads abuf here
    bf16* att = CL ? qbuf : abuf;
    const int ldatt = CL ? cx.L.ldq : cx.L.lda;
    for (int l = 0; l < args.layers; ++l) {
        const SlabTab* st = slabtab + l * 4;
        bf16* kvb = args.kv + (size_t)(l & 1) * args.n_frames * T * 2 * d + (size_t)f * T * 2 * d;
        // ---- qkv (LayerNorm 1 folded): q stays here, k and v go to the frame's exchange buffer
        if constexpr (CL) stats_of_rows(cx, d, args.eps);
        else round_rows_and_stats(cx, d, args.eps);
        consumer_sync();
        {
            const float* cv = pack_acquire();
            shrink(st[0], abuf, cx.L.lda, d, 3 * d, true, cv);
            const float4 s_lo = stats[cx.g], s_hi = stats[cx.g + 8];
            linear_rows<CL>(cx, abuf, cx.L.lda, d, 3 * d, LT_HD, st[0].n, d, true, hbuf, [&](int n0, float (&y)[2][4]) {
                float2 b[2], gs[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    b[q] = *reinterpret_cast<const float2*>(cv + n0 + 8 * q);
                    gs[q] = *reinterpret_cast<const float2*>(cv + 3 * d + n0 + 8 * q);
                }
                uint32_t lo[2], hi[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int n = n0 + 8 * q;
                    lo[q] = pk_bf16(s_lo.y * (y[q][0] - s_lo.x * gs[q].x) + b[q].x, s_lo.y * (y[q][1] - s_lo.x * gs[q].y) + b[q].y);
                    hi[q] = pk_bf16(s_hi.y * (y[q][2] - s_hi.x * gs[q].x) + b[q].x, s_hi.y * (y[q][3] - s_hi.x * gs[q].y) + b[q].y);
                    if (CL) continue;
                    if (n < d) {
                        *reinterpret_cast<uint32_t*>(qbuf + cx.g * cx.L.ldq + n) = lo[q];
                        *reinterpret_cast<uint32_t*>(qbuf + (cx.g + 8) * cx.L.ldq + n) = hi[q];
                    } else {
                        if (r0 + cx.g < T) *reinterpret_cast<uint32_t*>(kvb + (size_t)(r0 + cx.g) * 2 * d + (n - d)) = lo[q];
                        if (r0 + cx.g + 8 < T) *reinterpret_cast<uint32_t*>(kvb + (size_t)(r0 + cx.g + 8) * 2 * d + (n - d)) = hi[q];
                    }
                }
                if constexpr (CL) {
                    const uint4 v = quad_transpose(cx.t, lo, hi);
                    const int r = quad_row(cx), n = n0 + quad_col(cx);
                    if (n < d) *reinterpret_cast<uint4*>(qbuf + r * cx.L.ldq + n) = v;
                    else if (r0 + r < T) *reinterpret_cast<uint4*>(kvb + (size_t)(r0 + r) * 2 * d + (n - d)) = v;
                }
            });
            pack_release();
        }
        consumer_sync();                                     // all of q is in place
        // ---- attention, head by head.  Warp w: key range w / 2 of four, dims 32 (w % 2) .. + 31 of the head.
        // Keys and values of a head are one TMA box each ([tpad rows][64 dims], 128B swizzle; rows past the
        // frame hold a neighbour's rows or zeros and are masked below).
        {
            // shared tiles: eight key ranges, a warp takes all 64 dims; else four, the two warps of a pair split the dims
            // (with the count-in above as one release: 179 -> 176 us per frame)
            constexpr int RANGES = CL ? LT_CWARPS : LT_KSPLIT, ST = CL ? LT_ST / 2 : LT_ST, NP = CL ? 4 : 2;
            const int kr = CL ? cx.warp : cx.warp >> 1, dh = CL ? 0 : cx.warp & 1;
            const int n_t8 = tpad / 8;
            const int t8_lo = (n_t8 * kr) / RANGES, t8_hi = (n_t8 * (kr + 1)) / RANGES, n_t = t8_hi - t8_lo;   // <= ST tiles
            // a key tile is 8 rows of 128 bytes, so a lane's row keeps its swizzle phase (lane & 7) from tile
            // to tile: one address per k16 step (keys) or pair of dim tiles (values), plus a multiple of 1 KB
            const int l7 = cx.lane & 7, mi = cx.lane >> 3;
            uint32_t k_addr[2], v_addr[NP];
#pragma unroll
            for (int kp = 0; kp < 2; ++kp)                   // one fetch brings a tile's keys for two k16 steps (32 dims)
                k_addr[kp] = s_u32(smem + cx.L.kbuf) + (t8_lo * 8 + l7) * 128 + (((kp * 4 + mi) ^ l7) << 4);
#pragma unroll
            for (int n = 0; n < NP; ++n)
                v_addr[n] = s_u32(smem + cx.L.vbuf) + (t8_lo * 8 + (mi & 1) * 8 + l7) * 128 + (((dh * 4 + n * 2 + (mi >> 1)) ^ l7) << 4);
            float* part = reinterpret_cast<float*>(smem + cx.L.hbuf);
            for (int h = cx.rank; h < (CL ? cx.rank + 1 : args.heads); ++h, ++head_no) {
                uint32_t qa[4][4];
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    ldsm4(s_u32(qbuf) + ((cx.lane & 15) * cx.L.ldq + h * LT_HD + ks * 16 + (cx.lane >> 4) * 8) * 2,
                          qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3]);
                bar_wait(cx, kfull_bar(cx), head_no & 1u);
                float s[ST][4];
#pragma unroll
                for (int j = 0; j < ST; ++j) s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
                // tile by tile inside each k16 step: consecutive multiplications go to different accumulators
#pragma unroll
                for (int kp = 0; kp < 2; ++kp) {
                    uint32_t kf[ST][4];
#pragma unroll
                    for (int j = 0; j < ST; ++j)
                        if (j < n_t) ldsm4(k_addr[kp] + j * 1024, kf[j][0], kf[j][1], kf[j][2], kf[j][3]);
#pragma unroll
                    for (int j = 0; j < ST; ++j)
                        if (j < n_t) mma16816(s[j], qa[2 * kp], kf[j][0], kf[j][1]);
#pragma unroll
                    for (int j = 0; j < ST; ++j)
                        if (j < n_t) mma16816(s[j], qa[2 * kp + 1], kf[j][2], kf[j][3]);
                }
                __syncwarp();
                if (cx.lane == 0) bar_arrive(kempty_bar(cx));        // the next head's keys may land
                float m_lo = -INFINITY, m_hi = -INFINITY;
#pragma unroll
                for (int j = 0; j < ST; ++j) {
                    const int key = (t8_lo + j) * 8 + 2 * cx.t;
                    if (j >= n_t || (t8_lo + j) * 8 + 8 > T) {       // only the frame's last tile has keys to mask
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (!(j < n_t && key + (e & 1) < T)) s[j][e] = -INFINITY;
                    }
                    m_lo = fmaxf(m_lo, fmaxf(s[j][0], s[j][1]));
                    m_hi = fmaxf(m_hi, fmaxf(s[j][2], s[j][3]));
                }
                m_lo = fmaxf(m_lo, __shfl_xor_sync(0xFFFFFFFFu, m_lo, 1));
                m_lo = fmaxf(m_lo, __shfl_xor_sync(0xFFFFFFFFu, m_lo, 2));
                m_hi = fmaxf(m_hi, __shfl_xor_sync(0xFFFFFFFFu, m_hi, 1));
                m_hi = fmaxf(m_hi, __shfl_xor_sync(0xFFFFFFFFu, m_hi, 2));
                // the maxima in the exponent's units (1/sqrt(64) log2 e); a warp whose keys are all beyond the
                // frame contributes nothing (its maximum stays -inf)
                m_lo *= att_scale; m_hi *= att_scale;
                const float ms_lo = m_lo == -INFINITY ? 0.f : m_lo, ms_hi = m_hi == -INFINITY ? 0.f : m_hi;
                float l_lo = 0.f, l_hi = 0.f;
                uint32_t pa[ST / 2][4];
#pragma unroll
                for (int j = 0; j < ST; ++j) {
                    const float p0 = ex2(fmaf(s[j][0], att_scale, -ms_lo)), p1 = ex2(fmaf(s[j][1], att_scale, -ms_lo));
                    const float p2 = ex2(fmaf(s[j][2], att_scale, -ms_hi)), p3 = ex2(fmaf(s[j][3], att_scale, -ms_hi));
                    l_lo += p0 + p1;
                    l_hi += p2 + p3;
                    pa[j >> 1][(j & 1) * 2 + 0] = pk_bf16(p0, p1);
                    pa[j >> 1][(j & 1) * 2 + 1] = pk_bf16(p2, p3);
                }
                l_lo += __shfl_xor_sync(0xFFFFFFFFu, l_lo, 1);
                l_lo += __shfl_xor_sync(0xFFFFFFFFu, l_lo, 2);
                l_hi += __shfl_xor_sync(0xFFFFFFFFu, l_hi, 1);
                l_hi += __shfl_xor_sync(0xFFFFFFFFu, l_hi, 2);
                float o[2 * NP][4];
#pragma unroll
                for (int i = 0; i < 2 * NP; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
                bar_wait(cx, vfull_bar(cx), head_no & 1u);
                // 16-key steps of this warp's keys.  The second tile of the last step may belong to the next
                // range (its probabilities are 0 here) or lie behind the last key (the kilobyte of zeros)
#pragma unroll
                for (int kk = 0; kk < ST / 2; ++kk) {
                    if (2 * kk < n_t) {
#pragma unroll
                        for (int n = 0; n < NP; ++n) {           // pairs of 8-dim tiles
                            uint32_t b0, b1, b2, b3;
                            ldsm4t(v_addr[n] + kk * 2048, b0, b1, b2, b3);
                            mma16816(o[2 * n], pa[kk], b0, b1);
                            mma16816(o[2 * n + 1], pa[kk], b2, b3);
                        }
                    }
                }
                __syncwarp();
                if (cx.lane == 0) bar_arrive(vempty_bar(cx));
                // partial results: part[range][row][0..63] = o, [64] = max, [65] = sum
                float* pw = part + (size_t)kr * LT_ROWS * (LT_HD + 2);
#pragma unroll
                for (int i = 0; i < 2 * NP; ++i) {
                    const int c = dh * 32 + i * 8 + 2 * cx.t;
                    *reinterpret_cast<float2*>(pw + cx.g * (LT_HD + 2) + c) = make_float2(o[i][0], o[i][1]);
                    *reinterpret_cast<float2*>(pw + (cx.g + 8) * (LT_HD + 2) + c) = make_float2(o[i][2], o[i][3]);
                }
                if (dh == 0 && cx.t == 0) {
                    pw[cx.g * (LT_HD + 2) + 64] = m_lo; pw[cx.g * (LT_HD + 2) + 65] = l_lo;
                    pw[(cx.g + 8) * (LT_HD + 2) + 64] = m_hi; pw[(cx.g + 8) * (LT_HD + 2) + 65] = l_hi;
                }
                consumer_sync();
                {   // merge: thread -> (row, four dims)
                    const int r = threadIdx.x >> 4, c4 = (threadIdx.x & 15) * 4;
                    float m = -INFINITY;
#pragma unroll
                    for (int w = 0; w < RANGES; ++w) m = fmaxf(m, part[(w * LT_ROWS + r) * (LT_HD + 2) + 64]);
                    float den = 0.f, num[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int w = 0; w < RANGES; ++w) {
                        const float* pr = part + (w * LT_ROWS + r) * (LT_HD + 2);
                        const float e = pr[64] == -INFINITY ? 0.f : ex2(pr[64] - m);
                        den += e * pr[65];
#pragma unroll
                        for (int q = 0; q < 4; ++q) num[q] += e * pr[c4 + q];
                    }
                    const float inv = 1.f / den;                 // key 0 is always valid: den > 0
                    uint2 pkd;
                    pkd.x = pk_bf16(num[0] * inv, num[1] * inv);
                    pkd.y = pk_bf16(num[2] * inv, num[3] * inv);
                    bf16* dst = att + r * ldatt + h * LT_HD + c4;
                    if constexpr (CL) put_piece(cx, dst, pkd);
                    else *reinterpret_cast<uint2*>(dst) = pkd;
                }
                rows_sync<CL>(cx, LT_HD, true);
            }
        }
        // ---- proj (+ residual)
        {
            const float* cv = pack_acquire();
            shrink(st[1], att, ldatt, d, d, false, cv);
            linear_rows<CL>(cx, att, ldatt, d, d, LT_HD, st[1].n, d, false, hbuf, residual(cv, false));
            pack_release();
        }
        rows_sync<CL>(cx, LT_HD, true);
        // ---- fc1 (LayerNorm 2 folded, GELU) and fc2 (+ residual)
        if constexpr (CL) stats_of_rows(cx, d, args.eps);
        else round_rows_and_stats(cx, d, args.eps);
        consumer_sync();
        {
            const float* cv = pack_acquire();
            const int N = args.mlp;
            shrink(st[2], abuf, cx.L.lda, d, N, true, cv);
            const float4 s_lo = stats[cx.g], s_hi = stats[cx.g + 8];
            linear_rows<CL>(cx, abuf, cx.L.lda, d, N, mlp_part, st[2].n, d, false, nullptr, [&](int n0, float (&y)[2][4]) {
                float2 b[2], gs[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    b[q] = *reinterpret_cast<const float2*>(cv + n0 + 8 * q);
                    gs[q] = *reinterpret_cast<const float2*>(cv + N + n0 + 8 * q);
                }
                uint32_t lo[2], hi[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int n = n0 + 8 * q;
                    lo[q] = pk_bf16(gelu_fit(s_lo.y * (y[q][0] - s_lo.x * gs[q].x) + b[q].x), gelu_fit(s_lo.y * (y[q][1] - s_lo.x * gs[q].y) + b[q].y));
                    hi[q] = pk_bf16(gelu_fit(s_hi.y * (y[q][2] - s_hi.x * gs[q].x) + b[q].x), gelu_fit(s_hi.y * (y[q][3] - s_hi.x * gs[q].y) + b[q].y));
                    if (!CL) {
                        *reinterpret_cast<uint32_t*>(hbuf + cx.g * cx.L.ldh + n) = lo[q];
                        *reinterpret_cast<uint32_t*>(hbuf + (cx.g + 8) * cx.L.ldh + n) = hi[q];
                    }
                }
                if constexpr (CL) put_rows(cx, hbuf, cx.L.ldh, n0, lo, hi);
            });
            pack_release();
        }
        rows_sync<CL>(cx, mlp_part, true);
        {
            const float* cv = pack_acquire();
            shrink(st[3], hbuf, cx.L.ldh, args.mlp, d, false, cv);
            linear_rows<CL>(cx, hbuf, cx.L.ldh, args.mlp, d, LT_HD, st[3].n, d, false, qbuf, residual(cv, l == args.layers - 1));
            pack_release();
        }
        rows_sync<CL>(cx, LT_HD, l + 1 < args.layers);
    }

    if (CL) cluster_barrier();                                // no peer sends rows any more, aborted or not
    if (*abort_flag)
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);     // copies still in flight land before shared memory goes away
    if (*abort_flag || rt != 0 || cx.rank != 0) return;

    // ---- heads on the CLS row (row 0 of the frame's first CTA): final LayerNorm, base head, adapter heads
    float* z = reinterpret_cast<float*>(smem + cx.L.hbuf);
    const float* cls_row = CL ? xres + LT_ROWS * LT_LDX : xres;
    if (cx.warp == 0) {
        float v[12], sum = 0.f;
#pragma unroll
        for (int i = 0; i < 12; ++i) { const int c = cx.lane + 32 * i; v[i] = c < d ? cls_row[c] : 0.f; sum += v[i]; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        const float mean = sum / (float)d;
        float sq = 0.f;
#pragma unroll
        for (int i = 0; i < 12; ++i) if (cx.lane + 32 * i < d) { const float t = v[i] - mean; sq += t * t; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
        const float rstd = rsqrtf(sq / (float)d + args.eps);
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            const int c = cx.lane + 32 * i;
            if (c < d) z[c] = (v[i] - mean) * rstd * args.lnf_g[c] + args.lnf_b[c];
        }
    }
    float* srow = args.scores_out + (size_t)frame * args.n_classes;
    for (int k = threadIdx.x; k < args.n_classes; k += LT_CTHREADS) srow[k] = 0.f;
    consumer_sync();
    // one thread per head row: its d weights are independent 16-byte loads, all in flight at once
    auto dot = [&](const bf16* w) {
        float acc0 = 0.f, acc1 = 0.f;
        for (int c = 0; c < d; c += 8) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(w + c));
            const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc0 = fmaf(z[c + 2 * q], __bfloat162float(h2[q].x), acc0);
                acc1 = fmaf(z[c + 2 * q + 1], __bfloat162float(h2[q].y), acc1);
            }
        }
        return acc0 + acc1;
    };
    if (args.base_out) {
        for (int k = threadIdx.x; k < args.n_classes; k += LT_CTHREADS) {
            const float v = dot(args.head_wt + (size_t)k * d) + args.head_b[k];
            args.base_out[(size_t)frame * args.n_classes + k] = 1.f / (1.f + expf(-v));
        }
    }
    for (int i = 0; i < as->n; ++i) {
        const int a = as->id[i];
        for (int r = args.hoff[a] + threadIdx.x; r < args.hoff[a + 1]; r += LT_CTHREADS) {
            const float v = dot(args.hcat + (size_t)r * d) + args.hbias[r];
            // scores are positive: the maximum over adapters is an integer maximum of the bit patterns
            atomicMax(reinterpret_cast<int*>(srow + args.hcls[r]), __float_as_int(1.f / (1.f + expf(-v))));
        }
    }
}

// the most ring slots that fit beside everything else (0: the geometry does not fit at all)
int lat_ring_slots(int d, int mlp, int patch_dim, int tokens, int layers, bool shared) {
    const int room = 227 * 1024 - lat_layout(d, mlp, patch_dim, tokens, layers, 0, shared).total;
    const int slot = shared ? LT_SLOT_SHARED : LT_SLOT_BYTES;
    if (room < 2 * slot) return 0;
    return room / slot < LT_MAX_SLOTS ? room / slot : LT_MAX_SLOTS;
}

// CTAs per tile of 16 rows.  One per head (each takes its head and its part of every linear's outputs, and the rows are
// exchanged through distributed shared memory) while clusters for all tiles of the batch are resident at once, and where
// the hidden layer splits into parts of whole 128-column chunks; else one CTA does the whole tile.
int lat_share(const LatArgs& a, size_t smem) {
    const int c = a.heads;
    if (c < 2 || c > LT_MAX_SHARE || a.mlp % (128 * c) != 0) return 1;
    // clusters of c CTAs the device holds at once; the shared memory is that of one CTA per SM whatever the geometry
    static std::atomic<int> resident[64][LT_MAX_SHARE + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    std::atomic<int>& known = resident[dev & 63][c];
    if (const int n = known.load(std::memory_order_relaxed); n > 0) return a.n_frames * a.tiles_pf <= n ? c : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.n_frames * a.tiles_pf * c);
    cfg.blockDim = dim3(LT_THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)c;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, latency_forward_kernel<true>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    known.store(clusters, std::memory_order_relaxed);
    return a.n_frames * a.tiles_pf <= clusters ? c : 1;
}

}  // namespace

size_t latency_smem_bytes(int d, int mlp, int patch_dim, int tokens, int layers) {
    const int slots = lat_ring_slots(d, mlp, patch_dim, tokens, layers, false);
    if (!slots) return (size_t)1 << 30;
    return (size_t)lat_layout(d, mlp, patch_dim, tokens, layers, slots * LT_SLOT_BYTES, false).total;
}

// Sets `launched` once the kernel is on the stream.  cudaErrorNotSupported: this form does not apply to the geometry or the batch.
static cudaError_t launch_form(const Launch& L, const LatArgs& a, bool shared, bool& launched) {
    const int slots = lat_ring_slots(a.d, a.mlp, a.patch_dim, a.tokens, a.layers, shared);
    if (!slots) return shared ? cudaErrorNotSupported : cudaErrorInvalidValue;
    const int smem = lat_layout(a.d, a.mlp, a.patch_dim, a.tokens, a.layers, slots * (shared ? LT_SLOT_SHARED : LT_SLOT_BYTES), shared).total;
    static SmemGrant grant[2];
    if (cudaError_t e = shared ? grant[1].ensure(latency_forward_kernel<true>, smem) : grant[0].ensure(latency_forward_kernel<false>, smem);
        e != cudaSuccess) return e;
    const int share = shared ? lat_share(a, (size_t)smem) : 1;
    if (shared && share == 1) return cudaErrorNotSupported;
    const int ctas = a.n_frames * a.tiles_pf * share;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(LT_THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = L.st;
    // the CTAs of a frame wait for one another: all of them must be resident at once
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)share;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = share > 1 ? 2 : 1;
    LatArgs copy = a;
    copy.status = L.status;
    copy.ring_slots = slots;
    // the frames' arrival counters start at zero (an aborted launch may have left them anywhere)
    cudaError_t e = cudaMemsetAsync(a.bar, 0, sizeof(unsigned int) * a.n_frames * share, L.st);
    if (e != cudaSuccess) return e;
    e = share > 1 ? cudaLaunchKernelEx(&cfg, latency_forward_kernel<true>, copy) : cudaLaunchKernelEx(&cfg, latency_forward_kernel<false>, copy);
    if (e != cudaSuccess) return e;
    launched = true;
    BUMP(L);
    return cudaGetLastError();
}

cudaError_t launch_latency_forward(const Launch& L, const LatArgs& a) {
    if (a.layers * 4 > LT_THREADS) return cudaErrorInvalidValue;
    // Tiles shared by clusters where that applies, else, or where the launch of the clusters is refused (a profiler, or a
    // limit on the SMs, may leave room for fewer of them than the device), one CTA per tile.
    ProfScope ps(L, KC_GEMM);
    bool launched = false;
    const cudaError_t e = launch_form(L, a, true, launched);
    if (launched) return e;
    if (e != cudaErrorNotSupported) cudaGetLastError();
    return launch_form(L, a, false, launched);
}
