"""GPU parity of the single operators (through the C ABI) against the CPU oracle."""
import numpy as np
import pytest

import workloads as wl
from oracle import polymorph_oracle as po

pytestmark = pytest.mark.gpu

# bf16 build: inputs are bf16-exact, products accumulate in fp32, the output is rounded once to
# bf16 (relative 2^-9) and the LoRA intermediate t = s (x A) once more; fp32 debug build: fp32
# accumulation order only.
TOL = {0: dict(atol=1.5e-2, rtol=1.5e-2), 1: dict(atol=2e-4, rtol=2e-4)}


def tdtype(dtype):
    import torch
    return torch.bfloat16 if dtype == 0 else torch.float32


def to_dev(a, dtype):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda().to(tdtype(dtype)).contiguous()


def to_np(t):
    return t.float().cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("rows,d", [(1, 192), (1003, 384), (2 * 197 + 5, 768), (64, 1024)])
def test_layernorm(dtype, rows, d):
    import torch
    from paper_2507_14959_b200 import binding
    x = wl.normal((rows, d), 1.0, "ln_gpu", rows, d) * 3 + 0.5
    x = wl.round_bf16(x)
    g = wl.normal((d,), 0.2, "ln_gpu_g", d, mean=1.0)
    b = wl.normal((d,), 0.2, "ln_gpu_b", d)
    xd = to_dev(x, dtype)
    yd = torch.full_like(xd, float("nan"))
    binding.layernorm(xd, torch.from_numpy(g).cuda(), torch.from_numpy(b).cuda(), yd, 1e-6, dtype)
    torch.cuda.synchronize()
    want = po.layernorm(x.astype(np.float64), g.astype(np.float64), b.astype(np.float64), 1e-6)
    np.testing.assert_allclose(to_np(yd), want, **TOL[dtype])


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("frames,tokens,heads", [(3, 197, 3), (1, 577, 2), (2, 10, 1), (2, 64, 2), (1, 130, 1),
                                                 (2, 626, 2),      # beyond the tcgen05 kernels' 624 tokens
                                                 (1, 785, 1)])     # 448x448 frames: several query slices
def test_attention(dtype, frames, tokens, heads):
    import torch
    from paper_2507_14959_b200 import binding
    d = heads * 64
    qkv = wl.normal((frames * tokens, 3 * d), 1.0, "attn_gpu", frames, tokens, heads)
    qd = to_dev(qkv, dtype)
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=tdtype(dtype))
    binding.attention(qd, od, frames, tokens, heads, dtype)
    torch.cuda.synchronize()
    got = to_np(od)
    for f in range(frames):
        want = po.attention(qkv[f * tokens:(f + 1) * tokens].astype(np.float64), heads)
        np.testing.assert_allclose(got[f * tokens:(f + 1) * tokens], want, **TOL[dtype])


def test_attention_many_heads_several_query_tiles_per_cta():
    """With enough (frame, head) pairs to fill the GPU several times over, the kernel for 209..624 tokens
    gives each CTA all query tiles of its pair (instead of one tile per CTA): two key blocks and three
    query tiles here, the second and third tile reusing the score regions and O of the first.  Three
    frames of the batch are compared with the oracle."""
    import torch
    from paper_2507_14959_b200 import binding
    frames, tokens, heads = 50, 300, 12
    d = heads * 64
    qkv = wl.normal((frames * tokens, 3 * d), 1.0, "attn_gpu_many", frames, tokens, heads).astype(np.float32)
    qd = to_dev(qkv, 0)
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=tdtype(0))
    binding.attention(qd, od, frames, tokens, heads, 0)
    torch.cuda.synchronize()
    got = to_np(od)
    assert np.isfinite(got).all()
    for f in (0, 17, 49):
        want = po.attention(to_np(qd[f * tokens:(f + 1) * tokens]).astype(np.float64), heads)
        np.testing.assert_allclose(got[f * tokens:(f + 1) * tokens], want, **TOL[0])


def oracle_linear(cell_x, w, b, A, B, scale, tokens, offsets, ids, epilogue, residual):
    out = np.empty((cell_x.shape[0], w.shape[1]))
    w64, b64 = w.astype(np.float64), b.astype(np.float64)
    for f in range(len(offsets) - 1):
        rows = slice(f * tokens, (f + 1) * tokens)
        act = [(scale, A[a].astype(np.float64), B[a].astype(np.float64))
               for a in sorted(ids[offsets[f]:offsets[f + 1]])]
        out[rows] = po.lora_linear(cell_x[rows].astype(np.float64), w64, b64, act)
    if epilogue == 1:
        out = po.gelu(out)
    elif epilogue == 2:
        out = out + residual
    return out


LINEAR_CASES = [
    # k_in, n_out, frames, tokens, rank, n_adapters, epilogue, sets
    (192, 576, 2, 197, 4, 4, 0, [[0], [1, 3]]),
    (192, 192, 3, 197, 4, 4, 2, [[], [2], [0, 1, 2, 3]]),
    (384, 1536, 5, 197, 8, 6, 1, [[5], [5], [0, 2], [], [1, 3, 4]]),
    (768, 2304, 5, 197, 16, 8, 0, [[0], [0, 7], [1, 2, 3], [4], [4]]),
    (3072, 768, 3, 197, 16, 4, 2, [[0, 1], [2], [3]]),
    (768, 3072, 2, 577, 32, 5, 1, [[0, 4], [1, 2, 3]]),
    (768, 768, 3, 197, 64, 9, 0, [[0, 1, 2, 3, 4, 5, 6, 7], [8], [2, 8]]),
    (128, 256, 7, 10, 16, 3, 0, [[0], [1], [2], [0, 1], [], [1, 2], [0, 1, 2]]),   # many frames per tile
    (768, 2304, 4, 197, 16, 2, 0, [[], [], [], []]),                                # no LoRA at all
]


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("case", LINEAR_CASES, ids=[f"{c[0]}x{c[1]}_F{c[2]}_T{c[3]}_r{c[4]}_e{c[6]}" for c in LINEAR_CASES])
def test_lora_linear(dtype, case):
    import torch
    from paper_2507_14959_b200 import binding
    k_in, n_out, frames, tokens, rank, n_ad, epi, sets = case
    name = f"lin_gpu_{k_in}_{n_out}_{rank}"
    rows = frames * tokens
    x = wl.normal((rows, k_in), 1.0, name, "x")
    w = wl.normal((k_in, n_out), 0.02, name, "w")
    b = wl.normal((n_out,), 0.02, name, "b")
    A = [wl.normal((k_in, rank), 0.02, name, "A", a) for a in range(n_ad)]
    B = [wl.normal((rank, n_out), 0.02, name, "B", a) for a in range(n_ad)]
    res = wl.normal((rows, n_out), 1.0, name, "res")
    scale = 32.0 / rank
    off, ids = wl.sets_to_csr(sets)
    max_set = max(1, max(len(s) for s in sets))
    lin = binding.Linear(w, b, max_adapters=n_ad, max_rank=rank, max_set=max_set, max_frames=frames,
                         tokens=tokens, epilogue=epi, dtype=dtype)
    for a in range(n_ad):
        lin.register(a, rank, scale, A[a], B[a])
    xd = to_dev(x, dtype)
    rd = to_dev(res, dtype) if epi == 2 else None
    yd = torch.full((rows, n_out), float("nan"), device="cuda", dtype=tdtype(dtype))
    lin.forward(xd, frames, off, ids, yd, residual=rd)
    assert lin.status() == 0
    got = to_np(yd)
    want = oracle_linear(x, w, b, A, B, scale, tokens, off, ids, epi, res.astype(np.float64))
    np.testing.assert_allclose(got, want, **TOL[dtype])
    # a second call with the same sets reuses the cached plan and must give the same bits
    y2 = torch.full_like(yd, float("nan"))
    lin.forward(xd, frames, off, ids, y2, residual=rd)
    assert lin.status() == 0
    assert torch.equal(yd, y2)
    # LoRA really contributes where a set is non-empty
    if any(sets):
        base = oracle_linear(x, w, b, A, B, scale, tokens, np.zeros(frames + 1, np.int32), ids[:0], epi,
                             res.astype(np.float64))
        assert np.abs(want - base).max() > 0.05
    lin.close()


FULL_SIZE_CELLS = [
    # k_in, n_out, rank, clustered, epilogue
    (768, 2304, 16, False, 0),
    (3072, 768, 64, False, 2),      # rank 64 with up to 8 active adapters: the largest LoRA share
    (768, 3072, 64, False, 1),
    (768, 2304, 32, True, 0),       # Zipf-clustered sets
    (3072, 768, 8, True, 2),        # rank below one slab
]


@pytest.mark.parametrize("k_in,n_out,rank,clustered,epi", FULL_SIZE_CELLS,
                         ids=[f"{c[0]}x{c[1]}_r{c[2]}_{'zipf' if c[3] else 'unif'}_e{c[4]}" for c in FULL_SIZE_CELLS])
def test_lora_linear_full_size_sampled(k_in, n_out, rank, clustered, epi):
    """Cells of the single-linear grid at full size (256 frames x 197 tokens, 128 adapters of one
    rank, 1-8 active per frame) in the launch configuration the sweep times; the oracle computes
    sampled rows one by one: first and last row tiles, frame boundaries, the ragged tail, rows of
    the frames with the most active adapters, and random rows."""
    import torch
    from paper_2507_14959_b200 import binding
    cell = wl.linear_cell(k_in, n_out, 256, rank, clustered=clustered)
    lin = binding.Linear(cell.w, cell.b, max_adapters=128, max_rank=rank, max_set=8, max_frames=256,
                         tokens=cell.tokens, epilogue=epi, dtype=0)
    for a in range(128):
        lin.register(a, rank, cell.scale, cell.A[a], cell.B[a])
    rows = 256 * cell.tokens
    xd = to_dev(cell.x, 0)
    res = wl.normal((rows, n_out), 1.0, cell.name, "res") if epi == 2 else None
    rd = to_dev(res, 0) if epi == 2 else None
    yd = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    lin.forward(xd, 256, cell.set_offsets, cell.set_ids, yd, residual=rd)
    assert lin.status() == 0
    assert not torch.isnan(yd.float()).any()
    g = wl.rng_for("full_size_rows", k_in, n_out, rank)
    sizes = np.diff(cell.set_offsets)
    assert sizes.max() == 8
    widest = [int(f) for f in np.argsort(-sizes, kind="stable")[:3]]
    sample = sorted(set([0, 127, 128, 196, 197, 198, rows - 1, rows - 65, rows - 128, rows - 129]
                        + [f * cell.tokens + t for f in widest for t in (0, 100, 196)]
                        + [int(r) for r in g.integers(0, rows, 48)]))
    got = to_np(yd[sample])
    w64, b64 = cell.w.astype(np.float64), cell.b.astype(np.float64)
    for i, r in enumerate(sample):
        f = r // cell.tokens
        act = [(cell.scale, cell.A[a].astype(np.float64), cell.B[a].astype(np.float64))
               for a in sorted(cell.set_ids[cell.set_offsets[f]:cell.set_offsets[f + 1]])]
        want = po.lora_linear(cell.x[r:r + 1].astype(np.float64), w64, b64, act)[0]
        if epi == 1:
            want = po.gelu(want)
        elif epi == 2:
            want = want + wl.round_bf16(res[r]).astype(np.float64)
        np.testing.assert_allclose(got[i], want, **TOL[0])
    lin.close()


def test_gelu_epilogue_accuracy():
    """The GELU epilogue against the exact-erf definition: y = gelu(4 x) through an identity-like
    weight, x sweeping [-3, 3] (so the argument spans [-12, 12]); the bf16 result must be within one
    bf16 step of the exact value plus 3e-5 (the kernel evaluates a fitted form x (1/2 + 1/2 tanh(x q(x^2)))
    of x Phi(x) whose absolute error stays below 2.6e-5, with the hardware's approximate tanh)."""
    import torch
    from paper_2507_14959_b200 import binding
    n, rows = 64, 197 * 3
    w = 4.0 * np.eye(n, dtype=np.float32)
    x = wl.round_bf16(np.linspace(-3.0, 3.0, rows * n, dtype=np.float32).reshape(rows, n))
    lin = binding.Linear(w, np.zeros(n, np.float32), max_adapters=1, max_rank=16, max_set=1, max_frames=3,
                         tokens=197, epilogue=1, dtype=0)
    xd = to_dev(x, 0)
    yd = torch.full((rows, n), float("nan"), device="cuda", dtype=torch.bfloat16)
    lin.forward(xd, 3, np.zeros(4, np.int32), np.zeros(0, np.int32), yd)
    assert lin.status() == 0
    want = po.gelu(4.0 * x.astype(np.float64))
    got = to_np(yd)
    step = np.maximum(np.abs(want), 2.0 ** -20) * 2.0 ** -8          # one bf16 step at |want|
    assert np.all(np.abs(got - want) <= step + 3e-5)
    assert np.all(got[want > 11.0] == wl.round_bf16(want[want > 11.0].astype(np.float32)))   # saturated branch: x itself
    lin.close()


def test_linear_argument_errors():
    import torch
    from paper_2507_14959_b200 import binding
    w = wl.normal((64, 64), 0.02, "err_w")
    b = np.zeros(64, np.float32)
    lin = binding.Linear(w, b, max_adapters=2, max_rank=16, max_set=1, max_frames=2, tokens=8, dtype=0)
    lin.register(0, 16, 2.0, np.zeros((64, 16), np.float32), np.zeros((16, 64), np.float32))
    x = torch.zeros((16, 64), device="cuda", dtype=torch.bfloat16)
    y = torch.zeros_like(x)
    with pytest.raises(binding.PolymorphError) as e:      # unregistered adapter
        lin.forward(x, 2, [0, 1, 2], [0, 1], y)
    assert e.value.code == binding.PM_ERR_STATE
    with pytest.raises(binding.PolymorphError) as e:      # set larger than max_set
        lin.forward(x, 2, [0, 2, 2], [0, 0], y)
    assert e.value.code == binding.PM_ERR_CAPACITY
    with pytest.raises(binding.PolymorphError) as e:      # non-monotone CSR
        lin.forward(x, 2, [0, 1, 0], [0], y)
    assert e.value.code == binding.PM_ERR_ARG
    with pytest.raises(binding.PolymorphError) as e:      # too many frames
        lin.forward(x, 3, [0, 0, 0, 0], [], y)
    assert e.value.code == binding.PM_ERR_CAPACITY
    with pytest.raises(binding.PolymorphError) as e:      # rank above max_rank
        lin.register(1, 32, 1.0, np.zeros((64, 32), np.float32), np.zeros((32, 64), np.float32))
    assert e.value.code == binding.PM_ERR_CAPACITY
    lin.close()


def test_bounded_wait_gives_up_and_reports():
    """A wait on a barrier that nothing signals runs into its limit, records PM_ERR_TIMEOUT, takes the
    other warps of the CTA out through the abort flag and releases tensor memory; nothing faults and
    the next kernel on the device runs normally."""
    import torch
    from paper_2507_14959_b200 import binding
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    trace = torch.full((3,), -1, dtype=torch.int32, device="cuda")
    binding.selftest_wait_timeout(100000, status, trace)
    torch.cuda.synchronize()
    assert int(status.item()) == binding.PM_ERR_TIMEOUT
    assert trace.cpu().tolist() == [1, 3, 1]
    # the context is intact: an ordinary operator right after
    x = wl.normal((64, 128), 1.0, "after_timeout")
    y = torch.zeros((64, 128), device="cuda")
    binding.layernorm(torch.from_numpy(x).cuda(), torch.ones(128, device="cuda"), torch.zeros(128, device="cuda"),
                      y, 1e-6, 1)
    torch.cuda.synchronize()
    np.testing.assert_allclose(y.cpu().numpy(), po.layernorm(x.astype(np.float64), np.ones(128), np.zeros(128), 1e-6),
                               atol=2e-4)
    with pytest.raises(binding.PolymorphError):
        binding.selftest_wait_timeout(10 ** 12, status, trace)       # limits beyond 1e8 cycles are refused


def check_form(k_in, n_out, rows, epi, adapters, form):
    """The kernel, tile width and split of K that a test names are those of the rule (stated for 148 SMs)."""
    import torch
    from paper_2507_14959_b200 import binding
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert binding.linear_kernel(k_in, n_out, rows, epi, adapters)[:3] == form


@pytest.mark.parametrize("k_in,n_out,frames,tokens,rank,epi,form,what", [
    (768, 768, 1, 197, 16, 2, ("few rows", 64, 1), ""), (320, 576, 2, 130, 24, 0, ("few rows", 64, 1), "odd K blocks"),
    (768, 2304, 3, 197, 64, 0, ("few rows", 128, 1), "several slab groups"), (192, 1152, 16, 128, 16, 1, ("few rows", 128, 1), "whole row tiles"),
    (192, 1152, 24, 128, 16, 1, ("few rows", 192, 1), "whole row tiles"), (768, 3072, 6, 197, 16, 1, ("few rows", 256, 1), ""),
    (3072, 768, 1, 197, 16, 2, ("few rows", 64, 4), ""), (1600, 768, 3, 200, 16, 2, ("few rows", 128, 4), "odd K blocks"),
    (3072, 768, 6, 197, 8, 2, ("few rows", 128, 2), ""), (3072, 768, 8, 197, 48, 2, ("few rows", 192, 2), "several slab groups"),
    (3072, 768, 12, 197, 16, 2, ("few rows", 256, 2), ""), (3072, 768, 17, 197, 16, 2, ("few rows", 192, 1), "unsplit"),
    (768, 768, 33, 197, 16, 2, ("pair", 192, 1), "beyond one wave: shrink and pair GEMM"), (384, 1152, 30, 197, 16, 0, ("pair", 192, 1), "beyond one wave, short K"),
    (1600, 1536, 20, 197, 16, 2, ("pair", 192, 1), "shrink with K in four, odd K blocks"),
    (1536, 1536, 40, 197, 48, 2, ("pair", 256, 1), "shrink with K in two, several slab groups"),
    (320, 768, 70, 130, 64, 1, ("single", 256, 1), "shrink of one tile per SM, odd K blocks, slabs beyond the list"),
    (192, 768, 300, 100, 24, 0, ("single", 256, 1), "shrink of two tiles per SM"), (192, 256, 300, 197, 40, 1, ("single", 256, 1), "shrink of three tiles per SM"),
    (64, 64, 1, 1, 4, 0, ("few rows", 64, 1), "one row")])
def test_lora_linear_over_the_tile_rule(k_in, n_out, frames, tokens, rank, epi, form, what, most=6):
    """One case on each side of every line of the few-row kernel's tile rule for linears with adapters (on 148 SMs), sets of
    0 to 6 of 7 adapters, against float64 sums of the same bf16 inputs.  Tolerance: as for the other linears (one bf16 rounding of
    the output, one of t)."""
    import torch
    from paper_2507_14959_b200 import binding
    check_form(k_in, n_out, frames * tokens, epi, most > 0, form)
    gen = torch.Generator(device="cuda").manual_seed(k_in + n_out + frames)

    def draw(shape, std):
        return (torch.randn(shape, generator=gen, device="cuda") * std).bfloat16()
    rows, n_ad = frames * tokens, 7
    x, res, w, b = draw((rows, k_in), 1.0), draw((rows, n_out), 1.0), draw((k_in, n_out), 0.02), draw((n_out,), 0.02)
    A = [draw((k_in, rank), 0.02) for _ in range(n_ad)]
    B = [draw((rank, n_out), 0.02) for _ in range(n_ad)]
    g = np.random.default_rng(rows)
    sets = [sorted(int(a) for a in g.choice(n_ad, size=int(g.integers(0, most + 1)), replace=False)) for _ in range(frames)]
    off, ids = wl.sets_to_csr(sets)
    host = lambda t: t.float().cpu().numpy()  # noqa: E731
    lin = binding.Linear(host(w), host(b), max_adapters=n_ad, max_rank=rank, max_set=6, max_frames=frames, tokens=tokens, epilogue=epi)
    for a in range(n_ad):
        lin.register(a, rank, 2.0, host(A[a]), host(B[a]))
    y = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    lin.forward(x, frames, off, ids, y, residual=res if epi == 2 else None)
    assert lin.status() == 0
    want = x.double() @ w.double() + b.double()
    for f, s in enumerate(sets):
        r = slice(f * tokens, (f + 1) * tokens)
        for a in s:
            want[r] += 2.0 * (x[r].double() @ A[a].double()) @ B[a].double()
    if epi == 1:
        want = torch.nn.functional.gelu(want)
    elif epi == 2:
        want = want + res.double()
    np.testing.assert_allclose(to_np(y), want.cpu().numpy(), **TOL[0])
    lin.close()


@pytest.mark.parametrize("k_in,n_out,frames,tokens,rank,epi,form,rounds", [
    (768, 640, 31, 130, 16, 2, ("pair", 128, 1), 2), (832, 640, 70, 197, 40, 1, ("pair", 128, 1), 4), (768, 896, 100, 130, 24, 0, ("pair", 128, 1), 5),
    (3072, 768, 37, 197, 16, 2, ("pair", 192, 1), 2), (768, 576, 40, 200, 48, 2, ("pair", 192, 1), 2), (768, 768, 37, 197, 40, 1, ("pair", 192, 1), 2),
    (768, 576, 70, 197, 8, 0, ("pair", 192, 1), 3),
    (448, 1280, 60, 197, 8, 0, ("pair", 256, 1), 4), (768, 768, 50, 200, 48, 2, ("pair", 256, 1), 2), (768, 2304, 24, 130, 16, 1, ("pair", 256, 1), 2),
    (768, 768, 60, 197, 16, 2, ("pair", 256, 1), 2), (448, 640, 70, 197, 40, 1, ("single", 128, 1), 4)])
def test_pair_gemm_widths(k_in, n_out, frames, tokens, rank, epi, form, rounds):
    """The three tile widths of the CTA-pair GEMM, and the single-CTA kernel for a width that only 128 divides, with the plain,
    the GELU and the residual epilogue, ragged last row tiles, several rounds, up to 21 slabs.  (One round: the residuals
    without adapters below.  Folded LayerNorm and patch placement: the models' forwards.)"""
    rows = 256 if form[0] == "pair" else 128
    assert -(-(-(-frames * tokens // rows) * (n_out // form[1])) // (148 if form[0] == "single" else 74)) == rounds
    test_lora_linear_over_the_tile_rule(k_in, n_out, frames, tokens, rank, epi, form, "")


@pytest.mark.parametrize("k_in,n_out,frames,form", [
    (768, 768, 6, ("few rows", 64, 1)), (768, 768, 8, ("pair", 128, 1)), (512, 512, 24, ("few rows", 128, 1)), (512, 512, 28, ("pair", 256, 1)),
    (3072, 768, 6, ("few rows", 128, 2)), (2048, 512, 12, ("pair", 128, 1)), (2048, 512, 24, ("few rows", 128, 1)), (1600, 576, 9, ("few rows", 64, 1)),
    (1600, 576, 12, ("few rows", 192, 2)), (3072, 576, 16, ("pair", 192, 1)), (256, 256, 40, ("few rows", 128, 1)), (256, 256, 96, ("single", 256, 1))])
def test_residual_linear_without_adapters_around_the_few_row_rule(k_in, n_out, frames, form):
    """A residual and empty sets on both sides of each line of the few-row kernel's rule."""
    test_lora_linear_over_the_tile_rule(k_in, n_out, frames, 197, 8, 2, form, "", most=0)


@pytest.mark.parametrize("k_in,n_out,frames,tokens,rank,adapters", [(64, 256, 130, 197, 8, 0), (384, 512, 60, 130, 16, 0), (192, 768, 40, 200, 24, 5),
                                                                    (320, 384, 90, 197, 16, 0), (768, 768, 40, 197, 16, 5), (1536, 640, 30, 130, 16, 0)])
def test_residual_may_be_the_output_buffer(k_in, n_out, frames, tokens, rank, adapters):
    """y == residual through the single-CTA and the pair GEMM, ragged last row tiles: bit-equal to separate buffers, and within the
    tolerance of the other linears of float64 sums."""
    import torch
    from paper_2507_14959_b200 import binding
    assert binding.linear_kernel(k_in, n_out, frames * tokens, 2, adapters)[0] == ("single" if k_in <= 384 else "pair")
    gen = torch.Generator(device="cuda").manual_seed(k_in + n_out)
    rows = frames * tokens

    def draw(shape, std):
        return (torch.randn(shape, generator=gen, device="cuda") * std).bfloat16()
    x, res, w, b = draw((rows, k_in), 1.0), draw((rows, n_out), 1.0), draw((k_in, n_out), 0.02), draw((n_out,), 0.02)
    A = [draw((k_in, rank), 0.02) for _ in range(adapters)]
    B = [draw((rank, n_out), 0.02) for _ in range(adapters)]
    host = lambda t: t.float().cpu().numpy()  # noqa: E731
    lin = binding.Linear(host(w), host(b), max_adapters=max(1, adapters), max_rank=rank, max_set=1, max_frames=frames, tokens=tokens, epilogue=2)
    for a in range(adapters):
        lin.register(a, rank, 1.0, host(A[a]), host(B[a]))
    off, ids = wl.sets_to_csr([[f % adapters] if adapters else [] for f in range(frames)])
    y, z = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16), res.clone()
    lin.forward(x, frames, off, ids, y, residual=res)
    lin.forward(x, frames, off, ids, z, residual=z)
    assert lin.status() == 0
    assert torch.equal(y, z)
    want = x.double() @ w.double() + b.double() + res.double()
    for f in range(frames if adapters else 0):
        r = slice(f * tokens, (f + 1) * tokens)
        want[r] += (x[r].double() @ A[f % adapters].double()) @ B[f % adapters].double()
    np.testing.assert_allclose(to_np(y), want.cpu().numpy(), **TOL[0])
    lin.close()


@pytest.mark.parametrize("frames,rank,form", [(1, 16, ("few rows", 64, 4)), (1, 64, ("few rows", 64, 4)), (12, 64, ("few rows", 256, 2))])
def test_lora_linear_several_slab_groups_through_the_shortest_ring(frames, rank, form):
    """The few-row kernel's ring is shortest where a group of eight slabs and the exchange of partial sums take the
    rest of the shared memory; further groups of slabs then follow through those stages, x from one thread and the slabs
    from another.  Eight adapters on every frame: one to eight groups per tile.  Several calls in a row, against float64
    sums of the same bf16 inputs; tolerance as for the other linears."""
    import torch
    from paper_2507_14959_b200 import binding
    k_in, n_out, tokens, n_ad, rows = 3072, 768, 197, 16, frames * 197
    check_form(k_in, n_out, rows, 2, True, form)
    gen = torch.Generator(device="cuda").manual_seed(frames + rank)

    def draw(shape, std):
        return (torch.randn(shape, generator=gen, device="cuda") * std).bfloat16()
    x, res, w, b = draw((rows, k_in), 1.0), draw((rows, n_out), 1.0), draw((k_in, n_out), 0.02), draw((n_out,), 0.02)
    A = [draw((k_in, rank), 0.02) for _ in range(n_ad)]
    B = [draw((rank, n_out), 0.02) for _ in range(n_ad)]
    sets = [list(range(f % 2, n_ad, 2)) for f in range(frames)]
    off, ids = wl.sets_to_csr(sets)
    host = lambda t: t.float().cpu().numpy()  # noqa: E731
    lin = binding.Linear(host(w), host(b), max_adapters=n_ad, max_rank=rank, max_set=8, max_frames=frames, tokens=tokens, epilogue=2)
    for a in range(n_ad):
        lin.register(a, rank, 1.0, host(A[a]), host(B[a]))
    y = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    for _ in range(4):
        lin.forward(x, frames, off, ids, y, residual=res)
    assert lin.status() == 0
    want = x.double() @ w.double() + b.double() + res.double()
    for f, s in enumerate(sets):
        r = slice(f * tokens, (f + 1) * tokens)
        for a in s:
            want[r] += (x[r].double() @ A[a].double()) @ B[a].double()
    np.testing.assert_allclose(to_np(y), want.cpu().numpy(), **TOL[0])
    lin.close()


@pytest.mark.parametrize("frames,tokens,rank,n_ad,largest", [(300, 197, 32, 24, (33, 48)), (300, 197, 64, 24, (65, 96)), (1240, 32, 64, 40, (97, 160))])
def test_lora_linear_of_long_slab_lists_on_full_grids(frames, tokens, rank, n_ad, largest):
    """Three shrink CTAs per SM, sets of 0 to 8 adapters: row-tile pairs of up to 48 and 96 slabs, of which a tile's own
    masks and scales fit the prepared list or do not, and pairs of more slabs than are listed.  Twice, so that a slab
    left unwritten for a tile that does not use it would show; against float64 sums of the same bf16 inputs, tolerance as
    for the other linears."""
    import torch
    from paper_2507_14959_b200 import binding
    k_in, n_out, rows = 192, 256, frames * tokens
    gen = torch.Generator(device="cuda").manual_seed(frames + rank)

    def draw(shape, std):
        return (torch.randn(shape, generator=gen, device="cuda") * std).bfloat16()
    x, w, b = draw((rows, k_in), 1.0), draw((k_in, n_out), 0.02), draw((n_out,), 0.02)
    A = [draw((k_in, rank), 0.02) for _ in range(n_ad)]
    B = [draw((rank, n_out), 0.02) for _ in range(n_ad)]
    host = lambda t: t.float().cpu().numpy()  # noqa: E731
    lin = binding.Linear(host(w), host(b), max_adapters=n_ad, max_rank=rank, max_set=8, max_frames=frames, tokens=tokens, epilogue=0)
    for a in range(n_ad):
        lin.register(a, rank, 1.0, host(A[a]), host(B[a]))
    y = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    g = np.random.default_rng(rows + rank)
    for _ in range(2):
        sets = [sorted(int(a) for a in g.choice(n_ad, size=int(g.integers(0, 9)), replace=False)) for _ in range(frames)]
        union = [set().union(*sets[r // tokens:min(r + 255, rows - 1) // tokens + 1]) for r in range(0, rows, 256)]
        assert largest[0] <= max(len(u) for u in union) * rank // 16 <= largest[1]
        off, ids = wl.sets_to_csr(sets)
        lin.forward(x, frames, off, ids, y)
        assert lin.status() == 0
        want = x.double() @ w.double() + b.double()
        for f, s in enumerate(sets):
            r = slice(f * tokens, (f + 1) * tokens)
            for a in s:
                want[r] += (x[r].double() @ A[a].double()) @ B[a].double()
        np.testing.assert_allclose(to_np(y), want.cpu().numpy(), **TOL[0])
    lin.close()


@pytest.mark.parametrize("frames,form", [(1, ("few rows", 64, 4)), (2, ("few rows", 128, 4)), (4, ("few rows", 128, 2)), (8, ("few rows", 192, 2)),
                                         (12, ("few rows", 256, 2)), (33, ("pair", 192, 1))])
def test_lora_intermediate_of_a_split_k_is_not_rounded_share_by_share(frames, form):
    """t = s x A whose K shares cancel: x is 64 times as large on one part of each half of K and the halves take most of it
    back.  W = 0, so the output is t B.  Root mean square of the error against float64, relative to that of the
    output: one rounding of t and one of the output to bf16, 2^-9 each at most, give below 2^-8; shares rounded
    by themselves would leave about 64 * 2^-9."""
    import torch
    from paper_2507_14959_b200 import binding
    k_in, n_out, tokens, rank, rows = 3072, 768, 197, 16, frames * 197
    check_form(k_in, n_out, rows, 2, True, form)        # the last one: shrink with K in two
    gen = torch.Generator(device="cuda").manual_seed(frames)

    def draw(shape, std):
        return (torch.randn(shape, generator=gen, device="cuda") * std).bfloat16()
    x, A, B = draw((rows, k_in), 1.0), draw((k_in, rank), 0.02), draw((rank, n_out), 0.02)
    big = draw((rows, 768), 64.0)
    A[1536:2304] = A[:768]
    x[:, :768], x[:, 1536:2304] = big, (x[:, 1536:2304].float() - big.float()).bfloat16()
    lin = binding.Linear(np.zeros((k_in, n_out), np.float32), np.zeros(n_out, np.float32), max_adapters=1, max_rank=rank, max_set=1,
                         max_frames=frames, tokens=tokens, epilogue=2)
    lin.register(0, rank, 1.0, A.float().cpu().numpy(), B.float().cpu().numpy())
    y = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    off, ids = wl.sets_to_csr([[0]] * frames)
    lin.forward(x, frames, off, ids, y, residual=torch.zeros_like(y))
    assert lin.status() == 0
    want = (x.double() @ A.double()) @ B.double()
    assert float((y.double() - want).norm() / want.norm()) < 2.0 ** -8
    lin.close()


@pytest.mark.parametrize("k_in,n_out,frames", [(3072, 768, 1), (3072, 768, 4), (3072, 768, 8), (3072, 768, 12), (3072, 768, 15),
                                               (2048, 512, 24), (4096, 1024, 8)])
def test_lora_intermediate_of_a_split_k_is_held_in_more_than_16_bits(k_in, n_out, frames):
    """W = 0 and no cancellation: the output is t B.  The shares of t carry 16 significant bits, so the error is that of the one
    rounding of the output to bf16.  Rounding to 8 significant bits errs by at most 2^-8 / m relative to a value of mantissa m in [1, 2),
    uniformly; over mantissas of equal probability per logarithm E[1/m^2] = 3 / (8 ln 2), and the root mean square is 2^-8 * sqrt(E / 3) =
    2^-8 * 0.425.  A t rounded to bf16 would add as much again in the sum over its 16 ranks, 2^-8 * 0.60 in all.  The limit lies between."""
    import torch
    from paper_2507_14959_b200 import binding
    tokens, rank, rows = 197, 16, frames * 197
    assert binding.linear_kernel(k_in, n_out, rows, 2, True)[2] > 1
    gen = torch.Generator(device="cuda").manual_seed(frames)
    x = torch.randn((rows, k_in), generator=gen, device="cuda").bfloat16()
    A = (torch.randn((k_in, rank), generator=gen, device="cuda") * 0.02).bfloat16()
    B = (torch.randn((rank, n_out), generator=gen, device="cuda") * 0.02).bfloat16()
    lin = binding.Linear(np.zeros((k_in, n_out), np.float32), np.zeros(n_out, np.float32), max_adapters=1, max_rank=rank, max_set=1,
                         max_frames=frames, tokens=tokens, epilogue=2)
    lin.register(0, rank, 1.0, A.float().cpu().numpy(), B.float().cpu().numpy())
    y = torch.full((rows, n_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    off, ids = wl.sets_to_csr([[0]] * frames)
    lin.forward(x, frames, off, ids, y, residual=torch.zeros_like(y))
    assert lin.status() == 0
    want = (x.double() @ A.double()) @ B.double()
    error = float((y.double() - want).norm() / want.norm())
    assert error < 0.5 * 2.0 ** -8, error * 2.0 ** 8
    lin.close()


@pytest.mark.parametrize("frames,tokens,heads", [(1, 1, 1), (2, 16, 3), (1, 17, 2), (3, 49, 1), (1, 208, 12), (49, 33, 1),     # a few pairs
                                                 (50, 33, 1), (60, 1, 1), (20, 197, 3), (17, 208, 4), (13, 129, 12)])           # the pipelined kernel
def test_attention_of_one_key_block_on_both_sides_of_the_pair_limit(frames, tokens, heads):
    """Up to 208 tokens: few (frame, head) pairs run as one CTA per 16 query rows, more as the pipelined kernel (limit:
    49 pairs on 148 SMs); token counts at the edges of 16-key groups and query tiles.  Against the oracle."""
    import torch
    from paper_2507_14959_b200 import binding
    d = heads * 64
    qkv = wl.normal((frames * tokens, 3 * d), 1.0, "attn_gpu_few", frames, tokens, heads)
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    binding.attention(to_dev(qkv, 0), od, frames, tokens, heads, 0)
    torch.cuda.synchronize()
    got = to_np(od)
    for f in sorted({0, frames // 2, frames - 1}):
        want = po.attention(qkv[f * tokens:(f + 1) * tokens].astype(np.float64), heads)
        np.testing.assert_allclose(got[f * tokens:(f + 1) * tokens], want, **TOL[0])


@pytest.mark.parametrize("frames,tokens,heads", [(18, 197, 3), (1, 300, 2), (2, 577, 1)])
def test_attention_rows_whose_first_scores_are_far_below_the_largest(frames, tokens, heads):
    """The tensor-memory kernels take a row's exponentials relative to the maximum of its first 16 scores; a row with a
    score far above it is computed again with its true maximum.  Here keys 0..15 are zero and a later key of every row
    in the first frame's first head scores about 2000, in the last frame's last head moderate scores stay as they are: both
    kinds of rows against the oracle, in one launch."""
    import torch
    from paper_2507_14959_b200 import binding
    d = heads * 64
    qkv = wl.normal((frames * tokens, 3 * d), 1.0, "attn_gpu_far", frames, tokens, heads)
    qkv[:tokens, :64] = 16.0                                   # queries of frame 0, head 0
    qkv[:16, d:d + 64] = 0.0                                   # its keys 0..15
    qkv[tokens - 40, d:d + 64] = 16.0                          # score 16 * 16 * 64 / 8 = 2048
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    binding.attention(to_dev(qkv, 0), od, frames, tokens, heads, 0)
    torch.cuda.synchronize()
    got = to_np(od)
    for f in sorted({0, frames - 1}):
        want = po.attention(qkv[f * tokens:(f + 1) * tokens].astype(np.float64), heads)
        np.testing.assert_allclose(got[f * tokens:(f + 1) * tokens], want, **TOL[0])


@pytest.mark.parametrize("far", [50, 300, 540, 560, 700])
@pytest.mark.parametrize("frames,tokens,heads", [(18, 197, 3), (1, 300, 2), (2, 577, 1)])
def test_attention_rows_over_the_range_of_their_reference(frames, tokens, heads, far):
    """Rows whose later scores (q k) lie 50 to 700 above those of keys 0..15: exponentials up to 2^100 relative to the
    reference on one side of 550, computed again on the other.  Six far keys of nearby scores, in both shares of the key columns
    and in every key block; every other query row of the first frame's first head and all rows of the last frame's
    last head.  All rows of both frames against the oracle."""
    import torch
    from paper_2507_14959_b200 import binding
    d = heads * 64
    qkv = wl.normal((frames * tokens, 3 * d), 1.0, "attn_gpu_range", frames, tokens, heads)
    for f, h, rows in ((0, 0, slice(0, tokens, 2)), (frames - 1, heads - 1, slice(0, tokens))):
        x = qkv[f * tokens:(f + 1) * tokens]
        q, k = slice(h * 64, h * 64 + 64), slice(d + h * 64, d + h * 64 + 64)
        x[rows, q] = 1.0
        x[:16, k] = 0.0
        for i, key in enumerate((17, tokens // 3, tokens // 2, tokens // 2 + 30, tokens - 60, tokens - 2)):
            x[key, k] = far / 64 - i % 3 / 32          # q k = far, far - 2, far - 4 (bf16 steps at most)
    qkv = wl.round_bf16(qkv)
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    binding.attention(to_dev(qkv, 0), od, frames, tokens, heads, 0)
    torch.cuda.synchronize()
    got = to_np(od)
    for f in sorted({0, frames - 1}):
        want = po.attention(qkv[f * tokens:(f + 1) * tokens].astype(np.float64), heads)
        np.testing.assert_allclose(got[f * tokens:(f + 1) * tokens], want, **TOL[0])


@pytest.mark.parametrize("frames,tokens,heads", [(830, 17, 12), (450, 209, 12)])
def test_attention_rows_computed_again_in_late_tiles(frames, tokens, heads):
    """More tiles per CTA than a thread has bits for them: rows out of range in early, middle and last tiles.  Frames with
    such rows and their neighbours against the oracle."""
    import torch
    from paper_2507_14959_b200 import binding
    d = heads * 64
    gen = torch.Generator(device="cuda").manual_seed(tokens)
    qkv = torch.randn((frames, tokens, 3, heads, 64), generator=gen, device="cuda")
    far = (0, frames // 3, frames // 2, frames - 1)
    for f in far:
        qkv[f, 3::5, 0, f % heads] = 1.0
        qkv[f, :16, 1, f % heads] = 0.0
        qkv[f, tokens - 1, 1, f % heads] = 12.0
    qkv = qkv.bfloat16().reshape(frames * tokens, 3 * d)
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    binding.attention(qkv, od, frames, tokens, heads, 0)
    torch.cuda.synchronize()
    assert torch.isfinite(od.float()).all()
    for f in sorted({g for f in far for g in (f, min(f + 1, frames - 1))}):
        rows = slice(f * tokens, (f + 1) * tokens)
        np.testing.assert_allclose(to_np(od[rows]), po.attention(to_np(qkv[rows]), heads), **TOL[0])


@pytest.mark.parametrize("exponent", [40, 60, 100])
@pytest.mark.parametrize("frames,tokens,heads", [(18, 197, 3), (2, 577, 1)])
def test_attention_of_large_values_under_large_terms(frames, tokens, heads, exponent):
    """Terms of 2^92 relative to the reference (scores q k = 512 above those of keys 0..15) times values of 2^40 to 2^100:
    the unnormalised output overflows fp32, the quotient does not.  One value column per half of the head is large.
    Relative to the oracle, as for the other attention cases."""
    import torch
    from paper_2507_14959_b200 import binding
    d, scale = heads * 64, 2.0 ** exponent
    qkv = wl.normal((frames * tokens, 3 * d), 1.0, "attn_gpu_large", frames, tokens, heads)
    qkv[:tokens, :64] = 1.0
    qkv[:16, d:d + 64] = 0.0
    qkv[tokens - 40, d:d + 64] = 8.0
    qkv[tokens - 90, d:d + 64] = 8.0 - 1.0 / 32
    qkv = wl.round_bf16(qkv)
    large = (2 * d + 5, 2 * d + 50)
    sent = qkv.copy()
    sent[:tokens, large] *= scale
    od = torch.full((frames * tokens, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    binding.attention(to_dev(sent, 0), od, frames, tokens, heads, 0)
    torch.cuda.synchronize()
    got = to_np(od)[:tokens]
    got[:, (5, 50)] /= scale
    np.testing.assert_allclose(got, po.attention(qkv[:tokens].astype(np.float64), heads), **TOL[0])


def test_linear_alignment_of_operands():
    """x, y and a residual that is added must be 16-byte aligned, on few rows and on many, whatever the kernel; a residual that is
    not used may lie anywhere."""
    import torch
    from paper_2507_14959_b200 import binding
    for k_in, n_out, frames in ((64, 128, 1), (64, 128, 300), (1536, 768, 1), (768, 768, 60)):
        rows = frames * 197
        off, ids = np.zeros(frames + 1, np.int32), np.zeros(0, np.int32)
        wide = torch.randn((rows * max(k_in, n_out) + 8,), device="cuda").bfloat16()
        x, res = wide[:rows * k_in].view(rows, k_in), wide[:rows * n_out].view(rows, n_out)
        odd_x, odd_res = wide[1:1 + rows * k_in].view(rows, k_in), wide[1:1 + rows * n_out].view(rows, n_out)
        out = torch.zeros((rows * n_out + 8,), device="cuda", dtype=torch.bfloat16)
        y, odd_y = out[:rows * n_out].view(rows, n_out), out[1:1 + rows * n_out].view(rows, n_out)
        w = wl.normal((k_in, n_out), 0.02, "align", k_in)
        for epi in (0, 2):
            lin = binding.Linear(w, np.zeros(n_out, np.float32), max_adapters=1, max_rank=16, max_set=1, max_frames=frames, tokens=197, epilogue=epi)
            for a in ((odd_x, res, y), (x, res, odd_y)) + (((x, odd_res, y),) if epi == 2 else ()):
                with pytest.raises(binding.PolymorphError) as e:
                    lin.forward(a[0], frames, off, ids, a[2], residual=a[1])
                assert e.value.code == binding.PM_ERR_CUDA
            lin.forward(x, frames, off, ids, y, residual=odd_res if epi == 0 else res)
            assert lin.status() == 0
            want = x.float() @ torch.from_numpy(w).cuda() + (res.float() if epi == 2 else 0)
            np.testing.assert_allclose(to_np(y), want.double().cpu().numpy(), **TOL[0])
            lin.close()
