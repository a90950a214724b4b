"""pm_select (Algorithm 2 on the device) against the oracle's literal Algorithm 2: bit-exact adapter
sets over several chained time steps, on disjoint and overlapping class->adapter tables."""
import numpy as np
import pytest

import workloads as wl
from oracle import polymorph_oracle as po

pytestmark = pytest.mark.gpu


def small_model(contexts, accs, n_classes, max_frames):
    from paper_2507_14959_b200 import binding
    spec = wl.ModelSpec(img=32, d=64, heads=1, mlp=64, n_classes=n_classes, layers=1)
    bb = wl.make_backbone("select_gpu", spec)
    m = binding.Model(img=32, d=64, layers=1, heads=1, mlp=64, n_classes=n_classes, backbone=bb,
                      max_adapters=len(contexts), max_rank=16, max_set=4, max_frames=max_frames)
    for a, (c, ac) in enumerate(zip(contexts, accs)):
        m.register_adapter(a, rank=1, scale=1.0, A=[None] * 4, B=[None] * 4, class_ids=c,
                           head_w=np.zeros((64, len(c)), np.float32), head_b=np.zeros(len(c), np.float32),
                           acc=ac)
    return m


@pytest.mark.parametrize("n_ctx,n_labels,max_size,overlap,seed", [
    (8, 16, 4, False, 0), (12, 40, 6, True, 1), (70, 200, 9, True, 2), (64, 800, 25, True, 3),
    (5, 33, 3, False, 4)])
@pytest.mark.parametrize("context_copy", [False, True])
def test_select_chained_steps(n_ctx, n_labels, max_size, overlap, seed, context_copy):
    import torch
    ctxs, accs = wl.random_cover_table(seed, n_ctx, n_labels, max_size, overlap)
    keep = [i for i, c in enumerate(ctxs) if len(c)]
    ctxs, accs = [ctxs[i] for i in keep], [accs[i] for i in keep]
    F = 37
    m = small_model(ctxs, accs, n_labels, F)
    tau = 0.6
    m.set_cover(tau)
    g = wl.rng_for("select_scores", seed, context_copy)
    nw = (n_labels + 31) // 32
    labels = torch.zeros((F, nw), dtype=torch.int32, device="cuda")
    cap = F * len(ctxs)
    bufs = [(torch.zeros(F + 1, dtype=torch.int32, device="cuda"),
             torch.full((cap,), -1, dtype=torch.int32, device="cuda")) for _ in range(2)]
    Y_prev = [None] * F
    S_prev = [None] * F
    cur = None
    for step in range(5):
        scores = np.full((F, n_labels), 0.1, dtype=np.float32)
        for f in range(F):
            if step > 0 and g.random() < 0.5:
                scores[f] = last[f]                     # unchanged frame: Y_t = Y_{t-1}
                continue
            on = g.choice(n_labels, size=int(g.integers(0, 5)), replace=False)
            scores[f, on] = 0.9
            scores[f, g.integers(0, n_labels)] = 0.5    # exactly at the threshold: not a label
        last = scores
        want = []
        for f in range(F):
            Y = po.labels_from_scores(scores[f], 0.5)
            want.append(po.detect_contexts(Y, Y_prev[f], ctxs, accs, tau, S_prev[f], context_copy))
            Y_prev[f], S_prev[f] = Y, want[-1]
        nxt = bufs[step % 2]
        m.select(torch.from_numpy(scores).cuda(), 0.5, context_copy, step > 0, labels,
                 None if cur is None else cur[0], None if cur is None else cur[1], nxt[0], nxt[1])
        assert m.status() == 0
        off, ids = wl.sets_to_csr(want)
        np.testing.assert_array_equal(nxt[0].cpu().numpy(), off)
        np.testing.assert_array_equal(nxt[1].cpu().numpy()[:len(ids)], ids)
        # the label bit sets written back are Y_t
        lab = labels.cpu().numpy().view(np.uint32)
        for f in range(F):
            bits = {k for k in range(n_labels) if (lab[f, k // 32] >> (k % 32)) & 1}
            assert bits == Y_prev[f]
        cur = nxt
    m.close()


def test_select_capacity_overflow_sets_status():
    import torch
    from paper_2507_14959_b200 import binding
    ctxs = [np.array([k], np.int32) for k in range(6)]
    accs = [np.ones(1, np.float32) for _ in range(6)]
    m = small_model(ctxs, accs, 6, 2)
    m.set_cover(0.5)
    scores = torch.ones((2, 6), device="cuda")
    noff = torch.zeros(3, dtype=torch.int32, device="cuda")
    nids = torch.zeros(7, dtype=torch.int32, device="cuda")       # 12 needed
    m.select(scores, 0.5, False, False, None, None, None, noff, nids)
    assert m.status() == binding.PM_ERR_CAPACITY
    assert m.status() == 0                                         # cleared after reading
    np.testing.assert_array_equal(noff.cpu().numpy(), [0, 6, 12])
    m.close()


def test_select_needs_cover_table():
    import torch
    from paper_2507_14959_b200 import binding
    ctxs = [np.array([0, 1], np.int32)]
    m = small_model(ctxs, [np.ones(2, np.float32)], 4, 1)
    with pytest.raises(binding.PolymorphError) as e:
        m.select(torch.zeros((1, 4), device="cuda"), 0.5, False, False, None, None, None,
                 torch.zeros(2, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda"))
    assert e.value.code == binding.PM_ERR_STATE
    m.close()


@pytest.mark.parametrize("static", [False, True])
def test_select_frame_count_changes_between_calls(static):
    """One handle (or the one static scratch array), batches of 37, then 8, then 37 frames: the state
    the kernel keeps between launches must not depend on the batch size."""
    import torch
    from paper_2507_14959_b200 import binding
    ctxs, accs = wl.random_cover_table(5, 40, 120, 7, True)
    keep = [i for i, c in enumerate(ctxs) if len(c)]
    ctxs, accs = [ctxs[i] for i in keep], [accs[i] for i in keep]
    n_labels, tau, n_ad = 120, 0.6, len(ctxs)
    m = small_model(ctxs, accs, n_labels, 37)
    m.set_cover(tau)
    if static:
        import test_zz_no_alloc as tz
        first, provider = tz.cover_tables(ctxs, accs, n_labels, tau)
        first_d, prov_d = torch.from_numpy(first).cuda(), torch.from_numpy(provider.view(np.int64)).cuda()
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
    g = wl.rng_for("select_varying_frames", int(static))
    for F in (37, 8, 37, 1, 20):
        scores = np.full((F, n_labels), 0.1, dtype=np.float32)
        for f in range(F):
            scores[f, g.choice(n_labels, size=int(g.integers(1, 6)), replace=False)] = 0.9
        want = [po.detect_contexts(po.labels_from_scores(scores[f], 0.5), None, ctxs, accs, tau, None, False)
                for f in range(F)]
        noff = torch.full((F + 1,), -7, dtype=torch.int32, device="cuda")
        nids = torch.full((F * n_ad,), -1, dtype=torch.int32, device="cuda")
        sd = torch.from_numpy(scores).cuda()
        if static:
            binding.select_static(sd, n_ad, 0.5, False, False, None, None, None, first_d, prov_d, noff, nids,
                                  status_out=status)
            torch.cuda.synchronize()
            assert int(status.item()) == 0
        else:
            m.select(sd, 0.5, False, False, None, None, None, noff, nids)
            assert m.status() == 0
        off, ids = wl.sets_to_csr(want)
        np.testing.assert_array_equal(noff.cpu().numpy(), off)
        np.testing.assert_array_equal(nids.cpu().numpy()[:len(ids)], ids)
    m.close()


def test_select_reports_bad_previous_lists():
    """Ids outside the adapter range in S_{t-1} (or a malformed offset pair) are skipped and reported
    in the status word; the other frames' results are unaffected."""
    import torch
    from paper_2507_14959_b200 import binding
    ctxs = [np.array([2 * a, 2 * a + 1], np.int32) for a in range(6)]
    accs = [np.ones(2, np.float32) for _ in range(6)]
    m = small_model(ctxs, accs, 12, 3)
    m.set_cover(0.5)
    scores = np.full((3, 12), 0.1, np.float32)
    scores[0, 0] = scores[1, 5] = scores[2, 11] = 0.9
    sd = torch.from_numpy(scores).cuda()
    labels = torch.zeros((3, 1), dtype=torch.int32, device="cuda")
    noff = torch.zeros(4, dtype=torch.int32, device="cuda")
    nids = torch.full((18,), -1, dtype=torch.int32, device="cuda")
    for prev_off, prev_ids in (([0, 1, 2, 3], [0, 99, 5]), ([0, 1, 2, 3], [0, -4, 5]), ([0, 1, 100, 3], [0, 2, 5])):
        labels.zero_()
        po_ = torch.tensor(prev_off, dtype=torch.int32, device="cuda")
        pi_ = torch.tensor(prev_ids, dtype=torch.int32, device="cuda")
        m.select(sd, 0.5, True, True, labels, po_, pi_, noff, nids)
        assert m.status() == binding.PM_ERR_ARG
        assert m.status() == 0
        # frame 0 keeps {0} (copy: label 0 is covered by adapter 0); a bad previous set counts as empty,
        # so the greedy branch picks the provider of the frame's label
        assert noff.cpu().tolist() == [0, 1, 2, 3]
        assert nids.cpu().tolist()[:3] == [0, 2, 5]
    m.close()


def test_select_counts_eq7_eq8_on_the_device():
    import torch
    ctxs, accs = wl.random_cover_table(9, 20, 60, 5, True)
    keep = [i for i, c in enumerate(ctxs) if len(c)]
    ctxs, accs = [ctxs[i] for i in keep], [accs[i] for i in keep]
    F, K, tau = 11, 60, 0.6
    m = small_model(ctxs, accs, K, F)
    m.set_cover(tau)
    m.metrics_reset()
    g = wl.rng_for("select_metrics")
    labels = torch.zeros((F, 2), dtype=torch.int32, device="cuda")
    bufs = [(torch.zeros(F + 1, dtype=torch.int32, device="cuda"),
             torch.full((F * len(ctxs),), -1, dtype=torch.int32, device="cuda")) for _ in range(2)]
    seqs = [[] for _ in range(F)]
    Y_prev, S_prev = [None] * F, [None] * F
    scores = None
    for step in range(7):
        new = np.full((F, K), 0.1, np.float32)
        for f in range(F):
            if step > 0 and g.random() < 0.5:
                new[f] = scores[f]
            else:
                new[f, g.choice(K, size=int(g.integers(0, 4)), replace=False)] = 0.9
        scores = new
        for f in range(F):
            Y = po.labels_from_scores(scores[f], 0.5)
            S = po.detect_contexts(Y, Y_prev[f], ctxs, accs, tau, S_prev[f], True)
            seqs[f].append(S)
            Y_prev[f], S_prev[f] = Y, S
        prev, nxt = bufs[(step + 1) % 2], bufs[step % 2]
        m.select(torch.from_numpy(scores).cuda(), 0.5, True, step > 0, labels, prev[0], prev[1], nxt[0], nxt[1])
    frames, contexts, switches = m.metrics_read()
    assert m.status() == 0
    assert frames == 7 * F
    assert contexts / frames == pytest.approx(sum(po.avg_coverage(s) * len(s) for s in seqs) / (7 * F))
    assert switches == sum(po.switch_penalty(s) for s in seqs)
    m.metrics_reset()
    assert m.metrics_read() == (0, 0, 0)
    m.close()


@pytest.mark.parametrize("n_frames,n_labels,n_ctx", [(1, 1025, 3), (2049, 40, 65), (4096, 33, 130)])
def test_select_at_the_edges_of_its_passes(n_frames, n_labels, n_ctx):
    """More than 32 label words (a second pass over a frame's scores), more frames than one pass of the emission
    takes (2048), one to three mask words per frame: sets against the oracle, exactly."""
    import torch
    ctxs, accs = wl.random_cover_table(21, n_ctx, n_labels, 4, True)
    m = small_model(ctxs, accs, n_labels, n_frames)
    m.set_cover(0.6)
    g = wl.rng_for("select_edges", n_frames)
    scores = np.full((n_frames, n_labels), 0.1, np.float32)
    for f in range(n_frames):
        scores[f, g.choice(n_labels, size=int(g.integers(0, 4)), replace=False)] = 0.9
    scores[-1, -1] = 0.9                                     # the last label of the last frame
    off = torch.zeros(n_frames + 1, dtype=torch.int32, device="cuda")
    ids = torch.full((n_frames * n_ctx,), -1, dtype=torch.int32, device="cuda")
    m.select(torch.from_numpy(scores).cuda(), 0.5, False, False, None, None, None, off, ids)
    assert m.status() == 0
    o, i = off.cpu().numpy(), ids.cpu().numpy()
    for f in range(n_frames):
        want = po.detect_contexts(po.labels_from_scores(scores[f], 0.5), None, ctxs, accs, 0.6, None, False)
        assert sorted(want) == list(i[o[f]:o[f + 1]])
    m.close()


@pytest.mark.parametrize("n_frames,n_labels,n_ctx", [(1, 80, 200), (3, 33, 16), (70, 800, 200), (300, 1100, 70)])
@pytest.mark.parametrize("density", [0.02, 0.3, 1.0])
def test_select_with_few_and_many_labels_per_frame(n_frames, n_labels, n_ctx, density):
    """Frames of a few labels, whose words the lanes walk side by side, and of hundreds, which are taken word by word; batches of one
    and of several frames per thread of the emission.  Two steps (the second with context copy) against the oracle, exactly."""
    import torch
    ctxs, accs = wl.random_cover_table(33, n_ctx, n_labels, 12, True)
    m = small_model(ctxs, accs, n_labels, n_frames)
    m.set_cover(0.6)
    g = wl.rng_for("select_density", n_frames, n_labels, density)
    nw = (n_labels + 31) // 32
    labels = torch.zeros((n_frames, nw), dtype=torch.int32, device="cuda")
    lists = [(torch.zeros(n_frames + 1, dtype=torch.int32, device="cuda"),
              torch.full((n_frames * n_ctx,), -1, dtype=torch.int32, device="cuda")) for _ in range(2)]
    keep = g.random((n_frames, n_labels)) < density
    prev = [(None, None)] * n_frames
    for step in range(2):
        if step == 1:
            keep &= g.random((n_frames, n_labels)) < 0.9           # mostly covered by the sets in use
            keep[::3] = g.random(keep[::3].shape) < density
        scores = np.where(keep, 0.9, 0.1).astype(np.float32)
        old, new = lists[(step + 1) % 2], lists[step % 2]
        m.select(torch.from_numpy(scores).cuda(), 0.5, True, step > 0, labels, old[0], old[1], new[0], new[1])
        assert m.status() == 0
        o, i = new[0].cpu().numpy(), new[1].cpu().numpy()
        for f in range(n_frames):
            Y = po.labels_from_scores(scores[f], 0.5)
            want = po.detect_contexts(Y, prev[f][0], ctxs, accs, 0.6, prev[f][1], True)
            assert sorted(want) == list(i[o[f]:o[f + 1]]), (step, f)
            prev[f] = (Y, want)
    m.close()
