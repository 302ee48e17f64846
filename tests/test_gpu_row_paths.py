"""The row kernels' layouts and cuts at the sizes where they change, bit for
bit against the CPU oracle (tokens, windows, stored rows): rows per SM and
support sizes around the lines between the layouts, top-p cuts that the ids
with t > -22 leave open, rows that start off 16-byte boundaries, trees with
more groups than warps, and stored rows read back at odd capacities.

Every comparison is exact: the sampled integers and the fp32 probabilities
are defined operation by operation.
"""

import ctypes

import numpy as np
import pytest
import torch

from lockstep import Lockstep, TreeLockstep, config_of, device_logits, tree_inputs
from paper_2603_18599_gb300 import sjd
from paper_2603_18599_gb300 import workloads as wlm

pytestmark = pytest.mark.gpu

BASE = wlm.workloads()["b1w16v8192_f32"]


def run(w, steps, **kw):
    ls = Lockstep(w, **kw)
    c, u = ls.start_from_logits()
    ls.step(c, u)
    for t in range(1, steps):
        c, u, _, _ = ls.inputs(t)
        ls.step(c, u)
    return ls


@pytest.mark.parametrize("batch,window,vocab,top_k,top_p", [
    (8, 19, 640, 200, 1.0),      # 152 rows: one row per SM, 512 threads
    (3, 51, 640, 200, 1.0),      # 153 rows: two rows per SM, 256 threads
    (16, 19, 512, 129, 0.97),    # 304 rows, the smallest support beyond the narrow arrays
    (5, 61, 512, 200, 0.97),     # 305 rows with top-p: the narrow layout
    (5, 61, 512, 200, 1.0),      # 305 rows without: more rows than one wave of the wide one
    (3, 51, 2200, 2048, 1.0),    # a longer support with 256 threads
    (3, 51, 2200, 2049, 1.0),    # and one above
    (3, 51, 2600, 2500, 1.0),    # 256 threads beyond that
    (2, 4, 4088, 100, 0.9),      # few rows, small supports: 128 threads below 4096 ids,
    (2, 4, 4096, 100, 0.9),      # then 512
    (2, 4, 4096, 1, 1.0),
    (3, 51, 4096, 20, 0.9),      # and 256
    (16, 20, 760, 200, 1.0),     # 320 rows: 128 threads below 768 ids,
    (16, 20, 768, 200, 1.0),     # 256 from there
    (10, 31, 16384, 60, 0.95),   # long rows with top-p and a few rows too many
    (3, 51, 640, 128, 1.0),      # kept rows that fit the narrow arrays
])
def test_layouts_at_their_lines(batch, window, vocab, top_k, top_p):
    run(BASE.scaled(batch=batch, window=window, vocab=vocab, hi=vocab, top_k=top_k, top_p=top_p, sigma=0.6,
                    q_noise=0.4, dtype="bf16"), 2)


@pytest.mark.parametrize("vocab,lo,hi", [(4096, 0, 4096), (8200, 3, 8195)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_top_p_cut_left_open_by_the_large_weights(vocab, lo, hi, dtype):
    """Two equal maxima and everything else between t = -33 and -26, top-p
    0.5: whether the first id alone reaches half of the total depends on the
    small weights, so the cut is open and the row is streamed again."""
    w = BASE.scaled(batch=2, window=8, vocab=vocab, lo=lo, hi=hi, top_k=2000, top_p=0.5, cfg_scale=1.0, dtype=dtype)
    ls = Lockstep(w)
    rng = np.random.default_rng(11)

    def rows():
        x = np.full((2, 8, vocab), wlm.OUT_OF_RANGE_POISON, np.float32)
        x[:, :, lo:hi] = rng.uniform(-33.0, -26.0, (2, 8, hi - lo))
        for b in range(2):
            for j in range(8):
                x[b, j, rng.choice(np.arange(lo, hi), 2, replace=False)] = 0.0
        return wlm.bf16_round(x) if dtype == "bf16" else x

    c, q = rows(), rows()
    ls.start_from_logits((c, c, q, q))
    ls.step(c, c)
    c = rows()
    ls.step(c, c)
    assert ls.ctx.row_path() == 1 and ls.ctx.stats()[4] > 0


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("vocab,lo,hi,top_k", [
    (1003, 0, 1003, 300),     # both ends of the rows
    (1001, 7, 998, 300),      # inside them
    (999, 500, 503, 0),       # less than a chunk
    (1013, 8, 16, 0),         # one chunk, starting anywhere
    (10007, 5, 9001, 2000),
])
@pytest.mark.parametrize("fused", [True, False])
def test_rows_off_16_byte_boundaries(vocab, lo, hi, top_k, dtype, fused):
    run(BASE.scaled(batch=2, window=5, vocab=vocab, lo=lo, hi=hi, top_k=top_k, top_p=0.95, sigma=1.0, dtype=dtype), 2,
        fused=fused)


@pytest.mark.parametrize("dtype,off_c,off_u",
                         [("bf16", k, k) for k in range(8)] + [("f32", k, k) for k in range(4)] +
                         [("bf16", 0, 8), ("bf16", 0, 1), ("bf16", 5, 2), ("f32", 1, 5), ("f32", 0, 3), ("f32", 2, 1)])
@pytest.mark.parametrize("vocab", [1003, 1024])
def test_logits_inside_a_larger_buffer(vocab, dtype, off_c, off_u):
    """Logit tensors that begin off_c / off_u elements into an allocation (the
    elements around them hold a poison value), alike or not, give the bits of
    tensors of their own. The streaming kernel takes rows off 16-byte
    boundaries where cond and uncond lie alike, and rows on them."""
    w = BASE.scaled(batch=2, window=5, vocab=vocab, hi=vocab, top_k=300, sigma=1.0, dtype=dtype)
    per = 8 if dtype == "bf16" else 4
    streams = (off_c - off_u) % per == 0 if vocab == 1003 else off_c % per == 0 and off_u % per == 0
    dev = torch.device("cuda", torch.cuda.current_device())
    a, b = sjd.SJD(config_of(w), dev), sjd.SJD(config_of(w), dev)
    for t in range(3):
        c, u, _, _ = wlm.logits_step(w, t)
        dc, du = device_logits(w, (c, u), dev)
        ra = a.step(dc, du)
        inner = []
        for x, off in ((dc, off_c), (du, off_u)):
            buf = torch.full((x.numel() + 16,), wlm.OUT_OF_RANGE_POISON, dtype=x.dtype, device=dev)
            buf[off:off + x.numel()] = x.reshape(-1)
            inner.append((buf, ctypes.c_void_p(buf.data_ptr() + off * buf.element_size())))
        rb = tuple(torch.empty_like(x) for x in ra)
        assert b.step_raw(inner[0][1], inner[1][1], *[ctypes.c_void_p(x.data_ptr()) for x in rb]) == sjd.SJD_OK
        torch.cuda.synchronize()
        for x, y in zip(ra + a.get_window() + a.get_rows(), rb + b.get_window() + b.get_rows()):
            assert torch.equal(x, y), t
        assert b.rows_streamed() == (10 * (t + 1) if streams else 0)
    assert a.sync() == sjd.SJD_OK and b.sync() == sjd.SJD_OK
    assert a.rows_streamed() == a.stats()[0] == b.stats()[0] == 30


@pytest.mark.parametrize("K,D,W,top_k", [(2, 8, 12, 60), (8, 2, 5, 200), (4, 3, 3, 1), (2, 8, 400, 60)])
def test_trees_with_many_groups_or_few_rows(K, D, W, top_k):
    """127 and 7 drawn groups a row, a window no longer than the tree,
    single-id rows that leave every group after the first draw empty, and a
    window whose walk needs more shared memory than the candidates of 256 ids."""
    w = BASE.scaled(batch=1 if W > 100 else 2, window=W, vocab=256, hi=256, top_k=top_k, pd_k=K, pd_depth=D, sigma=0.4, dtype="bf16",
                    seed=K * 100 + D)
    ls = TreeLockstep(w)
    ls.start_from_logits()
    for t in range(2 if W > 100 else 4):
        c, u = tree_inputs(w, t + 1)
        ls.step(c, u)


@pytest.mark.parametrize("top_k", [1, 201, 1023, 1025])
def test_stored_rows_of_any_capacity(top_k):
    run(BASE.scaled(batch=2, window=4, vocab=2048, hi=2048, top_k=top_k, sigma=1.0, dtype="bf16"), 2)


@pytest.mark.parametrize("kind,over", [
    ("256 threads", dict(batch=4, window=50, vocab=2048, hi=2048, top_k=600)),
    ("list in the workspace", dict(batch=4, window=50, vocab=16384, hi=16384, top_k=2048, sigma=0.2)),
    ("ragged rows", dict(batch=4, window=50, vocab=2051, lo=3, hi=2045, top_k=600)),
    ("ragged narrow rows", dict(batch=8, window=60, vocab=2051, lo=3, hi=2045, top_k=300, top_p=0.95)),
    ("tree", dict(batch=2, window=12, vocab=2048, hi=2048, top_k=300)),
])
def test_overlapping_steps_on_every_route(kind, over):
    """Steps that start before the one in front of them has finished (the
    early-logits guarantee) give the bits of steps that wait."""
    tree = kind == "tree"
    w = BASE.scaled(**{**dict(sigma=0.6, q_noise=0.4, dtype="bf16"), **over})
    dev = torch.device("cuda", torch.cuda.current_device())
    steps = 6
    make = tree_inputs if tree else lambda w, t: wlm.logits_step(w, t)[:2]
    ins = [device_logits(w, make(w, t + 1), dev) for t in range(steps)]
    dq = device_logits(w, wlm.logits_step(w, 0)[2:], dev)
    cfg = config_of(w, pd_tree=1) if tree else config_of(w)
    a, b = sjd.SJD(cfg, dev), sjd.SJD(cfg, dev)
    for x in (a, b):
        x.draft_from_logits(*dq)
    b.set_early_logits(True)
    torch.cuda.synchronize()
    ref = []
    for t in range(steps):
        ref.append([x.clone() for x in a.step(*ins[t])])
        torch.cuda.synchronize()
    got = [b.step(*ins[t]) for t in range(steps)]
    torch.cuda.synchronize()
    assert a.sync() == sjd.SJD_OK and b.sync() == sjd.SJD_OK, (a.last_error(), b.last_error())
    for t in range(steps):
        for x, y in zip(ref[t], got[t]):
            assert torch.equal(x, y), (kind, t)
    for x, y in zip(a.get_window() + a.get_rows(), b.get_window() + b.get_rows()):
        assert torch.equal(x, y), kind


@pytest.mark.parametrize("early", [False, True])
@pytest.mark.parametrize("top_k", [60, 200])     # the 128-thread layout and a wide one
def test_rows_of_absent_tree_nodes_are_not_looked_at(top_k, early):
    """Node rows whose node does not exist hold NaN, all of them before the
    first tree: no status, no row streamed again, and the bits of the oracle,
    which evaluates existing nodes only; with the early-logits guarantee also
    in steps back to back."""
    w = BASE.scaled(batch=2, window=8, vocab=640, hi=640, top_k=top_k, pd_k=3, pd_depth=4, sigma=0.4, q_noise=0.4,
                    dtype="bf16")
    K, D, W = w.pd_k, w.pd_depth, w.window
    ls = TreeLockstep(w)
    waits = ls.ctx.step
    if early:
        ls.ctx.set_early_logits(True)
        ls.ctx.step = lambda *a: (torch.cuda.synchronize(), waits(*a))[1]  # (logits written before)
    ls.start_from_logits()
    ins, absent_seen = [], []
    for t in range(6):
        c, u = tree_inputs(w, t + 1)
        absent = 0
        for b, st in enumerate(ls.states):
            row = W
            for d in range(1, D):
                for i in range(1, K ** d):
                    if d >= len(st.tree) or i % K >= len(st.tree[d - 1][i // K]):
                        c[b, row] = u[b, row] = np.nan
                        absent += 1
                    row += 1
        ins.append((c, u))
        absent_seen.append(absent)
        ls.step(c, u)
    X = sum(K ** d - 1 for d in range(1, D))
    assert absent_seen[0] == 2 * X and min(absent_seen) < 2 * X
    if early:  # once more, without a wait between the steps
        ctx = sjd.SJD(config_of(w, pd_tree=1), ls.dev)
        ctx.draft_from_logits(*device_logits(w, wlm.logits_step(w, 0)[2:], ls.dev))
        ctx.set_early_logits(True)
        dl = [device_logits(w, x, ls.dev) for x in ins]
        torch.cuda.synchronize()
        for c, u in dl:
            ctx.step(c, u)
        assert ctx.sync() == sjd.SJD_OK, ctx.last_error()
        for x, y in zip(ctx.get_window() + ctx.get_rows() + ctx.get_tree(),
                        ls.ctx.get_window() + ls.ctx.get_rows() + ls.ctx.get_tree()):
            assert torch.equal(x, y)
        assert ctx.stats()[4:] == ls.ctx.stats()[4:]


@pytest.mark.parametrize("kernel", ["streaming", "general"])
@pytest.mark.parametrize("top", [1e8, -1e8, 1.5 * 2.0 ** 26, 4e6, 3.9e6])
@pytest.mark.parametrize("batch,window,top_k,n_max", [(2, 4, 50, 10), (2, 4, 200, 150), (3, 51, 200, 150)])
def test_top_k_among_ties_at_large_magnitudes(batch, window, top_k, n_max, top, kernel, monkeypatch):
    """Maxima of a magnitude at which fp32 values are up to 16 apart, 60 ties
    32 below them (weight 2 of 2^47 each) and the rest far below: the top-k
    cut lies among the ties (layouts of 128, 512 and 256 threads)."""
    if kernel == "general":
        monkeypatch.setenv("SJD_KERNEL", "general")
    else:
        monkeypatch.delenv("SJD_KERNEL", raising=False)
    vocab = 2048
    w = BASE.scaled(batch=batch, window=window, vocab=vocab, hi=vocab, top_k=top_k, top_p=1.0, cfg_scale=1.0,
                    dtype="f32")
    ls = Lockstep(w)
    assert ls.ctx.row_path() == (1 if kernel == "streaming" else 0)
    rng = np.random.default_rng(5)

    def rows():
        x = np.full((batch, window, vocab), np.float32(top) - np.float32(4096.0), np.float32)
        for r in x.reshape(-1, vocab):
            at = rng.permutation(vocab)
            r[at[:n_max]] = np.float32(top)
            r[at[n_max:n_max + 60]] = np.float32(top) - np.float32(32.0)
        return x

    c, q = rows(), rows()
    ls.start_from_logits((c, c, q, q))
    ls.step(c, c)
    _, _, n = ls.ctx.get_rows()
    assert int(n.max()) == top_k


@pytest.mark.parametrize("kind,over,size", [
    ("ragged", dict(batch=2, window=5, vocab=1003, hi=1003, top_k=300, top_p=0.95), 30464),
    ("tree", dict(batch=2, window=8, vocab=640, hi=640, top_k=200, pd_k=3, pd_depth=4), 64512),
])
def test_a_workspace_without_the_streaming_scratch(kind, over, size, monkeypatch):
    """Ragged rows and the full tree in a workspace that holds the decode
    state and the step's results alone: the general kernel, the same bits; a
    byte less is refused."""
    w = BASE.scaled(**{**dict(sigma=0.6, q_noise=0.4, dtype="bf16"), **over})
    monkeypatch.setattr(sjd, "workspace_size", lambda cfg: size)
    ls = (TreeLockstep if kind == "tree" else Lockstep)(w)
    ls.start_from_logits()
    for t in range(3):
        c, u = tree_inputs(w, t + 1) if kind == "tree" else ls.inputs(t + 1)[:2]
        ls.step(c, u)
    assert ls.ctx.row_path() == 0
    monkeypatch.setattr(sjd, "workspace_size", lambda cfg: size - 1)
    with pytest.raises(sjd.SJDError) as e:
        sjd.SJD(config_of(w, pd_tree=1 if kind == "tree" else 0), ls.dev)
    assert e.value.code == sjd.SJD_ERR_CAPACITY


def test_lists_beyond_shared_memory_with_a_small_top_k():
    """More candidates than the list's shared part, at supports where the
    row's scratch holds fewer entries than the list could have."""
    for k in (2, 128):
        run(BASE.scaled(batch=2, window=4, vocab=16384, hi=16384, top_k=k, sigma=0.3, cfg_scale=1.0, dtype="bf16",
                        ramp=-20.0), 2)


@pytest.mark.parametrize("over", [
    dict(batch=5, window=61, vocab=512, hi=512, top_k=200, top_p=0.97),                                 # kept rows, 128 threads
    dict(batch=2, window=4, vocab=16384, hi=16384, top_k=128, cfg_scale=1.0, sigma=0.3, ramp=-20.0),   # lists, 128 threads
    dict(batch=2, window=4, vocab=16384, hi=16384, top_k=200, cfg_scale=1.0, sigma=0.3, ramp=-20.0),   # 512
    dict(batch=3, window=51, vocab=16384, hi=16384, top_k=200, cfg_scale=1.0, sigma=0.3, ramp=-20.0),  # 256
])
def test_the_rows_scratch_needs_no_clearing(over):
    """sjd_init leaves the rows' scratch as it is (its size would cost more
    than the rest of the start), and what lies there does not reach a result."""
    w = BASE.scaled(**{**dict(sigma=0.6, q_noise=0.4, dtype="bf16"), **over})
    ls = Lockstep(w)
    ctx, cap = ls.ctx, ls.ctx.cfg.support_cap

    def up(x):
        return -(-x // 256) * 256

    row = up(32 * cap) + up(8 * (min(w.vocab, 16384) - min(w.vocab, 3072)))
    ctx.close()
    ctx.workspace.fill_(0xAB)
    assert ctx.L.sjd_init(ctypes.byref(ctx.cfg), ctypes.c_void_p(ctx.workspace.data_ptr()), ctx.workspace.numel(),
                          ctypes.c_void_p(ctx.stream.cuda_stream), ctypes.byref(ctx.ctx)) == sjd.SJD_OK
    scratch = ctx.workspace[-w.batch * w.window * row:]
    assert bool((scratch == 0xAB).all())
    c, u = ls.start_from_logits()
    ls.step(c, u)
    c, u, _, _ = ls.inputs(1)
    ls.step(c, u)
    assert not bool((scratch == 0xAB).all())     # the case does use it


@pytest.mark.parametrize("top_p", [0.5, 0.95, 0.9999])
@pytest.mark.parametrize("batch,window,vocab,top_k", [
    (2, 4, 2048, 100),     # 128 threads
    (2, 4, 8192, 200),     # 512
    (3, 51, 8192, 200),    # 256
])
def test_a_short_list_longer_than_k(batch, window, vocab, top_k, top_p):
    """The ids that the first round samples lie far below one maximum, so that
    the row is expected to have few ids with t > -22; the others hold three
    times k of them, with ties at the cut. The row is not streamed again."""
    w = BASE.scaled(batch=batch, window=window, vocab=vocab, hi=vocab, top_k=top_k, top_p=top_p, cfg_scale=1.0,
                    dtype="bf16")
    ls = Lockstep(w)
    rng = np.random.default_rng(7)

    def rows():
        x = rng.uniform(-30.0, -26.0, (batch, window, vocab)).astype(np.float32)
        for r in x.reshape(-1, vocab):
            r[rng.integers(0, vocab // 2)] = 0.0
            near = vocab // 2 + rng.permutation(vocab // 2)[:3 * top_k]
            r[near] = np.round(rng.uniform(-20.0, -1.0, 3 * top_k) * 4) / 4
        return wlm.bf16_round(x)

    c, q = rows(), rows()
    ls.start_from_logits((c, c, q, q))
    ls.step(c, c)
    c = rows()
    ls.step(c, c)
    assert ls.ctx.stats()[4] == 0


@pytest.mark.parametrize("batch,window", [(5, 61), (3, 51), (2, 4)])    # 128, 256, 512 threads
@pytest.mark.parametrize("top_k", [128, 129, 400])
def test_short_rows_after_long_ones(batch, window, top_k):
    """Rows of a few kept ids whose stored draft rows have up to top_k: the
    draft row is merged by the block from 129 entries on."""
    w = BASE.scaled(batch=batch, window=window, vocab=512, hi=512, top_k=top_k, top_p=0.999, q_noise=0.1, dtype="bf16")
    flat, sharp = w.scaled(sigma=0.1), w.scaled(sigma=5.0)
    ls = Lockstep(w)
    c, u, _, _ = wlm.logits_step(sharp, 0)
    _, _, qc, qu = wlm.logits_step(flat, 0)
    ls.start_from_logits((c, u, qc, qu))
    assert int(ls.ctx.get_rows()[2].max()) > 0.9 * top_k
    ls.step(c, u)
    assert int(ls.ctx.get_rows()[2].max()) <= 32
    ls.step(*wlm.logits_step(flat, 1)[:2])
    ls.step(*wlm.logits_step(sharp, 2)[:2])


@pytest.mark.parametrize("vocab,top_k,K", [(301, 200, 1), (1003, 500, 1), (1003, 128, 2), (1273, 500, 2), (1291, 500, 2),
                                           (1003, 500, 3), (2293, 500, 1), (2299, 500, 1)])
@pytest.mark.parametrize("sigma", [0.8, 4.0])
def test_ragged_rows_of_few_ids(vocab, top_k, K, sigma):
    """Ragged rows around the lines between the streaming and the general
    kernel, whose choice depends on the mode: a drafted window on one, its
    steps and split verification on the other."""
    ids = -(-(vocab + 7) // 8) * 8     # of a chunk grid that starts anywhere
    draft = top_k <= 128 or ids > 2304          # streamed?
    step = top_k <= 128 or K > 2 or ids > (2304 if K == 1 else 1280)
    w = BASE.scaled(batch=2, window=6, vocab=vocab, hi=vocab, top_k=top_k, top_p=0.95, cfg_scale=1.0, pd_k=K,
                    sigma=sigma, dtype="bf16")
    for fused in (True, False):
        ls = run(w, 2, fused=fused)
        assert ls.ctx.stats()[0] == 36
        assert ls.ctx.rows_streamed() == 12 * draft + 24 * step


@pytest.mark.parametrize("inference", [False, True])
def test_decode_loop_arguments_after_in_place_changes(inference):
    """A forward that reshapes its arguments in place finds them as documented
    at the next step, and the decode is the one of a forward that does not."""
    with torch.inference_mode(inference):
        _decode_with_in_place_changes()


def _decode_with_in_place_changes():
    w = BASE.scaled(batch=2, window=5, vocab=64, hi=64, top_k=20, dtype="bf16")
    dev = torch.device("cuda", torch.cuda.current_device())
    table = torch.randn((64, 64), generator=torch.Generator(dev).manual_seed(3), device=dev)
    seen = []

    def forward(win, prev, pos, cond, uncond, in_place):
        seen.append((win.shape, prev.shape, pos.shape))
        before = torch.cat([prev.view(2, 1), win.view(2, 5)[:, :-1]], dim=1).long()
        cond.copy_(table[before])
        uncond.copy_(table[before] * 0.5)
        if in_place:
            win.t_()
            prev.unsqueeze_(1)
            pos.unsqueeze_(0)

    grids = []
    for in_place in (False, True):
        ctx = sjd.SJD(config_of(w, max_steps=60), dev)
        cond = torch.empty((2, 5, 64), dtype=torch.bfloat16, device=dev)
        grid, _, steps = ctx.decode_loop(lambda *a: forward(*a, in_place), 24, cond, torch.empty_like(cond))
        grids.append(grid)
        assert steps > 3 and ctx.sync() == sjd.SJD_OK
    assert set(seen) == {((2, 5), (2,), (2,))}
    assert torch.equal(*grids)


@pytest.mark.parametrize("kind,top_p", [
    ("equal 2", 0.5), ("equal 100", 0.5), ("equal 100", 0.25), ("equal 128", 0.5), ("equal 129", 0.5),
    ("near 199", 0.9999), ("near 200", 0.9999), ("near 201", 0.9999), ("near 200", 0.75),
    ("rebuilt", 0.5), ("rebuilt", 0.95), ("rebuilt", 0.9999),
])
@pytest.mark.parametrize("batch,window,vocab", [(2, 4, 2048), (3, 51, 2048), (2, 4, 2051)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_top_p_cuts_at_their_bounds(kind, top_p, batch, window, vocab, dtype):
    """Targets on the boundary between two entries (equal maxima whose number
    times top-p is whole, from two to more than the head holds), exactly k
    ids, one less and one more above t = -22 with all others just below it,
    and heads rebuilt at t > -6 (220 ids above -9, 20 of them above -6)."""
    k = 200
    w = BASE.scaled(batch=batch, window=window, vocab=vocab, hi=vocab, top_k=k, top_p=top_p, cfg_scale=1.0, pd_k=4,
                    dtype=dtype)
    ls = Lockstep(w)
    rng = np.random.default_rng(3)

    def rows():
        x = np.empty((batch, window, vocab), np.float32)
        for r in x.reshape(-1, vocab):
            at = rng.permutation(vocab)
            if kind.startswith("equal"):
                n = int(kind.split()[1])
                r[:] = -50.0
                r[at[:n]] = 0.0
            elif kind.startswith("near"):
                n = int(kind.split()[1])
                r[:] = -22.0 - rng.integers(0, 8, vocab) * 0.125
                r[at[:n]] = -rng.integers(60, 176, n) * 0.125
                r[at[0]] = 0.0
            else:
                r[:] = -12.0 - rng.integers(0, 100, vocab) * 0.125
                r[at[:220]] = -6.0 - rng.integers(1, 24, 220) * 0.125
                r[at[:20]] = -rng.integers(0, 48, 20) * 0.125
        return x

    c, q = rows(), rows()
    ls.start_from_logits((c, c, q, q))
    ls.step(c, c)


@pytest.mark.parametrize("kind", ["plain", "split", "tree", "host"])
def test_captured_calls_replay_to_the_same_bits(kind):
    """The step with the reads of its results, captured into a graph (with
    copies and memsets between the kernels, and a fork to a second stream and
    back) and replayed, gives the bits of the same calls made one by one."""
    tree = kind == "tree"
    w = BASE.scaled(batch=2, window=8, vocab=1024, hi=1024, top_k=200, sigma=0.6, dtype="bf16", pd_k=3, pd_depth=2)
    dev = torch.device("cuda", torch.cuda.current_device())
    cfg = config_of(w, pd_tree=1 if tree else 0)
    side, other = torch.cuda.Stream(dev), torch.cuda.Stream(dev)
    ins = device_logits(w, tree_inputs(w, 1) if tree else wlm.logits_step(w, 1)[:2], dev)
    dq = device_logits(w, wlm.logits_step(w, 0)[2:], dev)
    host = [x.cpu().pin_memory() for x in ins]
    ctxs = [sjd.SJD(cfg, dev, stream=side) for _ in range(2)]
    made = []

    def calls(ctx, out, fork):
        if kind == "split":
            ctx.verify_step(*ins, out=out)
            ctx.draft_pd()
        elif kind == "host":
            ctx.step_host(*host, stages[ctxs.index(ctx)], out=out)
        else:
            ctx.step(*ins, out=out)
        if fork:    # another stream waits for the step and is waited for before the reads
            other.wait_stream(side)
            with torch.cuda.stream(other):
                out[1].add_(0)
            side.wait_stream(other)
        got = ctx.get_rows() + ctx.get_window()
        return got + ctx.get_tree() if tree else got

    with torch.cuda.stream(side):
        stages = [c.host_stage() for c in ctxs] if kind == "host" else []
        for c in ctxs:
            c.draft_from_logits(*dq)
            made.append(tuple(torch.zeros_like(x) for x in c.step(*ins)))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        got = calls(ctxs[1], made[1], True)
    for _ in range(4):
        with torch.cuda.stream(side):
            ref = calls(ctxs[0], made[0], False)
            graph.replay()
        torch.cuda.synchronize()
        for x, y in zip(ref + made[0], got + made[1]):
            assert torch.equal(x, y)
    assert [c.sync() for c in ctxs] == [sjd.SJD_OK] * 2


@pytest.mark.parametrize("top_p", [0.8, 1.0])
@pytest.mark.parametrize("kind", ["spread", "equal"])
@pytest.mark.parametrize("batch,window,vocab,lo,top_k", [
    (2, 2, 20000, 0, 2000),     # 512 threads
    (3, 51, 17000, 0, 200),     # 256
    (2, 2, 20011, 3, 100),      # 512, ragged
    (2, 153, 17000, 0, 60),     # 128
])
def test_few_candidates_among_many_ids_of_large_magnitude(batch, window, vocab, lo, top_k, kind, top_p):
    """Rows of magnitude 1.6e8 (where the list takes every value) with three
    candidates among more ids than the list holds, the others far below the
    maximum, spread or all alike: the rows are streamed again and keep the
    candidates, also after a step whose top-k cut lay at a higher value."""
    w = BASE.scaled(batch=batch, window=window, vocab=vocab, lo=lo, hi=vocab, top_k=top_k, top_p=top_p, cfg_scale=1.0,
                    dtype="f32")
    ls = Lockstep(w, check_batches=[batch - 1])
    rng = np.random.default_rng(13)

    def rows():
        x = np.full((batch, window, vocab), np.float32(1e8), np.float32)
        for r in x.reshape(-1, vocab):
            if kind == "spread":
                r[:] = rng.uniform(1e8, 1.5e8, vocab).astype(np.float32)
            at = lo + rng.permutation(vocab - lo)[:3]
            r[at] = np.float32(1.6e8) - np.float32(16.0) * rng.integers(0, 2, 3).astype(np.float32)
        return x

    def higher():
        x = np.full((batch, window, vocab), np.float32(1e8), np.float32)
        x[:, :, lo:lo + top_k + 50] = np.float32(3e8)
        return x

    c, q = higher(), rows()
    ls.start_from_logits((c, c, q, q))
    ls.step(c, c)
    for _ in range(2):
        c = rows()
        ls.step(c, c)
        n = ls.ctx.get_rows()[2]
        assert 1 <= int(n[n >= 0].min()) <= 3
        c = higher()
        ls.step(c, c)


@pytest.mark.parametrize("kernel", ["streaming", "general"])
@pytest.mark.parametrize("value", [np.inf, 3e38, 1e30, 4e13])
@pytest.mark.parametrize("top_k,top_p", [(0, 1.0), (0, 0.9), (50, 1.0)])
def test_infinite_and_huge_logits_are_contained(value, top_k, top_p, kernel, monkeypatch):
    """+inf is reported, also where the top-k cut keeps every id, and finite
    logits up to the largest fp32 value index nothing out of range: later
    steps on ordinary logits give what they give after any window."""
    if kernel == "general":
        monkeypatch.setenv("SJD_KERNEL", "general")
    else:
        monkeypatch.delenv("SJD_KERNEL", raising=False)
    w = BASE.scaled(batch=2, window=4, vocab=512, hi=512, top_k=top_k, top_p=top_p, dtype="f32")
    dev = torch.device("cuda", torch.cuda.current_device())
    ctx = sjd.SJD(config_of(w), dev)
    rng = np.random.default_rng(1)
    for t in range(3):
        c, u, _, _ = wlm.logits_step(w, t)
        for r in c.reshape(-1, 512):
            r[rng.permutation(512)[:3]] = np.float32(value) * np.asarray([1.0, 1.0 - 2.0 ** -22, 0.5], np.float32)
        ctx.step(*device_logits(w, (c, u), dev))
        code = ctx.sync()
        assert code == sjd.SJD_ERR_NONFINITE if value == np.inf else code in (
            sjd.SJD_OK, sjd.SJD_ERR_NONFINITE, sjd.SJD_ERR_INVALID_DRAFT), code
    ctx.draft_uniform()
    c, u, _, _ = wlm.logits_step(w, 9)
    ctx.step(*device_logits(w, (c, u), dev))
    assert ctx.sync() == sjd.SJD_OK
