"""GPU parity, recursion shaped by the values it computes (Section 6.2, last paragraph): a tree is grown top-down
from a seed state, a gate on every node's state decides whether the node is expanded.  The CUDA executor
(token waves and vector operators interleaved, through the C boundary) against the fp64 oracle: the state of every
generated tree's root, and the shape of every generated tree (invocations per function, read off the Call records).
The gate is a sign decision on an fp32 sum: an instance whose nearest decision is closer to zero than 1e-4 in the
oracle may legitimately grow a different tree in fp32; such instances are only required to be few, the others must
agree in shape exactly and in value within the fp32 tolerance."""
import numpy as np
import pytest

import workloads
import paper_2410_20225_b200 as rdf
from oracle import direct

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MARGIN = 1e-4
TOL = 1e-4


def oracle_run(P, tb, D):
    states, logs = [], []
    for b in range(tb.B):
        log = {}
        states.append(direct.topdown(P, int(tb.tok[b]), D, log))
        logs.append(log)
    return np.array(states), logs


def shapes_from_trace(tr, B, n_frames):
    """Per instance: number of Call firings per callee-site label, from the (frame, parent, label) records."""
    calls = tr[tr["kind"] == 0]
    frame = calls["tag"].astype(np.int64) & 0xFFFFFFFF
    parent = np.full(n_frames, -1, dtype=np.int64)
    parent[frame] = calls["parent"]
    inst = np.arange(n_frames, dtype=np.int64)
    inst[B:] = -1
    order = np.sort(frame)                       # frame ids grow with the wave: a parent has a smaller id than its callee
    for f in order:
        inst[f] = inst[parent[f]]
    per = {}
    for f, l in zip(frame, calls["label"]):
        per.setdefault(int(inst[f]), {}).setdefault(int(l), 0)
        per[int(inst[f])][int(l)] += 1
    return per


@pytest.mark.parametrize("H,D,B", [(64, 8, 256), (100, 6, 96), (256, 7, 64), (8, 10, 33)])
def test_topdown_recursion_states_and_shapes(H, D, B):
    V = 1000
    P = workloads.topdown_params(workloads.DEFAULT_SEED + H, V, H)
    tb = workloads.topdown_batch(workloads.DEFAULT_SEED + H, B, V)
    want, logs = oracle_run(P, tb, D)
    total = sum(1 + l["expand"] + l["child"] for l in logs)
    fs, r = rdf.topdown_program(D)
    g = rdf.Graph(fs, r, rdf.TAGS_FRAME)
    h, tr = g.eval_trees(rdf.Graph.device_trees(tb), rdf.Graph.device_params(P), rdf.F32, trace_capacity=4 * total + 64,
                         max_invocations=2 * total + 64)
    h = h.cpu().numpy()
    st = g.stats()
    decisive = np.array([l["margin"] > MARGIN for l in logs])
    assert decisive.mean() >= 0.9, decisive.mean()
    # shapes: per instance, one seed call, `expand` calls over its three sites, left and right calls
    per = shapes_from_trace(tr, B, B + 2 * total + 64)
    for b in np.flatnonzero(decisive):
        n_calls = sum(per[b].values())
        assert n_calls == 1 + logs[b]["expand"] + logs[b]["child"], (b, per[b], logs[b])
    if decisive.all():
        assert st["invocations"] == total
    # values
    err = np.abs(h[decisive] - want[decisive]).max() / np.abs(want[decisive]).max()
    assert err <= TOL, err
    # the generated trees differ in size across the batch: the control really followed the values
    assert len({l["expand"] for l in logs}) >= 4


def test_topdown_degenerate_gates():
    """Gate always open: every tree is the seed alone (three invocations: seed, expand, and nothing below).  Gate
    never open: the full tree down to the depth limit."""
    V, H, D, B = 50, 16, 4, 40
    P = workloads.topdown_params(7, V, H)
    tb = workloads.topdown_batch(7, B, V)
    fs, r = rdf.topdown_program(D)
    g = rdf.Graph(fs, r, rdf.TAGS_FRAME)
    for bias, per_instance in ((100.0, 2), (-100.0, 1 + (2 ** (D + 1) - 1) + (2 ** (D + 1) - 2))):
        P["b_s"][0] = bias
        want, logs = oracle_run(P, tb, D)
        h, _ = g.eval_trees(rdf.Graph.device_trees(tb), rdf.Graph.device_params(P), rdf.F32, max_invocations=B * per_instance + 8)
        assert g.stats()["invocations"] == B * per_instance
        assert np.abs(h.cpu().numpy() - want).max() / np.abs(want).max() <= TOL


def test_topdown_is_forward_fp32_only():
    V, H, D, B = 50, 16, 3, 8
    P = workloads.topdown_params(7, V, H)
    tb = workloads.topdown_batch(7, B, V)
    fs, r = rdf.topdown_program(D)
    g = rdf.Graph(fs, r, rdf.TAGS_FRAME)
    dt, dp = rdf.Graph.device_trees(tb), rdf.Graph.device_params(P)
    with pytest.raises(rdf.RdfError) as e:
        g.eval_trees(dt, dp, rdf.BF16, max_invocations=4096)
    assert e.value.code == -11
    with pytest.raises(rdf.RdfError) as e:
        g.grad_trees(dt, dp, rdf.F32, max_invocations=4096)
    assert e.value.code == -11
    # an undersized frame table is a status code and the graph stays usable
    with pytest.raises(rdf.RdfError) as e:
        g.eval_trees(dt, dp, rdf.F32, max_invocations=B)
    assert e.value.code == -6
    want, _ = oracle_run(P, tb, D)
    h, _ = g.eval_trees(dt, dp, rdf.F32, max_invocations=4096)
    assert np.abs(h.cpu().numpy() - want).max() / np.abs(want).max() <= TOL


def test_topdown_full_size_as_benchmarked():
    """The workload `bench.py --workload 6` times (8192 seeds, H = 128, depth limit 10, frame table of 256 frames per
    seed): every instance against the oracle -- the root state of each decisive instance, the number of invocations
    of the whole batch when every instance is decisive, else of the decisive ones through the Call records."""
    cfg = workloads.config(6)
    tb, P, D = cfg["trees"], cfg["params"], cfg["D"]
    want, logs = oracle_run(P, tb, D)
    total = sum(1 + l["expand"] + l["child"] for l in logs)
    fs, r = rdf.topdown_program(D)
    g = rdf.Graph(fs, r, rdf.TAGS_FRAME)
    h, _ = g.eval_trees(rdf.Graph.device_trees(tb), rdf.Graph.device_params(P), rdf.F32, max_invocations=cfg["max_invocations"])
    h = h.cpu().numpy()
    st = g.stats()
    decisive = np.array([l["margin"] > MARGIN for l in logs])
    assert decisive.mean() >= 0.99, decisive.mean()
    err = np.abs(h[decisive] - want[decisive]).max() / np.abs(want[decisive]).max()
    assert err <= TOL, err
    # an instance that is not decisive may have grown another tree: the totals then differ by at most its size
    slack = sum(2 * (2 ** (D + 1)) for d in decisive if not d)
    assert abs(st["invocations"] - total) <= slack, (st["invocations"], total, slack)


@pytest.mark.parametrize("H,D,B", [(4, 5, 40), (20, 6, 33), (124, 5, 30), (128, 5, 30), (132, 4, 30), (256, 4, 20),
                                   (20, 4, 440), (124, 4, 110), (124, 4, 112), (132, 4, 120)])
def test_topdown_hidden_sizes(H, D, B):
    """Hidden sizes on both sides of the warp tiles (16 outputs) and of the switch from weights in shared memory (H <= 128)
    to weights read through the cache; groups of one and of several warps along the items."""
    test_topdown_recursion_states_and_shapes(H, D, B)


def test_topdown_errors_in_one_cluster():
    """Calls that one thread-block cluster runs (small batches) and that end with a status in any of their waves -- the frame
    table full after each of many different numbers of invocations, a token that is no row of the table: every block leaves, and
    the next call has the states of an undisturbed one."""
    V, H, D, B = 50, 32, 7, 24
    P = workloads.topdown_params(7, V, H)
    P["b_s"][0] = -100.0                          # full trees
    tb = workloads.topdown_batch(7, B, V)
    total = B * (1 + (2 ** (D + 1) - 1) + (2 ** (D + 1) - 2))
    g = rdf.Graph(*rdf.topdown_program(D), rdf.TAGS_FRAME)
    dt, dp = rdf.Graph.device_trees(tb), rdf.Graph.device_params(P)
    want = g.eval_trees(dt, dp, rdf.F32, max_invocations=total)[0]
    bad = dict(dt, tok=dt["tok"].clone())
    bad["tok"][B // 2] = V

    def code(trees, max_invocations):
        try:
            g.eval_trees(trees, dp, rdf.F32, max_invocations=max_invocations)
        except rdf.RdfError as e:
            return e.code
        return 0

    for m in [B, B + 1, 3 * B] + list(range(5 * B, total, 311)) + [total - 1]:
        assert code(dt, m) == -6, m
    assert code(bad, total) == -2
    assert torch.equal(g.eval_trees(dt, dp, rdf.F32, max_invocations=total)[0], want)


def _full_trees(B, D, H, V=50):
    P = workloads.topdown_params(7, V, H)
    P["b_s"][0] = -100.0                          # the gate never stops: 2^d expansions per seed at depth d
    g = rdf.Graph(*rdf.topdown_program(D), rdf.TAGS_FRAME)
    tb = workloads.topdown_batch(7, B, V)
    total = B * (1 + (2 ** (D + 1) - 1) + (2 ** (D + 1) - 2))
    return g, P, tb, total


@pytest.mark.parametrize("B,D,H", [(1, 9, 128), (3, 12, 16), (8, 9, 100), (40, 6, 256), (1, 1, 4)])
def test_topdown_waves_that_outgrow_a_cluster(B, D, H):
    """A call that starts in one thread-block cluster and is handed to the whole grid at its first wide wave (tokens x H x H
    beyond 10 x 2^20, or more than 4096 tokens), and one that never gets there: states, invocations and waves."""
    g, P, tb, total = _full_trees(B, D, H)
    want = np.array([direct.topdown(P, int(t), D, {}) for t in tb.tok[:B]])
    dt, dp = rdf.Graph.device_trees(tb), rdf.Graph.device_params(P)
    for _ in range(2):
        h = g.eval_trees(dt, dp, rdf.F32, max_invocations=total)[0].cpu().numpy()
        st = g.stats()
        assert st["invocations"] == total and st["waves"] == 4 * (D + 1)
        assert np.abs(h - want).max() / np.abs(want).max() <= TOL


def test_topdown_errors_behind_a_cluster():
    """Calls that a cluster hands to the whole grid and that end with a status there, some in the first wave the grid runs: every
    block leaves, and the next call has the states of an undisturbed one."""
    g, P, tb, total = _full_trees(8, 9, 100)
    dt, dp = rdf.Graph.device_trees(tb), rdf.Graph.device_params(P)
    want = g.eval_trees(dt, dp, rdf.F32, max_invocations=total)[0]
    for m in list(range(8 * 31, total, 173)) + [total - 1]:
        with pytest.raises(rdf.RdfError) as e:
            g.eval_trees(dt, dp, rdf.F32, max_invocations=m)
        assert e.value.code == -6, m
    assert torch.equal(g.eval_trees(dt, dp, rdf.F32, max_invocations=total)[0], want)


def test_topdown_wide_waves_of_few_seeds_use_the_device():
    """64 seeds that grow full trees (waves of 65 536 tokens) take no longer than 512 of them."""
    ms = []
    for B in (64, 512):
        g, P, tb, total = _full_trees(B, 10, 128)
        dt, dp = rdf.Graph.device_trees(tb), rdf.Graph.device_params(P)
        for _ in range(3):
            g.eval_trees(dt, dp, rdf.F32, check=False, max_invocations=total)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(5):
            g.eval_trees(dt, dp, rdf.F32, check=False, max_invocations=total)
        e[1].record()
        torch.cuda.synchronize()
        g.stats()
        ms.append(e[0].elapsed_time(e[1]) / 5)
    assert ms[0] < ms[1], ms


@pytest.mark.parametrize("B,H,D", [(1, 16, 4), (40, 48, 5), (600, 112, 6), (3000, 128, 6), (700, 16, 7), (260, 256, 4), (900, 132, 3)])
def test_group_sizes_of_the_operators(B, H, D):
    """Two, four and eight items per thread, one to all warps along the outputs, weights in shared memory and through L1: every state is one
    fixed expression, so the groups that an operator falls into must not show.  A seed alone and the same seed in a batch agree bit by bit."""
    fs, r = rdf.topdown_program(D)
    gen = torch.Generator(device="cuda").manual_seed(B)
    p = {"E": torch.randn(50, H, device="cuda", generator=gen), "W": torch.randn(H, 2 * H, device="cuda", generator=gen) / (2 * H) ** 0.5,
         "b": torch.randn(H, device="cuda", generator=gen) * 0.1, "W_s": torch.randn(5, H, device="cuda", generator=gen) / H ** 0.5,
         "b_s": torch.full((5,), 0.3, device="cuda")}

    def run(tok):
        n = tok.numel()
        one = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        dt = {"tree_root": torch.arange(n, dtype=torch.int32, device="cuda"), "left": one, "right": one, "tok": tok, "label": one}
        h, _ = rdf.Graph(fs, r, rdf.TAGS_FRAME).eval_trees(dt, p, max_invocations=n * 4 * 2 ** D)
        return h
    tok = (torch.arange(B, device="cuda") * 7 % 50).int()
    h = run(tok)
    for t in (0, 7, 49):
        rows = h[tok == t]
        if rows.numel():
            alone = run(torch.tensor([t], dtype=torch.int32, device="cuda"))
            assert torch.equal(rows, alone.expand_as(rows))
