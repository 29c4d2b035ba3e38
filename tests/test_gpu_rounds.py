"""Several decoding rounds in a row with the acceptance history kept on the device (Eq. 15), and the round
captured in a CUDA graph."""
import numpy as np
import pytest
import torch

import graft_inputs as gi
import oracle
from helpers import compare_round, gpu_round, oracle_round

pytestmark = pytest.mark.gpu

DT = {"f32": 0, "bf16": 1}


def _graft(w):
    from paper_2608_20375_b200 import Graft
    g = Graft(w.V, w.L, w.K, w.m, w.hidden_dim, w.batch, w.budget_min, w.budget_max, w.budget_step, w.beta, 1,
              DT[w.logits_dtype], DT[w.hidden_dtype])
    tb = gi.tdes_tables(w)
    saba_kw = gi.saba_defaults(w)
    keep = [tb["P"].cuda(), tb["C"].cuda(), tb["u"].cuda()]
    g.set_tdes_tables(keep[0], keep[1], keep[2], tb["s"])
    g.set_saba(**saba_kw)
    return g, tb, saba_kw, keep


def _target_next_from_tree(rng, tree, V, p_follow=0.75):
    """Target next-token ids per node: mostly the token of one of the node's children, so that walks get somewhere."""
    n = int(tree["n_nodes"])
    tn = rng.integers(0, V, size=tree["token"].shape[0]).astype(np.int32)
    children = {}
    for i in range(1, n):
        children.setdefault(int(tree["parent"][i]), []).append(i)
    for i in range(n):
        if i in children and rng.random() < p_follow:
            tn[i] = tree["token"][children[i][int(rng.integers(len(children[i])))]]
    return tn


@pytest.mark.parametrize("hist_w", [1, 3, 8])
def test_rounds_with_device_resident_history(hist_w):
    rounds = 7
    base = dict(batch=5, L=6, V=3000, K=6, budget_min=8, budget_max=40, budget_step=8, m=16, hidden_dim=32)
    w0 = gi.small(**base)
    g, tb, saba_kw, keep = _graft(w0)
    window = torch.zeros((w0.batch, hist_w), dtype=torch.int32, device="cuda")
    count = torch.zeros(w0.batch, dtype=torch.int32, device="cuda")
    hist_dev = torch.zeros(w0.batch, dtype=torch.float32, device="cuda")
    g.set_hist_window(hist_w, window, count, hist_dev)
    rng = np.random.default_rng(77)
    accepted = [[] for _ in range(w0.batch)]  # the oracle's record of a_t per sequence
    a_len = torch.empty(w0.batch, dtype=torch.int32, device="cuda")
    a_path = torch.empty((w0.batch, w0.L), dtype=torch.int32, device="cuda")
    bonus = torch.empty(w0.batch, dtype=torch.int32, device="cuda")
    for r in range(rounds):
        w = gi.small(**base, seed=4100 + r)  # new drafter outputs every round
        x = gi.batch_inputs(w)
        hist_orc = np.array([oracle.hist_update(a, hist_w) for a in accepted], dtype=np.float32)
        assert np.array_equal(hist_dev.cpu().numpy(), hist_orc), f"round {r}: device history differs"
        x["hist"] = torch.from_numpy(hist_orc.copy())
        out = g.alloc_out(w.batch, debug=True)
        g.build_trees(x["logits"].cuda(), x["hidden"].cuda(), x["root_token"].cuda(), hist_dev, x["prefix_len"].cuda(),
                      None, out)
        torch.cuda.synchronize()
        gpu = out.cpu()
        orc = oracle_round(oracle, w, x, tb, saba_kw)
        stats = compare_round(oracle, w, x, tb, saba_kw, gpu, orc)
        assert stats["excused_tree"] == 0 and stats["excused_budget"] == 0, stats
        tn = np.stack([_target_next_from_tree(rng, {k: orc[k][b] for k in ("n_nodes", "token", "parent")}, w.V)
                       for b in range(w.batch)])
        g.accept(out, torch.from_numpy(tn).cuda(), a_len, a_path, bonus)
        torch.cuda.synchronize()
        for b in range(w.batch):
            a, path, bo = oracle.accept(int(orc["n_nodes"][b]), orc["token"][b], orc["parent"][b], tn[b], w.L)
            assert int(a_len[b]) == a and int(bonus[b]) == bo
            accepted[b].append(a)
        assert count.cpu().tolist() == [r + 1] * w.batch
    assert max(max(a) for a in accepted) >= 2  # the walks did get somewhere
    g.set_hist_window(0)
    g.destroy()


def test_round_in_a_cuda_graph():
    """build_trees + accept captured once and replayed: the library calls allocate nothing, synchronise nothing and
    keep no per-launch host state that a replay would miss."""
    w = gi.small(batch=4, L=8, V=6000, K=8, budget_min=16, budget_max=96, budget_step=16, m=32, hidden_dim=64,
                 logits_dtype="bf16", hidden_dtype="bf16")
    g, tb, saba_kw, keep = _graft(w)
    g.set_edge_rows(min(w.L, 8))
    xs = [gi.batch_inputs(gi.small(batch=4, L=8, V=6000, K=8, budget_min=16, budget_max=96, budget_step=16, m=32,
                                   hidden_dim=64, logits_dtype="bf16", hidden_dtype="bf16", seed=900 + i))
          for i in range(2)]
    stat = {k: xs[0][k].cuda().clone() for k in ("logits", "hidden", "root_token", "hist", "prefix_len")}
    out = g.alloc_out(w.batch)
    tn = torch.zeros((w.batch, g.nmax), dtype=torch.int32, device="cuda")
    a_len = torch.empty(w.batch, dtype=torch.int32, device="cuda")
    a_path = torch.empty((w.batch, w.L), dtype=torch.int32, device="cuda")
    bonus = torch.empty(w.batch, dtype=torch.int32, device="cuda")

    def round_():
        g.build_trees(stat["logits"], stat["hidden"], stat["root_token"], stat["hist"], stat["prefix_len"], None, out)
        g.accept(out, tn, a_len, a_path, bonus)

    # eager results for both input sets
    eager = []
    for x in xs:
        for k in stat:
            stat[k].copy_(x[k].cuda())
        round_()
        torch.cuda.synchronize()
        eager.append({k: v.copy() for k, v in out.cpu().items()})
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        round_()  # warm-up on the capture stream
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        round_()
    for rep in range(2):
        for i, x in enumerate(xs):
            for k in stat:
                stat[k].copy_(x[k].cuda())
            graph.replay()
            torch.cuda.synchronize()
            got = out.cpu()
            for k in ("n_nodes", "budget", "status", "token", "parent", "depth", "position", "path_score", "mask"):
                assert np.array_equal(got[k], eager[i][k]), (rep, i, k)
    g.destroy()


def test_micro_batches_on_streams_of_their_own():
    """Two micro-batches, each with its own context and stream, so that one's tree building overlaps the other's
    (stub) verification: every round's results are the sequential schedule's, bit for bit, and the sequential
    schedule's first and last rounds are the oracle's."""
    from paper_2608_20375_b200.pipeline import MicroBatch, join, run_rounds

    rounds, hist_w, n_micro = 5, 3, 2
    base = dict(batch=6, L=8, V=5000, K=8, budget_min=16, budget_max=96, budget_step=16, m=32, hidden_dim=64,
                logits_dtype="bf16", hidden_dtype="bf16")
    w0 = gi.small(**base)
    keys = ("n_nodes", "budget", "status", "token", "parent", "depth", "position", "path_score", "mask", "topk_id",
            "topk_lp", "lse", "edge", "state")
    ctxs = [_graft(w0) for _ in range(n_micro)]
    tb, saba_kw = ctxs[0][1], ctxs[0][2]
    hist_bufs = []
    for g, *_ in ctxs:
        bufs = (torch.zeros((w0.batch, hist_w), dtype=torch.int32, device="cuda"),
                torch.zeros(w0.batch, dtype=torch.int32, device="cuda"),
                torch.zeros(w0.batch, dtype=torch.float32, device="cuda"))
        g.set_hist_window(hist_w, *bufs)
        hist_bufs.append(bufs)
    micro = [MicroBatch(g, w0.batch, w0.L, out=g.alloc_out(w0.batch, debug=True)) for g, *_ in ctxs]
    ws = [[gi.small(**base, seed=5200 + 10 * i + r) for r in range(rounds)] for i in range(n_micro)]
    xs = [[gi.batch_inputs(w) for w in row] for row in ws]
    dev_x = [[{k: x[k].cuda() for k in ("logits", "hidden", "root_token", "prefix_len")} for x in row] for row in xs]
    burn = torch.randn(1024, 1024, device="cuda")
    tn_dev = {}   # (i, r) -> target ids, fixed by the sequential pass
    record = {}   # schedule -> (i, r) -> outputs
    rng = np.random.default_rng(11)

    def draft(i, r):
        return dict(dev_x[i][r], hist=hist_bufs[i][2])

    def run(schedule, overlap):
        for bufs in hist_bufs:
            for t in bufs:
                t.zero_()
        record[schedule] = {}

        def verify(i, r, out):
            y = burn
            for _ in range(4):  # stands in for the target model's forward pass on this stream
                y = torch.mm(y, burn) * 1e-3
            if (i, r) not in tn_dev:  # sequential pass only: choose the target ids from the tree just built
                torch.cuda.current_stream().synchronize()
                t = out.cpu()
                tn = np.stack([_target_next_from_tree(rng, {k: t[k][b] for k in ("n_nodes", "token", "parent")},
                                                      w0.V) for b in range(w0.batch)])
                tn_dev[(i, r)] = torch.from_numpy(tn).cuda()
            return tn_dev[(i, r)]

        def after(i, r, mb):
            snap = {k: getattr(mb.out, k).clone() for k in keys}
            snap["accept_len"] = mb.accept_len.clone()
            snap["hist"] = hist_bufs[i][2].clone()
            record[schedule][(i, r)] = snap

        run_rounds(micro, rounds, draft, verify, overlap=overlap, after_round=after)
        join(micro)
        torch.cuda.synchronize()

    run("sequential", False)
    run("overlapped", True)
    for key, snap in record["sequential"].items():
        for k, v in snap.items():
            assert torch.equal(v, record["overlapped"][key][k]), (key, k)
    assert max(int(s["accept_len"].max()) for s in record["sequential"].values()) >= 2
    # the sequential schedule against the oracle: the first round (no history yet) and the last (hist from the device)
    for i in range(n_micro):
        for r in (0, rounds - 1):
            snap = record["sequential"][(i, r)]
            x = dict(xs[i][r])
            prev = record["sequential"][(i, r - 1)]["hist"] if r > 0 else torch.zeros(w0.batch)
            x["hist"] = prev.cpu().float()
            orc = oracle_round(oracle, ws[i][r], x, tb, saba_kw)
            gpu = {k: snap[k].cpu().numpy() for k in keys}
            gpu["mask"] = gpu["mask"].view("uint32")
            stats = compare_round(oracle, ws[i][r], x, tb, saba_kw, gpu, orc)
            assert stats["excused_tree"] == 0 and stats["excused_budget"] == 0, stats
    for g, *_ in ctxs:
        g.set_hist_window(0)
        g.destroy()


@pytest.mark.parametrize("K,m,beta", [(32, 128, 0.2), (32, 128, 0.0), (8, 124, 0.2), (11, 64, 0.2)])
def test_a_later_smaller_context_takes_no_shared_memory_from_an_older_one(K, m, beta):
    """The limit on a kernel's dynamic shared memory is the kernel's on the device: a context of smaller sizes that runs
    the same instances, created while a larger one lives, must leave the larger one's rounds and training steps alone."""
    w = gi.small(batch=2, L=16, V=2003, K=K, budget_min=16, budget_max=400, budget_step=16, m=m, hidden_dim=32, beta=beta)
    g, _, _, keep = _graft(w)
    x = gi.batch_inputs(w)
    tr = gi.tdes_traces(w.V, w.L, K, 20, 30, 40, seed=3)
    groups = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in tr["groups"].items()}
    pairs, edges = torch.from_numpy(tr["pairs"]).cuda(), torch.from_numpy(tr["edges"]).cuda()
    loss = torch.empty((2, 4), dtype=torch.float64, device="cuda")

    def work(i):
        _, gpu = gpu_round(g, w, x)          # every depth scored ahead, the score array asked for
        _, plain = gpu_round(g, w, x, debug=False)
        g.tdes_loss(groups, pairs, edges, gamma=0.5, w1=4.0, lambda_kl=1.0, lambda_pair=1.0, lambda_bce=0.25, loss=loss[i])
        torch.cuda.synchronize()
        return gpu, plain

    before = work(0)
    small = gi.small(batch=2, L=4, V=2003, K=K, budget_min=16, budget_max=64, budget_step=16, m=16 if m == 64 else m,
                     hidden_dim=32, beta=beta)
    g2, _, _, keep2 = _graft(small)
    after = work(1)
    for a, b in zip(before, after):
        for k in a:
            assert np.array_equal(a[k], b[k], equal_nan=True), k
    assert torch.allclose(loss[0], loss[1], rtol=1e-12)  # (64-bit sums in no fixed order)
    g2.destroy()
    g.destroy()


@pytest.mark.parametrize("field", ["mask", "budget", "depth", "position", "path_score", "status"])
@pytest.mark.parametrize("wrong", ["cpu", "dtype", "strides"])
def test_accept_refuses_a_wrong_tree(field, wrong):
    """Every array of the tree is looked at, whether the walk reads it or not."""
    from paper_2608_20375_b200 import GraftError
    w = gi.small(batch=2, L=4, V=300, K=4, budget_min=8, budget_max=16, budget_step=8, m=16, hidden_dim=8)
    g, _, _, keep = _graft(w)
    out, _ = gpu_round(g, w, gi.batch_inputs(w))
    tn = torch.zeros((2, g.nmax), dtype=torch.int32, device="cuda")
    a, path, bonus = (torch.empty(s, dtype=torch.int32, device="cuda") for s in ((2,), (2, w.L), (2,)))
    g.accept(out, tn, a, path, bonus)
    t = getattr(out, field)
    setattr(out, field, t.cpu() if wrong == "cpu" else t.to(torch.int64) if wrong == "dtype" else
            torch.stack([t, t], -1)[..., 0])
    with pytest.raises(GraftError):
        g.accept(out, tn, a, path, bonus)
    torch.cuda.synchronize()
    g.destroy()


@pytest.mark.parametrize("K,m", [(32, 128), (16, 64), (8, 128)])
@pytest.mark.parametrize("fixed", [False, True])
def test_large_batches_build_the_trees_of_small_ones(K, m, fixed):
    """From some batch on, how many depths are scored ahead depends on the sequence, and past one sequence an SM so does the order in
    which the trees are built.  Neither shows: the same bits as in batches of forty, round after round."""
    from paper_2608_20375_b200 import Graft
    V, L, n, hd = 3000, 16, 330, 64
    gen = torch.Generator(device="cuda").manual_seed(K + m)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    height = 16.0 * torch.rand((n, 1, 1), generator=gen, device="cuda")  # mean top-1 probabilities from 0.01 to nearly 1
    rank = torch.rand((n, L, V), generator=gen, device="cuda").argsort(2).float()
    logits = (2.0 * rand(n, L, V) + height / (1.0 + rank)).to(torch.bfloat16)
    logits[7, 3, 5] = float("nan")  # a bad row
    P, Ct, u = rand(V, m), rand(V, m), 0.5 * rand(L, m)
    root = torch.randint(0, V, (n,), generator=gen, device="cuda", dtype=torch.int32)
    prefix = torch.randint(1, 4000, (n,), generator=gen, device="cuda", dtype=torch.int32)
    hidden, hist = rand(n, L, hd).to(torch.bfloat16), 8.0 * torch.rand(n, generator=gen, device="cuda")
    budget = torch.randint(1, 300, (n,), generator=gen, device="cuda", dtype=torch.int32)

    def graft(batch):
        g = Graft(V, L, K, m, hd, batch, 16, 304, 16, 0.2, 1)
        g.set_tdes_tables(P, Ct, u, 1.0)
        g.set_saba(phi_conf=-160.0, phi_degen=20.0, phi_hist=-5.0, phi_bias=200.0, tau_min=8.0, cost_mode=1,
                   pts_n=[0.0, 64.0, 1024.0], pts_t=[18.0, 18.0, 37.2])
        return g

    def build(g, lo, hi):
        o = g.alloc_out(hi - lo)
        part = lambda t: t[lo:hi].contiguous()  # noqa: E731
        g.build_trees(part(logits), None if fixed else part(hidden), part(root), None if fixed else part(hist), part(prefix),
                      part(budget) if fixed else None, o)
        torch.cuda.synchronize()
        return o.cpu()

    small = graft(40)
    want = [build(small, lo, min(lo + 40, n)) for lo in range(0, n, 40)]
    want = {k: np.concatenate([w[k] for w in want]) for k in want[0]}
    depth = want["depth"].max(axis=1)
    assert depth.min() <= 3 and depth.max() >= 9
    big = graft(n)
    for lo, hi in ((0, n), (0, n), (11, n), (30, 180), (0, 149), (0, 148), (5, 85), (0, n)):
        got = build(big, lo, hi)
        for k, w in want.items():
            assert np.array_equal(got[k], w[lo:hi]), (k, lo, hi)
    big.destroy()
    small.destroy()


@pytest.mark.parametrize("K,m,L", [(32, 128, 12), (16, 64, 16), (9, 32, 7)])
def test_large_batches_with_any_number_of_depths_scored_ahead(K, m, L):
    """Asked for a number of depths, or for the score array, large batches build the same trees as when they choose for themselves."""
    from paper_2608_20375_b200 import Graft
    V, n = 2000, 170
    gen = torch.Generator(device="cuda").manual_seed(K + L)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    height = 16.0 * torch.rand((n, 1, 1), generator=gen, device="cuda")
    rank = torch.rand((n, L, V), generator=gen, device="cuda").argsort(2).float()
    logits = (2.0 * rand(n, L, V) + height / (1.0 + rank)).to(torch.bfloat16)
    P, Ct, u = rand(V, m), rand(V, m), 0.5 * rand(L, m)
    root = torch.randint(0, V, (n,), generator=gen, device="cuda", dtype=torch.int32)
    prefix = torch.full_like(root, 200)
    budget = torch.randint(1, 250, (n,), generator=gen, device="cuda", dtype=torch.int32)
    g = Graft(V, L, K, m, 64, n, 16, 256, 16, 0.2, 1)
    g.set_tdes_tables(P, Ct, u, 1.0)

    def build(debug=False):
        o = g.alloc_out(n, debug=debug)
        g.build_trees(logits, None, root, None, prefix, budget, o)
        torch.cuda.synchronize()
        return o.cpu()

    want = build()
    with_edges = build(debug=True)
    for rows in (0, 3, 5, 7, 12, L):
        g.set_edge_rows(min(rows, L))
        for got in (build(), build(debug=True)):
            for k, w in want.items():
                assert np.array_equal(got[k], w), (k, rows)
            if "edge" in got:
                assert np.array_equal(got["edge"], with_edges["edge"])
    g.destroy()
