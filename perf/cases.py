"""The work that users of this library have it do, as cases that can be timed and compared.

Five paths, every one through the package's public entry points:

  round   one decoding round of a batch: Graft.build_trees (vocab pass, budget, edge scores, tree) and Graft.accept
  shard   the vocab pass of one rank of a vocabulary-parallel LM head: its shard, then the merge of all shards' pieces
  loss    one training step of the edge scorer: cleared gradient buffers, losses and gradients (Graft.tdes_loss)
  tables  the scorer's tables for both towers, once per model (Graft.tdes_precompute)
  fit     the least-squares fit of the budget models to replay logs (Graft.saba_fit)

Inputs follow graft_inputs.py (the same distributions, drawn on the GPU): logits 2 N(0,1) with a Zipf-ranked boost on 64
tokens a position, hidden rows that grow more similar along the block, N(0,1) tables, targets whose match rate falls
from 0.9 to 0.3 along the block, Zipf-distributed tokens in training traces.
"""
import math

import torch

from paper_2608_20375_b200 import Graft
from paper_2608_20375_b200.binding import BF16, F32, VOCAB_PARTIAL_BYTES
from paper_2608_20375_b200.vocab_parallel import vocab_range

_DTYPES = {"bf16": (torch.bfloat16, BF16, 2), "f32": (torch.float32, F32, 4)}


def _round(name, batch, L, V, K, hidden_dim, budget_min, budget_max, fixed=0, dtype="bf16", m=128, beta=0.2, root_edge=1,
           boost_lo=12.0, boost_hi=12.0):
    return dict(name=name, kind="round", batch=batch, L=L, V=V, K=K, hidden_dim=hidden_dim, budget_min=budget_min,
                budget_max=budget_max, fixed=fixed, dtype=dtype, m=m, beta=beta, root_edge=root_edge, boost_lo=boost_lo,
                boost_hi=boost_hi)


def listed():
    return [
        # one user at a small vocabulary, a fixed budget, fp32 logits: the latency of three dependent kernels and a walk
        _round("round_b1_v32000_f32", 1, 16, 32000, 8, 256, 64, 64, fixed=64, dtype="f32"),
        # one user of a large-vocabulary model, the budget chosen per round
        _round("round_b1_v151936", 1, 16, 151936, 32, 4096, 16, 512),
        # a lightly loaded server, narrower candidate sets and budgets
        _round("round_b16_v151936", 16, 16, 151936, 16, 2560, 16, 256),
        # confident and uncertain rounds in one batch (boost heights 6 to 14), so that budgets and depths vary
        _round("round_b64_v128256_mixed", 64, 16, 128256, 32, 4096, 16, 512, boost_lo=6.0, boost_hi=14.0),
        # the ordinary serving batch
        _round("round_b64_v151936", 64, 16, 151936, 32, 4096, 16, 512),
        # a server at its largest batch
        _round("round_b256_v151936", 256, 16, 151936, 32, 4096, 16, 512),
        # the product-of-probabilities tree (no edge scores) at sizes that divide by nothing: ragged rows and tails
        _round("ddtree_b37_v50021", 37, 11, 50021, 11, 1000, 16, 200, beta=0.0, m=64),
        # one of eight ranks of a tensor-parallel LM head
        dict(name="shard_1of8_b64_v151936", kind="shard", batch=64, L=16, V=151936, K=32, world=8, dtype="bf16"),
        # a training step of the scorer: forward and backward over groups, pairs and edges
        dict(name="loss_g32768_v151936", kind="loss", V=151936, L=16, K=32, m=128, groups=32768, pairs=131072, edges=262144),
        # the set-up step of a large model, embeddings as checkpoints keep them
        dict(name="tables_v151936_e4096", kind="tables", V=151936, E=4096, m=128, dtype="bf16"),
        # the same for a small model kept in fp32
        dict(name="tables_v32000_e2048_f32", kind="tables", V=32000, E=2048, m=128, dtype="f32"),
        # replay logs of some ten thousand rounds at 31 budgets, several prompts sets together
        dict(name="fit_n4000000", kind="fit", n=4000000),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round"] * 7 + ["shard", "loss", "tables", "fit"])
    if kind == "round":
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        L = rng.choice([16, 16, 16, 12, rng.randint(4, 8)])
        V = rng.choice([32000, 128256, 151936, _log_uniform(rng, 16000, 151936)])
        most = 256 * 16 * 151936 * 2 // (L * V * _DTYPES[dtype][2])  # no more bytes than the largest listed round
        batch = _log_uniform(rng, 1, min(256, most))
        K = rng.choice([8, 16, 32, 32, rng.randint(4, 32)])
        budget_max = rng.choice([256, 512, rng.randint(32, 512)])
        fixed = rng.choice([0, 0, 0, rng.randint(16, budget_max)])
        lo, hi = rng.choice([(12.0, 12.0), (12.0, 12.0), (6.0, 14.0)])
        c = _round("", batch, L, V, K, rng.choice([256, 2560, 4096, rng.randint(128, 4096)]), 16, budget_max, fixed, dtype,
                   rng.choice([128, 128, 128, 64]), rng.choice([0.2, 0.2, 0.2, 0.1, 0.0]), rng.choice([1, 1, 1, 0]), lo, hi)
        del c["name"]
        return c
    if kind == "shard":
        return dict(kind="shard", batch=_log_uniform(rng, 1, 128), L=rng.choice([16, rng.randint(4, 16)]),
                    V=rng.choice([128256, 151936, _log_uniform(rng, 32000, 151936)]), K=rng.choice([16, 32, rng.randint(4, 32)]),
                    world=rng.choice([2, 4, 8]), dtype=rng.choice(["bf16", "bf16", "f32"]))
    if kind == "loss":
        n = _log_uniform(rng, 500, 32768)
        return dict(kind="loss", V=rng.choice([151936, _log_uniform(rng, 16000, 151936)]), L=16, K=rng.choice([8, 16, 32, rng.randint(4, 32)]),
                    m=rng.choice([128, 128, 64]), groups=n, pairs=4 * n + rng.randint(0, 3), edges=8 * n + rng.randint(0, 3))
    if kind == "tables":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        return dict(kind="tables", V=_log_uniform(rng, 16000, 151936 if dtype == "bf16" else 64000),
                    E=rng.choice([1024, 2048, 4096 if dtype == "bf16" else 1536, 8 * rng.randint(100, 256)]), m=128, dtype=dtype)
    return dict(kind="fit", n=_log_uniform(rng, 20000, 4000000))


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _boosted_ids(gen, n, L, V):
    """[n, L, 64] distinct token ids a position, in the order of their boost."""
    start = torch.randint(0, V, (n, L, 1), generator=gen, device="cuda")
    stride = torch.randint(1, V // 64, (n, L, 1), generator=gen, device="cuda")
    return (start + stride * torch.arange(64, device="cuda")) % V


def _logits(gen, c, V, dtype):
    """([batch, L, V] logits, boosted ids)."""
    n, L = c["batch"], c["L"]
    ids = _boosted_ids(gen, n, L, V)
    lo, hi = c.get("boost_lo", 12.0), c.get("boost_hi", 12.0)
    height = lo + (hi - lo) * torch.rand((n, 1, 1), generator=gen, device="cuda")
    boost = (height - 0.4 * torch.arange(L, device="cuda")[:, None]) * torch.arange(1, 65, device="cuda") ** -1.1
    out = torch.empty((n, L, V), dtype=dtype, device="cuda")
    step = max(1, (1 << 27) // (L * V))
    for i in range(0, n, step):
        z = 2.0 * torch.randn((min(step, n - i), L, V), generator=gen, device="cuda")
        out[i:i + step] = z.scatter_add_(2, ids[i:i + step], boost[i:i + step].float())
    return out, ids


def _prepare_round(c, gen):
    n, L, V, m = c["batch"], c["L"], c["V"], c["m"]
    dtype, code, _ = _DTYPES[c["dtype"]]
    g = Graft(V, L, c["K"], m, c["hidden_dim"], n, c["budget_min"], c["budget_max"], 16, c["beta"], c["root_edge"], code, code)
    s = dict(g=g)
    if c["beta"] != 0:
        s["P"], s["C"] = (torch.randn((V, m), generator=gen, device="cuda") for _ in range(2))
        s["u"] = 0.5 * torch.randn((L, m), generator=gen, device="cuda")
        g.set_tdes_tables(s["P"], s["C"], s["u"], 1.0)
    s["logits"], ids = _logits(gen, c, V, dtype)
    s["root"] = torch.randint(0, V, (n,), generator=gen, device="cuda", dtype=torch.int32)
    s["prefix"] = torch.randint(128, 4097, (n,), generator=gen, device="cuda", dtype=torch.int32)
    if c["fixed"]:
        s["hidden"], s["hist"] = None, None
        s["fixed"] = torch.full((n,), c["fixed"], dtype=torch.int32, device="cuda")
    else:
        g.set_saba(phi_conf=-160.0, phi_degen=20.0, phi_hist=-5.0, phi_bias=200.0, tau_min=8.0, cost_mode=1,
                   pts_n=[0.0, 64.0, 1024.0], pts_t=[18.0, 18.0, 37.2])
        h = torch.randn((n, L, c["hidden_dim"]), generator=gen, device="cuda")
        for j in range(1, L):
            rho = 0.2 + 0.6 * j / (L - 1)
            h[:, j] = rho * h[:, j - 1] + math.sqrt(1.0 - rho * rho) * h[:, j]
        s["hidden"], s["fixed"] = h.to(dtype), None
        s["hist"] = 1.0 + 8.0 * torch.rand((n,), generator=gen, device="cuda")
    # the target model's continuation: the boosted token of Zipf-distributed rank, or any token
    rank = torch.multinomial(torch.arange(1, 65, device="cuda") ** -1.1, n * L, replacement=True, generator=gen).view(n, L, 1)
    p = 0.9 - 0.6 * torch.arange(L, device="cuda") / max(1, L - 1)
    match = torch.rand((n, L), generator=gen, device="cuda") < p
    y = torch.randint(0, V, (n, L + 1), generator=gen, device="cuda")
    y[:, :L] = torch.where(match, ids.gather(2, rank)[..., 0], y[:, :L])
    i32 = torch.int32
    s["out"] = g.alloc_out(n)
    s["len"] = torch.empty(n, dtype=i32, device="cuda")
    s["path"] = torch.empty((n, L), dtype=i32, device="cuda")
    s["bonus"] = torch.empty(n, dtype=i32, device="cuda")
    # the verifier's answer to the round's tree: the continuation's next token at every node's depth
    g.build_trees(s["logits"], s["hidden"], s["root"], s["hist"], s["prefix"], s["fixed"], s["out"])
    s["next"] = y.gather(1, s["out"].depth.long().clamp(min=0)).int()
    return s


def _run_round(s):
    g, o = s["g"], s["out"]
    g.build_trees(s["logits"], s["hidden"], s["root"], s["hist"], s["prefix"], s["fixed"], o)
    g.accept(o, s["next"], s["len"], s["path"], s["bonus"])
    return [o.n_nodes, o.budget, o.token, o.parent, o.depth, o.position, o.path_score, o.mask, o.status, s["len"], s["path"],
            s["bonus"]]


def _prepare_shard(c, gen):
    """Rank 0 of `world`: its slice of the logits, and the other ranks' pieces as the all-gather left them."""
    n, L, V, K, world = c["batch"], c["L"], c["V"], c["K"], c["world"]
    dtype, code, _ = _DTYPES[c["dtype"]]
    logits, _ = _logits(gen, c, V, dtype)
    parts = torch.empty((world, n * L, VOCAB_PARTIAL_BYTES), dtype=torch.uint8, device="cuda")
    s = dict(parts=parts, offsets=[vocab_range(V, r, world)[0] for r in range(world)])
    for r in reversed(range(world)):
        lo, hi = vocab_range(V, r, world)
        s["g"] = Graft(hi - lo, L, K, 128, 64, n, 16, 16, logits_dtype=code)
        s["shard"] = logits[:, :, lo:hi].contiguous()
        s["g"].vocab_pass_partial(s["shard"], parts[r])
    for k, shape, t in (("ids", (n, L, K), torch.int32), ("lp", (n, L, K), torch.float32), ("lse", (n, L), torch.float32),
                        ("status", (n, L), torch.int32)):
        s[k] = torch.empty(shape, dtype=t, device="cuda")
    return s


def _run_shard(s):
    s["g"].vocab_pass_partial(s["shard"], s["parts"][0])
    s["g"].vocab_merge(s["parts"], s["offsets"], s["ids"], s["lp"], s["lse"], s["status"])
    return [s["ids"], s["lp"], s["lse"], s["status"]]


def _prepare_loss(c, gen):
    V, L, K, m, n = c["V"], c["L"], c["K"], c["m"], c["groups"]
    perm = torch.randperm(V, generator=gen, device="cuda")
    cdf = torch.cumsum(torch.arange(1, V + 1, device="cuda", dtype=torch.float64) ** -1.1, 0)
    cdf /= cdf[-1].clone()

    def tokens(*shape):
        at = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
        return perm[torch.searchsorted(cdf, at).clamp(max=V - 1)].int()

    def depths(k):
        return torch.randint(1, L + 1, (k,), generator=gen, device="cuda", dtype=torch.int32)

    child = torch.empty((n, K), dtype=torch.int32, device="cuda")  # K distinct children a group
    for i in range(0, n, 8192):
        t = tokens(min(8192, n - i), 6 * K).sort(dim=1).values
        order = torch.rand(t.shape, generator=gen, device="cuda")
        order[:, 1:][t[:, 1:] == t[:, :-1]] = 2.0  # repeated tokens last
        child[i:i + 8192] = t.gather(1, order.argsort(dim=1)[:, :K])
    gaps = -1.0 / 1.4 * torch.log(1.0 - torch.rand((n, K), generator=gen, device="cuda"))
    groups = dict(parent=tokens(n), depth=depths(n), child=child, logq=-torch.cumsum(gaps, 1).float(),
                  ztgt=2.0 * torch.randn((n, K), generator=gen, device="cuda"))
    k = c["pairs"]
    pos = torch.stack([tokens(k), tokens(k), depths(k)], 1)
    swap = torch.rand(k, generator=gen, device="cuda") < 0.5
    neg = torch.stack([torch.where(swap, tokens(k), pos[:, 0]), torch.where(swap, pos[:, 1], tokens(k)), pos[:, 2]], 1)
    k = c["edges"]
    good = (torch.rand(k, generator=gen, device="cuda") < 0.15).int()
    edges = torch.stack([tokens(k), tokens(k), depths(k), good], 1).contiguous()
    s = dict(groups=groups, pairs=torch.cat([pos, neg], 1).contiguous(), edges=edges)
    s["P"], s["C"] = (torch.randn((V, m), generator=gen, device="cuda") for _ in range(2))
    s["u"] = 0.5 * torch.randn((L, m), generator=gen, device="cuda")
    s["g"] = Graft(V, L, K, m, 64, 1, 16, 16)
    s["g"].set_tdes_tables(s["P"], s["C"], s["u"], 1.0)
    s["loss"] = torch.empty(4, dtype=torch.float64, device="cuda")
    s["skipped"] = torch.empty(1, dtype=torch.int32, device="cuda")
    s["grads"] = [torch.empty(shape, device="cuda") for shape in ((V, m), (V, m), (L, m), (1,))]
    return s


def _run_loss(s):
    for t in s["grads"]:
        t.zero_()
    s["g"].tdes_loss(s["groups"], s["pairs"], s["edges"], gamma=0.5, w1=4.0, lambda_kl=1.0, lambda_pair=1.0, lambda_bce=0.25,
                     loss=s["loss"], skipped=s["skipped"], gP=s["grads"][0], gC=s["grads"][1], gu=s["grads"][2],
                     gs=s["grads"][3])
    return [s["loss"], s["skipped"]] + s["grads"]


def _prepare_tables(c, gen):
    V, E, m = c["V"], c["E"], c["m"]
    s = dict(g=Graft(V, 4, 4, m, 64, 1, 16, 16), emb=torch.empty((V, E), dtype=_DTYPES[c["dtype"]][0], device="cuda"))
    for i in range(0, V, 32768):
        s["emb"][i:i + 32768] = torch.randn((min(32768, V - i), E), generator=gen, device="cuda")
    for t in ("p", "c"):
        s["W" + t] = torch.randn((m, E), generator=gen, device="cuda") / math.sqrt(E)
        s["b" + t] = 0.1 * torch.randn((m,), generator=gen, device="cuda")
        s["out" + t] = torch.empty((V, m), device="cuda")
    return s


def _run_tables(s):
    for t in ("p", "c"):
        s["g"].tdes_precompute(s["emb"], s["W" + t], s["b" + t], s["out" + t])
    return [s["outp"], s["outc"]]


def _prepare_fit(c, gen):
    n = c["n"]
    state = torch.rand((n, 3), generator=gen, device="cuda") * torch.tensor([0.75, 0.9, 8.0], device="cuda")
    state += torch.tensor([0.2, 0.5, 0.0], device="cuda")
    budget = 32 + 16 * torch.randint(0, 31, (n,), generator=gen, device="cuda", dtype=torch.int32)
    prefix = torch.randint(16, 4097, (n,), generator=gen, device="cuda", dtype=torch.int32)
    tau = (state * torch.tensor([-160.0, 20.0, -5.0], device="cuda")).sum(1) + 200.0
    noise = 1.0 + 0.02 * torch.randn((2, n), generator=gen, device="cuda")
    gain = ((1.0 - torch.exp(-budget / tau.clamp(min=1.0))) * noise[0]).clamp(0.0, 1.0)
    latency = (6.0 + 0.012 * budget + 2.0e-6 * budget * prefix.float()) * noise[1]
    return dict(g=Graft(64, 4, 4, 4, 8, 1, 16, 512), args=(state, budget, gain, prefix, latency),
                out=torch.empty(10, dtype=torch.float64, device="cuda"))


def _run_fit(s):
    s["g"].saba_fit(*s["args"], s["out"])
    return [s["out"][:4], s["out"][4:7], s["out"][7:]]  # the gain model, the cost model, rounds used and status


_PREPARE = dict(round=_prepare_round, shard=_prepare_shard, loss=_prepare_loss, tables=_prepare_tables, fit=_prepare_fit)
_RUN = dict(round=_run_round, shard=_run_shard, loss=_run_loss, tables=_run_tables, fit=_run_fit)


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, _generator(seed))
    s["run"] = _RUN[case["kind"]]
    return s


def run(state):
    return state["run"](state)


def work(case):
    c = case
    if c["kind"] == "round":
        n, L, V, K, nmax = c["batch"], c["L"], c["V"], c["K"], c["budget_max"] + 1
        esz = _DTYPES[c["dtype"]][2]
        b = n * L * V * esz + n * nmax * (4 * 6 + 4 * ((nmax + 31) // 32))  # logits; tree arrays, masks and target ids
        if not c["fixed"]:
            b += n * L * c["hidden_dim"] * esz
        depths = 0 if c["beta"] == 0 else min(L, 4)  # the candidates of the first depths, which every tree reaches
        return {"bytes": b + n * depths * 2 * K * c["m"] * 4, "flops": 4.0 * n * L * V + 2.0 * n * depths * K * K * c["m"]}
    if c["kind"] == "shard":
        n, K, width = c["batch"] * c["L"], c["K"], vocab_range(c["V"], 0, c["world"])[1]
        return {"bytes": n * width * _DTYPES[c["dtype"]][2] + n * c["world"] * (24 + 8 * K) + n * (8 * K + 8), "flops": 4.0 * n * width}
    if c["kind"] == "loss":
        refs = c["groups"] * (K := c["K"]) + 2 * c["pairs"] + c["edges"]
        rows = min(c["V"], refs)
        traces = c["groups"] * (8 + 12 * K) + 24 * c["pairs"] + 16 * c["edges"]
        # both tables' rows read, both gradients cleared and written
        return {"bytes": traces + 2 * 4 * c["m"] * (2 * rows + c["V"]), "flops": 6.0 * refs * c["m"]}
    if c["kind"] == "tables":
        V, E, m = c["V"], c["E"], c["m"]
        return {"bytes": V * E * _DTYPES[c["dtype"]][2] + 2 * (m * E + m + V * m) * 4, "flops": 4.0 * V * E * m}
    return {"bytes": 36.0 * c["n"] + 80, "flops": 100.0 * c["n"]}


def tolerance(case):
    # Measured: a round against itself with the scale of the edge scores off by one part in 4 million, 2048 trees: the
    # same trees, path scores within 3e-8; path scores within 4e-6 of a 64-bit oracle at magnitudes near 10.  The losses
    # against 64-bit automatic differentiation: 3.7e-6, single entries 2.6e-4 (a row of the gradient is a sum of up to a
    # hundred thousand terms of both signs); tables against 64-bit products: 1.0e-6, single entries 6e-6.  The fit against
    # 64-bit normal equations in another order: 7e-12.
    return {
        "round": {"rel": 1e-6, "max": 1e-5, "differ": 0.0},
        "shard": {"rel": 1e-6, "max": 1e-5, "differ": 0.0},
        "loss": {"rel": 1.5e-5, "max": 1e-3},
        "tables": {"rel": 4e-6, "max": 4e-5},
        "fit": {"rel": 1e-10},
    }[case["kind"]]
