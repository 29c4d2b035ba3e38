"""Vocab pass with the rows held in shared memory, against the oracle, where its pieces can go wrong: rows shorter than a
vector, at the edges of a step of all threads and of a cluster's pieces, on no 16-byte boundary, and rows that overflow the
list of candidates in every way."""
import numpy as np
import pytest
import torch

import oracle
from helpers import tolerance

pytestmark = pytest.mark.gpu


def _row(style, V, g):
    z = 2.0 * torch.randn(V, generator=g)
    if style == "ascending":
        return z.sort().values
    if style == "descending":
        return z.sort(descending=True).values
    if style == "flat":
        return torch.full((V,), -1.5)
    if style == "masked":  # a few finite tokens more than K
        keep = torch.randperm(V, generator=g)[:40]
        out = torch.full((V,), -float("inf"))
        out[keep] = z[keep]
        return out
    if style == "ties":
        return (2.0 * z).round() / 2.0
    if style == "winners":  # fewer winners than K over an exactly flat rest
        z = torch.full((V,), -1.0)
        z[torch.randperm(V, generator=g)[:5]] = 4.0
        return z
    if style == "block":  # large elements side by side
        z[V // 3: V // 3 + V // 8] += 20.0
        return z
    if style == "ramps":
        return (torch.arange(V) % 1024).float() / 100.0 - 5.0
    return z


STYLES = ["random", "ascending", "descending", "flat", "masked", "ties", "winners", "block", "ramps"]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("batch,L,V,K,shift", [
    (2, 9, 41, 32, 1),         # five vectors a row, most rows on no 16-byte boundary
    (2, 9, 8176, 32, 0),       # bf16: one step of 256 threads with its two vectors of ragged ends, to the element
    (2, 9, 8177, 1, 3),        # and one element more
    (1, 9, 16001, 7, 1),
    (4, 10, 20011, 32, 0),     # a row a CTA, and more rows than stand alone
    (1, 9, 50021, 32, 5),      # four CTAs a row, uneven pieces; fp32: 200 KB
    (1, 9, 130003, 32, 0),     # rows that no CTA holds alone
    (5, 9, 54000, 32, 0),      # 512 threads a row (bf16: 108 KB; fp32: 216 KB)
])
def test_rows_in_shared_memory(batch, L, V, K, shift, dtype):
    from paper_2608_20375_b200 import Graft
    g = torch.Generator().manual_seed(V + K)
    z = torch.stack([_row(STYLES[r % len(STYLES)] if V > 1000 else "ties", V, g) for r in range(batch * L)]).to(dtype)
    flat = torch.empty(batch * L * V + 8, dtype=dtype, device="cuda")  # the rows begin `shift` elements behind a boundary
    x = flat[shift:shift + batch * L * V].view(batch, L, V)
    x.copy_(z.view(batch, L, V))
    gr = Graft(V, L, K, 16, 8, batch, 8, 8, 8, 0.0, 1, 1 if dtype == torch.bfloat16 else 0, 0)
    ids = torch.empty((batch, L, K), dtype=torch.int32, device="cuda")
    lp = torch.empty((batch, L, K), device="cuda")
    lse = torch.empty((batch, L), device="cuda")
    st = torch.empty((batch, L), dtype=torch.int32, device="cuda")
    gr.vocab_pass(x, ids, lp, lse, st)
    torch.cuda.synchronize()
    o_ids, o_lp, o_lse, o_st = oracle.vocab_pass(z, K)
    assert np.array_equal(st.cpu().numpy().reshape(-1), o_st)
    assert np.array_equal(ids.cpu().numpy().reshape(-1, K), o_ids)
    a, b = lp.cpu().numpy().reshape(-1, K).astype(np.float64), o_lp.astype(np.float64)
    assert np.array_equal(np.isneginf(a), np.isneginf(b))
    fin = np.isfinite(b)
    assert np.all(np.abs(a[fin] - b[fin]) <= tolerance(b[fin]))
    assert np.all(np.abs(lse.cpu().numpy().reshape(-1) - o_lse) <= tolerance(o_lse))


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_rows_in_shared_memory_report_bad_logits(bad):
    """A NaN, an infinity or nothing finite in any piece of a row marks that row and no other."""
    from paper_2608_20375_b200 import Graft
    L, V, K = 8, 60000, 8
    g = torch.Generator().manual_seed(3)
    z = 2.0 * torch.randn((1, L, V), generator=g)
    if bad == -float("inf"):
        z[0, 2] = bad
    else:
        z[0, 2, 1], z[0, 5, V - 2] = bad, bad
    gr = Graft(V, L, K, 16, 8, 1, 8, 8, 8, 0.0, 1, 0, 0)
    ids = torch.empty((1, L, K), dtype=torch.int32, device="cuda")
    lp, lse = torch.empty((1, L, K), device="cuda"), torch.empty((1, L), device="cuda")
    st = torch.empty((1, L), dtype=torch.int32, device="cuda")
    gr.vocab_pass(z.cuda(), ids, lp, lse, st)
    torch.cuda.synchronize()
    _, _, _, o_st = oracle.vocab_pass(z.view(L, V), K)
    assert np.array_equal(st.cpu().numpy().reshape(-1), o_st)
    assert o_st[2] == 1 and o_st[0] == 0


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("batch,V", [
    (2, 20011),    # a row a CTA
    (2, 75011),    # bf16: a row a CTA of 512 threads; fp32: clusters of four
    (1, 130003),   # clusters of four
    (20, 150001),  # the streaming kernel, whole rows and rows in pieces
])
def test_a_nan_among_masked_tokens_is_reported(batch, V, dtype):
    """Rows masked to -inf but for 40 tokens, and one NaN: at either ragged end, in the body, where no finite token is near it."""
    from paper_2608_20375_b200 import Graft
    L, K = 8, 32
    g = torch.Generator().manual_seed(7)
    z = torch.full((batch * L, V), -float("inf"))
    for r in range(batch * L):
        keep = torch.randint(V // 3, V // 2, (64,), generator=g).unique()[:40]
        z[r, keep] = torch.randn(len(keep), generator=g)
    places = [None, 0, V - 1, V // 4 + 13, 3 * V // 4 + 5, 9000, None, V - 2]
    for r in range(batch * L):
        if places[r % 8] is not None:
            z[r, places[r % 8]] = float("nan")
    z = z.to(dtype)
    gr = Graft(V, L, K, 16, 8, batch, 8, 8, 8, 0.0, 1, 1 if dtype == torch.bfloat16 else 0, 0)
    out = (torch.empty((batch, L, K), dtype=torch.int32, device="cuda"), torch.empty((batch, L, K), device="cuda"),
           torch.empty((batch, L), device="cuda"), torch.empty((batch, L), dtype=torch.int32, device="cuda"))
    gr.vocab_pass(z.view(batch, L, V).cuda(), *out)
    torch.cuda.synchronize()
    bad = np.array([places[r % 8] is not None for r in range(batch * L)]).astype(np.int32)
    assert np.array_equal(out[3].cpu().numpy().reshape(-1), bad)
    o_ids, _, _, o_st = oracle.vocab_pass(z[:8], K)
    assert np.array_equal(o_st, bad[:8])
    assert np.array_equal(out[0].cpu().numpy().reshape(-1, K)[:8][bad[:8] == 0], o_ids[bad[:8] == 0])


def _masked(batch, L, V, dtype, value, keep, g):
    z = torch.full((batch * L, V), value)
    for r in range(batch * L):
        at = torch.randperm(V, generator=g)[:keep]
        z[r, at] = torch.randn(keep, generator=g)
    if value > -float("inf"):  # elements just above and just below the value of the masked
        up = torch.tensor(value, dtype=dtype)
        z[0, V // 2] = torch.nextafter(up, torch.tensor(0.0, dtype=dtype)).float()
        z[1, ::7] = torch.nextafter(up, torch.tensor(-float("inf"), dtype=dtype)).float()
    return z.to(dtype).view(batch, L, V)


def _outputs(batch, L, K):
    return (torch.empty((batch, L, K), dtype=torch.int32, device="cuda"), torch.empty((batch, L, K), device="cuda"),
            torch.empty((batch, L), device="cuda"), torch.empty((batch, L), dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("value", [-float("inf"), -1e4, -17.3])
@pytest.mark.parametrize("V,keep", [(20011, 5), (20011, 40), (75000, 40), (130003, 5), (130003, 300)])
def test_masked_rows(V, keep, value, dtype):
    """Rows in which all but a few tokens hold one low value: fewer of them than K, a few more, more than the list takes."""
    from paper_2608_20375_b200 import Graft
    batch, L, K = 2, 4, 32
    z = _masked(batch, L, V, dtype, value, keep, torch.Generator().manual_seed(keep))
    gr = Graft(V, L, K, 16, 8, batch, 8, 8, 8, 0.0, 1, 1 if dtype == torch.bfloat16 else 0, 0)
    out = _outputs(batch, L, K)
    gr.vocab_pass(z.cuda(), *out)
    torch.cuda.synchronize()
    o_ids, o_lp, o_lse, o_st = oracle.vocab_pass(z.view(batch * L, V), K)
    assert np.array_equal(out[3].cpu().numpy().reshape(-1), o_st)
    assert np.array_equal(out[0].cpu().numpy().reshape(-1, K), o_ids)
    a, b = out[1].cpu().numpy().reshape(-1, K).astype(np.float64), o_lp.astype(np.float64)
    fin = np.isfinite(b)
    assert np.array_equal(np.isneginf(a), np.isneginf(b)) and np.all(np.abs(a[fin] - b[fin]) <= tolerance(b[fin]))
    assert np.all(np.abs(out[2].cpu().numpy().reshape(-1) - o_lse) <= tolerance(o_lse))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("batch,V", [(2, 151936), (16, 16000)])
@pytest.mark.parametrize("value", [-float("inf"), -1e4])
def test_masked_rows_take_no_longer_than_others(batch, V, value, dtype):
    """... or not much; by bisection 2 to 20 times as long."""
    from paper_2608_20375_b200 import Graft
    L, K = 16, 32
    gr = Graft(V, L, K, 16, 8, batch, 8, 8, 8, 0.0, 1, 1 if dtype == torch.bfloat16 else 0, 0)
    out = _outputs(batch, L, K)
    z = (2.0 * torch.randn((batch, L, V), device="cuda")).to(dtype)
    keep = torch.zeros((batch, L, V), dtype=torch.bool, device="cuda")
    keep.scatter_(2, torch.randint(0, V, (batch, L, 40), device="cuda"), True)
    times = []
    for x in (z, z.masked_fill(~keep, value)):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        best = float("inf")
        for _ in range(5):
            a.record()
            for _ in range(20):
                gr.vocab_pass(x, *out)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] < 2.0 * times[0], times


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("value", ["lowest", -1e30, -1e10, -1e9, -3e4])
@pytest.mark.parametrize("batch,V,shift", [(2, 20011, 1), (2, 75011, 3), (1, 130003, 1), (20, 150001, 1)])
def test_rows_masked_far_below(batch, V, shift, value, dtype):
    """Low values whose product with log2(e) is infinite or rounded by more than an exponent holds, with neighbours a spacing or
    a few apart, at the ragged ends of rows too: nothing is wrong with such rows."""
    from paper_2608_20375_b200 import Graft
    L, K, n = 8, 32, 8
    low = torch.tensor(torch.finfo(dtype).min if value == "lowest" else value, dtype=dtype)
    z = _masked(1, n, V, dtype, low.item(), 40, torch.Generator().manual_seed(9)).view(n, V)
    if value == "lowest":
        z[1] = z[0]  # (_masked puts infinities beside its second row's values)
    for r in range(2, 5):  # the masked of the row's second half a spacing up, two, three
        up = low
        for _ in range(r - 1):
            up = torch.nextafter(up, torch.tensor(0.0, dtype=dtype))
        half = z[r, V // 2:]
        half[half == low] = up
    flat = torch.empty(batch * L * V + 8, dtype=dtype, device="cuda")
    x = flat[shift:shift + batch * L * V].view(batch, L, V)
    x.copy_(z.cuda().expand(batch, L, V))
    gr = Graft(V, L, K, 16, 8, batch, 8, 8, 8, 0.0, 1, 1 if dtype == torch.bfloat16 else 0, 0)
    out = _outputs(batch, L, K)
    gr.vocab_pass(x, *out)
    torch.cuda.synchronize()
    o_ids, o_lp, o_lse, o_st = oracle.vocab_pass(z, K)
    assert not o_st.any()
    for b in range(batch):
        assert np.array_equal(out[3][b].cpu().numpy(), o_st)
        assert np.array_equal(out[0][b].cpu().numpy(), o_ids)
        assert np.all(np.abs(out[1][b].cpu().numpy().astype(np.float64) - o_lp) <= tolerance(o_lp))
        assert np.all(np.abs(out[2][b].cpu().numpy() - o_lse) <= tolerance(o_lse))


@pytest.mark.parametrize("batch,V", [(4, 99000), (3, 101003), (4, 151936), (5, 101003)])  # one turn of clusters, two in a round, streamed
def test_rows_of_a_round_and_of_a_call_of_its_own(batch, V):
    """fp32 rows near 390 KB, which rounds and calls of the vocab pass alone may cut in different ways: the same candidates."""
    from paper_2608_20375_b200 import Graft
    L, K = 16, 16
    g = torch.Generator(device="cuda").manual_seed(V)
    z = 2.0 * torch.randn((batch, L, V), generator=g, device="cuda")
    z[:, :, 7::1000] = 6.5  # (ties that decide)
    gr = Graft(V, L, K, 16, 64, batch, 16, 64, 16, 0.2, 1, 0, 0)
    P, Ct = (torch.randn((V, 16), generator=g, device="cuda") for _ in range(2))
    gr.set_tdes_tables(P, Ct, torch.randn((L, 16), generator=g, device="cuda"), 1.0)
    o = gr.alloc_out(batch, debug=True)
    ones = torch.ones(batch, dtype=torch.int32, device="cuda")
    gr.build_trees(z, None, ones, None, 100 * ones, 32 * ones, o)
    out = _outputs(batch, L, K)
    gr.vocab_pass(z, *out)
    torch.cuda.synchronize()
    assert torch.equal(o.topk_id.view(batch, L, K), out[0]) and not out[3].any() and not o.status.any()
    assert (o.topk_lp.view(batch, L, K) - out[1]).abs().max() <= 4e-6  # (two spacings at 10)
    o_ids, _, o_lse, _ = oracle.vocab_pass(z[0].cpu(), K)
    assert np.array_equal(out[0][0].cpu().numpy(), o_ids)
    assert np.all(np.abs(o.lse.view(batch, L)[0].cpu().numpy() - o_lse) <= tolerance(o_lse))
