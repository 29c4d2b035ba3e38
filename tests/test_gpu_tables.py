"""The table precompute beyond its parity with the oracle: where its scratch comes from, entries that bf16 parts cannot
hold, the parts themselves, and the way into the FMA kernel."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _graft(V, m):
    from paper_2608_20375_b200 import Graft
    return Graft(V, 4, 4, m, 64, 1, 16, 16)


def _inputs(V, E, m, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    emb = torch.randn((V, E), generator=g, device="cuda").to(DTYPES[dtype])
    W = torch.randn((m, E), generator=g, device="cuda") / E ** 0.5
    return emb, W, torch.randn(m, generator=g, device="cuda")


def _exact(emb, W, b=None):
    out = emb.double() @ W.double().T
    return out if b is None else out + b.double()


def _call(g, emb, W, b, m):
    out = torch.full((emb.shape[0], m), 7.0, device="cuda")
    g.tdes_precompute(emb, W, b, out)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_first_call_under_capture_and_a_larger_call_after_it(dtype):
    """A captured call stays good when a later call of the context needs more scratch than it did."""
    V, m = 700, 24
    emb, W, b = _inputs(V, 64, m, dtype, 1)
    big, W_big, _ = _inputs(V, 8192, m, dtype, 2)
    g = _graft(V, m)
    out = torch.zeros((V, m), device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        g.tdes_precompute(emb, W, b, out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, _call(_graft(V, m), emb, W, b, m))
    for E in (4096, 8192):  # (more scratch each time)
        got = _call(g, big[:, :E].contiguous(), W_big[:, :E].contiguous(), None, m)
        assert (got - _exact(big[:, :E], W_big[:, :E])).abs().max() < 2e-5
    emb.copy_(_inputs(V, 64, m, dtype, 3)[0])
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, _call(_graft(V, m), emb, W, b, m))
    del graph


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_no_memory_for_the_scratch(dtype):
    """The FMA kernel needs none and takes over."""
    V, E, m = 700, 64, 24
    emb, W, b = _inputs(V, E, m, dtype, 4)
    g = _graft(V, m)
    odd = _call(g, emb[:, :E - 1].contiguous(), W[:, :E - 1].contiguous(), b, m)  # (loads the FMA kernel)
    want, out = _exact(emb, W, b), torch.zeros((V, m), device="cuda")
    torch.cuda.synchronize()
    hold, size = [], 1 << 35
    while size >= 1 << 21:
        try:
            hold.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.cuda.OutOfMemoryError:
            size >>= 1
    try:
        g.tdes_precompute(emb, W, b, out)
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert (out - want).abs().max() < 2e-5
    assert (odd - _exact(emb[:, :E - 1], W[:, :E - 1], b)).abs().max() < 2e-5
    assert (_call(g, emb, W, b, m) - want).abs().max() < 2e-5  # and with memory again


@pytest.mark.parametrize("V,E,m", [(300, 64, 128), (19300, 1092, 40), (40003, 132, 256)])  # whole tiles, pieces, both
def test_fp32_entries_that_bf16_parts_cannot_hold(V, E, m):
    """Infinities, NaN and finite values that round past the largest bf16, in the embeddings and in W: what fp32 arithmetic
    gives, and nothing else is touched."""
    emb, W, b = _inputs(V, E, m, "f32", 5)
    inf, huge = float("inf"), 3.4e38
    emb[:, 0] *= 0.1  # (times -huge, below: finite, on the way too)
    for v, x in ((0, inf), (1, -inf), (2, huge), (3, -huge), (4, float("nan")), (V // 2, inf), (V - 1, huge)):
        emb[v, (7 * v) % E] = x
    emb[5, 3], emb[5, 9] = inf, -inf
    emb[6] = 0.0
    W[0, 5], W[m - 1, 0] = inf, -huge
    W[:, 1] = 0.0
    emb[7, 1] = inf       # (infinity times zero)
    got = _call(_graft(V, m), emb, W, b, m).double()
    want = _exact(emb, W, b)
    over = want.abs() > 3.4028234e38  # past fp32 (with the sums' rounding to either side of the limit, none is near it)
    want[over] = want[over].sign() * inf
    assert torch.equal(got.isnan(), want.isnan())
    assert torch.equal(got.isinf(), want.isinf()) and torch.equal(got[got.isinf()], want[want.isinf()])
    fin = want.isfinite()
    assert ((got - want)[fin].abs() <= 2e-5 + 2e-6 * want[fin].abs()).all()
