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


@pytest.mark.parametrize("V,E,m", [
    (130, 20, 32),       # less than a block of columns
    (500, 288, 128),     # nine blocks: the second chunk, on the accumulators' other side, has one
    (500, 544, 96),      # seventeen: three chunks, the last of one block
    (129, 32, 200),      # two blocks of m, the second of 72 columns; a row in the second tile
    (19000, 2080, 128),  # a whole tile and shares of the tiles left, which begin and end anywhere
    (57000, 1056, 64),   # several whole tiles a worker, an odd number of chunks each
])
def test_fp32_chunks_and_tiles_of_odd_lengths(V, E, m):
    """The large products' accumulators take turns on either side of the small ones', which last a tile: every chunk and every tile
    counts once.  The sums are about 1; the parts of order 2^-11 of every chunk are 1e-4 of them and more."""
    emb, W, b = _inputs(V, E, m, "f32", 11)
    got = _call(_graft(V, m), emb, W, b, m).double()
    want = _exact(emb, W, b)
    assert ((got - want).abs() <= 1e-5 + 1e-6 * want.abs()).all()  # (a sum's rounding: 2e-6 at most, measured)


@pytest.mark.parametrize("V,E,m,dtype", [(5, (1 << 22) + 64, 8, "f32"), (5, (1 << 22) + 64, 8, "bf16"), (130, (1 << 23) + 4, 4, "f32")])
def test_rows_of_many_million_columns(V, E, m, dtype):
    """Tables of any length that fits in memory go to the tensor cores (more than one kernel a table)."""
    emb, W, b = _inputs(V, E, m, dtype, 13)
    g = _graft(V, m)
    n = g.launch_count()
    got = _call(g, emb, W, b, m).double()
    assert g.launch_count() - n > 1
    want = b.double() + sum(_exact(emb[:, i:i + (1 << 19)], W[:, i:i + (1 << 19)]) for i in range(0, E, 1 << 19))
    assert ((got - want).abs() <= 2e-5 + 2e-6 * want.abs()).all()
    g.destroy()


@pytest.mark.parametrize("part", ["embedding", "W", "both"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_parts_of_every_order_count(part, dtype):
    """Terms +-(1 + 2^-10 + t 2^-19) whose leading parts cancel: what the last part holds (W beside bf16 embeddings: the third, fp32
    embeddings and their W: the second) is the whole result, exactly (all sums are short multiples of powers of two)."""
    if dtype == "bf16" and part != "W":
        pytest.skip("bf16 embeddings have one part")
    V, E, m = 1000, 2048, 128
    g = torch.Generator(device="cuda").manual_seed(6)
    sign = torch.where(torch.arange(E, device="cuda") % 2 == 0, 1.0, -1.0)
    third = lambda n: 1.0 + 2.0 ** -10 + 2.0 ** -19 * torch.randint(0, 3, (n, E), generator=g, device="cuda")  # noqa: E731
    emb = (third(V) if part != "W" else torch.ones((V, E), device="cuda")) * sign
    W = third(m) if part != "embedding" else torch.ones((m, E), device="cuda")
    got, want = _call(_graft(V, m), emb.to(DTYPES[dtype]), W, None, m).double(), _exact(emb, W)
    assert want.abs().max() > 1e-5
    # where both numbers have a part of some 2^-19, their product is left out: far below 2^-27 a term
    assert (got - want).abs().max() <= (2.0 ** -27 * E if part == "both" else 0.0)


@pytest.mark.parametrize("V,E,m,dtype", [(8192, 4096, 128, "bf16"), (8192, 2048, 128, "f32")])
def test_error_against_64_bit_products(V, E, m, dtype):
    """N(0, 1) embeddings, results of N(0, 1): twice the largest error seen over a million results (3.2e-6; in fp32 2.2e-6, with three
    bf16 parts 3.0e-6; a chain of fp32 multiply-adds 1.2e-5)."""
    emb, W, _ = _inputs(V, E, m, dtype, 8)
    assert (_call(_graft(V, m), emb, W, None, m) - _exact(emb, W)).abs().max() <= 6e-6


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("off", ["embedding", "out", "neither"])
def test_rows_off_the_16_byte_grid(dtype, off):
    """Pointers that the tensor cores' copies cannot take go to the FMA kernel."""
    V, E, m = 333, 72, 20
    emb, W, b = _inputs(V, E, m, dtype, 9)
    pad = torch.empty(V * E + 8, dtype=DTYPES[dtype], device="cuda")
    o_pad = torch.full((V * m + 8,), 7.0, device="cuda")
    i, j = (1 if off == "embedding" else 0), (1 if off == "out" else 0)
    e2, out = pad[i:i + V * E].view(V, E), o_pad[j:j + V * m].view(V, m)
    e2.copy_(emb)
    _graft(V, m).tdes_precompute(e2, W, b, out)
    torch.cuda.synchronize()
    assert (out - _exact(emb, W, b)).abs().max() < 1e-5
    assert (o_pad[:j] == 7.0).all() and (o_pad[j + V * m:] == 7.0).all()


@pytest.mark.parametrize("V,E,m", [(300, 64, 128), (19300, 1092, 40), (40003, 132, 256)])  # whole tiles, pieces, both
def test_fp32_rows_of_other_sizes(V, E, m):
    """Rows far larger or smaller than the others, rows of zeros, rows with one large entry, and columns of W of every size: an error
    of 2e-5 (the chain of fp32 multiply-adds: 1.2e-5) of a result's size, row by row."""
    emb, W, _ = _inputs(V, E, m, "f32", 11)
    size = torch.ones(V, device="cuda")
    for i, e in enumerate((-100, -40, -25, -19, -17, -12, -9, 5, 8, 9, 16, 40, 60)):
        size[(7919 * i) % V], size[V - 1 - i] = 2.0 ** e, 2.0 ** e
    emb *= size[:, None]
    emb[V // 3] = 0.0
    emb[V // 4, E // 2], emb[V // 5, 0] = 200.0, 3e4  # (beside entries of N(0, 1))
    size[V // 4], size[V // 5] = 4.0, 3e4 * E ** -0.5 + 1.0
    wide = 2.0 ** (torch.arange(m, device="cuda") % 50 - 30)
    W = W * wide[:, None]
    got = _call(_graft(V, m), emb, W, None, m).double()
    # (sums in fp32's denormals, the smallest rows and columns: half a spacing of 1.4e-45 an addition)
    bound = 2e-5 * size[:, None].double() * wide[None].double() + 0.7e-45 * E
    over = (got - _exact(emb, W)).abs() / bound
    assert over.max() <= 1.0, (over.max(), over.argmax() // m, size[over.argmax() // m], over.argmax() % m)


@pytest.mark.parametrize("row", ["a small piece", "a piece of two sizes"])
def test_fp32_rows_are_judged_tile_by_tile(row):
    """Three blocks of columns of the table, of which two are left over and cut along E while the third is worked out whole: a row that only
    the pieces' workers find unfit for fp16 parts keeps its results in the third block, whatever else is worked out again there."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m, E = 384, 2048
    tiles = next(t for t in range(sms + 1, sms + 10) if t % 3 == 0 and (t - sms) % 3 != 0)
    V = tiles // 3 * 128
    emb, W, _ = _inputs(V, E, m, "f32", 12)
    if row == "a small piece":
        emb[10, 256:512] *= 2.0 ** -25
    else:
        emb[10, 256:288] *= 2.0 ** -9
        emb[10, 320:352] *= 2.0 ** 6
    g = _graft(V, m)
    want = _call(g, emb, W, None, m)
    emb[20, 0] = float("inf")  # (its results are not finite: the third block's tile of these rows is looked through)
    got = _call(g, emb, W, None, m)
    rest = torch.arange(V, device="cuda") != 20
    assert torch.equal(got[rest], want[rest])
    assert not got[20].isfinite().any()


def _row_error(got, emb, W):
    """The largest error, of results of N(0, 1) for rows of N(0, 1), over the size of the row."""
    size = emb.double().pow(2).mean(1, keepdim=True).sqrt().clamp(min=1e-300)
    return ((got.double() - _exact(emb, W)).abs() / size).max().item()


def _best_time(f):
    best = float("inf")
    for _ in range(4):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("factor", [300.0, 1000.0, 1e-3, 1e7])
@pytest.mark.parametrize("column", [5, 1000])  # in the block of columns by which a row is scaled, and not
def test_fp32_column_of_another_size(column, factor):
    """One column far larger or smaller than the others: no less precise than N(0, 1) alone (6e-6 of a row's size), and as fast as that
    where fp16 parts hold it; where they do not (1e7 times), faster than the FMA kernel."""
    V, E, m = 32000, 2048, 128
    emb, W, _ = _inputs(V, E, m, "f32", 13)
    out, g = torch.zeros((V, m), device="cuda"), _graft(V, m)
    pad = torch.zeros(V * m + 4, device="cuda")
    ordinary = _best_time(lambda: g.tdes_precompute(emb, W, None, out))
    fma = _best_time(lambda: g.tdes_precompute(emb, W, None, pad[1:1 + V * m].view(V, m)))  # (off the 16-byte grid)
    emb[:, column] *= factor
    assert _row_error(_call(g, emb, W, None, m), emb, W) <= 6e-6
    taken = _best_time(lambda: g.tdes_precompute(emb, W, None, out))
    assert taken < (2.5 * ordinary if factor < 1e6 else fma), (ordinary, fma, taken)
    # W made the other way round, so that all columns count as much
    W[:, column] /= factor
    like = emb.clone()
    like[:, column] /= factor
    got, want = _call(g, emb, W, None, m).double(), _exact(emb, W)
    size = like.double().pow(2).mean(1, keepdim=True).sqrt()
    assert ((got - want).abs() / size).max() <= 6e-6


@pytest.mark.parametrize("V,E,m", [(300, 64, 128), (19300, 1092, 40), (40003, 132, 256)])  # whole tiles, pieces, both
def test_fp32_rows_of_other_sizes_are_as_precise(V, E, m):
    """Rows of every size, rows that begin with zeros, blocks of a row of other sizes than its first: twice the largest error of
    N(0, 1) (6e-6 of a row's size; one chain of fp32 multiply-adds is off by 1.2e-5)."""
    emb, W, _ = _inputs(V, E, m, "f32", 14)
    W = W.clone()
    for i, e in enumerate((-90, -60, -30, -19, -12, -7, 7, 8, 9, 16, 40, 60)):
        emb[(7919 * i) % V] *= 2.0 ** e
        emb[V - 1 - i, E // 2:] *= 2.0 ** e
        emb[(4001 * i + 17) % V, :32] *= 2.0 ** e
    emb[V // 2, :40], emb[V // 3, :32] = 0.0, 0.0
    emb[V // 3] *= 2.0 ** 20
    emb[V // 4, :33] = 1e-39
    assert _row_error(_call(_graft(V, m), emb, W, None, m), emb, W) <= 6e-6
