"""Parity of graft_saba_fit (least-squares fit of the SABA models, Eq. 16-17) with the oracle, through the C ABI."""
import numpy as np
import pytest
import torch

import graft_inputs as gi
import oracle

pytestmark = pytest.mark.gpu

# both sides work in fp64 on the same fp32 logs; the library solves the normal equations (columns scaled), the oracle
# an SVD: the difference is the conditioning of the scaled normal equations times fp64 rounding
RTOL = 1e-8


def _ctx():
    from paper_2608_20375_b200 import Graft
    return Graft(1000, 4, 4, 16, 8, 1, 8, 8, 8, 0.0, 1, 0, 0)


def _fit(g, lg):
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in lg.items()}
    out = torch.full((10,), 7.0, dtype=torch.float64, device="cuda")
    g.saba_fit(dev["state"], dev["budget"], dev["gain"], dev["prefix_len"], dev["latency"], out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("n,seed,noise", [(7, 1, 0.02), (1000, 2, 0.02), (100003, 3, 0.05), (2_000_000, 4, 0.02),
                                          (5000, 5, 0.0)])
def test_fit_matches_the_oracle(n, seed, noise):
    g = _ctx()
    lg = gi.saba_replay_logs(n, seed=seed, noise=noise)
    ref = oracle.saba_fit(**lg)
    for _ in range(2):  # the accumulators clear themselves: a second call gives the same answer
        got = _fit(g, lg)
        assert got[9] == 0.0
        assert got[7] == ref["n_gain"] and got[8] == ref["n_cost"]
        scale_phi = np.abs(ref["phi"]).max()
        assert np.all(np.abs(got[:4] - ref["phi"]) <= RTOL * scale_phi * 10), (got[:4], ref["phi"])
        assert np.all(np.abs(got[4:7] - ref["c"]) <= RTOL * np.maximum(np.abs(ref["c"]), 1e-9) * 100), (got[4:7], ref["c"])
    g.destroy()


def test_degenerate_logs_are_reported():
    g = _ctx()
    lg = gi.saba_replay_logs(50, seed=8)
    lg["gain"][:] = 1.0               # nothing to fit the gain model to
    lg["budget"][:] = 64              # one budget: the cost columns are dependent
    lg["prefix_len"][:] = 100
    got = _fit(g, lg)
    assert int(got[9]) == 3 and not np.any(got[:7])
    assert got[7] == 0 and got[8] == 50
    # a usable call afterwards is not disturbed by the failed one
    lg2 = gi.saba_replay_logs(500, seed=9)
    ref = oracle.saba_fit(**lg2)
    got2 = _fit(g, lg2)
    assert got2[9] == 0.0 and np.allclose(got2[4:7], ref["c"], rtol=1e-6)
    g.destroy()


def test_unaligned_arrays_take_the_scalar_path():
    g = _ctx()
    lg = gi.saba_replay_logs(3001, seed=12)
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in lg.items()}
    out = torch.zeros(10, dtype=torch.float64, device="cuda")
    # views that start one round in: 4 bytes (12 for the state) past a 16-byte boundary
    g.saba_fit(dev["state"][1:], dev["budget"][1:], dev["gain"][1:], dev["prefix_len"][1:], dev["latency"][1:], out)
    torch.cuda.synchronize()
    ref = oracle.saba_fit(**{k: v[1:] for k, v in lg.items()})
    got = out.cpu().numpy()
    assert got[9] == 0.0 and got[8] == 3000
    assert np.allclose(got[:4], ref["phi"], rtol=1e-7) and np.allclose(got[4:7], ref["c"], rtol=1e-7)
    g.destroy()


@pytest.mark.parametrize("g0", [1e-42, 2.0 ** -60, 2.0 ** -29, 2.0 ** -10, 2.0 ** -9, 0.25, 0.5, 0.625, 1 - 2.0 ** -9, 1 - 2.0 ** -22])
def test_logarithms_of_gains(g0):
    """Gains around one value, on both sides of where the logarithm's table changes its entry or its way: the gain model is a
    regression of -B / ln(1 - g), so an error there shows in it."""
    rng = np.random.default_rng(13)
    n = 4003
    gain = (np.float64(g0) * (1.0 + rng.integers(-4, 5, n) * (2.0 ** -4 if g0 < 0.5 else 2.0 ** -24))).astype(np.float32)
    lg = dict(state=rng.random((n, 3), dtype=np.float32), budget=rng.integers(16, 513, n).astype(np.int32),
              gain=np.minimum(gain, np.float32(1 - 2.0 ** -24)), prefix_len=rng.integers(1, 4096, n).astype(np.int32),
              latency=rng.random(n, dtype=np.float32) + 1)
    ref = oracle.saba_fit(**lg)
    g = _ctx()
    got = _fit(g, lg)
    assert got[9] == 0.0 and got[7] == ref["n_gain"] == n
    assert np.all(np.abs(got[:4] - ref["phi"]) <= RTOL * np.abs(ref["phi"]).max()), (got[:4], ref["phi"])
    g.destroy()


@pytest.mark.parametrize("n", [2047, 2049, 303103, 303109, 606211])  # rounds of a thread, of all CTAs once and twice: one less, some more
def test_sizes_around_whole_turns_back_to_back(n):
    """Calls that follow one another at once, on other logs: each has its own sums."""
    g = _ctx()
    logs = [gi.saba_replay_logs(n + 3 * k, seed=20 + k) for k in range(3)]
    dev = [{k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in lg.items()} for lg in logs]
    outs = torch.zeros((6, 10), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for i in range(6):
        d = dev[i % 3]
        g.saba_fit(d["state"], d["budget"], d["gain"], d["prefix_len"], d["latency"], outs[i])
    got = outs.cpu().numpy()
    for i in range(6):
        ref = oracle.saba_fit(**logs[i % 3])
        assert got[i, 9] == 0.0 and got[i, 7] == ref["n_gain"] and got[i, 8] == ref["n_cost"]
        assert np.all(np.abs(got[i, :4] - ref["phi"]) <= RTOL * np.abs(ref["phi"]).max() * 10)
        assert np.all(np.abs(got[i, 4:7] - ref["c"]) <= RTOL * np.maximum(np.abs(ref["c"]), 1e-9) * 100)
    g.destroy()


@pytest.mark.parametrize("n,odd", [(257, False), (1021, True), (131056, False), (131060, False), (131063, False), (32767, True), (32768, True)])
def test_sizes_where_the_thread_blocks_change(n, odd):
    """The last size of the smaller thread blocks and the first of the larger, with four rounds a turn and with one."""
    g = _ctx()
    lg = gi.saba_replay_logs(n, seed=n)
    ref = oracle.saba_fit(**lg)
    dev = {}
    for k, v in lg.items():  # (four bytes behind a boundary: one round a turn)
        flat = torch.from_numpy(np.ascontiguousarray(v)).reshape(-1)
        buf = torch.zeros(flat.numel() + 1, dtype=flat.dtype, device="cuda")
        part = buf[1:] if odd else buf[:-1]
        part.copy_(flat)
        dev[k] = part.view(v.shape)
    out = torch.zeros((3, 10), dtype=torch.float64, device="cuda")
    for i in range(3):
        g.saba_fit(dev["state"], dev["budget"], dev["gain"], dev["prefix_len"], dev["latency"], out[i])
    for got in out.cpu().numpy():
        assert got[9] == 0.0 and got[7] == ref["n_gain"] and got[8] == ref["n_cost"]
        assert np.all(np.abs(got[:4] - ref["phi"]) <= RTOL * np.abs(ref["phi"]).max() * 10)
        assert np.all(np.abs(got[4:7] - ref["c"]) <= RTOL * np.maximum(np.abs(ref["c"]), 1e-9) * 100)
    g.destroy()


def test_first_call_on_a_stream_of_its_own_behind_a_busy_default_stream():
    """A context is ready when its creation returns: the first call need not wait for the default stream, nor for what is queued there."""
    lg = gi.saba_replay_logs(900, seed=3)
    ref = oracle.saba_fit(**lg)
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in lg.items()}
    out = torch.zeros((20, 10), dtype=torch.float64, device="cuda")
    a = torch.ones((4096, 4096), device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    made = []
    for i in range(20):
        for _ in range(20):
            a.mul_(1.0)
        made.append(_ctx())
        with torch.cuda.stream(side):
            made[-1].saba_fit(dev["state"], dev["budget"], dev["gain"], dev["prefix_len"], dev["latency"], out[i])
    torch.cuda.synchronize()
    for got in out.cpu().numpy():
        assert got[9] == 0.0 and got[7] == ref["n_gain"] and got[8] == ref["n_cost"]
        assert np.all(np.abs(got[:4] - ref["phi"]) <= RTOL * np.abs(ref["phi"]).max() * 10)
    for g in made:
        g.destroy()
