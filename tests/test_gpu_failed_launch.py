"""A launch that fails on the host: the call says so, and what the kernels ahead of it left in the context does not harm the
next calls.

No kernel goes wrong here.  A child process loads a small library ahead of the CUDA runtime that answers one call of
cudaLaunchKernelExC with an error instead of handing it on; programmatic launches are made through that call."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
static int wanted = 0, calls = 0;
int shim_calls(void) { return calls; }
void shim_fail(int nth) { wanted = nth; calls = 0; }  /* the nth call from here on; 0: none */
int cudaLaunchKernelExC(const void* config, const void* func, void** args) {
    static int (*real)(const void*, const void*, void**);
    if (!real) *(void**)&real = dlsym(dlopen("libcudart.so.12", RTLD_NOW | RTLD_NOLOAD), "cudaLaunchKernelExC");
    if (++calls == wanted) return 701; /* cudaErrorLaunchOutOfResources */
    return real(config, func, args);
}
"""


@pytest.mark.parametrize("case", ["round", "loss"])
def test_calls_after_a_launch_that_failed(tmp_path, case):
    src, so = os.path.join(str(tmp_path), "shim.c"), os.path.join(str(tmp_path), "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-O1", "-o", so, src, "-ldl"])
    r = subprocess.run([sys.executable, os.path.abspath(__file__), case, so], env=dict(os.environ, LD_PRELOAD=so), cwd=ROOT,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    assert "fine" in r.stdout


def _round(shim):
    """More sequences than SMs: the edge-score kernel counts them into an order that the tree kernel follows and clears."""
    import numpy as np
    import torch
    from paper_2608_20375_b200 import Graft, GraftError
    V, L, K, m, n, hd = 1500, 16, 8, 128, 330, 32
    gen = torch.Generator(device="cuda").manual_seed(4)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    g = Graft(V, L, K, m, hd, n, 16, 64, 16, 0.2, 1)
    P, Ct, u = rand(V, m), rand(V, m), 0.5 * rand(L, m)
    g.set_tdes_tables(P, Ct, u, 1.0)
    logits = (6.0 * rand(n, L, V) * torch.rand((n, 1, 1), generator=gen, device="cuda")).to(torch.bfloat16)
    root = torch.randint(0, V, (n,), generator=gen, device="cuda", dtype=torch.int32)
    prefix, fixed = torch.full_like(root, 100), torch.full_like(root, 48)

    def build():
        o = g.alloc_out(n)
        for t in (o.token, o.parent, o.n_nodes):
            t.fill_(-7)
        g.build_trees(logits, None, root, None, prefix, fixed, o)
        torch.cuda.synchronize()
        return o.cpu()

    want = build()
    shim.shim_fail(0)
    build()
    last = shim.shim_calls()  # the tree kernel's launch is the round's last
    assert last >= 2
    for _ in range(3):
        shim.shim_fail(last)
        try:
            build()
            raise SystemExit("the call did not report the launch that failed")
        except GraftError:
            pass
        torch.cuda.synchronize()
    shim.shim_fail(0)
    for _ in range(2):
        got = build()
        for k, w in want.items():
            if w is not None:
                assert np.array_equal(got[k], w), k


def _loss(shim):
    """Many traces: two kernels whose thread blocks count themselves; the last of all of them writes the losses."""
    import torch
    from paper_2608_20375_b200 import Graft, GraftError
    V, L, K, m, n = 3000, 16, 16, 128, 9000
    gen = torch.Generator(device="cuda").manual_seed(5)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    ints = lambda lo, hi, *s: torch.randint(lo, hi, s, generator=gen, device="cuda", dtype=torch.int32)  # noqa: E731
    g = Graft(V, L, K, m, 32, 1, 8, 16)
    P, Ct, u = rand(V, m), rand(V, m), 0.5 * rand(L, m)
    g.set_tdes_tables(P, Ct, u, 1.0)
    groups = dict(parent=ints(0, V, n), depth=ints(1, L + 1, n), child=ints(0, V, n, K), logq=rand(n, K), ztgt=rand(n, K))
    pairs = torch.stack([ints(0, V, n), ints(0, V, n), ints(1, L + 1, n), ints(0, V, n), ints(0, V, n), ints(1, L + 1, n)], 1).contiguous()
    edges = torch.stack([ints(0, V, n), ints(0, V, n), ints(1, L + 1, n), ints(0, 2, n)], 1).contiguous()

    def step():
        out = dict(loss=torch.zeros(4, dtype=torch.float64, device="cuda"), skipped=torch.zeros(1, dtype=torch.int32, device="cuda"),
                   gP=torch.zeros((V, m), device="cuda"), gC=torch.zeros((V, m), device="cuda"),
                   gu=torch.zeros((L, m), device="cuda"), gs=torch.zeros(1, device="cuda"))
        g.tdes_loss(groups, pairs, edges, gamma=0.5, w1=4.0, lambda_kl=1.0, lambda_pair=1.0, lambda_bce=0.25, **out)
        torch.cuda.synchronize()
        return out

    want = step()
    for _ in range(3):
        shim.shim_fail(1)  # (the second of the two kernels: the first is launched the ordinary way)
        try:
            step()
            raise SystemExit("the call did not report the launch that failed")
        except GraftError:
            pass
        torch.cuda.synchronize()
    shim.shim_fail(0)
    for _ in range(2):
        got = step()
        assert got["skipped"].item() == 0
        assert torch.allclose(got["loss"], want["loss"], rtol=1e-12, atol=0.0), (got["loss"], want["loss"])
        for k in ("gP", "gC", "gu"):
            assert ((got[k] - want[k]).abs().max() <= 1e-4 * want[k].abs().max()).item(), k


if __name__ == "__main__":
    import ctypes
    sys.path.insert(0, ROOT)
    {"round": _round, "loss": _loss}[sys.argv[1]](ctypes.CDLL(sys.argv[2]))
    print("fine")
