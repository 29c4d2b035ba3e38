"""A bounded device-side wait that runs out: the kernel must return, say so in the rows' status words, and leave the
device usable.

The vocab pass waits on shared-memory barriers with an iteration limit; when a wait gives up, the thread block
raises a flag, stops waiting, drains its copies in flight and finishes, and every row it finishes or leaves a piece of
carries GRAFT_ST_INTERNAL.  To make a wait run out without faulting, trapping or hanging anything, this test compiles
a SECOND copy of the vocab pass (one source file, into a temporary folder) with a tiny iteration limit and a build flag
under which one thread block never issues the copy of its third tile.  The shipped library is not touched.  A second flag
lets the other thread blocks leave their records of shared rows some milliseconds late, after block 0 has given up: the
block that merges block 0's row has seen no time-out itself and knows of it from block 0's record alone.  A third keeps
one block of every cluster from saying that the rest of its list of candidates is there.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

ST_INTERNAL = 8


def _build_test_library(tmp_path, *flags, withheld="-DGRAFT_TEST_WITHHOLD_TILE=2"):
    from paper_2608_20375_b200 import build as b
    out = os.path.join(str(tmp_path), "libgraft_waittest.so")
    cmd = [os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *b.NVCC_FLAGS, "-DGRAFT_SPIN_LIMIT=512u",
           withheld, *flags, "-I", os.path.join(b.HERE, "..", "include"), "-shared",
           os.path.join(b.CSRC, "vocab_pass.cu"), "-o", out, "-lcudart"]
    subprocess.check_call(cmd, stderr=subprocess.DEVNULL)
    return out


@pytest.mark.parametrize("Bt,L,flagged_rows", [
    (8, 16, [0]),       # fewer rows than SMs, one whole row of ten tiles per thread block
    (12, 16, [0, 1]),   # more rows than SMs, equal shares: block 0 has row 0 and, visited first, three tiles of row 1
])
def test_a_wait_that_runs_out_is_reported_and_the_device_stays_usable(tmp_path, Bt, L, flagged_rows):
    _case(_build_test_library(tmp_path), Bt, L, flagged_rows)


@pytest.mark.parametrize("Bt,V,block,flagged_rows", [
    (4, 50021, 5, [5]),     # a row a thread block of 256 threads, six tiles
    (4, 75000, 0, [0]),     # of 512 threads, four tiles
    (1, 151936, 4, [1]),    # a row a cluster of four, four tiles each: the block that ranks the row's candidates
    (1, 151936, 6, [1]),    # and another, which tells the first with its number of candidates
])
def test_a_wait_that_runs_out_on_a_row_in_shared_memory_is_reported(tmp_path, Bt, V, block, flagged_rows):
    _case(_build_test_library(tmp_path, f"-DGRAFT_TEST_WITHHOLD_CTA={block}"), Bt, 16, flagged_rows, V=V)


def test_a_wait_that_runs_out_is_reported_by_the_block_that_merges_the_row(tmp_path):
    # rows too long for a cluster's shared memory: nine pieces a row, a thread block each, which meet through records in global memory
    _case(_build_test_library(tmp_path, "-DGRAFT_TEST_LATE_RECORDS=20"), 1, 16, [0], V=480000)


def test_a_wait_that_runs_out_after_the_lists_were_sent_is_reported(tmp_path):
    # clusters of four; one row has over 32 candidates in every piece and the arrival behind a piece's list never comes: the first
    # block of that cluster gives up when all counts are there.  Other rows' lists are short and nothing waits for that arrival.
    _case(_build_test_library(tmp_path, withheld="-DGRAFT_TEST_WITHHOLD_LISTS"), 1, 16, [3], ties=3)


def _case(so, Bt, L, flagged_rows, V=151936, ties=None):
    lib = C.CDLL(so)
    vp = C.c_void_p
    lib.graft_vocab_pass_static.argtypes = [C.c_int32, C.c_int32, C.c_int32, C.c_int32, C.c_int, vp, vp, vp, vp, vp, vp]
    K = 16
    g = torch.Generator().manual_seed(5)
    z = (2.0 * torch.randn((Bt, L, V), generator=g)).to(torch.bfloat16)
    if ties is not None:
        z.view(-1, V)[ties, ::620] = 20.0  # (61 in every quarter of the row)
    zc = z.cuda()
    ids = torch.full((Bt, L, K), -7, dtype=torch.int32, device="cuda")
    lp = torch.zeros((Bt, L, K), dtype=torch.float32, device="cuda")
    lse = torch.zeros((Bt, L), dtype=torch.float32, device="cuda")
    rs = torch.full((Bt, L), -7, dtype=torch.int32, device="cuda")
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = lib.graft_vocab_pass_static(Bt, L, V, K, 1, zc.data_ptr(), ids.data_ptr(), lp.data_ptr(), lse.data_ptr(),
                                     rs.data_ptr(), stream)
    assert rc == 0                      # the call only enqueues: host-side status
    torch.cuda.synchronize()            # the kernel came back by itself, and without a device error
    st = rs.cpu().numpy().reshape(-1)
    assert (st >= 0).all()              # every row's status word was written
    flagged = (st & ST_INTERNAL) != 0
    # the rows of thread block 0 and no others
    assert np.flatnonzero(flagged).tolist() == flagged_rows, "the wait that ran out was not reported as it should be"
    # rows that no block with a failed wait touched are correct
    o_ids, o_lp, o_lse, o_st = oracle.vocab_pass(z.reshape(Bt * L, V), K)
    ok = ~flagged
    assert np.array_equal(st[ok], o_st[ok])
    assert np.array_equal(ids.cpu().numpy().reshape(Bt * L, K)[ok], o_ids[ok])
    assert np.abs(lse.cpu().numpy().reshape(-1)[ok] - o_lse[ok]).max() <= 1e-5
    # the device and the shipped library are fine afterwards: an ordinary call gives the oracle's rows
    from paper_2608_20375_b200 import vocab_pass_static
    vocab_pass_static(zc, K, ids, lp, lse, rs)
    torch.cuda.synchronize()
    assert np.array_equal(rs.cpu().numpy().reshape(-1), o_st)
    assert np.array_equal(ids.cpu().numpy().reshape(Bt * L, K), o_ids)
    assert np.abs(lp.cpu().numpy().reshape(Bt * L, K) - o_lp).max() <= 1e-5
