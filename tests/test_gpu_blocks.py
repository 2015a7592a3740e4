"""Shrink cycles in blocks (csrc/block_kernels.cu): streams that end at and beside the edges of a block, of a shrink and of the groups that
the kernels work in, the smallest and largest sketches and rows, and what changes the form of pass 1 in the middle of a block. Against the
oracle with the path's tolerances; however the rows are cut into calls, the sketch is the same to the bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_02470_b200 as sage

from helpers import compare, gpu_run
from test_gpu_parity import lowrank_rows

pytestmark = pytest.mark.gpu


def _block(ell):
    """Rows until the first block (one shrink) ends, and rows of each block after it."""
    return 2 * ell, max(4, 352 // (ell + 1)) * (ell + 1)


EDGES = [(2, 1, 0), (2, 63, 1), (3, 64, -1), (16, 65, 0), (21, 127, 17), (32, 300, 1), (64, 129, -1), (64, 2056, 65), (65, 520, 0), (80, 136, 3), (128, 264, -1),
         (129, 200, 0)]


@pytest.mark.parametrize("dtype,ell,D,extra", [(dt,) + e for dt in (torch.float32, torch.bfloat16) for e in EDGES] + [(torch.bfloat16, 256, 640, 1)])
def test_streams_that_end_at_the_edges_of_a_block(dtype, ell, D, extra):
    first, rest = _block(ell)
    N = first + rest + extra
    ld = D + (-D) % 8
    rows = lowrank_rows(N, D, min(5, D), 0.4, N + D + ell, dtype, ld)
    whole = gpu_run(rows, D, ell, 0.1)
    ref = oracle.run(rows, D, ell, 0.1, route=1)
    compare(whole, ref, rows, D, 0.1, label="block edge")
    assert whole["stats"]["shrinks"] == ref["stats"]["shrinks"] and whole["stats"]["device_flags"] == 0
    cuts = [first - 1, 1, ell, 1, 2 * ell, rest - 3 * ell - 1 + min(extra, 0)] + ([extra] if extra > 0 else [])
    parts = gpu_run(rows[:, :D].contiguous(), D, ell, 0.1, chunks=cuts)               # and packed: rows on odd boundaries
    assert np.array_equal(parts["S"], whole["S"]) and np.array_equal(parts["sigma"], whole["sigma"])


@pytest.mark.parametrize("dtype,ell,D", [(torch.float32, 16, 260), (torch.bfloat16, 64, 1032), (torch.bfloat16, 9, 515)])
@pytest.mark.parametrize("cut", [3, 1, 0])                                                # rows into the first block, the second's first cycle, its third
def test_form_of_pass_1_changed_in_the_middle(dtype, ell, D, cut):
    """Option 4 switched off (cycle by cycle on CUDA cores) and on again, and a checkpoint written in either form read by the other: each
    goes on from the rows that the other held."""
    first, rest = _block(ell)
    at = {3: ell + 3, 1: first + ell // 2, 0: first + 2 * (ell + 1) + 5}[cut]
    N = first + rest + 40
    rows = lowrank_rows(N, D, 5, 0.4, N + at, dtype)
    g = rows.cuda()
    ref = oracle.run(rows, D, ell, 0.1, route=1)

    def finish(fd):
        fd.finalize()
        S, sigma = fd.sketch()
        scores = fd.score(g)
        st = fd.stats()
        out = {"S": S.double().cpu().numpy(), "alpha": scores.double().cpu().numpy(), "idx": sage.sage_select(scores, 0.1).cpu().numpy()}
        fd.close()
        compare(out, ref, rows, D, 0.1)
        assert st["shrinks"] == ref["stats"]["shrinks"] and st["device_flags"] == 0 and np.isclose(st["sum_delta"], ref["stats"]["sum_delta"], rtol=1e-4)

    fd = sage.SageFD(D, ell, dtype, 0)
    fd.update(g[:at])
    fd.set_option(4, 0)
    blob = fd.export_state()                                                             # rows of the buffer
    fd.update(g[at:at + ell])
    fd.set_option(4, 1)
    fd.update(g[at + ell:])
    finish(fd)
    fd = sage.SageFD(D, ell, dtype, 0)
    fd.import_state(blob)
    fd.update(g[at:])
    in_block = sage.SageFD(D, ell, dtype, 0)
    in_block.update(g[:at])
    blob = in_block.export_state()
    in_block.close()
    finish(fd)
    fd = sage.SageFD(D, ell, dtype, 0)
    fd.set_option(4, 0)
    fd.import_state(blob)
    fd.update(g[at:])
    finish(fd)


def test_dense_and_structured_rows_in_one_block():
    """bfloat16 rows of both kinds: products take two planes a row, rows given before them are moved."""
    C, F, ell, N = 4, 40, 16, 300
    D = C * F + C
    r = torch.Generator().manual_seed(4)
    q, h = torch.randn(N, C, generator=r).bfloat16(), torch.randn(N, F, generator=r).bfloat16()
    outer = torch.cat([(q.float()[:, :, None] * h.float()[:, None, :]).reshape(N, -1), q.float()], 1)
    dense = lowrank_rows(N, D, 5, 0.4, 9, torch.bfloat16)
    A = torch.cat([dense[:50].float(), outer[50:120], dense[120:130].float(), outer[130:]])
    fd = sage.SageFD(D, ell, torch.bfloat16, 0)
    qd, hd, dd = q.cuda(), h.cuda(), dense.cuda()
    for _ in range(2):
        fd.reset()
        fd.update(dd[:50])
        fd.update_outer(qd[50:120], hd[50:120], C, F)
        fd.update(dd[120:130])
        fd.update_outer(qd[130:], hd[130:], C, F)
        fd.finalize()
        S, _ = fd.sketch()
        ref = oracle.run(A, D, ell, 0.1, route=1)
        from oracle import metrics
        assert metrics.signed_gram_norm(S.double().cpu().numpy(), ref["S"]) / float(A.double().norm()) ** 2 <= 1e-4
        assert fd.stats()["shrinks"] == ref["stats"]["shrinks"]
    fd.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_captured_updates_replay(dtype):
    """Rows of whole cycles, captured in the middle of a block and between two calls that go on with it: the graph finds the handle each
    time as it was when it was captured."""
    ell, D = 8, 104
    rows = lowrank_rows(2 * ell + 5 * (ell + 1) + 4 + 3 * 18 + 50, D, 4, 0.4, 8, dtype)
    g, at = rows.cuda(), 2 * ell + 5 * (ell + 1) + 4
    feed = torch.empty(18, D, dtype=dtype, device="cuda")
    fd = sage.SageFD(D, ell, dtype, 0)
    fd.update(g[:at])
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        fd.update(feed)
    for r in range(3):
        feed.copy_(g[at + 18 * r:at + 18 * (r + 1)])
        graph.replay()
    torch.cuda.synchronize()
    fd.update(g[at + 54:])
    fd.finalize()
    S, _ = fd.sketch()
    scores = fd.score(g)
    ref = oracle.run(rows, D, ell, 0.1, route=1)
    out = {"S": S.double().cpu().numpy(), "alpha": scores.double().cpu().numpy(), "idx": sage.sage_select(scores, 0.1).cpu().numpy()}
    compare(out, ref, rows, D, 0.1)
    fd.close()


def test_rows_without_a_finite_norm_are_flagged():
    """Finite values whose squares are not: an error at the freeze, and a sketch of finite values."""
    D, ell = 200, 8
    rows = lowrank_rows(420, D, 4, 0.3, 3)
    rows[37] = 3e37
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.update(rows.cuda())
    with pytest.raises(sage.SageError) as e:
        fd.finalize()
    assert e.value.status == 7 and bool(torch.isfinite(fd.sketch()[0]).all())
    fd.close()
