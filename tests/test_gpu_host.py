"""Rows in host memory, taken in by one call: pieces that stay on the device (default), chunks that do not, sizes around both,
and calls from several threads at a time. Rows, sketch and scores are those of the device path, so the results are too."""
import threading

import pytest
import torch

import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu


def _device(rows, D, ell, keep):
    fd = sage.SageFD(D, ell, rows.dtype, 0)
    g = rows.cuda()
    fd.update(g)
    fd.finalize()
    a = fd.score(g)
    idx = sage.sage_select(a, keep)
    out = a.cpu(), idx.cpu()
    fd.close()
    return out


def _rows(N, D, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    return ((torch.randn(N, 5, generator=g) + 0.3) @ torch.randn(5, D, generator=g) + 0.3 * torch.randn(N, D, generator=g)).to(dtype).pin_memory()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("N,D,ell,chunk", [(1, 9, 4, 0), (7, 130, 4, 0), (8, 131, 4, 3), (129, 264, 64, 0), (1001, 264, 64, 0), (1001, 264, 64, 1001), (1000, 264, 64, 999)])
def test_host_rows_equal_device_rows(dtype, N, D, ell, chunk):
    rows = _rows(N, D, dtype, N + D)
    a, idx = _device(rows, D, ell, 0.3)
    b, jdx = sage.sage_select_from_host(rows, D, ell, 0.3, chunk)
    # the same sketch bit for bit; a pass that scores in chunks adds the consensus in another order (fp64 sums of fp32 partials)
    assert torch.max(torch.abs(a - b)) <= 2e-6
    if chunk in (0, N):
        assert torch.equal(a, b) and torch.equal(idx, jdx)


def test_calls_from_several_threads():
    jobs = [_rows(900 + 50 * i, 260, torch.float32, i) for i in range(4)]
    want = [_device(r, 260, 32, 0.2) for r in jobs]
    got = [[] for _ in jobs]

    def work(i):
        for _ in range(3):
            got[i].append(sage.sage_select_from_host(jobs[i], 260, 32, 0.2))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, (a, idx) in enumerate(want):
        assert len(got[i]) == 3
        for b, jdx in got[i]:
            assert torch.equal(a, b) and torch.equal(idx, jdx)
