"""The merged form once its cycles are replayed as graphs: many cycles per sketch, rows in calls that cut blocks and cycles at
every place, options changed in between, against the same rows with direct launches (per-kernel timing switches the replay off):
the same kernels on the same data, so the sketches agree bit for bit."""
import threading

import pytest
import torch

import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu


def _sketch(rows, D, ell, P, block, cuts, timed, repeat=1, change=None):
    fd = sage.SageFD(D, ell, rows.dtype, 0)
    fd.set_option(6, P)
    if block:
        fd.set_option(7, block)
    for again in range(repeat):
        if again:
            fd.reset()
        if timed:
            fd.set_option(3, 1)
        r0 = 0
        for i, c in enumerate(cuts):
            if change and i == len(cuts) // 2:
                fd.set_option(*change)
            fd.update(rows[r0:r0 + c])
            r0 += c
        fd.finalize()
    S, sigma = fd.sketch()
    st = fd.stats()
    fd.close()
    assert st["device_flags"] == 0
    return S, sigma, st


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("D,ell,P,block,cuts", [(130, 8, 2, None, [700]), (130, 8, 3, 5, [333, 1, 2, 364]), (100, 5, 4, 40, [97] * 10),
                                                (260, 33, 2, None, [2300]), (64, 4, 16, None, [50] * 30)])
def test_replayed_cycles_equal_direct_launches(dtype, D, ell, P, block, cuts):
    g = torch.Generator().manual_seed(D + ell)
    rows = torch.randn(sum(cuts), D, generator=g).to(dtype).cuda()
    S0, sg0, st0 = _sketch(rows, D, ell, P, block, cuts, True)
    S1, sg1, st1 = _sketch(rows, D, ell, P, block, cuts, False, repeat=2)
    S2, sg2, _ = _sketch(rows, D, ell, P, block, cuts, False, change=(9, 1))
    assert torch.equal(S0, S1) and torch.equal(sg0, sg1) and torch.equal(S0, S2) and torch.equal(sg0, sg2)
    assert st0["shrinks"] == st1["shrinks"] and st0["kernel_launches"] == st1["kernel_launches"]


def test_other_threads_may_synchronise_meanwhile():
    """New handles whose cycles become graphs in the middle of a pass, while another thread synchronises the device all the time."""
    g = torch.Generator().manual_seed(5)
    rows = torch.randn(3000, 100, generator=g).cuda()
    want = _sketch(rows, 100, 8, 8, None, [3000], True)[0]
    other = sage.SageFD(64, 4, torch.float32, 0)
    stop, errors, turns = threading.Event(), [], [0]

    def synchronise():
        while not stop.is_set():
            try:
                torch.cuda.synchronize()
                other.stats()
            except Exception as e:                                  # noqa: BLE001
                errors.append(e)
            turns[0] += 1

    t = threading.Thread(target=synchronise)
    t.start()
    try:
        for _ in range(6):
            assert torch.equal(_sketch(rows, 100, 8, 8, None, [3000], False)[0], want)
    finally:
        stop.set()
        t.join()
    other.close()
    assert not errors and turns[0] > 0


def test_captured_updates_of_a_sketch_with_graphs():
    """Rows that bring every sketch back to where it stood (a cycle per buffer copy each): captured once the cycles are graphs, the
    updates replay like any others."""
    g = torch.Generator().manual_seed(6)
    ell, P, D = 8, 2, 100
    warm, again = torch.randn(P * (2 * ell + 30 * (ell + 1)), D, generator=g).cuda(), torch.randn(2 * P * (ell + 1), D, generator=g).cuda()

    def fill(fd):
        fd.set_option(6, P)
        fd.update(warm[:P * 2 * ell])
        fd.update(warm[P * 2 * ell:])

    want = sage.SageFD(D, ell, torch.float32, 0)
    fill(want)
    for _ in range(3):
        want.update(again)
    want.finalize()
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fill(fd)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        fd.update(again)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    fd.finalize()
    assert torch.equal(fd.sketch()[0], want.sketch()[0])
    fd.close()
    want.close()
