"""The merged form once its cycles are replayed as graphs: many cycles per sketch, rows in calls that cut blocks and cycles at
every place, options changed in between, against the same rows with direct launches (per-kernel timing switches the replay off):
the same kernels on the same data, so the sketches agree bit for bit."""
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
