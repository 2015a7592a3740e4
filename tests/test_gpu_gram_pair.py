"""The Gram matrix of buffers of more than 128 rows, computed by pairs of SMs: row counts at the edges of the 128-row halves and the
256-row tiles, and row lengths of one K tile, of ragged last tiles, of fewer tiles than slices and of several runs a slice."""
import numpy as np
import pytest
import torch

import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [20, 32, 100, 2052, 5130, 40004])
@pytest.mark.parametrize("n", [129, 130, 131, 200, 255, 256, 257, 258, 383, 384, 400, 511, 512])
def test_spectrum_of_wide_buffers(n, D):
    """n rows frozen: without a shrink up to 256 rows (ell = n), with one to ell = 256 beyond. The singular values are those of the
    Gram matrix, and the sketch's rows are orthogonal with these norms. Bound, relative to the largest eigenvalue: at most 96
    additions between two drains of an accumulator, each truncated by 2^-24 (5.7e-6), dropped products below 2^-22, and the fp32
    eigen-solve: 9e-6 as in the direct solve's tests, twice that for the sketch, whose rebuild truncates as often."""
    g = torch.Generator().manual_seed(n * 100003 + D)
    decay = torch.exp(-torch.arange(n) / (0.3 * n))[torch.randperm(n, generator=g)][:, None]
    rows = torch.randn(n, D, generator=g) * decay
    ell = min(n, 256)
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.update(rows.cuda())
    fd.finalize()
    S, sigma = fd.sketch()
    st = fd.stats()
    fd.close()
    # a factorisation takes its Gram matrix and its rebuild on tensor cores, the direct solve between them; 512 rows shrink, then freeze
    assert st["device_flags"] == 0 and st["shrinks"] == (1 if n > 256 else 0)
    assert st["tensor_core_launches"] == (4 if n == 512 else 2) and st["last_sweeps"] == 0
    lam = np.zeros(n)
    sv = np.linalg.svd(rows.double().numpy(), compute_uv=False) ** 2
    lam[:len(sv)] = sv
    expect = np.clip(lam[:ell] - (lam[ell - 1] if n > 256 else 0.0), 0.0, None)
    S, sigma = S.double().cpu().numpy(), sigma.double().cpu().numpy()
    assert np.max(np.abs(sigma ** 2 - expect)) <= 9e-6 * lam[0]
    assert np.linalg.norm(S @ S.T - np.diag(sigma ** 2), 2) <= 18e-6 * lam[0]


@pytest.mark.parametrize("n", [200, 512])
def test_the_same_rows_give_the_same_bits(n):
    """Two CTAs hand operands and accumulators to one another many times per launch; every order of events has one result."""
    g = torch.Generator().manual_seed(n)
    rows = torch.randn(n, 40004, generator=g).cuda()
    first = None
    for _ in range(12):
        fd = sage.SageFD(40004, min(n, 256), torch.float32, 0)
        fd.update(rows)
        fd.finalize()
        S, sigma = fd.sketch()
        assert fd.stats()["device_flags"] == 0
        fd.close()
        if first is None:
            first = S, sigma
        assert torch.equal(S, first[0]) and torch.equal(sigma, first[1])
