"""The rebuild of buffers of more than 256 rows: the smallest of them (one half of the output rows), output widths that end inside
and at a group of 16, the largest one, and row lengths from one column tile to several a block with a ragged last one."""
import numpy as np
import pytest
import torch

import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [128, 600, 18944, 18948, 40004])
@pytest.mark.parametrize("ell", [129, 130, 145, 161, 200, 256])
def test_rebuild_of_wide_sketches(ell, D):
    """2 ell rows shrink once, so that the frozen sketch is the rebuilt buffer: compared with the same factors applied in fp64.
    S = W B with W = diag(sqrt(1 - delta / lambda)) U^T, |W| <= 1 in the 2-norm. B is held as it is; the operands are split into
    parts of 11 bits whose dropped product is below 2^-22 of the whole, and a run's 60 additions truncate by 2^-24 each: with
    the runs' own roundings 66 * 2^-24 = 4e-6 of the largest |W| |B|, and 9e-6 with the Gram matrix behind W (the bound that
    the direct solve's tests derive for it)."""
    g = torch.Generator().manual_seed(ell * 1000 + D)
    n = 2 * ell
    low = torch.randn(n, 24, generator=g) @ torch.randn(24, D, generator=g) / 24 ** 0.5
    rows = low + 0.3 * torch.randn(n, D, generator=g)
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.update(rows.cuda())
    fd.finalize()
    S, _ = fd.sketch()
    st = fd.stats()
    fd.close()
    # a shrink and the freeze of what it left, each a Gram matrix and a rebuild on tensor cores
    assert st["device_flags"] == 0 and st["shrinks"] == 1 and st["tensor_core_launches"] == 4 and st["last_sweeps"] == 0
    S = S.double().cpu().numpy()
    A = rows.double().numpy()
    lam, U = np.linalg.eigh(A @ A.T)
    lam, U = lam[::-1], U[:, ::-1]
    kept = np.clip(lam - lam[ell - 1], 0.0, None)[:ell]
    # through the row space, so that the comparison stays ell-sized: S^T S = A^T U diag(kept / lam) U^T A
    P = (S @ A.T) @ U[:, :n]                                # rows of S against the left vectors: S A^T = W A A^T
    err = np.linalg.norm(P.T @ P - np.diag(np.concatenate([kept, np.zeros(n - ell)]) * lam), 2) / lam[0] ** 2
    norm = abs(np.linalg.norm(S) ** 2 - kept.sum()) / lam[0]
    assert err <= 9e-6 and norm <= 9e-6 * ell, (err, norm)
