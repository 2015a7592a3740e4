"""The projection of fp32 rows onto sketches of at most 64 rows: row counts at the edges of the 128-row halves and of the 256-row tiles
of a pair of SMs, K lengths from one K tile on with ragged ends, and sizes at which row tiles are whole, cut once and cut many times."""
import numpy as np
import pytest
import torch

import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ell", [2, 31, 33, 64])
@pytest.mark.parametrize("N,D", [(1, 20), (127, 32), (129, 100), (255, 2052), (257, 5132), (700, 20000), (18944, 64), (19000, 260), (40000, 1028)])
def test_scores_of_fp32_rows(N, D, ell):
    """Scores of all rows against a loaded sketch of unit rows, compared with fp64. Every product of the split operands is taken, and an
    accumulator takes 24 additions truncated by 2^-24 between drains, so that a component of z_i = S g_i is off by at most
    24 * 2^-24 |g_i| = 1.5e-6 |g_i| and a direction z_i / |z_i| by b_i = 1.5e-6 sqrt(ell) |g_i| / |z_i|. A score is that
    direction times the normalised sum of all of them: off by b_i + sum(b) / |sum|. The rows share a part c S with |c| = 1, so that
    neither |z_i| nor the sum is small."""
    g = torch.Generator().manual_seed(N + 7 * D + ell)
    used = min(ell, D)
    S = torch.zeros(ell, D)
    S[:used] = torch.linalg.qr(torch.randn(D, used, generator=g, dtype=torch.float64))[0].T.float()
    c = torch.randn(used, generator=g)
    rows = torch.zeros(N, (D + 3) // 4 * 4)
    rows[:, :D] = torch.randn(N, D, generator=g) / D ** 0.5 + (c / c.norm()) @ S[:used]
    dev = rows.cuda()
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.load_sketch(S.cuda())
    a = fd.score(dev[:, :D]).double().cpu().numpy()
    st = fd.stats()
    fd.close()
    G = rows[:, :D].double().numpy()
    Z = G @ S.double().numpy().T
    zn = np.linalg.norm(Z, axis=1)
    total = (Z / zn[:, None]).sum(axis=0)
    b = 1.5e-6 * used ** 0.5 * np.linalg.norm(G, axis=1) / zn
    err = np.abs(a - Z @ total / zn / np.linalg.norm(total))
    assert st["device_flags"] == 0 and st["tensor_core_launches"] == 1           # one projection, all rows in one launch
    assert np.all(err <= b + b.sum() / np.linalg.norm(total) + 2e-7), np.max(err / b)
