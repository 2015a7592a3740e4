"""The direct eigen-solve of a shrink (Householder tridiagonalisation, fp64 multisection, recurrences) at the sizes where its
tiles, clusters and padding change, on spectra that are hard for it: repeated eigenvalues, low rank, grading."""
import numpy as np
import pytest
import torch

import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu


def _rows(kind, N, D, seed):
    r = np.random.default_rng(seed)
    Q = np.linalg.qr(r.standard_normal((D, N)))[0].T
    if kind == "equal":                    # all eigenvalues of the Gram matrix equal
        A = Q
    elif kind == "steps":                  # two clusters: half the eigenvalues 1, half 1/4
        A = np.where(r.permutation(N) < N // 2, 0.5, 1.0)[:, None] * Q
    elif kind == "fifths":                 # five clusters, of which a shrink keeps two and a half, between rows at no right angles
        A = np.linalg.qr(r.standard_normal((N, N)))[0] @ (np.sqrt([1.0, 0.7, 0.5, 0.3, 0.25])[np.arange(N) % 5][:, None] * Q)
    elif kind == "pairs":                  # every row twice: half the eigenvalues zero, the others distinct
        A = np.repeat(r.standard_normal(((N + 1) // 2, D)), 2, axis=0)[:N]
    elif kind == "graded":                 # six orders of magnitude in the eigenvalues
        A = (10.0 ** (-3.0 * np.arange(N) / N))[:, None] * (np.linalg.qr(r.standard_normal((N, N)))[0] @ Q)
    else:
        A = r.standard_normal((N, D)) @ np.diag(np.exp(-np.arange(D) / D))
    return torch.from_numpy(np.ascontiguousarray(A, dtype=np.float32))


@pytest.mark.parametrize("kind", ["random", "equal", "steps", "fifths", "pairs", "graded"])
@pytest.mark.parametrize("ell", [2, 3, 5, 31, 32, 33, 63, 64, 65, 95, 127, 128, 129, 200, 255, 256])
def test_one_shrink_and_one_freeze(kind, ell):
    """2 ell rows shrink once; the first ell rows alone are frozen without a shrink. Bounds, relative to the largest
    eigenvalue: the fp32 Gram matrix of the CUDA-core kernels and the fp32 reduction are each accurate to a few 1e-7, 3e-6
    leaves a factor of about five; the tensor-core Gram matrix adds up to 96 truncations of 2^-24 between two drains of its
    accumulator (5.7e-6). Clusters of equal eigenvalues have the same bounds: their vectors are computed one by one, and two whose
    eigenvalues are as close as rounding leaves them live at different places of the tridiagonal matrix."""
    D = 600
    rows = _rows(kind, 2 * ell, D, 1000 + ell)
    for N, tensor_cores, bound in ((2 * ell, 0, 3e-6), (ell, 0, 3e-6), (2 * ell, 1, 9e-6), (ell, 1, 9e-6)):
        fd = sage.SageFD(D, ell, torch.float32, 0)
        fd.set_option(4, tensor_cores)
        fd.update(rows[:N].cuda())
        fd.finalize()
        S, sigma = fd.sketch()
        st = fd.stats()
        fd.close()
        A = rows[:N].double().numpy()
        lam, V = np.linalg.eigh(A.T @ A)
        delta = lam[-ell] if N == 2 * ell else 0.0
        kept = np.clip(lam - delta, 0.0, None)
        S, sigma = S.double().cpu().numpy(), sigma.double().cpu().numpy()
        expect = np.sort(kept)[::-1][:ell]
        err = np.linalg.norm(S.T @ S - (V * kept) @ V.T, 2) / lam[-1]
        err_sigma = np.max(np.abs(sigma ** 2 - expect)) / lam[-1]
        assert st["device_flags"] == 0 and st["shrinks"] == (1 if N == 2 * ell else 0)
        # each factorisation (a full buffer shrinks, what is left is frozen) takes two tensor-core kernels, or none, and the direct solve
        assert st["tensor_core_launches"] == tensor_cores * 2 * (2 if N == 2 * ell else 1) and st["last_sweeps"] == 0
        assert err <= bound and err_sigma <= bound, (N, tensor_cores, err, err_sigma)


@pytest.mark.parametrize("ell", [5, 8, 33, 64, 100, 128, 129, 200, 256])
def test_small_rows_beside_large_ones(ell):
    """ell rows of norms spread over three decades, in no order, frozen without a shrink: every row counts as much as in a sketch of
    rows of one size. Scaled to unit rows the Gram matrix is that of random rows of 4,000 values, whose condition number is below 3,
    so that an entry's rounding (fp32 sums folded every 2,048 terms: below 4e-7 of the product of the two norms) moves a singular
    value by 6e-7 of itself; twice that is allowed. Two rows of the sketch mix as far as the reflections round small against
    large: 1e-4 was met in this order of rows over all sizes, 1e-2 in another."""
    D = 4000
    r = np.random.default_rng(ell)
    rows = r.standard_normal((ell, D)) * (10.0 ** (-3.0 * r.permutation(ell) / ell) / D ** 0.5)[:, None]
    rows = torch.from_numpy(rows.astype(np.float32))
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.set_option(4, 0)
    fd.update(rows.cuda())
    fd.finalize()
    S, sigma = fd.sketch()
    st = fd.stats()
    fd.close()
    expect = np.linalg.svd(rows.double().numpy(), compute_uv=False)
    S, sigma = S.double().cpu().numpy(), sigma.double().cpu().numpy()
    norm = np.linalg.norm(S, axis=1)
    cosines = (S / norm[:, None]) @ (S / norm[:, None]).T - np.eye(ell)
    assert st["device_flags"] == 0 and st["last_rank"] == ell
    assert np.max(np.abs(sigma / expect - 1.0)) <= 1.2e-6
    assert np.max(np.abs(norm / expect - 1.0)) <= 1.2e-6 and np.max(np.abs(cosines)) <= 2e-4
