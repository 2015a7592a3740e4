"""Selections at the sizes where the sort behind them changes: whole slots and blocks of the one-launch form, its largest size
and one more, one and two passes over the class. Integer work: exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from oracle import cb
import paper_2510_02470_b200 as sage

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("N", [1, 33, 8191, 8192, 8193, 57344 + 5, 131071, 131072, 131073, 262144, 262145, 1050001])
def test_selection_at_the_edges(N):
    r = np.random.default_rng(N)
    a = np.where(r.uniform(size=N) < 0.3, r.integers(-6, 7, N) / 6.0, r.uniform(-1, 1, N)).astype(np.float32)   # ties at many places
    s = torch.from_numpy(a).to(DEV)
    for rate in (1.0 / N, min(8192, N) / N, min(8193, N) / N, 0.37, 0.5, 0.51, 1.0):
        assert np.array_equal(sage.sage_select(s, rate).cpu().numpy(), oracle.select(a.astype(np.float64), rate)), rate


@pytest.mark.parametrize("N,C", [(8193, 255), (8192, 256), (131072, 255), (131073, 10), (140000, 300), (3000, 65535), (1, 256), (98304, 300), (98305, 300)])
def test_selection_by_class_at_the_edges(N, C):
    r = np.random.default_rng(N + C)
    a = (r.integers(-50, 51, size=N) / 50.0).astype(np.float32)
    labels = r.integers(-1, C + 1, size=N).astype(np.int32)
    labels[: N // 3] = C // 2                                        # one large class
    idx, kc = sage.sage_select_classes(torch.from_numpy(a).to(DEV), torch.from_numpy(labels).to(DEV), C, 0.23)
    idx_ref, kc_ref = cb.select(a.astype(np.float64), labels, C, 0.23)
    assert kc == kc_ref.tolist() and np.array_equal(idx.cpu().numpy(), idx_ref)


@pytest.mark.parametrize("n,rate", [(11, 0.04545454545454545), (25, 0.019999999999999997), (35, 0.014285714285714284), (44, 0.011363636363636362)])
def test_quota_of_the_classes_is_the_count_of_a_selection(n, rate):
    """floor(rate n + 0.5) with the product rounded first: a fused multiply-add gives one less here."""
    a = np.linspace(-1.0, 1.0, n).astype(np.float32)
    labels = np.zeros(n, dtype=np.int32)
    idx, kc = sage.sage_select_classes(torch.from_numpy(a).to(DEV), torch.from_numpy(labels).to(DEV), 3, rate)
    assert sage.sage_select_count(n, rate) == 1 and kc == [1, 0, 0] and idx.cpu().tolist() == [n - 1]


@pytest.mark.parametrize("N,C,ell", [(1, 1, 4), (9000, 255, 33), (9000, 256, 16), (132000, 12, 8), (2000, 20000, 5)])
def test_class_centroids_at_the_edges(N, C, ell):
    """The centroid is a sum in fp64 of the library's own fp32 projections, rounded once: 2^-24, and 1e-6 for the fp32 dot
    product of a score."""
    D = 20
    r = np.random.default_rng(N + C)
    labels = r.integers(-1, C + 1, size=N).astype(np.int32)
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.load_sketch(torch.from_numpy(r.standard_normal((ell, D)).astype(np.float32)).to(DEV))
    fd.score(torch.from_numpy((r.standard_normal((N, D)) + 0.3).astype(np.float32)).to(DEV))
    zhat = fd.intermediates(N)[0].double().cpu().numpy()
    a = fd.score_classes(torch.from_numpy(labels).to(DEV), C)
    U, cnt = fd.class_centroids()
    fd.close()
    a_ref, U_ref, cnt_ref = cb.class_scores(zhat, labels, C)
    assert np.array_equal(cnt.cpu().numpy(), cnt_ref)
    assert np.max(np.abs(U.double().cpu().numpy() - U_ref)) <= 6.1e-8
    assert np.max(np.abs(a.double().cpu().numpy() - a_ref)) <= 1e-6


@pytest.mark.parametrize("N,C,ell", [(2, 1, 4), (100, 1000, 64), (255, 3, 32), (256, 2, 33), (257, 300, 65), (511, 7, 256), (512, 1, 64), (512, 1, 65), (512, 700, 130), (2048, 40, 64), (2049, 40, 64), (2048, 9765, 8), (2048, 9766, 8)])
def test_class_centroids_of_few_rows(N, C, ell):
    """Around the size from which rows are grouped by class first; bounds as above. The launch counter follows the path."""
    D = 20
    r = np.random.default_rng(N * 7 + C)
    labels = r.integers(-1, C + 1, size=N).astype(np.int32)
    labels[N // 2:] = C - 1                                          # one large class
    fd = sage.SageFD(D, ell, torch.float32, 0)
    fd.load_sketch(torch.from_numpy(r.standard_normal((ell, D)).astype(np.float32)).to(DEV))
    fd.score(torch.from_numpy((r.standard_normal((N, D)) + 0.3).astype(np.float32)).to(DEV))
    zhat = fd.intermediates(N)[0].double().cpu().numpy()
    n0 = fd.stats()["kernel_launches"]
    a = fd.score_classes(torch.from_numpy(labels).to(DEV), C)
    launches = fd.stats()["kernel_launches"] - n0
    U, cnt = fd.class_centroids()
    fd.close()
    a_ref, U_ref, cnt_ref = cb.class_scores(zhat, labels, C)
    assert np.array_equal(cnt.cpu().numpy(), cnt_ref)
    assert np.max(np.abs(U.double().cpu().numpy() - U_ref)) <= 6.1e-8
    assert np.max(np.abs(a.double().cpu().numpy() - a_ref)) <= 1e-6
    few = N <= 2048 and N * max(32, 1 << (ell - 1).bit_length()) <= 32768 * C and N * C <= 20000000
    assert launches == (2 if few else (3 if C > 255 else 1) + (3 if C <= 8192 else 2))
