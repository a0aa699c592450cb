"""The Tikhonov control matrix on both of its routes (compressed D, dense D) at the edges of their
tiles, against the oracle (tolerance of the banded test: 1e-10 of the largest element; the random
matrices' condition is below 1e4, so LAPACK's own error stays under 1e-11)."""
import numpy as np
import pytest

import oracle
from paper_1608_00386_gb300 import build, mcao

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()


def _check(D, alpha):
    import torch
    ref, lam_ref = oracle.tikhonov_reconstructor(D, alpha)
    got, lam = mcao.tikhonov_reconstructor(torch.from_numpy(D).cuda(), alpha, fp64=True)
    assert lam == pytest.approx(lam_ref, rel=1e-12)
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-10 * np.max(np.abs(ref))
    r32, _ = mcao.tikhonov_reconstructor(torch.from_numpy(D).cuda(), alpha)
    assert torch.equal(r32, got.float())


@pytest.mark.parametrize("fill", [0.05, 0.3, 0.4, 1.0])   # the route changes at one third
@pytest.mark.parametrize("n_slopes,n_cmd", [(1, 1), (33, 31), (64, 32), (65, 63), (200, 64), (190, 65), (321, 129), (400, 193)])
def test_edges(n_slopes, n_cmd, fill):
    rng = np.random.default_rng(n_slopes * 1000 + n_cmd)
    D = rng.standard_normal((n_slopes, n_cmd)) * (rng.random((n_slopes, n_cmd)) < fill)
    D[0, 0] = 1.0
    _check(D.astype(np.float32), 0.05)


def test_empty_rows_and_columns_and_long_rows():
    rng = np.random.default_rng(7)
    D = np.zeros((700, 600), np.float32)
    D[5:650:3, 100:140] = rng.standard_normal((215, 40))
    D[17] = rng.standard_normal(600)          # more nonzeros than a block has threads
    D[:, 300] = rng.standard_normal(700)      # a full column
    _check(D, 0.3)


def test_not_positive_definite_is_refused():
    import torch
    with pytest.raises(mcao.McaoError) as e:
        mcao.tikhonov_reconstructor(torch.zeros((100, 70), device="cuda"), 1e-2)
    assert e.value.status == 7
