"""Noise-free slopes and their derivatives straight from the field's lags (k_lag.cu): every sensor
shape with and without elongation against the oracle and against the image route, a dark frame, the
matrix's padding columns, and the products at the edges of the vector groups with a rotated DM."""
import numpy as np
import pytest

import oracle
from paper_1608_00386_gb300 import build, inputs, mcao

from _helpers import mcao_small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()
    oracle.build()


def _one_sensor(n_sub, n_px, n_fft, n_bin, na_fwhm, photons=1000.0):
    cfg = mcao_small()
    kind = "lgs" if na_fwhm else "ngs"
    cfg["wfs"] = [inputs._wfs(kind, (10 * inputs.ARCSEC, 0.0), n_sub, n_px, n_fft, n_bin, 589e-9, photons,
                              height=90e3 if na_fwhm else 0.0, na_fwhm=na_fwhm, launch=(4.2, -1.0) if na_fwhm else (0.0, 0.0),
                              valid_thr=0.3)]
    cfg["dms"] = [inputs.dm_spec(cfg, 0.0, 1.0, 0.3), inputs.dm_spec(cfg, 5000.0, 1.4, 0.3)]
    return cfg


def _loaded(cfg, screens, **kw):
    s = mcao.Sim(cfg, **kw)
    s.load_atmosphere(screens)
    s.load_dms()
    return s


@pytest.mark.parametrize("shape", [(7, 8, 16, 2), (9, 8, 16, 1), (5, 8, 32, 2), (5, 16, 32, 2), (3, 32, 64, 4)])
@pytest.mark.parametrize("na_fwhm", [0.0, 10e3])
def test_slopes_match_oracle_and_image_route(shape, na_fwhm):
    cfg = _one_sensor(*shape, na_fwhm)
    screens = inputs.make_screens(cfg)
    c = (np.random.default_rng(2).standard_normal(inputs.n_commands(cfg)) * 0.3).astype(np.float32)
    o = oracle.Sim(cfg, screens)
    o.set_commands(c.astype(np.float64))
    ref = o.measure()
    for keep in (False, True):   # lags, image
        g = _loaded(cfg, screens, keep_frames=keep)
        g.set_commands(c)
        assert np.abs(g.measure() - ref).max() <= 2e-5   # px: the loop's bar for every slope


def test_dark_frame_has_no_slopes():
    cfg = _one_sensor(5, 8, 32, 2, 10e3, photons=0.0)
    screens = inputs.make_screens(cfg)
    assert not np.any(_loaded(cfg, screens).measure())


def test_matrix_padding_and_product_groups():
    import torch
    cfg = mcao_small()
    g = _loaded(cfg, inputs.make_screens(cfg))
    g.set_misregistration(1, 0.1, -0.05, 0.02, 1.01)   # one separable and one rotated DM
    nc, ns = g.query(mcao.Q_COMMANDS), g.query(mcao.Q_SLOPES)
    D = g.interaction_matrix()
    P = torch.full((ns, nc + 3), float("nan"), device="cuda")
    g._ck(mcao.lib().mcao_interaction_matrix(g.h, P.data_ptr(), nc + 3))
    assert torch.equal(P[:, :nc], D) and not P[:, nc:].any()
    v = torch.randn((17, ns), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    full, phase = g.slopes_vjp(v, phase=True)
    want = v.double() @ D.double()
    # float32 sums of at most ns * 9 * 9 terms per command, and the weights below 1e-10 each side leaves out
    assert float((full.double() - want).norm() / want.norm()) <= 1e-5
    for n in (1, 8, 9):
        part, _ = g.slopes_vjp(v[:n])
        assert float((part.double() - want[:n]).norm() / want[:n].norm()) <= 1e-5
    # a phase gradient is what the same vector's command gradient is made of: alone and together
    alone = g.slopes_vjp(v[16], commands=False, phase=True)[1]
    assert torch.equal(alone, phase[16])
