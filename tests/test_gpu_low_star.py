"""A laser star set below a DM's altitude: its beam crosses its own axis under that DM and samples it in
descending order.  Slopes on both noise-free routes, the interaction matrix and the command products
against the oracle, with the tolerances of the tests of stars above every DM."""
import numpy as np
import pytest

import oracle
from paper_1608_00386_gb300 import build, inputs, mcao

from _helpers import mcao_small, wide_lgs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()
    oracle.build()


# DM at 5 km: the beam there is -0.25, -1 and -1.5 times the pupil (samples -0.25, -1 and -1.5 surface samples apart)
@pytest.mark.parametrize("height", [4000.0, 2500.0, 2000.0])
@pytest.mark.parametrize("npx", [8, 16])
def test_star_below_a_dm_matches_oracle(height, npx):
    import torch
    cfg = mcao_small()
    if npx == 16:
        cfg["wfs"][0] = dict(wide_lgs()["wfs"][0], theta=cfg["wfs"][0]["theta"])
    cfg["wfs"][0]["na_fwhm"] = 0.0
    cfg["layers"][1]["alt"] = 1000.0
    for lay in cfg["layers"]:
        lay["pixel"] = 0.125   # pupil samples at most one grid sample apart on every grid
    cfg["dms"][1] = inputs.dm_spec(cfg, 5000.0, 1.1, 0.3)
    screens = inputs.make_screens(cfg)
    o = oracle.Sim(dict(cfg, wfs=[dict(cfg["wfs"][0], height=height), cfg["wfs"][1]]), screens)
    c = np.random.default_rng(6).normal(0.0, 0.3, o.n_cmd).astype(np.float32)
    o.set_commands(c.astype(np.float64))
    ref = o.measure()
    for keep in (False, True):   # lags, image
        g = mcao.Sim(cfg, keep_frames=keep)
        g.load_atmosphere(screens)
        g.load_dms()
        g.set_sodium(0, height, 0.0)
        g.set_commands(c)
        assert np.abs(g.measure() - ref).max() <= 2e-5
        phase = o.wfs_phase(0)
        assert np.abs(g.wfs_phase(0) - phase).max() <= 2e-5 * np.abs(phase).max()
    D = g.interaction_matrix()
    Do = oracle.jacobian_fd(o, 1e-3)
    assert np.linalg.norm(D.cpu().numpy() - Do) <= 1e-5 * np.linalg.norm(Do)
    v = torch.from_numpy(np.random.default_rng(7).normal(size=(2, o.n_slopes)).astype(np.float32)).cuda()
    want = v.double() @ D.double()
    assert float((g.slopes_vjp(v)[0].double() - want).norm() / want.norm()) <= 1e-5
