"""Sensing launches shared by several sensors, product launches shared by several slices, and the
pair-wise Poisson search: bit-identical to a launch per sensor, and to the oracle's sampler from dark
to bright frames."""
import numpy as np
import pytest

import oracle
from paper_1608_00386_gb300 import build, inputs, mcao

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()
    oracle.build()


def _system(n_lgs, mixed):
    """20 m-like system cut to 16 x 16 subapertures: n_lgs laser stars, optionally one of another
    shape between them, and a low-order star."""
    cfg = inputs.mcao_20m(noise=True)
    cfg["D"] = 8.0
    lgs = [dict(cfg["wfs"][i % 3], n_sub=16, theta=(1e-4 * i, -5e-5 * i)) for i in range(n_lgs)]
    if mixed:
        lgs[n_lgs // 2] = dict(lgs[n_lgs // 2], n_fft=16, n_bin=2)
    cfg["wfs"] = lgs + [cfg["wfs"][3]]
    cfg["layers"] = [dict(l, n=256) for l in cfg["layers"][:2]]
    cfg["science"] = [dict(cfg["science"][0], n_px=128)]
    cfg["dms"] = [inputs.dm_spec(cfg, 0.0, 0.5, 0.3)]
    return cfg


def _control(cfg, screens):
    o = oracle.Sim(cfg, screens)
    n = o.n_slopes
    o.close()
    return inputs.random_reconstructor(inputs.n_commands(cfg), n, 1e-3, 3)


@pytest.mark.parametrize("dtype", [mcao.DTYPE_F32, mcao.DTYPE_BF16, mcao.DTYPE_FP8_E4M3])
@pytest.mark.parametrize("n_lgs,mixed", [(3, False), (4, True), (7, False)])
def test_shared_launches_are_bit_identical(n_lgs, mixed, dtype):
    cfg = _system(n_lgs, mixed)
    screens = inputs.make_screens(cfg)
    R = _control(cfg, screens)
    out = []
    for blocks in (1, 2, 8):   # warps at once: every sensor fits one launch, or few of them do
        s = mcao.make_sim(cfg, screens, R, r_dtype=dtype)
        s.set_tuning(sense_blocks_per_sm=blocks)
        s.step(4)
        out.append((s.slopes(), s.commands(), np.array(s.psf(0, with_image=False)[1:])))
        s.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("photons", [0.0, 0.3, 40.0, 2000.0, 3e5])
@pytest.mark.parametrize("read_noise", [0.0, 3.0])
def test_counts_match_the_sampler(photons, read_noise):
    cfg = _system(2, True)
    cfg["wfs"] = [dict(w, n_photons=photons, read_noise=read_noise) for w in cfg["wfs"]]
    screens = inputs.make_screens(cfg)
    R = _control(cfg, screens)
    g = mcao.make_sim(cfg, screens, R, keep_frames=True)
    g.step(2)
    for w, p in enumerate(cfg["wfs"]):
        lam, fr = g.frames(w)
        ref = oracle.noise_frame(lam.ravel(), read_noise, 0, 1, w, cfg["seed"], frame_px=(p["n_fft"] // p["n_bin"]) ** 2)
        assert np.array_equal(fr.ravel(), ref)
