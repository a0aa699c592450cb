"""The autotuner and the science's start: with one sensing launch the knob has no effect, so it is not tried
and stays as it was; with several both values are."""
import re

import pytest

from paper_1608_00386_gb300 import build, inputs, mcao

from _helpers import mcao_small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()


@pytest.mark.parametrize("launches", [1, 2])
@pytest.mark.parametrize("set_to", [0, 1])
def test_tried_where_it_has_an_effect(launches, set_to):
    cfg = mcao_small()
    if launches == 2:   # laser stars of two detector shapes
        cfg["wfs"].insert(1, dict(cfg["wfs"][0], n_fft=32))
    g = mcao.Sim(cfg)
    g.load_atmosphere(inputs.make_screens(cfg))
    g.load_dms()
    g.load_reconstructor(inputs.random_reconstructor(g.query(mcao.Q_COMMANDS), g.query(mcao.Q_SLOPES), 1e-3, 4))
    g.set_tuning(science_after_aux=set_to)
    chosen, report = g.autotune(steps_per_trial=5)
    tried = re.findall(r"(\d)=", re.search(r"science_after_aux:(.*?) ->", report).group(1))
    assert tried == ([str(set_to)] if launches == 1 else ["0", "1"])
    assert launches == 2 or chosen["science_after_aux"] == set_to
