"""Reference slopes are in place when mcao_load_reconstructor returns: the caller's buffer may be written
over at once, and a step on the caller's stream, which nothing orders behind the library's own streams,
subtracts the values that were passed."""
import numpy as np
import pytest

from paper_1608_00386_gb300 import build, inputs, mcao

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()


@pytest.mark.parametrize("n_real", [1, 2])
@pytest.mark.parametrize("where", ["pinned", "device"])
def test_first_step_on_the_callers_stream_sees_them(where, n_real):
    import torch
    cfg = inputs.scao_tiny()
    screens = inputs.make_screens(cfg)
    R = torch.from_numpy(inputs.random_reconstructor(inputs.n_commands(cfg), 416, 0.01, 2))
    ref = torch.from_numpy(np.random.default_rng(3).normal(size=416).astype(np.float32))

    def first_slopes(s_ref, matrix, stream=None, spoil=False):
        s = mcao.Sim(cfg, n_real=n_real, stream=stream)
        for r in range(n_real):
            s.load_atmosphere(screens, realization=r)
        s.set_realization(0)
        s.load_dms()
        s.load_reconstructor(matrix, s_ref)
        if spoil:
            s_ref.fill_(1e3)
        s.step(1)
        return s.slopes()

    want = first_slopes(ref.numpy(), R.numpy())
    plain = first_slopes(None, R.numpy())
    assert np.abs(plain - want - ref.numpy()).max() <= 1e-5   # a float32 subtraction of values up to 4
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(stream):
            mine, matrix = (ref.clone().pin_memory(), R) if where == "pinned" else (ref.cuda(), R.cuda())
            assert np.array_equal(first_slopes(mine, matrix, stream, spoil=True), want)
