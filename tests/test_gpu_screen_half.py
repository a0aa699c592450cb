"""Half-spectrum screen passes (256 .. 4096) against the oracle at the sizes and tolerances of the
device screens' own test, and the general passes for a screen that starts on 4 bytes only."""
import ctypes as C

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
    oracle.build()


def _close(got, ref):
    rms = np.sqrt(np.mean(ref ** 2))
    assert np.abs(got - ref).max() <= 1e-4 * rms
    assert np.sqrt(np.mean((got - ref) ** 2)) <= 1e-5 * rms


@pytest.mark.parametrize("n", [256, 512, 1024, 2048])
@pytest.mark.parametrize("seed", [3, (1 << 40) + 17])
def test_matches_oracle(n, seed):
    got = mcao.generate_screen(n, 0.05, 0.15, 25.0, seed).cpu().numpy()
    c = oracle.screen_coeffs(n, 0.05, 0.15, 25.0, seed)
    _close(got, np.real(np.fft.ifft2(c)) * n * n)


@pytest.mark.parametrize("n", [256, 1024])
def test_unaligned_screen_takes_the_general_passes(n):
    import torch
    buf = torch.zeros(n * n + 1, device="cuda")
    out = buf[1:]
    err = C.create_string_buffer(256)
    st = mcao.lib().mcao_generate_screen(n, 0.05, 0.15, 25.0, 9, C.c_void_p(out.data_ptr()), None, err, 256)
    assert st == 0, err.value
    torch.cuda.synchronize()
    ref = mcao.generate_screen(n, 0.05, 0.15, 25.0, 9).cpu().numpy()
    assert buf[0] == 0.0
    _close(out.cpu().numpy().reshape(n, n), ref.astype(np.float64))
