"""Calls whose faster route wants more device memory than their plain one, where the device has room for
the plain one alone: the same results as with room to spare."""
import contextlib
import ctypes as C

import numpy as np
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


@contextlib.contextmanager
def _only(wanted):
    """All of the device's free memory taken but `wanted` bytes, to 4 MB."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = []
    try:
        for _ in range(8):
            spare = torch.cuda.mem_get_info()[0] - wanted
            if spare >= 2 << 20:
                try:
                    hog.append(torch.empty(spare - spare % (2 << 20), dtype=torch.uint8, device="cuda"))
                except torch.OutOfMemoryError:
                    hog.append(torch.empty(spare // 2, dtype=torch.uint8, device="cuda"))
        left = torch.cuda.mem_get_info()[0]
        if abs(left - wanted) > 4 << 20:
            pytest.skip(f"device memory could not be taken: {left} bytes left")
        yield
    finally:
        hog.clear()
        torch.cuda.empty_cache()


def test_control_matrix_without_room_for_the_compressed_matrix():
    import torch
    n_slopes, n_cmd = 20000, 1024
    gen = torch.Generator(device="cuda").manual_seed(5)
    D = torch.randn((n_slopes, n_cmd), device="cuda", generator=gen)
    D *= torch.rand((n_slopes, n_cmd), device="cuda", generator=gen) < 0.3
    want, lam = mcao.tikhonov_reconstructor(D, 0.1, fp64=True)
    # the two square arrays take 17 MB, the nonzeros 123 MB more; the result is allocated before
    assert 20 * int((D != 0).sum()) > 100 << 20
    out = torch.empty((n_cmd, n_slopes), dtype=torch.float64, device="cuda")
    lam2, err = C.c_double(), C.create_string_buffer(256)
    with _only(50 << 20):
        st = mcao.lib().mcao_tikhonov_reconstructor(D.data_ptr(), n_slopes, n_cmd, D.stride(0), 0.1, out.data_ptr(), n_slopes, 1,
                                                    None, C.byref(lam2), err, 256)
    assert st == 0, err.value.decode()
    assert lam2.value == pytest.approx(lam, rel=1e-12)
    # sums of the same terms in another order: the tolerance of both routes against the oracle
    assert float((out - want).abs().max()) <= 1e-10 * float(want.abs().max())


def test_psf_image_without_room_for_a_second_one():
    def stepped():
        cfg = mcao_small()
        cfg["science"][0].update(n_px=512, pad=4)   # 2048 x 2048 doubles, 33 MB
        s = mcao.Sim(cfg)
        s.load_atmosphere(inputs.make_screens(cfg))
        s.load_dms()
        s.load_reconstructor(inputs.random_reconstructor(s.query(mcao.Q_COMMANDS), s.query(mcao.Q_SLOPES), 1e-3, 4))
        s.step(2)
        return s

    want = stepped().psf(0)
    s = stepped()
    s.sync()
    with _only(16 << 20):
        got = s.psf(0)
    assert np.array_equal(got[0], want[0]) and got[1:] == want[1:]
    assert np.array_equal(s.psf(0)[0], want[0])   # and with room again


def test_command_gradients_without_room_for_a_whole_group():
    import torch

    def loaded():
        cfg = inputs.mcao_20m()
        s = mcao.Sim(cfg)
        s.load_atmosphere(inputs.make_screens(cfg))
        s.load_dms()
        s.set_commands(np.random.default_rng(1).normal(0.0, 0.3, s.query(mcao.Q_COMMANDS)).astype(np.float32))
        return s

    a, b = loaded(), loaded()
    v = torch.randn((8, a.query(mcao.Q_SLOPES)), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    want = a.slopes_vjp(v)[0]
    out = torch.empty_like(want)
    with _only(12 << 20):   # the derivatives take 2 MB, eight vectors 13 MB more
        b._ck(mcao.lib().mcao_slopes_vjp(b.h, v.data_ptr(), 8, out.data_ptr(), None, None))
    assert torch.equal(out, want)   # no sum crosses vectors
