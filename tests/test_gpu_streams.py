"""Steps and readouts on the caller's stream, and readouts straight into page-locked buffers: the same
values as the getters whatever streams, buffers and calls are mixed."""
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


def _sim(stream=None):
    cfg = inputs.scao_tiny(noise=True)
    return mcao.make_sim(cfg, inputs.make_screens(cfg), inputs.random_reconstructor(inputs.n_commands(cfg), 416, 0.01, 2),
                         stream=stream)


def _history(n):
    s = _sim()
    out = []
    for _ in range(n):
        s.step(1)
        out.append((s.commands(), np.array(s.psf(0, with_image=False)[1:])))
    return out


def test_streams_and_buffers_may_change_between_calls():
    import torch
    steps = 24
    ref = _history(steps)
    streams = [None, torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]
    s = _sim()
    nc = s.query(mcao.Q_COMMANDS)
    pinned = [torch.zeros(nc).pin_memory() for _ in range(steps)]
    sr = [torch.zeros((1, 2), dtype=torch.float64).pin_memory() for _ in range(steps)]
    pageable = np.zeros((steps, nc), np.float32)
    odd = torch.zeros(4 * nc + 2, dtype=torch.uint8).pin_memory().numpy()[2:]   # not aligned to a float
    for k in range(steps):
        if streams[k % 4] is not None:
            s.set_stream(streams[k % 4])
        s.step(1)
        if k % 3 == 0:
            s.read_async(pageable[k], sr[k])       # ring, then direct readouts behind it
            s.read_async(pinned[k])
        elif k % 3 == 1:
            s.read_async(pinned[k], sr[k])
        else:
            s.read_async(np.frombuffer(odd, np.float32, nc))
            s.read_async(pinned[k], sr[k])
        if k % 5 == 4:
            assert np.array_equal(s.commands(), ref[k][0])
    s.sync()
    for k in range(steps):
        assert np.array_equal(pinned[k].numpy(), ref[k][0])
        assert np.array_equal(sr[k].numpy()[0], ref[k][1])
        if k % 3 == 0:
            assert np.array_equal(pageable[k], ref[k][0])
    assert np.array_equal(np.frombuffer(odd, np.float32, nc), ref[23][0])


def test_one_buffer_holds_the_latest_readout():
    import torch
    ref = _history(12)
    s = _sim(torch.cuda.Stream())
    c = torch.zeros(s.query(mcao.Q_COMMANDS)).pin_memory()
    sr = np.zeros((1, 2))                                  # pageable: this call goes through the ring
    for k in range(12):
        s.step(1)
        if k % 2:
            s.read_async(c)
        else:
            s.read_async(c, sr)
    s.sync()
    assert np.array_equal(c.numpy(), ref[11][0])


def test_callers_stream_sees_the_readout():
    import torch
    ref = _history(3)
    st = torch.cuda.Stream()
    s = _sim(st)
    c = torch.zeros(s.query(mcao.Q_COMMANDS)).pin_memory()
    with torch.cuda.stream(st):
        s.step(3)
        s.read_async(c)
        d = c.to("cuda", non_blocking=True)               # queued behind the readout on the same stream
    st.synchronize()
    assert np.array_equal(d.cpu().numpy(), ref[2][0])


@pytest.mark.parametrize("n_px,pad", [(8, 3), (40, 2), (72, 1), (128, 2)])
def test_psf_image_order(n_px, pad):
    """The image is the accumulator shifted by half its side (odd sides too) and transposed."""
    cfg = inputs.scao_tiny()
    cfg["science"] = [dict(cfg["science"][0], n_px=n_px, pad=pad)]
    screens = inputs.make_screens(cfg)
    s = mcao.make_sim(cfg, screens, inputs.random_reconstructor(inputs.n_commands(cfg), 416, 0.01, 2))
    s.step(2)
    M = n_px * pad
    acc = np.frombuffer(s.get_state()[-8 * M * M:], np.float64).reshape(M, M)
    img = s.psf(0)[0]
    x = (np.arange(n_px) - (n_px - 1) / 2) * 8.0 / n_px
    A = (x[:, None] ** 2 + x ** 2 <= 16.0).sum()
    j = (np.arange(M) + M // 2) % M
    assert np.array_equal(img, acc.T[np.ix_(j, j)] * (1.0 / (2.0 * float(A) * float(A))))
