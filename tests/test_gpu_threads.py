"""Objects of different sizes side by side, from one host thread and from several: each launch is admitted
whatever sizes the others launch, and the results are those of the object by itself."""
import threading

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


def _together(calls, times):
    """Runs every call `times` times, a thread each; the first error of any is raised."""
    errors, start = [], threading.Barrier(len(calls))

    def work(call):
        try:
            start.wait()
            for _ in range(times):
                call()
        except Exception as e:   # handed to the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_control_matrices_of_different_sizes():
    import torch

    def call(n_slopes, n_cmd, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        D = torch.randn((n_slopes, n_cmd), device="cuda", generator=gen)
        D *= torch.rand((n_slopes, n_cmd), device="cuda", generator=gen) < 0.1
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        want, _ = mcao.tikhonov_reconstructor(D, 0.1, stream=stream)

        def run():
            got, _ = mcao.tikhonov_reconstructor(D, 0.1, stream=stream)
            assert torch.equal(got, want)
        return run

    _together([call(900, 400, 1), call(60, 20, 2), call(300, 100, 3)], 200)


def test_interaction_matrices_of_different_systems():
    import torch

    def call(n_dms, npx):
        cfg = mcao_small()
        cfg["dms"] = cfg["dms"][:n_dms]
        if npx == 8:
            cfg["wfs"] = cfg["wfs"][:1]
        g = mcao.Sim(cfg)
        g.load_atmosphere(inputs.make_screens(cfg))
        g.load_dms()
        g.set_commands(np.random.default_rng(n_dms).normal(0.0, 0.3, g.query(mcao.Q_COMMANDS)).astype(np.float32))
        want = g.interaction_matrix()

        def run():
            assert torch.equal(g.interaction_matrix(), want)
        return run

    _together([call(2, 32), call(1, 8), call(2, 8)], 200)


@pytest.mark.parametrize("what", ["science", "batch", "screen"])
def test_a_smaller_object_made_later(what):
    import torch

    def sim(big):
        cfg = mcao_small()
        n_real = 1
        if what == "science":   # 960 and 80 points: sizes without a transform of their own
            cfg["science"][0].update({"n_px": 120, "pad": 8} if big else {"n_px": 40, "pad": 2})
        else:
            n_real = 33 if big else 2
        s = mcao.Sim(cfg, n_real=n_real)
        screens = inputs.make_screens(cfg)
        for r in range(n_real):
            s.load_atmosphere(screens, realization=r)
        s.set_realization(0)
        s.load_dms()
        R = inputs.random_reconstructor(s.query(mcao.Q_COMMANDS), s.query(mcao.Q_SLOPES), 1e-3, 4)
        s.load_reconstructor(R, dtype=mcao.DTYPE_BF16 if what == "batch" else mcao.DTYPE_F32)
        return s

    if what == "screen":
        want = mcao.generate_screen(3000, 0.06, 0.15, 25.0, 1)

        def call(n, w):
            stream = torch.cuda.Stream()
            torch.cuda.synchronize()

            def run():
                with torch.cuda.stream(stream):
                    out = mcao.generate_screen(n, 0.06, 0.15, 25.0, 1, stream=stream)
                    assert w is None or torch.equal(out, w)
            return run
        _together([call(3000, want), call(100, None)], 300)
        return
    alone = sim(True)
    alone.step(1)
    big = sim(True)
    sim(False).step(1)
    big.step(1)
    assert np.array_equal(big.commands(), alone.commands()) and big.psf(0)[1:] == alone.psf(0)[1:]
