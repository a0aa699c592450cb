"""Where a NaN in a vector goes: into the commands of its row, and no further."""
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


def _case():
    cfg = inputs.mcao_20m(noise=False)
    cfg["layers"] = cfg["layers"][:1]
    g = mcao.Sim(cfg)
    g.load_atmosphere(inputs.make_screens(cfg))
    g.load_dms()
    g.set_commands(np.zeros(g.query(mcao.Q_COMMANDS), np.float32))
    return cfg, g


@pytest.mark.parametrize("rotated", [False, True])
def test_a_nan_in_a_vector_reaches_the_commands_of_its_row(rotated):
    import torch
    cfg, g = _case()
    if rotated:
        g.set_misregistration(1, 0.0, 0.0, 0.02, 1.0)
    D = g.interaction_matrix().double().cpu().numpy()
    row = g.query(mcao.Q_VALID, 0) // 2
    v = np.random.default_rng(2).normal(size=(1, D.shape[0])).astype(np.float32)
    want = v.astype(np.float64) @ D
    v[0, row] = np.nan
    got = g.slopes_vjp(torch.from_numpy(v).cuda())[0].cpu().numpy()[0]
    # the row's actuators on each DM: the columns and rows that have a value (their far corners may underflow)
    off, col = np.ones(D.shape[1], bool), 0
    for m in cfg["dms"]:
        ok = np.asarray(m["valid"]).reshape(m["ny"], m["nx"]).astype(bool)
        grid = np.zeros(ok.shape, bool)
        n = int(ok.sum())
        grid[ok] = D[row, col:col + n] != 0.0
        off[col:col + n] = ~(grid.any(axis=1)[:, None] & grid.any(axis=0)[None, :])[ok]
        col += n
    assert 0.2 < off.mean() < 1.0
    assert np.isfinite(got[off]).all() and np.linalg.norm(got[off] - want[0, off]) <= 1e-5 * np.linalg.norm(want)
    assert np.isnan(got[np.abs(D[row]) > 1e-6 * np.abs(D[row]).max()]).all()
