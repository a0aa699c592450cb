"""Where NaN in a screen or in a vector goes: into the derivatives and products of the subapertures that see
it, and no further."""
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


def _case(spoil):
    """The 20 m system with one layer, its screen spoiled at one point over the pupil or not."""
    cfg = inputs.mcao_20m(noise=False)
    cfg["layers"] = cfg["layers"][:1]
    n = cfg["layers"][0]["n"]
    screen = inputs.make_screens(cfg)[0]
    if spoil:
        screen[n // 2 + 70, n // 2 + 60] = np.nan
    g = mcao.Sim(cfg)
    g.load_atmosphere([screen])
    g.load_dms()
    g.set_commands(np.zeros(g.query(mcao.Q_COMMANDS), np.float32))
    return cfg, g


def _blind_rows(cfg, g):
    """True for the slopes of every subaperture with a NaN sample."""
    out = []
    for w, ww in enumerate(cfg["wfs"]):
        n, p = ww["n_sub"], ww["n_px"]
        bad = np.isnan(g.wfs_phase(w)).reshape(n, p, n, p).any(axis=(1, 3)).ravel()[g.valid(w)]
        out += [bad, bad]
    return np.concatenate(out)


def test_a_spoiled_screen_spoils_the_matrix_rows_that_see_it():
    import torch
    _, good = _case(False)
    D0 = good.interaction_matrix().cpu().numpy()
    cfg, g = _case(True)
    blind = _blind_rows(cfg, g)
    assert 0 < blind.sum() < blind.size // 4
    D = g.interaction_matrix().cpu().numpy()
    assert np.array_equal(D[~blind], D0[~blind])
    # the blind rows' entries are NaN wherever they have a sizeable value without the spoiled point
    assert np.isnan(D[blind][np.abs(D0[blind]) > 1e-6 * np.abs(D0).max()]).all()
    # vectors that leave those slopes out have finite products, with the values of the other rows
    v = torch.from_numpy(np.random.default_rng(1).normal(size=(2, blind.size)).astype(np.float32)).cuda()
    v[:, torch.from_numpy(blind).cuda()] = 0.0
    want = v.double().cpu().numpy()[:, ~blind] @ D[~blind].astype(np.float64)
    for phase in (False, True):
        gc, gp = g.slopes_vjp(v, phase=phase)
        assert np.linalg.norm(gc.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
        assert gp is None or bool(torch.isnan(gp).any())   # 0 times NaN, sample by sample
    # a vector that has them does not hide them
    v[:] = 1.0
    assert np.isnan(g.slopes_vjp(v)[0].cpu().numpy()).any()


@pytest.mark.parametrize("rotated", [False, True])
def test_a_nan_in_a_vector_reaches_the_commands_of_its_row(rotated):
    import torch
    cfg, g = _case(False)
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
