"""Column chunks of the allocation-free update: at the edges of the shortest chunk, of the largest
chunk and of the scratch array, against the product in float64 on two calls in a row."""
import pytest

from paper_1608_00386_gb300 import build, mcao

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cmd,n_slopes", [
    (1, 1), (33, 255), (33, 256), (33, 257), (7, 515), (300, 4096), (300, 4097), (31, 20002), (2500, 1030),
    (40000, 3000), (524288, 260)])   # the scratch holds 13 chunks of 40000 rows and one of 524288
def test_split_matches_float64_product(n_cmd, n_slopes):
    import torch
    build.build()
    g = torch.Generator(device="cuda").manual_seed(n_cmd + n_slopes)
    ld = (n_slopes + 3) // 4 * 4
    Rp = torch.full((n_cmd, ld), float("nan"), device="cuda")
    Rp[:, :n_slopes] = torch.randn((n_cmd, n_slopes), generator=g, device="cuda") * 0.01
    R = Rp[:, :n_slopes]
    c = torch.randn(n_cmd, generator=g, device="cuda")
    ref, R64 = c.double(), R.double()
    for _ in range(2):
        s = torch.randn(n_slopes, generator=g, device="cuda")
        mcao.reconstruct_noalloc(R, s, c, 0.37)
        ref = ref + 0.37 * (R64 @ s.double())
    torch.cuda.synchronize()
    # sums of up to n_slopes float products, each rounded: 2^-24 of the terms' size per addition in a chain
    # of at most 4096 / 32 / 4 x 4 + 13, far below 1e-5 of the result's size
    assert float((c.double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max())


def test_beyond_the_scratch_is_refused():
    import torch
    build.build()
    R = torch.zeros((1 << 19) + 1, 4, device="cuda")
    with pytest.raises(mcao.McaoError):
        mcao.reconstruct_noalloc(R, torch.zeros(4, device="cuda"), torch.zeros((1 << 19) + 1, device="cuda"), 0.5)
