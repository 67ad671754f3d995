"""GPU: panels on the short side of a long matrix, whose chunk plans are not those of the long side."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402


@pytest.mark.parametrize("long_side", [16448, 17000, 53248])
def test_the_probe_leaves_the_saved_panel_alone(long_side):
    # A panel of 16384 rows is 512 chunks of the probe, a layout for 16448 rows holds 258.  The saved panel lies behind them:
    # a pivot that fails (nearly parallel columns) must find it as it was.
    rows, r = 16384, 96
    g = torch.Generator(device="cuda"); g.manual_seed(long_side)
    P = torch.randn(rows, 1, generator=g, device="cuda") + 1e-4 * torch.randn(rows, r, generator=g, device="cuda")
    outs = []
    for n_total in (rows, long_side):
        U = P.clone()
        flag = torch.zeros(1, dtype=torch.int32, device="cuda")
        with binding.Dion() as opt:
            opt.orthonormalize(rows, r, n_total, U, flag)
            assert opt.get_status() == (0, 0) and int(flag.item()) == 0 and opt.fallbacks() == 1
        outs.append(U)
    assert torch.equal(outs[0], outs[1])
    U, D = outs[1].double(), P.double()
    # Gram-Schmidt twice in fp32: orthonormal to a few roundings per column, and U R = P to those of a column's sums
    assert (U.t() @ U - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max().item() <= 1e-5
    assert ((U @ (U.t() @ D) - D).norm(dim=0) <= 1e-5 * D.norm(dim=0)).all()
