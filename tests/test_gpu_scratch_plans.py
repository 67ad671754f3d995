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


@pytest.mark.parametrize("m,n,r,transposed", [(9792, 9472, 148, False), (9472, 9792, 148, True), (4288, 4160, 520, False)])
def test_the_column_sums_leave_the_sum_alone(m, n, r, transposed):
    # A right factor of 9472 rows is 296 chunks of the column sums, a layout for 9792 rows holds 289: behind them lie the column
    # norms and M + G, which the error feedback reads afterwards.
    g = torch.Generator(device="cuda"); g.manual_seed(r)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    X, M, G, Q = rn(m, n) * 0.02, rn(m, n) * 0.3, rn(m, n) * 0.1, rn(m if transposed else n, r)
    Q /= Q.norm(dim=0)
    B = (M + G).double()
    Bt = B.t() if transposed else B
    U, T = torch.linalg.qr(Bt @ Q.double())
    U *= torch.sign(torch.diagonal(T))
    R = Bt.t() @ U
    Qr = R / R.norm(dim=0)
    Mr = B - 0.05 * (R @ U.t() if transposed else U @ R.t())
    d = torch.zeros(r, device="cuda")
    with binding.Dion(mu=0.95) as opt:
        opt.step(X, M, G, Q, 0.01, colnorm_out=d, transposed=transposed)
        assert opt.get_status() == (0, 0)
    # entry by entry: the library's 1e-4 of the largest one
    for got, want in ((M, Mr), (Q, Qr), (d, R.norm(dim=0))):
        assert (got.double() - want).abs().max().item() <= 1e-4 * want.abs().max().item()


def test_what_an_earlier_call_left_in_the_scratch_does_not_matter():
    # Blocked solves (r > 3072) on half pairs scale the inverses of 512-column squares by their largest entry: below the diagonal
    # there must be zeros, not the saved panel of an earlier call of another shape, which lies where the inverses go.
    g = torch.Generator(device="cuda"); g.manual_seed(1)
    rows, r = 14336, 3584
    P = torch.randn(rows, r, generator=g, device="cuda")
    big = torch.randn(73728, 512, generator=g, device="cuda") * 1e15
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    outs = []
    for before in (False, True):
        U = P.clone()
        with binding.Dion(workspace_bytes=6 << 30) as opt:
            if before:
                opt.orthonormalize(73728, 512, 73728, big, flag)
                assert opt.get_status() == (0, 0)
            opt.orthonormalize(rows, r, rows, U, flag)
            assert opt.get_status() == (0, 0) and opt.fallbacks() == 0
        outs.append(U)
    assert torch.equal(outs[0], outs[1])
