"""GPU: the factorization's launch where its row blocks, taken one or two at a time, end: panels and inverses of odd and even numbers of
64-row blocks, with a last one that is short, for one matrix and for a chain."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402
from test_gpu_orth_sizes import test_against_float64 as check  # noqa: E402

# rows, r: the panel solved in the launch (1 to 5 row blocks, 2 to 5 column blocks), then the inverse (rows r > 1.1e6)
PANELS = [(128, 65), (129, 65), (192, 128), (193, 128), (256, 132), (260, 132), (1027, 250), (900, 257), (4100, 320), (5000, 321),
          (8200, 192), (8192, 196)]


@pytest.mark.parametrize("rows,r", PANELS)
def test_pairs_of_row_blocks(rows, r):
    check(rows, r, 4 * r)


@pytest.mark.parametrize("rows,r", [(257, 200), (320, 320), (451, 387)])
def test_pairs_of_row_blocks_in_adaptive_rounds(rows, r):
    check(rows, r, r)


@pytest.mark.parametrize("m,n,r,count", [(448, 640, 112, 9), (832, 1090, 208, 5), (200, 260, 200, 3)])
def test_chain_equals_single_steps(m, n, r, count):
    g = torch.Generator(device="cuda"); g.manual_seed(m + r)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    mats = [(rn(m, n), rn(m, n), rn(m, n), torch.nn.functional.normalize(rn(n, r), dim=0)) for _ in range(count)]
    single = [tuple(t.clone() for t in a) for a in mats]
    with binding.Dion() as opt:
        for X, M, G, Q in single:
            opt.step(X, M, G, Q, 0.01)
        opt.step_grouped(mats, 0.01)
        assert opt.get_status() == (0, 0)
    for k, (a, b) in enumerate(zip(single, mats)):
        for name, u, v in zip("XMGQ", a, b):
            assert torch.equal(u, v), f"matrix {k}: {name}"


@pytest.mark.parametrize("rows,r", [(70, 66), (900, 83), (2111, 1023)])
def test_probe_of_ranks_that_are_no_multiple_of_four(rows, r):
    # (its decision shows in the rounds: one for a Gaussian panel, two where columns are nearly parallel)
    g = torch.Generator(device="cuda"); g.manual_seed(rows)
    P = torch.randn(rows, r, generator=g, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    with binding.Dion(orth=binding.ORTH_CHOLQR2) as opt:
        opt.orth_rounds()
        for spread, rounds in ((1.0, (1, 1 if rows > 3 * r // 2 else 2)), (2e-3, (2, 2))):
            A = P[:, :1] + spread * P if spread < 1 else P.clone()
            opt.orthonormalize(rows, r, rows, A, flag)
            torch.cuda.synchronize()
            assert rounds[0] <= opt.orth_rounds() <= rounds[1], spread
        assert opt.get_status() == (0, 0)


@pytest.mark.parametrize("r", [4, 22, 64])
def test_partial_sums_of_one_block_take_no_launch_of_their_own(r):
    # rows as the inner dimension: the Gram product is cut in 8, 11 and 16 parts
    launches = []
    with binding.Dion(orth=binding.ORTH_CHOLQR2) as opt:
        flag = torch.zeros(1, dtype=torch.int32, device="cuda")
        for rows in (1024, 2048, 4096):
            g = torch.Generator(device="cuda"); g.manual_seed(rows + r)
            P = torch.randn(rows, r, generator=g, device="cuda")
            l0 = opt.launch_count()
            opt.orthonormalize(rows, r, rows, P, flag)
            torch.cuda.synchronize()
            launches.append(opt.launch_count() - l0)
            E = P.double().t() @ P.double() - torch.eye(r, device="cuda", dtype=torch.float64)
            assert E.norm().item() <= 2 * 3e-5 * r ** 0.5      # (as in test_gpu_orth_sizes.py)
        assert opt.get_status() == (0, 0)
    assert len(set(launches)) == 1, launches
