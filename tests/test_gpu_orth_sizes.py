"""GPU: the orthonormalization at the edges of its tiles, against the QR factorization of the same panel in float64."""
import math

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402

# rows, r, short side of the matrix (4 r <= short side: CholeskyQR2, else the adaptive rounds)
SIZES = [(4, 1, 4), (70, 1, 64), (513, 63, 256), (513, 64, 256), (520, 65, 264), (777, 127, 520), (640, 129, 520), (2048, 193, 800),
         (2111, 513, 2100), (1100, 1030, 4120), (5000, 260, 1040), (200, 63, 63), (192, 65, 65), (300, 193, 193), (1030, 1030, 1030),
         (520, 512, 512), (1216, 1026, 1026)]


@pytest.mark.parametrize("rows,r,short", SIZES)
def test_against_float64(rows, r, short):
    g = torch.Generator(device="cuda"); g.manual_seed(rows * 7 + r)
    P0 = torch.randn(rows, r, generator=g, device="cuda")
    if 4 * r > min(rows, short):      # graded columns: the first round's pivots are floored
        P0 *= torch.logspace(0, -3, r, device="cuda")
    P = P0.clone()
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    with binding.Dion() as opt:
        opt.orthonormalize(rows, r, short, P, flag)
        torch.cuda.synchronize()
        assert opt.get_status() == (0, 0) and int(flag.item()) == 0
    U, D = P.double(), P0.double()
    # A panel is done when |U^T U - I|_F <= 3e-5 sqrt(r) by an estimate of 8 probes (relative spread sqrt(2 / 8): twice that
    # value is beyond two deviations).
    E = U.t() @ U - torch.eye(r, device="cuda", dtype=torch.float64)
    assert E.norm().item() <= 2 * 3e-5 * math.sqrt(r)
    # U R = P with R upper triangular and a positive diagonal: the backward error of products with 22-bit operands and
    # chains of 1024 (8e-6 relative per product), two per round.
    R = U.t() @ D
    scale = D.norm(dim=0)
    assert ((U @ R - D).norm(dim=0) <= 4e-5 * scale).all()
    # U^T P is U^T U R: below the diagonal it carries E R
    assert (torch.tril(R, -1).norm(dim=0) <= (4e-5 + E.norm().item()) * scale).all()
    assert (torch.diagonal(R) > 0).all()
