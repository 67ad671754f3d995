"""GPU: steps on scaled half pairs at the edges of their range, against the step in float64; and chains long enough that the
products add their K splits inside a work item, against single steps (the same bits)."""
import math

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402


def problem(m, n, r, seed, transposed=False, g_dtype=torch.float32):
    g = torch.Generator(device="cuda"); g.manual_seed(seed)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    Q = rn(m if transposed else n, r)
    return rn(m, n) * 0.02, rn(m, n) * 0.3, (rn(m, n) * 0.1).to(g_dtype), Q / Q.norm(dim=0)


def reference(X, M, G, Q, lr, mu, transposed):
    X, B, Q = X.double(), M.double() + G.double(), Q.double()
    Bt = B.t() if transposed else B
    U, R = torch.linalg.qr(Bt @ Q)
    U = U * torch.sign(torch.diagonal(R))
    R = Bt.t() @ U
    Qn = R / R.norm(dim=0)
    L, Lx = (R @ U.t(), Qn @ U.t()) if transposed else (U @ R.t(), U @ Qn.t())
    return X - lr * math.sqrt(X.shape[0] / X.shape[1]) * Lx, B - (1 - mu) * L, Qn


# the smallest shapes that take them, column counts beside the tiles' 64, 128, 192 and 256, odd row tiles, G in bf16
SIZES = [(256, 256, 64, False), (256, 264, 64, False), (264, 256, 64, True), (512, 1536, 64, False), (768, 1000, 72, False), (1000, 768, 136, True), (776, 1544, 128, False), (2056, 768, 192, False),
         (1032, 1040, 248, True), (1096, 1032, 256, False)]


@pytest.mark.parametrize("m,n,r,transposed", SIZES)
@pytest.mark.parametrize("scale_q,aligned", [(1.0, True), (300.0, False)])
def test_step_against_float64(m, n, r, transposed, scale_q, aligned):
    X, M, G, Q = problem(m, n, r, m + r, transposed, torch.bfloat16 if n % 16 else torch.float32)
    Q = Q * scale_q      # (nothing bounds the caller's right factor)
    if not aligned:
        hold = torch.zeros(Q.shape[0] * (r + 1) + 1, device="cuda")
        Qv = hold[1:].view(Q.shape[0], r + 1)[:, :r]
        Qv.copy_(Q)
        Q = Qv
    Xr, Mr, Qr = reference(X, M, G, Q, 0.01, 0.95, transposed)
    with binding.Dion(mu=0.95) as opt:
        opt.step(X, M, G, Q, 0.01, transposed=transposed)
        assert opt.get_status() == (0, 0)
    rel = lambda a, b: ((a.double() - b).norm() / b.norm()).item()
    # 2^-22 operands, chains of at most 1024 (1e-6), a Gaussian panel (condition <= 3): below 1e-5 of R; M takes a twentieth of
    # it; X the rounding of its factors to 11 bits (2^-11 of a change of 1e-2 of X)
    assert rel(Q, Qr) <= 1e-5 and rel(M, Mr) <= 1e-6 and rel(X, Xr) <= 1e-5


@pytest.mark.parametrize("m,n,r,count", [(768, 768, 192, 14), (768, 768, 200, 28), (256, 3072, 72, 30), (500, 260, 24, 40), (333, 515, 83, 24),
                                         (384, 384, 48, 30)])
def test_long_chain_equals_single_steps(m, n, r, count):
    single = [problem(m, n, r, k) for k in range(count)]
    chain = [tuple(t.clone() for t in p) for p in single]
    with binding.Dion(mu=0.95) as opt:
        for X, M, G, Q in single:
            opt.step(X, M, G, Q, 0.01)
        opt.step_grouped(chain, 0.01)
        assert opt.get_status() == (0, 0)
    for k, (a, b) in enumerate(zip(single, chain)):
        for name, u, v in zip("XMGQ", a, b):
            assert torch.equal(u, v), f"matrix {k}: {name}"
