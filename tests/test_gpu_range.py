"""GPU: matrices with a block of rows, columns or both far below the rest.  What the calls make of the block is as accurate
against float64, relative to the block itself, as what they make of the whole."""
import math

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402

MU, LR = 0.95, 0.01


def problem(m, n, r, axis, exponent, transposed=False, seed=3):
    g = torch.Generator(device="cuda"); g.manual_seed(seed)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    X, M, G, Q = rn(m, n) * 0.02, rn(m, n) * 0.3, rn(m, n) * 0.1, rn(m if transposed else n, r)
    at = block(axis, m, n)
    for t in (X, M, G):
        t[at] *= 2.0 ** exponent
    # (the right factor that such a matrix has had for a while: its small rows belong to the small rows or columns)
    if axis == ("rows" if transposed else "cols"):
        Q[Q.shape[0] // 2:] *= 2.0 ** exponent
    return X, M, G, Q / Q.norm(dim=0)


def block(axis, m, n):
    return {"rows": (slice(m // 2, m), slice(None)), "cols": (slice(None), slice(n // 2, n)), "none": (slice(None), slice(None))}[axis]


def reference(M, G, Q, transposed):
    B, Q = M.double() + G.double(), Q.double()
    Bt = B.t() if transposed else B
    U, T = torch.linalg.qr(Bt @ Q)
    U = U * torch.sign(torch.diagonal(T))
    R = Bt.t() @ U
    return B, (R @ U.t() if transposed else U @ R.t()), R / R.norm(dim=0)


def off(a, b):
    return ((a.double() - b).norm() / b.norm()).item()


def check(M, Q, ref, axis, transposed):
    B, low, Qr = ref
    at = block(axis, *B.shape)
    # Factors of 16 significant bits (2^-17 of an entry) and chains of at most 1024 terms (8e-6), twice, on a panel of condition
    # at most 3; M carries (1 - mu) of it.
    assert off(((B - M.double()) / (1 - MU))[at], low[at]) <= 4e-5 + 1e-6 / (1 - MU)      # (M rounded to 24 bits)
    assert off(M[at], (B - (1 - MU) * low)[at]) <= 2e-6
    rows = slice(Q.shape[0] // 2, None) if axis == ("rows" if transposed else "cols") else slice(None)
    assert off(Q[rows], Qr[rows]) <= 4e-5


CASES = [("none", 0), ("rows", -18), ("cols", -18), ("rows", -26), ("cols", -26), ("rows", -40), ("cols", -40)]


@pytest.mark.parametrize("m,n,r,transposed", [(256, 512, 64, False), (1536, 512, 64, True), (1032, 1040, 136, False)])
@pytest.mark.parametrize("axis,exponent", CASES)
def test_step(m, n, r, transposed, axis, exponent):
    X, M, G, Q = problem(m, n, r, axis, exponent, transposed)
    ref = reference(M, G, Q, transposed)
    with binding.Dion(mu=MU) as opt:
        opt.step(X, M, G, Q, LR, transposed=transposed)
        assert opt.get_status() == (0, 0)
    check(M, Q, ref, axis, transposed)


@pytest.mark.parametrize("axis,exponent", CASES)
def test_data_parallel_and_sharded_calls(axis, exponent):
    m, n, r = 768, 640, 128
    X, M, G, Q = problem(m, n, r, axis, exponent)
    ref = reference(M, G, Q, False)
    P, W = torch.zeros(m, r, device="cuda"), torch.zeros(n, r, device="cuda")
    sums, flag = torch.zeros(r, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    for sharded in (False, True):
        Xk, Mk, Qk = X.clone(), M.clone(), Q.clone()
        desc = binding.matrix_desc(Xk, Mk, G, Qk)
        with binding.Dion(mu=MU) as opt:
            if sharded:
                opt.shard_project(desc, n, P, flag)
                opt.orthonormalize(m, r, n, P, flag)
                opt.shard_factor(desc, n, P, W, sums, flag)
                opt.shard_finish(desc, n, P, W, sums, flag, LR)
            else:
                opt.dp_project(desc, P, flag)
                opt.dp_factor(desc, P, W, flag)
                opt.dp_finish(desc, P, W, flag, LR)
            assert opt.get_status() == (0, 0)
        check(Mk, Qk, ref, axis, False)


def test_a_chain_of_both_kinds_equals_single_steps():
    m, n, r = 512, 768, 96
    kinds = [("none", 0), ("rows", -30), ("none", 0), ("cols", -24), ("rows", -17), ("none", 0)]
    single = [problem(m, n, r, a, e, seed=k) for k, (a, e) in enumerate(kinds)]
    chain = [tuple(t.clone() for t in p) for p in single]
    with binding.Dion(mu=MU) as opt:
        for X, M, G, Q in single:
            opt.step(X, M, G, Q, LR)
        opt.step_grouped(chain, LR)
        assert opt.get_status() == (0, 0)
    for k, (a, b) in enumerate(zip(single, chain)):
        for name, u, v in zip("XMGQ", a, b):
            assert torch.equal(u, v), f"matrix {k}: {name}"


@pytest.mark.parametrize("exponent", [-30, 40])
def test_columns_of_the_right_factor_of_any_scale(exponent):
    # the caller's right factor spans the same space whatever its columns' lengths
    m, n, r = 512, 640, 64
    X, M, G, Q = problem(m, n, r, "none", 0)
    ref = reference(M, G, Q, False)
    Q[:, r // 2:] *= 2.0 ** exponent
    with binding.Dion(mu=MU) as opt:
        opt.step(X, M, G, Q, LR)
        assert opt.get_status() == (0, 0)
    check(M, Q, ref, "none", False)


def test_zero_rows_and_columns_are_no_wide_range():
    # rows of an embedding that no token touched: exact zeros do not ask for more range, the results keep 22 bits (1e-5 with 17)
    m, n, r = 1024, 512, 64
    X, M, G, Q = problem(m, n, r, "none", 0)
    M[100:300] = 0; G[100:300] = 0; M[:, 7:40] = 0; G[:, 7:40] = 0
    B, low, Qr = reference(M, G, Q, False)
    with binding.Dion(mu=MU) as opt:
        opt.step(X, M, G, Q, LR)
        assert opt.get_status() == (0, 0)
    assert off(Q, Qr) <= 2e-6
    assert torch.equal(M[100:300], torch.zeros_like(M[100:300])) and torch.equal(Q[7:40], torch.zeros_like(Q[7:40]))


@pytest.mark.parametrize("refresh", [True, False])
@pytest.mark.parametrize("m,n,r", [(640, 768, 128), (1288, 648, 136)])
@pytest.mark.parametrize("axis,exponent", CASES)
def test_lazy_step(m, n, r, refresh, axis, exponent):
    X, M, G, Q = problem(m, n, r, axis, exponent)
    at = block(axis, m, n)
    if not refresh:      # the factor of an earlier refresh
        Q = torch.linalg.qr(Q)[0].contiguous()
    B, X0, Qr = M.double() + G.double(), X.double(), Q.double()
    if refresh:
        Qr, T = torch.linalg.qr(B.t() @ (B @ Qr))
        Qr = Qr * torch.sign(torch.diagonal(T))
    W = B @ Qr
    low, dX = W @ Qr.t(), LR * math.sqrt(m / n) * (W / W.norm(dim=0)) @ Qr.t()
    with binding.Dion(mu=MU) as opt:
        opt.lazy_step(X, M, G, Q, LR, refresh=refresh)
        assert opt.get_status() == (0, 0)
    # products of 22 significant bits and chains of at most 1024 terms (8e-6), three in a row on a well-conditioned panel
    assert off(((B - M.double()) / (1 - MU))[at], low[at]) <= 4e-5 + 1e-6 / (1 - MU)
    assert off(M[at], (B - (1 - MU) * low)[at]) <= 2e-6
    assert ((X.double() - X0 + dX)[at]).norm() <= 4e-5 * dX[at].norm() + 2.0 ** -24 * X0[at].norm()
    rows = slice(n // 2, None) if axis == "cols" else slice(None)
    assert off(Q[rows], Qr[rows]) <= 4e-5


def test_lazy_step_of_graded_columns_and_of_a_breakdown():
    m, n, r = 512, 768, 128
    # T = (M + G) Q with columns 2^-24 of others: only Z has to see them
    X, M, G, Q = problem(m, n, r, "none", 0)
    Q[:, r // 2:] *= 2.0 ** -24
    B = M.double() + G.double()
    want, T = torch.linalg.qr(B.t() @ (B @ Q.double()))
    with binding.Dion(mu=MU) as opt:
        opt.lazy_step(X, M, G, Q, LR, refresh=True)
        assert opt.get_status() == (0, 0)
        assert off(Q, want * torch.sign(torch.diagonal(T))) <= 4e-5
        # a panel of rank one less than its width cancels the step, on either kind of product
        for exponent in (0, -30):
            X, M, G, Q = problem(m, n, r, "rows", exponent)
            Q[:, 5] = Q[:, 3]
            before = [t.clone() for t in (X, M, Q)]
            opt.lazy_step(X, M, G, Q, LR, refresh=True)
            assert opt.get_status() == (binding.STATUS_BREAKDOWN, 1)
            for a, b in zip(before, (X, M, Q)):
                assert torch.equal(a, b)


@pytest.mark.parametrize("exponent", [-37, -38, -40, -42])
def test_adaptive_rounds_of_columns_beyond_the_pair(exponent):
    # At 2^-38 of the others a column's half pair is a few odd bits or zero, and so is its entry of the Gram matrix: the first round
    # leaves it as it is, the next one sees it beside columns of norm 1.  The split lies inside a block of 64 columns.
    rows, r = 4096, 1032
    g = torch.Generator(device="cuda"); g.manual_seed(r)
    P = torch.randn(rows, r, generator=g, device="cuda")
    P[:, r // 2:] *= 2.0 ** exponent
    want, T = torch.linalg.qr(P.double())
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    with binding.Dion() as opt:
        opt.orthonormalize(rows, r, rows, P, flag)
        assert opt.get_status() == (0, 0) and int(flag.item()) == 0
    assert off(P, want * torch.sign(torch.diagonal(T))) <= 4e-5      # 22 bits, chains of at most 1024 terms, twice


@pytest.mark.parametrize("axis,exponent", CASES)
@pytest.mark.parametrize("rows,r,short", [(4096, 768, 4096), (4104, 1024, 4104), (4096, 1032, 4096), (8192, 512, 2048)])
def test_panel(rows, r, short, axis, exponent):
    # panels whose Gram matrix, and the product that takes them to U, run on half pairs (the third: adaptive rounds)
    g = torch.Generator(device="cuda"); g.manual_seed(r)
    P = torch.randn(rows, r, generator=g, device="cuda")
    at = block(axis, rows, r)
    P[at] *= 2.0 ** exponent
    want, T = torch.linalg.qr(P.double())
    want *= torch.sign(torch.diagonal(T))
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    with binding.Dion() as opt:
        opt.orthonormalize(rows, r, short, P, flag)
        assert opt.get_status() == (0, 0) and int(flag.item()) == 0
    # 22 bits, chains of at most 1024 terms, twice; condition at most 3
    assert off(P[at], want[at]) <= 4e-5
