"""GPU: the two rank-r updates of a step side by side (one launch of the FMA engine, or two branches of a replayed graph) against the
same step with one after the other, which is what a profiled step launches: the same bits."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402

# m, n, r: tiles of 64 x 64, of 128 x 32 (few columns) and of 128 x 128 (from 148 of them and r = 96 on), the first size on either side;
# then shapes that are replayed as a graph, rounded factors in half and in TF32
FMA = [(1001, 333, 83), (70, 66, 5), (4100, 32, 20), (4100, 33, 20), (1601, 1603, 97), (1601, 1603, 95), (1537, 1409, 130)]
REPLAYED = [(256, 512, 64), (520, 264, 72), (2048, 2048, 128), (260, 388, 68)]


@pytest.mark.parametrize("m,n,r", FMA + REPLAYED)
@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("g_dtype", [torch.float32, torch.bfloat16])
def test_same_bits_as_one_after_the_other(m, n, r, transposed, g_dtype):
    g = torch.Generator(device="cuda"); g.manual_seed(m + r)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    start = (rn(m, n), rn(m, n), rn(m, n).to(g_dtype), torch.nn.functional.normalize(rn(m if transposed else n, r), dim=0))
    results, launches = [], []
    for profiled in (False, True):
        X, M, G, Q = (t.clone() for t in start)
        with binding.Dion() as opt:
            opt.profile_enable(profiled)
            for _ in range(3):
                l0 = opt.launch_count()
                opt.step(X, M, G, Q, 0.01, transposed=transposed)
            torch.cuda.synchronize()
            launches.append(opt.launch_count() - l0)
            assert opt.get_status() == (0, 0)
        results.append((X, M, Q))
    for name, a, b in zip("XMQ", *results):
        assert torch.equal(a, b), name
    if (m, n, r) in FMA:
        assert launches[0] == launches[1] - 1      # (both updates in one launch)
