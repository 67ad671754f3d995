"""GPU: the factorization's launch where a wait for tensor-core products runs out for some threads of a block only.  (The threads report
it while the products are done: nothing is in flight when the block leaves.)  The block leaves as a whole, the launch ends with
DION_STATUS_TIMEOUT, and the next call is not touched by it."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2504_05295_b200 import binding  # noqa: E402

TIMEOUT = binding.STATUS_TIMEOUT
# rows, r, short side: the panel solved in the launch, one product behind it (inverse), adaptive rounds, r no multiple of four
PANELS = [(1536, 384, 1536), (4096, 512, 4096), (512, 512, 512), (1100, 386, 1600)]


def _lose(opt, cta, threads):
    fn = binding.load_library().dion_debug_flow_lose
    fn.argtypes, fn.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int], ctypes.c_int
    assert fn(opt._ctx, cta, threads) == 0


def _check(rows, r, short, cta, threads):
    g = torch.Generator(device="cuda"); g.manual_seed(rows + r)
    P0 = torch.randn(rows, r, generator=g, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    with binding.Dion() as opt:
        def call():
            P = P0.clone()
            opt.orthonormalize(rows, r, short, P, flag)
            torch.cuda.synchronize()
            return P
        before = call()
        assert opt.get_status() == (0, 0)
        _lose(opt, cta, threads)
        call()
        assert opt.get_status()[0] & TIMEOUT
        _lose(opt, 0, 0)
        flag.zero_()
        assert torch.equal(call(), before)
        assert opt.get_status() == (0, 0) and int(flag.item()) == 0


@pytest.mark.parametrize("rows,r,short", PANELS)
@pytest.mark.parametrize("threads", [1, 40, 65, 200, 256])
def test_helpers_leave_as_a_whole(rows, r, short, threads):
    _check(rows, r, short, -1, threads)


@pytest.mark.parametrize("rows,r,short", PANELS + [(640, 112, 448)])
@pytest.mark.parametrize("threads", [1, 65, 256, 257, 300])
def test_runner_leaves_as_a_whole(rows, r, short, threads):
    # (threads 256 on: its service warps too)
    _check(rows, r, short, 0, threads)
