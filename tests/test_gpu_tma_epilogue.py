"""GPU: the TMA epilogue of the rank-r updates against the register epilogue (bit 3 of the hook's variant word keeps that
one): the same operations per element, so the same bits, and nothing written outside the output."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from test_gpu_gemm_engines import GemmArgs, lib  # noqa: E402,F401


def product(lib, M, N, K, epi, c2_dtype, pairs, pad, variant):
    g = torch.Generator(device="cuda"); g.manual_seed(M + 7 * N + K)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    A, B = rn(M, K), rn(N, K)
    Ah, Bh = A.to(torch.bfloat16), B.to(torch.bfloat16)
    Al, Bl = (A - Ah.float()).to(torch.bfloat16), (B - Bh.float()).to(torch.bfloat16)
    Cb = torch.full((M + 8, N + pad), 7.0, device="cuda")
    Cb[:M, :N] = rn(M, N)
    C0 = Cb.clone()
    C2 = torch.zeros(M, N + pad, device="cuda", dtype=c2_dtype)
    C2[:, :N] = rn(M, N).to(c2_dtype)
    a = GemmArgs()
    a.M, a.N, a.K = M, N, K
    a.A, a.a_si, a.a_sk = Ah.data_ptr(), K, 1
    a.B, a.b_sk, a.b_sn = Bh.data_ptr(), 1, K
    if pairs:
        a.A16lo, a.B16lo = Al.data_ptr(), Bl.data_ptr()
    a.C, a.ldc, a.epi = Cb.data_ptr(), N + pad, epi
    a.C2, a.ldc2, a.c2_mode = C2.data_ptr(), N + pad, 1 if c2_dtype == torch.float32 else 2
    a.alpha, a.ab16, a.variant = 0.05, 1, variant
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = lib.dion_debug_gemm(2, 1, ctypes.byref(a), None, 0, status.data_ptr(), int(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0 and int(status.item()) == 0
    assert torch.equal(Cb[M:], C0[M:]) and torch.equal(Cb[:, N:], C0[:, N:])
    if pairs:
        acc = A.double() @ B.double().t()
    else:
        acc = Ah.double() @ Bh.double().t()
    base = {1: C0[:M, :N].double(), 2: C0[:M, :N].double() + C2[:, :N].double(), 3: C2[:, :N].double()}[epi]
    want = base - 0.05 * acc
    return Cb[:M, :N].clone(), float((Cb[:M, :N].double() - want).norm() / want.norm())


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("M,N,K,pad", [(512, 256, 64, 0), (520, 264, 72, 8), (1000, 1304, 1024, 0), (648, 392, 328, 8), (4096, 512, 128, 0),
                                       (5000, 4104, 64, 16)])
def test_same_bits_as_the_register_epilogue(lib, M, N, K, pad, pairs):  # noqa: F811
    for epi, dt in [(1, torch.float32), (2, torch.float32), (2, torch.bfloat16), (3, torch.float32)]:
        got, err = product(lib, M, N, K, epi, dt, pairs, pad, 0)
        # 2^-16 operand error of the pairs (bf16 arrays: none), relative to a result of norm >= that of the product x 0.05
        assert err < 1e-5, (epi, dt, err)
        ref, _ = product(lib, M, N, K, epi, dt, pairs, pad, 8)
        assert torch.equal(got, ref), (epi, dt)
