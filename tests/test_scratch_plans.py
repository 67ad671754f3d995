"""The row chunks of the panel passes fit the scratch that is laid out for them, whichever side of the matrix the panel is."""
import ctypes

import pytest

from paper_2504_05295_b200 import binding, build


@pytest.fixture(scope="module")
def chunks():
    build.build()
    fn = ctypes.CDLL(binding.LIB_PATH).dion_debug_chunks
    fn.argtypes = [ctypes.c_int64] * 4 + [ctypes.c_int, ctypes.POINTER(ctypes.c_int64)]
    out = (ctypes.c_int64 * 4)()

    def call(m, n, r, rows, sms):
        assert fn(m, n, r, rows, sms, out) == 0
        return list(out)

    return call


def sides():
    some = sorted({k * s for k in (64, 4288, 4160, 9472, 9792) for s in (1, 2, 3, 5)} | {1, 31, 333, 16384, 16385, 16448, 53248})
    return [(m, n) for m in some for n in some]


def test_probe_chunks_fit(chunks):
    # 16384 rows take 512 chunks, 16448 take 257: a layout for the long side holds fewer than the short side would use
    for m, n in sides():
        for r in {1, min(m, n, 148), min(m, n, 1024)}:
            for rows in (m, n):
                used, room = chunks(m, n, r, rows, 148)[2:]
                assert 0 < used <= room, (m, n, r, rows)


def test_column_normalization_chunks_fit(chunks):
    # 148 SMs, r = 148: 9472 rows (the right factor of 9792 x 9472) take 296 chunks of 32, 9792 take 288 of 34
    for sms in (132, 148):
        for m, n in sides():
            for r in {1, min(m, n, 148), min(m, n, 520)}:
                for rows in (m, n):
                    used, room = chunks(m, n, r, rows, sms)[:2]
                    assert 0 < used <= room, (m, n, r, rows, sms)
