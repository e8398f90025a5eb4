"""The stage kernel's chunks along s, on the CPU: for one plane to very many, one tile to many, and
batches up to the largest, the chunk length lies in the planes, the launch stays within the grid's
third dimension wherever chunks of 128 planes do, a small grid is cut to fill the slots, and a large
one is not cut short."""
import ctypes

import pytest

from host_build import build


@pytest.fixture(scope="module")
def chunk(tmp_path_factory):
    L = ctypes.CDLL(build("host_chunks.cpp", tmp_path_factory.mktemp("chunks") / "libchunks.so", shared=True))
    L.host_s_chunk.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_double,
                               ctypes.c_int, ctypes.c_int]
    return L.host_s_chunk


@pytest.mark.parametrize("nk", [1, 2, 5, 6, 7, 33, 97, 127, 128, 129, 401, 70000, 9000000])
@pytest.mark.parametrize("nb", [1, 8, 1024])
@pytest.mark.parametrize("tiles", [1, 10, 85, 4257])
@pytest.mark.parametrize("slots,warm,b,extra", [(304, 3.6, 6, 6), (152, 1.0, 6, 1), (152, 0.3, 1, 1)])
def test_chunk_length(chunk, nk, nb, tiles, slots, warm, b, extra):
    n = chunk(tiles * nb, nk, nb, slots, warm, b, extra)
    assert 1 <= n <= min(nk, 128)
    if -(-nk // 128) * nb <= 65535:
        assert -(-nk // n) * nb <= 65535
    if nk >= 97 and tiles * nb * nk <= slots:   # fewer block-planes than slots: as many blocks as planes allow
        assert n == 1
    if tiles * nb >= 20 * slots and nk >= 128:  # many rounds: the queues' fill counts, not the last round
        assert n >= 24 * warm / 3.6
