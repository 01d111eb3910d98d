"""The radix sort's grid: a look-back word counts a block's keys of one digit in 24 bits, so a
block's run of chunks stays below 2^24 keys on a device of any size, for every accepted capacity."""
import ctypes as C

import pytest

from tests import native_probe

CHUNK = 4096


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    p = native_probe.load(tmp_path_factory.mktemp("sort_grid"), """
extern "C" int grid(long long capacity, int sms) { return gs::sort_grid(capacity, sms); }
extern "C" int chunk() { return gs::kSortChunk; }
extern "C" size_t words_end(long long capacity, int bits) { return gs::sort_lookback_bytes(capacity, bits); }
extern "C" size_t group_bytes() { return gs::kSortGroupBytes; }
""")
    p.grid.argtypes = [C.c_longlong, C.c_int]
    p.words_end.argtypes, p.words_end.restype = [C.c_longlong, C.c_int], C.c_size_t
    p.group_bytes.restype = C.c_size_t
    return p


@pytest.mark.parametrize("sms", [1, 8, 16, 64, 100, 127, 128, 148, 152, 300])
@pytest.mark.parametrize("capacity", [0, 1, CHUNK, CHUNK + 1, 10_000_000, 2 ** 24, 2 ** 28 + 17, 2 ** 31, 2 ** 32 - 1])
def test_a_blocks_run_fits_its_look_back_words(probe, sms, capacity):
    assert probe.chunk() == CHUNK
    g = probe.grid(capacity, sms)
    chunks = -(-capacity // CHUNK)
    assert 1 <= g <= 512 and g <= max(1, chunks)
    # counts at and below the capacity: run t of a pass over nch chunks by min(nch, g) blocks
    for nch in {chunks, chunks - 1, chunks // 2, chunks // 3}:
        blocks = min(nch, g)
        if blocks > 0:
            assert -(-nch // blocks) * CHUNK < 2 ** 24
    # the words of every block lie inside the sized region, and the resident blocks stay as they were
    assert probe.group_bytes() + 4 * g * 512 <= max(probe.words_end(capacity, 9), probe.group_bytes() + 4 * 512)
    if sms >= 148:
        assert g == max(1, min(chunks, 2 * sms, 512))
