"""A radix sort pass whose look-back waits give up (here: at once) sorts as one whose waits end."""
import ctypes as C

import numpy as np
import pytest
import torch

from tests import native_probe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    p = native_probe.load(tmp_path_factory.mktemp("sort_wait"), """
// keys[0] / vals[0] sorted by the low passes * 8 (or 9, 32-bit keys) bits, through keys[1] / vals[1];
// tmp: zeroed scratch
extern "C" int sort(void* k0, void* k1, void* v0, void* v1, void* tmp, long long n, int wide, int bits, int passes,
                    int spin, int tag, void* stream) {
    gs::SortArgs a;
    char* b = static_cast<char*>(tmp);
    a.keys[0] = k0; a.keys[1] = k1;
    a.vals[0] = static_cast<uint32_t*>(v0); a.vals[1] = static_cast<uint32_t*>(v1);
    a.counters = reinterpret_cast<gs::Counters*>(b);
    a.count = &a.counters->n_pairs;
    a.tickets = reinterpret_cast<uint32_t*>(b + 256);
    a.hist = reinterpret_cast<uint32_t*>(b + 512);
    a.lookback = reinterpret_cast<unsigned long long*>(b + 512 + 4 * gs::kSortMaxPasses * gs::kSortMaxBins);
    a.capacity = n;
    a.spin = spin;
    a.tag = tag;
    int shifts[8], nb[8];
    for (int p = 0; p < passes; p++) { shifts[p] = bits * p; nb[p] = bits; }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!wide) return gs::launch_sort32(a, passes, shifts, nb, st);   // the caller filled hist[0]
    const cudaError_t e = gs::launch_sort_count64(a, 0, st);
    return e != cudaSuccess ? e : gs::launch_sort64(a, passes, shifts, st);
}
extern "C" long long tmp_bytes(long long n) {
    return 512 + 4 * gs::kSortMaxPasses * gs::kSortMaxBins + gs::sort_lookback_bytes(n, 9);
}
""")
    p.tmp_bytes.argtypes, p.tmp_bytes.restype = [C.c_longlong], C.c_longlong
    p.sort.argtypes = [C.c_void_p] * 5 + [C.c_longlong] + [C.c_int] * 5 + [C.c_void_p]
    return p


@pytest.mark.parametrize("spin", [0, 1, 1 << 20])
@pytest.mark.parametrize("wide,bits,passes", [(1, 8, 8), (0, 8, 4), (0, 9, 2)])
@pytest.mark.parametrize("n", [1, 4096, 4097, 70_001, 300_000, 2_500_001])
def test_sort_with_waits_that_give_up(probe, n, wide, bits, passes, spin):
    rng = np.random.default_rng(n + bits)
    pool = rng.integers(0, 1 << (63 if wide else 32), size=max(2, n // 50), dtype=np.uint64)
    keys = pool[rng.integers(0, pool.shape[0], n)].astype(np.uint64 if wide else np.uint32)
    vals = rng.permutation(n).astype(np.uint32)
    low = keys if bits * passes >= (64 if wide else 32) else keys & np.uint32((1 << bits * passes) - 1)
    order = np.argsort(low, kind="stable")
    k = [torch.as_tensor(keys.view(np.int64 if wide else np.int32)).cuda(), None]
    v = [torch.as_tensor(vals.view(np.int32)).cuda(), None]
    k[1], v[1] = torch.full_like(k[0], -1), torch.full_like(v[0], -1)
    tmp = torch.zeros(probe.tmp_bytes(n), dtype=torch.uint8, device="cuda")
    tmp[8:16].view(torch.int64).fill_(n)               # Counters::n_pairs
    if not wide:
        hist = np.bincount(keys & np.uint32((1 << bits) - 1), minlength=512).astype(np.int32)
        tmp[512:512 + 2048].view(torch.int32).copy_(torch.as_tensor(hist))
    st = torch.cuda.current_stream().cuda_stream
    assert probe.sort(k[0].data_ptr(), k[1].data_ptr(), v[0].data_ptr(), v[1].data_ptr(), tmp.data_ptr(), n, wide, bits,
                      passes, spin, 3, st) == 0
    torch.cuda.synchronize()
    out_k, out_v = k[passes % 2].cpu().numpy(), v[passes % 2].cpu().numpy()
    np.testing.assert_array_equal(out_k.view(keys.dtype), keys[order])
    np.testing.assert_array_equal(out_v.view(np.uint32), vals[order])
    assert int(tmp[0:4].view(torch.int32)[0]) == 0     # no error
