"""Scans of the binning whose waits run out: the first chunk is handed to nobody, so every later
chunk waits for it in vain.  The kernels return, the status says so, and the workspace's next call
works."""
import ctypes as C

import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests import native_probe
from tests.gpu_helpers import planes_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    p = native_probe.load(tmp_path_factory.mktemp("scan_wait"), """
// scratch: zeroed; the look-back words of both scans, then digit counts and tickets
extern "C" int scan(const gs_ws_layout* L, void* ws, int tile, void* scratch, int pairs, int spin, void* stream) {
    using namespace gs;
    auto at = [&](size_t off) { return static_cast<char*>(ws) + off; };
    BinArgs b;
    b.n = L->n; b.n_views = L->n_views; b.tile = tile; b.max_pairs = L->max_pairs;
    b.views = reinterpret_cast<View*>(at(L->views));
    b.proj = reinterpret_cast<float4*>(at(L->proj));
    b.vis_bits = reinterpret_cast<uint32_t*>(at(L->vis_bits));
    b.entry_scan = static_cast<unsigned long long*>(scratch);
    b.pair_scan = b.entry_scan + entry_scan_words(L->n, L->n_views);
    uint32_t* w = reinterpret_cast<uint32_t*>(b.pair_scan + pair_scan_words(L->n, L->n_views));
    b.ehist = w; b.phist = w + kSortMaxBins; b.phist_mask = 0;
    b.tickets = w + 2 * kSortMaxBins;
    b.ekeys = reinterpret_cast<uint32_t*>(at(L->ekeys0));
    b.evals = reinterpret_cast<uint32_t*>(at(L->evals0));
    b.entries = reinterpret_cast<uint32_t*>(at(L->entries));
    b.erect = reinterpret_cast<uint4*>(at(L->erect));
    b.sorted_evals = b.evals;
    b.pkeys = reinterpret_cast<uint32_t*>(at(L->keys0));
    b.pvals = reinterpret_cast<uint32_t*>(at(L->vals0));
    b.poff = reinterpret_cast<uint32_t*>(at(L->ekeys1));
    b.chunk_first = reinterpret_cast<uint32_t*>(at(L->emit_tmp));
    b.srt = reinterpret_cast<uint32_t*>(at(L->geo2d));
    b.counters = reinterpret_cast<Counters*>(at(L->counters));
    b.spin = spin;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t one = 1;   // chunk 0 is taken already, by nobody
    cudaError_t e = cudaMemcpyAsync(b.tickets + pairs, &one, 4, cudaMemcpyHostToDevice, st);
    return e != cudaSuccess ? e : pairs ? launch_emit(b, st) : launch_entries(b, st);
}
extern "C" long long scratch_bytes(long long n, int views) {
    return 8 * (gs::entry_scan_words(n, views) + gs::pair_scan_words(n, views)) + 4 * (2 * gs::kSortMaxBins + 2);
}
""")
    p.scratch_bytes.argtypes, p.scratch_bytes.restype = [C.c_longlong, C.c_int], C.c_longlong
    p.scan.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_int, C.c_int, C.c_void_p]
    return p


@pytest.mark.parametrize("spin", [1, 2000])
@pytest.mark.parametrize("pairs", [0, 1])
def test_a_wait_that_runs_out(probe, pairs, spin):
    n, cams = 60_000, [synth.camera(320, 240, 300.0)]
    planes = planes_of(synth.uniform_box_scene(73, n, sh_degree=0))
    ws = gs.Workspace(n, cams, gs.default_opts(), 300 * n)
    ws.project(planes, 0)
    ws.bin_sort()
    want = ws.counters()
    assert want.status == 0 and want.n_entries > 4096        # several chunks of either scan
    entries = ws.region("entries", torch.int32, want.n_entries).clone()
    tiles, vals = ws.sorted_pairs(want.n_pairs)
    tiles, vals = tiles.clone(), vals.clone()
    scratch = torch.zeros(probe.scratch_bytes(n, 1), dtype=torch.uint8, device="cuda")
    assert probe.scan(C.addressof(ws.layout), ws.buf.data_ptr(), 16, scratch.data_ptr(), pairs, spin,
                      torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert ws.counters().status == 4                         # GS_ERR_TIMEOUT
    ws.project(planes, 0)
    ws.bin_sort()
    c = ws.counters()
    assert c.status == 0 and c.n_entries == want.n_entries and c.n_pairs == want.n_pairs
    assert torch.equal(ws.region("entries", torch.int32, c.n_entries), entries)
    again = ws.sorted_pairs(c.n_pairs)
    assert torch.equal(again[0], tiles) and torch.equal(again[1], vals)
