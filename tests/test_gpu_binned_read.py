"""Large batches of reads from large arrays go through bins (2^25 reads and
more): random, ascending, windowed and mixed batches, indices out of range,
a batch that ends inside a tile, arrays with empty LFVectors and arrays the
L2 holds, several streams at once, and a stream being captured (which reads
directly), against indexing the flattened array."""

import pytest
import torch

from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

N_READS = (1 << 25) + 1234


def grown(E, elements, slab, L=700):
    """An array of about `elements` self-describing elements; every seventh LFVector is empty."""
    g = gga.GGArray(L, 256, 1024, E, slab)
    counts = torch.zeros((1, L, 256), dtype=torch.int32, device="cuda")
    per = elements // L // 256
    counts[0] = (torch.arange(L * 256, device="cuda") % 3 + per - 1).reshape(L, 256).int()
    counts[0, ::7] = 0
    n = int(counts.sum().item())
    values = wl.encode_values_t(wl.splitmix_at_t(3, torch.arange(n, device="cuda")), E)
    g.insert(counts, values)
    assert g.size() == (n, gga.GGA_OK)
    return g, n


def batch(kind, n):
    i = torch.arange(N_READS, device="cuda")
    idx = wl.uniform_indices_t(5, N_READS, n, "cuda")
    if kind == "ascending":
        idx = idx.sort().values
    elif kind == "window":
        idx = (i * (n - (1 << 16)) // N_READS + idx % (1 << 16)).contiguous()
    elif kind == "mixed":
        idx = torch.where((i // 5000) % 2 == 0, idx, idx.sort().values)
    return idx


def same(got, flat, idx):
    for a in range(0, N_READS, 1 << 24):
        b = min(N_READS, a + (1 << 24))
        assert torch.equal(got[a:b], flat[idx[a:b]])


@pytest.mark.parametrize("E", [4, 8])
@pytest.mark.parametrize("kind", ["uniform", "ascending", "window", "mixed"])
def test_reads_equal_the_flattened_array(E, kind):
    g, n = grown(E, (300 << 20) // E, 600 << 20)
    flat = g.flatten()
    idx = batch(kind, n)
    same(g.read(idx), flat, idx)
    assert g.last_error() == gga.GGA_OK
    g.close()


def test_indices_out_of_range_read_zero_and_latch():
    g, n = grown(4, 75 << 20, 600 << 20)
    flat = g.flatten()
    idx = batch("uniform", n)
    bad = torch.zeros(N_READS, dtype=torch.bool, device="cuda")
    bad[::1001] = True
    bad[4096 * 3:4096 * 4] = True                      # a whole tile
    idx[bad] = idx[bad] + n
    idx[7] = -1                                        # 2^64 - 1
    bad[7] = True
    got = g.read(idx)
    assert g.last_error() == gga.GGA_ERR_OUT_OF_RANGE
    assert int(got[bad].abs().max()) == 0
    assert torch.equal(got[~bad], flat[idx[~bad]])
    g.close()


@pytest.mark.parametrize("E", [4, 8])
@pytest.mark.parametrize("kind", ["all", "tiles", "all but one"])
def test_tiles_with_no_index_in_range_read_zero(E, kind):
    """Scattered indices out of range, with no scattered tile beside them
    that holds a valid one ("all but one": a single index of the batch)."""
    g, n = grown(E, (300 << 20) // E, 600 << 20)
    flat = g.flatten()
    beyond = batch("uniform", n) + n
    idx, bad = beyond, torch.ones(N_READS, dtype=torch.bool, device="cuda")
    if kind == "tiles":
        idx, bad = batch("ascending", n), ~bad
        for tile in (0, 777, N_READS // 4096):        # the last one ends with the batch
            bad[4096 * tile:4096 * (tile + 1)] = True
        idx = torch.where(bad, beyond, idx)
    elif kind == "all but one":
        idx[N_READS // 2], bad[N_READS // 2] = n - 1, False
    out = gga.elem_tensor(N_READS, E).fill_(-7)
    g.read(idx, out)
    assert g.last_error() == gga.GGA_ERR_OUT_OF_RANGE
    assert int(out[bad].abs().max()) == 0
    assert torch.equal(out[~bad], flat[idx[~bad]])
    g.close()


def test_small_and_empty_arrays_in_a_large_slab():
    g, n = grown(4, 5 << 20, 600 << 20)                # the L2 holds it
    flat = g.flatten()
    idx = batch("uniform", n)
    same(g.read(idx), flat, idx)
    g.clear()
    assert int(g.read(idx).abs().max()) == 0
    assert g.last_error() == gga.GGA_ERR_OUT_OF_RANGE
    g.close()


def test_streams_at_once_and_capture():
    g, n = grown(8, 40 << 20, 600 << 20)
    flat = g.flatten()
    batches = [batch("uniform", n), batch("mixed", n)]
    outs = [torch.empty(N_READS, dtype=torch.int64, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(4)]
    for rep in range(3):
        for k, s in enumerate(streams):
            with torch.cuda.stream(s):
                g.read(batches[k % 2], outs[k])
    torch.cuda.synchronize()
    for k in range(4):
        same(outs[k], flat, batches[k % 2])
    out = torch.zeros(N_READS, dtype=torch.int64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.read(batches[0], out)
    graph.replay()
    torch.cuda.synchronize()
    same(out, flat, batches[0])
    g.close()
