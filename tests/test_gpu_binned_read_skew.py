"""Large batches of reads whose indices meet in a small part of a large array --
a few elements, hot pieces scattered over it, one place -- are read directly,
also with indices out of range among them: against indexing the flattened
array; and what they cost beside uniform indices."""

import pytest
import torch

from paper_2209_00103_gb300 import gga

from test_gpu_binned_read import N_READS, grown, same
from test_gpu_count_means import COEFFS, microseconds

pytestmark = pytest.mark.gpu


def power_law(n, s, count=N_READS):
    """Ranks 0, 1, ... with probability about (rank + 1)^-s."""
    torch.manual_seed(3)
    u = torch.rand(count, device="cuda", dtype=torch.float64)
    return (((1 - u) * (float(n) ** (1 - s) - 1) + 1) ** (1 / (1 - s))).long().clamp_(1, n) - 1


def indices(kind, n, E, count=N_READS):
    torch.manual_seed(4)
    u = torch.rand(count, device="cuda", dtype=torch.float64)
    if kind == "few":
        return power_law(n, 1.3, count)
    if kind == "few, scattered":
        return (power_law(n, 1.3, count) * 2654435761) % n
    if kind == "pieces":                              # 256 pieces of 64 KB
        hot, piece = (16 << 20) // E, (64 << 10) // E
        k = (u * hot).long()
        return (k // piece) * (n // 256) + k % piece
    if kind == "one place":
        return (n / 2 + torch.randn(count, device="cuda", dtype=torch.float64) * n * 0.03).long().clamp_(0, n - 1)
    return (u * n).long()


@pytest.mark.parametrize("E", [4, 8])
@pytest.mark.parametrize("kind", ["few", "few, scattered", "pieces", "one place", "uniform"])
def test_reads_equal_the_flattened_array(E, kind):
    g, n = grown(E, (400 << 20) // E, 900 << 20)
    flat = g.flatten()
    idx = indices(kind, n, E)
    same(g.read(idx), flat, idx)
    assert g.last_error() == gga.GGA_OK
    bad = torch.zeros(N_READS, dtype=torch.bool, device="cuda")
    bad[::977] = True
    bad[4096 * 9:4096 * 10] = True
    far = torch.where(bad, idx + n, idx)
    out = gga.elem_tensor(N_READS, E).fill_(-7)
    g.read(far, out)
    assert g.last_error() == gga.GGA_ERR_OUT_OF_RANGE
    assert int(out[bad].abs().max()) == 0
    assert torch.equal(out[~bad], flat[idx[~bad]])
    g.close()


def test_skewed_reads_cost_less_than_uniform_ones():
    """2^26 reads of 0.96 GB: grouped by ranges all the same, the reads of a few
    neighbouring elements took three times as long as uniform ones, those of hot
    pieces as long."""
    E, count = 4, 1 << 26
    g = gga.GGArray(1024, 512, 4096, E, int(1.1 * (1 << 30)))
    g.insert_generated(gga.make_gen_spec(5, "uniform3", COEFFS), 490)
    n, rc = g.size()
    assert rc == gga.GGA_OK
    out = gga.elem_tensor(count, E)

    def read(kind):
        idx = indices(kind, n, E, count)
        return microseconds(lambda: g.read(idx, out))

    uniform = read("uniform")
    assert read("few") < 0.9 * uniform
    assert read("pieces") < 0.9 * uniform
    assert g.last_error() == gga.GGA_OK
    g.close()
    # LFVectors of uneven sizes: a search per read, which the grouping shortens.
    g, n = grown(E, (960 << 20) // E, int(2.2 * (1 << 30)))
    uniform = read("uniform")
    assert read("few") < 0.9 * uniform
    assert read("pieces") < 1.1 * uniform
    g.close()
