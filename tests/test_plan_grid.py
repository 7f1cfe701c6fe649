"""The grid of large counts (host only): 32-bit entry indices bound each catalogue, not their sum."""
import pytest

import paper_1911_08275_gb300 as cf

LIMIT = 2 ** 31 - 64


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n1,n2", [(1_080_000_000, 1_080_000_000), (100_000_000, 2_050_000_000),
                                   (2_050_000_000, 100_000_000), (2_000_000_000, None)])
def test_large_counts_keep_their_columns(n1, n2, periodic):
    # box / Rmax = 40 less the float32 margin, refine 4
    grid = cf.debug_grid(n1, n2, extent=(1000.0,) * 3, boxsize=1000.0, rmax=25.0, periodic=periodic)
    assert grid[:2] == (156, 156)


@pytest.mark.parametrize("n2", [None, 1000])
def test_padding_never_passes_the_index_range(n2):
    for n1 in (LIMIT - 10_000, LIMIT - 100_000, LIMIT - 10_000_000):
        ncx, ncy, _ = cf.debug_grid(n1, n2, boxsize=1000.0, rmax=2.0, refine=(4, 4, 1))
        assert (n1 + 31 * ncx * ncy + 31) // 32 * 32 <= LIMIT


def test_bad_arguments():
    for kw in (dict(n1=-1, rmax=1.0), dict(n1=5, n2=-2, rmax=1.0), dict(n1=5, rmax=0.0), dict(n1=5, rmax=float("inf"))):
        with pytest.raises(cf.CfError):
            cf.debug_grid(boxsize=10.0, **kw)
