"""Device memory of an FP32 context: tables of the flat launch only where the lattice can take it.

(Host only.)  Besides the populations, the density history and the step tilings' tables, a lattice of
thousands of tiles per SM reserves nothing for the flat launch, and a small one no more than its tiles:
at most 3 rounds of 2 CTAs on 152 SMs, each a table entry and a cache line.
"""
import pytest

from paper_2009_05264_gb300 import lbm

FLAT_TILE, LINE = 160, 128  # no less than the entry's size; a done count's line


def rest(nx, ny):
    """Bytes besides populations, history and the step tilings' tables (two entries and a count a tile)."""
    pitch = -(-nx // 32) * 32
    tiles = -(-nx // 56) * -(-ny // 4)
    return lbm.load().lbm_required_bytes(nx, ny, lbm.FP32) - pitch * ny * 4 * 37 - tiles * (2 * 32 + 8)


FIXED = 1024 * 12 * 8 + 16384  # diagnostics ring; descriptors, state, alignment


@pytest.mark.parametrize("nx,ny", [(4000, 400), (8000, 800), (3000, 300), (20000, 64)])
def test_large_lattices_reserve_nothing_for_it(nx, ny):
    assert rest(nx, ny) <= FIXED


@pytest.mark.parametrize("nx,ny", [(130, 20), (1000, 100), (600, 80), (1800, 160), (60, 4)])
def test_small_lattices_reserve_their_tiles(nx, ny):
    strips = -(-nx // 60) + 1
    tiles = min(912, strips * -(-ny // 4))
    assert 0 < rest(nx, ny) <= FIXED + 4096 + tiles * (FLAT_TILE + LINE)
