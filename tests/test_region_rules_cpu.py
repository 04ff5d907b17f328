"""Which domains the region launches serve: the rule alone, without a GPU."""
import pytest

WIDEST = 1 << 23  # elements per row; the pitch is a caller's (a multiple of 32)


@pytest.mark.parametrize("rows", [2, 4, 8])
@pytest.mark.parametrize("warps", [4, 16])
def test_pitch_fits_32_bit_offsets(rows, warps):
    """A region's offsets are 32-bit products of a row count and the pitch, so
    a wide pitch leaves the domain to the single-step kernel."""
    from . import regions

    def t(pitch):
        return regions.tiles(regions.shape(100, 90, pitch=pitch), rows, warps, 1)

    for pitch in (128, 1 << 20, WIDEST):
        g = t(pitch)
        assert g.rows == rows and g.gx > 0 and g.gy > 0
        # the rows of a region and one to either side, from any column
        assert (rows * warps + 2) * pitch + 64 < 1 << 32
    for pitch in (WIDEST + 32, 1 << 25, 1 << 26, 1 << 27, 1 << 32, 1 << 40):
        assert t(pitch).rows == 0
    # a context's pitch follows its width
    assert regions.tiles(regions.shape(WIDEST, 90), rows, warps, 1).rows == rows
    assert regions.tiles(regions.shape(WIDEST + 1, 90), rows, warps, 1).rows == 0
