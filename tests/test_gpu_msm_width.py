"""The default window width on both sides of 2^19.5 entries: 127-bit weights change to 16 bits there,
full scalars do not."""
import pytest

from paper_2506_08781_gb300 import poslo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,words,width", [((1 << 19) - 1, 4, 13), (741_454, 4, 15), (741_455, 4, 16),
                                           ((1 << 20) - 1, 4, 16), (741_455, 8, 15)])
def test_default_width(n, words, width):
    import __graft_entry__
    __graft_entry__.build()
    with poslo.Context(device=0) as cx:
        assert cx.msm_get_plan(n, words)[0] == width
