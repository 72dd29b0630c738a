"""Field arithmetic at the edges of its 32-bit limbs, through the C ABI: points whose y has limbs
of all ones, all zeros or a single bit, or lies next to 0 and p, are decoded (255 squarings
each) and summed (unified additions of those coordinates), and the encoded sum is the oracle's."""
import numpy as np
import pytest

from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

LIMBS = (0, 1, 0x7FFFFFFF, 0x80000000, 0xFFFFFFDA, 0xFFFFFFFF)


def _candidates(kind):
    if kind == "near_zero":
        return list(range(2, 80))
    if kind == "near_p":
        return [O.P - k for k in range(2, 80)]
    if kind == "bits":
        return [1 << k for k in range(1, 255)] + [O.P - (1 << k) for k in range(1, 254)]
    w = synth.words(11, "limbs", 8 * 300)
    ys = [sum(LIMBS[int(w[8 * i + k] >> np.uint64(32)) % len(LIMBS)] << (32 * k) for k in range(8)) for i in range(300)]
    return [y & ((1 << 255) - 1) for y in ys]


def _points(kind):
    """Encodings with the candidates as y, both signs, that are points of the curve."""
    out = []
    for y in _candidates(kind):
        for sign in (0, 1):
            b = (y | sign << 255).to_bytes(32, "little")
            if y < O.P and O.decode_point(b) is not None:
                out.append(b)
    return out


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = poslo.Context(device=0)
    yield c
    c.close()


@pytest.mark.parametrize("kind", ["near_zero", "near_p", "bits", "limbs"])
def test_sums_of_points_at_limb_edges(ctx, kind):
    pts = _points(kind)
    # one sign of each, so that the sum does not cancel
    half = pts[::2]
    assert len(half) >= 20
    acc = O.IDENTITY
    for b in half:
        acc = O.point_add(acc, O.decode_point(b))
    _, got = ctx.agg(np.zeros(32 * len(half), np.uint8), b"".join(half))
    assert got == O.encode_point(acc)
    # every point alone keeps its encoding
    for b in half[:24]:
        assert ctx.agg(np.zeros(32, np.uint8), b)[1] == b
