"""e_t at the edges of the hashing kernel's tiles (256 entries) and groups (one tile per group,
several groups per block in POSLO+, every group looping once the grid is full), both
instantiations, against the oracle's definition; lengths on both sides of the last class the
kernel sorts by (31 blocks)."""
import numpy as np
import pytest

from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

NAMES = {poslo.INST_SHA256: "POSLO", poslo.INST_AES: "POSLO+"}


@pytest.fixture(scope="module", params=[poslo.INST_SHA256, poslo.INST_AES])
def ctx(request):
    import __graft_entry__
    __graft_entry__.build()
    c = poslo.Context(device=0, instantiation=request.param)
    c.inst = request.param
    yield c
    c.close()


def _check(ctx, msgs, sample, first=3, n2=8):
    D = 5
    while (1 << D) * n2 < first + msgs.n:
        D += 1
    root = synth.random_bytes(31, "root", 16).tobytes()
    ds = O.ds_root(root, D)
    b = ctx.make_batch(poslo.VARIANT_F, n2, O.encode_point(O.G), msgs.data, msgs.offs, bytes(32 * msgs.n),
                       bytes(32 * msgs.n), O.ds_serialize(ds), first_index=first)
    e = ctx.hash_entries(b).reshape(-1, 32)
    with O.instantiation(NAMES[ctx.inst]):
        for t in sample:
            assert int.from_bytes(bytes(e[t]), "little") == O.entry_scalar(ds, n2, first + t, msgs.entry(t)), t


@pytest.mark.parametrize("n", [1, 127, 129, 256, 257, 1025])
def test_every_entry_at_tile_edges(ctx, n):
    _check(ctx, synth.messages(n, n, 0, 40), range(n))


def test_lengths_around_the_last_class(ctx):
    lens = [440, 463, 464, 479, 480, 481, 496, 1831, 1832, 1895, 1896, 1897, 2100, 0]
    entries = [synth.random_bytes(7, f"m{i}", L).tobytes() for i, L in enumerate(lens * 11)]
    _check(ctx, synth.pack(entries), range(len(entries)))


def test_groups_that_loop_over_tiles(ctx):
    n = 400_001   # more tiles than the 1,216 groups of the largest grid
    sample = [0, 255, 256, 155_647, 155_648, 311_295, 311_296, n - 2, n - 1]
    _check(ctx, synth.messages(9, n, 0, 24), sample)
