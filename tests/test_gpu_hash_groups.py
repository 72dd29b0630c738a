"""The hashing's groups where a batch has just more tiles than the chip has SMs, twice and four
times as many: e_t of entries on both sides of the places where the next tile goes to another
group of a block, both instantiations, alone (several groups a block in POSLO+) against the
oracle's definition, and beside the decoding through Distill of a signed log with flipped
entries."""
import numpy as np
import pytest

from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

NAMES = {poslo.INST_SHA256: "POSLO", poslo.INST_AES: "POSLO+"}
TILE, SMS = 256, 152
SIZES = [SMS * TILE + 1, 2 * SMS * TILE + 1, 4 * SMS * TILE + 1]


@pytest.fixture(scope="module", params=[poslo.INST_SHA256, poslo.INST_AES])
def ctx(request):
    import __graft_entry__
    __graft_entry__.build()
    c = poslo.Context(device=0, instantiation=request.param)
    c.inst = request.param
    yield c
    c.close()


def _edges(n):
    tiles = {0, 1, SMS - 1, SMS, 2 * SMS - 1, 2 * SMS, 4 * SMS - 1, 4 * SMS}
    return sorted({t for k in tiles for t in (TILE * k, TILE * k + 255) if t < n} | {n - 1})


@pytest.mark.parametrize("n", SIZES)
def test_hashes_where_the_groups_change(ctx, n):
    msgs = synth.messages(13, n, 0, 24)
    n2, d = 8, 15
    root = synth.random_bytes(33, "root", 16).tobytes()
    ds = O.ds_root(root, d)
    b = ctx.make_batch(poslo.VARIANT_F, n2, O.encode_point(O.G), msgs.data, msgs.offs, bytes(32 * n), bytes(32 * n),
                       O.ds_serialize(ds))
    e = ctx.hash_entries(b).reshape(-1, 32)
    with O.instantiation(NAMES[ctx.inst]):
        for t in _edges(n):
            assert int.from_bytes(bytes(e[t]), "little") == O.entry_scalar(ds, n2, t, msgs.entry(t)), t


@pytest.mark.parametrize("n", SIZES)
def test_distill_where_the_groups_change(ctx, n):
    n2, d = 256, 11
    km = synth.key_material(41, v=16)
    msgs = synth.messages(41, n, 1, 24)
    Y, bpv_R = ctx.keygen_f(km.y, km.bpv_r)
    s, R = ctx.sign_f(km.y, km.root, d, n2, km.bpv_r, bpv_R, synth.bpv_subsets(41, n, v=16, k=4), msgs.data, msgs.offs)
    flips = _edges(n)
    data = np.array(msgs.data)
    for t in flips:
        data[int(msgs.offs[t])] ^= 0x20
    ds = ctx.disclose(km.root, d, (n - 1) // n2)
    idx = ctx.distill(ctx.make_batch(poslo.VARIANT_F, n2, Y, data, msgs.offs, s, R, ds))[0]
    assert [int(t) for t in idx] == flips
