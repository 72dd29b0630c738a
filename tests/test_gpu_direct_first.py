"""Small batches checked entry by entry at once: Distill and the many-signer call at the sizes
where the number of lanes per check, the path or the block's list handling changes, against the
C++ oracle: flips, malformed entries, every entry invalid, more invalid entries than the first
copy of the list holds, and a list longer than the caller's room."""
import numpy as np
import pytest

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

D, N2 = 12, 4


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = poslo.Context(device=0, verifier_seed=synth.verifier_seed(15))
    yield c
    c.close()


def _log(seed, n, first=0):
    km = synth.key_material(seed, v=16)
    msgs = synth.messages(seed, n, 1, 50)
    sub = synth.bpv_subsets(seed, n, v=16, k=4)
    s, R = X.sign_f(km.y, km.root, D, N2, km.bpv_r, sub, msgs.data, msgs.offs, first)
    return X.base_mult(int.from_bytes(km.y, "little")), msgs, s, R, O.ds_serialize(O.ds_root(km.root, D))


@pytest.mark.parametrize("n,flips", [(1, 0), (1, 1), (31, 31), (257, 3), (2048, 40), (2049, 0), (2049, 700),
                                     (4096, 4096), (4097, 5)])
def test_distill_at_the_edges(ctx, n, flips):
    Y, msgs, s, R, ds = _log(n, n, first=3)
    s, R = s.copy(), R.copy()
    bad = synth.apply_tamper(msgs, synth.tamper_plan(n, msgs, flips)) if flips else msgs
    if n > 200:
        s[32 * 7:32 * 8] = 0xFF                                            # not canonical
        R[32 * 11:32 * 12] = np.frombuffer((O.P + 1).to_bytes(32, "little"), np.uint8)   # does not decode
    want = X.distill_f(Y, bad.data, bad.offs, 3, N2, s.tobytes(), R.tobytes(), ds)
    b = ctx.make_batch(poslo.VARIANT_F, N2, Y, bad.data, bad.offs, s, R, ds, first_index=3)
    for _ in range(2):
        idx, cs, cR = ctx.distill(b)
        assert ([int(t) for t in idx], cs, cR) == want
    if len(want[0]) > 1:
        with pytest.raises(poslo.PosloError) as e:
            ctx.distill(b, cap=len(want[0]) - 1)
        assert e.value.code == poslo.POSLO_EBUFSMALL


@pytest.mark.parametrize("sizes,flips", [([1], 1), ([0, 3, 0, 40], 2), ([700, 1, 1347], 600), ([2049], 1),
                                         ([4000, 0, 97], 1), ([5000, 3192], 3), ([5000, 3193], 3)])
def test_many_signers_at_the_edges(ctx, sizes, flips):
    logs = [_log(50 + d, n, first=5 * d) if n else None for d, n in enumerate(sizes)]
    spare = _log(49, 1)
    keys = [x[0] if x else spare[0] for x in logs]
    stacks = [x[4] if x else spare[4] for x in logs]
    live = [x for x in logs if x]
    data = np.concatenate([x[1].data for x in live])
    lens = np.concatenate([(x[1].offs[1:] - x[1].offs[:-1]) for x in live])
    offs = np.zeros(len(lens) + 1, np.uint64)
    np.cumsum(lens, out=offs[1:])
    msgs = synth.Messages(data, offs)
    bad = synth.apply_tamper(msgs, synth.tamper_plan(3, msgs, flips))
    s, R = np.concatenate([x[2] for x in live]), np.concatenate([x[3] for x in live])
    want, start = [], 0
    for d, n in enumerate(sizes):
        if n:
            o = bad.offs[start:start + n + 1]
            got = X.distill_f(keys[d], bad.data[int(o[0]):int(o[-1])], o - o[0], 5 * d, N2,
                              s[32 * start:32 * (start + n)].tobytes(), R[32 * start:32 * (start + n)].tobytes(),
                              stacks[d])[0]
            want += [(d, t) for t in got]
        start += n
    args = (keys, sizes, [5 * d for d in range(len(sizes))], [N2] * len(sizes), stacks, bad.data, bad.offs, s, R)
    for _ in range(3):
        acc, pairs = ctx.aver_multi(*args)
        assert [(int(a), int(b)) for a, b in pairs] == want
        assert list(acc) == [all(d != w[0] for w in want) for d in range(len(sizes))]
    if len(want) > 1:
        with pytest.raises(poslo.PosloError) as e:
            ctx.aver_multi(*args, cap=1)
        assert e.value.code == poslo.POSLO_EBUFSMALL


@pytest.mark.parametrize("n,flips", [(8192, 0), (8192, 9), (8192, 8192), (8193, 9)])
def test_distill_at_the_upper_edge(ctx, n, flips):
    Y, msgs, s, R, ds = _log(n, n, first=3)
    bad = synth.apply_tamper(msgs, synth.tamper_plan(n, msgs, flips)) if flips else msgs
    want = X.distill_f(Y, bad.data, bad.offs, 3, N2, s.tobytes(), R.tobytes(), ds)
    b = ctx.make_batch(poslo.VARIANT_F, N2, Y, bad.data, bad.offs, s, R, ds, first_index=3)
    for _ in range(2):
        idx, cs, cR = ctx.distill(b)
        assert ([int(t) for t in idx], cs, cR) == want
