"""Many signers above the direct-check size: flagged signers of up to 16,384 entries together are
settled beside the confirmation, more behind it, and a confirmation that fails (errors that cancel
inside a signer's unit aggregate) settles every signer, against the C++ oracle."""
import numpy as np
import pytest

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

D, N2 = 13, 4


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = poslo.Context(device=0, verifier_seed=synth.verifier_seed(21))
    yield c
    c.close()


def _shift(s, t, delta):
    v = (int.from_bytes(s[32 * t:32 * t + 32].tobytes(), "little") + delta) % O.Q
    s[32 * t:32 * t + 32] = np.frombuffer(v.to_bytes(32, "little"), np.uint8)


# sizes; entries (of the whole batch) with a flipped byte; a pair of entries shifted by +-delta
@pytest.mark.parametrize("sizes,flips,pair", [
    ([9000, 500, 300], [], None),
    ([9000, 500, 300], [9100], None),
    ([9000, 0, 500], [4, 9499], None),
    ([8000, 8384, 5], [7999, 8000], None),
    ([8000, 8385, 5], [7999, 8000], None),
    ([9000, 500, 300], [9100], (17, 8000)),
    ([9000, 500, 300], [], (17, 8000)),
    ([16385, 500, 300], [], None),
    ([16385, 500, 300], [16500], None),
    ([16385, 500, 300], [16500], (17, 8000)),
    ([16385, 500, 300], [5, 17100], None),
    ([9000, 7384], [8999], None),
    ([9000, 7385], [8999], None),
])
def test_flagged_signers_beside_and_behind(ctx, sizes, flips, pair):
    data, lens, ss, Rs, keys, stacks = [], [], [], [], [], []
    for d, n in enumerate(sizes):
        km = synth.key_material(70 + d, v=16)
        msgs = synth.messages(70 + d, max(n, 1), 1, 40)
        keys.append(X.base_mult(int.from_bytes(km.y, "little")))
        stacks.append(O.ds_serialize(O.ds_root(km.root, D)))
        if n == 0:
            continue
        s, R = X.sign_f(km.y, km.root, D, N2, km.bpv_r, synth.bpv_subsets(70 + d, n, v=16, k=4), msgs.data, msgs.offs, 0)
        data.append(msgs.data), lens.append(msgs.offs[1:] - msgs.offs[:-1]), ss.append(s), Rs.append(R)
    data, s, R = np.concatenate(data), np.concatenate(ss), np.concatenate(Rs)
    offs = np.zeros(sum(sizes) + 1, np.uint64)
    np.cumsum(np.concatenate(lens), out=offs[1:])
    for t in flips:
        data[int(offs[t])] ^= 1
    if pair:
        _shift(s, pair[0], 12345)
        _shift(s, pair[1], -12345)
    start = np.concatenate([[0], np.cumsum(sizes)])
    bad = sorted(set(flips) | set(pair or ()))
    want = [(int(np.searchsorted(start, t, side="right")) - 1, t) for t in bad]
    want = [(d, int(t - start[d])) for d, t in want]
    for d, n in enumerate(sizes):   # the oracle says the same of every signer
        if n:
            lo, hi = int(start[d]), int(start[d + 1])
            o = offs[lo:hi + 1]
            got = X.distill_f(keys[d], data[int(o[0]):int(o[-1])], o - o[0], 0, N2, s[32 * lo:32 * hi].tobytes(),
                              R[32 * lo:32 * hi].tobytes(), stacks[d])[0]
            assert [int(t) for t in got] == [t for dd, t in want if dd == d]
    for _ in range(3):
        acc, pairs = ctx.aver_multi(keys, sizes, [0] * len(sizes), [N2] * len(sizes), stacks, data, offs, s, R)
        assert [(int(a), int(b)) for a, b in pairs] == want
        assert list(acc) == [all(d != w[0] for w in want) for d in range(len(sizes))]
