"""Served batches above the size whose entries are checked one by one, with flagged requests small
enough to be settled beside the confirmation, too large for it, or cancelling so that the
confirmation fails: the clean requests' answers are published without waiting for the flagged
ones', and every answer is the C++ oracle's."""
import numpy as np
import pytest

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

D, N2 = 13, 4


def _request(seed, n, flips=(), pair=()):
    km = synth.key_material(seed, v=16)
    msgs = synth.messages(seed, n, 1, 24)
    s, R = X.sign_f(km.y, km.root, D, N2, km.bpv_r, synth.bpv_subsets(seed, n, v=16, k=4), msgs.data, msgs.offs, 0)
    data, s = np.array(msgs.data), np.array(s)
    for t in flips:
        data[int(msgs.offs[t])] ^= 4
    for t, delta in zip(pair, (777, -777)):
        v = (int.from_bytes(s[32 * t:32 * t + 32].tobytes(), "little") + delta) % O.Q
        s[32 * t:32 * t + 32] = np.frombuffer(v.to_bytes(32, "little"), np.uint8)
    Y, ds = X.base_mult(int.from_bytes(km.y, "little")), O.ds_serialize(O.ds_root(km.root, D))
    want = [int(t) for t in X.distill_f(Y, data, msgs.offs, 0, N2, s.tobytes(), np.array(R).tobytes(), ds)[0]]
    assert want == sorted(set(flips) | set(pair))
    return Y, (data, msgs.offs, s, np.array(R), ds), want


@pytest.mark.parametrize("flagged", [
    [(9_000, (0, 8_999), ()), (40, (7,), ())],
    [(17_000, (16_384,), ())],
    [(9_000, (), (5, 8_000))],
    [(9_000, (1,), ()), (8_000, (), (0, 7_999))],
], ids=["beside", "behind", "cancelling", "flipped and cancelling"])
def test_clean_requests_beside_flagged_ones(flagged):
    import __graft_entry__
    __graft_entry__.build()
    reqs = [_request(60 + i, n) for i, n in enumerate((300, 8_500, 1, 7_000))]
    reqs[2:2] = [_request(80 + i, *f) for i, f in enumerate(flagged)]
    with poslo.Context(device=0, verifier_seed=synth.verifier_seed(5)) as cx:
        cx.serve_start(workers=1)
        kid = [cx.register_key(Y) for Y, _, _ in reqs]
        largest = 0
        for _ in range(6):
            tickets = [cx.submit(k, N2, 0, *a) for k, (_, a, _) in zip(kid, reqs)]
            for t, (_, _, want) in reversed(list(zip(tickets, reqs))):
                accept, idx = cx.poll(t, wait_ms=60_000)
                assert (accept, [int(x) for x in idx]) == (not want, want)
            largest = max([largest] + [b["entries"] for b in cx.serve_timeline()])
        cx.serve_stop()
    assert largest > 16_384   # some batch took the weighted check
