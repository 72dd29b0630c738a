"""Many signers above the size whose entries are checked one by one: the combined weighted check with
the full weights and window by window, on the same device buffers with other contents each call, so
that the launch sequence captured from one call is replayed on the next ones' inputs: valid, flipped,
malformed and cancelling entries, against the C++ oracle.  Which path a call takes is read off the
kernel timers."""
import numpy as np
import pytest
import torch

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

D, N2 = 13, 4
SIZES = [9000, 0, 700, 6500, 185]   # 16,385 entries
START = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)


def _logs():
    data, lens, ss, Rs, keys, stacks = [], [], [], [], [], []
    for d, n in enumerate(SIZES):
        km = synth.key_material(90 + d, v=16)
        msgs = synth.messages(90 + d, max(n, 1), 1, 40)
        keys.append(X.base_mult(int.from_bytes(km.y, "little")))
        stacks.append(O.ds_serialize(O.ds_root(km.root, D)))
        if n:
            s, R = X.sign_f(km.y, km.root, D, N2, km.bpv_r, synth.bpv_subsets(90 + d, n, v=16, k=4), msgs.data,
                            msgs.offs, 0)
            data.append(msgs.data), lens.append(msgs.offs[1:] - msgs.offs[:-1]), ss.append(s), Rs.append(R)
    offs = np.zeros(sum(SIZES) + 1, np.uint64)
    np.cumsum(np.concatenate(lens), out=offs[1:])
    return keys, stacks, np.concatenate(data), offs, np.concatenate(ss), np.concatenate(Rs)


def _put(a, t, v):
    a[32 * t:32 * t + 32] = np.frombuffer(v.to_bytes(32, "little"), np.uint8)


def _scalar(s, t):
    return int.from_bytes(s[32 * t:32 * t + 32].tobytes(), "little")


def _contents(data, offs, s, R):
    """The inputs of each call and the batch positions that are invalid in it."""
    out = [((data, s, R), [])]
    f = data.copy()
    for t in (3, 9700 + 6499):
        f[int(offs[t])] ^= 1
    out.append(((f, s, R), [3, 16_199]))
    s2, R2 = s.copy(), R.copy()
    _put(s2, 9001, _scalar(s2, 9001) + O.Q)   # not canonical
    _put(R2, 16_384, O.P + 1)                 # not a point
    out.append(((data, s2, R2), [9001, 16_384]))
    s3 = s.copy()
    _put(s3, 17, (_scalar(s3, 17) + 12345) % O.Q)   # errors that cancel in the signer's unit sum
    _put(s3, 8000, (_scalar(s3, 8000) - 12345) % O.Q)
    out.append(((data, s3, R), [17, 8000]))
    return out + out[:2] + out[3:] + out[:1]


@pytest.mark.parametrize("limit", [0, 1 << 40])
def test_weighted_check_replayed_on_other_contents(limit):
    import __graft_entry__
    __graft_entry__.build()
    keys, stacks, data, offs, s, R = _logs()
    dev = [torch.from_numpy(np.array(a)).cuda() for a in (data, offs.view(np.int64), s, R)]
    args = (keys, SIZES, [0] * len(SIZES), [N2] * len(SIZES), stacks)
    with poslo.Context(device=0, verifier_seed=synth.verifier_seed(23)) as cx:
        cx.set_multi_window_limit(limit)
        calls = _contents(data, offs, s, R)
        for (m, si, Ri), bad in calls:
            for d, n in enumerate(SIZES):   # the oracle finds the same entries
                if n and any(START[d] <= t < START[d + 1] for t in bad):
                    lo, hi = int(START[d]), int(START[d + 1])
                    o = offs[lo:hi + 1]
                    got = X.distill_f(keys[d], m[int(o[0]):int(o[-1])], o - o[0], 0, N2, si[32 * lo:32 * hi].tobytes(),
                                      Ri[32 * lo:32 * hi].tobytes(), stacks[d])[0]
                    assert [int(t) + lo for t in got] == [t for t in bad if lo <= t < hi]
            for t, a in zip((dev[0], dev[2], dev[3]), (m, si, Ri)):
                t.copy_(torch.from_numpy(np.array(a)))
            torch.cuda.synchronize()
            acc, pairs = cx.aver_multi(*args, *dev)
            owner = [int(np.searchsorted(START, t, side="right")) - 1 for t in bad]
            assert [(int(a), int(b)) for a, b in pairs] == [(d, int(t - START[d])) for d, t in zip(owner, bad)]
            assert list(acc) == [d not in owner for d in range(len(SIZES))]
        # the first call builds the keys' tables, the second is the first of the shape that repeats,
        # the third is captured and the others replay it
        assert cx.graph_stats() == (1, len(calls) - 3)


@pytest.mark.parametrize("sizes,weighted", [([16_384, 0], False), ([16_384, 1], True)])
def test_which_check_a_batch_takes(sizes, weighted):
    import __graft_entry__
    __graft_entry__.build()
    km = synth.key_material(90, v=16)
    n = sum(sizes)
    msgs = synth.messages(90, n, 1, 8)
    s, R = X.sign_f(km.y, km.root, D, N2, km.bpv_r, synth.bpv_subsets(90, n, v=16, k=4), msgs.data, msgs.offs, 0)
    Y, ds = X.base_mult(int.from_bytes(km.y, "little")), O.ds_serialize(O.ds_root(km.root, D))
    with poslo.Context(device=0) as cx:
        cx.set_profiling(True)
        acc, pairs = cx.aver_multi([Y, Y], sizes, [0, sizes[0]], [N2, N2], [ds, ds], msgs.data, msgs.offs, s, R)
        assert list(acc) == [True, True] and len(pairs) == 0
        assert (cx.kernel_time("segment_sums")[1] > 0) == weighted
        assert (cx.kernel_time("localise")[1] > 0) == (not weighted)
