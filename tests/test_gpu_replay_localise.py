"""Distill of a tampered device-resident batch above the direct-check size, called several times
with the same buffers: the first stage is captured on the second call and replayed afterwards,
and the localisation behind it (launched outside the graph) gives the same result each time."""
import numpy as np
import pytest
import torch

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 16_400])
def test_localisation_behind_a_replayed_first_stage(n):
    import __graft_entry__
    __graft_entry__.build()
    D, n2 = 13, 4
    km = synth.key_material(5, v=16)
    msgs = synth.messages(5, n, 1, 40)
    s, R = X.sign_f(km.y, km.root, D, n2, km.bpv_r, synth.bpv_subsets(5, n, v=16, k=4), msgs.data, msgs.offs, 0)
    Y = X.base_mult(int.from_bytes(km.y, "little"))
    ds = O.ds_serialize(O.ds_root(km.root, D))
    plan = synth.tamper_plan(5, msgs, 3)
    bad = synth.apply_tamper(msgs, plan)
    want = X.distill_f(Y, bad.data, bad.offs, 0, n2, s.tobytes(), R.tobytes(), ds)
    dev = [torch.from_numpy(np.array(a)).cuda() for a in (bad.data, bad.offs.view(np.int64), s, R)]
    with poslo.Context(device=0, verifier_seed=synth.verifier_seed(6)) as cx:
        b = cx.make_batch(poslo.VARIANT_F, n2, Y, dev[0], dev[1], dev[2], dev[3], ds)
        for _ in range(6):
            idx, cs, cR = cx.distill(b)
            assert ([int(t) for t in idx], cs, cR) == want
        assert cx.graph_stats()[1] >= 2
        # a valid batch in the same buffers replays the same graph
        dev[0].copy_(torch.from_numpy(np.array(msgs.data)))
        idx, cs, cR = cx.distill(b)
        assert len(idx) == 0 and (cs, cR) == X.distill_f(Y, msgs.data, msgs.offs, 0, n2, s.tobytes(), R.tobytes(), ds)[1:]
