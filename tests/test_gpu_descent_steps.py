"""Distill's descent at sizes whose tree has an odd and an even number of levels, with so few
failing entries that a step jumps many levels, with so many that it takes the least (two), and with
the last step left a single level, against the C++ oracle."""
import numpy as np
import pytest

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16_385, 33_000])
@pytest.mark.parametrize("share", [0, 3, 40, 500])   # 1 / share of the entries flipped; 0: one entry
def test_steps_of_the_descent(n, share):
    import __graft_entry__
    __graft_entry__.build()
    D, n2 = 14, 4
    km = synth.key_material(31, v=16)
    msgs = synth.messages(31, n, 1, 20)
    s, R = X.sign_f(km.y, km.root, D, n2, km.bpv_r, synth.bpv_subsets(31, n, v=16, k=4), msgs.data, msgs.offs, 0)
    Y = X.base_mult(int.from_bytes(km.y, "little"))
    ds = O.ds_serialize(O.ds_root(km.root, D))
    bad = synth.apply_tamper(msgs, synth.tamper_plan(31, msgs, n // share if share else 1))
    want = X.distill_f(Y, bad.data, bad.offs, 0, n2, s.tobytes(), R.tobytes(), ds)
    with poslo.Context(device=0, verifier_seed=synth.verifier_seed(8)) as cx:
        b = cx.make_batch(poslo.VARIANT_F, n2, Y, bad.data, bad.offs, s, R, ds)
        idx, cs, cR = cx.distill(b)
        assert ([int(t) for t in idx], cs, cR) == want
