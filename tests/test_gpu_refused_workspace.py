"""A workspace that the memory budget refuses in the middle of a call, while other streams work on
the caller's arrays: Distill's confirmation of more than 4,096 flagged entries, and the entry
checks of flagged signers beside their confirmation.  The call fails with ENOMEM and has nothing
running when it returns, so the caller may overwrite its arrays, and the next call on the same
context gives the oracle's answer."""
import numpy as np
import pytest
import torch

from oracle import cpp_oracle as X
from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

D, N2 = 13, 4
ENOMEM = -2


class Log:
    """A signer's log of n entries, `flips` of them with a flipped byte, on the device."""

    def __init__(self, seed, n, flips):
        km = synth.key_material(seed, v=16)
        msgs = synth.messages(seed, n, 1, 20)
        s, R = X.sign_f(km.y, km.root, D, N2, km.bpv_r, synth.bpv_subsets(seed, n, v=16, k=4), msgs.data, msgs.offs, 0)
        bad = synth.apply_tamper(msgs, synth.tamper_plan(seed, msgs, flips)) if flips else msgs
        self.Y = X.base_mult(int.from_bytes(km.y, "little"))
        self.ds = O.ds_serialize(O.ds_root(km.root, D))
        self.data, self.offs, self.s, self.R, self.n = np.array(bad.data), np.array(bad.offs), np.array(s), np.array(R), n
        self.want = X.distill_f(self.Y, bad.data, bad.offs, 0, N2, s.tobytes(), R.tobytes(), self.ds)


def _device(*arrays):
    return [torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).cuda() for a in arrays]


def _budget_refusing(workspace, call):
    """A memory budget at which call(context) is refused `workspace` and nothing before it."""
    lo, hi = 0, 1 << 28   # at lo an earlier workspace (or the context) is refused, at hi none
    seen = []
    for _ in range(28):
        mid = (lo + hi) // 2
        cx = _context(mid)
        try:
            call(cx)
            hi = mid
        except poslo.PosloError as e:
            assert e.code == ENOMEM, e
            name = str(e).split("'")[1]
            if name == workspace:
                return mid
            if name not in seen:
                seen.append(name)
            if name in AFTER[workspace]:
                hi = mid
            else:
                lo = mid
        finally:
            cx.close()
    raise AssertionError(f"no budget refuses {workspace} first; refused: {seen}")


# the workspaces that are asked for after the one sought
AFTER = {"confirm_gpts": {"confirm_gz", "confirm_gskip"}, "m_idx": {"flag_cnt", "flag_off"}}


def _context(budget):
    cx = poslo.Context(device=0, verifier_seed=synth.verifier_seed(4), mem_budget=budget)
    cx.set_key_cache(0)
    return cx


def test_distill_refused_its_confirmation():
    import __graft_entry__
    __graft_entry__.build()
    many, few = Log(3, 20_000, 5_000), Log(4, 9_000, 7)
    d = _device(many.data, many.offs, many.s, many.R)
    batch = poslo.Context.make_batch(poslo.VARIANT_F, N2, many.Y, *d, many.ds)
    budget = _budget_refusing("confirm_gpts", lambda cx: cx.distill(batch))
    other = poslo.Context.make_batch(poslo.VARIANT_F, N2, few.Y, *_device(few.data, few.offs, few.s, few.R), few.ds)
    with _context(budget) as cx:
        for _ in range(4):
            with pytest.raises(poslo.PosloError) as e:
                cx.distill(batch)
            assert e.value.code == ENOMEM
            for a in d[2:]:
                a.zero_()   # nothing reads the caller's signatures any more
            idx, cs, cR = cx.distill(other)
            assert ([int(t) for t in idx], cs, cR) == few.want
            torch.cuda.synchronize()
            for a, h in zip(d[2:], (many.s, many.R)):
                a.copy_(torch.from_numpy(h))
            torch.cuda.synchronize()
    with _context(0) as cx:
        idx, cs, cR = cx.distill(batch)
        assert ([int(t) for t in idx], cs, cR) == many.want


def test_many_signers_refused_their_localisation():
    import __graft_entry__
    __graft_entry__.build()
    logs = [Log(11, 9_000, 0), Log(12, 9_000, 3), Log(13, 400, 0)]
    offs = [np.uint64(0) * logs[0].offs[:1]]
    for g in logs:
        offs.append(g.offs[1:] + offs[-1][-1])
    data, offs = np.concatenate([g.data[:int(g.offs[-1])] for g in logs]), np.concatenate(offs)
    s, R = np.concatenate([g.s for g in logs]), np.concatenate([g.R for g in logs])
    d = _device(data, offs, s, R)
    args = ([g.Y for g in logs], [g.n for g in logs], [0] * 3, [N2] * 3, [g.ds for g in logs])
    budget = _budget_refusing("m_idx", lambda cx: cx.aver_multi(*args, *d))
    small = logs[2]
    with _context(budget) as cx:
        for _ in range(4):
            with pytest.raises(poslo.PosloError) as e:
                cx.aver_multi(*args, *d)
            assert e.value.code == ENOMEM
            for a in d[2:]:
                a.zero_()
            b = cx.make_batch(poslo.VARIANT_F, N2, small.Y, small.data, small.offs, small.s, small.R, small.ds)
            idx, cs, cR = cx.distill(b)
            assert ([int(t) for t in idx], cs, cR) == small.want
            torch.cuda.synchronize()
            for a, h in zip(d[2:], (s, R)):
                a.copy_(torch.from_numpy(h))
            torch.cuda.synchronize()
    with _context(0) as cx:
        acc, pairs = cx.aver_multi(*args, *d)
        assert list(acc) == [True, False, True]
        assert [(int(a), int(b)) for a, b in pairs] == [(1, t) for t in logs[1].want[0]]
