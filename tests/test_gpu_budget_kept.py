"""Memory budgets that are enough for POSLO-C Distill and SeBVer with very many umbrellas (measured as
the least accepted before their checks got workspaces of their own): the calls keep to them, and
give what they give without a budget."""
import numpy as np
import pytest
import torch

from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

# entries per epoch, epochs, umbrellas -> bytes for distill_c, and for SeBVer in its three modes
BUDGETS = [
    ((1, 4096, 1), 844_800, {"V": 411_392, "U": 411_392, "I": 525_056}),
    ((1, 4096, 4096), 1_106_944, {"V": 411_392, "U": 1_208_832, "I": 525_056}),
    ((4, 1000, 1), 358_912, {"V": 253_184, "U": 253_184, "I": 280_320}),
    ((4, 1000, 1000), 422_912, {"V": 253_184, "U": 446_976, "I": 280_320}),
    ((256, 64, 64), 634_112, {"V": 623_360, "U": 634_624, "I": 624_896}),
]


@pytest.mark.parametrize("shape,budget,seb", BUDGETS)
def test_ccd_within_its_budget(shape, budget, seb):
    import __graft_entry__
    __graft_entry__.build()
    n2, epochs, umbrellas = shape
    n, depth = n2 * epochs, max(1, (epochs - 1).bit_length()) + 1
    km = synth.key_material(77, v=16)
    msgs = synth.messages(77, n, 16, 64)

    def context(bytes_):
        cx = poslo.Context(device=0, mem_budget=bytes_)
        cx.set_key_cache(0)
        return cx

    with context(0) as cx:
        Y, epoch_R = cx.keygen_c(km.y, km.r, depth, n2)
        s = cx.sign_c(km.y, km.r, km.root, depth, n2, msgs.data, msgs.offs, 0, epochs)
        ds = cx.disclose(km.root, depth, epochs - 1)
        data = np.array(msgs.data)
        flipped = list(range(0, epochs, 7))
        for e in flipped:
            data[int(msgs.offs[n2 * e])] ^= 8
        dev = [torch.from_numpy(a).cuda() for a in (data, np.array(msgs.offs).view(np.int64), s,
                                                    np.array(epoch_R[:32 * epochs]))]
        b = cx.make_batch(poslo.VARIANT_C, n2, Y, dev[0], dev[1], dev[2], dev[3], ds)
        want = cx.distill_c(b, umbrellas)
        assert want[1]["invalid"] == flipped and want[0].count(False) == len(flipped)
    with context(budget) as cx:
        for _ in range(2):
            assert cx.distill_c(b, umbrellas) == want
    for mode, bytes_ in seb.items():
        with context(bytes_) as cx:
            assert cx.sebver_c(b, umbrellas, want[1], mode) == [mode != "I"] * len(
                {"V": [0], "U": want[1]["umbrellas"], "I": flipped}[mode])
