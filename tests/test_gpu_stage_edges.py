"""e_t where the hashing's copy of a tile's messages to shared memory starts and ends: tiles of empty
messages, of one byte, of exactly the bytes the copy takes (40,832) and of one byte more (read in
place), at every alignment of the first byte within 16, against the oracle's definition."""
import numpy as np
import pytest
import torch

from oracle import poslo_oracle as O
from paper_2506_08781_gb300 import poslo, synth

pytestmark = pytest.mark.gpu

D, N2, TILE = 6, 8, 256


def _even(total):
    """A tile's 256 lengths, as even as they come, that sum to `total`."""
    q, r = divmod(total, TILE)
    return [q + (k < r) for k in range(TILE)]


@pytest.mark.parametrize("lens", [[0] * TILE, [0] * 200 + [1] + [0] * 55, [0] * 300 + [7] * 3, _even(40_832),
                                  _even(40_833), [0] * TILE + _even(40_832)[::-1] + _even(40_833)],
                         ids=["empty", "one byte", "empty then some", "largest copied", "one more", "all three"])
def test_hashes_at_the_edges_of_the_copy(lens):
    import __graft_entry__
    __graft_entry__.build()
    n = len(lens)
    d = D
    while (N2 << d) < n:
        d += 1
    root = synth.random_bytes(31, "root", 16).tobytes()
    ds = O.ds_root(root, d)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    data = synth.random_bytes(7, "data", int(offs[-1]) + 16)
    sample = range(n) if offs[-1] < 100 else sorted({0, 1, 127, 128, 200, 255, n // 2, n - 2, n - 1})
    with poslo.Context(device=0) as cx:
        zeros = torch.zeros(32 * n, dtype=torch.uint8, device="cuda")
        d_offs = torch.from_numpy(offs.view(np.int64)).cuda()
        for shift in (0, 1, 2, 3, 5, 15):
            buf = torch.zeros(len(data) + 32, dtype=torch.uint8, device="cuda")
            buf[shift:shift + len(data)] = torch.from_numpy(np.array(data)).cuda()
            b = cx.make_batch(poslo.VARIANT_F, N2, O.encode_point(O.G), buf[shift:], d_offs, zeros, zeros,
                              O.ds_serialize(ds))
            out = torch.empty(32 * n, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            cx.hash_entries(b, out)
            e = out.cpu().numpy().reshape(-1, 32)
            for t in sample:
                m = bytes(data[int(offs[t]):int(offs[t + 1])])
                assert int.from_bytes(bytes(e[t]), "little") == O.entry_scalar(ds, N2, t, m), (shift, t)
