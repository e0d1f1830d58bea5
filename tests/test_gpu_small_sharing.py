"""Small batches with the library's default, repeated trees built once per
batch, and without it, whatever an earlier test left the switch at: sizes
where shared and own trees go through the same launches with FORS_Sign beside
them, against the oracle."""
import numpy as np
import pytest

from paper_2512_23969_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


# two keys: shared from 4 messages on; FORS a thread per leaf up to 27 messages
# at 192f and 17 at 256f (152 SMs)
@pytest.mark.parametrize("sharing", [True, False])
@pytest.mark.parametrize("ps,count", [("128f", 3), ("128f", 4), ("128f", 5), ("192f", 27), ("192f", 28), ("256f", 17), ("256f", 18),
                                      ("robust-128f", 9), ("shake-192f", 5), ("192s", 4), ("toy", 9)])
def test_sign_small(hs, O, ps, count, sharing):
    wl = inputs.make(ps, count, num_keys=2, lengths=("uniform", 0, 200), seed=720 + count, key_mode="random")
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    try:
        hs.hs_set_tree_sharing(sharing)
        got = hs.hs_sign_batch(ps, sk, _dev(wl.msgs), _dev(wl.lens), key_idx=_dev(wl.key_idx)).cpu().numpy()
    finally:
        hs.hs_set_tree_sharing(True)
    osk = [O.keygen(ps, bytes(s))[1] for s in wl.seeds]
    for i in sorted({0, count // 2, count - 1}):
        assert got[i].tobytes() == O.sign(ps, osk[wl.key_idx[i]], wl.message(i)), i
