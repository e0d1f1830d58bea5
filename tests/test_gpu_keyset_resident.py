"""Keysets whose resident keys are many (the scratch of a call holds none of
their key blocks), and keysets without prebuilt layers, whose calls build the
trees that several messages share in their own scratch.  Signatures are
byte-identical to hs_sign_batch's without sharing, and to the oracle's."""
import numpy as np
import pytest

from paper_2512_23969_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("ps,count,layers", [("128f", 1, 1), ("128f", 300, 2), ("256f", 5, 1)])
def test_many_keys_pageable_host_buffers(hs, ps, count, layers):
    wl = inputs.make(ps, count, num_keys=1000, lengths=("uniform", 0, 200), seed=310 + count, key_mode="random")
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    ref = hs.hs_sign_batch(ps, sk, _dev(wl.msgs), _dev(wl.lens), key_idx=_dev(wl.key_idx), num_keys=1000).cpu().numpy()
    with hs.KeySet(ps, sk, cache_layers=layers) as ks:
        got = np.asarray(ks.sign(wl.msgs, wl.lens, key_idx=wl.key_idx))      # staged behind the scratch
    assert np.array_equal(got, ref)


# both TREE_Sign forms (chain-parallel, per leaf), trees of one warp and wide
# ones, one and two shared layers, and a batch too small to share any
@pytest.mark.parametrize("ps,count,keys", [("128f", 40, 2), ("128f", 3, 2), ("192f", 70, 3), ("256f", 70, 1), ("128s", 6, 2),
                                           ("256s", 5, 2), ("shake-128f", 40, 2), ("robust-128f", 40, 2), ("toy", 50, 3)])
def test_no_cached_layers(hs, O, ps, count, keys):
    import torch
    from paper_2512_23969_gb300 import autotune
    wl = inputs.make(ps, count, num_keys=keys, lengths=("uniform", 0, 200), seed=330 + count, key_mode="random")
    wl.key_idx[1] = keys                                     # an invalid key among them
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    m, l, k = _dev(wl.msgs), _dev(wl.lens), _dev(wl.key_idx)
    saved = autotune.get(ps, "tree_split_below")
    try:
        hs.hs_set_tree_sharing(False)
        ref = hs.hs_sign_batch(ps, sk, m, l, key_idx=k, num_keys=keys).cpu()
        hs.hs_set_tree_sharing(True)
        for ck in (2, 0):
            hs.hs_set_chain_checkpoint(ck)
            with hs.KeySet(ps, sk) as ks:
                for split in (0, 1 << 20):
                    autotune.set(ps, "tree_split_below", split)
                    assert torch.equal(ks.sign(m, l, key_idx=k).cpu(), ref), (ck, split)
    finally:
        hs.hs_set_tree_sharing(True)
        hs.hs_set_chain_checkpoint(2)
        autotune.set(ps, "tree_split_below", saved)
        hs.hs_check_status()
    osk = [O.keygen(ps, bytes(s))[1] for s in wl.seeds]
    for i in (0, count - 1):
        assert ref[i].numpy().tobytes() == O.sign(ps, osk[wl.key_idx[i]], wl.message(i))
