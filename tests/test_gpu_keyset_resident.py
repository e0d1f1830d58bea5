"""Keysets whose resident keys are many: the scratch of a call holds none of
their key blocks.  Signatures are byte-identical to hs_sign_batch's."""
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
