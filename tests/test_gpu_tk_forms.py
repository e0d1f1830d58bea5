"""T_k (the FORS public key) in its two forms: by groups of 32 messages up to
7 groups per SM (34048 messages on 152 SMs; robust sets 5, 24320), above that
a thread per message.  A batch just past the line signs and verifies like its
messages in small batches, and like the oracle."""
import numpy as np
import pytest

from paper_2512_23969_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("ps,per_sm", [("toy", 7), ("192f", 7), ("shake-128f", 7), ("robust-128f", 5)])
def test_past_the_line(hs, O, ps, per_sm):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = per_sm * 32 * sms + 77                          # the last block is partly full
    wl = inputs.make(ps, count, num_keys=2, lengths=32, seed=410 + per_sm, key_mode="random")
    wl.key_idx[count - 5] = 2                                # an invalid key among them
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    m, l, k = _dev(wl.msgs), _dev(wl.lens), _dev(wl.key_idx)
    sigs = hs.hs_sign_batch(ps, sk, m, l, key_idx=k)
    ok = hs.hs_verify_batch(ps, pk, m, l, sigs, key_idx=k).cpu().numpy()
    hs.hs_check_status()
    assert ok[count - 5] == 0 and int(ok.sum()) == count - 1
    for at in (0, count // 2, count - 64):
        part = slice(at, at + 60)
        few = hs.hs_sign_batch(ps, sk, m[at * 32:(at + 60) * 32], l[part], key_idx=k[part])
        hs.hs_check_status()
        assert torch.equal(few, sigs[part])
    i = count - 1
    osk = O.keygen(ps, bytes(wl.seeds[wl.key_idx[i]]))[1]
    assert sigs[i].cpu().numpy().tobytes() == O.sign(ps, osk, wl.message(i))
