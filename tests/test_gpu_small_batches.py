"""Batches at the lines between the kernels' forms: signing around the sizes
where FORS_Sign, TREE_Sign and tree sharing change form, key generation in
both of its forms, and verification around the line between the walk over
the layers and the layer-by-layer form.  Signatures and keys are compared
byte for byte with the oracle, and with the other form where the library can
be told to take it; verification has to accept every signature and reject
every one with a flipped bit in any of its parts."""
import numpy as np
import pytest

from paper_2512_23969_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _sign(hs, ps, sk, wl):
    import torch
    s = hs.hs_sign_batch(ps, sk, _dev(wl.msgs), _dev(wl.lens), key_idx=_dev(wl.key_idx), num_keys=wl.num_keys)
    torch.cuda.synchronize()
    return s.cpu()


# a tree group holds 4 trees at 128f / 192f, 2 at 256f; FORS a thread per leaf
# up to 17 messages at 256f, 27 at 192f (152 SMs)
@pytest.mark.parametrize("ps,count", [("128f", 1), ("128f", 2), ("128f", 3), ("128f", 5), ("192f", 1), ("192f", 27), ("192f", 28), ("256f", 1),
                                      ("256f", 17), ("256f", 18), ("robust-128f", 2), ("shake-192f", 3),
                                      ("192s", 1), ("toy", 9)])
def test_sign_small(hs, O, ps, count):
    wl = inputs.make(ps, count, num_keys=2, lengths=("uniform", 0, 200), seed=700 + count, key_mode="random")
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    got = _sign(hs, ps, sk, wl)
    osk = [O.keygen(ps, bytes(s))[1] for s in wl.seeds]
    for i in sorted({0, count // 2, count - 1}):
        assert got[i].numpy().tobytes() == O.sign(ps, osk[wl.key_idx[i]], wl.message(i)), i


# the top layer holds one tree per key: shared from 2 * keys messages on
@pytest.mark.parametrize("ps,count,keys", [("128f", 31, 16), ("128f", 32, 16), ("128f", 33, 16), ("256f", 65, 2),
                                           ("128s", 4, 2), ("toy", 8, 1)])
def test_sharing_line(hs, ps, count, keys):
    import torch
    wl = inputs.make(ps, count, num_keys=keys, lengths=32, seed=900 + count, key_mode="random")
    wl.key_idx[1] = keys + 3                              # an invalid key among them
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    try:
        hs.hs_set_tree_sharing(True)
        on = _sign(hs, ps, sk, wl)
        hs.hs_set_tree_sharing(False)
        off = _sign(hs, ps, sk, wl)
    finally:
        hs.hs_set_tree_sharing(True)
        hs.hs_check_status()
    assert torch.equal(on, off)
    assert int(on[1].sum()) == 0 and int(on[0].sum()) != 0


@pytest.mark.parametrize("ps,count", [("128f", 1), ("128f", 34), ("128f", 35), ("192f", 4), ("256f", 3), ("128s", 1), ("256s", 2),
                                      ("shake-128f", 5), ("robust-192f", 3), ("toy", 9)])
def test_keygen_forms(hs, O, ps, count):
    import torch
    from paper_2512_23969_gb300 import autotune
    wl = inputs.make(ps, 1, num_keys=count, seed=40 + count)
    saved = autotune.get(ps, "tree_step_us"), autotune.get(ps, "tree_split_ns")
    try:
        out = []
        for step, ns in ((0, 0), (1 << 20, 1)):           # a thread per leaf; chain-parallel
            autotune.set(ps, "tree_step_us", step)
            autotune.set(ps, "tree_split_ns", ns)
            pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
            torch.cuda.synchronize()
            out.append((pk.cpu(), sk.cpu()))
    finally:
        autotune.set(ps, "tree_step_us", saved[0])
        autotune.set(ps, "tree_split_ns", saved[1])
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    for k in {0, count - 1}:
        opk, osk = O.keygen(ps, bytes(wl.seeds[k]))
        assert out[1][0][k].numpy().tobytes() == opk and out[1][1][k].numpy().tobytes() == osk


# the walk takes 3500 (SHAKE: 3000) chains a layer: 100 signatures at n = 16
# (SHAKE 85), 68 at n = 24, 52 at n = 32; 32 signatures to a block; above 5
# groups of 32 signatures per SM (24320 on 152) T_len runs a thread per item
@pytest.mark.parametrize("ps,count", [("128f", 1), ("128f", 33), ("128f", 100), ("128f", 101), ("192f", 68),
                                      ("256f", 52), ("256f", 53), ("shake-128f", 85), ("shake-256f", 2),
                                      ("robust-128f", 34), ("128s", 3), ("256s", 2), ("toy", 40),
                                      ("toy", 24400)])
def test_verify_forms(hs, O, ps, count):
    import torch
    wl = inputs.make(ps, count, num_keys=2, lengths=("uniform", 0, 100), seed=60 + count, key_mode="random")
    pk, sk = hs.hs_keygen(ps, _dev(wl.seeds))
    sigs = _sign(hs, ps, sk, wl)
    S = sigs.shape[1]
    args = (_dev(wl.msgs), _dev(wl.lens))
    kidx = wl.key_idx.copy()
    ok = hs.hs_verify_batch(ps, pk, *args, sigs.cuda(), key_idx=_dev(kidx)).cpu().numpy()
    assert ok.tolist() == [1] * count
    # a flipped bit anywhere: R, the first and last FORS bytes, and bytes spread over all layers
    rng = np.random.default_rng(count)
    bad, where = sigs.clone(), {}
    spots = [0, hs.N_BYTES[ps], S - 1] + [int(x) for x in np.linspace(hs.N_BYTES[ps] + 1, S - 1, 40)]
    for n, i in enumerate(rng.permutation(count)[:max(1, count - 2)]):
        where[int(i)] = spots[n % len(spots)]
        bad[int(i), where[int(i)]] ^= 1 << int(rng.integers(0, 8))
    kidx[count - 1] = 7 if count > 1 else kidx[0]          # an invalid key index
    ok = hs.hs_verify_batch(ps, pk, *args, bad.cuda(), key_idx=_dev(kidx)).cpu().numpy()
    hs.hs_check_status()
    want = [0 if i in where or (count > 1 and i == count - 1) else 1 for i in range(count)]
    assert ok.tolist() == want
