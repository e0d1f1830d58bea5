"""The forms a server batch takes beside other batches (T_l a thread per item,
FORS_Sign by lane groups above 2 trees per SM, launches in plain order) and
alone give the same bytes as hs_sign_batch: requests of three sets at once,
with batches of up to 4 messages (FORS a thread per leaf in both) and up to 24
(9 messages are 2 trees per SM at k = 33 on 152 SMs)."""
import numpy as np
import pytest

from paper_2512_23969_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("sets,layers,max_batch", [(("128f", "192f", "256f"), 0, 24), (("128f", "192f", "256f"), 2, 24),
                                                   (("128f", "192f", "256f"), 1, 4),
                                                   (("shake-128f", "robust-192f", "toy"), 0, 24),
                                                   (("128s", "robust-256f", "shake-192f"), 1, 24)])
def test_overlapping_batches(hs, sets, layers, max_batch):
    count, work = 60, {}
    for i, ps in enumerate(sets):
        wl = inputs.make(ps, count, num_keys=3, lengths=("uniform", 0, 300), seed=510 + i, key_mode="random")
        sk = hs.hs_keygen(ps, _dev(wl.seeds))[1]
        ref = hs.hs_sign_batch(ps, sk, _dev(wl.msgs), _dev(wl.lens), key_idx=_dev(wl.key_idx)).cpu().numpy()
        work[ps] = wl, sk, ref
    with hs.Server({ps: w[1] for ps, w in work.items()}, max_inflight=4, max_batch=max_batch, mem_budget=2 << 30,
                   cache_layers=layers) as srv:
        reqs = [(ps, i, *srv.submit(ps, int(work[ps][0].key_idx[i]), work[ps][0].message(i)))
                for i in range(count) for ps in sets]
        for ps, i, rid, out in reqs:
            srv.wait(rid)
            assert out.tobytes() == work[ps][2][i].tobytes(), (ps, i)
        assert srv.stats()["max_inflight_batches"] >= 2      # batches ran beside each other


def test_form_changed_while_serving(hs):
    """Tuning knobs may change at any time: a batch's scratch and its
    TREE_Sign form come from one look at them."""
    import threading
    from paper_2512_23969_gb300 import autotune
    wl = inputs.make("128f", 64, num_keys=3, lengths=("uniform", 0, 100), seed=540, key_mode="random")
    sk = hs.hs_keygen("128f", _dev(wl.seeds))[1]
    ref = hs.hs_sign_batch("128f", sk, _dev(wl.msgs), _dev(wl.lens), key_idx=_dev(wl.key_idx)).cpu().numpy()
    saved, stop = autotune.get("128f", "tree_split_below"), threading.Event()

    def toggle():
        while not stop.is_set():
            for v in (0, 1 << 20):
                autotune.set("128f", "tree_split_below", v)
    t = threading.Thread(target=toggle)
    t.start()
    try:
        with hs.Server({"128f": sk}, max_inflight=4, max_batch=16, mem_budget=64 << 20) as srv:
            for _ in range(4):
                reqs = [srv.submit("128f", int(wl.key_idx[i]), wl.message(i)) for i in range(64)]
                for i, (rid, out) in enumerate(reqs):
                    srv.wait(rid)
                    assert out.tobytes() == ref[i].tobytes(), i
    finally:
        stop.set()
        t.join()
        autotune.set("128f", "tree_split_below", saved)
