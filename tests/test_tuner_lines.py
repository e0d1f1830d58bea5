"""The tuner's lines between two forms, with made-up times in place of the
GPU's: the line gives away least over the sizes measured, and lies just behind
a size, not at the next one; the chain-parallel form's line keeps its chain
ends within SPLIT_BYTES; the batches timed share no trees."""
import os
import subprocess
import sys

import pytest

from paper_2512_23969_gb300 import autotune, hs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_form_line():
    f = autotune.form_line
    assert f((8, 16, 32), (1, 1, 1), (2, 2, 2)) == 64
    assert f((8, 16, 32), (2, 2, 2), (1, 1, 1)) == 0
    assert f((8, 16, 32), (1, 1, 3), (2, 2, 2)) == 17
    assert f((8, 16, 32), (1, 1, 1), (1, 1, 1)) == 0                       # no difference: form b
    assert f((64, 256, 512, 1024), (1, 1, 1.2, 1), (2, 2, 1, 1.1)) == 257   # a late win of less than the loss
    assert f((64, 256, 512, 1024), (1, 1, 1.05, 1), (2, 2, 1, 1.1)) == 2048


@pytest.mark.parametrize("ps", ["128f", "192f", "256f"])
def test_split_line_ends_at_the_last_win(monkeypatch, ps):
    knobs = {"tree_split_below": 0}
    split = {8: 0.3, 64: 0.8, 256: 2.54, 1024: 9.99, 2048: 19.0}     # ms; 2048: one more win
    leaf = {8: 0.96, 64: 0.96, 256: 2.71, 1024: 8.88, 2048: 19.1}
    monkeypatch.setattr(autotune, "_batch", lambda p, count, seed=0: (count, None, None, None))
    monkeypatch.setattr(autotune, "_stage_ms", lambda p, wl, *a: (split if wl < knobs["tree_split_below"] else leaf)[wl])
    monkeypatch.setattr(autotune, "set", lambda p, k, v: knobs.update({k: v}))
    assert autotune.tune_split(ps, counts=(8, 64, 256, 1024, 2048), verbose=False)["best"] == 257
    assert knobs["tree_split_below"] == 257


@pytest.mark.parametrize("ps", ["shake-256f", "robust-256f", "shake-192f", "256s", "128f"])
def test_split_line_bounds_the_chain_ends(monkeypatch, ps):
    seen = []
    monkeypatch.setattr(autotune, "_batch", lambda p, count, seed=0: (count, None, None, None))
    monkeypatch.setattr(autotune, "set", lambda p, k, v: seen.append(v) if k == "tree_split_below" else None)
    monkeypatch.setattr(autotune, "_stage_ms", lambda *a: 1.0 if seen[-1] else 2.0)     # chain-parallel always ahead
    best = autotune.tune_split(ps, verbose=False)["best"]
    d, leaves = autotune._shape(ps)
    n = hs.N_BYTES[ps]
    assert 0 < (best - 1) * d * leaves * (2 * n + 3) * n <= autotune.SPLIT_BYTES


@pytest.mark.parametrize("count", [1, 3, 110, 16384])
def test_tuner_batches_share_no_trees(monkeypatch, count):
    """Trees are shared from two messages per key on (plan_dedup)."""
    class Made(Exception):
        pass

    def make(ps, n, num_keys, *a, **k):
        assert n == count and 2 * num_keys > n
        raise Made
    monkeypatch.setattr(autotune.inputs, "make", make)
    with pytest.raises(Made):
        autotune._batch("128f", count)


def test_default_message_line_is_two_warps_per_sub_partition():
    """Beyond two warps per SM sub-partition (8 per SM, 152 SMs) the message
    stage's warp form is behind at long messages: the default line stops
    there.  (A process of its own: other tests set the knob.)"""
    out = subprocess.run([sys.executable, "-c", "from paper_2512_23969_gb300 import autotune, hs\n"
                          "for ps in hs.PARAMS: print(ps, autotune.get(ps, 'msg_warp_below'))"],
                         cwd=ROOT, check=True, capture_output=True, text=True).stdout
    lines = dict(row.split() for row in out.splitlines())
    assert len(lines) == len(hs.PARAMS)
    for ps, line in lines.items():
        assert int(line) == 0 if ps.startswith("shake") else 0 < int(line) <= 8 * 152 + 1, ps
