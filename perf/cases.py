"""The workloads the signer is timed on, each one call of a user's program
through the public entry points of ``paper_2512_23969_gb300.hs``.

A case is a dict of plain values:

  kind       "sign" (hs_sign_batch), "slh" (hs_slh_sign_batch), "verify"
             (hs_verify_batch), "mixed" (hs_sign_mixed), "serve" (hs.Server:
             submit every request, wait for all), "keygen" (hs_keygen)
  params     the parameter set ("mixed" and "serve": drawn per message over
             128f / 192f / 256f)
  count      messages (keygen: keys)
  keys       signing keys (mixed and serve: split over the three sets)
  lo, hi     message lengths in bytes: uniform in [lo, hi], or log-uniform
             with "log"
  ctx        bytes of the FIPS 205 context string ("slh")
  host       buffers in page-locked host memory instead of device memory

The sizes are those of the repository's own workload recipes (inputs.py) and
tests: 64 and 16384 messages of 32 bytes at 128f, batches of U[32, 1024]
bytes at 192f / 256f, the 96-message mixed batch of log-U[16 B, 64 KB], the
60/25/15 serving mix over 1024 keys, and single calls.
"""
import math

import numpy as np
import torch

from paper_2512_23969_gb300 import hs, inputs

F_SETS = ("128f", "192f", "256f")
# n, layers d, tree height h', FORS height a, FORS trees k
SHAPE = {"128f": (16, 22, 3, 6, 33), "192f": (24, 22, 3, 8, 33), "256f": (32, 17, 4, 9, 35),
         "128s": (16, 7, 9, 12, 14), "192s": (24, 7, 9, 14, 17), "256s": (32, 8, 8, 14, 22)}
SETS = list(SHAPE) + ["shake-" + s for s in SHAPE] + ["robust-" + s for s in F_SETS]


def _case(name, kind, params, count, keys=1, lo=32, hi=32, log=False, ctx=0, host=False):
    c = {"kind": kind, "params": params, "count": count, "keys": keys, "lo": lo, "hi": hi, "log": log, "ctx": ctx,
         "host": host}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one signature while a caller waits for it
        _case("sign_128f_1", "sign", "128f", 1),
        # a small batch under one key
        _case("sign_128f_64", "sign", "128f", 64),
        # bulk signing: the benchmark's batch
        _case("sign_128f_16384", "sign", "128f", 16384, keys=16),
        # bulk signing of documents of mixed length at the middle security level
        _case("sign_192f_4096", "sign", "192f", 4096, keys=16, lo=32, hi=1024),
        # standard (FIPS 205) signing from an application's host buffers
        _case("slh_256f_1021_host", "slh", "256f", 1021, keys=16, lo=32, hi=1024, ctx=20, host=True),
        # short signatures, as for firmware and certificates
        _case("sign_128s_200", "sign", "128s", 200, keys=4, lo=32, hi=1024),
        # the SHAKE instantiation
        _case("sign_shake128f_1000", "sign", "shake-128f", 1000, keys=16, lo=32, hi=1024),
        # a small batch over several sets with long messages among it
        _case("mixed_96", "mixed", "", 96, keys=64, lo=16, hi=65536, log=True),
        # requests of many keys through the server
        _case("serve_256", "serve", "", 256, keys=1024, lo=16, hi=4096, log=True),
        # bulk verification
        _case("verify_128f_16384", "verify", "128f", 16384, keys=16),
        # verifying a handful of signatures while a caller waits
        _case("verify_256f_7", "verify", "256f", 7, keys=3, lo=32, hi=1024),
        # issuing keys
        _case("keygen_128f_1024", "keygen", "128f", 1024),
    ]


def _ops(family, n, blocks, tl=False):
    """ALU operations (rotations and 3-input logic on 32-bit lanes) of a hash
    of the given number of blocks: 1024 per SHA-256 block, 2624 per SHA-512
    block, 4320 per Keccak-f[1600]."""
    if family == "shake":
        return 4320 * blocks
    return (2624 if tl and n > 16 else 1024) * blocks


def _distinct(keys, bits, count):
    """Expected distinct values of count draws over keys * 2**bits."""
    u = keys * 2.0 ** bits
    return u * -math.expm1(count * math.log1p(-1.0 / u)) if u > 1 else 1.0


def _set_work(kind, ps, count, keys, mean_len):
    """(bytes, operations) of count messages of one set."""
    family, base = (ps.split("-") if "-" in ps else ("sha2", ps))
    n, d, hp, a, k = SHAPE[base]
    length = 2 * n + 3
    leaves = 1 << hp
    block = 136 if family == "shake" else (128 if n > 16 else 64)
    f = _ops(family, n, 2 if family == "robust" else 1)
    h = _ops(family, n, 2 if family == "robust" else 1, True)
    tl_blocks = lambda m: ((n + 32 + m * n) // 136 + 1 if family == "shake"          # noqa: E731
                           else (22 + m * n + (17 if n > 16 else 9) + block - 1) // block)
    tl = lambda m: _ops(family, n, tl_blocks(m) * (2 if family == "robust" else 1), True)   # noqa: E731
    leaf = length * 16 * f + tl(length)
    tree = leaves * leaf + (leaves - 1) * h
    msg = _ops(family, n, 6 + 2 * int(mean_len) // block, True)
    sig = n * (1 + k * (a + 1) + d * (length + hp))
    if kind == "keygen":
        return count * 9 * n, count * tree
    if kind == "verify":
        ops = msg + k * (f + a * h) + tl(k) + d * (length * 7.5 * f + tl(length) + hp * h)
        return count * (sig + mean_len + 13) + keys * 2 * n, count * ops
    ops = count * (msg + k * ((2 << a) * f + ((1 << a) - 1) * h) + tl(k))
    for j in range(d):                       # a tree that several messages sign with is needed once
        ops += _distinct(keys, hp * (d - 1 - j), count) * tree
    return count * (sig + mean_len + 12) + keys * 4 * n, ops


def _mean_len(case):
    lo, hi = case["lo"], case["hi"]
    return (hi - lo) / math.log(hi / lo) if case["log"] and hi > lo else 0.5 * (lo + hi)


def _split(total, mix):
    out = [max(1, int(round(total * m))) for m in mix]
    return out[:-1] + [max(1, total - sum(out[:-1]))]


MIX = {"mixed": (0.5, 0.3, 0.2), "serve": (0.6, 0.25, 0.15)}


def work(case):
    kind = case["kind"]
    if kind in MIX:
        parts = [_set_work("sign", ps, c, k, _mean_len(case)) for ps, c, k in
                 zip(F_SETS, _split(case["count"], MIX[kind]), _split(case["keys"], MIX[kind]))]
    else:
        parts = [_set_work(kind, case["params"], case["count"], case["keys"], _mean_len(case))]
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


def draw(rng):
    """One more case: the kinds as they are used, the plain SHA-2 f sets most
    often, sizes spread over their logarithm and up to the largest listed."""
    cap = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["sign"] * 5 + ["slh"] * 2 + ["verify"] * 4 + ["mixed", "serve", "keygen"])
        sets = [s for s in SETS if not (kind == "slh" and s.startswith("robust"))]
        params = "" if kind in MIX else rng.choice(F_SETS if rng.random() < 0.5 else sets)
        top = {"mixed": 2048, "serve": 1024, "keygen": 4096}.get(kind, 16384)
        least = {"mixed": 12, "serve": 12, "verify": 3}.get(kind, 1)
        count = int(round(math.exp(rng.uniform(math.log(least), math.log(top)))))
        keys = int(round(math.exp(rng.uniform(0, math.log(64)))))
        keys = 64 if kind == "mixed" else (1024 if kind == "serve" else min(keys, count))
        log = kind in MIX or rng.random() < 0.25
        lo, hi = rng.choice([(32, 32), (32, 1024), (1, 200), (16, 4096)])
        if kind == "mixed":
            lo, hi = 16, 65536
        elif kind == "serve":
            lo, hi = 16, 4096
        host = kind in ("sign", "slh", "verify", "keygen") and rng.random() < 0.2
        c = _case(None, kind, params, count, keys, lo, hi, log, rng.randint(0, 255) if kind == "slh" else 0, host)
        if work(c)["flops"] <= cap:
            return c


class _State:
    pass


def _tensor(x, host):
    t = torch.from_numpy(np.ascontiguousarray(x))
    return t.pin_memory() if host else t.cuda()


def _out(n, host):
    return torch.empty(n, dtype=torch.uint8, pin_memory=True) if host else \
        torch.empty(n, dtype=torch.uint8, device="cuda")


def _batch(case, seed, params, count, keys, host):
    """One set's inputs: keys, packed messages, lengths, key indices and the
    signature buffer."""
    if case["log"]:
        lengths = ("loguniform", case["lo"], case["hi"])
    else:
        lengths = ("uniform", case["lo"], case["hi"])
    wl = inputs.make(params, count, num_keys=keys, lengths=lengths, seed=seed, key_mode="random")
    pk, sk = hs.hs_keygen(params, _tensor(wl.seeds, False))
    b = _State()
    b.params = params
    b.pk, b.sk = (pk.cpu().pin_memory(), sk.cpu().pin_memory()) if host else (pk, sk)
    b.msgs, b.lens, b.key_idx = (_tensor(x, host) for x in (wl.msgs, wl.lens.view(np.int64),
                                                            wl.key_idx.view(np.int32)))
    b.sigs = _out(count * hs.sig_bytes(params), host)
    return b


def prepare(case, seed):
    st = _State()
    st.kind, count, keys, host = case["kind"], case["count"], case["keys"], case["host"]
    rng = np.random.default_rng(seed + 1)
    if st.kind in MIX:
        mix = MIX[st.kind]
        split, counts = _split(keys, mix), _split(count, mix)
    if st.kind == "keygen":
        n = hs.N_BYTES[case["params"]]
        st.params = case["params"]
        st.seeds = _tensor(np.frombuffer(rng.bytes(3 * n * count), np.uint8).reshape(count, 3 * n).copy(), host)
        st.pk, st.sk = _out(count * 2 * n, host), _out(count * 4 * n, host)
    elif st.kind == "mixed":
        st.jobs = []
        for i, ps in enumerate(F_SETS):
            b = _batch(case, seed * 8 + i, ps, counts[i], split[i], False)
            st.jobs.append({"params": ps, "sk": b.sk, "msgs": b.msgs, "lens": b.lens, "key_idx": b.key_idx,
                            "sigs": b.sigs})
    elif st.kind == "serve":
        keysets = {}
        for i, ps in enumerate(F_SETS):
            n = hs.N_BYTES[ps]
            seeds = np.frombuffer(rng.bytes(3 * n * split[i]), np.uint8).reshape(split[i], 3 * n).copy()
            keysets[ps] = hs.hs_keygen(ps, _tensor(seeds, False))[1]
        st.server = hs.Server(keysets, max_inflight=4, max_batch=1024, mem_budget=4 << 30)
        lens = inputs.log_uniform_lengths(rng, sum(counts), case["lo"], case["hi"])
        st.sigs = [np.empty((c, hs.sig_bytes(ps)), np.uint8) for ps, c in zip(F_SETS, counts)]
        rows = [(i, r) for i, c in enumerate(counts) for r in range(c)]
        rng.shuffle(rows)                                            # the sets arrive mixed
        st.requests = [(F_SETS[i], int(rng.integers(0, split[i])), rng.bytes(int(n)), st.sigs[i][r])
                       for (i, r), n in zip(rows, lens)]
    else:
        b = st.b = _batch(case, seed, case["params"], count, keys, host)
        st.ctx = rng.bytes(case["ctx"])
        if st.kind == "verify":
            b.sigs = hs.hs_sign_batch(b.params, b.sk, b.msgs, b.lens, key_idx=b.key_idx, sigs=b.sigs)
            bad = np.nonzero(rng.random(count) < min(0.5, max(2 / count, 1 / 64)))[0]      # a few do not verify
            at = rng.integers(0, hs.sig_bytes(b.params), size=bad.size)
            dev = b.sigs.device
            b.sigs[torch.from_numpy(bad).to(dev), torch.from_numpy(at).to(dev)] ^= 1
            b.ok = _out(count, host)
    torch.cuda.synchronize()
    return st


def run(state):
    if state.kind == "keygen":
        pk, sk = hs.hs_keygen(state.params, state.seeds, pk=state.pk, sk=state.sk)
        return [pk, sk]
    if state.kind == "mixed":
        return hs.hs_sign_mixed(state.jobs)
    if state.kind == "serve":
        ids = [state.server.submit(ps, key, msg, out)[0] for ps, key, msg, out in state.requests]
        for i in ids:
            state.server.wait(i)
        state.server.poll()                                          # collected: the server forgets them
        return state.sigs
    b = state.b
    if state.kind == "sign":
        return hs.hs_sign_batch(b.params, b.sk, b.msgs, b.lens, key_idx=b.key_idx, sigs=b.sigs)
    if state.kind == "slh":
        return hs.hs_slh_sign_batch(b.params, b.sk, b.msgs, b.lens, ctx=state.ctx, key_idx=b.key_idx, sigs=b.sigs)
    return hs.hs_verify_batch(b.params, b.pk, b.msgs, b.lens, b.sigs, key_idx=b.key_idx, ok=b.ok)


def exact(case, seed):
    """Every output is bytes: there is no value in 64 bits beside them."""
    return None
