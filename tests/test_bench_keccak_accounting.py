"""The executed ALU work of a one-permutation SHAKE hash in bench.py against
a lane-by-lane enumeration: theta, rho, pi, chi and iota of FIPS 202 on 32-bit
halves, three-input logic and funnel shifts one operation each, the input's
constant lanes folded in the first round and the last round reduced to the
lanes the output needs."""
import pytest

import bench

SETS = ("128f", "192f", "256f", "128s", "192s", "256s")


def _rho_offsets():
    off, x, y = {0: 0}, 1, 0
    for t in range(24):
        off[x + 5 * y] = (t + 1) * (t + 2) // 2 % 64
        x, y = y, (2 * x + 3 * y) % 5
    return off


def _pi_source(lane):
    x, y = lane % 5, lane // 5                       # B[x, y] = A[(x + 3y) mod 5, x]
    return (x + 3 * y) % 5 + 5 * x


def _enumerate(n, payload):
    data, rho = (n + 32 + payload) // 8, _rho_offsets()
    ops = 0
    halves = [set(range(data)) | {data}, set(range(data)) | {16}]     # nonzero: data, pad byte; data, last pad bit
    for nonzero in halves:                           # first round
        for x in range(5):
            terms = [i for i in range(x, 25, 5) if i in nonzero]
            while len(terms) > 1:                    # parity, three terms at a time
                terms = terms[3:] + ["sum"] if len(terms) >= 3 else ["sum"]
                ops += 1
        zero_columns = set()
        for i in range(25):                          # theta into each lane; zero lanes of a column alike
            if i in nonzero:
                ops += 1
            else:
                zero_columns.add(i % 5)
        ops += len(zero_columns)
        ops += 5                                     # parities rotated by one
        ops += sum(1 for i in range(25) if rho[i] % 32)
        ops += 25                                    # chi
    ops += 1                                         # iota: round constant 1
    ops += 22 * 180
    out = n // 8
    lanes = sorted({(x + d) % 5 for x in range(out) for d in range(3)})
    src = [_pi_source(b) for b in lanes]
    parities = {(s + 4) % 5 for s in src} | {(s + 1) % 5 for s in src}
    ops += 2 * (2 * len(parities) + len({s % 5 for s in src}) + len(src) + sum(1 for s in src if rho[s] % 32) + out)
    return ops + 2                                   # iota: both halves of the last constant


@pytest.mark.parametrize("n", [16, 24, 32])
def test_one_permutation_hash(n):
    for payload in (n, 2 * n):
        assert bench._keccak_hash_alu(n, payload) == _enumerate(n, payload)


def test_executed_work_of_the_stages():
    for ps in SETS:
        for st in ("tree", "fors"):
            e, f = bench.exec_alu_per_sig("shake-" + ps, st), bench.alu_ops_per_sig("shake-" + ps, st)
            assert 0.95 * f < e < f, (ps, st)
    # shake-128f FORS: 33 trees of 64 leaves (PRF, F) and 63 nodes, T_k of 5 permutations
    assert bench.exec_alu_per_sig("shake-128f", "fors") == 33 * (128 * _enumerate(16, 16) + 63 * _enumerate(16, 32)) + 5 * 4320
