"""The rule that cuts K for split-precision products (one function, for a product's own launch
and for the waves' grouped products) against its definition: over all splits into whole
slices, the fewest K blocks on the critical path."""
import ctypes as C

import numpy as np
import pytest

from ._helpers import hostsim_lib


def _definition(kind, M, N, Kpad, table, scratch, sms, bn):
    mt = -(-M // 128)
    bn = bn if bn in (128, 144) else 256
    if bn == 256 and table and 2 * mt * -(-N // 256) <= sms:
        bn = 128
    kb = Kpad // ((128 if bn != 256 else 64) // (2 if kind == 1 else 4))
    tiles = mt * -(-N // bn)
    if tiles >= sms or kb < 8 or scratch <= 0:
        return bn, kb
    cost = {}
    for sk in range(1, min(kb // 4, 64) + 1):
        per = -(-kb // sk)
        real = -(-kb // per)
        if real > 1 and real * M * N > scratch:
            break
        cost.setdefault(-(-tiles * real // sms) * (per + 4), per)
    return bn, cost[min(cost)]


@pytest.mark.parametrize("kind", [1, 2], ids=["bf16x3", "tf32x3"])
def test_k_slices_follow_the_definition(kind):
    lib = hostsim_lib()
    rng = np.random.default_rng(kind)
    split = 0
    for _ in range(400):
        M, N = (int(2 ** rng.uniform(0, 13)) for _ in range(2))
        Kpad = 64 * int(2 ** rng.uniform(0, 9))
        table, scratch = int(rng.integers(2)), int(rng.choice([0, 1 << 16, 8 << 20]))
        bn = int(rng.choice([128, 144, 256]))
        got = C.c_int(bn)
        per = lib.rcc_test_split(kind, M, N, Kpad, table, C.c_longlong(scratch), 152, C.byref(got))
        want = _definition(kind, M, N, Kpad, table, scratch, 152, bn)
        assert (got.value, per) == want
        split += per < Kpad // 64
    assert split > 50
