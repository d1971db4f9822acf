"""RCCSDT_Q_FP32 takes FP32 for the products only: the spin sum, the denominators, their
quotients and the sum over tuples and quadruples are FP64.  With integer integrals and
amplitudes every FP32 product and sum is exact, so the energy equals the FP64 one bit for
bit (the operations are the same, in the same order)."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B

from ._helpers import gpu_lib


@pytest.mark.gpu
@pytest.mark.parametrize("o,v", [(2, 2), (2, 5), (3, 4), (4, 3), (5, 3), (6, 2)])
def test_exact_products_give_the_fp64_energy(o, v):
    rng = np.random.default_rng(10 * o + v)
    n, nonzero = o + v, 0
    for _ in range(4):
        L = rng.integers(-1, 2, size=(1, n, n)).astype(float)
        L = np.triu(L[0]) + np.triu(L[0], 1).T
        e = np.concatenate([np.sort(-0.5 - rng.random(o)), np.sort(0.3 + rng.random(v))])
        t2 = rng.integers(-1, 2, size=(o, o, v, v)).astype(float)
        t2 = t2 + t2.transpose(1, 0, 3, 2)
        t3c = rng.integers(-1, 2, size=(oc.n3(o), v, v, v)).astype(float)
        ctx = B.Context(gpu_lib(), o, v, 1)
        ctx.set_hamiltonian(e, L[None])
        ctx.set_amplitudes(np.zeros((o, v)), t2, t3c)
        e64, e32 = ctx.q_energy(B.Q_FP64)[0], ctx.q_energy(B.Q_FP32)[0]
        ctx.close()
        assert e32 == e64
        nonzero += e64 != 0.0
    assert nonzero
