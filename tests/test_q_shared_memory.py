"""(Q) where the tiled kernel's dynamic shared memory is just below 48 KB: its static tables
count too, so these sizes need the opt-in (o = 5, v = 35 and 36 in FP32 did not launch).
Against the FP64 energy of the same amplitudes (FP32 bar 1e-5), or its neighbours' form."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B

from ._helpers import gpu_lib


@pytest.mark.gpu
@pytest.mark.parametrize("o,v", [(5, 34), (5, 35), (5, 36), (5, 37)])
def test_sizes_at_48_kilobytes(o, v):
    rng = np.random.default_rng(v)
    n, naux = o + v, 3
    L = 0.1 * rng.standard_normal((naux, n, n))
    L = L + L.transpose(0, 2, 1)
    e = np.concatenate([np.sort(-0.5 - rng.random(o)), np.sort(0.3 + rng.random(v))])
    t2 = 0.01 * rng.standard_normal((o, o, v, v))
    t2 = t2 + t2.transpose(1, 0, 3, 2)
    t3c = 0.001 * rng.standard_normal((oc.n3(o), v, v, v))
    ctx = B.Context(gpu_lib(), o, v, naux, diis_space=0)
    ctx.set_hamiltonian(e, L)
    ctx.set_amplitudes(np.zeros((o, v)), t2, t3c)
    e64, e32 = ctx.q_energy(B.Q_FP64)[0], ctx.q_energy(B.Q_FP32)[0]
    ctx.close()
    assert e64 != 0.0 and abs(e32 - e64) <= 1e-5 * abs(e64)
