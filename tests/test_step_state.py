"""What is accepted after an iteration that reported a non-finite residual does not depend on
whether the iteration was launched or replayed: the intermediates and the residual are those
of the amplitudes, so rccsdt_residual and rccsdt_postprocess run (the latter with the same
report), and new amplitudes start afresh."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib, hostsim_lib

BACKENDS = [pytest.param("hostsim", id="hostsim"), pytest.param("gpu", id="gpu", marks=pytest.mark.gpu)]


@pytest.mark.parametrize("kind", BACKENDS)
@pytest.mark.parametrize("prec", [B.FP64, B.SPLIT_BF16X3], ids=["fp64", "bf16x3"])
def test_calls_after_a_nonfinite_residual(kind, prec):
    o, v, naux = 2, 5, 10
    lib = gpu_lib() if kind == "gpu" else hostsim_lib()
    inst = make_instance(o, v, naux, seed=2, scale=0.3)
    t1, t2, t3 = (0.05 * x for x in random_amplitudes(o, v, seed=3))
    t3c = oc.pack(t3)
    bad = t1.copy()
    bad[1, 2] = np.nan
    ctx = B.Context(lib, o, v, naux, precision=prec)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    norms = []
    for _ in range(4):
        ctx.set_amplitudes(bad, t2, t3c)
        with pytest.raises(B.RccsdtError) as ei:
            ctx.iterate()
        assert ei.value.status == B.ERR_NONFINITE
        ctx.residual()
        with pytest.raises(B.RccsdtError) as ei:
            ctx.postprocess()
        assert ei.value.status == B.ERR_NONFINITE
        ctx.set_amplitudes(t1, t2, t3c)
        with pytest.raises(B.RccsdtError) as ei:
            ctx.residual()  # no intermediates of these amplitudes yet
        assert ei.value.status == B.ERR_STATE
        norms.append(ctx.iterate()[1])
        with pytest.raises(B.RccsdtError) as ei:
            ctx.postprocess()  # the update has changed the amplitudes
        assert ei.value.status == B.ERR_STATE
    ctx.close()
    assert all(np.array_equal(x, norms[0]) for x in norms)
