"""FP64 residuals at sizes where some contractions gather their operands in the GEMM and others
read packed panels (they share operands), against the oracle at the FP64 bar of the other
parity tests (1e-11 of the largest element), alone and as instances of a batch."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib

SIZES = [(2, 40, 50), (3, 31, 40), (4, 28, 44), (1, 62, 70)]


def _error(ctx, o, v, naux):
    inst = make_instance(o, v, naux, seed=v)
    t1, t2, t3 = random_amplitudes(o, v, seed=o)
    t3c = oc.pack(t3)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, t3c)
    ctx.build_intermediates()
    ctx.residual()
    ctx.postprocess()
    r1, r2, r3 = ctx.residuals()
    R1, R2, R3 = oc.residuals_compact(inst.L, inst.fock_diag, t1, t2, t3c)
    scale = max(1.0, np.abs(R3).max())
    return max(np.abs(r1 - R1).max(), np.abs(r2 - R2).max(),
               np.abs(oc.postprocess(r3, o) - oc.postprocess(R3, o)).max()) / scale


@pytest.mark.gpu
@pytest.mark.parametrize("o,v,naux", SIZES)
def test_gathered_and_packed_operands_alone(o, v, naux):
    ctx = B.Context(gpu_lib(), o, v, naux)
    assert _error(ctx, o, v, naux) < 1e-11
    ctx.close()


@pytest.mark.gpu
def test_gathered_and_packed_operands_in_a_batch():
    batch = B.Batch(gpu_lib(), SIZES, max_iter=2)
    for ctx, size in zip(batch.instances, SIZES):
        assert _error(ctx, *size) < 1e-11
    batch.close()
