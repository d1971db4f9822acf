"""What a context with digit planes holds, and with it the form of its products, follows from
its sizes and options: the planes of both operands (six or seven BF16 words per panel
element) and nothing that depends on the memory free at its creation."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [B.FP64, B.SPLIT_BF16X3], ids=["fp64", "bf16x3"])
@pytest.mark.parametrize("o,v,naux", [(2, 33, 64), (5, 36, 60), (6, 48, 100)])
def test_planes_are_all_that_the_option_adds(prec, o, v, naux):
    held = []
    for f64_tc in (0, 1, 2, 3):
        ctx = B.Context(gpu_lib(), o, v, naux, precision=prec, f64_tc=f64_tc, diis_space=2)
        held.append(ctx.device_bytes())
        ctx.close()
    six, seven = held[1] - held[0], held[3] - held[0]
    assert six > 0 and held[2] == held[1] and 7 * six == 6 * seven


@pytest.mark.gpu
@pytest.mark.parametrize("f64_tc,bar", [(1, 1e-10), (2, 1e-10), (3, 1e-11)])
@pytest.mark.parametrize("o,v,naux", [(2, 40, 50), (5, 36, 60), (3, 50, 60)])
def test_dense_products_in_the_panels_memory(o, v, naux, f64_tc, bar):
    inst = make_instance(o, v, naux, seed=v)
    t1, t2, t3 = random_amplitudes(o, v, seed=o)
    t3c = oc.pack(t3)
    ctx = B.Context(gpu_lib(), o, v, naux, f64_tc=f64_tc)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, t3c)
    for _ in range(2):  # the second evaluation finds the panels as the first one left them
        ctx.build_intermediates()
        ctx.residual()
        ctx.postprocess()
    r1, r2, r3 = ctx.residuals()
    ctx.close()
    R1, R2, R3 = oc.residuals_compact(inst.L, inst.fock_diag, t1, t2, t3c)
    scale = max(1.0, np.abs(R3).max())
    err = max(np.abs(r1 - R1).max(), np.abs(r2 - R2).max(), np.abs(oc.postprocess(r3, o) - oc.postprocess(R3, o)).max())
    assert err / scale < bar
