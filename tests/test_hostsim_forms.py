"""The host simulation runs the forms the GPU runs: small intermediates as five waves of grouped
products and their grouped combines, R3's FP64 products with operands gathered in the GEMM,
the split residual as one grouped product.  Residuals against the oracle at the bars of the
other parity tests, alone and as an instance of a batch (whole K slices)."""
import ctypes as C

import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import hostsim_lib


def _evaluate(ctx, o, v, naux):
    inst = make_instance(o, v, naux, seed=v)
    t1, t2, t3 = random_amplitudes(o, v, seed=o)
    t3c = oc.pack(t3)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, t3c)
    forms = (C.c_longlong * 4)()
    ctx.lib.rcc_test_forms(forms)
    ctx.build_intermediates()
    ctx.residual()
    ctx.postprocess()
    ctx.lib.rcc_test_forms(forms)
    r1, r2, r3 = ctx.residuals()
    R1, R2, R3 = oc.residuals_compact(inst.L, inst.fock_diag, t1, t2, t3c)
    scale = max(1.0, np.abs(R3).max())
    err = max(np.abs(r1 - R1).max(), np.abs(r2 - R2).max(), np.abs(oc.postprocess(r3, o) - oc.postprocess(R3, o)).max())
    return err / scale, list(forms)


@pytest.mark.parametrize("prec,bar", [(B.FP64, 1e-11), (B.SPLIT_BF16X3, 5e-5), (B.SPLIT_TF32X3, 5e-6)],
                         ids=["fp64", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("batch", [False, True], ids=["alone", "batch"])
def test_waves_and_grouped_combines_on_the_host(prec, bar, batch):
    o, v, naux = 2, 9, 20
    lib = hostsim_lib()
    group = B.Batch(lib, [(o, v, naux), (1, 4, 6)], precision=prec, max_iter=2) if batch else None
    ctx = group.instances[0] if batch else B.Context(lib, o, v, naux, precision=prec)
    err, (gather, waves64, split, combines) = _evaluate(ctx, o, v, naux)
    (group or ctx).close()
    assert err < bar
    assert combines >= 13
    if prec == B.FP64:
        assert waves64 == 5 and split == 0 and gather > 5
    else:
        assert split == 6 and waves64 == 0 and gather == 0
