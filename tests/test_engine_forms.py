"""rccsdt_engine_info names the forms that a context runs: grouped intermediates, digit planes,
captured sequences (so that a test of replays knows that it replays)."""
import ctypes as C

import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib, hostsim_lib

BACKENDS = [pytest.param("hostsim", id="hostsim"), pytest.param("gpu", id="gpu", marks=pytest.mark.gpu)]


@pytest.mark.parametrize("kind", BACKENDS)
@pytest.mark.parametrize("prec,f64_tc,waves,planes", [(B.FP64, 0, 1, 0), (B.FP64, 1, 1, 6), (B.FP64, 2, 0, 6), (B.FP64, 3, 1, 7),
                                                      (B.SPLIT_BF16X3, 0, 2, 0), (B.SPLIT_TF32X3, 1, 2, 6)])
def test_forms_of_a_context(kind, prec, f64_tc, waves, planes):
    o, v, naux = 2, 5, 10
    lib = gpu_lib() if kind == "gpu" else hostsim_lib()
    inst = make_instance(o, v, naux, seed=2, scale=0.3)
    t1, t2, t3 = (0.05 * x for x in random_amplitudes(o, v, seed=3))
    ctx = B.Context(lib, o, v, naux, precision=prec, f64_tc=f64_tc)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, oc.pack(t3))
    held = []
    for _ in range(4):
        ctx.iterate()
        held.append(ctx.engine_info()["sequences"])
    info = ctx.engine_info()
    assert (info["waves"], info["planes"]) == (waves, planes)
    assert held == [0, 2, 2, 2]  # the residual and the update, from the second call on
    ctx.enable_timing()
    ctx.iterate()
    out = np.zeros(20, dtype=np.int64)
    assert lib.rccsdt_engine_info(ctx.h, out.ctypes.data_as(C.c_void_p), 13) == 13
    ctx.close()
