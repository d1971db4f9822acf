"""A context takes larger panels for its grouped intermediates only where they fit: at the
memory's limit it is created without them and gives the same results (split precisions bit
for bit, FP64 at the parity bar).  On the host simulation, whose device memory can be limited."""
import ctypes as C

import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import hostsim_lib


def _memory(lib, limit):
    lib.rcc_test_memory.restype = C.c_longlong
    lib.rcc_test_memory.argtypes = [C.c_longlong]
    return lib.rcc_test_memory(limit)


def _intermediates(ctx, o, v, naux):
    inst = make_instance(o, v, naux, seed=3)
    t1, t2, t3 = random_amplitudes(o, v, seed=4)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, oc.pack(t3))
    ctx.build_intermediates()
    return ctx.debug_copy("Fvv", (v, v)), ctx.debug_copy("Wvvvo", (v, v, v, o))


@pytest.mark.parametrize("prec", [B.FP64, B.SPLIT_BF16X3], ids=["fp64", "bf16x3"])
@pytest.mark.parametrize("batch", [False, True], ids=["alone", "batch"])
def test_created_without_the_larger_panels(prec, batch):
    lib = hostsim_lib()
    o, v, naux = (2, 12, 168) if prec else (5, 12, 204)
    opt = dict(precision=prec, diis_space=2, max_iter=2)

    def create():
        return B.Batch(lib, [(o, v, naux), (1, 3, 5)], **opt) if batch else B.Context(lib, o, v, naux, **opt)

    base = _memory(lib, 0)
    full = create()
    used = _memory(lib, 0) - base
    want = _intermediates(full.instances[0] if batch else full, o, v, naux)
    full.close()
    assert _memory(lib, 0) == base
    _memory(lib, base + used - 300000)
    try:
        lean = create()
        got = _intermediates(lean.instances[0] if batch else lean, o, v, naux)
        held = _memory(lib, 0) - base
        lean.close()
    finally:
        _memory(lib, 0)
    assert held < used
    for x, y in zip(got, want):
        assert np.array_equal(x, y) if prec else np.abs(x - y).max() <= 1e-11 * max(1.0, np.abs(y).max())


def test_a_context_that_does_not_fit_is_refused():
    lib = hostsim_lib()
    base = _memory(lib, 0)
    _memory(lib, base + (8 << 20))
    try:
        with pytest.raises(B.RccsdtError) as ei:
            B.Context(lib, 2, 12, 168)
    finally:
        left = _memory(lib, 0)
    assert ei.value.status == B.ERR_OOM and left == base


@pytest.mark.parametrize("prec", [B.SPLIT_BF16X3, B.SPLIT_TF32X3], ids=["bf16x3", "tf32x3"])
@pytest.mark.parametrize("o,v,naux", [(2, 12, 168), (4, 9, 150)])
def test_waves_are_bitwise_the_products_one_by_one(prec, o, v, naux):
    lib = hostsim_lib()
    lib.rcc_test_memory.restype = C.c_longlong
    lib.rcc_test_memory.argtypes = [C.c_longlong]
    inst = make_instance(o, v, naux, seed=3)
    t1, t2, t3 = random_amplitudes(o, v, seed=4)
    base, out, forms = lib.rcc_test_memory(0), [], (C.c_longlong * 4)()
    for limit in (0, 1):
        if limit:
            lib.rcc_test_memory(base + used - 300000)
        try:
            ctx = B.Context(lib, o, v, naux, precision=prec, diis_space=2)
        finally:
            used = lib.rcc_test_memory(0) - base
        ctx.set_hamiltonian(inst.fock_diag, inst.L)
        ctx.set_amplitudes(t1, t2, oc.pack(t3))
        lib.rcc_test_forms(forms)
        ctx.build_intermediates()
        lib.rcc_test_forms(forms)
        assert (forms[2] == 0) == bool(limit)
        out.append([ctx.debug_copy(n, s) for n, s in (("Fvv", (v, v)), ("Wvvvo", (v, v, v, o)), ("Wb_ovov", (o, v, o, v)))])
        ctx.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


def test_digit_planes_do_not_grow_with_the_panels():
    """The planes are cut from the plans' own operands, not from what the waves add."""
    lib = hostsim_lib()
    o, v, naux = 2, 12, 168
    base, held = _memory(lib, 0), {}
    for f64_tc in (0, 1):
        for lean in (False, True):
            _memory(lib, base + used - 300000 if lean else 0)
            try:
                ctx = B.Context(lib, o, v, naux, precision=B.SPLIT_BF16X3, diis_space=2, f64_tc=f64_tc)
            finally:
                used = _memory(lib, 0) - base
            held[f64_tc, lean] = ctx.device_bytes()
            ctx.close()
    assert held[0, True] < held[0, False]
    assert held[1, False] - held[0, False] == held[1, True] - held[0, True] > 0
