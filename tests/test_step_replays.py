"""Replayed iterations and solves equal the same ones launched one by one, bit for bit (a
context with timing on never captures), on the engines beyond the default one: products one
by one in the split precisions, digit planes of every kind, DIIS on a virtual subspace."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib

ENGINES = {
    "per-plan-bf16x3": ((3, 20, 24), dict(precision=B.SPLIT_BF16X3, grouped_bytes=0)),
    "per-plan-tf32x3": ((2, 33, 40), dict(precision=B.SPLIT_TF32X3, grouped_bytes=0)),
    "six-planes": ((3, 20, 24), dict(f64_tc=2)),
    "six-planes-large": ((4, 36, 40), dict(f64_tc=1)),
    "seven-planes": ((4, 36, 40), dict(f64_tc=3)),
    "units-large": ((4, 36, 40), dict()),
    "subspace-fp64": ((3, 20, 24), dict(diis_t3_nvir=9)),
    "subspace-bf16x3": ((3, 20, 24), dict(precision=B.SPLIT_BF16X3, diis_t3_nvir=8)),
}


def _run(size, opt, timed, solve):
    o, v, naux = size
    ctx = B.Context(gpu_lib(), o, v, naux, tol=1e-7, max_iter=8 if solve else 100, **opt)
    if timed:
        ctx.enable_timing()
    out = []
    for seed in (1, 2):
        inst = make_instance(o, v, naux, seed=seed, scale=0.3)
        ctx.set_hamiltonian(inst.fock_diag, inst.L)
        t1, t2, t3 = (0.02 * x for x in random_amplitudes(o, v, seed=seed))
        for _ in range(2 if solve else 1):
            ctx.set_amplitudes(t1, t2, oc.pack(t3))
            if solve:
                out.append(np.array([float(x) for x in ctx.solve()]))
        for _ in range(0 if solve else 5):
            e, norms = ctx.iterate()
            out.append(np.concatenate([[e], norms]))
        out += list(ctx.amplitudes())
    ctx.close()
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("engine", list(ENGINES))
def test_replayed_iterations_equal_plain_launches(engine):
    for x, y in zip(_run(*ENGINES[engine], False, False), _run(*ENGINES[engine], True, False)):
        assert np.array_equal(x, y)


@pytest.mark.gpu
@pytest.mark.parametrize("engine", ["per-plan-bf16x3", "seven-planes", "subspace-fp64"])
def test_replayed_solves_equal_plain_launches(engine):
    for x, y in zip(_run(*ENGINES[engine], False, True), _run(*ENGINES[engine], True, True)):
        assert np.array_equal(x, y)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [B.SPLIT_BF16X3, B.SPLIT_TF32X3], ids=["bf16x3", "tf32x3"])
def test_converging_split_solves_equal_plain_launches(prec):
    """Through the split iterations to the FP64 ones (other sequences of one solve)."""
    o, v, naux = 3, 12, 40
    inst = make_instance(o, v, naux, seed=3)
    out = []
    for timed in (False, True):
        ctx = B.Context(gpu_lib(), o, v, naux, precision=prec, tol=1e-7, max_iter=60)
        if timed:
            ctx.enable_timing()
        ctx.set_hamiltonian(inst.fock_diag, inst.L)
        for _ in range(3):
            ctx.init_mp2()
            out.append(ctx.solve())
        ctx.close()
    assert out[0][3] and all(x == out[0] for x in out)
