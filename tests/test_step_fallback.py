"""Iterations whose captured sequence cannot be captured, or not be launched, run launch by
launch: the same results, no error.  On the host simulation, whose captures and graph
launches can be made to fail (a replay there runs the sequence without its effects on the
context's flags)."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import hostsim_lib

O, V, NAUX = 2, 5, 10


def _iterations(lib, fail_from, fail, solve=False):
    inst = make_instance(O, V, NAUX, seed=2, scale=0.3)
    t1, t2, t3 = (0.05 * x for x in random_amplitudes(O, V, seed=3))
    ctx = B.Context(lib, O, V, NAUX, tol=1e-9, max_iter=40)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, oc.pack(t3))
    lib.rcc_test_graphs(0)
    out = []
    try:
        for it in range(6):
            if it == fail_from:
                lib.rcc_test_graphs(fail)
            if solve:
                ctx.init_mp2()
                out.append(np.array([float(x) for x in ctx.solve()[:3]]))
            else:
                e, norms = ctx.iterate()
                out.append(np.concatenate([[e], norms]))
    finally:
        replays = lib.rcc_test_graphs(0)
    out += list(ctx.amplitudes())
    ctx.close()
    return out, replays


@pytest.mark.parametrize("solve", [False, True], ids=["iterate", "solve"])
@pytest.mark.parametrize("fail_from,fail", [(0, 1), (0, 2), (3, 2)], ids=["capture", "launch", "later-launch"])
def test_a_failed_graph_falls_back_to_plain_launches(fail_from, fail, solve):
    lib = hostsim_lib()
    want, replays = _iterations(lib, 99, 0, solve)
    assert replays > 0
    got, replays = _iterations(lib, fail_from, fail, solve)
    assert replays == 0  # (counted from the failure on)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
