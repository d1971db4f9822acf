"""The flop count of rccsdt_q_energy names the form that ran: 12 joint permutations where the
tiled kernel takes the sizes (FP32 2 <= o <= 8, FP64 2 <= o <= 7 at these sizes), else 24."""
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib


@pytest.mark.gpu
@pytest.mark.parametrize("o,v,n64,n32", [(1, 6, 24, 24), (2, 5, 12, 12), (7, 4, 12, 12), (8, 3, 24, 12), (9, 3, 24, 24)])
def test_flop_of_the_form_that_ran(o, v, n64, n32):
    naux = o + v
    inst = make_instance(o, v, naux, seed=o)
    t1, t2, t3 = random_amplitudes(o, v, seed=v)
    ctx = B.Context(gpu_lib(), o, v, naux)
    ctx.set_hamiltonian(inst.fock_diag, inst.L)
    ctx.set_amplitudes(t1, t2, oc.pack(t3))
    for arith, n in ((B.Q_FP64, n64), (B.Q_FP32, n32)):
        info = ctx.q_energy(arith)[1]
        assert info["flop"] == 2.0 * n * o ** 4 * (2 * v + 2 * o) * info["quadruples"]
    ctx.close()
