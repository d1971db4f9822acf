"""FP64 contexts with the default options form every contraction in FP64: an element of the
residual is as accurate as the terms of its own sums, however large other elements of the
amplitudes are.

Two groups of virtual orbitals, without integrals between them: the residual of the second
group does not depend on the first one's amplitudes, which are 2^40 times as large in the
rows that both share.  The oracle's own sums multiply them by exact zeros."""
import numpy as np
import pytest

from oracle import compact as oc
from paper_2607_00981_gb300 import binding as B
from paper_2607_00981_gb300.synth import make_instance, random_amplitudes

from ._helpers import gpu_lib, hostsim_lib

BACKENDS = [pytest.param("hostsim", 2, 9, 16, id="hostsim"), pytest.param("gpu", 2, 33, 64, id="gpu", marks=pytest.mark.gpu),
            pytest.param("gpu", 3, 40, 60, id="gpu-o3v40", marks=pytest.mark.gpu)]


@pytest.mark.parametrize("kind,o,v,naux", BACKENDS)
def test_small_amplitudes_beside_large_ones_keep_fp64_accuracy(kind, o, v, naux):
    inst = make_instance(o, v, naux, seed=v)
    t1, t2, t3 = random_amplitudes(o, v, seed=o)
    g = v // 3
    big = np.ones(v)
    big[:g] = 2.0 ** 20
    L = inst.L.copy()
    first = slice(o, o + g)
    rest = np.r_[0:o, o + g:o + v]
    L[:, first, rest] = 0.0
    L[:, rest, first] = 0.0
    t1 = np.zeros_like(t1)
    t2 = t2.copy()
    t2[:, :, :g, :] = 0.0
    t2[:, :, :, :g] = 0.0
    t3c = oc.pack(t3 * big[:, None, None] * big[:, None] * big)
    ctx = B.Context(gpu_lib() if kind == "gpu" else hostsim_lib(), o, v, naux)
    ctx.set_hamiltonian(inst.fock_diag, L)
    ctx.set_amplitudes(t1, t2, t3c)
    ctx.build_intermediates()
    ctx.residual()
    ctx.postprocess()
    _, _, r3 = ctx.residuals()
    ctx.close()
    _, _, R3 = oc.residuals_compact(L, inst.fock_diag, t1, t2, t3c)
    r3, R3 = (oc.postprocess(x, o)[:, g:, g:, g:] for x in (r3, R3))
    assert np.abs(R3).max() < 1e3
    assert np.abs(r3 - R3).max() / max(1.0, np.abs(R3).max()) < 1e-11
