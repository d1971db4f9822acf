"""A grouped combine launch takes combines of up to four dimensions that do not depend on each
other, and refuses the rest when a context is built: random pairs of views of one array
against their element sets, on the host simulation."""
import ctypes as C
import itertools

import numpy as np

from paper_2607_00981_gb300 import binding as B

from ._helpers import hostsim_lib


def _elements(shape, offset, strides):
    return {offset + sum(i * s for i, s in zip(idx, strides)) for idx in itertools.product(*map(range, shape))}


def _status(lib, items, size=4096):
    flat = [v for shape, oo, os_, io, is_ in items for v in (len(shape), *shape, oo, *os_, io, *is_)]
    x = np.zeros(size)
    return lib.rcc_test_group(x.ctypes.data_as(C.c_void_p), np.array(flat, dtype=np.int64).ctypes.data_as(C.c_void_p))


def test_dependent_combines_are_refused_and_others_taken():
    lib = hostsim_lib()
    rng = np.random.default_rng(1)
    taken = refused = interleaved = 0
    for _ in range(1500):
        shape = tuple(int(n) for n in rng.integers(1, 5, size=rng.integers(1, 5)))
        # a dense layout with room between its rows, or any strides
        strides, step = [], 1
        for n in reversed(shape):
            strides.insert(0, step)
            step *= n + int(rng.integers(0, 3))
        off = int(rng.integers(0, 1200))
        items = []
        for q in range(2):
            oo = off + (int(rng.integers(-40, 41)) if q else 0)
            io = int(rng.integers(2500, 2600)) if rng.integers(4) else int(rng.integers(0, 1300))
            items.append((shape, max(oo, 0), strides, io, [int(s) for s in rng.permutation(strides)]))
        outs = [_elements(i[0], i[1], i[2]) for i in items]
        ins = [_elements(i[0], i[3], i[4]) for i in items]
        depend = bool(outs[0] & outs[1] or outs[0] & ins[1] or outs[1] & ins[0])
        st = _status(lib, items)
        if depend:
            assert st == B.ERR_ARG
            refused += 1
        else:  # (views of other strides are refused where their ranges overlap)
            close = any(min(a) <= max(b) and min(b) <= max(a) for a, b in ((outs[0], ins[1]), (outs[1], ins[0])))
            assert st == B.OK or close
            taken += st == B.OK
            interleaved += st == B.OK and min(outs[0]) <= max(outs[1]) and min(outs[1]) <= max(outs[0])
    assert taken > 200 and refused > 200 and interleaved > 20


def test_five_dimensions_are_refused():
    lib = hostsim_lib()
    s5, st5 = (2, 2, 2, 2, 2), (16, 8, 4, 2, 1)
    s4, st4 = (2, 2, 2, 2), (8, 4, 2, 1)
    other = (s4, 1000, st4, 1100, st4)
    assert _status(lib, [(s4, 0, st4, 100, st4), other]) == B.OK
    assert _status(lib, [(s5, 0, st5, 100, st5), other]) == B.ERR_ARG
