"""A species in more reactions of a chunk than its runs in one warp hold (eight runs of seven): the runs
beyond are added by atomics.  On the CPU (lane_emulator.h) against the oracle; f to 1e-12 of its gross
terms, the parity tests' bound, d f / d n to 1e-12 of the rows' largest gross term."""
import os

import numpy as np
import pytest

from tests import emulated
from tests.conftest import GOLDEN
from tests.gpu_helpers import gross_f

TINY = os.path.join(GOLDEN, "tiny_hon7.mech")


@pytest.mark.parametrize("team,block", [(64, 64), (128, 128)])
def test_more_than_eight_runs_of_a_species(tmp_path, team, block):
    from oracle import oracle as O
    lines = open(TINY).read().splitlines()
    i = [k for k, l in enumerate(lines) if l.startswith("REACTIONS")][0]
    extra = ["R ELEM 2 H 1 O2 1 2 O 1 OH 1 %g 0.%d %g" % (1e9 + 1e7 * k, k % 10, 9000.0 + 50.0 * k) for k in range(70)]
    extra += ["R ELEM 1 OH 2 2 O 1 H2O 1 %g 0.1 %g" % (1e8 + 1e6 * k, 700.0 + k) for k in range(40)]
    lines[i] = "REACTIONS %d" % (6 + len(extra))
    lines[-1:-1] = extra
    spec = str(tmp_path / "many.mech")
    with open(spec, "w") as fh:
        fh.write("\n".join(lines) + "\n")
    om = O.Mechanism(spec)
    n = 3
    rng = np.random.default_rng(12)
    T, P = rng.uniform(1000.0, 1500.0, n), np.full(n, 101325.0)
    Y = rng.uniform(0.02, 1.0, (n, om.ns))
    Y /= Y.sum(axis=1, keepdims=True)
    y = om.state_from_TY(T, Y)
    e = emulated.Emulated(tmp_path, emulated.host_program(tmp_path, emulated.EMIT), spec, team, block, emulated.EVAL)
    src = open(e.exe + ".cpp").read()
    words = [int(w) for w in src[src.index("mk_oseg["):].split("{", 1)[1].split("}};")[0].replace("u", "").replace("{", "").replace("}", "").split(",")]
    assert any(w & 0x1000 for w in words[::4]) and any(w & 0x800 for w in words[::4])  # atomics and plain stores
    for order in (1, -1):
        f, J = e.eval(T, P, y[:, 1:], om.nr, order=order)
        fo, Jo = om.source(y, P), om.jacobian(y, P)
        for c in range(n):
            gross = np.abs(gross_f(om, y[c], P[c]))
            assert (np.abs(f[c] - fo[c]) <= 1e-12 * (np.abs(fo[c]) + gross)).all()
            rows = gross.max() / y[c, 1:].min()  # d q / d n is q over the moles of a species
            assert (np.abs(J[c] - Jo[c])[:, 1:] <= 1e-12 * rows).all()
