"""Error weights atol + rtol |y| too small to have a reciprocal (an absent species and a denormal atol), on
the CPU (lane_emulator.h) against the oracle."""
import os

import numpy as np
import pytest

from tests import emulated
from tests.conftest import GOLDEN
from tests.gpu_helpers import weighted_norm

TINY = os.path.join(GOLDEN, "tiny_hon7.mech")


@pytest.mark.parametrize("team,block", [(32, 32), (64, 64)])
def test_denormal_weight_of_an_absent_species(tmp_path, team, block):
    from oracle import oracle as O
    lines = open(TINY).read().splitlines()
    i = [k for k, l in enumerate(lines) if l.startswith("SPECIES")][0]
    lines[i] = "SPECIES 8"
    i = [k for k, l in enumerate(lines) if l.startswith("SP N2 ")][0]
    a = " 2.5 0.0 0.0 0.0 0.0 -745.0 4.4"
    lines[i:i] = ["SP AR 39.948 0 0 0 300.0 1000.0 5000.0 0.0 18.6", "LO" + a, "HI" + a]
    spec = str(tmp_path / "ar.mech")
    with open(spec, "w") as fh:
        fh.write("\n".join(lines) + "\n")
    om = O.Mechanism(spec)
    n, dt = 2, 1e-6
    rng = np.random.default_rng(4)
    T, P = rng.uniform(1000.0, 1500.0, n), np.full(n, 101325.0)
    Y = rng.uniform(0.02, 1.0, (n, om.ns))
    Y[:, 6] = 0.0
    Y /= Y.sum(axis=1, keepdims=True)
    emit = emulated.host_program(tmp_path, emulated.EMIT)
    e = emulated.Emulated(tmp_path, emit, spec, team, block, emulated.INTEGRATE)
    T1, Y1, _, _, status, att = e.integrate(T, P, Y, dt, rtol=1e-6, atol=1e-310)
    yo, info = om.integrate(om.state_from_TY(T, Y), P, dt, rtol=1e-6, atol=1e-310)
    assert (info["status"] == 0).all() and (status == 0).all()
    assert (att == info["attempts"]).all()
    assert (weighted_norm(yo, om.state_from_TY(T1, Y1)) <= 1e-5).all()
