"""Vector-Jacobian products where a rate constant has no normal reciprocal, on the CPU (lane_emulator.h)
against the oracle's Jacobian."""
import os

import numpy as np

from tests import emulated
from tests.conftest import GOLDEN

TINY = os.path.join(GOLDEN, "tiny_hon7.mech")


def test_falloff_with_a_denormal_high_pressure_limit(tmp_path):
    """k_inf = exp(23 - 738) at 176 K (a dissociation of 259 kcal/mol), k_0 [M] / k_inf of about 1e75: the reaction
    adds nothing, so the oracle's mechanism is the one without it; by the VJP tests' bound of 1e-11 of the
    gross terms."""
    from oracle import oracle as O
    text = open(TINY).read()
    new = text.replace("1 H2O 1 1.0e10 0.0 0.0", "1 H2O 1 1.0e10 0.0 259000.0").replace("LOW 1.0e16 -1.0 0.0",
                                                                                         "LOW 1.0e16 -1.0 200000.0")
    assert new.count("259000.0") == 1 and new.count("200000.0") == 1
    spec = str(tmp_path / "cold.mech")
    with open(spec, "w") as fh:
        fh.write(new)
    without = str(tmp_path / "without.mech")
    with open(without, "w") as fh:
        fh.write(text[:text.index("R TROE")].replace("REACTIONS 6", "REACTIONS 5") + "END\n")
    om = O.Mechanism(without)
    rng = np.random.default_rng(2)
    n = 3
    T, P = np.array([174.5, 175.5, 176.0]), np.full(n, 101325.0)
    Y = rng.uniform(0.02, 1.0, (n, om.ns))
    Y /= Y.sum(axis=1, keepdims=True)
    y = om.state_from_TY(T, Y)
    v = rng.normal(size=y.shape) / np.maximum(np.abs(om.source(y, P)), 1e-30)
    e = emulated.Emulated(tmp_path, emulated.host_program(tmp_path, emulated.EMIT), spec, 32, 32, emulated.VJP, adjoint=True)
    gy, gp = e.vjp(T, P, y[:, 1:], v)
    J = om.jacobian(y, P)
    assert np.isfinite(J).all()
    for c in range(n):
        ref, scale = J[c].T @ v[c], np.abs(J[c]).T @ np.abs(v[c])
        assert np.isfinite(gy[c]).all() and np.isfinite(gp[c]).all() and abs(gp[c, 5]) < 1e-200
        assert (np.abs(gy[c] - ref) <= 1e-11 * (np.abs(ref) + scale)).all(), c
