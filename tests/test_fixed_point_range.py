"""Mechanisms and run-time ln A at the ends of the fixed-point logarithms' range, on the CPU (lane_emulator.h)
against the oracle: what does not fit takes the FP64 functions.  f to 1e-12 of its gross terms, the parity
tests' bound."""
import os

import numpy as np
import pytest

from tests import emulated
from tests.conftest import GOLDEN
from tests.gpu_helpers import gross_f

TINY = os.path.join(GOLDEN, "tiny_hon7.mech")


@pytest.fixture(scope="module")
def emit(tmp_path_factory):
    return emulated.host_program(tmp_path_factory.mktemp("emit"), emulated.EMIT)


def _state(om, T, seed=9):
    rng = np.random.default_rng(seed)
    Y = rng.uniform(0.02, 1.0, (len(T), om.ns))
    Y /= Y.sum(axis=1, keepdims=True)
    return np.full(len(T), 101325.0), om.state_from_TY(T, Y)


def _check(f, fo, gross):
    for c in range(len(f)):
        assert np.isfinite(f[c]).all() and (np.abs(f[c] - fo[c]) <= 1e-12 * (np.abs(fo[c]) + gross[c])).all(), (c, f[c], fo[c])


def test_run_time_ln_a_far_from_the_file(emit, tmp_path):
    """log2 k_f = -1,900 and K_c = 2^340 at 257 K: within the range with the file's A of 1, not with exp(-490)."""
    from oracle import oracle as O
    text = open(TINY).read()
    new = text.replace("R ELEM 1 OH 2 2 O 1 H2O 1 2.0e9 0.0 1000.0", "R ELEM 2 H 1 OH 1 1 H2O 1 1.0 -60.0 247000.0")
    assert new != text
    spec = str(tmp_path / "cold.mech")
    with open(spec, "w") as fh:
        fh.write(new)
    om = O.Mechanism(spec)
    T = np.array([257.0, 300.0, 1200.0])
    P, y = _state(om, T)
    lnA = om.lnA.copy()
    lnA[3] = -490.0
    lnA[0] += 0.5
    e = emulated.Emulated(tmp_path, emit, spec, 32, 32, emulated.EVAL)
    f, _ = e.eval(T, P, y[:, 1:], om.nr, lnA=lnA)
    gross = np.abs([gross_f(om, y[c], P[c]) for c in range(3)])
    _check(f, om.source(y, P, lnA=lnA), 2.0 * gross)  # reaction 0 is e^0.5 faster


def test_thermodynamic_polynomial_beyond_the_format(emit, tmp_path):
    """The polynomial part of log2 exp(s/R - h/RT) is 2,150 for one species and 2,030 for another, beyond and
    within the format, while the sums with the terms in log T and 1/T are 980 and 860 at 260 K."""
    from oracle import oracle as O
    lines = open(TINY).read().splitlines()
    i = [k for k, l in enumerate(lines) if l.startswith("SPECIES")][0]
    lines[i] = "SPECIES 9"
    i = [k for k, l in enumerate(lines) if l.startswith("SP N2 ")][0]
    for name, lg in (("X", 2150.0), ("Y", 2030.0)):
        a = " -60.0 0.0 0.0 0.0 0.0 124000.0 %r" % float(lg * np.log(2.0) - 60.0)
        lines[i:i] = ["SP %s 15.999 0 1 0 300.0 1000.0 5000.0 0.0 0.0" % name, "LO" + a, "HI" + a]
    i = [k for k, l in enumerate(lines) if l.startswith("REACTIONS")][0]
    lines[i:i + 1] = ["REACTIONS 7", "R ELEM 2 X 1 O 1 2 Y 1 O 1 1.0e-20 0.0 0.0"]
    spec = str(tmp_path / "poly.mech")
    with open(spec, "w") as fh:
        fh.write("\n".join(lines) + "\n")
    om = O.Mechanism(spec)
    T = np.array([258.0, 260.0, 262.0])
    P, y = _state(om, T)
    f, _ = emulated.Emulated(tmp_path, emit, spec, 32, 32, emulated.EVAL).eval(T, P, y[:, 1:], om.nr)
    _check(f, om.source(y, P), np.abs([gross_f(om, y[c], P[c]) for c in range(3)]))
