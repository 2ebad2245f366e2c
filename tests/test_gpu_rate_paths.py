"""The reaction loop's paths: reactions beyond A + B = C + D (equal species, third order, a species on
both sides), the FP64 functions outside the fixed-point range, run-time ln A, in every kind of
team; against the oracle with the parity tests' bound of 1e-12 of the gross row magnitude."""
import numpy as np
import pytest

from tests.conftest import states
from tests.gpu_helpers import gpu_mech, gross_f, to_dev

pytestmark = pytest.mark.gpu

EXTRA = """R ELEM 2 H 2 O 1 1 H2O 1 1.0e15 -0.5 100.0
R ELEM 2 H 2 H2O 1 2 H2 1 H2O 1 6.0e15 -1.2 0.0
R ELEM 1 HO 2 2 O 1 H2O 1 4.0e9 1.1 500.0
R ELEM 1 O 3 2 O2 1 O 1 1.0e14 0.0 0.0
R THIRD 1 HO 2 1 H2O2 1 2.0e15 -0.7 0.0
EFF 2 H2O 6.0 H 2.5
R LIND 1 HO 2 1 H2O2 1 7.0e12 -0.4 0.0
EFF 1 N2 0.7
LOW 2.0e17 -0.9 -1500.0
"""


@pytest.fixture(scope="module")
def odd_mech(mech_path, tmp_path_factory):
    from oracle import oracle as O
    lines = open(mech_path("h2_13")).read().splitlines()
    i = [k for k, l in enumerate(lines) if l.startswith("REACTIONS")][0]
    lines[i] = "REACTIONS %d" % (int(lines[i].split()[1]) + 6)
    lines[-1:-1] = EXTRA.splitlines()
    path = str(tmp_path_factory.mktemp("odd") / "odd.mech")
    open(path, "w").write("\n".join(lines) + "\n")
    return path, O.Mechanism(path)


def _check(om, g, T, st, y, lnA=None):
    y = y.copy()
    y[:, 0] = T
    kw = {} if lnA is None else {"lnA": to_dev(lnA)}
    okw = {} if lnA is None else {"lnA": lnA}
    args = (to_dev(y[:, 0]), to_dev(st.P), to_dev(y[:, 1:].T))
    f = g.eval_source(*args, **kw).cpu().numpy().T
    J = g.eval_jacobian(*args, **kw).cpu().numpy().T.reshape(len(T), om.N, om.N)
    fo = om.source(y, st.P, **okw)
    Jo = om.jacobian(y, st.P, threads=4, **okw)
    for c in range(len(T)):
        gr = gross_f(om, y[c], st.P[c]) if lnA is None else np.abs(fo[c]).max() + np.abs(f[c]).max()
        assert (np.abs(f[c] - fo[c]) <= 1e-12 * (np.abs(fo[c]) + gr)).all(), (c, T[c])
        row = np.abs(Jo[c]).max(axis=1, keepdims=True)
        assert (np.abs(J[c] - Jo[c]) <= 1e-12 * (np.abs(Jo[c]) + row)).all(), (c, T[c])


@pytest.mark.parametrize("team,block", [(1, 32), (4, 64), (16, 64), (32, 64), (64, 64), (256, 256)])
def test_reaction_forms_and_temperature_range(odd_mech, team, block):
    path, om = odd_mech
    g = gpu_mech(path, team=team, block=block)
    n = 48
    st = states("h2_13", n, "h2_fresh", 31)
    y = om.state_from_TY(st.T, st.Y)
    # both sides of the fixed-point range's ends (256 and 8192 K) and inside it
    T = np.resize([300.0, 255.9, 256.0, 256.1, 999.9, 1000.0, 1600.0, 4000.0, 8191.9, 8192.0, 8200.0, 240.0], n)
    _check(om, g, T, st, y)


def test_ln_a_outside_the_fixed_point_range(odd_mech):
    path, om = odd_mech
    g = gpu_mech(path, team=64, block=64)
    n = 16
    st = states("h2_13", n, "h2_fresh", 32)
    y = om.state_from_TY(st.T, st.Y)
    lnA = om.lnA.copy()
    lnA[::3] -= 620.0  # beyond |ln A| = 500: these reactions take the FP64 functions
    lnA[1::3] += 0.5
    _check(om, g, st.T, st, y, lnA)


@pytest.mark.parametrize("team,block", [(4, 64), (64, 64)])
def test_mechanism_outside_the_fixed_point_range(odd_mech, tmp_path, team, block):
    """An activation temperature beyond the fixed-point format: every rate takes the FP64 functions."""
    from oracle import oracle as O
    path, _ = odd_mech
    text = open(path).read()
    cold = text.replace("2 O2 1 O 1 1.0e14 0.0 0.0", "2 O2 1 O 1 1.0e14 0.0 900000.0")
    assert cold != text
    p = tmp_path / "cold.mech"
    p.write_text(cold)
    om = O.Mechanism(str(p))
    st = states("h2_13", 24, "h2_fresh", 33)
    _check(om, gpu_mech(str(p), team=team, block=block), st.T, st, om.state_from_TY(st.T, st.Y))
