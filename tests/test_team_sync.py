"""Synchronisation of the kernels' lanes, on the CPU: lane_emulator.h lets one end of the block run ahead
as far as the barriers allow, so that a missing one gives wrong numbers, and reports lanes that wait for
others which never come."""
import os

import numpy as np
import pytest

from tests import emulated
from tests.conftest import GOLDEN

TINY = os.path.join(GOLDEN, "tiny_hon7.mech")


@pytest.fixture(scope="module")
def emit(tmp_path_factory):
    return emulated.host_program(tmp_path_factory.mktemp("emit"), emulated.EMIT)


def _states(om, n, seed):
    rng = np.random.default_rng(seed)
    T = rng.uniform(1000.0, 1500.0, n)
    Y = rng.uniform(0.02, 1.0, (n, om.ns))
    Y /= Y.sum(axis=1, keepdims=True)
    return T, np.full(n, 101325.0), Y, om.state_from_TY(T, Y)


@pytest.mark.parametrize("order", [1, -1])
@pytest.mark.parametrize("team", [64, 128])
def test_cached_factors_are_those_of_the_iteration_matrix(emit, omech, tmp_path, team, order):
    """A W-method attempt leaves the plain factors of I/(gamma h) - J in the cell's cache: L U = P M, whichever
    warp gets to the in-place inversion of the diagonal blocks first.  Rounding: growth of a 7 x 7
    elimination with partial pivoting, well below 1e-12 of the largest entry."""
    om = omech("tiny_hon7.mech")
    T, P, Y, y = _states(om, 3, 5)
    e = emulated.Emulated(tmp_path, emit, TINY, team, team, emulated.INTEGRATE, tableau=5)
    n = om.N
    _, _, C, _, status, att = e.integrate(T, P, Y, 1e-9, cache=True, order=order)
    assert (status == 0).all() and (att == 1).all()
    J = om.jacobian(y, P)
    gamma = 1.0 + 1.0 / np.sqrt(2.0)
    ints = (n + 1) // 2
    for c in range(len(T)):
        lu = C[c, :n * n].reshape(n, n)
        perm = np.ascontiguousarray(C[c, n * n:n * n + ints]).view(np.int32)[:n]
        h = C[c, n * n + 2 * ints]
        assert h == 1e-9
        L, U = np.tril(lu, -1) + np.eye(n), np.triu(lu)
        np.fill_diagonal(U, 1.0 / np.diag(lu))
        M = np.eye(n) / (gamma * h) - J[c]
        assert np.abs(L @ U - M[perm]).max() <= 1e-12 * np.abs(M).max()


@pytest.mark.parametrize("order", [1, -1])
@pytest.mark.parametrize("ns,team,block", [(7, 16, 64), (2, 16, 64), (2, 8, 32), (2, 4, 32)])
def test_teams_that_share_a_warp_wait_for_their_own_lanes_only(emit, omech, tmp_path, ns, team, block, order):
    """Several cells per warp, with row sums split over lanes of the team (at most half as many species as
    lanes) and a cell count that leaves the last warp's teams with different numbers of cells: no team may
    wait for another, and f and J agree with the oracle to rounding of their largest term."""
    from oracle import oracle as O
    spec = TINY
    if ns == 2:
        spec = str(tmp_path / "h.mech")
        with open(spec, "w") as fh:
            fh.write(_two_species())
    om = O.Mechanism(spec)
    n = 2 * (block // team) + 1
    T, P, _, y = _states(om, n, 6)
    f, J = emulated.Emulated(tmp_path, emit, spec, team, block, emulated.EVAL).eval(T, P, y[:, 1:], om.nr, order=order)
    fo, Jo = om.source(y, P), om.jacobian(y, P)
    for c in range(n):
        assert np.abs(f[c] - fo[c]).max() <= 1e-12 * np.abs(fo[c]).max()
        assert np.abs(J[c] - Jo[c]).max() <= 1e-12 * np.abs(Jo[c]).max()



def _two_species():
    """H and H2 of the seven-species mechanism with their recombination."""
    lines = open(TINY).read().splitlines()
    out = ["MECHANISM h 0", "ELEMENTS H O N", "SPECIES 2"]
    for s in ("H", "H2"):
        i = [k for k, l in enumerate(lines) if l.startswith("SP %s " % s)][0]
        out += lines[i:i + 3]
    return "\n".join(out + ["REACTIONS 1", "R THIRD 1 H 2 1 H2 1 1.0e13 -0.5 0.0", "EFF 1 H2 2.0", "END", ""])
