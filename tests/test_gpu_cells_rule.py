"""Both sides of the lines by which a call without a configuration gets its lanes per cell from the number
of cells; integrated states against the oracle with the parity tests' bound (1e-5 of the solver's
tolerance, cells with the oracle's attempt count)."""
import os

import numpy as np
import pytest

from tests.conftest import GOLDEN, states
from tests.gpu_helpers import gpu_mech, gpu_state, gross_f, to_dev, weighted_norm

pytestmark = pytest.mark.gpu


def _integrate(g, om, T, P, Y, dt, sample):
    """A call on all cells; the sampled ones against the oracle."""
    import torch
    n = len(T)
    dT, dP, dY = to_dev(T), to_dev(P), to_dev(Y.T)
    att = torch.zeros(n, dtype=torch.int32, device=dT.device)
    status = torch.full((n,), -1, dtype=torch.int32, device=dT.device)
    g.integrate(dT, dP, dY, dt, status=status, opts=g.opts(attempts=att))
    assert (status.cpu().numpy() == 0).all()
    y0 = om.state_from_TY(T[sample], Y[sample])
    yo, info = om.integrate(y0, P[sample], dt, threads=16)
    assert (info["status"] == 0).all()
    same = info["attempts"] == att.cpu().numpy()[sample]
    assert same.sum() >= len(sample) - max(1, len(sample) // 50)  # accept/reject flips
    e = weighted_norm(yo, gpu_state(om, dT, dY)[sample])
    assert (e[same] <= 1e-5).all(), e.max()


def _sm_count():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("per_sm", [12, 160])
@pytest.mark.parametrize("over", [0, 1])
def test_seven_species(omech, per_sm, over):
    """Fewer than half as many species as lanes at 16 lanes per cell; 64, 16 and 8 lanes."""
    om = omech("tiny_hon7.mech")
    n = per_sm * _sm_count() + over
    rng = np.random.default_rng(per_sm + over)
    T = rng.uniform(1000.0, 1500.0, n)
    Y = rng.uniform(0.02, 1.0, (n, om.ns))
    Y /= Y.sum(axis=1, keepdims=True)
    g = gpu_mech(os.path.join(GOLDEN, "tiny_hon7.mech"))
    _integrate(g, om, T, np.full(n, 101325.0), Y, 1e-5, np.unique(np.linspace(0, n - 1, 200).astype(int)))


@pytest.mark.parametrize("team,block", [(16, 64), (16, 32), (8, 32), (4, 64)])
def test_seven_species_jacobian_in_shared_warps(omech, team, block):
    """f and J where several teams share a warp, with a last warp that is not full: f to 1e-12 of its gross
    terms, which come to 9e3 times the net sums in these states, so J to 1e-8 of its largest entry."""
    om = omech("tiny_hon7.mech")
    g = gpu_mech(os.path.join(GOLDEN, "tiny_hon7.mech"), team=team, block=block)
    n = 1001
    rng = np.random.default_rng(3)
    T = rng.uniform(300.0, 2500.0, n)
    P = np.full(n, 101325.0)
    Y = rng.uniform(0.02, 1.0, (n, om.ns))
    Y /= Y.sum(axis=1, keepdims=True)
    y = om.state_from_TY(T, Y)
    a = (to_dev(T), to_dev(P), to_dev(y[:, 1:].T))
    f = g.eval_source(*a).cpu().numpy().T
    J = g.eval_jacobian(*a).cpu().numpy().T.reshape(n, om.N, om.N)
    fo, Jo = om.source(y, P), om.jacobian(y, P, threads=4)
    gross = np.array([gross_f(om, y[c], P[c]) for c in range(n)])
    assert (np.abs(f - fo) <= 1e-12 * (np.abs(fo) + gross)).all()
    assert (np.abs(J - Jo).max(axis=(1, 2)) <= 1e-8 * np.abs(Jo).max(axis=(1, 2))).all()


@pytest.mark.parametrize("per_sm", [12, 160])
@pytest.mark.parametrize("over", [0, 1])
def test_thirteen_species(mech_path, omech, per_sm, over):
    n = per_sm * _sm_count() + over
    st = states("h2_13", n, "h2_fresh", 51)
    _integrate(gpu_mech(mech_path("h2_13")), omech("h2_13"), st.T, st.P, st.Y, 1e-7,
               np.unique(np.linspace(0, n - 1, 200).astype(int)))


@pytest.mark.parametrize("over", [0, 1])
def test_fifty_three_species(mech_path, omech, over):
    n = 4 * _sm_count() + over
    st = states("ch4_53", n, "ch4_partial", 52)
    _integrate(gpu_mech(mech_path("ch4_53")), omech("ch4_53"), st.T, st.P, st.Y, 1e-7,
               np.unique(np.linspace(0, n - 1, 60).astype(int)))
