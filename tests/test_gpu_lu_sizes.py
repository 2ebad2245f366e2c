"""The blocked factorisation and stage solves at matrix sizes around their tiles (panels of eight
columns, update tiles of 16 rows, 32 rows per warp) and with teams of one and of several panel warps,
with and without warps to spare for the look-ahead; integrated states against the oracle with the
parity tests' bound (1e-5 of the solver's tolerance, cells with the oracle's attempt count)."""
import numpy as np
import pytest

from tests.gpu_helpers import gpu_mech, gpu_state, to_dev, weighted_norm

pytestmark = pytest.mark.gpu

CASES = [(33, 64), (40, 64), (41, 128), (48, 256), (56, 64), (63, 64), (64, 64), (64, 128), (65, 128),
         (96, 128), (97, 256), (128, 128), (128, 256)]


@pytest.mark.parametrize("ns,team", CASES)
def test_integrate_at_matrix_sizes(tmp_path, ns, team):
    import torch
    from oracle import oracle as O
    from paper_2205_05681_gb300 import synth
    mech = synth.make_mechanism(ns, 3 * ns, 6, 6, 4, ("C", "H", "O", "N"), 7000 + ns, name="lu%d" % ns)
    path = str(tmp_path / ("lu%d.mech" % ns))
    synth.write_spec(mech, path)
    om = O.Mechanism(path)
    g = gpu_mech(path, team=team, block=team, cache_dir=None)
    n = 12
    st = synth.make_states(mech, n, "ch4_partial", 41)
    T, P, Y = to_dev(st.T), to_dev(st.P), to_dev(st.Y.T)
    att = torch.zeros(n, dtype=torch.int32, device=T.device)
    status = torch.full((n,), -1, dtype=torch.int32, device=T.device)
    g.integrate(T, P, Y, 1e-7, status=status, opts=g.opts(attempts=att))
    y0 = om.state_from_TY(st.T, st.Y)
    yo, info = om.integrate(y0, st.P, 1e-7, threads=16)
    assert (status.cpu().numpy() == 0).all() and (info["status"] == 0).all()
    same = info["attempts"] == att.cpu().numpy()
    assert same.sum() >= n - 1  # one accept/reject flip at most
    e = weighted_norm(yo, gpu_state(om, T, Y))
    assert (e[same] <= 1e-5).all(), (ns, team, e)
    assert info["attempts"].max() >= 3
