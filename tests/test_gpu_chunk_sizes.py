"""Launch configurations whose chunk of reactions is cut down to leave room for the cells (not a multiple
of the team's lanes), the largest mechanism among them; integrated states against the oracle with the
parity tests' bound (1e-5 of the solver's tolerance, cells with the oracle's attempt count)."""
import pytest

from tests.gpu_helpers import gpu_mech, gpu_state, to_dev, weighted_norm

pytestmark = pytest.mark.gpu

CASES = [(113, 0, 0), (54, 4, 32), (24, 4, 128), (79, 16, 64)]


def _mechanism(tmp_path, ns):
    from paper_2205_05681_gb300 import synth
    mech = synth.make_mechanism(ns, 3 * ns, 6, 6, 4, ("C", "H", "O", "N"), 7000 + ns, name="ch%d" % ns)
    path = str(tmp_path / ("ch%d.mech" % ns))
    synth.write_spec(mech, path)
    return path, synth.make_states(mech, 12, "ch4_partial", 43)


def _integrate(g, st):
    import torch
    T, P, Y = to_dev(st.T), to_dev(st.P), to_dev(st.Y.T)
    att = torch.zeros(len(st.T), dtype=torch.int32, device=T.device)
    status = torch.full_like(att, -1)
    g.integrate(T, P, Y, 1e-7, status=status, opts=g.opts(attempts=att))
    assert (status.cpu().numpy() == 0).all()
    return T, Y, att.cpu().numpy()


@pytest.mark.parametrize("ns,team,block", CASES)
def test_integrate_with_short_chunks(tmp_path, ns, team, block):
    from oracle import oracle as O
    path, st = _mechanism(tmp_path, ns)
    om = O.Mechanism(path)
    T, Y, att = _integrate(gpu_mech(path, team=team, block=block, cache_dir=None), st)
    yo, info = om.integrate(om.state_from_TY(st.T, st.Y), st.P, 1e-7, threads=8)
    assert (info["status"] == 0).all()
    same = info["attempts"] == att
    assert same.sum() >= len(same) - 1  # one accept/reject flip at most
    e = weighted_norm(yo, gpu_state(om, T, Y))
    assert (e[same] <= 1e-5).all(), (ns, team, e)
    assert info["attempts"].max() >= 3


def test_the_largest_mechanism(tmp_path):
    """164 species fill an SM's shared memory; beyond the oracle's 128, so the block of 256 lanes is compared
    with a warp per cell (another factorisation, other sums) by the same bound."""
    from oracle import oracle as O
    path, st = _mechanism(tmp_path, 164)
    om = O.Mechanism(path)
    y = []
    for kw in ({}, {"team": 32, "block": 32}):
        T, Y, att = _integrate(gpu_mech(path, cache_dir=None, **kw), st)
        y.append((om.state_from_TY(T.cpu().numpy(), Y.cpu().numpy().T), att))
    same = y[0][1] == y[1][1]
    assert same.sum() >= len(same) - 1
    assert (weighted_norm(y[0][0], y[1][0])[same] <= 1e-5).all()
    assert y[0][1].max() >= 3
