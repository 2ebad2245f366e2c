"""The adjoint on both sides of the line by number of cells (17 to 64 species: 128 lanes per cell up to four
cells per SM, 64 above)."""
import numpy as np
import pytest

from tests.conftest import states
from tests.gpu_helpers import gpu_mech, to_dev

pytestmark = pytest.mark.gpu


def _tape(g, n, dt=1e-7):
    import torch
    st = states("ch4_53", n, "ch4_ign", 61)
    T, P, Y = to_dev(st.T), to_dev(st.P), to_dev(st.Y.T)
    tape = g.make_tape(n, 512, 8)
    status = torch.full((n,), -1, dtype=torch.int32, device=T.device)
    g.integrate_ckpt(T, P, Y, dt, tape, status=status)
    assert (status.cpu().numpy() == 0).all()
    gY = torch.zeros_like(Y)
    gY[1] = 1.0
    return P, 2.0 * (T - 1500.0), gY, tape


def _outputs(g, n):
    import torch
    return tuple(torch.full(s, float("nan"), dtype=torch.float64, device="cuda") for s in ((g.nr,), (n,), (g.ns, n)))


@pytest.mark.parametrize("setup", [0, 1])
def test_set_up_by_one_call_serves_a_capture_of_another_size(mech_path, setup):
    """chem_adjoint_noalloc is called once, on many cells or on none, before the calls that must not allocate
    (a stream capture among them); those may have any number of cells."""
    import ctypes as C
    import torch
    from paper_2205_05681_gb300 import chem
    g = gpu_mech(mech_path("ch4_53"))
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    n = 16
    args = _tape(g, n)
    if setup == 0:
        ptr = [C.c_void_p(x.data_ptr()) for x in (*args[:3], *_outputs(g, n))]
        none = chem.TapeStruct(args[3].buf.data_ptr(), args[3].buf.numel(), 0, 512, 8)
        rc = g._lib.chem_adjoint_noalloc(g._h, 0, *ptr[:3], 0, C.byref(none), None, *ptr[3:],
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0, g._lib.chem_last_error()
    else:
        many = 4 * sm + 8
        g.adjoint_noalloc(*_tape(g, many), *_outputs(g, many))
    out = _outputs(g, n)
    with torch.cuda.graph(torch.cuda.CUDAGraph()):  # the first capture of a process takes memory of its own
        out[0].fill_(0.0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.adjoint_noalloc(*args, *out, stream=torch.cuda.current_stream())
        taken = free - torch.cuda.mem_get_info()[0]
    graph.replay()
    torch.cuda.synchronize()
    assert taken < 8 << 20, taken  # a second module's scratch array alone is 8 MiB
    for a, b in zip(g.adjoint(*args), out):
        a, b = a.cpu().numpy(), b.cpu().numpy()
        assert np.all(np.isfinite(b))
        assert np.allclose(b, a, rtol=1e-9, atol=1e-12 * np.abs(a).max())  # other sums of the same terms


@pytest.mark.parametrize("lanes", [128, 64])
def test_directional_derivatives_vs_complex_step(mech_path, omech, lanes):
    """Few cells take 128 lanes each by default; the same with the 64 that many cells get.  Against the oracle's
    complex step along the accepted steps, by the adjoint tests' bound of 1e-6 of the gradient's scale."""
    om = omech("ch4_53")
    g = gpu_mech(mech_path("ch4_53"))
    n, dt = 3, 1e-6
    P, gT, gY, tape = _tape(g, n, dt)
    opts = g.opts() if lanes == 128 else g.opts(team=64, block=64)
    g_lnA, gT0, gY0 = [x.cpu().numpy() for x in g.adjoint(P, gT, gY, tape, opts=opts)]
    gT, gY = gT.cpu().numpy(), gY.cpu().numpy().T
    nacc, hs = tape.n_accepted().cpu().numpy(), tape.step_sizes().cpu().numpy()
    st = states("ch4_53", n, "ch4_ign", 61)
    y0 = om.state_from_TY(st.T, st.Y)
    gy0 = np.concatenate([gT0[:, None], gY0.T[:, :-1] * om.W[:-1]], axis=1)
    rng = np.random.default_rng(8)
    for _ in range(3):
        dy = rng.normal(size=(n, om.N)) * np.maximum(np.abs(y0), 1e-12)
        dl = rng.normal(size=om.nr)
        ref = 0.0
        for c in range(n):
            y = om.replay_cplx(y0[c] + 1e-30j * dy[c], st.P[c], hs[:nacc[c], c], lnA=om.lnA + 1e-30j * dl)
            d = y.imag / 1e-30
            # L = gT T + sum_k gY_k Y_k, the last mass fraction from the closure
            ref += gT[c] * d[0] + ((gY[c, :-1] - gY[c, -1]) * om.W[:-1]) @ d[1:]
        got = (gy0 * dy).sum() + g_lnA @ dl
        scale = np.abs(gy0 * dy).sum() + np.abs(g_lnA * dl).sum()
        assert abs(got - ref) <= 1e-6 * scale, (got, ref, scale)
