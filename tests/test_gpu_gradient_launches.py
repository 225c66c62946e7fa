"""Reverse mode on handles whose forward launch is kind 8, kind 9 or the autotuner's pick:
the forward pass, the recomputed segments and the buffers that nobody zeroes."""
import numpy as np
import pytest

import oracle as O
from paper_1406_6438_gb300 import workloads as W
from paper_1406_6438_gb300._binding import Launch
from tests._gpu import solver, torch_cuda

pytestmark = pytest.mark.gpu

# D2Q9 (odd rows and columns, walls, a moving wall) and D3Q19, small enough for a cluster
CASES = {
    "channel": W.adjoint_channel(nx=64, ny=48)[0],
    "periodic": W.params(q=9, nx=61, ny=33, wall_mask=0, tau=0.7, g=(5e-5, 2e-5, 0), drag_mode=2, k_mode=0,
                         d_p=W.D_P),
    "moving": W.params(q=9, nx=37, ny=20, wall_mask=2, tau=0.9, g=(1e-4, 0, 0), drag_mode=2, k_mode=2, K=4.0,
                       u_wall=(0.01, 0, 0)),
    "duct": W.params(q=19, nx=12, ny=8, nz=6, wall_mask=6, tau=0.7, g=(1e-4, 0, 0), drag_mode=2, k_mode=0, d_p=5.0),
}
LAUNCHES = {"kind0": None, "kind8": Launch(1, 16, 16, 8), "kind9x2": Launch(2, 4, 2, 9), "kind9x4": Launch(2, 4, 4, 9),
            "auto": "auto"}
GRID = [(c, k) for c in CASES for k in LAUNCHES if c != "duct" or not k.startswith("kind9")]


def _solver(case, launch):
    p = CASES[case]
    eps = W.smoothed_noise((p["nz"], p["ny"], p["nx"]), 4.0, 0.4, 1.0, seed=p["ny"])
    L = LAUNCHES[launch]
    s = solver(p, eps, None if L == "auto" else L)
    if L == "auto":
        s.autotune()
    return p, eps, s


def _populations(s, state):
    s.set_state(state)
    return s.populations()


@pytest.mark.parametrize("case,launch", GRID)
def test_segments_are_recomputed_bit_for_bit(case, launch):
    """seg[k] holds the populations that step_single(k) leads to."""
    torch = torch_cuda()
    p, eps, s = _solver(case, launch)
    s.step(7)
    start, n = s.get_state(), 6
    states = []
    for k in range(n + 1):
        s.set_state(start)
        s.step_single(k)
        states.append(s.populations())
    seg = torch.full((n + 1, s.state_floats), float("nan"), device="cuda")
    lam, tmp = torch.full((2, s.state_floats), float("nan"), device="cuda")
    acc = torch.full((s.grad_floats(),), float("nan"), device="cuda")
    s.set_state(start)
    s.step_single(n)
    s.flux_seed(p["nx"] - 1, lam, acc)
    s.adjoint_segment(start, seg, n, lam, tmp, acc)
    for k in range(n + 1):
        assert torch.equal(_populations(s, seg[k]), states[k]), k


@pytest.mark.parametrize("case,launch", GRID)
def test_gradient(case, launch, monkeypatch):
    """Within 1e-4 of the oracle's adjoint (the tolerance of the default launch), the same
    bits whatever the checkpoint interval, and whatever fresh buffers hold."""
    torch = torch_cuda()
    from paper_1406_6438_gb300.adjoint import outlet_flux
    p, eps, s = _solver(case, launch)
    n = 24

    def grad(every):
        e = torch.from_numpy(eps).cuda().requires_grad_(True)
        J = outlet_flux(e, s, n, every)
        (g,) = torch.autograd.grad(J, e)
        return g.cpu().numpy().astype(np.float64)
    g = grad(7)
    g_o = O.adjoint(O.Params(**p), eps.astype(np.float64), n, p["nx"] - 1)[1]
    assert np.abs(g - g_o).max() <= 1e-4 * np.abs(g_o).max()
    for every in (24, 5):
        assert np.array_equal(grad(every), g)
    empty, empty_like = torch.empty, torch.empty_like
    monkeypatch.setattr(torch, "empty", lambda *a, **k: empty(*a, **k).fill_(float("nan")))
    monkeypatch.setattr(torch, "empty_like", lambda *a, **k: empty_like(*a, **k).fill_(float("nan")))
    assert np.array_equal(grad(7), g)
