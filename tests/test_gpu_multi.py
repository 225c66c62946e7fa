"""Several steps per launch (kind 9) against the FP64 oracle and against itself.

Tolerance: 2e-7 on populations, as for the single-step kinds (they lie below 0.5,
one ulp is 3e-8; the stored deviations are 1e-2 of that, so ten steps stay within
a few ulps of f)."""
import numpy as np
import pytest

from paper_1406_6438_gb300 import workloads as W
from paper_1406_6438_gb300._binding import Launch, VansError
from tests._gpu import gpu_run, oracle_run, rel_u, solver, torch_cuda

pytestmark = pytest.mark.gpu

LAUNCHES = [Launch(2, 4, t, 9, c) for t in (2, 3, 4) for c in (0, 1)]

# (ny, nx): one cell; rows and columns fewer than the steps of a launch; one column
# block less and more one cell (60 stored columns for 2 steps, 56 for 3 and 4), blocks
# that fit and that wrap; strips of one row and of many
SHAPES = [(1, 1), (2, 3), (3, 60), (4, 61), (5, 56), (7, 57), (8, 64), (9, 113), (13, 120),
          (40, 37), (23, 700), (300, 65)]


def _case(ny, nx, walls, moving, k_mode, seed):
    p = W.params(q=9, nx=nx, ny=ny, wall_mask=2 if walls else 0, tau=0.7, g=(3e-4, -1e-4, 0.0),
                 drag_mode=2, k_mode=k_mode, d_p=6.0, K=2.5, F_eps=0.3,
                 u_wall=(0.02, 0.004, 0.0) if moving else (0.0, 0.0, 0.0))
    eps = W.smoothed_noise((1, ny, nx), 2.0, 0.4, 1.0, seed)
    return p, eps, W.random_state(9, eps, seed + 100, amp=0.02)


@pytest.mark.parametrize("walls,moving,k_mode", [(False, False, 0), (True, False, 2),
                                                 (True, True, 1)])
@pytest.mark.parametrize("ny,nx", SHAPES)
def test_matches_oracle(ny, nx, walls, moving, k_mode):
    """10 steps (4+3+3, 4 x 3-step minus two, 5 x 2): every population and moment."""
    p, eps, f0 = _case(ny, nx, walls, moving, k_mode, seed=ny + nx)
    rho_o, u_o, f_o = oracle_run(p, eps, 10, f0)
    for L in LAUNCHES:
        rho, u, f = gpu_run(p, eps, 10, f0, launch=L)
        assert np.abs(f - f_o).max() <= 2e-7, (L, np.abs(f - f_o).max())
        assert np.abs(rho - rho_o).max() <= 1e-6, L
        assert rel_u(u, u_o) <= 1e-5, (L, rel_u(u, u_o))


@pytest.mark.parametrize("walls", [False, True])
def test_result_does_not_depend_on_the_launch(walls):
    """Bit for bit the same for 2, 3 and 4 steps per launch, for other strips, and
    for one call of 12 steps or calls of 2, 4 and 6 (even: 2 per launch leaves no
    single step, which is another kernel)."""
    torch = torch_cuda()
    p, eps, f0 = _case(50, 150, walls, walls, 0, seed=3)
    out = []
    for L in LAUNCHES + [Launch(2, 4, 4, 9, 2)]:
        for calls in ((12,), (2, 4, 6)):
            s = solver(p, eps, L)
            s.set_populations(torch.from_numpy(f0).cuda())
            for n in calls:
                s.step(n)
            out.append(s.populations())
            s.close()
    for f in out[1:]:
        assert torch.equal(f, out[0])


@pytest.mark.parametrize("walls", [False, True])
def test_result_does_not_depend_on_calls_of_two_steps_or_more(walls):
    """The same for odd counts: 11 steps in one call or in calls of at least two."""
    torch = torch_cuda()
    p, eps, f0 = _case(50, 150, walls, walls, 0, seed=4)
    out = []
    for L in LAUNCHES:
        for calls in ((11,), (2, 9), (3, 3, 5), (7, 4)):
            s = solver(p, eps, L)
            s.set_populations(torch.from_numpy(f0).cuda())
            for n in calls:
                s.step(n)
            out.append(s.populations())
            s.close()
    for f in out[1:]:
        assert torch.equal(f, out[0])


def test_single_steps_and_refusals():
    """vans_step(h, 1), step_raw and step_single run the single-step launch; plates
    on nodes, D3Q19 and shapes that are not built are refused."""
    torch = torch_cuda()
    p, eps, f0 = _case(20, 90, True, False, 0, seed=5)
    f0 = torch.from_numpy(f0).cuda()
    a, b = solver(p, eps, Launch(2, 4, 4, 9)), solver(p, eps, Launch(4, 4, 1))
    for s in (a, b):
        s.set_populations(f0)
        s.step(1)
        s.step_single(5)
    assert torch.equal(a.populations(), b.populations())
    for bad in (Launch(2, 4, 1, 9), Launch(2, 4, 5, 9), Launch(4, 4, 2, 9), Launch(2, 8, 2, 9),
                Launch(2, 4, 2, 9, 3)):
        with pytest.raises(VansError):
            a.launch = bad
    q, eps3 = W.duct_3d(nx=16, ny=6, nz=5)[:2]
    with pytest.raises(VansError):
        solver(q, eps3, Launch(2, 4, 2, 9))
    q, epsc, = W.couette_80(n=20, nx=16, wall_kind=1)
    with pytest.raises(VansError) as e:
        solver(q, epsc, Launch(2, 4, 2, 9))
    assert e.value.status == -5


@pytest.mark.parametrize("L", [Launch(2, 4, 2, 9), Launch(2, 4, 3, 9, 1), Launch(2, 4, 4, 9, 1),
                               Launch(2, 4, 4, 9, 2)])
@pytest.mark.parametrize("nsteps", [5, 14])
def test_batch_matches_oracle(L, nsteps):
    """Uneven domains (walls, moving wall, periodic; one of a single row and column,
    one of several strips) in one batch, each against the oracle."""
    torch = torch_cuda()
    import paper_1406_6438_gb300 as V
    cases = [_case(ny, nx, w, m, k, seed=ny) for ny, nx, w, m, k in
             [(40, 130, True, False, 0), (1, 1, True, False, 0), (150, 61, True, True, 1),
              (33, 300, False, False, 2), (97, 56, True, False, 2), (5, 20, False, False, 0)]]
    b = V.Batch([p for p, _, _ in cases])
    for d, (_, eps, _) in enumerate(cases):
        b.set_eps(d, torch.from_numpy(eps).cuda().view(-1))
    b.launch = L
    b.step(nsteps)
    for d, (p, eps, _) in enumerate(cases):
        rho_o, u_o, f_o = oracle_run(p, eps, nsteps)
        rho, u = b.moments(d)
        f = b.populations(d)
        torch.cuda.synchronize()
        assert np.abs(f.cpu().numpy() - f_o).max() <= 2e-7, (d, L)
        assert rel_u(u.cpu().numpy(), u_o) <= 1e-5, (d, L)
    assert b.launch == L
