"""D3Q19 reverse steps in tiles of other widths: the same bits as in 128-cell tiles (a
cell's arithmetic does not depend on its tile)."""
import numpy as np
import pytest

from paper_1406_6438_gb300 import workloads as W
from paper_1406_6438_gb300._binding import Launch, VansError
from tests._gpu import solver, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [0, 2, 6])
@pytest.mark.parametrize("nx", [1, 33, 64, 65, 96, 150, 161, 223, 224, 225, 330])
def test_tile_width_does_not_change_the_gradient(nx, walls):
    torch = torch_cuda()
    shape = (3, 4, nx)
    p = W.params(q=19, nx=nx, ny=4, nz=3, wall_mask=walls, tau=0.7, g=(3e-4, -1e-4, 2e-4), drag_mode=2,
                 k_mode=0, d_p=6.0, u_wall=(0.02, 0.0, -0.01) if walls & 2 else (0.0, 0.0, 0.0))
    eps = W.smoothed_noise(shape, 2.0, 0.4, 1.0, nx)
    f0 = torch.from_numpy(W.random_state(19, eps, nx + 1, amp=0.02)).cuda()
    out = []
    for warps in (4, None, 2, 3, 5, 6, 7):
        s = solver(p, eps)
        s.set_populations(f0)
        if warps:
            s.set_adjoint_launch(Launch(1, warps, 2, 1))
        lam, tmp, st = s.new_state(), s.new_state(), s.get_state()
        acc = torch.empty(s.grad_floats(), dtype=torch.float32, device="cuda")
        s.flux_seed(nx - 1, lam, acc, state=st)
        for _ in range(3):
            s.step_adjoint(st, lam, tmp, acc)
            lam, tmp = tmp, lam
        out.append((acc.clone(), s.grad_finalize(lam, acc).clone()))
        s.close()
    assert np.isfinite(out[0][1].cpu().numpy()).all()
    for a, g in out[1:]:
        assert torch.equal(a, out[0][0]) and torch.equal(g, out[0][1])


@pytest.mark.parametrize("q,shapes", [(9, [(1, 2), (1, 4), (2, 4)]), (19, [(1, w) for w in range(2, 8)])])
def test_a_reverse_shape_that_is_accepted_runs(q, shapes):
    """Two stages up to the most that shared memory holds; one more is refused where it is set."""
    p = W.params(q=q, nx=40, ny=5, nz=1 if q == 9 else 3, wall_mask=2, tau=0.7, g=(3e-4, 0.0, 0.0),
                 drag_mode=2, k_mode=0, d_p=6.0)
    eps = W.smoothed_noise((p["nz"], 5, 40), 2.0, 0.4, 1.0, 1)
    torch = torch_cuda()
    s = solver(p, eps)
    lam, tmp, st = s.new_state(), s.new_state(), s.get_state()
    acc = torch.zeros(s.grad_floats(), dtype=torch.float32, device="cuda")
    for cpt, warps in shapes:
        stage = (21 if q == 9 else 47) * (32 * warps * cpt + 16) * 4
        for stages in range(2, 9):
            L = Launch(cpt, warps, stages, 1)
            if 128 + stages * stage > 227 * 1024:
                with pytest.raises(VansError) as e:
                    s.set_adjoint_launch(L)
                assert e.value.status == -1
                continue
            s.set_adjoint_launch(L)
            s.step_adjoint(st, lam, tmp, acc)
