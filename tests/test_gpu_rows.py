"""D3Q19 rows that are one tile of a kind 6 or 7 pipeline: staged without halo
columns, the last sector stored whole.

Tolerances as for the other single-step kinds: 2e-7 on populations, 1e-5 on u."""
import numpy as np
import pytest

from paper_1406_6438_gb300 import workloads as W
from paper_1406_6438_gb300._binding import Launch
from tests._gpu import gpu_run, oracle_run, rel_u, solver, torch_cuda

pytestmark = pytest.mark.gpu

# nx at the ends of the tiles' and the sectors' ranges, and launches that take it as one
# tile or (the last) as two
CASES = [(nx, [Launch(1, (nx + 31) // 32, 2, 6)] * (nx > 32) + [Launch(1, 8, 3, 6), Launch(2, 4, 2, 7)])
         for nx in (1, 2, 7, 8, 9, 33, 64, 65, 95, 96, 127, 150, 153, 160, 191, 223, 224, 255, 256)]
CASES += [(257, [Launch(1, 5, 2, 6), Launch(2, 5, 2, 7)]), (319, [Launch(1, 5, 3, 6), Launch(2, 5, 2, 7)])]


def _case(nx, walls, seed):
    p = W.params(q=19, nx=nx, ny=4, nz=3, wall_mask=walls, tau=0.7, g=(3e-4, -1e-4, 2e-4), drag_mode=2,
                 k_mode=0, d_p=6.0, u_wall=(0.02, 0.0, -0.01) if walls & 2 else (0.0, 0.0, 0.0))
    eps = W.smoothed_noise((3, 4, nx), 2.0, 0.4, 1.0, seed)
    return p, eps, W.random_state(19, eps, seed + 100, amp=0.02)


@pytest.mark.parametrize("walls", [0, 2, 6])
@pytest.mark.parametrize("nx,launches", CASES)
def test_matches_oracle(nx, launches, walls):
    p, eps, f0 = _case(nx, walls, seed=nx)
    rho_o, u_o, f_o = oracle_run(p, eps, 5, f0)
    for L in launches:
        rho, u, f = gpu_run(p, eps, 5, f0, launch=L)
        assert np.abs(f - f_o).max() <= 2e-7, (L, np.abs(f - f_o).max())
        assert rel_u(u, u_o) <= 1e-5, (L, rel_u(u, u_o))


@pytest.mark.parametrize("nx", [150, 96, 33])
def test_halo_copies_serve_the_other_kinds(nx):
    """Kinds that read the halo columns and kinds that do not, in turn, leave the
    bits that one of them alone leaves."""
    torch = torch_cuda()
    p, eps, f0 = _case(nx, 2, seed=nx)
    f0 = torch.from_numpy(f0).cuda()
    row, other = Launch(1, (nx + 31) // 32, 2, 6), Launch(1, 4, 1)
    out = []
    for turn in ([other] * 6, [row, other] * 3, [other, row] * 3, [row] * 6):
        s = solver(p, eps, turn[0])
        s.set_populations(f0)
        for L in turn:
            s.launch = L
            s.step(1)
        out.append(s.populations())
        s.close()
    for f in out[1:]:
        assert torch.equal(f, out[0])


@pytest.mark.parametrize("nx", [1, 24, 31, 32])
def test_the_narrowest_tile_takes_short_rows(nx):
    """Rows of at most half the 64-cell tile, which autotune offers them."""
    p, eps, f0 = _case(nx, 6, seed=nx)
    rho_o, u_o, f_o = oracle_run(p, eps, 5, f0)
    for stages in (2, 3):
        rho, u, f = gpu_run(p, eps, 5, f0, launch=Launch(1, 2, stages, 6))
        assert np.abs(f - f_o).max() <= 2e-7 and rel_u(u, u_o) <= 1e-5


@pytest.mark.parametrize("shape", [(61, 67, 250), (64, 75, 221), (80, 100, 129)])
def test_last_sectors_stored_whole_of_a_domain_beyond_the_l2(shape):
    """More than a million cells, where tiles that a row fills to 4/5 store its last sector
    whole: kind 6 leaves the bits of the register-load kernel, which stores cells and halo
    copies alone, whoever steps next; the strip kinds agree within 2e-7."""
    torch = torch_cuda()
    nz, ny, nx = shape
    p = W.params(q=19, nx=nx, ny=ny, nz=nz, wall_mask=2, tau=0.7, g=(3e-4, -1e-4, 2e-4), drag_mode=2, k_mode=0,
                 d_p=6.0)
    eps = W.smoothed_noise(shape, 2.0, 0.4, 1.0, nx)
    plain, fit = Launch(1, 4, 1), Launch(1, (nx + 31) // 32, 2, 6)
    out = []
    for turn in ([plain] * 6, [fit] * 6, [fit, plain] * 3, [Launch(2, 4, 2, 2), Launch(1, 8, 2, 4)] * 3,
                 [Launch(1, 4, 3, 4), fit] * 3):
        s = solver(p, eps, turn[0])
        for L in turn:
            s.launch = L
            s.step(1)
        out.append(s.populations())
        s.close()
    assert torch.equal(out[1], out[0]) and torch.equal(out[2], out[0])
    for f in out[3:]:
        assert float((f - out[0]).abs().max()) <= 2e-7
