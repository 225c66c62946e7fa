"""D2Q9 moments by rows and by cells: the choice between them by the lanes that a row uses."""
import numpy as np
import pytest

from paper_1406_6438_gb300 import workloads as W
from tests._gpu import gpu_run, oracle_run, rel_u

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("nx", [1, 2, 3, 79, 80, 81, 127, 128, 129, 159, 160, 161, 239, 240, 256, 257, 400])
def test_moments_match_the_oracle(nx, moving):
    """Either side of 5/8 of the lanes of one, two and three warps a row; tolerances as for
    the step kernels (1e-6 on rho, 1e-5 relative on u)."""
    ny = 7
    p = W.params(q=9, nx=nx, ny=ny, wall_mask=2, tau=0.7, g=(3e-4, -1e-4, 0.0), drag_mode=2, k_mode=0, d_p=6.0,
                 u_wall=(0.02, 0.0, 0.0) if moving else (0.0, 0.0, 0.0))
    eps = W.smoothed_noise((1, ny, nx), 2.0, 0.4, 1.0, nx)
    f0 = W.random_state(9, eps, nx + 100, amp=0.02)
    rho_o, u_o, _ = oracle_run(p, eps, 0, f0)
    rho, u, _ = gpu_run(p, eps, 0, f0)
    assert np.abs(rho - rho_o).max() <= 1e-6
    assert rel_u(u, u_o) <= 1e-5
