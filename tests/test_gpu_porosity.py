"""Porosity fields: the range check, the padded rows and the update in place, and the
emissions between launches of several steps."""
import numpy as np
import pytest

from paper_1406_6438_gb300 import workloads as W
from paper_1406_6438_gb300._binding import Launch, VansError
from tests._gpu import solver, torch_cuda

pytestmark = pytest.mark.gpu

# (q, (nz, ny, nx)): rows and fields off the vectors of four, one cell, one row
SHAPES = [(9, (1, 1, 1)), (9, (1, 3, 2)), (9, (1, 7, 129)), (9, (1, 64, 256)), (19, (2, 3, 1)), (19, (5, 4, 37))]


def _case(q, shape, seed, moving=False):
    nz, ny, nx = shape
    p = W.params(q=q, nx=nx, ny=ny, nz=nz, wall_mask=2, tau=0.7, g=(3e-4, 0.0, 0.0), drag_mode=2,
                 k_mode=0, d_p=6.0, u_wall=(0.02, 0.0, 0.0) if moving else (0.0, 0.0, 0.0))
    eps = W.smoothed_noise(shape, 2.0, 0.4, 1.0, seed)
    return p, eps, W.random_state(q, eps, seed + 1, amp=0.02)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("q,shape", SHAPES)
def test_update_keeps_the_populations_or_refuses(q, shape, offset):
    """update_eps leaves f as it was (one rounding of a deviation: 2e-7) and steps as a
    handle set to the new field does (10 x that); a value outside (0, 1] anywhere,
    the last included, is refused and changes nothing."""
    torch = torch_cuda()
    p, eps, f0 = _case(q, shape, 3, moving=True)
    new = W.smoothed_noise(shape, 2.0, 0.4, 1.0, 9)
    n = new.size
    buf = torch.empty(n + offset, device="cuda")
    buf[offset:] = torch.from_numpy(new).cuda().view(-1)
    field = buf[offset:]
    s, ref = solver(p, eps), solver(p, new)
    f0 = torch.from_numpy(f0).cuda()
    s.set_populations(f0)
    before = s.get_state()
    for bad in (0.0, -1.0, 1.5, float("nan")):
        for at in {0, n // 2, n - 1}:
            worse = field.clone()
            worse[at] = bad
            with pytest.raises(VansError):
                s.update_eps(worse)
            assert torch.equal(s.get_state(), before)
    s.update_eps(field)
    assert float((s.populations() - f0.view_as(s.populations())).abs().max()) <= 2e-7
    ref.set_populations(f0)
    for h in (s, ref):
        h.step(4)
    assert float((s.populations() - ref.populations()).abs().max()) <= 2e-6


@pytest.mark.parametrize("q,shape", SHAPES)
def test_set_eps_refuses_out_of_range(q, shape):
    torch = torch_cuda()
    p, eps, _ = _case(q, shape, 4)
    s = solver(p, eps)
    for at in {0, eps.size // 2, eps.size - 1}:
        worse = torch.from_numpy(eps).cuda().view(-1).clone()
        worse[at] = 1.0001
        with pytest.raises(VansError):
            s.set_eps(worse)
        s.set_eps_async(worse)
        with pytest.raises(VansError):
            s.check()
        s.set_eps(torch.from_numpy(eps).cuda().view(-1))


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 9, 130), (1, 64, 256), (1, 33, 77)])
@pytest.mark.parametrize("every,n", [(2, 7), (5, 20), (10, 10)])
def test_emissions_between_launches_of_several_steps(shape, every, n):
    """rho and u of the last emission are those of the state that its step reads, the
    maximum is that over all emissions, and the final state is that of n steps: 2e-6 for
    the launches that group the steps otherwise, 1e-5 relative on u."""
    torch = torch_cuda()
    p, eps, f0 = _case(9, shape, 6, moving=True)
    f0 = torch.from_numpy(f0).cuda()
    a, b = solver(p, eps, Launch(2, 4, 4, 9)), solver(p, eps, Launch(4, 4, 1))
    for s in (a, b):
        s.set_populations(f0)
    rho, u, st = a.step_monitored(n, every)
    done, norm = 0, 0.0
    while done < n:
        plain = min(every - 1, n - done - 1)
        b.step(plain)
        rho_b, u_b = b.moments()
        norm = max(norm, float(u_b.double().pow(2).sum(0).sqrt().max()))
        b.step(1)
        done += plain + 1
    scale = float(u_b.abs().max())
    assert float((u - u_b).abs().max()) <= 1e-5 * scale
    assert float((rho - rho_b).abs().max()) <= 1e-6
    assert float((a.populations() - b.populations()).abs().max()) <= 2e-6
    assert abs(float(st[1]) - norm) <= 1e-5 * scale
    assert float(st[3]) == -(-n // every)
