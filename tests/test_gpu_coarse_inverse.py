"""Both ways to the coarse inverse: elimination of node columns, and the banded LU
that takes over where the elimination's check (the componentwise backward error
of one product with a vector of signs, 2e-12) refuses it."""
import numpy as np
import pytest

from oracle import mesh
from tests.gpu_util import lib, seeded_state

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context(dn, ob, nu, dt, amp, precision=0):
    o = ob or (-1, -1)
    c = dn.Context(level_solve=2, precision=precision, obstacle_i0=o[0], obstacle_j0=o[1],
                   obstacle_level=1 if len(o) > 2 else 0, nu=nu, dt=dt, persistent_vcycle=0)
    assert c.lib.dnnmg_coarse_lu(c.h) == -1
    c.linearize(torch.from_numpy(seeded_state(mesh.Level(2, obstacle=ob), 9, amp=amp)).cuda())
    return c


@pytest.mark.parametrize("ob,nu,dt,amp,lu", [
    ((2, 1), 0.01, 0.01, 0.3, 0), ((13, 1), 0.004, 0.02, 0.3, 0), (None, 0.02, 0.005, 0.3, 0),
    ((2, 1), 1e-4, 2.0, 3.0, 1), ((2, 1), 1e-5, 20.0, 0.3, 1)])
def test_coarse_inverse_by_either_way(ob, nu, dt, amp, lu):
    """Ordinary flows take the elimination, strong convection at large steps the LU.
    Either inverse X has columns of backward error 2e-12 at most (the check's
    tolerance; the LU's is smaller), so that |A X b - b| stays below 2e-12
    |A| |A^-1| |b| plus the product's own rounding (891 units of 1.1e-16 of |A| |X| |b|);
    five times that here, because the check's vector is only one."""
    dn = lib()
    c = _context(dn, ob, nu, dt, amp)
    assert c.lib.dnnmg_coarse_lu(c.h) == lu
    n = mesh.Level(1, obstacle=ob).ndof
    A = np.empty((n, n))
    e = torch.zeros(n, dtype=torch.float64, device="cuda")
    for k in range(n):
        e.zero_()
        e[k] = 1.0
        A[:, k] = c.apply(1, e).cpu().numpy()
    spread = np.abs(A) @ np.abs(np.linalg.inv(A))
    for seed in range(3):
        b = np.random.default_rng(seed).standard_normal(n)
        x = c.vcycle(1, torch.from_numpy(b).cuda()).cpu().numpy()
        assert (np.abs(A @ x - b) <= 5 * (2e-12 + 1e-13) * (spread @ np.abs(b))).all()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("i0,lu", [(6, 0), (7, 1)])
def test_part_solid_patches_take_the_lu(precision, i0, lu):
    """A square snapped to level 1 at an odd offset leaves part-solid patches there,
    whose column blocks can be singular; at an even offset they are whole."""
    dn = lib()
    c = _context(dn, (i0, 2, 1), 0.01, 0.01, 0.3, precision)
    assert c.lib.dnnmg_coarse_lu(c.h) == lu
