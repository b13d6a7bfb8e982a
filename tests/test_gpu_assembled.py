"""The persistent V-cycle works from assembled coefficients (vnode.cuh), the
one-launch-per-stage cycle evaluates the operator cell by cell: one cycle of
each must agree to rounding for every pattern of fluid cells and patches
around a node (walls, corners, outflow, obstacles at both ends of the
channel and snapped to level 1), for every stabilisation form with a regular
Jacobian, and for right-hand sides that do not vanish on constrained
unknowns.  Bars: 1e-10 in FP64 and, for FP32 cycles whose own rounding is
about 2e-6, 2e-5."""
import pytest

from oracle import mesh
from tests.gpu_util import lib, rel, seeded_state

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,tol", [(0, 1e-10), (1, 2e-5)])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("L,ob,kw", [(2, (1, 1), {}), (2, (13, 1), dict(nu1=1, nu2=1)),
                                     (3, None, dict(lps_mode=1)), (3, (7, 2, 1), {}),
                                     (4, (2, 1), dict(nu1=0, nu2=3)),
                                     (3, (1, 1), dict(nu1=1, nu2=0)), (5, (2, 1), {})])
def test_assembled_cycle_matches_cell_by_cell_cycle(precision, tol, mode, L, ob, kw):
    dn = lib()
    o = ob or (-1, -1)
    common = dict(level_solve=L, precision=precision, obstacle_i0=o[0], obstacle_j0=o[1],
                  obstacle_level=1 if len(o) > 2 else 0, nu=0.007, dt=0.008, **kw)
    lev = mesh.Level(L, obstacle=ob)
    x = torch.from_numpy(seeded_state(lev, 81 + L)).cuda()
    staged = dn.Context(persistent_vcycle=0, **common)
    walk = dn.Context(persistent_vcycle=L, persistent_mode=mode, **common)
    g = torch.Generator().manual_seed(5 + L)
    b = torch.randn(lev.ndof, generator=g, dtype=torch.float64).to(staged.vdtype).cuda()
    out = []
    for c in (staged, walk):
        c.linearize(x)
        out.append(c.vcycle(L, b).double().cpu().numpy())
    assert rel(out[1], out[0]) < tol, rel(out[1], out[0])
    # the tiles wait for each other's updates one by one: the same values whatever the order
    for _ in range(20):
        assert (walk.vcycle(L, b).double().cpu().numpy() == out[1]).all()


@pytest.mark.parametrize("L,nu,dt", [(2, 0.004, 0.02), (3, 0.01, 0.005), (5, 0.0065, 0.005)])
def test_fp32_rows_act_on_differences(L, nu, dt):
    """FP32 rows are applied to differences of the iterate, so that a cycle's
    error against FP64 stays at a few of the result's own roundings (6e-8)
    instead of their amplification by a smooth pressure (1e-6 and more)."""
    dn = lib()
    lev = mesh.Level(L, obstacle=(2, 1))
    x = torch.from_numpy(seeded_state(lev, 7)).cuda()
    g = torch.Generator().manual_seed(17 + L)
    b = torch.randn(lev.ndof, generator=g, dtype=torch.float64).float()
    out = []
    for precision in (0, 1):
        c = dn.Context(level_solve=L, precision=precision, obstacle_i0=2, obstacle_j0=1, nu=nu,
                       dt=dt, persistent_vcycle=L, persistent_mode=0)
        c.linearize(x)
        out.append(c.vcycle(L, b.to(c.vdtype).cuda()).double().cpu().numpy())
    assert rel(out[1], out[0]) < 1e-6, rel(out[1], out[0])


@pytest.mark.parametrize("nu1,nu2,modes", [(2, 2, (0,)), (0, 2, (0, 1)), (1, 0, (1,))])
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
def test_batched_cycle_matches_single_cycles(precision, tol, nu1, nu2, modes):
    """Problems whose finest levels differ wait for each other's updates of no
    level but their own: every problem's cycle is that of its own context."""
    dn = lib()
    levels = (1, 3, 2, 4, 3)
    kw = [dict(level_solve=L, precision=precision, obstacle_i0=2, obstacle_j0=1, nu=0.006 + 0.001 * p,
               dt=0.01, nu1=nu1, nu2=nu2, lps_mode=modes[p % len(modes)]) for p, L in enumerate(levels)]
    B = dn.Batch([dn.default_config(**k) for k in kw])
    g = torch.Generator().manual_seed(3)
    bvec = torch.zeros(B.length, dtype=B.vdtype, device="cuda")
    single = []
    for p, L in enumerate(levels):
        lev = mesh.Level(L, obstacle=(2, 1))
        x = torch.from_numpy(seeded_state(lev, 40 + p)).cuda()
        b = torch.randn(lev.ndof, generator=g, dtype=torch.float64).to(B.vdtype).cuda()
        off = B.layout(p)[1]
        bvec[off:off + lev.ndof] = b
        B.set_state(p, x)
        c = dn.Context(persistent_vcycle=max(L, 2), persistent_mode=0, **kw[p])
        c.linearize(x)
        single.append((off, lev.ndof, c.vcycle(L, b).double().cpu().numpy()))
    B.linearize()
    first = B.vcycle(bvec).clone()
    for off, n, ref in single:
        got = first[off:off + n].double().cpu().numpy()
        assert rel(got, ref) < tol, rel(got, ref)
    for _ in range(10):
        assert torch.equal(B.vcycle(bvec), first)


@pytest.mark.parametrize("ob,more", [((2, 1), {}), (None, {}), ((1, 1), dict(nu=0.001, dt=2.0)),
                                     ((13, 1), dict(nu=0.02, dt=1e-3)),
                                     ((6, 2, 1), dict(nu=0.001, dt=0.5))])
def test_coarse_inverse_solves_the_coarse_system(ob, more):
    """The coarse inverse by elimination of node columns, checked on the device
    to 2e-12 per entry of A Ainv - 1 (the band LU takes over otherwise): with 891 unknowns the residual of a solve stays
    below 891 * 2e-12 of the right-hand side's largest entry."""
    dn = lib()
    o = ob or (-1, -1)
    kw = dict(dict(nu=0.01, dt=0.01), **more)
    c = dn.Context(level_solve=2, precision=0, obstacle_i0=o[0], obstacle_j0=o[1],
                   obstacle_level=1 if len(o) > 2 else 0, **kw)
    c.linearize(torch.from_numpy(seeded_state(mesh.Level(2, obstacle=ob), 9)).cuda())
    n = mesh.Level(1, obstacle=ob).ndof
    b = torch.randn(n, generator=torch.Generator().manual_seed(2), dtype=torch.float64).cuda()
    r = c.apply(1, c.vcycle(1, b)) - b
    assert float(r.abs().max() / b.abs().max()) < 891 * 2e-12
