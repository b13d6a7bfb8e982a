"""V-cycles at the edges of what the calls accept: very many smoothing sweeps,
linearisation points that are not finite, and waits that hit their bound."""
import pytest

from oracle import mesh
from tests.gpu_util import lib, rel, seeded_state

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nu1,nu2", [(33, 32), (0, 64), (64, 64)])
@pytest.mark.parametrize("precision,tol", [(0, 1e-10), (1, 2e-5)])
def test_batched_cycle_with_many_sweeps(precision, tol, nu1, nu2):
    """4 (nu1 + nu2) + 1 updates of a level's iterate per cycle, 257 and more: no
    cycle may take a value that the one before left behind.  Right-hand sides
    alternate, so that such a value would show.  The bars are those between the
    assembled and the cell-by-cell cycle (1e-10 in FP64, 2e-5 in FP32); FP32 results
    that differ by more, where the roundings of so many sweeps add up, may be no
    further from the FP64 cycle than the cell-by-cell FP32 cycle is."""
    dn = lib()
    levels = (2, 3)
    kw = [dict(level_solve=L, obstacle_i0=2, obstacle_j0=1, nu=0.007, dt=0.008, nu1=nu1, nu2=nu2)
          for L in levels]
    B = dn.Batch([dn.default_config(precision=precision, **k) for k in kw])
    g = torch.Generator().manual_seed(11)
    rhs = [torch.zeros(B.length, dtype=B.vdtype, device="cuda") for _ in range(2)]
    staged = []
    for p, L in enumerate(levels):
        lev = mesh.Level(L, obstacle=(2, 1))
        x = torch.from_numpy(seeded_state(lev, 50 + p)).cuda()
        B.set_state(p, x)
        off = B.layout(p)[1]
        for k, b in enumerate(rhs):
            b[off:off + lev.ndof] = torch.randn(lev.ndof, generator=g, dtype=torch.float64).cuda()
            ref = []
            for prec in (precision, 0):
                c = dn.Context(persistent_vcycle=0, precision=prec, **kw[p])
                c.linearize(x)
                v = b[off:off + lev.ndof].to(c.vdtype)
                ref.append(c.vcycle(L, v).double().cpu().numpy())
            staged.append((k, off, lev.ndof, ref))
    B.linearize()
    first = [B.vcycle(b).clone() for b in rhs]
    for k, off, n, (ref, ref64) in staged:
        got = first[k][off:off + n].double().cpu().numpy()
        assert rel(got, ref) < tol or rel(got, ref64) <= rel(ref, ref64), (rel(got, ref),
                                                                           rel(got, ref64))
    for k in range(20):
        assert torch.equal(B.vcycle(rhs[k % 2]), first[k % 2])


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("node", [(7, 5), (8, 8), (38, 19)])
def test_linearisation_at_a_non_finite_state_is_an_error(precision, node, bad):
    """A velocity that is not finite makes local matrices without an inverse, on the
    finest level only ((7, 5): a node of no coarser level) or on all of them, and
    linearize reports it, for one problem and in a batch."""
    dn = lib()
    L = 3
    lev = mesh.Level(L, obstacle=(5, 1))
    good = torch.from_numpy(seeded_state(lev, 3)).cuda()
    x = good.clone()
    x[node[1] * lev.nnx + node[0]] = bad
    kw = dict(level_solve=L, precision=precision, obstacle_i0=5, obstacle_j0=1, nu=0.01, dt=0.01)
    c = dn.Context(**kw)
    B = dn.Batch([dn.default_config(**kw), dn.default_config(**kw)])
    for tries in range(2):  # the first linearisation, and one after a good one
        with pytest.raises(dn.DnnmgError) as e:
            c.linearize(x)
        assert e.value.code == dn.ERR_NUMERICAL
        B.set_state(0, good)
        B.set_state(1, x)
        with pytest.raises(dn.DnnmgError) as e:
            B.linearize()
        assert e.value.code == dn.ERR_NUMERICAL
        B.set_state(1, good)
        B.linearize()
        c.linearize(good)


DEFAULT_POLLS = 1 << 21


def _timeout(dn, call):
    with pytest.raises(dn.DnnmgError) as e:
        call()
    assert e.value.code == dn.ERR_TIMEOUT


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
def test_cycle_whose_waits_run_out_is_reported(precision, mode):
    """With no polls allowed every wait gives up (the kernel still runs to its end):
    the next linearisation and the step itself say so, once, and cycles with the
    default bound give the same values as before."""
    dn = lib()
    L = 3
    lev = mesh.Level(L, obstacle=(2, 1))
    x = torch.from_numpy(seeded_state(lev, 5)).cuda()
    c = dn.Context(level_solve=L, precision=precision, obstacle_i0=2, obstacle_j0=1, nu=0.01, dt=0.01,
                   persistent_vcycle=L, persistent_mode=mode)
    c.linearize(x)
    b = torch.randn(lev.ndof, generator=torch.Generator().manual_seed(1),
                    dtype=torch.float64).to(c.vdtype).cuda()
    ref = c.vcycle(L, b).clone()
    c.linearize(x)  # nothing to report
    c._check(c.lib.dnnmg_vcycle_polls(c.h, 0))
    c.vcycle(L, b)
    _timeout(dn, lambda: c.linearize(x))
    c.linearize(x)  # reported once
    _timeout(dn, c.step)
    c._check(c.lib.dnnmg_vcycle_polls(c.h, DEFAULT_POLLS))
    c.linearize(x)
    assert torch.equal(c.vcycle(L, b), ref)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("graphs", [0, 1])
def test_batched_cycle_whose_waits_run_out_is_reported(precision, graphs):
    dn = lib()
    levels = (2, 3)
    B = dn.Batch([dn.default_config(level_solve=L, precision=precision, obstacle_i0=2, obstacle_j0=1,
                                    nu=0.01, dt=0.01) for L in levels])
    B._check(B.lib.dnnmg_batch_graphs(B.h, graphs))
    states = [torch.from_numpy(seeded_state(mesh.Level(L, obstacle=(2, 1)), 6 + L)).cuda()
              for L in levels]
    b = torch.randn(B.length, generator=torch.Generator().manual_seed(2),
                    dtype=torch.float64).to(B.vdtype).cuda()

    def start():
        for p, x in enumerate(states):
            B.set_state(p, x)
        B.linearize()

    start()
    off = B.layout(1)[1]
    b1 = b[off:off + mesh.Level(3).ndof].clone()
    ref, ref1 = B.vcycle(b).clone(), B.vcycle_inst(1, b1).clone()
    for _ in range(2):  # eager iterations first, then graphs
        B.step()
    B._check(B.lib.dnnmg_batch_vcycle_polls(B.h, 0))
    start()
    for call in (lambda: B.vcycle(b), lambda: B.vcycle_inst(1, b1), B.step):
        _timeout(dn, call)
    B._check(B.lib.dnnmg_batch_vcycle_polls(B.h, DEFAULT_POLLS))
    start()
    assert torch.equal(B.vcycle(b), ref) and torch.equal(B.vcycle_inst(1, b1), ref1)
    B.step()


def test_batched_fp32_stabilisation_is_rounded_once():
    """A batch scales one stabilisation table by every problem's alpha0 / nu.  At
    alpha0 / nu = 1 + 3 2^-24 (times a power of two) FP32 rounds that scale up by
    2^-24, and the table's entries (multiples of 1/6) by 2^-25: entries rounded twice
    are 8.9e-8 too large, entries rounded once at most 2^-24 = 6.0e-8.  The error
    of the FP32 cycle along its derivative to alpha0, for right-hand sides of rough
    pressures, on which the stabilisation acts; the median of eight, because other
    roundings project on it too."""
    dn = lib()
    L = 4
    lev = mesh.Level(L, obstacle=(2, 1))
    x = torch.from_numpy(seeded_state(lev, 8)).cuda()
    cons = torch.from_numpy(lev.cons).cuda()
    alpha0, eta = 0.125 * (1 + 3 * 2.0 ** -24), 1e-3
    kw = dict(level_solve=L, obstacle_i0=2, obstacle_j0=1, nu=2.0 ** -7, dt=2.0 ** -7, lps_mode=1)
    exact, moved = (dn.Context(precision=0, alpha0=a, **kw) for a in (alpha0, alpha0 * (1 + eta)))
    for c in (exact, moved):
        c.linearize(x)
    B = dn.Batch([dn.default_config(precision=1, alpha0=alpha0, **kw)])
    B.set_state(0, x)
    B.linearize()
    along = []
    for seed in range(8):
        g = torch.Generator().manual_seed(seed)
        rough = torch.zeros(lev.ndof, dtype=torch.float64, device="cuda")
        rough[2 * lev.nn:] = torch.randn(lev.nn, generator=g, dtype=torch.float64).cuda()
        rough[cons] = 0
        b = torch.zeros(B.length, device="cuda")
        b[: lev.ndof] = exact.apply(L, rough).float()
        ref = exact.vcycle(L, b[: lev.ndof].double())
        deriv = (moved.vcycle(L, b[: lev.ndof].double()) - ref) / eta
        err = B.vcycle(b)[: lev.ndof].double() - ref
        along.append(abs(float(err @ deriv / (deriv @ deriv))))
    assert sorted(along)[4] < 2.0 ** -24, along


@pytest.mark.parametrize("L,precision,tol", [(6, 0, 1e-10), (6, 1, 2e-5), (7, 1, 2e-5), (8, 1, 2e-5)])
def test_persistent_cycle_of_large_levels(L, precision, tol):
    """Where a level's tiles outnumber the warps and its index arithmetic grows (4.2 M
    nodes on level 8): the persistent cycle against that of one launch per stage, with
    the bars they have on the smaller levels."""
    dn = lib()
    nnx, nny = (16 << L) + 1, (4 << L) + 1
    y = torch.linspace(0, 1, nny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.linspace(0, 4, nnx, dtype=torch.float64, device="cuda")[None, :]
    s = torch.zeros(3, nny, nnx, dtype=torch.float64, device="cuda")
    s[0] = 6 * y * (1 - y) * (1 + 0.2 * torch.sin(2 * x))
    s[1] = 0.2 * torch.sin(3 * x) * torch.sin(3.14159265358979 * y)
    g = torch.Generator(device="cuda").manual_seed(L)
    b = torch.randn(s.numel(), generator=g, dtype=torch.float64, device="cuda")
    common = dict(level_solve=L, precision=precision, obstacle_i0=3, obstacle_j0=1, nu=0.0065,
                  dt=0.005, gmres_m=2)
    out = []
    for kw in (dict(persistent_vcycle=0), dict(persistent_vcycle=L, persistent_mode=0)):
        c = dn.Context(**common, **kw)
        c.linearize(s.reshape(-1))
        assert c.lib.dnnmg_vcycle_split(c.h) == kw["persistent_vcycle"]
        out.append(c.vcycle(L, b.to(c.vdtype)).double())
        again = c.vcycle(L, b.to(c.vdtype)).double()
        assert torch.equal(again, out[-1])
        c.close()
    assert 0 < float((out[1] - out[0]).norm() / out[0].norm()) < tol
