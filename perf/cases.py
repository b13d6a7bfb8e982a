"""The calls that a program makes of this library, with their sizes, inputs and 64-bit results.

A case is a dict of plain values.  Its "kind" is one of

  infer     one recurrent step of the patch network over P patches
            (Context.patch_infer): the network's share of a time step;
  grad      loss and gradient of a training batch (dnnmg_train_grad), for a
            program with its own optimiser;
  train     one Adam step on a batch (Context.train_step) and the new weights;
  vcycle    one V(2,2) cycle (Context.vcycle): the preconditioner, the call
            most time is spent in;
  newton    the linear algebra of one Newton step for a program with its own
            Krylov loop: residual, linearisation, V-cycle, operator;
  batch     one V-cycle of many channels at once (Batch.vcycle);
  plain     one classical time step (Context.step(PLAIN));
  dnnmg     one time step with the network's correction (Context.step(NET)).

Channel sizes, obstacle positions, viscosities, time steps and network sizes
are those of the repository's benchmark and tests.  Level l of the channel
has (16 * 2^l) x (4 * 2^l) cells.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2106_07687_gb300 import dnnmg

MLP = 128        # width of the network's hidden dense layer
LEARNING_RATE = 1e-3


def listed():
    return [
        # the 64x16 channel's 960 fluid patches: a handful of tiles, all latency
        dict(name="infer_960", kind="infer", patches=960, hidden=64, layers=2, replaced=1),
        # every fluid cell of the 512x128 channel, the benchmark's step
        dict(name="infer_61440", kind="infer", patches=61440, hidden=64, layers=2, replaced=1),
        # two replaced levels (104 inputs, 50 outputs): the large workload's network
        dict(name="infer_two_levels", kind="infer", patches=61440, hidden=64, layers=2, replaced=2),
        # a small network on a short batch whose rows do not fill the last tile
        dict(name="grad_32x2_ragged", kind="grad", batch=1040, steps=7, hidden=32, layers=2,
             replaced=1),
        # the benchmark's training step: 19,456 sequences of 10 steps
        dict(name="train_64x2", kind="train", batch=19456, steps=10, hidden=64, layers=2,
             replaced=1),
        # the 128x32 channel in FP64: the smallest configured solver
        dict(name="vcycle_fp64_l3", kind="vcycle", level=3, precision=0, obstacle=2, nu=0.01,
             dt=0.01),
        # 512x128 in mixed precision: the cycle of the benchmark's step
        dict(name="vcycle_mixed_l5", kind="vcycle", level=5, precision=1, obstacle=3, nu=0.0065,
             dt=0.005),
        # 1024x256 in mixed precision: the cycle of the fine solve and of the corpus
        dict(name="vcycle_mixed_l6", kind="vcycle", level=6, precision=1, obstacle=2, nu=0.0065,
             dt=0.005),
        # one Newton step's linear algebra on the 256x64 channel in FP64
        dict(name="newton_fp64_l4", kind="newton", level=4, precision=0, obstacle=3, nu=0.01,
             dt=0.01),
        # twelve channels of uneven size in one batch, in mixed precision
        dict(name="batch_mixed", kind="batch", count=12, level=5, precision=1, nu=0.01, dt=0.005),
        # a classical FP64 time step of the 128x32 channel: the smallest whole call
        dict(name="plain_step_fp64_l3", kind="plain", level=3, precision=0, obstacle=2, nu=0.01,
             dt=0.01),
        # the benchmark's whole step: solve on 512x128, network on 1024x256
        dict(name="dnnmg_step_l5", kind="dnnmg", level=5, precision=1, obstacle=3, nu=0.0065,
             dt=0.005),
    ]


def draw(rng):
    kind = rng.choice(["infer", "infer", "grad", "train", "vcycle", "vcycle", "vcycle", "newton",
                       "batch"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    net = dict(hidden=rng.choice([32, 64]), layers=rng.choice([1, 2, 3]), replaced=1)
    if kind == "infer":
        if net["layers"] < 3 and rng.random() < 0.3:
            net["replaced"] = 2
        return dict(kind=kind, patches=log_int(1, 61440), **net)
    if kind in ("grad", "train"):
        return dict(kind=kind, batch=16 * log_int(1, 800), steps=rng.randint(1, 10), **net)
    phys = dict(nu=round(rng.uniform(0.004, 0.02), 4), dt=rng.choice([0.005, 0.01, 0.02]))
    precision = rng.choice([0, 1, 1])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 10), level=rng.choice([3, 4]),
                    precision=precision, **phys)
    top = 5 if precision == 0 else 6
    if kind == "newton":
        top -= 1
    return dict(kind=kind, level=rng.randint(2, top), precision=precision,
                obstacle=rng.choice([-1, 2, 3, 5, 8]), **phys)


# ---- inputs -------------------------------------------------------------------


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * salt + 7919 * int(seed) + 11)
    return g


def _dims(level):
    nx, ny = 16 << level, 4 << level
    return nx, ny, nx + 1, ny + 1


def _masks(level, obstacle):
    """(solid [ny][nx], velocity-Dirichlet [nny][nnx], pressure-fixed [nny][nnx])
    of the channel with the square of 2x2 level-0 cells at cell (obstacle, 1)."""
    nx, ny, nnx, nny = _dims(level)
    solid = torch.zeros(ny, nx, dtype=torch.bool, device="cuda")
    if obstacle >= 0:
        solid[1 << level:3 << level, obstacle << level:(obstacle + 2) << level] = True
    touch_solid = torch.zeros(nny, nnx, dtype=torch.bool, device="cuda")
    touch_fluid = torch.zeros_like(touch_solid)
    for dj in (0, 1):
        for di in (0, 1):
            touch_solid[dj:dj + ny, di:di + nx] |= solid
            touch_fluid[dj:dj + ny, di:di + nx] |= ~solid
    vdir = touch_solid
    vdir[:, 0] = True
    vdir[0, :] = True
    vdir[-1, :] = True
    return solid, vdir, ~touch_fluid


def _flow(level, obstacle, seed, salt=0, amp=0.3):
    """A state [3][nny][nnx] (FP64): the channel's parabola and a few smooth
    modes, the boundary values imposed, and a rough pressure."""
    _, _, nnx, nny = _dims(level)
    g = _gen(seed, salt + 1)
    y = torch.linspace(0, 1, nny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.linspace(0, 4, nnx, dtype=torch.float64, device="cuda")[None, :]
    s = torch.zeros(3, nny, nnx, dtype=torch.float64, device="cuda")
    s[0] = 6 * y * (1 - y)
    c = torch.randn(3, 2, 4, generator=g, dtype=torch.float64, device="cuda").cpu()
    for kx in range(1, 4):
        for ky in range(1, 3):
            a, b, e, f = (float(v) for v in c[kx - 1, ky - 1])
            s[0] += amp * a * torch.sin(kx * math.pi * x / 4 + e) * torch.sin(ky * math.pi * y)
            s[1] += amp * b * torch.sin(kx * math.pi * x / 4 + f) * torch.sin(ky * math.pi * y)
    s[2] = 0.1 * torch.randn(nny, nnx, generator=g, dtype=torch.float64, device="cuda")
    _, vdir, pfix = _masks(level, obstacle)
    s[0][vdir] = 0
    s[1][vdir] = 0
    s[0][:, 0] = (6 * y * (1 - y))[:, 0]
    s[2][pfix] = 0
    return s


def _rhs(level, obstacle, seed, dtype, salt=0):
    """A vector like a Krylov basis vector: unit norm, zero on constrained unknowns."""
    _, _, nnx, nny = _dims(level)
    b = torch.randn(3, nny, nnx, generator=_gen(seed, salt + 2), dtype=torch.float64,
                    device="cuda")
    _, vdir, pfix = _masks(level, obstacle)
    b[:2, vdir] = 0
    b[2, pfix] = 0
    return (b / b.norm()).reshape(-1).to(dtype)


def _net_dims(case):
    k = 2 ** case["replaced"] + 1
    return 4 * k * k + 4, 2 * k * k


def _weights(case, seed, scale=0.2):
    c_in, c_out = _net_dims(case)
    m, n = case["hidden"], case["layers"]
    count = sum(3 * m * (c_in if l == 0 else m) + 3 * m * m + 6 * m for l in range(n))
    count += MLP * m + MLP + c_out * MLP + c_out
    w = torch.rand(count, generator=_gen(seed, 3), device="cuda") * 2 - 1
    return (scale * w).cpu()


def _batch_data(case, seed):
    c_in, c_out = _net_dims(case)
    B, T = case["batch"], case["steps"]
    g = _gen(seed, 4)
    X = torch.randn(B, T, c_in, generator=g, device="cuda").to(torch.bfloat16)
    Y = 0.3 * torch.randn(B, T, c_out, generator=g, device="cuda")
    return X, Y


def _patch_data(case, seed):
    c_in, _ = _net_dims(case)
    P, m, n = case["patches"], case["hidden"], case["layers"]
    g = _gen(seed, 5)
    x = torch.randn(P, c_in, generator=g, device="cuda").to(torch.bfloat16)
    h = torch.tanh(0.5 * torch.randn(n, P, m, generator=g, device="cuda"))
    return x, h


def _batch_levels(case):
    return [case["level"] - (2 - p % 3) % 3 for p in range(case["count"])]


def _context(case, **more):
    return dnnmg.Context(level_solve=case["level"], precision=case["precision"],
                         obstacle_i0=case["obstacle"], obstacle_j0=1 if case["obstacle"] >= 0 else -1,
                         nu=case["nu"], dt=case["dt"], **more)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "infer":
        s["ctx"] = dnnmg.Context(level_solve=2, replaced_levels=case["replaced"],
                                 hidden=case["hidden"], gru_layers=case["layers"])
        s["ctx"].set_weights(_weights(case, seed))
        s["x"], s["h"] = _patch_data(case, seed)
    elif kind in ("grad", "train"):
        s["ctx"] = dnnmg.Context(level_solve=2, hidden=case["hidden"], gru_layers=case["layers"],
                                 train_batch=case["batch"], train_seq=case["steps"])
        s["ctx"].set_weights(_weights(case, seed))
        s["X"], s["Y"] = _batch_data(case, seed)
        s["grad"] = torch.empty(s["ctx"].num_params(), device="cuda")
    elif kind == "vcycle":
        s["ctx"] = _context(case)
        s["ctx"].linearize(_flow(case["level"], case["obstacle"], seed).reshape(-1))
        s["b"] = _rhs(case["level"], case["obstacle"], seed, s["ctx"].vdtype)
    elif kind == "newton":
        s["ctx"] = _context(case)
        x = _flow(case["level"], case["obstacle"], seed).reshape(-1)
        s["ctx"].linearize(x)  # a program's previous Newton step
        s["x"] = x
        s["f"] = _old_rhs(case, _flow(case["level"], case["obstacle"], seed, salt=50))
    elif kind == "batch":
        levels = _batch_levels(case)
        cfgs = [dnnmg.default_config(level_solve=l, precision=case["precision"],
                                     obstacle_i0=2 + p % 2, obstacle_j0=1,
                                     nu=case["nu"] * (1 + 0.1 * (p % 4)), dt=case["dt"])
                for p, l in enumerate(levels)]
        B = s["batch"] = dnnmg.Batch(cfgs)
        s["b"] = torch.zeros(B.length, dtype=B.vdtype, device="cuda")
        for p, l in enumerate(levels):
            B.set_state(p, _flow(l, 2 + p % 2, seed, salt=60 + p).reshape(-1))
            lev, off = B.layout(p)
            v = _rhs(l, 2 + p % 2, seed, B.vdtype, salt=90 + p)
            s["b"][off:off + v.numel()] = v
        B.linearize()
    elif kind == "plain":
        s["ctx"] = _context(case)
        s["ctx"].set_state(_flow(case["level"], case["obstacle"], seed, amp=0.1).reshape(-1))
        for _ in range(5):  # past the start's transient
            s["ctx"].step(dnnmg.PLAIN)
    elif kind == "dnnmg":
        # a flow that has developed over some larger steps
        start = _context(dict(case, dt=0.02))
        start.set_state(_flow(case["level"], case["obstacle"], seed, amp=0.1).reshape(-1))
        for _ in range(15):
            start.step(dnnmg.PLAIN)
        s["ctx"] = _context(case)
        s["ctx"].set_state(start.get_state())
        start.close()
        # a trained network's corrections are a few thousandths of the velocity
        net = dict(hidden=64, layers=2, replaced=1)
        w = _weights(net, seed, 0.1)
        last = MLP * 18 + 18
        w[-last:] *= 0.01
        s["ctx"].set_weights(w)
        for _ in range(5):  # the network's memory has filled
            s["ctx"].step(dnnmg.NET)
    else:
        raise ValueError(kind)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "infer":
        return {"out": s["ctx"].patch_infer(s["x"], s["h"]), "h": s["h"]}
    if kind == "grad":
        ctx, loss = s["ctx"], ctypes.c_float()
        ctx._check(ctx.lib.dnnmg_train_grad(
            ctx.h, s["X"].data_ptr(), s["Y"].data_ptr(), case["batch"], case["steps"],
            s["grad"].data_ptr(), ctypes.byref(loss)))
        return {"grad": s["grad"], "loss": np.float32(loss.value)}
    if kind == "train":
        loss = s["ctx"].train_step(s["X"], s["Y"], case["batch"], case["steps"], LEARNING_RATE)
        return {"weights": s["ctx"].get_weights(), "loss": np.float32(loss)}
    if kind == "vcycle":
        return {"x": s["ctx"].vcycle(case["level"], s["b"])}
    if kind == "newton":
        ctx, lev = s["ctx"], case["level"]
        r = ctx.residual(s["x"], s["f"])
        ctx.linearize(s["x"])
        z = ctx.vcycle(lev, r.to(ctx.vdtype))
        return {"r": r, "z": z, "Az": ctx.apply(lev, z)}
    if kind == "batch":
        return {"x": s["batch"].vcycle(s["b"])}
    if kind == "plain":
        s["ctx"].step(dnnmg.PLAIN)
        return {"x": s["ctx"].get_state()}
    # the fields as a program writes them to its output file, in single precision
    s["ctx"].step(dnnmg.NET)
    return {"x": s["ctx"].get_state().float(), "v": s["ctx"].get_fine_velocity().float()}


# ---- what a pass cannot do without ----------------------------------------------


def _macs(case):
    c_in, c_out = _net_dims(case)
    m = case["hidden"]
    return sum(3 * m * (c_in if l == 0 else m) + 3 * m * m for l in range(case["layers"])) \
        + MLP * m + c_out * MLP


def _nodes(level):
    _, _, nnx, nny = _dims(level)
    return nnx * nny


def _cycle_work(level, precision):
    """The vectors, the linearisation velocities and the local inverses read once
    each; 16 colour passes of assembled rows and 12x12 products per level."""
    size = 8 if precision == 0 else 4
    by, fl = size * 6 * _nodes(level) + 8 * 891 ** 2, 2 * 891 ** 2
    for l in range(2, level + 1):
        nx, ny, _, _ = _dims(l)
        by += size * (2 * _nodes(l) + 144 * nx * ny)
        fl += 2 * 17 * 97 * _nodes(l) + 4 * 2 * 144 * nx * ny
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "infer":
        c_in, c_out = _net_dims(case)
        P, mn = case["patches"], case["hidden"] * case["layers"]
        return {"bytes": P * (2 * c_in + 8 * mn + 4 * c_out) + 2 * _macs(case),
                "flops": 2 * P * _macs(case)}
    if kind in ("grad", "train"):
        c_in, c_out = _net_dims(case)
        rows = case["batch"] * case["steps"]
        skipped = 3 * case["hidden"] * c_in  # the inputs need no gradient
        return {"bytes": rows * (2 * c_in + 4 * c_out) + 8 * _macs(case),
                "flops": 2 * rows * (3 * _macs(case) - skipped)}
    if kind == "batch":
        got = [_cycle_work(l, case["precision"]) for l in _batch_levels(case)]
        return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}
    by, fl = _cycle_work(case["level"], case["precision"])
    n = _nodes(case["level"])
    if kind == "newton":  # two operators, and the local inverses written before they are read
        cells = sum(_dims(l)[0] * _dims(l)[1] for l in range(2, case["level"] + 1))
        return {"bytes": by + 8 * 9 * n, "flops": fl + 2 * 2 * 97 * n + 2 * 12 ** 3 * cells}
    if kind in ("plain", "dnnmg"):
        its = 6  # two Newton steps of three V-cycles
        extra = 0
        if kind == "dnnmg":
            net = dict(patches=15 * _dims(case["level"])[0] * _dims(case["level"])[1] // 16,
                       hidden=64, layers=2, replaced=1, kind="infer")
            extra = work(net)
            return {"bytes": its * by + extra["bytes"] + 8 * 6 * _nodes(case["level"] + 1),
                    "flops": its * fl + extra["flops"]}
        return {"bytes": its * by, "flops": its * fl}
    return {"bytes": by, "flops": fl}


# ---- the same in 64 bits ------------------------------------------------------------


def _net_params(case, seed):
    c_in, c_out = _net_dims(case)
    m, flat, o, p = case["hidden"], _weights(case, seed).double().cuda(), 0, []
    shapes = []
    for l in range(case["layers"]):
        shapes += [(3 * m, c_in if l == 0 else m), (3 * m, m), (3 * m,), (3 * m,)]
    shapes += [(MLP, m), (MLP,), (c_out, MLP), (c_out,)]
    for sh in shapes:
        k = int(np.prod(sh))
        p.append(flat[o:o + k].reshape(sh).clone())
        o += k
    return p


def _net_step(case, p, x, h):
    """One step of the stacked GRUs and the dense head; (output, new states)."""
    m, new = case["hidden"], []
    for l in range(case["layers"]):
        wi, wh, bi, bh = p[4 * l:4 * l + 4]
        gi, gh = x @ wi.T + bi, h[l] @ wh.T + bh
        r = torch.sigmoid(gi[:, :m] + gh[:, :m])
        z = torch.sigmoid(gi[:, m:2 * m] + gh[:, m:2 * m])
        n = torch.tanh(gi[:, 2 * m:] + r * gh[:, 2 * m:])
        x = (1 - z) * n + z * h[l]
        new.append(x)
    w1, b1, w2, b2 = p[-4:]
    return torch.relu(x @ w1.T + b1) @ w2.T + b2, new


def _net_gradient(case, seed):
    """(flat gradient, loss) of the mean squared error, in pieces of the batch."""
    X, Y = _batch_data(case, seed)
    p = [q.requires_grad_(True) for q in _net_params(case, seed)]
    B, T = case["batch"], case["steps"]
    total = 0.0
    for b0 in range(0, B, 4096):
        x, y = X[b0:b0 + 4096].double(), Y[b0:b0 + 4096].double()
        h = [torch.zeros(x.shape[0], case["hidden"], dtype=torch.float64, device="cuda")
             for _ in range(case["layers"])]
        loss = 0.0
        for t in range(T):
            out, h = _net_step(case, p, x[:, t], h)
            loss = loss + ((out - y[:, t]) ** 2).sum()
        loss = loss / Y.numel()
        loss.backward()
        total += float(loss.detach())
    return torch.cat([q.grad.reshape(-1) for q in p]), total


class _Level:
    """One level's operator in FP64: 3x3 node stencils of 3x3 blocks, K[c][d][dj][di]
    at every node, and the 5x5 stencil S[dj][di] of the pressure stabilisation."""

    def __init__(self, level, obstacle, nu, dt, vel):
        nx, ny, nnx, nny = _dims(level)
        self.nx, self.ny, self.nnx, self.nny = nx, ny, nnx, nny
        h = 4.0 / nx
        opts = dict(dtype=torch.float64, device="cuda")
        self.solid, vdir, pfix = _masks(level, obstacle)
        fluid = (~self.solid).double()
        self.free = torch.stack([~vdir, ~vdir, ~pfix]).double()
        g = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0))
        phi, dx, dy = np.zeros((4, 4)), np.zeros((4, 4)), np.zeros((4, 4))
        for q in range(4):
            gx, gy = g[q & 1], g[q >> 1]
            for a in range(4):
                fx, sx = (gx, 1.0) if a & 1 else (1 - gx, -1.0)
                fy, sy = (gy, 1.0) if a >> 1 else (1 - gy, -1.0)
                phi[q, a], dx[q, a], dy[q, a] = fx * fy, sx * fy / h, fx * sy / h
        w = 0.25 * h * h
        mass = w * phi.T @ phi
        stiff = w * (dx.T @ dx + dy.T @ dy)
        self.E, self.Dx, self.Dy = mass / dt + nu * stiff, w * phi.T @ dx, w * phi.T @ dy
        self.phi, self.dx, self.dy, self.w = (torch.tensor(v, **opts) for v in (phi, dx, dy, w))
        self.fluid, self.mass = fluid, mass
        if vel is not None:
            self._assemble(vel, opts)
        # stabilisation: alpha kappa^T K9 kappa on the 2x2-cell patches
        pi = np.zeros((9, 9))
        for t in range(3):
            for s_ in range(3):
                for ct in (0, 2):
                    for cs in (0, 2):
                        pi[s_ + 3 * t, cs + 3 * ct] = (1 - abs(s_ - cs) / 2) * (1 - abs(t - ct) / 2)
        k9 = np.zeros((9, 9))
        for c in range(4):
            loc = [((c & 1) + (a & 1)) + 3 * ((c >> 1) + (a >> 1)) for a in range(4)]
            k9[np.ix_(loc, loc)] += stiff
        kap = np.eye(9) - pi
        s9 = 0.1 * h * h / nu * kap.T @ k9 @ kap
        patch = fluid[::2, ::2]
        self.S = torch.zeros(5, 5, nny, nnx, **opts)
        for a in range(9):
            for b in range(9):
                at = self.S[b // 3 - a // 3 + 2, b % 3 - a % 3 + 2]
                ax, ay = a % 3, a // 3
                at[ay:ay + ny - 1:2, ax:ax + nx - 1:2] += s9[a, b] * patch

    def _cell(self, f):
        return torch.stack([f[(a >> 1):(a >> 1) + self.ny, (a & 1):(a & 1) + self.nx]
                            for a in range(4)])

    def _assemble(self, vel, opts):
        ub, vb = self._cell(vel[0]), self._cell(vel[1])

        def at_gauss(m, f):
            return torch.einsum("qa,ayx->qyx", m, f)

        U, V = at_gauss(self.phi, ub), at_gauss(self.phi, vb)
        grads = [[at_gauss(d, f) for d in (self.dx, self.dy)] for f in (ub, vb)]
        self.K = torch.zeros(3, 3, 3, 3, self.nny, self.nnx, **opts)
        for a in range(4):
            for b in range(4):
                conv = sum(self.w * self.phi[q, a] * (self.dx[q, b] * U[q] + self.dy[q, b] * V[q])
                           for q in range(4))
                at = (slice(None), slice(None), (b >> 1) - (a >> 1) + 1, (b & 1) - (a & 1) + 1,
                      slice(a >> 1, (a >> 1) + self.ny), slice(a & 1, (a & 1) + self.nx))
                K = self.K[at]
                for c in range(2):
                    K[c, c] += (self.E[a, b] + conv) * self.fluid
                    for d in range(2):
                        K[c, d] += self.fluid * sum(
                            self.w * self.phi[q, a] * self.phi[q, b] * grads[c][d][q]
                            for q in range(4))
                K[0, 2] -= self.Dx[b, a] * self.fluid
                K[1, 2] -= self.Dy[b, a] * self.fluid
                K[2, 0] += self.Dx[a, b] * self.fluid
                K[2, 1] += self.Dy[a, b] * self.fluid

    def stabilise(self, p):
        pp = torch.nn.functional.pad(p, (2, 2, 2, 2))
        return sum(self.S[j, i] * pp[j:j + self.nny, i:i + self.nnx]
                   for j in range(5) for i in range(5))

    def apply(self, w):
        """Identity rows and columns on constrained unknowns."""
        wf = torch.nn.functional.pad(w * self.free, (1, 1, 1, 1))
        y = torch.zeros_like(w)
        for j in range(3):
            for i in range(3):
                v = wf[:, j:j + self.nny, i:i + self.nnx]
                for c in range(3):
                    y[c] += (self.K[c, :, j, i] * v).sum(0)
        y[2] += self.stabilise(w[2] * self.free[2])
        return y * self.free + w * (1 - self.free)

    def blocks(self):
        """The 12x12 restriction of the operator to every cell's unknowns."""
        A = torch.zeros(self.ny, self.nx, 12, 12, dtype=torch.float64, device="cuda")
        fr = torch.stack([self._cell(self.free[c]) for c in range(3)])
        for a in range(4):
            ya, xa = slice(a >> 1, (a >> 1) + self.ny), slice(a & 1, (a & 1) + self.nx)
            for b in range(4):
                j, i = (b >> 1) - (a >> 1), (b & 1) - (a & 1)
                for c in range(3):
                    for d in range(3):
                        v = self.K[c, d, j + 1, i + 1, ya, xa]
                        if c == 2 and d == 2:
                            v = v + self.S[j + 2, i + 2, ya, xa]
                        v = v * fr[c, a] * fr[d, b]
                        if c == d and a == b:
                            v = v + 1 - fr[c, a]
                        A[:, :, 4 * c + a, 4 * d + b] = v
        return A

    def dense(self):
        n = 3 * self.nny * self.nnx
        eye = torch.eye(n, dtype=torch.float64, device="cuda")
        return torch.stack([self.apply(eye[k].reshape(3, self.nny, self.nnx)).reshape(-1)
                            for k in range(n)], dim=1)

    def operator(self, x):
        """The nonlinear operator's rows at x."""
        c = [self._cell(x[k]) for k in range(3)]
        y = torch.zeros_like(x)
        U, V = (torch.einsum("qa,ayx->qyx", self.phi, f) for f in c[:2])
        for k in range(2):
            gx, gy = (torch.einsum("qa,ayx->qyx", d, c[k]) for d in (self.dx, self.dy))
            for a in range(4):
                D = self.Dx if k == 0 else self.Dy
                row = sum(float(self.E[a, b]) * c[k][b] - float(D[b, a]) * c[2][b]
                          for b in range(4))
                row = row + sum(self.w * self.phi[q, a] * (U[q] * gx[q] + V[q] * gy[q])
                                for q in range(4))
                div = sum(float(D[a, b]) * c[k][b] for b in range(4))
                at = (slice(a >> 1, (a >> 1) + self.ny), slice(a & 1, (a & 1) + self.nx))
                y[k][at] += row * self.fluid
                y[2][at] += div * self.fluid
        y[2] += self.stabilise(x[2])
        return y

    def old_rhs(self, x, dt):
        f = torch.zeros_like(x)
        for k in range(2):
            c = self._cell(x[k])
            for a in range(4):
                row = sum(float(self.mass[a, b]) / dt * c[b] for b in range(4))
                f[k][(a >> 1):(a >> 1) + self.ny, (a & 1):(a & 1) + self.nx] += row * self.fluid
        return f


def _old_rhs(case, x_old):
    lev = _Level(case["level"], case["obstacle"], case["nu"], case["dt"], None)
    return lev.old_rhs(x_old, case["dt"]).reshape(-1)


def _exact_cycle(level, obstacle, nu, dt, vel, b):
    """One V(2,2) cycle with the four-colour cell smoother (damping 0.8)."""
    lev = _Level(level, obstacle, nu, dt, vel)
    if level == 1:
        return torch.linalg.solve(lev.dense(), b.reshape(-1)).reshape(b.shape)
    inv = torch.linalg.inv(lev.blocks())
    x = torch.zeros_like(b)

    def smooth():
        for colour in range(4):
            cx, cy = colour & 1, colour >> 1
            d = b - lev.apply(x)
            loc = torch.stack([lev._cell(d[c])[a] for c in range(3) for a in range(4)], dim=-1)
            u = 0.8 * torch.einsum("yxij,yxj->yxi", inv[cy::2, cx::2], loc[cy::2, cx::2])
            u = u * (~lev.solid[cy::2, cx::2]).double()[..., None]
            ny, nx = u.shape[:2]
            for c in range(3):
                for a in range(4):
                    y0, x0 = cy + (a >> 1), cx + (a & 1)
                    x[c][y0:y0 + 2 * ny - 1:2, x0:x0 + 2 * nx - 1:2] += u[..., 4 * c + a]

    smooth()
    smooth()
    d = (b - lev.apply(x)) * lev.free
    # bilinear transfers on free unknowns
    k1 = torch.tensor([0.5, 1.0, 0.5], dtype=torch.float64, device="cuda")
    k2 = (k1[:, None] * k1[None, :])[None, None]
    bc = torch.nn.functional.conv2d(d[:, None], k2, stride=2, padding=1)[:, 0]
    _, vdir, pfix = _masks(level - 1, obstacle)
    cfree = torch.stack([~vdir, ~vdir, ~pfix]).double()
    xc = _exact_cycle(level - 1, obstacle, nu, dt, vel[:, ::2, ::2], bc * cfree) * cfree
    x += torch.nn.functional.conv_transpose2d(xc[:, None], k2, stride=2, padding=1)[:, 0] * lev.free
    smooth()
    smooth()
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "infer":
        x, h = _patch_data(case, seed)
        out, new = _net_step(case, _net_params(case, seed), x.double(), list(h.double()))
        return {"out": out, "h": torch.stack(new)}
    if kind == "grad":
        g, loss = _net_gradient(case, seed)
        return {"grad": g, "loss": loss}
    if kind == "train":
        g, loss = _net_gradient(case, seed)
        w = _weights(case, seed).double().cuda()
        # the first Adam step: both bias-corrected moments are those of g
        return {"weights": w - LEARNING_RATE * g / (g.abs() + 1e-8), "loss": loss}
    if kind in ("vcycle", "newton"):
        level, ob = case["level"], case["obstacle"]
        _, _, nnx, nny = _dims(level)
        x = _flow(level, ob, seed)
        args = (level, ob, case["nu"], case["dt"], x[:2])
        if kind == "vcycle":
            dtype = torch.float64 if case["precision"] == 0 else torch.float32
            b = _rhs(level, ob, seed, dtype).double().reshape(3, nny, nnx)
            return {"x": _exact_cycle(*args, b).reshape(-1)}
        lev = _Level(*args)
        r = (lev.old_rhs(_flow(level, ob, seed, salt=50), case["dt"]) - lev.operator(x)) * lev.free
        z = _exact_cycle(*args, r)
        return {"r": r.reshape(-1), "z": z.reshape(-1), "Az": lev.apply(z).reshape(-1)}
    if kind == "batch":
        dtype = torch.float64 if case["precision"] == 0 else torch.float32
        out, end = [], 0
        for p, l in enumerate(_batch_levels(case)):
            _, _, nnx, nny = _dims(l)
            ob = 2 + p % 2
            b = _rhs(l, ob, seed, dtype, salt=90 + p).double().reshape(3, nny, nnx)
            vel = _flow(l, ob, seed, salt=60 + p)[:2]
            x = _exact_cycle(l, ob, case["nu"] * (1 + 0.1 * (p % 4)), case["dt"], vel, b)
            # every problem's part of the vector is padded to 1024 elements
            x = torch.nn.functional.pad(x.reshape(-1), (0, -x.numel() % 1024))
            out.append(x)
        return {"x": torch.cat(out)}
    return None  # a whole step iterates to a tolerance
