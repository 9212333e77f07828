"""Performance cases: the calls a user's program makes, over the sizes and options it makes them with.

Sizes are the benchmark workloads of paper_2504_14494_gb300/workloads.py (the 64^2 and 4096^2 Taylor-Green BGK runs,
the 1024^2 GNN-LBM inference, the training batch of 256^2 lattices, the serving batch of uneven lattices), the channel
lattices of the Poiseuille study and of train.ChannelPairBank, and odd or ragged sizes of the same ranges.

A case is {"kind": ..., sizes, options}; prepare() makes what a program holds before the call (states, parameters,
workspaces, a plan), run() makes the call through the public binding, exact() restates the method in FP64 with torch.
"""
import math

import numpy as np
import torch

from paper_2504_14494_gb300 import inputs
from paper_2504_14494_gb300 import lib as L
from paper_2504_14494_gb300.autograd import GnnFunction

E = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
DEV = "cuda"


def listed():
    return [
        # The 64^2 Taylor-Green run of 1000 steps (the accuracy workload; also what parameter studies loop over).
        {"name": "bgk_64_1000steps", "kind": "bgk", "nx": 64, "ny": 64, "nb": 1, "steps": 1000, "taus": False,
         "totals": False},
        # The bandwidth workload: a 4096^2 lattice advanced some steps between two outputs.
        {"name": "bgk_4096_20steps", "kind": "bgk", "nx": 4096, "ny": 4096, "nb": 1, "steps": 20, "taus": False,
         "totals": False},
        # A stack of odd-sized lattices with their own viscosities and FP64 totals at the end (stability studies).
        {"name": "bgk_odd_stack_10steps", "kind": "bgk", "nx": 1023, "ny": 517, "nb": 3, "steps": 10, "taus": True,
         "totals": True},
        # The Poiseuille study: a narrow channel of 32 rows run to its steady state in long calls.
        {"name": "channel_4x32_2000steps", "kind": "channel", "nx": 4, "ny": 32, "nb": 1, "steps": 2000,
         "taus": False, "totals": False},
        # One GNN-LBM step of the inference workload.
        {"name": "gnn_1024", "kind": "gnn", "nx": 1024, "ny": 1024, "nb": 1, "variant": 0, "taus": False,
         "totals": False},
        # Two odd-sized lattices with the conserving correction, their own relaxation times, and totals.
        {"name": "gnn_odd_stack", "kind": "gnn", "nx": 301, "ny": 217, "nb": 2, "variant": 2, "taus": True,
         "totals": True},
        # The smallest call: one GNN-LBM step of a 64^2 lattice, where launches and latency count.
        {"name": "gnn_64", "kind": "gnn", "nx": 64, "ny": 64, "nb": 1, "variant": 0, "taus": False, "totals": False},
        # The network without message passing (the paper's Fig. 2) on the large lattice, as one fused step.
        {"name": "mlp_4096", "kind": "mlp", "nx": 4096, "ny": 4096, "nb": 1, "variant": 3, "taus": False,
         "totals": False},
        # The training workload: one supervised step on 64 pairs of 256^2 coarse nodes.
        {"name": "train_64x256", "kind": "train", "nx": 256, "ny": 256, "nb": 64, "variant": 0},
        # The channel network's training step: 64 small channels of the training bank (20,000 such steps a run).
        {"name": "train_channel_64x32x8", "kind": "train_channel", "nx": 8, "ny": 32, "nb": 64, "variant": 0},
        # The network through torch.autograd: forward and backward on a few odd lattices inside a user's own loss.
        {"name": "autograd_4x100x96", "kind": "autograd", "nx": 100, "ny": 96, "nb": 4, "variant": 0},
        # Serving: lattices of uneven size, half BGK and half GNN-LBM, advanced together by one plan.
        {"name": "batch_48_uneven", "kind": "batch", "n": 48, "side_lo": 32, "side_hi": 640, "lattice_seed": 7,
         "steps": 4},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sides(lo, hi, most):
        while True:
            nx, ny, nb = log(lo, hi), log(lo, hi), rng.choice((1, 1, 1, 2, 3, 5))
            if rng.random() < 0.4:  # rows of whole vectors as well as any size
                nx = max(4, nx // 4 * 4)
            if nx * ny * nb <= most:
                return nx, ny, nb

    kind = rng.choice(("bgk", "bgk", "channel", "gnn", "gnn", "mlp", "train", "train_channel", "autograd", "batch"))
    if kind == "bgk":
        nx, ny, nb = sides(32, 4096, 4096 * 4096)
        most = min(1000, int(20 * 4096 * 4096 / (nx * ny * nb)))
        return {"kind": kind, "nx": nx, "ny": ny, "nb": nb, "steps": log(1, max(2, most)),
                "taus": rng.random() < 0.4, "totals": rng.random() < 0.4}
    if kind == "channel":
        ny = rng.choice((4, 8, 16, 32, 33, 96))
        nx, nb = (rng.choice((4, 4, 8)), 1) if rng.random() < 0.5 else (rng.choice((8, 24)), rng.choice((4, 8)))
        return {"kind": kind, "nx": nx, "ny": ny, "nb": nb, "steps": log(2, 2000), "taus": rng.random() < 0.4,
                "totals": rng.random() < 0.4}
    if kind in ("gnn", "mlp"):
        nx, ny, nb = sides(32, 1024, 1024 * 1024) if kind == "gnn" else sides(64, 4096, 4096 * 4096)
        return {"kind": kind, "nx": nx, "ny": ny, "nb": nb,
                "variant": rng.choice((0, 2, 4) if kind == "gnn" else (1, 3, 5)), "taus": rng.random() < 0.4,
                "totals": rng.random() < 0.4}
    if kind == "train":
        n = rng.choice((32, 48, 64, 100, 128, 256))
        return {"kind": kind, "nx": n, "ny": n, "nb": rng.choice((1, 4, 9, 16)), "variant": rng.choice((0, 2, 4))}
    if kind == "train_channel":
        return {"kind": kind, "nx": rng.choice((4, 8, 12)), "ny": rng.choice((16, 32, 33)),
                "nb": rng.choice((8, 16, 32, 64)), "variant": rng.choice((0, 2))}
    if kind == "autograd":
        nx, ny, nb = sides(32, 200, 4 * 100 * 96)
        return {"kind": kind, "nx": nx, "ny": ny, "nb": nb, "variant": 0}
    return {"kind": kind, "n": rng.randint(4, 48), "side_lo": 32, "side_hi": rng.choice((128, 320, 640)),
            "lattice_seed": rng.randint(0, 10**6), "steps": rng.randint(1, 4)}


# ---- inputs ----------------------------------------------------------------------------------------------------
def tgv_state(nx, ny, nb, g, noise=1e-4):
    """Post-collision states [9, nb, ny, nx] (FP32): Taylor-Green vortices of random wave number, amplitude and phase
    with the consistent pressure, plus a non-equilibrium part and small multiplicative noise."""
    r = torch.rand(4, nb, 1, 1, generator=g, device=DEV)
    mult = (2.0 ** torch.floor(3 * r[0]))
    u0 = 0.01 + 0.07 * r[1]
    x = torch.arange(nx, device=DEV).view(1, 1, nx)
    y = torch.arange(ny, device=DEV).view(1, ny, 1)
    ax = 2 * math.pi * (mult * x / nx + r[2])
    ay = 2 * math.pi * (mult * y / ny + r[3])
    ux = u0 * torch.cos(ax) * torch.sin(ay)
    uy = -u0 * torch.sin(ax) * torch.cos(ay)
    rho = 1 - 0.75 * u0 * u0 * (torch.cos(2 * ax) + torch.cos(2 * ay))
    f = torch.empty(9, nb, ny, nx, device=DEV)
    usq = 1.5 * (ux * ux + uy * uy)
    neq = 0.02 * u0 * torch.sin(ax) * torch.sin(ay)  # shear stress of the vortex: opposite sign on x and y
    for q, (ex, ey) in enumerate(E):
        eu = ex * ux + ey * uy
        f[q] = W[q] * rho * (1 + 3 * eu + 4.5 * eu * eu - usq) + W[q] * (ex * ex - ey * ey) * neq
        f[q] *= 1 + noise * (2 * torch.rand(nb, ny, nx, generator=g, device=DEV) - 1)
    return f


def channel_state(nx, ny, nb, g, force, tau):
    """Post-collision states of channels on their way to the parabolic profile."""
    yy = (torch.arange(ny, device=DEV) + 0.5).view(1, ny, 1)
    grown = 0.2 + 0.8 * torch.rand(nb, 1, 1, generator=g, device=DEV)
    ux = (grown * force.view(-1, 1, 1) / (2 * (tau.view(-1, 1, 1) - 0.5) / 3) * yy * (ny - yy)).expand(nb, ny, nx)
    f = torch.empty(9, nb, ny, nx, device=DEV)
    for q, (ex, _) in enumerate(E):
        eu = ex * ux
        f[q] = W[q] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * ux * ux)
        f[q] *= 1 + 1e-4 * (2 * torch.rand(nb, ny, nx, generator=g, device=DEV) - 1)
    return f


def taus_of(case, g):
    """Relaxation times of the TGV draws (Re 100 to 5000), one per lattice."""
    return 0.505 + 0.5 * torch.rand(case["nb"], generator=g, device=DEV)


def gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def empty_bytes(n):
    return torch.empty(n, dtype=torch.uint8, device=DEV)


def network(seed, variant):
    return inputs.xavier_params(seed, variant=variant, bias_scale=0.05)


def lattice_draws(case):
    return inputs.batch_lattices(case["n"], case["lattice_seed"], case["side_lo"], case["side_hi"])


def fields(case, seed):
    """The random inputs of a case, from the seed alone (shared by prepare and exact)."""
    g, kind = gen(seed), case["kind"]
    if kind == "batch":
        return {"f": [tgv_state(d["side"], d["side"], 1, g) for d in lattice_draws(case)]}
    nx, ny, nb = case["nx"], case["ny"], case["nb"]
    d = {"tau": 0.8}
    if kind == "channel" or kind == "train_channel":
        per = kind == "train_channel" or case.get("taus")
        tau = 0.55 + 0.9 * torch.rand(nb if per else 1, generator=g, device=DEV)
        # forces giving centre-line velocities of 0.03 to 0.07
        peak = 0.03 + 0.04 * torch.rand(nb if kind == "train_channel" else 1, generator=g, device=DEV)
        nu = (tau - 0.5) / 3
        force = 8 * (nu if kind == "train_channel" else nu.min()) * peak / ny ** 2
        d["taus"], d["tau"] = (tau, 0.0) if per else (None, float(tau[0]))
        d["force"] = force
        d["f"] = channel_state(nx, ny, nb, g, force, tau)
    else:
        d["taus"] = taus_of(case, g) if case.get("taus") or kind == "train" else None
        d["f"] = tgv_state(nx, ny, nb, g)
    if kind in ("train", "train_channel"):
        # the pair's target: the plain step plus the small smooth difference to a refined run
        step = bgk_exact if kind == "train" else channel_exact
        t = d["taus"].double().view(-1, 1, 1)
        chunk = max(1, (1 << 20) // (nx * ny))
        tgt = torch.empty_like(d["f"])
        for b in range(0, nb, chunk):
            fb = d["f"][:, b:b + chunk].double()
            more = () if kind == "train" else (d["force"][b:b + chunk].double().view(-1, 1, 1),)
            tgt[:, b:b + chunk] = step(fb, t[b:b + chunk], *more).float()
        smooth = 2e-5 * torch.sin(torch.arange(nx, device=DEV) * (2 * math.pi / nx)).view(1, 1, nx)
        for q in range(9):
            tgt[q] *= 1 + smooth + 5e-6 * (2 * torch.rand(nb, ny, nx, generator=g, device=DEV) - 1)
        d["target"] = tgt
    return d


def prepare(case, seed):
    kind = case["kind"]
    d = fields(case, seed)
    st = {"kind": kind}
    if kind == "batch":
        lat = lattice_draws(case)
        st["plan"] = L.lbm_batch_plan_create(
            [(x["side"], x["side"], int(x["gnn"]), 0.5 + 3 * x["nu"]) for x in lat])
        n = L.lbm_batch_nodes(st["plan"])
        off = L.lbm_batch_offsets(st["plan"], case["n"])
        buf = torch.empty(9, n, device=DEV)
        for o, f in zip(off, d["f"]):
            buf[:, o:o + f[0].numel()] = f.reshape(9, -1)
        st.update(f_in=buf.reshape(-1), f_out=torch.empty(9 * n, device=DEV), f_tmp=torch.empty(9 * n, device=DEV),
                  steps=case["steps"], packed=empty_bytes(L.gnn_packed_bytes()),
                  ws=empty_bytes(max(16, L.lbm_batch_workspace_bytes(st["plan"]))))
        st["keep"] = Plan(st["plan"])
        L.gnn_pack(torch.from_numpy(network(seed, 0)).to(DEV), st["packed"])
        return st
    s = L.shape(case["nx"], case["ny"], case["nb"])
    f = d["f"].reshape(-1)
    st.update(s=s, f_in=f, taus=d["taus"], tau=d["tau"])
    if case.get("totals"):
        st["totals"] = torch.zeros(5, dtype=torch.float64, device=DEV)
    if kind in ("bgk", "channel"):
        st.update(steps=case["steps"], f_out=torch.empty_like(f),
                  f_tmp=torch.empty_like(f) if case["steps"] > 1 else None)
        if kind == "channel":
            st["force"] = float(d["force"][0] if d["force"].dim() else d["force"])
        return st
    theta = torch.from_numpy(network(seed, case["variant"])).to(DEV)
    if kind == "autograd":
        n = case["nx"] * case["ny"] * case["nb"]
        st.update(f_in=f.requires_grad_(), params=theta.requires_grad_(),
                  dy=torch.randn(10, n, generator=gen(seed + 1), device=DEV))
        return st
    st["packed"] = empty_bytes(L.gnn_packed_bytes())
    L.gnn_pack(theta, st["packed"])
    if kind in ("gnn", "mlp"):
        st["f_out"] = torch.empty_like(f)
        if kind == "gnn":
            st["ws"] = empty_bytes(L.gnn_step_workspace_bytes(s))
        return st
    nt = L.gnn_trainable_count()
    st.update(target=d["target"].reshape(-1), params=theta, m=torch.zeros(nt, device=DEV),
              v=torch.zeros(nt, device=DEV), loss=torch.zeros(1, dtype=torch.float64, device=DEV),
              grads=torch.zeros(nt, device=DEV), ws=empty_bytes(L.gnn_train_workspace_bytes(s)), step=0,
              forces=d.get("force"))
    return st


class Plan:
    """Gives a batch plan back when its state is dropped."""

    def __init__(self, plan):
        self.plan = plan

    def __del__(self):
        torch.cuda.synchronize()
        L.lbm_batch_plan_destroy(self.plan)


# ---- one pass --------------------------------------------------------------------------------------------------
def run(st):
    kind, tot = st["kind"], st.get("totals")
    if kind == "bgk":
        L.lbm_step_bgk(st["f_in"], st["f_out"], st["f_tmp"], st["s"], st["tau"], st["taus"], st["steps"], tot)
    elif kind == "channel":
        L.lbm_step_channel(st["f_in"], st["f_out"], st["f_tmp"], st["s"], st["tau"], st["taus"], st["force"],
                           st["steps"], tot)
    elif kind == "gnn":
        L.lbm_step_gnn(st["f_in"], st["f_out"], st["s"], st["tau"], st["taus"], st["packed"], tot, st["ws"])
    elif kind == "mlp":
        L.lbm_step_gnn_mlp(st["f_in"], st["f_out"], st["s"], st["tau"], st["taus"], st["packed"], tot)
    elif kind == "batch":
        L.lbm_batch_run(st["plan"], st["f_in"], st["f_out"], st["f_tmp"], st["steps"], st["packed"], st["ws"])
    elif kind == "autograd":
        y = GnnFunction.apply(st["f_in"], st["params"], st["s"])
        return [y.detach(), *torch.autograd.grad(y, (st["f_in"], st["params"]), st["dy"])]
    else:
        st["step"] += 1
        more = (st["params"], st["packed"], st["m"], st["v"], st["step"], 1e-3, 1e-2, st["loss"], st["grads"],
                st["ws"])
        if kind == "train":
            L.gnn_train_step(st["f_in"], st["target"], st["s"], st["tau"], st["taus"], *more)
        else:
            L.gnn_train_step_channel(st["f_in"], st["target"], st["s"], 0.0, st["taus"], 0.0, st["forces"], None,
                                     *more)
        return [st["loss"], st["grads"], st["params"], st["m"], st["v"]]
    return [st["f_out"]] if tot is None else [st["f_out"], tot]


# ---- what one pass cannot do without ---------------------------------------------------------------------------
def work(case):
    """Bytes: states read once and written once (36 B a node each), targets, gradients and parameters once.
    Operations: about 200 per node and step for a collision; the network's dense layers (76,544 per node) and its
    1,024 edge and 256 node activations at 10 each; the backward at twice the forward."""
    net = 76544 + 1280 * 10
    mlp = 2 * (12 * 64 + 64 * 64 + 640) + 128 * 10
    kind = case["kind"]
    if kind == "batch":
        lat = lattice_draws(case)
        n = sum(x["side"] ** 2 for x in lat)
        n_gnn = sum(x["side"] ** 2 for x in lat if x["gnn"])
        return {"bytes": 72 * n, "flops": case["steps"] * (200 * n + net * n_gnn)}
    n = case["nx"] * case["ny"] * case["nb"]
    if kind in ("bgk", "channel"):
        return {"bytes": 72 * n, "flops": 200 * n * case["steps"]}
    if kind in ("gnn", "mlp"):
        return {"bytes": 72 * n, "flops": (200 + (net if kind == "gnn" else mlp)) * n}
    params = 4 * 38922
    if kind == "autograd":
        return {"bytes": (36 + 40 + 40 + 36) * n + 2 * params, "flops": 3 * net * n}
    return {"bytes": 72 * n + 8 * params, "flops": (3 * net + 400) * n}


# ---- the same in 64 bits, in plain torch -----------------------------------------------------------------------
def moments(f, force=None):
    rho = f.sum(0)
    jx = sum(E[q][0] * f[q] for q in range(9) if E[q][0])
    jy = sum(E[q][1] * f[q] for q in range(9) if E[q][1])
    if force is not None:
        jx = jx + 0.5 * force
    return rho, jx / rho, jy / rho


def equilibrium(q, rho, ux, uy):
    eu = E[q][0] * ux + E[q][1] * uy
    return W[q] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))


def pull(f):
    return torch.stack([torch.roll(f[q], (E[q][1], E[q][0]), (-2, -1)) for q in range(9)])


def pull_walls(f):
    out = pull(f)
    for q in range(9):
        if E[q][1] > 0:
            out[q][..., 0, :] = f[OPP[q]][..., 0, :]
        elif E[q][1] < 0:
            out[q][..., -1, :] = f[OPP[q]][..., -1, :]
    return out


def guo(q, ux, uy, force):
    ex, ey = E[q]
    return W[q] * (3 * (ex - ux) + 9 * (ex * ux + ey * uy) * ex) * force


def bgk_exact(f, tau):
    f = pull(f)
    m = moments(f)
    for q in range(9):
        f[q] -= (f[q] - equilibrium(q, *m)) / tau
    return f


def channel_exact(f, tau, force):
    f = pull_walls(f)
    m = moments(f, force)
    for q in range(9):
        f[q] += (1 - 0.5 / tau) * guo(q, m[1], m[2], force) - (f[q] - equilibrium(q, *m)) / tau
    return f


def totals_exact(f):
    rho, ux, uy = moments(f)
    return torch.stack([rho.sum(), (rho * ux).sum(), (rho * uy).sum(), (0.5 * rho * (ux * ux + uy * uy)).sum(),
                        torch.zeros((), dtype=torch.float64, device=f.device)])


def weights64(theta):
    """The parameter vector as FP64 leaves: matrices rounded to BF16 first, as the network uses them."""
    out, o = [], 0
    for shape in inputs.PARAM_SHAPES:
        n = int(np.prod(shape))
        v = theta[o:o + n].view(shape)
        v = v.bfloat16() if len(shape) == 2 else v
        out.append(v.double().requires_grad_(theta.requires_grad))
        o += n
    return out, theta[o:].double()


def gelu(z):
    return 0.5 * z * (1 + torch.tanh(0.7978845608028654 * (z + 0.044715 * z ** 3)))


def net_exact(f_pre, p, fixed, walls=False, force=None):
    """Head output [N, 10] of the network on pre-collision populations [9, nb, ny, nx]."""
    nb, ny, nx = f_pre.shape[1:]
    rho, ux, uy = moments(f_pre, force)
    x = torch.cat([f_pre, rho[None], ux[None], uy[None]]).reshape(12, -1).T
    x = (x - fixed[:12]) / fixed[12:24]
    mlp_only = int(fixed[25]) & 1
    act = torch.relu if mlp_only else gelu
    h = act(act(x @ p[0].T + p[1]) @ p[2].T + p[3])
    for r in range(0 if mlp_only else 2):
        we, be, wn, bn = p[4 + 4 * r:8 + 4 * r]
        a_i, b_j = h @ we[:, :64].T, (h @ we[:, 64:128].T).view(nb, ny, nx, 64)
        a = 0
        for k in range(1, 9):
            ex, ey = E[k]
            z = torch.roll(b_j, (-ey, -ex), (1, 2)).reshape(-1, 64) + (ex * we[:, 128] + ey * we[:, 129] + be) + a_i
            m = gelu(z)
            if walls and ey:
                keep = torch.ones(nb, ny, nx, 1, dtype=torch.float64, device=f_pre.device)
                keep[:, -1 if ey > 0 else 0] = 0
                m = m * keep.view(-1, 1)
            a = a + m
        h = h + gelu(torch.cat([h, a], 1) @ wn.T + bn)
    return h @ p[12].T + p[13]


def collide_exact(f, y, tau, fixed, force=None):
    """Eq. 3 on pre-collision populations with the head output y [N, 10]."""
    variant = int(fixed[25])
    y = y.T.reshape((10,) + f.shape[1:])
    t = tau * (1.0 if variant & 4 else 0.5 + torch.sigmoid(y[0]))
    d = fixed[24] * y[1:]
    if variant & 2:
        s = d.sum(0)
        sx = sum(E[q][0] * d[q] for q in range(9))
        sy = sum(E[q][1] * d[q] for q in range(9))
        d = torch.stack([d[q] - s / 9 - E[q][0] * sx / 6 - E[q][1] * sy / 6 for q in range(9)])
    m = moments(f, force)
    out = []
    for q in range(9):
        v = f[q] - (f[q] - equilibrium(q, *m)) / t + d[q]
        out.append(v if force is None else v + (1 - 0.5 / t) * guo(q, m[1], m[2], force))
    return torch.stack(out)


def step_exact(f, p, fixed, tau):
    """One GNN-LBM step of [9, nb, ny, nx]; large Fig. 2 lattices in slabs of rows."""
    f = pull(f)
    if int(fixed[25]) & 1:
        out = torch.empty_like(f)
        rows = max(1, (1 << 20) // (f.shape[1] * f.shape[3]))
        for y in range(0, f.shape[2], rows):
            fs = f[:, :, y:y + rows].contiguous()
            out[:, :, y:y + rows] = collide_exact(fs, net_exact(fs, p, fixed), tau, fixed)
        return out
    return collide_exact(f, net_exact(f, p, fixed), tau, fixed)


def exact(case, seed):
    kind = case["kind"]
    d = fields(case, seed)
    if kind == "batch":
        p, fixed = weights64(torch.from_numpy(network(seed, 0)).to(DEV))
        lat = lattice_draws(case)
        order = [i for i, x in enumerate(lat) if not x["gnn"]] + [i for i, x in enumerate(lat) if x["gnn"]]
        out = []
        for i in order:
            f, tau = d["f"][i].double(), float(np.float32(0.5 + 3 * lat[i]["nu"]))
            for _ in range(case["steps"]):
                f = step_exact(f, p, fixed, tau) if lat[i]["gnn"] else bgk_exact(f, tau)
            out.append(f.reshape(9, -1))
        return [torch.cat(out, 1).reshape(-1)]
    f = d["f"].double()
    tau = float(np.float32(d["tau"])) if d["taus"] is None else d["taus"].double().view(-1, 1, 1)
    if kind in ("bgk", "channel"):
        force = None if kind == "bgk" else float(d["force"].reshape(-1)[0])
        for _ in range(case["steps"]):
            f = bgk_exact(f, tau) if force is None else channel_exact(f, tau, force)
        return [f.reshape(-1)] + ([totals_exact(f)] if case.get("totals") else [])
    theta = torch.from_numpy(network(seed, case["variant"])).to(DEV)
    if kind in ("gnn", "mlp"):
        p, fixed = weights64(theta)
        f = step_exact(f, p, fixed, tau)
        return [f.reshape(-1)] + ([totals_exact(f)] if case.get("totals") else [])
    p, fixed = weights64(theta.requires_grad_())
    p = [v.detach().requires_grad_() for v in p]
    fixed = fixed.detach()
    if kind == "autograd":
        f.requires_grad_()
        y = net_exact(f, p, fixed)
        dy = torch.randn(10, y.shape[0], generator=gen(seed + 1), device=DEV).double()
        got = torch.autograd.grad((y.T * dy).sum(), [f] + p)
        dp = torch.cat([v.reshape(-1) for v in got[1:]] + [torch.zeros(26, dtype=torch.float64, device=DEV)])
        return [y.detach().T, got[0].reshape(-1), dp]
    # training: loss and gradient lattice by lattice (they are independent), then the first AdamW update
    nb, n = case["nb"], case["nx"] * case["ny"]
    chunk = max(1, (1 << 18) // n)
    loss, grad = 0.0, None
    for b in range(0, nb, chunk):
        part = slice(b, b + chunk)
        walls = kind == "train_channel"
        force = d["force"][part].double().view(-1, 1, 1) if walls else None
        fp = pull_walls(f[:, part]) if walls else pull(f[:, part])
        pred = collide_exact(fp, net_exact(fp, p, fixed, walls, force), tau[part], fixed, force)
        ls = ((pred - d["target"][:, part].double()) ** 2).sum() / (9 * nb * n)
        g = torch.autograd.grad(ls, p, allow_unused=True)
        g = torch.cat([(torch.zeros_like(v) if x is None else x).reshape(-1) for x, v in zip(g, p)])
        loss, grad = loss + ls.detach(), g if grad is None else grad + g
    th = theta.detach().double()
    new = th.clone()
    new[:grad.numel()] = th[:grad.numel()] * (1 - 1e-5) - 1e-3 * grad / (grad.abs() + 1e-8)
    return [loss.reshape(1), grad, new, 0.1 * grad, 0.001 * grad * grad]
