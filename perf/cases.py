"""What the framework's speed is measured on: single passes through the public
entry points of paper_2006_14952_gb300.hfmm, over the sizes and options its
users run (the workloads of workloads.py, the learned-acceptance training of
train_mac.py, the kick-drift-kick step, the host-buffer call).

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  what a program has in hand before the call
    run(state)           one pass, and its outputs
    work(case)           bytes and flops no implementation can do without
    exact(case, seed)    the same outputs in 64 bits, in plain torch

Particle sets are drawn on the GPU with the statistics of workloads.py: uniform;
clustered (a share of the particles in NFW haloes, dN/dM ~ M^-1.9 over three
decades, the rest uniform); a displaced lattice with haloes.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2006_14952_gb300 as _package
from paper_2006_14952_gb300 import hfmm

RS_CELLS, RCUT_RS = 1.25, 4.5  # the split scale and cut-off of every workload in workloads.py
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(_package.__file__)), "weights", "mac_weights.bin")

# kind: which entry points a pass calls
#   forces  build_tree + short_range_forces (the benchmark's step)
#   host    short_range_forces_host on pinned host buffers
#   step    one kick-drift-kick step of a simulation
#   pm      pm_long_range on a built tree
#   train   one full-batch Adam step of the learned-acceptance network
_SET = dict(kind="forces", dist="nfw", n=0, haloes=0, halo_frac=0.7, box=1.0, pm_grid=32, theta=0.35, order=6,
            leaf_max=48, tree=0, split=0, mac_mode=0, m2l_precision=0, use_graph=0, equal_mass=True)


def _case(**kw):
    unknown = set(kw) - set(_SET) - {"name"}
    assert not unknown, unknown
    return {**_SET, **kw}


def listed():
    return [
        # the smallest call: a test particle set, dominated by launches and the calls' synchronisations
        _case(name="forces uniform 1k", dist="uniform", n=1000, theta=0.5, order=4, leaf_max=16),
        # the small uniform workload (N = 32^3, PM 32^3), as listed in workloads.py
        _case(name="forces uniform 32k", dist="uniform", n=32 ** 3, theta=0.5, order=4, leaf_max=16),
        # the benchmark: N = 128^3, 70% in 2000 haloes, the setting that meets 1e-4
        _case(name="forces nfw 2m", n=128 ** 3, haloes=2000, pm_grid=128),
        # the large set one GPU takes in sink batches: displaced lattice of 256^3, 40% in haloes
        _case(name="forces zeldovich 16m", dist="zeldovich", n=256 ** 3, haloes=1000, halo_frac=0.4, pm_grid=256),
        # the benchmark's other arm: learned acceptance with 3xTF32 tensor-core M2L
        _case(name="learned tf32 nfw 2m", n=128 ** 3, haloes=2000, pm_grid=128, theta=0.5, mac_mode=1,
              m2l_precision=1),
        # the paper's own tree on the benchmark's set
        _case(name="kd nfw 2m", n=128 ** 3, haloes=2000, pm_grid=128, tree=1),
        # the polynomial truncation in a box of 100 length units, unequal masses, odd sizes, lower accuracy
        _case(name="poly nfw 300k box 100", n=300_007, haloes=301, halo_frac=0.85, box=100.0, pm_grid=67,
              theta=0.5, order=5, leaf_max=32, split=1, equal_mass=False),
        # a host program without CUDA of its own: pinned buffers in, accelerations out
        _case(name="host nfw 262k", kind="host", n=1 << 18, haloes=250, pm_grid=64),
        # a simulation's step as one graph, benchmark set
        _case(name="step graph nfw 2m", kind="step", n=128 ** 3, haloes=2000, pm_grid=128, use_graph=1),
        # a small simulation stepping by direct launches, odd mesh
        _case(name="step uniform 100k", kind="step", dist="uniform", n=100_003, pm_grid=45, theta=0.5, order=4,
              leaf_max=24),
        # the mesh half alone: deposit, transforms, interpolation
        _case(name="pm nfw 2m", kind="pm", n=128 ** 3, haloes=2000, pm_grid=128),
        # training of the learned acceptance: the 400k pairs train_mac.py collects
        _case(name="train 400k", kind="train", n=400_000),
    ]


def draw(rng):
    """One more case: sizes log-uniform over what the listed cases span below the
    largest one, the options mixed the way the solver accepts them."""
    kind = rng.choice(["forces"] * 7 + ["host", "step", "step", "pm", "train"])
    if kind == "train":
        return _case(kind=kind, n=int(round(math.exp(rng.uniform(math.log(20_000), math.log(600_000))))))
    n = int(round(math.exp(rng.uniform(math.log(1_000), math.log(2_500_000)))))
    dist = rng.choice(["uniform", "nfw", "nfw"])
    side = n ** (1.0 / 3.0)
    # about one mesh cell per mean particle spacing, never so coarse that R_c reaches box / 3
    pm = max(20, int(round(side * rng.uniform(0.85, 1.15))))
    theta, order = rng.choice([(0.5, 4), (0.5, 5), (0.4, 5), (0.35, 6)])
    leaf = rng.choice([16, 24, 32, 48]) if n < 200_000 else rng.choice([32, 48, 64])
    if n >= 200_000 and order == 6 and leaf < 48:
        leaf = 48
    case = _case(kind=kind, dist=dist, n=n, haloes=max(1, n // 1000) if dist == "nfw" else 0,
                 halo_frac=rng.choice([0.4, 0.7, 0.85]), box=rng.choice([1.0, 1.0, 100.0, 0.5]), pm_grid=pm,
                 theta=theta, order=order, leaf_max=leaf, equal_mass=rng.random() < 0.7)
    if kind == "step":
        case["use_graph"] = rng.choice([0, 1])
    if kind == "forces":
        option = rng.choice(["plain", "plain", "graph", "kd", "kd", "poly", "learned", "tf32"])
        if option == "graph":
            case["use_graph"] = 1
        elif option == "kd":
            case["tree"] = 1
            case["split"] = rng.choice([0, 0, 1])
        elif option == "poly":
            case["split"] = 1
        elif option in ("learned", "tf32"):
            case["m2l_precision"] = rng.choice([1, 2]) if option == "tf32" else 0
            if option == "learned":
                case.update(mac_mode=1, theta=0.5, order=6, leaf_max=48)
    return case


# ------------------------------------------------------------------ particle sets
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _halo_positions(g, n, haloes, n_total):
    """n particles in NFW haloes, unit box: masses dN/dM ~ M^-1.9 over three decades,
    concentrations U[5, 15], truncated at r_200 of 200 times the mean density."""
    a = 0.9
    m = (1.0 - _rand(g, haloes) * (1.0 - 10.0 ** (-3.0 * a))) ** (-1.0 / a)
    edge = torch.cumsum(m, 0) / m.sum()
    edge[-1] = 1.0
    where = torch.bucketize((torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n, edge)
    count = torch.bincount(where, minlength=haloes).double()
    centre, c = _rand(g, 3, haloes), 5.0 + 10.0 * _rand(g, haloes)
    r200 = (3.0 * count / n_total / (4.0 * math.pi * 200.0)) ** (1.0 / 3.0)
    cw = c[where]

    def enclosed(x):
        return torch.log1p(x) - x / (1.0 + x)

    u = _rand(g, n) * enclosed(cw)
    lo, hi = torch.zeros_like(cw), cw.clone()
    for _ in range(44):  # bisection on the enclosed mass
        mid = 0.5 * (lo + hi)
        below = enclosed(mid) < u
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    r = 0.5 * (lo + hi) / cw * r200[where]
    d = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64)
    return centre[:, where] + r * d / d.norm(dim=0)


def _displaced_lattice(g, side):
    """side^3 lattice moved by a Gaussian field, P(k) ~ k^-2 exp(-(k / k_Nyq)^2), RMS 0.3 spacings."""
    x = torch.arange(side, device="cuda", dtype=torch.float64) / side
    pos = torch.stack(torch.meshgrid(x, x, x, indexing="ij")).reshape(3, -1)
    dk = torch.fft.rfftn(torch.randn(side, side, side, generator=g, device="cuda"))
    kf = torch.fft.fftfreq(side, 1.0 / side, device="cuda")
    kz = torch.fft.rfftfreq(side, 1.0 / side, device="cuda")
    k = (kf[:, None, None], kf[None, :, None], kz[None, None, :])
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    dk *= torch.sqrt(torch.exp(-k2 / (side / 2.0) ** 2) / k2)
    dk[0, 0, 0] = 0.0
    move = torch.stack([torch.fft.irfftn(1j * q * dk / k2, s=(side,) * 3).reshape(-1) for q in k]).double()
    return pos + move * (0.3 / side / move.square().sum(0).mean().sqrt())


def _particles(case, seed):
    """Positions [3][n] float64 in [0, box) and masses [n] float32 (total about 1)."""
    g, n, box = _generator(seed), case["n"], case["box"]
    if case["dist"] == "zeldovich":
        side = round(n ** (1.0 / 3.0))
        pos = _displaced_lattice(g, side)
    else:
        pos = _rand(g, 3, n)
    nh = int(round(case["halo_frac"] * n)) if case["dist"] != "uniform" else 0
    if nh:
        # the particles stay in no spatial order: a snapshot's order says nothing about place
        pos[:, torch.randperm(n, generator=g, device="cuda")[:nh]] = _halo_positions(g, nh, case["haloes"], n)
    pos = torch.remainder(pos, 1.0) * box
    pos = torch.where(pos >= box, torch.zeros_like(pos), pos).contiguous()
    mass = torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float32)
    if not case["equal_mass"]:
        mass = mass * (0.5 + torch.rand(n, generator=g, device="cuda"))
    return pos, mass, g


def _velocities(case, g):
    """Velocities and the accelerations of the step before, float32 [3][n]."""
    n, box = case["n"], case["box"]
    vel = 0.05 * box * torch.randn(3, n, generator=g, device="cuda")
    acc = torch.randn(3, n, generator=g, device="cuda") / box ** 2
    return vel, acc


_DT = 1e-4


def _training_batch(case, seed):
    """Pair features as the acceptance network sees them, labels of a rule of the same kind, a training run under way."""
    g, n = _generator(seed), case["n"]

    def u(lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda")

    def normal(scale):
        return scale * torch.randn(n, generator=g, device="cuda")

    sc, ha, hb = u(0.1, 4.0), u(0.05, 0.5), u(0.05, 0.5)
    level = torch.randint(-2, 3, (n,), generator=g, device="cuda").float() / 8.0
    x = torch.stack([sc, 0.6 * sc, 0.3 * sc, ha, hb, torch.maximum(ha, hb), level, u(0.1, 1.0), u(0.1, 1.0),
                     normal(0.2).abs(), normal(0.1).abs(), sc / RCUT_RS], dim=1).contiguous()
    open_, order = x[:, 5] > 0.42, 1 + (10.0 * x[:, 5] + 4.0 * x[:, 9] + 0.5 * normal(1.0)).floor().clamp(0, 4)
    y = torch.where(open_, torch.zeros_like(order), order).to(torch.int32).contiguous()
    w = torch.zeros(hfmm.MLP_WEIGHTS, device="cuda")
    at = 0
    for fan_in, fan_out in ((12, 64), (64, 64), (64, 8)):
        w[at:at + fan_in * fan_out] = (2.0 / fan_in) ** 0.5 * torch.randn(fan_in * fan_out, generator=g, device="cuda")
        at += fan_in * fan_out + fan_out
    m1 = 1e-3 * torch.randn(hfmm.MLP_WEIGHTS, generator=g, device="cuda")
    m2 = 1e-5 * (0.5 + torch.rand(hfmm.MLP_WEIGHTS, generator=g, device="cuda"))
    count = torch.bincount(y.long(), minlength=8).float()
    cw = torch.where(count > 0, (count.sum() / (8 * count.clamp(min=1))) ** 0.5, torch.zeros_like(count))
    return x, y, cw, w, m1, m2


# ------------------------------------------------------------------ the passes
def _solver(case):
    s = hfmm.Solver(box=case["box"], pm_grid=case["pm_grid"], rs_cells=RS_CELLS, rcut_rs=RCUT_RS,
                    theta=case["theta"], order=case["order"], leaf_max=case["leaf_max"], tree=case["tree"],
                    split=case["split"], mac_mode=case["mac_mode"], m2l_precision=case["m2l_precision"],
                    use_graph=case["use_graph"])
    if case["mac_mode"] == 1:
        s.load_mlp(np.fromfile(WEIGHTS, dtype=np.uint16))
    return s


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "train":
        x, y, cw, w, m1, m2 = _training_batch(case, seed)
        state.update(solver=hfmm.Solver(), x=x, y=y, cw=cw, w=w, m1=m1, m2=m2, step=100,
                     wb=torch.empty(hfmm.MLP_WEIGHTS, device="cuda", dtype=torch.bfloat16))
        return state
    pos, mass, g = _particles(case, seed)
    state["solver"] = s = _solver(case)
    if case["kind"] == "host":
        state.update(pos=pos.cpu().pin_memory(), mass=mass.cpu().pin_memory(),
                     acc=torch.empty(3, case["n"], dtype=torch.float32, pin_memory=True))
        return state
    state.update(pos=pos, mass=mass)
    if case["kind"] == "forces":
        state["acc"] = torch.empty(3, case["n"], dtype=torch.float32, device="cuda")
    else:
        s.build_tree(pos, mass)
    if case["kind"] == "step":
        vel, acc = _velocities(case, g)
        # every pass is the first step after this snapshot
        state.update(vel=vel, acc=acc, now=(pos.clone(), vel.clone(), acc.clone()))
    return state


def run(state):
    s, kind = state["solver"], state["case"]["kind"]
    if kind == "forces":
        s.build_tree(state["pos"], state["mass"])
        return {"acc": s.short_range_forces(state["acc"])}
    if kind == "host":
        return {"acc": s.short_range_forces_host(state["pos"], state["mass"], state["acc"])}
    if kind == "pm":
        return {"acc": s.pm_long_range()}
    if kind == "step":
        pos, vel, acc = state["now"]
        pos.copy_(state["pos"])
        vel.copy_(state["vel"])
        acc.copy_(state["acc"])
        s.step(pos, vel, acc, _DT)
        return {"pos": pos, "vel": vel, "acc": acc}
    grad, loss = s.mlp_grad(state["w"], state["x"], state["y"], state["cw"])
    state["step"] += 1
    hfmm.mlp_adam(grad, 3e-3, state["step"], state["w"], state["m1"], state["m2"], state["wb"])
    return {k: state[k] for k in ("w", "m1", "m2", "wb")} | {"grad": grad, "loss": loss}


def work(case):
    n = case["n"]
    if case["kind"] == "train":
        # features, labels; forward 2, backward 4 flops per weight and sample (less for the first layer's input)
        return {"bytes": 52.0 * n + 5512 * 34.0, "flops": float(n) * (6 * (64 * 64 + 64 * 8) + 4 * 12 * 64)}
    mesh = case["pm_grid"] ** 3
    pm = {"bytes": 24.0 * n + 4 * n + 24 * n, "flops": n * 8.0 * (4 + 7) + 4 * 2.5 * mesh * math.log2(mesh)}
    if case["kind"] == "pm":
        return pm
    # Particle pairs the tree leaves to the direct sum: about 50 leaf_max per particle on the
    # clustered benchmark set (theta 0.35), fewer where theta is larger, never more than lie within
    # R_c of a uniform set's particle times the clustering; 42 flops a pair (21 with the polynomial
    # split), and M2L with C(p + 6, 6) multiply-adds for about 8 pairs a particle at leaves of 48.
    rc = RS_CELLS * RCUT_RS / case["pm_grid"]
    near = 50.0 * case["leaf_max"] * (0.35 / case["theta"]) ** 2
    if case["dist"] == "uniform":
        near = min(0.5 * near, n * 4.0 / 3.0 * math.pi * rc ** 3)
    per_pair = 21.0 if case["split"] == 1 else 42.0
    m2l = 2.0 * math.comb(case["order"] + 6, 6) * 8.0 * (48.0 / case["leaf_max"]) ** 1.5
    total = {"bytes": 24.0 * n + 4 * n + 12 * n, "flops": n * (per_pair * near + m2l)}
    if case["kind"] == "step":
        total = {"bytes": (24 + 12 + 12) * 2.0 * n + 4 * n, "flops": total["flops"] + pm["flops"] + 24.0 * n}
    return total


# ------------------------------------------------------------------ the same in 64 bits
def _direct_forces(case, pos, mass, most=4e10):
    """The truncated pair sum over all pairs within R_c, in cells of side >= R_c; None above `most` candidates."""
    n, box = case["n"], case["box"]
    rs = RS_CELLS * box / case["pm_grid"]
    rc = RCUT_RS * rs
    nc = int(box / rc)
    assert nc >= 3
    cell = torch.clamp((pos * (nc / box)).long(), 0, nc - 1)
    flat = (cell[0] * nc + cell[1]) * nc + cell[2]
    order = torch.argsort(flat, stable=True)
    x, m = pos[:, order].contiguous(), mass[order].double()
    count = torch.bincount(flat, minlength=nc ** 3).reshape(nc, nc, nc)
    around = sum(torch.roll(count, (a, b, c), (0, 1, 2)) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1))
    if float((count.double() * around).sum()) > most:
        return None
    cnt = count.reshape(-1).cpu().numpy()
    start = np.concatenate([[0], np.cumsum(cnt)])
    out = torch.zeros(3, n, device="cuda", dtype=torch.float64)
    for q in np.nonzero(cnt)[0]:
        i, j, k = q // (nc * nc), (q // nc) % nc, q % nc
        parts = []
        for a in (-1, 0, 1):
            for b in (-1, 0, 1):
                row = ((i + a) % nc * nc + (j + b) % nc) * nc
                if 0 < k < nc - 1:
                    parts.append(slice(start[row + k - 1], start[row + k + 2]))
                else:
                    parts += [slice(start[row + (k + c) % nc], start[row + (k + c) % nc + 1]) for c in (-1, 0, 1)]
        src, ms = torch.cat([x[:, p] for p in parts], 1), torch.cat([m[p] for p in parts])
        mid = torch.tensor([(v + 0.5) * box / nc for v in (i, j, k)], dtype=torch.float64).cuda()[:, None]
        src = src - box * torch.round((src - mid) / box)  # the image next to this cell
        step = max(1, int(4e7 // max(1, src.shape[1])))
        for lo in range(start[q], start[q + 1], step):
            sl = slice(lo, min(lo + step, start[q + 1]))
            d = [x[e, sl, None] - src[e][None, :] for e in range(3)]
            r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
            inside = (r2 > 0) & (r2 < rc * rc)
            r2 = torch.where(inside, r2, torch.full_like(r2, rc * rc))
            r = torch.sqrt(r2)
            if case["split"] == 1:
                f = -1.0 / (r2 * r) + 5.0 / (2.0 * rc ** 3) - 3.0 * r2 / (2.0 * rc ** 5)
            else:
                f = -(torch.erfc(r / (2.0 * rs)) + r / (rs * math.sqrt(math.pi)) * torch.exp(-r2 / (4.0 * rs * rs)))
                f = f / (r2 * r)
            f = torch.where(inside, f, torch.zeros_like(f)) * ms[None, :]
            for e in range(3):
                out[e, sl] = (f * d[e]).sum(1)
    back = torch.empty_like(out)
    back[:, order] = out
    return back


def _mesh_forces(case, pos, mass):
    """Cloud-in-cell mass, 4 pi exp(-k^2 r_s^2) / k^2 over the squared window, spectral gradient, interpolation."""
    ng, box = case["pm_grid"], case["box"]
    rs = RS_CELLS * box / ng
    u = pos * (ng / box)
    base = torch.floor(u)
    d = u - base
    base = base.long()
    corners = []
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                at = [(base[e] + o) % ng for e, o in enumerate((a, b, c))]
                w = [d[e] if o else 1.0 - d[e] for e, o in enumerate((a, b, c))]
                corners.append(((at[0] * ng + at[1]) * ng + at[2], w[0] * w[1] * w[2]))
    rho = torch.zeros(ng ** 3, device="cuda", dtype=torch.float64)
    for at, w in corners:
        rho.index_add_(0, at, w * mass.double())
    mk = torch.fft.rfftn(rho.reshape(ng, ng, ng))
    kf = torch.fft.fftfreq(ng, 1.0 / ng, device="cuda", dtype=torch.float64) * (2.0 * math.pi / box)
    kr = torch.fft.rfftfreq(ng, 1.0 / ng, device="cuda", dtype=torch.float64) * (2.0 * math.pi / box)
    k = [kf[:, None, None], kf[None, :, None], kr[None, None, :]]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    window = 1.0
    for q in k:
        window = window * torch.sinc(q * (box / ng / (2.0 * math.pi)))
    green = 4.0 * math.pi * torch.exp(-k2 * rs * rs) / (k2 * window ** 4) / box ** 3
    green[0, 0, 0] = 0.0
    out = []
    for e in range(3):
        q = k[e].clone()
        if ng % 2 == 0:
            q.reshape(-1)[ng // 2] = 0.0
        a = torch.fft.irfftn(1j * q * green * mk, s=(ng, ng, ng), norm="forward").reshape(-1)
        out.append(sum(w * a[at] for at, w in corners))
    return torch.stack(out)


def _exact_training(case, seed):
    x, y, cw, w, m1, m2 = (t.double() if t.is_floating_point() else t.long() for t in _training_batch(case, seed))

    def bf(t):
        return t.to(torch.float32).to(torch.bfloat16).double()

    n, wr, at, part = case["n"], bf(w), 0, []
    for fan_in, fan_out in ((12, 64), (64, 64), (64, 8)):
        part.append((wr[at:at + fan_in * fan_out].reshape(fan_out, fan_in),
                     wr[at + fan_in * fan_out:at + fan_in * fan_out + fan_out]))
        at += fan_in * fan_out + fan_out
    grad, loss = torch.zeros_like(w), torch.zeros((), device="cuda", dtype=torch.float64)
    for lo in range(0, n, 65536):
        xb, yb = bf(x[lo:lo + 65536]), y[lo:lo + 65536]
        z1 = xb @ part[0][0].T + part[0][1]
        h1 = bf(z1.clamp(min=0))
        z2 = h1 @ part[1][0].T + part[1][1]
        h2 = bf(z2.clamp(min=0))
        p = torch.softmax(h2 @ part[2][0].T + part[2][1], 1)
        wt = cw[yb]
        loss += (-wt * torch.log(p.gather(1, yb[:, None])[:, 0].clamp(min=1e-30))).sum()
        d3 = p.clone()
        d3[torch.arange(len(yb), device="cuda"), yb] -= 1.0
        d3 *= wt[:, None]
        d2 = (d3 @ part[2][0]) * (z2 > 0)
        d1 = (d2 @ part[1][0]) * (z1 > 0)
        grad += torch.cat([t.reshape(-1) for t in (d1.T @ xb, d1.sum(0), d2.T @ h1, d2.sum(0), d3.T @ h2, d3.sum(0))])
    grad, loss = grad / n, loss / n
    m1, m2 = 0.9 * m1 + 0.1 * grad, 0.999 * m2 + 0.001 * grad * grad
    w = w - 3e-3 * (m1 / (1.0 - 0.9 ** 101)) / (torch.sqrt(m2 / (1.0 - 0.999 ** 101)) + 1e-8)
    return {"w": w, "m1": m1, "m2": m2, "wb": w.clone(), "grad": grad, "loss": loss.reshape(1)}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_training(case, seed)
    pos, mass, g = _particles(case, seed)
    if case["kind"] == "pm":
        return {"acc": _mesh_forces(case, pos, mass)}
    if case["kind"] != "step":
        acc = _direct_forces(case, pos, mass)
        return None if acc is None else {"acc": acc}
    vel, acc = (t.double() for t in _velocities(case, g))
    vel = vel + 0.5 * _DT * acc
    pos = torch.remainder(pos + _DT * vel, case["box"])
    acc = _direct_forces(case, pos, mass)
    if acc is None:
        return {"pos": pos, "vel": None, "acc": None}
    acc = acc + _mesh_forces(case, pos, mass)
    return {"pos": pos, "vel": vel + 0.5 * _DT * acc, "acc": acc}
