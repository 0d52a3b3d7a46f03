"""Performance cases: the work that users of this package have it do, each
through the public entry points, over the range of sizes in use.

``listed()`` gives the named cases, ``draw(rng)`` further ones of the same
ranges, ``prepare(case, seed)`` what a program has in hand before the call,
``run(state)`` one pass, ``work(case)`` the bytes and operations that a pass
cannot do without, and ``exact(case, seed)`` the outputs in 64 bits, written
with plain torch and none of the package's code.

Kinds of case:

* ``dam``: a dam break (optionally with obstacles) is uploaded from device
  arrays, advanced by ``steps`` time steps and read back by particle id:
  SPH stepping as a program does it.  Default formulation (Wendland C2,
  symplectic: two force evaluations per step) or the paper's (cubic spline,
  Verlet: one).
* ``ensemble``: many small dam breaks advanced in lockstep.
* ``subdomain``: the selection of a sub-domain's edge particles (Sec. 4.3),
  the data a decomposition along x sends to build its neighbours' halos.
* ``sort``: the stable (key, value) radix sort.
* ``forward``: one call of the learned surrogate (graph, encoders,
  message-passing layers, decoder).
* ``train``: forward and backward of the surrogate, returning the gradients.
* ``edge_layer``: one fused edge update of a message-passing layer.

Particles in motion: the generated lattices are jittered and given a smooth
velocity field with noise, and densities around the hydrostatic profile, as
a dam break has them once it moves.
"""
import functools
import math

import numpy as np
import torch

from paper_1210_1017_gb300 import cases as C
from paper_1210_1017_gb300 import sph as S
from paper_1210_1017_gb300 import surrogate as U

DEV = "cuda"
H_OVER_DP = 1.3
NEIGHBOURS = 4.0 / 3.0 * math.pi * (2 * H_OVER_DP) ** 3     # in the bulk of the fluid
LATENT, KIN, KOUT = 128, 16, 16


def listed():
    return [
        # the smallest configured dam break (6,000 fluid particles): latency
        # and launches count
        dict(name="dam_6k", kind="dam", tank="plain", dp=0.02, paper=False, steps=20),
        # a medium-size run in the paper's own formulation, at a ragged size
        dict(name="dam_60k_paper", kind="dam", tank="plain", dp=0.0093, paper=True, steps=10),
        # the one-million-particle case with obstacles
        dict(name="dam_obstacles_1m", kind="dam", tank="obstacles", dp=0.00733, paper=False, steps=4),
        # the headline workload: 35.4M particles
        dict(name="dam_32m", kind="dam", tank="plain", dp=0.00114, paper=False, steps=1),
        # 256 uneven dam breaks in lockstep (5.5M particles)
        dict(name="ensemble_256", kind="ensemble", members=256, steps=2),
        # what one of two slabs along x sends to its neighbour (2.1M particles)
        dict(name="subdomain_2m", kind="subdomain", dp=0.003, lo=0.0, hi=0.5),
        # 24-bit labels with 32-bit values, the size of a medium run
        dict(name="sort_4m", kind="sort", n=4000037, bits=24),
        # the fastest surrogate variant on the one-million-particle case
        dict(name="forward_1m_2_layers", kind="forward", tank="obstacles", dp=0.00733, layers=2,
             radius=0.65),
        # the configured network (10 layers, radius 2h) on the smallest case
        dict(name="forward_17k_10_layers", kind="forward", tank="plain", dp=0.02, layers=10,
             radius=1.0),
        # its training step on the smallest case
        dict(name="train_17k_10_layers", kind="train", tank="plain", dp=0.02, layers=10, radius=1.0),
        # one edge update as training keeps it (z written), ragged last tile
        dict(name="edge_layer_1500k", kind="edge_layer", edges=1500037, nodes=75001, z=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dp_for(fluid):
    return round((0.4 * 0.4 * 0.3 / fluid) ** (1.0 / 3.0), 6)


def draw(rng):
    kind = rng.choice(["dam", "dam", "dam", "dam", "ensemble", "subdomain", "sort", "forward",
                       "forward", "train", "edge_layer"])
    if kind == "dam":
        if rng.random() < 0.25:
            dp = round(_log(rng, 0.005, 0.02), 6)
            return dict(kind=kind, tank="obstacles", dp=dp, paper=rng.random() < 0.3,
                        steps=rng.randint(1, 4))
        fluid = _log(rng, 1500, 8e6)
        return dict(kind=kind, tank="plain", dp=_dp_for(fluid), paper=rng.random() < 0.3,
                    steps=max(1, min(30, int(4e6 / fluid * rng.uniform(0.3, 1.0)))))
    if kind == "ensemble":
        return dict(kind=kind, members=int(_log(rng, 3, 256)), steps=rng.randint(1, 4))
    if kind == "subdomain":
        lo = round(rng.uniform(0.0, 0.4), 3)
        return dict(kind=kind, dp=_dp_for(_log(rng, 2e4, 4e6)), lo=lo,
                    hi=round(lo + rng.uniform(0.25, 0.5), 3))
    if kind == "sort":
        return dict(kind=kind, n=int(_log(rng, 1e3, 3e7)), bits=rng.choice([8, 15, 16, 24, 32]))
    if kind == "forward":
        return dict(kind=kind, tank="plain", dp=_dp_for(_log(rng, 3e3, 4e5)),
                    layers=rng.randint(1, 6), radius=rng.choice([0.5, 0.65, 0.75, 1.0]))
    if kind == "train":
        return dict(kind=kind, tank="plain", dp=_dp_for(_log(rng, 3e3, 3e4)),
                    layers=rng.randint(1, 6), radius=rng.choice([0.65, 1.0]))
    edges = int(_log(rng, 2e3, 8e6))
    return dict(kind=kind, edges=edges, nodes=max(64, edges // rng.randint(12, 80)),
                z=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs --

@functools.lru_cache(maxsize=4)
def _geometry(tank, dp):
    """The generated lattice (no seed in it)."""
    return C.c2_dam_break_obstacles(dp=dp) if tank == "obstacles" else \
        C.dam_break(tank=(1.0, 0.4, 0.6), fluid=(0.4, 0.4, 0.3), dp=dp)


@functools.lru_cache(maxsize=2)
def _ensemble(members):
    return C.dam_break_ensemble(members)


def _moving(pos, rho, fluid, dp, seed):
    """Device arrays of a lattice set in motion: fluid positions jittered by
    up to 0.15 dp per axis, a velocity field of three smooth modes (up to
    about 1 m/s) with 5% noise, densities with 0.05% noise."""
    g = torch.Generator(DEV).manual_seed(int(seed))
    x = torch.from_numpy(pos).to(DEV)
    n = x.shape[0]
    f = fluid.to(torch.float64)[:, None]
    jit = torch.rand((n, 3), device=DEV, dtype=torch.float64, generator=g)
    x = x + f * ((jit - 0.5) * (0.3 * dp))
    del jit
    k = torch.rand((3, 3), device=DEV, dtype=torch.float64, generator=g) * 12.0
    ph = torch.rand((3, 3), device=DEV, dtype=torch.float64, generator=g) * 6.28
    vel = torch.empty((n, 3), device=DEV, dtype=torch.float32)
    for a in range(3):
        v = sum(torch.sin(x[:, b] * k[a, b] + ph[a, b]) for b in range(3)) / 3.0
        vel[:, a] = v.float()
    vel += 0.05 * torch.randn((n, 3), device=DEV, generator=g)
    vel *= fluid[:, None]
    r = torch.from_numpy(rho).to(DEV)
    r = r * (1.0 + 5e-4 * torch.randn(n, device=DEV, generator=g))
    return x.contiguous(), vel.contiguous(), r.contiguous()


def _params(case):
    g = _geometry(case["tank"], case["dp"])
    p = g.params()
    if case.get("paper"):
        p.update(kernel="cubic", integrator="verlet")
    return g, p


def _dam_inputs(case, seed):
    g, p = _params(case)
    fluid = torch.arange(g.n, device=DEV) >= g.n_bound
    pos, vel, rho = _moving(g.pos, g.rho, fluid, g.dp, seed)
    ids = torch.arange(g.n, device=DEV, dtype=torch.int32)
    return g, p, fluid, pos, vel, rho, ids


def _buffers(n):
    return dict(pos=torch.empty((n, 3), device=DEV, dtype=torch.float64),
                vel=torch.empty((n, 3), device=DEV, dtype=torch.float32),
                rho=torch.empty(n, device=DEV, dtype=torch.float32))


@functools.lru_cache(maxsize=1)
def _stream():
    """One stream for the program's simulations."""
    return torch.cuda.Stream()


def _layer_shapes(layers):
    s = [(KIN, LATENT, 1), (LATENT, LATENT, 1), (KIN, LATENT, 1), (LATENT, LATENT, 1)]
    for _ in range(layers):
        s += [(LATENT, LATENT, 0), (LATENT, LATENT, 0), (LATENT, LATENT, 1), (LATENT, LATENT, 1),
              (2 * LATENT, LATENT, 1), (LATENT, LATENT, 1)]
    return s + [(LATENT, LATENT, 1), (LATENT, KOUT, 1)]


def _weights(layers, seed):
    """Random weights at the scale of a trained network: residual branches
    small, the aggregated input of the node update scaled down."""
    rng = np.random.default_rng([int(seed), 7])
    out = []
    for k, (a, b, bias) in enumerate(_layer_shapes(layers)):
        last = 4 <= k < 4 + 6 * layers and (k - 4) % 6 in (3, 5)
        w = rng.standard_normal((a, b)) * ((0.2 if last else 1.0) / math.sqrt(a))
        if a == 2 * LATENT:
            w[LATENT:] *= 0.1
        out.append(w.ravel())
        if bias:
            out.append(0.05 * rng.standard_normal(b))
    return np.concatenate(out).astype(np.float32)


def _surrogate_inputs(case, seed):
    g, p, fluid, pos, vel, rho, ids = _dam_inputs(case, seed)
    gen = torch.Generator(DEV).manual_seed(int(seed) + 1)
    # five velocities, oldest first: the current one with a little drift
    drift = 0.05 * torch.randn((g.n, 5, 3), device=DEV, generator=gen)
    hist = ((vel[:, None, :] + drift) * fluid[:, None, None]).reshape(g.n, 15).contiguous()
    target = torch.randn((g.n, 3), device=DEV, generator=gen)
    return g, p, fluid, pos, vel, rho, ids, hist, target, _weights(case["layers"], seed)


def _edge_inputs(case, seed):
    gen = torch.Generator(DEV).manual_seed(int(seed))
    M, N = case["edges"], case["nodes"]

    def bf(*shape, scale=1.0):
        return (scale * torch.randn(shape, device=DEV, generator=gen)).to(torch.bfloat16)

    # edges sorted by receiving node, sending nodes nearby in the cell order
    src = (torch.arange(M, device=DEV, dtype=torch.int64) * N) // M
    dst = (src + torch.randint(-2000, 2001, (M,), device=DEV, generator=gen)) % N
    return dict(E=bf(M, LATENT), W1t=bf(LATENT, LATENT, scale=0.09), W2t=bf(LATENT, LATENT, scale=0.09),
                b1=0.05 * torch.randn(LATENT, device=DEV, generator=gen),
                b2=0.05 * torch.randn(LATENT, device=DEV, generator=gen),
                P=bf(N, LATENT), Q=bf(N, LATENT), src=src.to(torch.int32), dst=dst.to(torch.int32))


def _sort_inputs(case, seed):
    gen = torch.Generator(DEV).manual_seed(int(seed))
    n, bits = case["n"], case["bits"]
    keys = torch.randint(0, 1 << bits, (n,), device=DEV, generator=gen, dtype=torch.int64)
    vals = torch.randint(0, 1 << 31, (n,), device=DEV, generator=gen, dtype=torch.int64)
    return keys.to(torch.int32), vals.to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("dam", "subdomain"):
        case = dict(dict(tank="plain"), **case)
        g, p, _, pos, vel, rho, ids = _dam_inputs(case, seed)
        sim = S.Simulation(p, g.n, stream=_stream())
        st = dict(kind=kind, sim=sim, inp=(pos, vel, rho, ids))
        sim.upload(*st["inp"])
        sim.build_cells()
        if kind == "dam":
            sim.autotune()
            st.update(steps=case["steps"], out=_buffers(g.n))
            return st
        # room for every particle; what is not selected stays zero
        st.update(lo=case["lo"], hi=case["hi"], out=_buffers(g.n),
                  oid=torch.zeros(g.n, device=DEV, dtype=torch.int32))
        for v in st["out"].values():
            v.zero_()
        sim.synchronize()
        return st
    if kind == "ensemble":
        ens = _ensemble(case["members"])
        base = torch.from_numpy(ens.id_base).to(DEV)
        nb = torch.tensor([m["n_bound"] for m in ens.members], device=DEV)
        ids = torch.arange(ens.n, device=DEV)
        q = torch.searchsorted(base, ids, right=True) - 1
        fluid = ids - base[q] >= nb[q]
        pos, vel, rho = _moving(ens.pos, ens.rho, fluid, ens.cases[0].dp, seed)
        sim = S.Simulation(ens.params, ens.n, members=ens.members, stream=_stream())
        st = dict(kind="dam", sim=sim, inp=(pos, vel, rho, ids.to(torch.int32)), steps=case["steps"],
                  out=_buffers(ens.n))
        sim.upload(*st["inp"])
        sim.build_cells()
        sim.autotune()
        return st
    if kind == "sort":
        keys, vals = _sort_inputs(case, seed)
        nb = int(S.lib().sph_radix_sort_scratch_bytes(case["n"]))
        return dict(kind=kind, keys=keys, vals=vals, ko=torch.empty_like(keys),
                    vo=torch.empty_like(vals), n=case["n"], bits=case["bits"], nb=nb,
                    scratch=torch.empty(nb, device=DEV, dtype=torch.uint8))
    if kind in ("forward", "train"):
        g, p, _, pos, vel, rho, ids, hist, target, w = _surrogate_inputs(case, seed)
        sim = S.Simulation(p, g.n, stream=_stream())
        sim.upload(pos, vel, rho, ids)
        sim.build_cells()
        sur = U.Surrogate(sim, layers=case["layers"], train=kind == "train", v_scale=0.5,
                          radius=case["radius"],
                          edges_per_node=int(90 * case["radius"] ** 3) + 8)
        sur.set_params(w)
        return dict(kind=kind, sim=sim, sur=sur, hist=hist, target=target,
                    acc=torch.empty((g.n, 3), device=DEV, dtype=torch.float32))
    if kind == "edge_layer":
        t = _edge_inputs(case, seed)
        return dict(kind=kind, M=case["edges"], Z=torch.empty_like(t["E"]) if case["z"] else None,
                    Eout=torch.empty_like(t["E"]), **t)
    raise ValueError(kind)


def run(st):
    kind = st["kind"]
    if kind == "dam":
        sim, out = st["sim"], st["out"]
        sim.upload(*st["inp"])
        sim.step(st["steps"])
        sim.download_by_id(out["pos"], out["vel"], out["rho"])
        return out
    if kind == "subdomain":
        out = st["out"]
        counts = S.sph_subdomain_select(st["sim"].ctx, S.SPH_SUBDOMAIN_EDGE, st["lo"], st["hi"],
                                        st["oid"].shape[0], out["pos"], out["vel"], out["rho"],
                                        st["oid"])
        return dict(counts=counts.astype(np.int64), ids=st["oid"], **out)
    if kind == "sort":
        S.sph_radix_sort_pairs(st["keys"], st["vals"], st["ko"], st["vo"], st["n"], st["bits"],
                               st["scratch"], st["nb"], torch.cuda.current_stream().cuda_stream)
        return [st["ko"], st["vo"]]
    if kind == "forward":
        st["sur"].forward(st["hist"], st["acc"])
        return st["acc"]
    if kind == "train":
        st["sur"].forward(st["hist"], st["acc"])
        loss = st["sur"].backward(st["target"])
        return dict(acc=st["acc"], loss=loss, grads=st["sur"].grads())
    U.sur_edge_layer(st["E"], st["W1t"], st["W2t"], st["b1"], st["b2"], st["P"], st["Q"], st["src"],
                     st["dst"], st["M"], st["Z"], st["Eout"], torch.cuda.current_stream().cuda_stream)
    return [st["Eout"]] + ([st["Z"]] if st["Z"] is not None else [])


# -------------------------------------------------------------------- work --

def _size(case):
    if case["kind"] == "ensemble":
        return _ensemble(case["members"]).n
    dp = case["dp"]
    fluid = (0.8 * 1.0 * 0.5 if case.get("tank") == "obstacles" else 0.4 * 0.4 * 0.3) / dp ** 3
    # two layers of boundary particles on the floor and the four walls
    if case.get("tank") == "obstacles":
        wall = 3.2 * 1.0 + 2 * (3.2 + 1.0) * 0.8
    else:
        wall = 1.0 * 0.4 + 2 * (1.0 + 0.4) * 0.6
    return fluid + 2 * wall / dp ** 2


def work(case):
    kind = case["kind"]
    if kind in ("dam", "ensemble"):
        n, steps = _size(case), case["steps"]
        evals = steps * (1 if case.get("paper") else 2)
        # state in (position, velocity, density, id), state out; 50 flop a pair
        return dict(bytes=n * (44 + 40), flops=n * NEIGHBOURS * 50 * evals)
    if kind == "subdomain":
        n = _size(case)
        share = 2 * (2 * H_OVER_DP * case["dp"]) / 1.0
        return dict(bytes=n * 8 + 2 * 44 * n * share, flops=2 * n)
    if kind == "sort":
        return dict(bytes=16.0 * case["n"], flops=0.0)
    if kind == "edge_layer":
        M, N = case["edges"], case["nodes"]
        return dict(bytes=M * LATENT * 2 * (3 if case["z"] else 2) + 8 * M + 2 * N * LATENT * 2,
                    flops=2 * 2.0 * M * LATENT * LATENT)
    n = _size(case)
    edges = n * NEIGHBOURS * case["radius"] ** 3 * 0.8
    nl = case["layers"]
    flops = 2.0 * edges * LATENT * (KIN + LATENT + nl * 2 * LATENT) + \
        2.0 * n * LATENT * (KIN + LATENT + nl * 5 * LATENT + LATENT + KOUT)
    # positions, histories in, accelerations out, weights
    byt = n * (24 + 60 + 12) + 4.0 * sum(a * b for a, b, _ in _layer_shapes(nl))
    return dict(bytes=byt * (2 if kind == "train" else 1), flops=flops * (3 if kind == "train" else 1))


# ------------------------------------------------------------- 64-bit values --

class _Pairs:
    """Neighbour pairs |r_ij| < rc by cells of size rc (per group of
    particles; the grid has a margin of one cell), delivered as index lists
    with at most one pair per i each."""

    def __init__(self, pos, rc, group=None):
        self.pos, self.rc2 = pos, rc * rc
        lo = pos.min(0).values - rc
        c = torch.floor((pos - lo) / rc).to(torch.int64)
        dims = (c.max(0).values + 2).tolist()
        self.nx, self.ny, self.nz = dims
        cell = c[:, 0] + self.nx * (c[:, 1] + self.ny * c[:, 2])
        total = self.nx * self.ny * self.nz
        if group is not None:
            cell = cell + group * total
            total *= int(group.max()) + 1
        self.order = torch.argsort(cell)
        cnt = torch.bincount(cell, minlength=total)
        self.start = torch.cumsum(cnt, 0) - cnt
        self.cnt, self.cell, self.total = cnt, cell, total
        self.most = int(cnt.max())

    def lists(self):
        p = self.pos
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    nb = self.cell + dx + self.nx * (dy + self.ny * dz)
                    ok = (nb >= 0) & (nb < self.total)
                    nb = nb.clamp(0, self.total - 1)
                    s, m = self.start[nb], torch.where(ok, self.cnt[nb], 0)
                    for k in range(self.most):
                        i = (m > k).nonzero()[:, 0]
                        if i.numel() == 0:
                            break
                        j = self.order[s[i] + k]
                        d = p[i] - p[j]
                        r2 = (d * d).sum(1)
                        keep = (r2 < self.rc2) & (i != j)
                        i, j, d, r2 = i[keep], j[keep], d[keep], r2[keep]
                        if i.numel():
                            yield i, j, d, r2


def _rates(p, c0, pos, vel, rho, fluid, q, nq, cubic):
    """Accelerations, density rates and the CFL terms of Eqs. 7 and 9."""
    h = p["h"]
    eta2 = p["eta2_coef"] * h * h
    x = rho / p["rho0"]
    pr = c0 ** 2 * p["rho0"] / 7.0 * (x ** 7 - 1.0) / rho ** 2
    c = c0 * x ** 3
    n = pos.shape[0]
    a = torch.zeros((n, 3), device=DEV, dtype=torch.float64)
    dr = torch.zeros(n, device=DEV, dtype=torch.float64)
    mu = torch.zeros(n, device=DEV, dtype=torch.float64)
    for i, j, d, r2 in _Pairs(pos, 2 * h, q if nq > 1 else None).lists():
        s = torch.sqrt(r2) / h
        if cubic:
            F = torch.where(s < 1, 2.25 * s - 3.0, -0.75 * (2 - s) ** 2 / s) / (math.pi * h ** 5)
        else:
            F = -5.0 * 21.0 / (16.0 * math.pi * h ** 5) * (1 - 0.5 * s) ** 3
        vr = ((vel[i] - vel[j]) * d).sum(1)
        dr[i] += vr * F
        nu = h * vr / (r2 + eta2)
        visc = torch.where(vr < 0, -p["alpha"] * (c[i] + c[j]) * nu / (rho[i] + rho[j]), 0.0)
        a[i] -= ((pr[i] + pr[j] + visc) * F)[:, None] * d
        mu[i] = torch.maximum(mu[i], nu.abs())
    g = torch.tensor(p["gravity"], device=DEV, dtype=torch.float64)
    a = torch.where(fluid[:, None], p["mass"] * a + g, 0.0)
    mu = torch.where(fluid, mu, 0.0)

    def most(v):
        return torch.zeros(nq, device=DEV, dtype=torch.float64).scatter_reduce_(0, q, v, "amax")

    am = torch.sqrt(most((a * a).sum(1)))
    dt = p["cfl"] * torch.minimum(torch.sqrt(h / am), h / (most(c) + most(mu)))
    return a, p["mass"] * dr, dt[q]


def _advance(p, c0, pos, vel, rho, fluid, q, nq, steps, paper):
    f = fluid[:, None].to(torch.float64)
    pv, prho = vel, rho
    for k in range(steps):
        a, dr, dt = _rates(p, c0, pos, vel, rho, fluid, q, nq, paper)
        D = dt[:, None]
        if paper:   # Verlet; the first step, and every 40th, is an Euler step
            euler = k % int(p["verlet_every"]) == 0
            v1 = vel + D * a if euler else pv + 2 * D * a
            r1 = rho + dt * dr if euler else prho + 2 * dt * dr
            pos = pos + f * (D * vel + 0.5 * D * D * a)
            pv, prho = vel, rho
            vel, rho = torch.where(fluid[:, None], v1, vel), r1
            continue
        ph, vh, rh = pos + f * (0.5 * D * vel), vel + 0.5 * D * a, rho + 0.5 * dt * dr
        a, dr, _ = _rates(p, c0, ph, vh, rh, fluid, q, nq, paper)
        v1 = vel + D * a
        pos = pos + f * (0.5 * D * (v1 + vel))
        eps = -dr * dt / rh
        vel, rho = v1, rho * (2 - eps) / (2 + eps)
    return dict(pos=pos, vel=vel, rho=rho)


def _network(w, layers, xn, xe, src, dst):
    """The surrogate's outputs (normalised) from its flat parameters."""
    at, mats = 0, []
    for a, b, bias in _layer_shapes(layers):
        W = w[at:at + a * b].reshape(a, b)
        at += a * b
        mats.append((W, w[at:at + b] if bias else None))
        at += b if bias else 0

    def lin(k, v):
        W, b = mats[k]
        return v @ W if b is None else v @ W + b

    h = lin(1, torch.relu(lin(0, xn)))
    e = lin(3, torch.relu(lin(2, xe)))
    for k in range(4, 4 + 6 * layers, 6):
        z = torch.relu(lin(k, h)[src] + lin(k + 1, h)[dst] + lin(k + 2, e))
        e = e + lin(k + 3, z)
        agg = torch.zeros_like(h).index_add(0, src, e)
        h = h + lin(k + 5, torch.relu(lin(k + 4, torch.cat([h, agg], 1))))
    k = 4 + 6 * layers
    return lin(k + 1, torch.relu(lin(k, h)))[:, :3]


def exact(case, seed):
    kind = case["kind"]
    f64 = torch.float64
    if kind == "dam":
        if _size(case) * case["steps"] > 9e6:
            return None
        g, p, fluid, pos, vel, rho, _ = _dam_inputs(case, seed)
        q = torch.zeros(g.n, device=DEV, dtype=torch.int64)
        c0 = torch.full((g.n,), g.c0, device=DEV, dtype=f64)
        return _advance(p, c0, pos, vel.to(f64), rho.to(f64), fluid, q, 1, case["steps"],
                        bool(case.get("paper")))
    if kind == "ensemble":
        ens = _ensemble(case["members"])
        if ens.n * case["steps"] > 9e6:
            return None
        base = torch.from_numpy(ens.id_base).to(DEV)
        nb = torch.tensor([m["n_bound"] for m in ens.members], device=DEV)
        cs = torch.tensor([m["c0"] for m in ens.members], device=DEV, dtype=f64)
        ids = torch.arange(ens.n, device=DEV)
        q = torch.searchsorted(base, ids, right=True) - 1
        fluid = ids - base[q] >= nb[q]
        pos, vel, rho = _moving(ens.pos, ens.rho, fluid, ens.cases[0].dp, seed)
        return _advance(ens.params, cs[q], pos, vel.to(f64), rho.to(f64), fluid, q,
                        len(ens.members), case["steps"], False)
    if kind == "subdomain":
        g, p, _, pos, vel, rho, _ = _dam_inputs(dict(case, tank="plain"), seed)
        x, w = pos[:, 0], 2.0 * p["h"]
        a = ((x >= case["lo"]) & (x < case["lo"] + w)).nonzero()[:, 0]
        b = ((x >= case["hi"] - w) & (x < case["hi"])).nonzero()[:, 0]
        k = torch.cat([a, b])

        def padded(v):
            t = torch.zeros(v.shape, device=DEV, dtype=f64)
            t[:k.numel()] = v[k].to(f64)
            return t

        return dict(counts=None, ids=None, pos=padded(pos), vel=padded(vel), rho=padded(rho))
    if kind == "edge_layer":
        t = _edge_inputs(case, seed)
        s, d = t["src"].long(), t["dst"].long()
        E = t["E"].to(f64)
        z = torch.relu(E @ t["W1t"].to(f64).T + t["b1"].to(f64) + t["P"].to(f64)[s] + t["Q"].to(f64)[d])
        out = E + z @ t["W2t"].to(f64).T + t["b2"].to(f64)
        return [out, z] if case["z"] else [out]
    if kind in ("forward", "train"):
        if _size(case) * case["radius"] ** 3 * case["layers"] > 2e6:
            return None
        g, p, fluid, pos, _, _, _, hist, target, wf = _surrogate_inputs(case, seed)
        rc = case["radius"] * 2.0 * p["h"]
        got = list(_Pairs(pos, rc).lists())
        src, dst = (torch.cat([v[k] for v in got]) for k in (0, 1))
        d, r = torch.cat([v[2] for v in got]), torch.sqrt(torch.cat([v[3] for v in got]))
        xe = torch.zeros((src.numel(), KIN), device=DEV, dtype=f64)
        xe[:, :3], xe[:, 3] = d / (2 * p["h"]), r / (2 * p["h"])
        xn = torch.cat([hist.to(f64) / 0.5, (~fluid)[:, None].to(f64)], 1)
        w = torch.from_numpy(wf.astype(np.float64)).to(DEV).requires_grad_(kind == "train")
        out = _network(w, case["layers"], xn, xe, src, dst)
        if kind == "forward":
            return out
        loss = ((out - target.to(f64)) ** 2)[fluid].sum() / int(fluid.sum())
        loss.backward()
        return dict(acc=out.detach(), loss=loss.detach(), grads=w.grad)
    return None
