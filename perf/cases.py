"""Timed cases of the framework's public entry points (Domain, Batch), over the
range of sizes, lattices, precisions, geometries and options in use.

A case's pass advances a prepared simulation by some time steps and reads its
fields back, as a user's program does between two frames of output.  The next
pass on the same state goes on from there.  Fields come back in the precision
the domain works in (float16 for FP16 population storage), the type a program
keeps its frames in.

`exact` integrates the same model in plain torch float64: lattice-order sums,
populations N and B streamed separately, halfway bounce-back, ghost colors from
the fluid point x_G + n.
"""
import functools
import math

import numpy as np
import torch

from paper_2605_30878_gb300 import lbm
from paper_2605_30878_gb300 import workloads as wl

_PRECISION = {"fp64": lbm.FP64, "fp32": lbm.FP32, "fp16": lbm.FP16}
_FRAME = {"fp64": np.float64, "fp32": np.float32, "fp16": np.float16}
_VALUE_BYTES = {"fp64": 8, "fp32": 4, "fp16": 4}        # phi, u
_MOVING_BYTES = {"fp64": 8, "fp32": 4, "fp16": 2}       # a stored moving population


def listed():
    return [
        # validation against the paper in FP64 on its smallest grid: a few
        # steps at a time, bound by launches and latency
        dict(name="cylinder 64x64 fp64", kind="cylinder", nx=64, ny=64, nz=1, precision="fp64", ratio=1.0, rule=0,
             gravity=0.0, steps=16, fields="phi u p", geometry=0, domains=1),
        # stepping one step at a time with a look at the fields after each
        # (a driver that couples the step to something else)
        dict(name="cylinder 201x201 one step", kind="cylinder", nx=201, ny=201, nz=1, precision="fp32", ratio=1000.0,
             rule=0, gravity=0.0, steps=1, fields="phi", geometry=1, domains=1),
        # the paper's drop on a cylinder (odd grid, density ratio 1000)
        dict(name="cylinder 401x401 fp32", kind="cylinder", nx=401, ny=401, nz=1, precision="fp32", ratio=1000.0,
             rule=0, gravity=0.0, steps=200, fields="phi", geometry=2, domains=1),
        # the paper's drop on a plate between walls, FP64 as the paper runs it
        dict(name="plate 500x300 fp64", kind="plate", nx=500, ny=300, nz=1, precision="fp64", ratio=1000.0, rule=0,
             gravity=1e-5, steps=20, fields="phi u", geometry=0, domains=1),
        # its larger grid in the production precision
        dict(name="plate 1000x600 fp32", kind="plate", nx=1000, ny=600, nz=1, precision="fp32", ratio=1000.0, rule=0,
             gravity=0.0, steps=400, fields="phi", geometry=0, domains=1),
        # a small ragged 3D box with the comparison scheme's ghost rule
        dict(name="sphere 49x52x47 fp32", kind="sphere", nx=49, ny=52, nz=47, precision="fp32", ratio=10.0, rule=1,
             gravity=1e-5, steps=50, fields="phi u", geometry=3, domains=1),
        # 3D validation in FP64
        dict(name="sphere 64^3 fp64", kind="sphere", nx=64, ny=64, nz=64, precision="fp64", ratio=1000.0, rule=0,
             gravity=1e-5, steps=6, fields="phi u", geometry=4, domains=1),
        # the production run: 3D drop on a sphere at density ratio 1000
        dict(name="sphere 192^3 fp32", kind="sphere", nx=192, ny=192, nz=192, precision="fp32", ratio=1000.0, rule=0,
             gravity=0.0, steps=400, fields="phi", geometry=5, domains=1),
        # the same with half-width populations, for runs bound by memory size
        dict(name="sphere 192^3 fp16", kind="sphere", nx=192, ny=192, nz=192, precision="fp16", ratio=1000.0, rule=0,
             gravity=0.0, steps=400, fields="phi", geometry=5, domains=1),
        # imbibition into a porous sphere packing: bounce-back and ghost nodes
        # everywhere, no density contrast
        dict(name="packing 128^3 fp32", kind="packing", nx=128, ny=128, nz=128, precision="fp32", ratio=1.0, rule=0,
             gravity=0.0, steps=100, fields="phi", geometry=1, domains=1),
        # a parameter sweep: ragged 3D domains of all density ratios in one batch
        dict(name="batch of 12 spheres fp32", kind="sphere", nx=72, ny=76, nz=70, precision="fp32", ratio=0.0, rule=0,
             gravity=0.0, steps=50, fields="phi", geometry=6, domains=12),
        # a serving chunk: 2D requests stepped together
        dict(name="batch of 16 cylinders fp32", kind="cylinder", nx=260, ny=300, nz=1, precision="fp32", ratio=0.0,
             rule=0, gravity=0.0, steps=100, fields="phi", geometry=7, domains=16),
    ]


def draw(rng):
    """One more case: any family, sizes and node updates log-uniform over the listed range."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["cylinder", "plate", "sphere", "sphere", "packing"])
    precision = rng.choice(["fp32", "fp32", "fp16", "fp64"])
    domains = 1
    if kind == "packing":
        n = size(64, 160)
        nx = ny = nz = n
        ratio = 1.0
    else:
        ratio = rng.choice([1.0, 10.0, 1000.0])
        if kind == "sphere":
            nx, ny, nz = size(32, 190), size(32, 190), size(32, 190)
        else:
            nx, ny, nz = size(64, 1000), size(64, 600), 1
        if kind != "plate" and nx * ny * nz < 500000 and precision != "fp64" and rng.random() < 0.4:
            domains = rng.randint(2, 16)
            ratio = 0.0
    nodes = nx * ny * nz * domains
    most = {"fp64": 2e7, "fp32": 1.4e9, "fp16": 1.4e9}[precision]
    least = max(1.0, 2e5 / nodes)
    steps = int(min(100 if kind == "packing" else 400, max(1, round(math.exp(rng.uniform(math.log(least), math.log(max(least, most / nodes))))))))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, ratio=ratio, rule=rng.choice([0, 0, 0, 1]),
                gravity=0.0 if kind == "packing" else rng.choice([0.0, 1e-6]), steps=steps, fields="phi",
                geometry=rng.randint(10, 99), domains=domains)


# ---------------------------------------------------------------- inputs
def _sizes(case):
    """(nx, ny, nz) of each domain: the case's for one domain, spread by +/- 30% in a batch."""
    rng = np.random.default_rng(1000 + case["geometry"])
    out = []
    for _ in range(case["domains"]):
        f = 1.0 if case["domains"] == 1 else float(rng.uniform(0.7, 1.3))
        nz = 1 if case["nz"] == 1 else max(24, int(round(case["nz"] * f)))
        out.append((max(24, int(round(case["nx"] * f))), max(24, int(round(case["ny"] * f))), nz))
    return out


@functools.lru_cache(maxsize=4)
def _geometry(kind, geometry, nx, ny, nz):
    """Solid mask, ghost list and where the drop goes: (solid, (nodes, normals), center, R)."""
    rng = np.random.default_rng(geometry)
    lattice = 9 if nz == 1 else 19
    shape = (nz, ny, nx)
    if kind == "plate":
        solid, ghosts = wl.wall_domain(9, shape, 1, 1)
        return solid, ghosts, (nx / 2.0, 0.5, 0.0), 0.0
    if kind == "packing":
        reservoir = max(12, nx // 8)
        centers, radii = wl.sphere_packing(nx, r_min=8.0, r_max=16.0, porosity=0.45, reservoir=reservoir, seed=geometry)
        solid, ghosts = wl.packing_domain(centers, radii, nx)
        return solid, ghosts, (reservoir / 2.0, 0.0, 0.0), float(reservoir)
    small = min(nx, ny) if nz == 1 else min(nx, ny, nz)
    R = (0.2 if kind == "cylinder" else 1.0 / 6.0) * small
    center = tuple(n / 2.0 + float(rng.uniform(-0.5, 0.5)) for n in ((nx, ny) if nz == 1 else (nx, ny, nz)))
    center += (0.0,) * (3 - len(center))
    solid, ghosts = wl.sphere_domain(lattice, shape, center, R)
    return solid, ghosts, center, R


def _domain_inputs(case, seed):
    """Per domain: (params, solid, ghosts, initial color or (drop centre, radius))."""
    rng = np.random.default_rng([seed, case["geometry"]])
    out = []
    for nx, ny, nz in _sizes(case):
        solid, ghosts, center, R = _geometry(case["kind"], case["geometry"], nx, ny, nz)
        theta = math.radians(float(rng.uniform(40.0, 140.0)))
        ratio = case["ratio"] or float(rng.choice([1.0, 10.0, 1000.0]))
        params = dict(lattice=9 if nz == 1 else 19, nx=nx, ny=ny, nz=nz, periodic=5 if case["kind"] == "plate" else 7,
                      rho_l=ratio, rho_g=1.0, mu_l=0.1 * (100.0 if ratio == 1000.0 else 1.0), mu_g=0.1, sigma=0.005,
                      W=4.0, M_phi=0.02, theta=theta, ghost_rule=case["rule"],
                      g=(0.0, 0.0, -case["gravity"]) if nz > 1 else (0.0, -case["gravity"], 0.0),
                      precision=_PRECISION[case["precision"]])
        jitter = rng.uniform(-1.0, 1.0, 3)
        if case["kind"] == "packing":                  # a liquid slab in the reservoir
            width = R / 2.0 + 0.5 * jitter[0]
            x = np.arange(nx)
            d = np.abs((x - center[0] + nx / 2.0) % nx - nx / 2.0)
            phi = np.broadcast_to(0.5 * (1.0 + np.tanh(2.0 * (width - d) / 4.0)), (nz, ny, nx)).copy()
            out.append((params, solid, ghosts, phi))
            continue
        if case["kind"] == "plate":                    # a spreading cap
            r0 = 0.3 * min(nx / 2.0, ny) + jitter[2]
            drop = (center[0] + jitter[0], center[1] + 0.3 * r0 + 0.2 * jitter[1], 0.0)
        else:                                          # a drop near its place on the solid
            r0 = 0.75 * R * (1.0 + 0.03 * jitter[2])
            drop = wl.droplet_on_sphere_center(center, R, r0, theta + 0.2 * jitter[0], axis=1 if nz == 1 else 2)
            drop[0] += 0.3 * jitter[1]
        out.append((params, solid, ghosts, (tuple(drop), float(r0))))
    return out


def prepare(case, seed):
    doms = []
    for params, solid, ghosts, start in _domain_inputs(case, seed):
        d = lbm.Domain(params, solid, ghosts)
        if isinstance(start, tuple):
            d.init_droplet(*start)
        else:
            d.init_phi(start)
        doms.append(d)
    batch = lbm.Batch(doms) if case["domains"] > 1 else None
    if batch is not None and case["nz"] > 1:
        batch.set_variant(5)                           # the shape the tuner keeps for 3D batches
    return dict(domains=doms, batch=batch, steps=case["steps"], fields=case["fields"].split(),
                frame=_FRAME[case["precision"]])


def run(state):
    (state["batch"] or state["domains"][0]).step(state["steps"])
    return [{f: d.read(f).astype(state["frame"], copy=False) for f in state["fields"]} for d in state["domains"]]


def work(case):
    """Every step reads and writes the state that the next one needs: the moving
    populations of N, the color, the velocity, and the recolouring flux (a vector)
    that with N and the color makes up B."""
    s, m = _VALUE_BYTES[case["precision"]], _MOVING_BYTES[case["precision"]]
    nodes = sum(_fluid_share(case) * nx * ny * nz for nx, ny, nz in _sizes(case))
    Q, D = (9, 2) if case["nz"] == 1 else (19, 3)
    per_node = 2 * ((Q - 1) * m + s + 2 * D * s)
    flops = 210 if Q == 9 else 520                     # one step of one node, multiply-adds as two
    return {"bytes": nodes * per_node * case["steps"], "flops": nodes * flops * case["steps"]}


def _fluid_share(case):
    return {"packing": 0.52, "plate": 0.99, "cylinder": 0.87, "sphere": 0.98}[case["kind"]]


# ---------------------------------------------------------------- the model in 64 bits
def _lattice(Q):
    if Q == 9:
        c = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    else:
        pairs = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
        c = [(0, 0, 0)] + [v for p in pairs for v in (p, tuple(-a for a in p))]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    return c, w, [c.index(tuple(-a for a in v)) for v in c]


def _at(f, c):
    """f(x + c), periodic."""
    return torch.roll(f, shifts=(-c[2], -c[1], -c[0]), dims=(-3, -2, -1))


def _ghost_points(solid, nodes, normals, c, dev):
    """Corners (flat fluid node indices) and weights of each ghost's fluid point."""
    nz, ny, nx = solid.shape
    dims = torch.tensor([nx, ny, nz], device=dev)
    xyz = torch.stack([nodes % nx, (nodes // nx) % ny, nodes // (nx * ny)], 1)
    D = 2 if nz == 1 else 3
    flat = ~solid.reshape(-1)
    point = xyz.double() + normals
    base = torch.floor(point)
    frac = point - base
    index, weight = [], []
    for k in range(1 << D):
        at, wt = [], torch.ones(len(nodes), dtype=torch.float64, device=dev)
        for a in range(3):
            bit = (k >> a) & 1 if a < D else 0
            at.append((base[:, a].long() + bit) % dims[a] if a < D else torch.zeros_like(nodes))
            if a < D:
                wt = wt * (frac[:, a] if bit else 1.0 - frac[:, a])
        node = at[0] + nx * (at[1] + ny * at[2])
        index.append(node)
        weight.append(torch.where(flat[node], wt, torch.zeros_like(wt)))
    index, weight = torch.stack(index), torch.stack(weight)
    total = weight.sum(0)
    # no fluid corner: the fluid neighbour most aligned with the normal, ties to the smaller index
    best = torch.full((len(nodes),), -1e300, dtype=torch.float64, device=dev)
    where = torch.full_like(nodes, -1)
    for v in c[1:]:
        at = (xyz + torch.tensor(v, device=dev)) % dims
        node = at[:, 0] + nx * (at[:, 1] + ny * at[:, 2])
        dot = normals[:, 0] * v[0] + normals[:, 1] * v[1] + normals[:, 2] * v[2]
        take = flat[node] & ((dot > best) | ((dot == best) & (node < where)))
        best, where = torch.where(take, dot, best), torch.where(take, node, where)
    lost = total <= 0
    index[0] = torch.where(lost, where, index[0])
    weight[0] = torch.where(lost, torch.ones_like(total), weight[0])
    return index, weight / torch.where(lost, torch.ones_like(total), total)


def _integrate(P, solid_np, ghosts, start, steps):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    Q = P["lattice"]
    c, w, opp = _lattice(Q)
    D, cs2 = (2, 1 / 3) if Q == 9 else (3, 1 / 3)
    nz, ny, nx = solid_np.shape
    solid = torch.from_numpy(solid_np.astype(bool)).to(dev)
    fluid = ~solid
    nodes = torch.from_numpy(np.asarray(ghosts[0], np.int64)).to(dev)
    normals = torch.from_numpy(np.asarray(ghosts[1], np.float64).reshape(-1, 3)).to(dev)
    corner, weight = _ghost_points(solid, nodes, normals, c, dev)
    alpha = 1.0 - 2.0 * P["M_phi"] * (1.0 - w[0]) / cs2
    if Q == 9:
        chi = [alpha] + [(1 - alpha) / 5] * 4 + [(1 - alpha) / 20] * 4
    else:
        chi = [alpha] + [(1 - alpha) * wi / (1 - w[0]) for wi in w[1:]]
    W, sigma = P["W"], P["sigma"]
    rho_l, rho_g = P["rho_l"], P["rho_g"]
    nu_l, nu_g = P["mu_l"] / rho_l, P["mu_g"] / rho_g
    eps = -(4.0 / W) * math.cos(P["theta"])
    if isinstance(start, tuple):
        (ctr, R0), grid = start, [torch.arange(n, dtype=torch.float64, device=dev) for n in (nx, ny, nz)]
        d2 = torch.zeros((nz, ny, nx), dtype=torch.float64, device=dev)
        for a in range(D):
            v, n = grid[a] - ctr[a], (nx, ny, nz)[a]
            if P["periodic"] & (1 << a):
                v = v - n * torch.floor(v / n + 0.5)
            d2 += (v * v).reshape([-1 if 2 - a == k else 1 for k in range(3)])
        phi = 0.5 * (1.0 + torch.tanh(2.0 * (R0 - torch.sqrt(d2)) / W))
    else:
        phi = torch.from_numpy(np.ascontiguousarray(start)).to(dev)
    phi = torch.where(solid, torch.zeros_like(phi), phi)
    phi.view(-1)[nodes] = 0.5 * (1.0 + math.cos(P["theta"]))
    zero = torch.zeros_like(phi)
    N = [torch.full_like(phi, x) for x in chi]
    u, p = [zero.clone() for _ in range(3)], zero.clone()
    contrast = rho_l != rho_g
    from_solid = [_at(solid, tuple(-a for a in v)) for v in c]
    for _ in range(steps):
        phi_f = (phi.view(-1)[corner] * weight).sum(0)
        if P["ghost_rule"] == 0:
            phi.view(-1)[nodes] = phi_f / (phi_f + (1.0 - phi_f) * math.exp(eps))
        else:
            a = 1.0 + 0.5 * eps
            phi.view(-1)[nodes] = 4.0 * phi_f / (a + torch.sqrt(a * a - 2.0 * eps * phi_f)) - phi_f
        grad, lap = [zero.clone() for _ in range(3)], zero.clone()
        du = [[zero.clone() if contrast and a < D and b < D else None for b in range(3)] for a in range(3)]
        for i in range(1, Q):
            ph = _at(phi, c[i])
            lap += 6.0 * w[i] * (ph - phi)
            for a in range(D):
                if c[i][a]:
                    grad[a] += 3.0 * w[i] * c[i][a] * ph
                    if contrast:
                        for b in range(D):
                            du[a][b] += 3.0 * w[i] * c[i][a] * _at(u[b], c[i])
        rho = rho_l * phi + rho_g * (1.0 - phi)
        nu = 1.0 / (phi / nu_l + (1.0 - phi) / nu_g)
        tau = 0.5 + nu / cs2
        u0 = [sum((N[i] * c[i][a] for i in range(1, Q) if c[i][a]), zero) for a in range(3)]
        moving = sum((N[i] - chi[i] for i in range(1, Q)), zero)      # less the rest state: p is small

        def pressure(v):
            return (moving * cs2 - 0.5 * w[0] * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])) / (1.0 - w[0])
        mu = (48.0 / W) * phi * (1.0 - phi) * (phi - 0.5) + 1.5 * W * lap
        p0 = pressure(u0)
        F = []
        for a in range(3):
            f = -sigma * mu * grad[a] + rho * P["g"][a]
            if contrast and a < D:
                visc = sum(((du[a][b] + du[b][a]) * grad[b] for b in range(D)), zero)
                f = f + (rho_l - rho_g) * (cs2 * (tau - 0.5) * visc - p0 * grad[a])
            F.append(f if a < D else zero)
        u = [torch.where(solid, zero, u0[a] + F[a] / (2.0 * rho)) for a in range(3)]
        p = torch.where(solid, zero, pressure(u))
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        neq = []
        for i in range(Q):
            if i == 0:
                neq.append(chi[0] - (1.0 - w[0]) * p / cs2 - 1.5 * w[0] * uu)
            else:
                cu = sum((u[a] * c[i][a] for a in range(D) if c[i][a]), zero)
                neq.append(chi[i] + w[i] * (3.0 * p + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu))
        rows = []
        for v in c:
            v2 = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
            rows.append((v[0] ** 2 - v[1] ** 2, v[0] * v[1]) if D == 2 else
                        (3 * v[0] ** 2 - v2, v[1] ** 2 - v[2] ** 2, v[0] * v[1], v[1] * v[2], v[0] * v[2]))
        size = [sum(r[k] ** 2 for r in rows) for k in range(len(rows[0]))]
        stress = [sum(((N[i] - neq[i]) * rows[i][k] for i in range(Q) if rows[i][k]), zero) / size[k]
                  for k in range(len(size))]
        om = 1.0 - 1.0 / tau
        norm = torch.sqrt(grad[0] ** 2 + grad[1] ** 2 + grad[2] ** 2).clamp(min=1e-6)
        seg = (2.0 / W) * phi * (1.0 - phi) / norm
        post, blue = [], []
        for i in range(Q):
            v = neq[i] + om * sum((stress[k] * rows[i][k] for k in range(len(size)) if rows[i][k]), zero)
            if i:
                v = v + 1.5 * w[i] * sum((F[a] * c[i][a] for a in range(D) if c[i][a]), zero) / rho
            post.append(v)
            b = phi * v
            if i:
                b = b + seg * sum((grad[a] * c[i][a] for a in range(D) if c[i][a]), zero) * (chi[i] + 3.0 * w[i] * p)
            blue.append(b)
        new = zero.clone()
        for i in range(Q):
            back = tuple(-a for a in c[i])
            N[i] = torch.where(from_solid[i], post[opp[i]], _at(post[i], back))
            new += torch.where(from_solid[i], blue[opp[i]], _at(blue[i], back))
        phi = torch.where(fluid, new, phi)
    return {"phi": phi, "u": torch.stack(u), "p": p}


def exact(case, seed):
    nodes = sum(nx * ny * nz for nx, ny, nz in _sizes(case))
    if nodes * case["steps"] > 6e8 or case["steps"] * case["domains"] > 1700:     # over about 20 s
        return None
    out = []
    for params, solid, ghosts, start in _domain_inputs(case, seed):
        got = _integrate(params, solid, ghosts, start, case["steps"])
        out.append({f: got[f].reshape(3, -1) if f == "u" else got[f].reshape(-1) for f in case["fields"].split()})
    return out
