"""The work a user of the contact library has it do, as cases to be timed.

A case is a particle state (kind of shapes, number, resolution, volume
fraction), the options of the context and the way it is called:

  call  Contact.step             one checked step, results on the device
  step  Contact.step_async       the time loop's step: enqueued on the context's stream
  host  Contact.step_host        page-locked host poses in, host forces out
  grad  contact_forces + autograd   forces, torques and their adjoint

States are periodic boxes of the kinds the workloads module stands for: random
sequential addition of volume-equivalent spheres, shapes of uniform random
orientation at those centres, a share of the particles moved into touch with
their nearest neighbour.  A box of more than ~2000 particles is a periodic
block repeated `tiles` times per axis with every position jittered and every
orientation drawn anew.  `exact` evaluates the same method in 64 bits with
plain torch operations.
"""
import itertools
import math

import numpy as np
import torch

from paper_2401_10878_gb300 import workloads as W
from paper_2401_10878_gb300.contact import Contact, contact_forces

YOUNG, POISSON = 5.0e3, 0.3        # the workloads' material
RESTITUTION, MU_S, MU_K, U_K = 0.926, 0.32, 0.16, 0.001   # the paper's contact law (Sec. 5.1)
ROUGH = math.sqrt(0.75)            # rough-detection threshold of the box pipeline, cells


def _case(name, mode, kind, block, tiles=1, edge=12.0, phi=0.3, touch=0.0, smooth=0, fp64=0, box=0, law=0, walls=0,
          inflate=0.0):
    c = dict(mode=mode, kind=kind, block=block, tiles=tiles, edge=edge, phi=phi, touch=touch, smooth=smooth, fp64=fp64,
             box=box, law=law, walls=walls, inflate=inflate)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest state of the configurations: 27 spheres and cubes in 64^3, one checked call
        _case("mixed27_call", "call", "grid27", 27),
        # a dilute settling box in its time loop, with the paper's whole contact law
        # (velocities, damping from the contact history, friction)
        _case("cubes400_law", "step", "cubes", 400, phi=0.1, touch=0.15, law=1),
        # the headline state: 1934 cubes at 30 %, the time loop's step
        _case("cubes1934_step", "step", "cubes", 1934),
        # the same state called by a host program (a fluid solver on the CPU): poses and forces in host memory
        _case("cubes1934_host", "host", "cubes", 1934),
        # spheres, cubes and polytopes (12-20 faces) in the same box
        _case("mixed1934_step", "step", "mixed", 1934),
        # fitting or control through the contact: smoothed indicator, forward and adjoint
        _case("cubes1934_grad", "grad", "cubes", 1934, smooth=1),
        # the paper's own sample set (N_c = 8, dx/5 enlargement) between a floor and a ceiling, whole contact law
        _case("cubes1934_box8", "step", "cubes", 1934, box=8, law=1, walls=1, inflate=0.2),
        # the all-FP64 form, for runs that check the FP32 one
        _case("cubes1934_fp64", "step", "cubes", 1934, fp64=1),
        # the finest resolution of the sweep: 500 cubes of 24 cells at 20 %
        _case("cubes500_e24", "step", "cubes", 500, edge=24.0, phi=0.2, touch=0.15),
        # a larger suspension of spheres and cuboids with the whole contact law
        _case("sc15472_law", "step", "sc", 1934, tiles=2, law=1),
        # the adjoint of a larger mixed box (smoothed, velocities and friction)
        _case("mixed15472_grad", "grad", "mixed", 1934, tiles=2, smooth=1, law=1),
        # the largest: 52218 cubes at 30 % in 669^3
        _case("cubes52218_step", "step", "cubes", 1934, tiles=3),
    ]


def draw(rng):
    """A case of the same ranges: 27 to 52218 particles, 8 to 27 cells per edge, 10 to 30 %, every kind and option."""
    mode = rng.choice(["step", "step", "step", "call", "host", "grad"])
    kind = rng.choice(["cubes", "spheres", "sc", "mixed"])
    opt = rng.choice(["", "", "", "fp64", "box"]) if mode == "step" else ""
    most = {"fp64": 1934, "box": 1934}.get(opt, {"grad": 15472, "call": 15472, "host": 15472}.get(mode, 52218))
    n = int(round(math.exp(rng.uniform(math.log(27), math.log(most)))))
    tiles = 1
    while n > 1934 * tiles ** 3:
        tiles += 1
    block = max(27, n // tiles ** 3)
    edge = round(math.exp(rng.uniform(math.log(8.0), math.log(27.0))), 2)
    box = 0
    if opt == "fp64":     # the work grows with the nodes of the boxes
        edge = min(edge, round(12.0 * (1934.0 / block) ** (1.0 / 3.0), 2))
    elif opt == "box":    # with the samples
        box = rng.choice([4, 6, 8, 11, 16])
        block = min(block, int(1934 * (8.0 / box) ** 3))
    else:                 # with the lines
        edge = min(edge, round(max(8.0, 12.0 * math.sqrt(52218.0 / (block * tiles ** 3))), 2))
    return _case(None, mode, kind, block, tiles, edge, round(rng.uniform(0.1, 0.3), 3), rng.choice([0.0, 0.1, 0.15]),
                 smooth=1 if mode == "grad" else int(rng.random() < 0.25), fp64=int(opt == "fp64"), box=box,
                 law=int(rng.random() < 0.4), walls=int(rng.random() < 0.25),
                 inflate=rng.choice([0.0, 0.0, 0.2]))


# ---------------------------------------------------------------------------- states

def _rsa(n, d, L, gen, dev):
    """Centres of n spheres of diameter d in a periodic cube of side L, none closer than d (batches on the device)."""
    pts = torch.zeros((0, 3), dtype=torch.float64, device=dev)
    for _ in range(4000):
        c = torch.rand((2048, 3), dtype=torch.float64, device=dev, generator=gen) * L
        if len(pts):
            e = c[:, None, :] - pts[None, :, :]
            e -= L * torch.round(e / L)
            c = c[(e.square().sum(-1) >= d * d).all(1)]
        e = c[:, None, :] - c[None, :, :]
        e -= L * torch.round(e / L)
        near = torch.tril(e.square().sum(-1) < d * d, -1)   # an earlier one of the batch is too close
        pts = torch.cat([pts, c[~near.any(1)]])[:n]
        if len(pts) == n:
            return pts
    raise RuntimeError("the box does not take %d spheres" % n)


def _state(case, seed):
    """The case's particle state as plain arrays: shapes, material, poses, velocities, walls, lattice."""
    kind, edge = case["kind"], case["edge"]
    rng = np.random.default_rng(seed)
    if kind == "grid27":
        st = W.mixed_grid_27(seed=seed)
        types, params, species = st.shape_type, st.shape_param, np.zeros(st.n, np.int64)
        polys, pos, quat, ncell = [], st.pos, st.quat, int(st.n_cells[0])
    else:
        dev = torch.device("cuda")
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        block, tiles = case["block"], case["tiles"]
        d_eq = edge * (6.0 / math.pi) ** (1.0 / 3.0)
        # the shapes of a suspension: spheres of d_eq, cubes or cuboids of the edge, a dozen polytopes
        half = {"cubes": (0.5, 0.5, 0.5), "mixed": (0.5, 0.5, 0.5), "sc": (0.62, 0.5, 0.4), "spheres": (0.5,) * 3}[kind]
        rmax = edge * max(math.sqrt(sum(h * h for h in half)), 0.92) + max(1.0, case["inflate"] + ROUGH)
        side = max((block * edge ** 3 / case["phi"]) ** (1.0 / 3.0), (4.0 * rmax + 4.0) / tiles)
        ncell = int(math.ceil(side * tiles))
        side = ncell / tiles
        pts = _rsa(block, (0.95 if kind == "spheres" else 1.0) * d_eq, side, gen, dev).cpu().numpy()
        off = np.stack(np.meshgrid(*[np.arange(tiles)] * 3, indexing="ij"), -1).reshape(-1, 1, 3) * side
        pos = (pts[None] + off).reshape(-1, 3)
        n = len(pos)
        quat = rng.normal(size=(n, 4))
        quat /= np.linalg.norm(quat, axis=1, keepdims=True)
        perm = rng.permutation(n)
        pos = pos[perm] + (rng.normal(0.0, 0.05, size=(n, 3)) if tiles > 1 else 0.0)
        if case["touch"] > 0:   # a share of them moved to just under one diameter from their nearest neighbour
            m = rng.choice(n, size=int(round(case["touch"] * n)), replace=False)
            p = torch.tensor(pos, device=dev)
            pm, at = p[torch.tensor(m, device=dev)], []
            for c in pm.split(256):
                e = c[:, None, :] - p[None]
                e -= ncell * torch.round(e / ncell)
                q = e.square().sum(-1)
                q[q < 1e-9] = 1e30
                at.append(q.argmin(1))
            at = torch.cat(at).cpu().numpy()
            e = pos[m] - pos[at]
            e -= ncell * np.round(e / ncell)
            e /= np.linalg.norm(e, axis=1, keepdims=True)
            pos[m] = pos[at] + e * (0.93 * d_eq)
        species = np.zeros(n, np.int64)
        kinds = {"cubes": [1], "spheres": [0], "sc": [0, 1], "mixed": [0, 1, 2]}[kind]
        types = np.array(kinds, np.int32)[np.arange(n) % len(kinds)]
        params = np.zeros((n, 3))
        params[types == 0] = [d_eq / 2, 0.0, 0.0]
        params[types == 1] = np.array(half) * edge
        polys = []
        if 2 in kinds:
            polys = [W.random_polytope(rng, int(rng.integers(12, 21)), float(rng.uniform(8.0, 11.0)) * edge / 12.0)[0]
                     for _ in range(12)]
            species[types == 2] = rng.integers(0, len(polys), size=int((types == 2).sum()))
    L = float(ncell)
    pos = np.mod(pos, L)
    pos[pos >= L] = 0.0
    n = len(pos)
    s = dict(n=n, ncell=ncell, types=np.asarray(types, np.int32), params=np.ascontiguousarray(params, np.float64),
             species=species, polys=polys, pos=np.ascontiguousarray(pos), quat=np.ascontiguousarray(quat),
             vel=None, walls=np.zeros((0, 4)))
    if case["law"]:   # velocities of a settling suspension in lattice units: a few u_K of slip
        s["vel"] = np.concatenate([rng.normal(0.0, 2e-3, size=(n, 3)), rng.normal(0.0, 2e-4, size=(n, 3))], axis=1)
    if case["walls"]:   # a floor and a ceiling that the outermost particles press into
        z = pos[:, 2]
        s["walls"] = np.array([[0.0, 0.0, 1.0, z.min() - 0.2 * edge], [0.0, 0.0, -1.0, -(z.max() + 0.2 * edge)]])
    s["weights"] = rng.uniform(-1.0, 1.0, size=(2, n, 3))   # the loss's gradient at the forces and torques
    return s


def _max_pairs(n):
    return max(64, 16 * n)


_stream = None


def _loop_stream():
    """The one stream of the user's time loop (every context enqueues on it)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    s = _state(case, seed)
    n, nw = s["n"], len(s["walls"])
    planes = [s["polys"][k] for k, t in zip(s["species"], s["types"]) if t == 2]
    nf = np.zeros(n, np.int64)
    nf[s["types"] == 2] = [len(p) for p in planes]
    opts = {}
    if case["law"]:
        opts = dict(history=case["mode"] != "grad", restitution=RESTITUTION, friction=True, mu_s=MU_S, mu_k=MU_K, u_k=U_K)
        if case["mode"] == "grad":
            opts["damping_c"] = 0.5
    model = Contact(
        s["types"], s["params"], np.concatenate([[0], np.cumsum(nf)]).astype(np.int32),
        np.concatenate(planes) if planes else np.zeros((0, 4)), np.full(n, YOUNG), np.full(n, POISSON),
        [s["ncell"]] * 3, 1.0, indicator=case["smooth"], inflate=case["inflate"], precision=case["fp64"],
        walls=s["walls"] if nw else None, wall_young=np.full(nw, YOUNG), wall_poisson=np.full(nw, POISSON),
        box_mode=int(case["box"] > 0), contact_resolution=case["box"] or 8, max_pairs=_max_pairs(n),
        stream=_loop_stream(), **opts)
    state = dict(mode=case["mode"], model=model)
    if case["mode"] == "host":
        pin = lambda a: torch.tensor(a).pin_memory()  # noqa: E731
        state.update(pos=pin(s["pos"]), quat=pin(s["quat"]), vel=None if s["vel"] is None else pin(s["vel"]),
                     force=torch.zeros((n, 3), dtype=torch.float64).pin_memory(),
                     torque=torch.zeros((n, 3), dtype=torch.float64).pin_memory())
        return state
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    state.update(pos=dev(s["pos"]), quat=dev(s["quat"]), vel=None if s["vel"] is None else dev(s["vel"]))
    if case["mode"] == "grad":
        state["pos"].requires_grad_(True)
        state["quat"].requires_grad_(True)
        state.update(wf=dev(s["weights"][0]), wt=dev(s["weights"][1]))
    torch.cuda.synchronize()
    return state


def run(state):
    model, pos, quat, vel = state["model"], state["pos"], state["quat"], state["vel"]
    mode = state["mode"]
    if mode in ("step", "call"):   # outputs in the context's buffers (pair rows past n_pairs stay zero)
        if mode == "step":
            model.step_async(pos, quat, vel)
            n_pairs = model.n_pairs
        else:
            n_pairs = model.step(pos, quat, vel)["n_pairs"]
        return dict(force=model.force, torque=model.torque, n_pairs=n_pairs, pair_ij=model.pair_ij,
                    pair_out=model.pair_out)
    if mode == "host":
        return model.step_host(pos, quat, vel, force=state["force"], torque=state["torque"])
    force, torque = contact_forces(model, pos, quat, vel)
    gpos, gquat = torch.autograd.grad((force, torque), (pos, quat), (state["wf"], state["wt"]))
    return dict(force=force.detach(), torque=torque.detach(), grad_pos=gpos, grad_quat=gquat)


def work(case):
    """Poses (and velocities) in, forces, torques and the pairs' results out; the FP32 operations of the nodes that
    add to the sums (estimates per particle from the settling boxes: 3.4 candidate pairs at 30 %, ~14 nodes at 12
    cells per edge) and in the box pipeline of its samples."""
    n = case["block"] * case["tiles"] ** 3
    dense = case["phi"] / 0.3
    pairs = {"cubes": 3.4, "spheres": 2.0, "sc": 2.6, "mixed": 1.7, "grid27": 2.5}[case["kind"]] * dense * n
    nodes = 14.0 * (case["edge"] / 12.0) ** 2 * dense * n
    bytes_ = (7 + 6 + (6 if case["law"] else 0)) * 8.0 * n
    if case["mode"] in ("step", "call"):
        bytes_ += 96.0 * pairs
    ops = {"cubes": 30.0, "spheres": 14.0, "sc": 22.0, "mixed": 60.0, "grid27": 22.0}[case["kind"]]
    flops = 2.0 * ops * nodes
    if case["box"]:
        flops += 2.0 * ops * 0.25 * pairs * case["box"] ** 3
    if case["mode"] == "grad":
        bytes_ += (7 + 6) * 8.0 * n
        flops += 2.0 * 150.0 * nodes
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------------------- the method in 64 bits

def _offset_box_vertices(planes, delta):
    """Vertices of {y : n . y <= d + delta} (numpy): plane triples, kept when inside every half-space."""
    t = np.array(list(itertools.combinations(range(len(planes)), 3)))
    A, b = planes[t][:, :, :3], planes[t][:, :, 3] + delta
    ok = np.abs(np.linalg.det(A)) > 1e-12
    v = np.linalg.solve(A[ok], b[ok][..., None])[..., 0]
    inside = (v @ planes[:, :3].T <= planes[:, 3] + delta + 1e-9 * max(1.0, np.abs(planes[:, 3] + delta).max())).all(1)
    return v[inside]


class _Exact:
    """One state in 64 bits: faces of every species (a cuboid's six, a polytope's own; spheres have none)."""

    def __init__(self, case, s):
        self.case, self.s, self.n, self.L = case, s, s["n"], float(s["ncell"])
        dev = self.dev = torch.device("cuda")
        f8 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        box = next((p for p, t in zip(s["params"], s["types"]) if t == 1), np.ones(3))
        cub = np.array([[sg * (k == a) for k in range(3)] + [box[a]] for a in range(3) for sg in (1.0, -1.0)])
        shapes = [cub] + list(s["polys"])
        F = max(len(p) for p in shapes)
        tab = np.zeros((len(shapes) + len(s["walls"]), F, 4))
        tab[:, :, 3] = 1e30
        for k, p in enumerate(shapes):
            tab[k, :len(p)] = p
        for w, m in enumerate(s["walls"]):   # a wall: one face in the world frame, at the origin
            tab[len(shapes) + w, 0] = m
        self.inflate, self.w = float(case["inflate"]), 1.0
        band = 0.5 if case["smooth"] else 0.0
        if case["box"]:
            band = max(band, ROUGH)
        self.delta = self.inflate + band
        nw = len(s["walls"])
        self.tab = f8(tab)
        sp = np.where(s["types"] == 2, s["species"] + 1, 0)
        self.species = torch.tensor(np.concatenate([sp, len(shapes) + np.arange(nw)]), device=dev)
        self.sphere = torch.tensor(np.concatenate([s["types"] == 0, np.zeros(nw, bool)]), device=dev)
        self.any_sphere = bool((s["types"] == 0).any())
        self.rad = f8(np.concatenate([s["params"][:, 0], np.zeros(nw)]))
        self.pos, self.quat = f8(s["pos"]), f8(s["quat"])
        self.vel = None if s["vel"] is None else torch.cat([f8(s["vel"]), f8(np.zeros((nw, 6)))])
        # node ranges: extents of the widened shapes
        R = self.rot(self.quat)
        ext_hi = torch.zeros((self.n, 3), dtype=torch.float64, device=dev)
        t = torch.tensor(s["types"], device=dev)
        prm = f8(s["params"])
        ext_hi[t == 0] = (prm[t == 0, :1] + self.delta).expand(-1, 3)
        ext_hi[t == 1] = (R[t == 1].abs() @ (prm[t == 1] + self.delta)[..., None])[..., 0]
        ext_lo = -ext_hi
        rmax = 0.0
        for k, p in enumerate(s["polys"]):
            sel = (t == 2) & (self.species[:self.n] == k + 1)
            v = f8(_offset_box_vertices(p, self.delta))
            e = R[sel] @ v.T
            ext_hi[sel], ext_lo[sel] = e.amax(-1), e.amin(-1)
        rmax = float(ext_hi.abs().max()) * math.sqrt(3.0)
        self.lo, self.hi = torch.ceil(self.pos + ext_lo), torch.floor(self.pos + ext_hi)
        # candidate pairs, sorted by (i, j): node ranges that share a node, the partner in its nearest image
        ii, jj = [], []
        for rows in torch.arange(self.n, device=dev).split(max(1, 40_000_000 // self.n)):
            d = self.pos[None, :, :] - self.pos[rows][:, None, :]
            d -= self.L * torch.round(d / self.L)
            near = (d.abs().amax(-1) <= 2 * rmax + 2) & (torch.arange(self.n, device=dev)[None] > rows[:, None])
            a, b = near.nonzero(as_tuple=True)
            ii.append(rows[a])
            jj.append(b)
        i, j = torch.cat(ii), torch.cat(jj)
        shift = torch.round((self.pos[j] - self.pos[i]) / self.L)
        lo = torch.maximum(self.lo[i], self.lo[j] - shift * self.L)
        hi = torch.minimum(self.hi[i], self.hi[j] - shift * self.L)
        ok = (lo <= hi).all(1)
        i, j, shift, lo, hi = i[ok], j[ok], shift[ok], lo[ok], hi[ok]
        for w, m in enumerate(s["walls"]):   # along z: clipped to the nodes below h + delta
            up = m[2] > 0
            b = (m[3] + self.delta) / m[2]
            wlo, whi = self.lo.clone(), self.hi.clone()
            if up:
                whi[:, 2] = torch.clamp(whi[:, 2], max=math.floor(b))
            else:
                wlo[:, 2] = torch.clamp(wlo[:, 2], min=math.ceil(b))
            p = (wlo <= whi).all(1).nonzero()[:, 0]
            i, j = torch.cat([i, p]), torch.cat([j, torch.full_like(p, self.n + w)])
            shift = torch.cat([shift, torch.zeros((len(p), 3), dtype=torch.float64, device=dev)])
            lo, hi = torch.cat([lo, wlo[p]]), torch.cat([hi, whi[p]])
        order = torch.argsort(i * (self.n + nw + 1) + j)
        self.i, self.j, self.shift, self.plo, self.phi_ = i[order], j[order], shift[order], lo[order], hi[order]

    @staticmethod
    def rot(q):
        w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        return torch.stack([
            torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], 1),
            torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], 1),
            torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)], 1)

    def frames(self, pos, quat):
        """Positions and rotations of the particles and the walls (at the origin)."""
        nw = len(self.s["walls"])
        eye = torch.eye(3, dtype=torch.float64, device=self.dev).expand(nw, 3, 3)
        return (torch.cat([pos, torch.zeros((nw, 3), dtype=torch.float64, device=self.dev)]),
                torch.cat([self.rot(quat), eye]))

    def face(self, pid, y):
        """Index of the largest face value of each point (body frame), and the value."""
        best = torch.full((len(pid),), -1e300, dtype=torch.float64, device=self.dev)
        at = torch.zeros(len(pid), dtype=torch.int64, device=self.dev)
        sp = self.species[pid]
        for f in range(self.tab.shape[1]):
            e = self.tab[sp, f]
            v = (e[:, :3] * y).sum(1) - e[:, 3]
            up = v > best
            best = torch.where(up, v, best)
            at = torch.where(up, torch.full_like(at, f), at)
        return at, best

    def sdf(self, pid, r, R, grad):
        """Signed distance at r = x - X (reduced by inflate), its gradient if asked for."""
        y = (R.transpose(1, 2) @ r[..., None])[..., 0]
        with torch.no_grad():
            at, _ = self.face(pid, y.detach())
        e = self.tab[self.species[pid], at]
        v = (e[:, :3] * y).sum(1) - e[:, 3]
        g = (R @ e[:, :3, None])[..., 0] if grad else None
        if self.any_sphere:
            sph = self.sphere[pid]
            nr = torch.where(sph[:, None], r, torch.ones_like(r)).norm(dim=1)
            v = torch.where(sph, nr - self.rad[pid], v)
            if grad:
                g = torch.where(sph[:, None], r / nr[:, None], g)
        return v - self.inflate, g

    def nodes(self, X, R, limit):
        """(pair, node, index in the pair box) of the box nodes with both distances below limit."""
        dim = (self.phi_ - self.plo + 1).to(torch.int64)
        vol = dim.prod(1)
        out = []
        start = torch.cumsum(vol, 0)
        p0, P = 0, len(vol)
        cum = start.cpu().numpy()
        while p0 < P:
            base = cum[p0 - 1] if p0 else 0
            p1 = max(p0 + 1, int(np.searchsorted(cum, base + 3_000_000, side="right")))
            v = vol[p0:p1]
            q = torch.repeat_interleave(torch.arange(p0, p1, device=self.dev), v)
            k = torch.arange(len(q), device=self.dev) - torch.repeat_interleave(start[p0:p1] - v - int(base), v)
            d = dim[q]
            c = torch.stack([k % d[:, 0], (k // d[:, 0]) % d[:, 1], k // (d[:, 0] * d[:, 1])], 1).to(torch.float64)
            x = self.plo[q] + c
            a = self.i[q]
            fa, _ = self.sdf(a, x - X[a], R[a], False)
            keep = fa < limit
            q, k, x = q[keep], k[keep], x[keep]
            b = self.j[q]
            fb, _ = self.sdf(b, x - (X[b] - self.shift[q] * self.L), R[b], False)
            keep = fb < limit
            out.append((q[keep], k[keep], x[keep]))
            p0 = p1
        return [torch.cat(t) for t in zip(*out)] if out else None

    def deepest(self, P, q, depth, ok):
        """Row of each pair's deepest point (-1: none), the first of equals."""
        best = torch.full((P,), -1e300, dtype=torch.float64, device=self.dev)
        best.scatter_reduce_(0, q[ok], depth[ok], "amax")
        row = torch.full((P,), len(q), dtype=torch.int64, device=self.dev)
        hit = ok & (depth == best[q])
        row.scatter_reduce_(0, q[hit], hit.nonzero()[:, 0], "amin")
        return torch.where(row < len(q), row, torch.full_like(row, -1))

    def sums(self, q, P, x, X, R, weight, origin):
        """Per pair: volume, contact point, band vector G, depth and whether it overlaps, from points x (world)
        of pairs q that each weigh `weight` [P]."""
        a, b = self.i[q], self.j[q]
        fa, ga = self.sdf(a, x - X[a], R[a], True)
        fb, gb = self.sdf(b, x - (X[b] - self.shift[q] * self.L), R[b], True)
        ta, tb = (0.5 - fa / self.w).clamp(0.0, 1.0), (0.5 - fb / self.w).clamp(0.0, 1.0)
        if self.case["smooth"]:
            ha, hb = ta * ta * (3 - 2 * ta), tb * tb * (3 - 2 * tb)
        else:
            ha, hb = (fa <= 0).to(torch.float64), (fb <= 0).to(torch.float64)
        h = ha * hb
        zero = torch.zeros(P, dtype=torch.float64, device=self.dev)
        z3 = torch.zeros((P, 3), dtype=torch.float64, device=self.dev)
        S0 = zero.index_add(0, q, h)
        S1 = z3.index_add(0, q, h[:, None] * (x - origin[q]))
        Sg = z3.index_add(0, q, (ta * (1 - ta) * hb)[:, None] * ga - (ha * tb * (1 - tb))[:, None] * gb)
        V = weight * S0
        has = S0.detach() > 0
        xc = origin + S1 / torch.where(has, S0, torch.ones_like(S0))[:, None]
        G = (0.5 * weight * 6.0 / self.w)[:, None] * Sg
        row = self.deepest(P, q, -(fa + fb).detach(), (h > 0).detach())
        depth = torch.where(row >= 0, (-(fa + fb))[row.clamp(min=0)], zero)
        return V, xc, G, depth.clamp(min=0.0), has

    def law(self, V, xc, G, d, has, X, grad):
        """Pair outputs [P, 11] and particle forces and torques [N, 3] of the overlapping pairs."""
        P, o = len(V), has.nonzero()[:, 0]
        i, j = self.i[o], self.j[o]
        V, xc, G, d = V[o], xc[o], G[o], d[o]
        XA, XB = X[i], X[j] - self.shift[o] * self.L
        gn = G.norm(dim=1)
        line = XB - XA
        wall = j >= self.n
        fall = line / line.norm(dim=1, keepdim=True).clamp(min=1e-300)
        if wall.any():
            m = self.tab[self.species[j], 0][:, :3]
            fall = torch.where(wall[:, None], -m, fall)
        n = torch.where((gn > 1e-12)[:, None], G / gn.clamp(min=1e-300)[:, None], fall)
        estar = 1.0 / (2.0 * (1.0 - POISSON ** 2) / YOUNG)
        rA, rB = xc - XA, xc - XB
        damp, ut = torch.ones_like(V), None
        if self.vel is not None:
            va, vb = self.vel[i], self.vel[j]
            u = (va[:, :3] + torch.cross(va[:, 3:], rA, dim=1)) - (vb[:, :3] + torch.cross(vb[:, 3:], rB, dim=1))
            dd = (u * n).sum(1)
            if grad:
                c = torch.full_like(dd, 0.5)
            else:   # a contact's first step: c = K / u0 for an approach, else 0
                K = 1.5 * (1.0 - RESTITUTION) * (11.0 - RESTITUTION) / (1.0 + 9.0 * RESTITUTION)
                c = torch.where(dd > 0, K / torch.where(dd > 0, dd, torch.ones_like(dd)), torch.zeros_like(dd))
            damp = (1.0 + c * dd).clamp(min=0.0)
            ut = u - dd[:, None] * n
        vd = V * d
        fmag = 4.0 / (3.0 * math.pi) * estar * torch.sqrt(vd.clamp(min=1e-300)) * damp * (vd.detach() > 0)
        F = fmag[:, None] * n
        if ut is not None:
            mus = MU_S * (1.0 - 0.09 * (MU_K / MU_S) ** 4)
            un = ut.norm(dim=1)
            a2 = (un / U_K) ** 2
            f = (2 * mus - MU_K) * a2 / (a2 * a2 + 1) + MU_K * a2 / (a2 + 1)
            F = F + (f * fmag / un.clamp(min=1e-300))[:, None] * ut
        TA, TB = -torch.cross(rA, F, dim=1), torch.cross(rB, F, dim=1)
        rows = len(self.species)
        z = torch.zeros((rows, 3), dtype=torch.float64, device=self.dev)
        force = z.index_add(0, j, F).index_add(0, i, -F)[:self.n]
        torque = z.index_add(0, j, TB).index_add(0, i, TA)[:self.n]
        out = torch.zeros((P, 11), dtype=torch.float64, device=self.dev)
        out[o] = torch.cat([V[:, None], xc, n, d[:, None], F], 1).detach()
        return out, force, torque

    def clip(self, pid, p, X, R, k, sgn):
        """Interval [t0, t1] of the lines p + t sgn e_k inside the particles (or walls) pid."""
        t0 = torch.full((len(pid),), -1e30, dtype=torch.float64, device=self.dev)
        t1 = -t0
        r, sp = p - X, self.species[pid]
        for f in range(self.tab.shape[1]):
            e = self.tab[sp, f]
            nrm = (R @ e[:, :3, None])[..., 0]
            a = (nrm * r).sum(1) - e[:, 3] - self.inflate
            b = sgn * nrm[:, k]
            t = -a / torch.where(b == 0, torch.ones_like(b), b)
            t1 = torch.where(b > 0, torch.minimum(t1, t), t1)
            t0 = torch.where(b < 0, torch.maximum(t0, t), t0)
            t0 = torch.where((b == 0) & (a > 0), torch.full_like(t0, 1e30), t0)
        if self.any_sphere:
            b = sgn * r[:, k]
            disc = b * b - r.square().sum(1) + (self.rad[pid] + self.inflate) ** 2
            sq = disc.clamp(min=0).sqrt()
            sph = self.sphere[pid]
            t0 = torch.where(sph, torch.where(disc < 0, torch.full_like(b, 1e30), -b - sq), t0)
            t1 = torch.where(sph, torch.where(disc < 0, torch.full_like(b, -1e30), -b + sq), t1)
        return t0, t1

    def box_points(self, X, R):
        """The box pipeline: pairs with a rough contact, their corrected boxes (lo, hi)."""
        q, _, x = self.nodes(X, R, ROUGH)
        P = len(self.i)
        lo = torch.full((P, 3), 1e30, dtype=torch.float64, device=self.dev)
        hi = -lo
        at = q[:, None].expand(-1, 3)
        lo.scatter_reduce_(0, at, x, "amin")
        hi.scatter_reduce_(0, at, x, "amax")
        o = (lo[:, 0] <= hi[:, 0]).nonzero()[:, 0]
        lo, hi = lo[o] - ROUGH, hi[o] + ROUGH
        nc = self.case["box"]
        g = (torch.arange(nc, dtype=torch.float64, device=self.dev) + 0.5) / nc
        cut = []
        ids = torch.repeat_interleave(torch.arange(len(o), device=self.dev), nc * nc)
        A, B = self.i[o][ids], self.j[o][ids]
        XB = X[B] - self.shift[o][ids] * self.L
        for f in range(6):
            k, side = f // 2, f % 2
            u, v = [c for c in range(3) if c != k]
            p = torch.empty((len(o), nc * nc, 3), dtype=torch.float64, device=self.dev)
            p[:, :, k] = (lo if side == 0 else hi)[:, k:k + 1]
            p[:, :, u] = lo[:, u:u + 1] + g.repeat_interleave(nc)[None] * (hi - lo)[:, u:u + 1]
            p[:, :, v] = lo[:, v:v + 1] + g.repeat(nc)[None] * (hi - lo)[:, v:v + 1]
            p = p.reshape(-1, 3)
            sgn = 1.0 if side == 0 else -1.0
            a0, a1 = self.clip(A, p, X[A], R[A], k, sgn)
            b0, b1 = self.clip(B, p, XB, R[B], k, sgn)
            tin = torch.maximum(a0, b0).clamp(min=0)
            tout = torch.minimum(torch.minimum(a1, b1), (hi - lo)[:, k][ids])
            t = torch.where(tin <= tout, tin, torch.full_like(tin, 1e30)).reshape(len(o), -1).amin(1)
            cut.append(torch.where(t < 1e29, t, torch.zeros_like(t)))
        nlo, nhi = lo + torch.stack(cut[0::2], 1), hi - torch.stack(cut[1::2], 1)
        bad = ~(nlo <= nhi)
        return o, torch.where(bad, lo, nlo), torch.where(bad, hi, nhi)


def exact(case, seed):
    n_all = case["block"] * case["tiles"] ** 3
    if n_all * case["edge"] ** 3 > 1.2e8 or (case["kind"] == "mixed" and n_all * case["edge"] ** 3 > 3e7):
        return None   # takes too long
    s = _state(case, seed)
    grad = case["mode"] == "grad"
    E = _Exact(case, s)
    pos, quat = E.pos.clone().requires_grad_(grad), E.quat.clone().requires_grad_(grad)
    P = len(E.i)
    with torch.no_grad():
        X, R = E.frames(E.pos, E.quat)
    if case["box"]:
        with torch.no_grad():
            o, lo, hi = E.box_points(X, R)
            nc = case["box"]
            V, xc = torch.zeros(P, dtype=torch.float64, device=E.dev), torch.zeros((P, 3), dtype=torch.float64, device=E.dev)
            G, d, has = torch.zeros_like(xc), torch.zeros_like(V), torch.zeros(P, dtype=torch.bool, device=E.dev)
            g = (torch.arange(nc, dtype=torch.float64, device=E.dev) + 0.5) / nc
            pts = torch.stack([g.repeat(nc * nc), g.repeat_interleave(nc).repeat(nc), g.repeat_interleave(nc * nc)], 1)
            size = max(1, 2_000_000 // nc ** 3)
            for c0 in range(0, len(o), size):
                sl = slice(c0, c0 + size)
                x = (lo[sl][:, None] + pts[None] * (hi - lo)[sl][:, None]).reshape(-1, 3)
                q = torch.repeat_interleave(o[sl], nc ** 3)
                w, org = torch.zeros_like(V), torch.zeros_like(xc)
                w[o[sl]], org[o[sl]] = ((hi - lo)[sl] / nc).prod(1), lo[sl]
                r = E.sums(q, P, x, X, R, w, org)
                m = o[sl]
                V[m], xc[m], G[m], d[m], has[m] = (t[m] for t in r)
            out, force, torque = E.law(V, xc, G, d, has, X, False)
    else:
        with torch.no_grad():
            got = E.nodes(X, R, 0.5)
        q, _, x = got
        Xg, Rg = E.frames(pos, quat)
        one = torch.ones(P, dtype=torch.float64, device=E.dev)
        V, xc, G, d, has = E.sums(q, P, x, Xg, Rg, one, E.plo)
        out, force, torque = E.law(V, xc, G, d, has, Xg, grad)
    if grad:
        gp, gq = torch.autograd.grad((force, torque), (pos, quat),
                                     [torch.tensor(w, device=E.dev) for w in s["weights"]])
        return dict(force=force.detach(), torque=torque.detach(), grad_pos=gp, grad_quat=gq)
    if case["mode"] == "host":
        return dict(force=force.cpu(), torque=torque.cpu(), n_pairs=P)
    ij = torch.stack([E.i, E.j], 1).to(torch.int32)
    full_ij = torch.zeros((_max_pairs(E.n), 2), dtype=torch.int32, device=E.dev)
    full = torch.zeros((_max_pairs(E.n), 11), dtype=torch.float64, device=E.dev)
    full_ij[:P], full[:P] = ij, out
    return dict(force=force, torque=torque, pair_ij=full_ij, pair_out=full,
                n_pairs=P if case["mode"] == "call" else torch.tensor([P], dtype=torch.int32, device=E.dev))
