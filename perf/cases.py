"""Workloads of the coupled lattice-Boltzmann / immersed-boundary step, for
timing and for comparing results.

A case is one simulation as a user's program sets it up (a seeded suspension
in a box between moving plates, a channel, a pipe, a closed chamber under a
moving lid or a wall-free box with the Lees-Edwards boundary) and one pass
over it: a number of coupled steps followed by a read-out of every field,
with `grad` a recorded run with its deformation loss and the reverse sweep
before the read-out.  Consecutive passes continue the simulation, as a
program that steps and reads out does.

Cells start deformed (a volume-preserving stretch per cell), as cells in flow
are; from the rest shape the membrane forces of the first steps would be
rounding noise.

Fields of a case: geom (box, channel, pipe, chamber, lees), nx, ny, nz, cells (red
cells of 642 vertices), platelets (162 vertices), precision (f64, f32, f16,
bf16), steps (per pass), every (membrane forces every that many steps),
integrator (euler, ab2), visc (internal viscosity ratio, 1 = off), grad.
"""
import math

import numpy as np
import torch

from paper_2305_02752_gb300 import hemo, inputs

UMAX = 0.02        # centreline velocity of the driven flows
WALL_SPEED = 0.01  # plates of the shear box
LE_SPEED = 0.02    # Lees-Edwards image velocity
LID_SPEED = 0.02   # lid of the closed chamber
RED_CELL_VOLUME = 744.0  # lattice units (93 um^3 at dx = 0.5 um)


def _case(name, geom, nx, ny, nz, cells, precision, steps, platelets=0, every=1, integrator='euler', visc=1.0,
          grad=False):
    c = dict(geom=geom, nx=nx, ny=ny, nz=nz, cells=cells, platelets=platelets, precision=precision, steps=steps,
             every=every, integrator=integrator, visc=visc, grad=grad)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a single cell between plates in double precision: validation runs,
        # where launches and single-CTA latency count
        _case('box32_f64', 'box', 32, 32, 32, 1, 'f64', 4),
        # the smallest single-precision call: one step and a read-out of four
        # cells, as an interactive or control loop makes it
        _case('box48_f32', 'box', 48, 48, 48, 4, 'f32', 1),
        # wall-free shear of a few cells, the boundary used for rheology
        _case('lees48_f32', 'lees', 48, 48, 48, 6, 'f32', 10),
        # a channel with an odd wall distance in double precision: reference
        # solutions of a suspension
        _case('channel_f64', 'channel', 48, 39, 64, 30, 'f64', 2),
        # the suspension channel, single precision, default options
        _case('channel_f32', 'channel', 64, 64, 256, 440, 'f32', 10),
        # a ragged closed chamber under a moving lid, no axis periodic, with the
        # time scales separated: forces every fourth step, Adams-Bashforth
        _case('chamber_ab2_f32', 'chamber', 101, 83, 119, 240, 'f32', 8, every=4, integrator='ab2'),
        # the channel with a cytosol five times as viscous as the plasma
        _case('channel_visc_f32', 'channel', 64, 64, 256, 440, 'f32', 10, visc=5.0),
        # a vessel of red cells and platelets with 16-bit populations
        _case('vessel_bf16', 'channel', 128, 128, 512, 4460, 'bf16', 10, platelets=446),
        # the largest run: a 100 um pipe at 45 % haematocrit, single precision
        # and with 16-bit populations
        _case('pipe_f32', 'pipe', 1000, 208, 208, 19600, 'f32', 5),
        _case('pipe_f16', 'pipe', 1000, 208, 208, 19600, 'f16', 5),
        # parameter gradients of a deformation loss, both precisions
        _case('grad48_f32', 'box', 48, 48, 48, 4, 'f32', 40, grad=True),
        _case('grad32_f64', 'box', 32, 32, 32, 1, 'f64', 8, grad=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _eight(n):
    return max(8, 8 * int(round(n / 8.0)))


def draw(rng):
    """Periodic axes are whole blocks of eight nodes, as every configuration
    of this package has them; axes between walls are not."""
    geom = rng.choice(['box', 'channel', 'channel', 'channel', 'pipe', 'chamber', 'lees', 'grad'])
    ht = rng.uniform(0.08, 0.42)
    if geom in ('box', 'lees', 'grad'):
        n = _eight(rng.randint(28, 64 if geom != 'grad' else 48))
        nz = n if geom == 'lees' else rng.randint(27, n + 9)
        most = max(1, int(0.3 * n * n * nz / RED_CELL_VOLUME))
        cells = min(_log_int(rng, 1, 12), most)
        if geom == 'grad':
            return _case(None, 'box', n, n, nz, min(cells, 6), rng.choice(['f32', 'f32', 'f64']), 2 * rng.randint(4, 16),
                         grad=True)
        return _case(None, geom, n, _eight(rng.randint(28, n)), nz, cells, rng.choice(['f32', 'f32', 'f64']),
                     rng.randint(1, 8))
    if geom == 'pipe':
        d = _log_int(rng, 48, 208)
        nx = _eight(_log_int(rng, 96, 1000))
        cells = max(1, int(ht * nx * math.pi * (d / 2.0 - 6.0) ** 2 / RED_CELL_VOLUME))
        return _case(None, 'pipe', nx, d, d, cells, rng.choice(['f32', 'f16', 'bf16']), rng.randint(2, 5))
    prec = rng.choice(['f32', 'f32', 'f32', 'f16', 'bf16', 'f64'])
    big = 512 if prec != 'f64' else 96
    nx, ny, nz = _log_int(rng, 30, min(big, 160)), _log_int(rng, 30, min(big, 128)), _log_int(rng, 40, big)
    if geom == 'channel':
        nx, nz = _eight(nx), _eight(nz)
    cells = max(1, int(ht * nx * (ny - 4) * nz / RED_CELL_VOLUME))
    every, integ = rng.choice([(1, 'euler'), (1, 'euler'), (2, 'euler'), (4, 'ab2')])
    return _case(None, geom, nx, ny, nz, cells, prec, rng.randint(2, 8), platelets=rng.choice([0, 0, cells // 10]),
                 every=every, integrator=integ, visc=rng.choice([1.0, 1.0, 5.0]))


def _sites(rng, lo, hi, count, inside=None):
    """`count` centres on a jittered grid over the box, at even density
    (membranes of neighbours may intersect, as in the pipe's dense packing)."""
    lo, hi = np.asarray(lo, float), np.asarray(hi, float)
    span = np.maximum(hi - lo, 1e-3)
    h = (np.prod(np.maximum(span, 4.0)) / max(count, 1)) ** (1.0 / 3.0)
    for _ in range(60):
        n = np.maximum(1, np.floor(span / h)).astype(int)
        g = np.stack(np.meshgrid(*[np.arange(k) + 0.5 for k in n], indexing='ij'), -1).reshape(-1, 3)
        p = lo + g * (span / n)
        if inside is not None:
            p = p[inside(p)]
        if len(p) >= count:
            break
        h *= 0.97
    p = p[np.sort(rng.permutation(len(p))[:count])] if len(p) >= count else lo + rng.random((count, 3)) * span
    jit = p + (rng.random(p.shape) - 0.5) * 0.25 * h
    return np.clip(jit, lo, hi)


def _placements(rng, count):
    """Random rotations times a volume-preserving stretch of -10 to +12 %."""
    q = rng.normal(size=(count, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    rot = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                    2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                    2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).reshape(-1, 3, 3)
    s = rng.uniform(0.90, 1.12, size=count)
    axis = rng.integers(0, 2, size=count)  # along a diameter of the disc
    diag = np.repeat((1.0 / np.sqrt(s))[:, None], 3, axis=1)
    diag[np.arange(count), axis] = s
    return rot * diag[:, None, :]


def _config(case, seed):
    """The simulation's inputs as an inputs.Config."""
    rng = np.random.default_rng([int(seed), 77])
    nx, ny, nz, geom = case['nx'], case['ny'], case['nz'], case['geom']
    kbt = inputs.kbt_lattice(1.0)
    v, t = inputs.rbc_mesh()
    spec = (kbt, inputs.LINK_PERSISTENCE_UM / inputs.DX_UM, inputs.LINK_MAX_STRAIN)
    meshes = [inputs.MeshType('rbc', v, t, 15.0, 80.0, 5.0, 20.0, *spec)]
    kinds = [0] * case['cells']
    if case['platelets']:
        pv, pt = inputs.platelet_mesh()
        meshes.append(inputs.MeshType('platelet', pv, pt, 150.0, 800.0, 5.0, 20.0, *spec))
        kinds += [1] * case['platelets']
    mask, u0, wv, g = None, None, np.zeros((2, 3)), np.zeros(3)
    reach = 10.0  # a stretched cell's largest half-extent and the stencil's first node
    if geom == 'box':
        periodic = (1, 1, 0)
        mask = inputs.plate_mask(nx, ny, nz, axis=2, lo_id=inputs.WALL_A, hi_id=inputs.WALL_B)
        wv = np.array([[-WALL_SPEED, 0, 0], [WALL_SPEED, 0, 0]], float)
        lo, hi, keep = (0, 0, reach), (nx, ny, nz - 1 - reach), None
    elif geom == 'channel':
        periodic = (1, 0, 1)
        mask = inputs.plate_mask(nx, ny, nz, axis=1)
        g[0] = 8.0 / 6.0 * UMAX / (ny - 2.0) ** 2
        u0 = inputs.channel_profile(nx, ny, nz, 1, 0.5, ny - 1.5, UMAX)
        lo, hi, keep = (0, reach, 0), (nx, ny - 1 - reach, nz), None
    elif geom == 'pipe':
        periodic = (1, 0, 0)
        cy, cz, r = (ny - 1) / 2.0, (nz - 1) / 2.0, ny / 2.0 - 4.0
        mask = inputs.cylinder_mask(nx, ny, nz, r, cy, cz)
        g[0] = 4.0 / 6.0 * UMAX / r ** 2
        u0 = inputs.pipe_profile(nx, ny, nz, r, cy, cz, UMAX)
        rc = r - 8.0
        lo, hi = (0, cy - rc, cz - rc), (nx, cy + rc, cz + rc)

        def keep(p):
            return (p[:, 1] - cy) ** 2 + (p[:, 2] - cz) ** 2 <= rc * rc
    elif geom == 'chamber':
        periodic = (0, 0, 0)
        mask = np.zeros((nz, ny, nx), np.uint8)
        mask[nz - 1] = inputs.WALL_B
        wv = np.array([[0, 0, 0], [LID_SPEED, 0, 0]], float)
        lo, hi, keep = (reach,) * 3, (nx - 1 - reach, ny - 1 - reach, nz - 1 - reach), None
    else:
        periodic = (1, 1, 1)
        lo, hi, keep = (0, 0, 0), (nx, ny, nz), None
    centers = _sites(rng, lo, hi, len(kinds), keep)
    order = rng.permutation(len(kinds))
    return inputs.Config(geom, nx, ny, nz, 1.0, periodic, mask, wv, g, u0, meshes, np.array(kinds, np.int64),
                         centers[order], _placements(rng, len(kinds)), case['steps'], int(seed))


def prepare(case, seed):
    cfg = _config(case, seed)
    sim = hemo.Simulation.from_config(cfg, case['precision'])
    if case['geom'] == 'lees':
        sim.set_lees_edwards(LE_SPEED)
    if case['every'] != 1 or case['integrator'] != 'euler':
        sim.set_time_scales(case['every'], case['integrator'])
    if case['visc'] != 1.0:
        sim.set_viscosity_ratio(case['visc'])
    real = torch.float64 if case['precision'] == 'f64' else torch.float32
    shape = (cfg.nz, cfg.ny, cfg.nx)
    out = {'rho': torch.zeros(shape, dtype=real, device='cuda'),
           'u': torch.zeros(shape + (3,), dtype=real, device='cuda'),
           'X': torch.zeros((cfg.n_vertices, 3), dtype=torch.float64, device='cuda'),
           'Fv': torch.zeros((cfg.n_vertices, 3), dtype=torch.float64, device='cuda'),
           'cellstats': torch.zeros((len(cfg.centers), 6), dtype=torch.float64, device='cuda')}
    return {'sim': sim, 'case': case, 'out': out}


def run(state):
    sim, case = state['sim'], state['case']
    res = {}
    if case['grad']:
        sim.record(case['steps'])
        sim.step(case['steps'])
        loss, dX = sim.deformation_loss()
        res = {'loss': np.array([loss]), 'dX': dX, 'grad': sim.backward(dX)}
    else:
        sim.step(case['steps'])
    out = sim.get_fields(out=state['out'])
    if case['precision'] == 'f64':
        return {**res, **{k: out[k] for k in ('rho', 'u', 'X', 'Fv', 'cellstats')}}
    # values in the precision they were computed in
    res = {k: a.astype(np.float32) for k, a in res.items()}
    return {**res, 'rho': out['rho'], 'u': out['u'], 'X': out['X'].float(), 'Fv': out['Fv'].float(),
            'cellstats': out['cellstats'].float()}


def work(case):
    """Per step the populations of the fluid nodes in and out, the vertices'
    positions in and out; once per pass the fields that are read out.  Flops:
    collision and velocity per node, 64-node stencils twice and the membrane
    terms per vertex.  The reverse sweep: the forward steps again, and per
    step the adjoint populations in and out with about three times the
    arithmetic."""
    nx, ny, nz = case['nx'], case['ny'], case['nz']
    N = nx * ny * nz
    fluid = {'box': nx * ny * (nz - 2), 'channel': nx * (ny - 2) * nz, 'lees': N, 'chamber': nx * ny * (nz - 1),
             'pipe': int(nx * math.pi * (ny / 2.0 - 4.0) ** 2)}[case['geom']]
    nv = 642 * case['cells'] + 162 * case['platelets']
    pop = {'f64': 8, 'f32': 4, 'f16': 2, 'bf16': 2}[case['precision']]
    real = 8 if case['precision'] == 'f64' else 4
    step_bytes = fluid * 38 * pop + nv * 6 * real
    step_flops = fluid * 300.0 + nv * (2 * 64 * 6 + 700.0)
    k = case['steps']
    if case['grad']:
        return {'bytes': float(3 * k * step_bytes + 4 * N * real + nv * 72), 'flops': float(5 * k * step_flops)}
    return {'bytes': float(k * step_bytes + 4 * N * real + nv * 48), 'flops': float(k * step_flops)}


# ---------------------------------------------------------------------------
# The same passes in plain double-precision torch
# ---------------------------------------------------------------------------
_C = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if abs(x) + abs(y) + abs(z) <= 2]
_W = [{0: 1.0 / 3.0, 1: 1.0 / 18.0, 2: 1.0 / 36.0}[abs(x) + abs(y) + abs(z)] for x, y, z in _C]
_OPP = [_C.index((-x, -y, -z)) for x, y, z in _C]


def _peskin(t):
    """Weights of the nodes floor(X) - 1 .. floor(X) + 2, t = X - floor(X)."""
    w = []
    for k in (-1, 0, 1, 2):
        r = (t - k).abs()
        near = (3 - 2 * r + (1 + 4 * r - 4 * r * r).clamp_min(0).sqrt()) / 8
        far = (5 - 2 * r - (-7 + 12 * r - 4 * r * r).clamp_min(1e-30).sqrt()) / 8
        w.append(near if k in (0, 1) else far)
    return w


class _Mesh:
    """Edges, rest geometry and the energy of one membrane type."""

    def __init__(self, m, dev):
        first = {}
        edges = []
        for a, b, c in np.asarray(m.tri).tolist():
            for i, j, o in ((a, b, c), (b, c, a), (c, a, b)):
                if (j, i) in first:
                    edges[first[(j, i)]].append(o)
                else:
                    first[(i, j)] = len(edges)
                    edges.append([i, j, o])
        self.e = torch.tensor(edges, device=dev).T
        self.t = torch.tensor(np.asarray(m.tri, np.int64), device=dev).T
        rest = torch.tensor(np.asarray(m.rest), dtype=torch.float64, device=dev)[None]
        rest = rest - rest.mean(1, keepdim=True)
        self.L0, self.th0 = self._edges(rest)
        A0, V0 = self._area_volume(rest)
        self.A0, self.V0 = float(A0), float(V0)
        self.moduli = torch.tensor([m.k_link, m.k_bend, m.k_area, m.k_volume], dtype=torch.float64, device=dev)
        self.kbt, self.p, self.m2 = m.kbt, m.persistence, m.max_strain ** 2
        self.rest = torch.tensor(np.asarray(m.rest), dtype=torch.float64, device=dev)

    def _edges(self, X):
        p0, p1, pa, pb = (X[:, i] for i in self.e)
        e = p1 - p0
        L = e.square().sum(-1).sqrt()
        n1 = torch.linalg.cross(e, pa - p0)
        n2 = torch.linalg.cross(-e, pb - p1)
        th = torch.atan2((torch.linalg.cross(n1, n2) * e).sum(-1) / L, (n1 * n2).sum(-1))
        return L, th

    def _area_volume(self, X):
        p0, p1, p2 = (X[:, i] for i in self.t)
        n = torch.linalg.cross(p1 - p0, p2 - p0)
        A = 0.5 * n.square().sum(-1).sqrt().sum(-1)
        return A, (p0 * torch.linalg.cross(p1, p2)).sum(-1).sum(-1) / 6

    def energy(self, X, k):
        X = X - X.mean(1, keepdim=True).detach()
        L, th = self._edges(X)
        A, V = self._area_volume(X)
        eps = L / self.L0 - 1
        link = (k[0] * self.kbt / self.p * self.L0 * (eps * eps / 2 - 0.5 * torch.log1p(-eps * eps / self.m2))).sum()
        bend = 0.5 * k[1] * self.kbt * (th - self.th0).square().sum()
        area = 0.5 * k[2] * ((A - self.A0) / self.A0).square().sum()
        return link + bend + area + 0.5 * k[3] * ((V - self.V0) / self.V0).square().sum()

    def forces(self, X, k, graph):
        if graph:
            return -torch.autograd.grad(self.energy(X, k), X, create_graph=True)[0]
        out = []
        for x in X.split(2000):
            with torch.enable_grad():
                x = x.detach().requires_grad_()
                out.append(-torch.autograd.grad(self.energy(x, k), x)[0])
        return torch.cat(out)


def _gyration_index(X):
    d = X - X.mean(1, keepdim=True)
    lam = torch.linalg.eigvalsh(torch.einsum('cvi,cvj->cij', d, d) / X.shape[1]).clamp_min(0).sqrt()
    return (lam[:, 2] - lam[:, 0]) / (lam[:, 2] + lam[:, 0])


class _Reference:
    def __init__(self, case, seed):
        self.case, cfg = case, _config(case, seed)
        self.cfg, dev = cfg, torch.device('cuda')
        self.dims, self.per = (cfg.nx, cfg.ny, cfg.nz), cfg.periodic
        self.shape = (cfg.nz, cfg.ny, cfg.nx)
        self.mesh = [_Mesh(m, dev) for m in cfg.meshes]
        # cells of each type, and their vertices' places in the whole order
        sizes = np.array([len(m.rest) for m in cfg.meshes])
        first = np.concatenate([[0], np.cumsum(sizes[cfg.cell_type])])[:-1]
        self.moving = case['geom'] in ('box', 'chamber')
        self.groups, X = [], torch.zeros((cfg.n_vertices, 3), dtype=torch.float64, device=dev)
        for k, m in enumerate(self.mesh):
            cells = np.nonzero(cfg.cell_type == k)[0]
            idx = torch.tensor(first[cells][:, None] + np.arange(sizes[k]), device=dev)
            R = torch.tensor(cfg.rotations[cells], dtype=torch.float64, device=dev)
            c = torch.tensor(cfg.centers[cells], dtype=torch.float64, device=dev)
            X[idx] = torch.einsum('cij,vj->cvi', R, m.rest) + c[:, None]
            self.groups.append((torch.tensor(cells, device=dev), idx))
        self.X = X
        mask = torch.zeros(self.shape, dtype=torch.uint8, device=dev)
        if cfg.mask is not None:
            mask = torch.tensor(np.ascontiguousarray(cfg.mask), device=dev)
        self.mask, self.wall = mask, mask != 0
        self.uw = torch.zeros((4, 3), dtype=torch.float64, device=dev)
        self.uw[2:] = torch.tensor(cfg.wall_velocity, dtype=torch.float64)
        self.g = torch.tensor(cfg.body_force, dtype=torch.float64, device=dev)
        self.from_wall = []  # per direction: wall id of the node x - c_i (0 fluid)
        for c in _C:
            src = torch.roll(mask, (c[2], c[1], c[0]), (0, 1, 2))
            for d, ax in ((0, 2), (1, 1), (2, 0)):
                if c[d] and not self.per[d]:
                    src.select(ax, 0 if c[d] > 0 else self.dims[d] - 1).fill_(1)
            self.from_wall.append(src)
        u = torch.zeros((3,) + self.shape, dtype=torch.float64, device=dev)
        if cfg.init_velocity is not None:
            u = torch.tensor(cfg.init_velocity, device=dev).permute(3, 0, 1, 2).contiguous()
        uu = u.square().sum(0)
        self.f = []
        for c, w in zip(_C, _W):
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            self.f.append(w * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu))
        self.step_no, self.Up, self.Fv = 0, None, torch.zeros_like(X)
        self.moduli = [m.moduli for m in self.mesh]

    def _membrane(self, X, moduli, graph=False):
        F = torch.zeros_like(X)
        for (_, idx), m, k in zip(self.groups, self.mesh, moduli):
            F = F.index_put((idx.reshape(-1),), m.forces(X[idx], k, graph).reshape(-1, 3))
        return F

    def _layers(self, X, D):
        """Per stencil z-layer: node z, its weight, the x and y stencils
        (indices, weights) and the image's velocity; `live` masks nodes
        beyond a non-periodic edge."""
        def axis(x, d):
            j = x.detach().floor()
            w, idx, live = _peskin(x - j), [], []
            for k in range(4):
                q = j.long() + (k - 1)
                ok = torch.ones_like(q, dtype=torch.bool)
                if not self.per[d]:
                    ok = (q >= 0) & (q < self.dims[d])
                idx.append(q.remainder(self.dims[d]))
                live.append(ok)
            return idx, w, live
        ax, ay, az = axis(X[:, 0], 0), axis(X[:, 1], 1), axis(X[:, 2], 2)
        for k in range(4):
            if D is None:
                yield az[0][k], az[1][k], az[2][k], ax, ay, None
            else:
                q = X[:, 2].floor().long() + (k - 1)
                up, dn = (q >= self.dims[2]).double(), (q < 0).double()
                yield az[0][k], az[1][k], az[2][k], axis(X[:, 0] - D * up + D * dn, 0), ay, LE_SPEED * (up - dn)

    def _nodes(self, X, D):
        for jz, wz, lz, (jx, wx, lx), (jy, wy, ly), du in self._layers(X, D):
            for b in range(4):
                for a in range(4):
                    w = wz * wy[b] * wx[a] * (lz & ly[b] & lx[a])
                    yield (jz * self.dims[1] + jy[b]) * self.dims[0] + jx[a], w, du

    def _spread(self, X, Fv, D):
        F = torch.zeros((self.wall.numel(), 3), dtype=torch.float64, device=X.device)
        for n, w, _ in self._nodes(X, D):
            F = F.index_add(0, n, w[:, None] * Fv) if Fv.requires_grad else F.index_add_(0, n, w[:, None] * Fv)
        return F.T.reshape((3,) + self.shape)

    def _interpolate(self, X, u, D):
        uf, U = u.reshape(3, -1), torch.zeros_like(X)
        for n, w, du in self._nodes(X, D):
            v = uf[:, n].T
            if du is not None:
                v = torch.stack([v[:, 0] + du, v[:, 1], v[:, 2]], 1)
            U = U + w[:, None] * v
        return U

    def _inside(self, X):
        """Nodes with a net signed count of membrane crossings above them."""
        nx, ny, nz = self.dims
        tog = torch.zeros(self.wall.numel(), dtype=torch.int64, device=X.device)
        for (_, idx), m in zip(self.groups, self.mesh):
            P = X[idx][:, m.t].reshape(-1, 3, m.t.shape[1], 3).permute(0, 2, 1, 3).reshape(-1, 3, 3)
            n = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
            s = n[:, 2].sign()
            lo = P[..., :2].amin(1).ceil()
            for kx in range(3):
                for ky in range(3):
                    q = lo + torch.tensor([kx, ky], dtype=torch.float64, device=X.device)
                    ok = s != 0
                    for i in range(3):
                        a, b = P[:, i, :2], P[:, (i + 1) % 3, :2]
                        ok &= s * ((b[:, 0] - a[:, 0]) * (q[:, 1] - a[:, 1]) - (b[:, 1] - a[:, 1]) * (q[:, 0] - a[:, 0])) > 0
                    z = P[:, 0, 2] - (n[:, 0] * (q[:, 0] - P[:, 0, 0]) + n[:, 1] * (q[:, 1] - P[:, 0, 1])) / n[:, 2]
                    j = [q[:, 0].long(), q[:, 1].long(), torch.where(ok, z, 0).ceil().long()]
                    for d in range(3):
                        if self.per[d]:
                            j[d] = j[d].remainder(self.dims[d])
                        else:
                            j[d] = j[d].clamp_min(0) if d == 2 else j[d]
                            ok = ok & (j[d] >= 0) & (j[d] < self.dims[d])
                    tog.index_add_(0, ((j[2] * ny + j[1]) * nx + j[0])[ok], -s[ok].long())
        c = tog.reshape(self.shape).cumsum(0)
        return c > c.amin(0).clamp_max(0)

    def _le_pull(self, fs, i, D):
        """Populations of direction i across the displaced plane."""
        cx, cy, cz = _C[i]
        up = cz < 0  # the top layer pulls from the image above
        src, dU = (0, LE_SPEED) if up else (self.dims[2] - 1, -LE_SPEED)
        plane = [p[src] for p in fs]
        rho = sum(plane)
        u = [sum(c[d] * p for c, p in zip(_C, plane)) / rho for d in range(3)]

        def feq(ux):
            cu = cx * ux + cy * u[1] + cz * u[2]
            return _W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + u[1] ** 2 + u[2] ** 2))
        val = torch.roll(plane[i] + feq(u[0] + dU) - feq(u[0]), cy, 0)
        xs = torch.arange(self.dims[0], dtype=torch.float64, device=rho.device) - cx + (-D if up else D)
        fl = xs.floor()
        w, k = xs - fl, fl.long()
        return (1 - w) * val[:, k.remainder(self.dims[0])] + w * val[:, (k + 1).remainder(self.dims[0])]

    def lattice(self, f, F, uw, omega, D):
        rho = sum(f)
        u = [(sum(c[d] * p for c, p in zip(_C, f) if c[d]) + 0.5 * F[d]) / rho for d in range(3)]
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        fs = []
        for i, (c, w) in enumerate(zip(_C, _W)):
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            cF = c[0] * F[0] + c[1] * F[1] + c[2] * F[2]
            eq = w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
            fs.append((1 - omega) * f[i] + omega * eq + (1 - 0.5 * omega) * w * (3 * (cF - uF) + 9 * cu * cF))
        new = []
        for i, c in enumerate(_C):
            p = torch.roll(fs[i], (c[2], c[1], c[0]), (0, 1, 2))
            if D is not None and c[2]:
                p[self.dims[2] - 1 if c[2] < 0 else 0] = self._le_pull(fs, i, D)
            if i != _OPP[i] and D is None:
                src, o = self.from_wall[i], _OPP[i]
                cw = (uw * torch.tensor(_C[o], dtype=torch.float64, device=uw.device)).sum(1)
                back = fs[o] - 6 * _W[i] * rho * cw[src.long()] if self.moving else fs[o]
                p = torch.where(src != 0, back, p)
            new.append(torch.where(self.wall, _W[i], p))
        rho = sum(new)
        u = torch.stack([(sum(c[d] * p for c, p in zip(_C, new) if c[d]) + 0.5 * F[d]) / rho for d in range(3)])
        if self.case['geom'] != 'lees':
            u = torch.where(self.wall, uw[self.mask.long()].permute(3, 0, 1, 2) if self.moving else 0.0, u)
        return new, u

    def step(self):
        D = None
        if self.case['geom'] == 'lees':
            D = LE_SPEED * self.step_no % self.dims[0]
            for _, idx in self.groups:
                z = self.X[idx][..., 2].mean(1)
                hop = (z >= self.dims[2]).double() - (z < 0).double()
                self.X[idx] -= hop[:, None, None] * torch.tensor([D, 0.0, self.dims[2]], dtype=torch.float64, device=z.device)
        if self.step_no % self.case['every'] == 0:
            self.Fv = self._membrane(self.X, self.moduli)
        omega = 1.0
        if self.case['visc'] != 1.0:
            omega = 1.0 + (1.0 / (0.5 + 0.5 * self.case['visc']) - 1.0) * self._inside(self.X).double()
        F = self._spread(self.X, self.Fv, D) + self.g[:, None, None, None]
        F.masked_fill_(self.wall, 0.0)
        self.f, self.u = self.lattice(self.f, F, self.uw, omega, D)
        U = self._interpolate(self.X, self.u, D)
        ab2 = self.case['integrator'] == 'ab2' and self.Up is not None
        self.X = self.X + (1.5 * U - 0.5 * self.Up if ab2 else U)
        self.Up = U
        self.step_no += 1

    def stats(self):
        out = torch.zeros((len(self.cfg.centers), 6), dtype=torch.float64, device=self.X.device)
        for (cells, idx), m in zip(self.groups, self.mesh):
            X = self.X[idx]
            c = X.mean(1)
            A, V = m._area_volume(X - c[:, None])
            out[cells] = torch.cat([c, A[:, None], V[:, None], _gyration_index(X)[:, None]], 1)
        return out

    def fields(self):
        rho = torch.where(self.wall, 0.0, sum(self.f))
        return {'rho': rho, 'u': self.u.permute(1, 2, 3, 0).contiguous(), 'X': self.X, 'Fv': self.Fv,
                'cellstats': self.stats()}

    def gradient(self):
        """Loss, its gradient by the vertices and the parameter gradients, by
        automatic differentiation of the steps."""
        from torch.utils.checkpoint import checkpoint
        k = [m.moduli.clone().requires_grad_() for m in self.mesh]
        s = torch.ones((), dtype=torch.float64, device=self.X.device, requires_grad=True)
        g = self.g.clone().requires_grad_()
        c0 = [self.X[idx].mean(1) for _, idx in self.groups]

        def one(X, s, g, *rest):
            kk, f = rest[:len(k)], rest[len(k):]
            if not X.requires_grad:
                X = X.requires_grad_()
            F = self._spread(X, self._membrane(X, kk, True), None) + g[:, None, None, None]
            f, u = self.lattice(list(f), torch.where(self.wall, 0.0, F), self.uw * s, 1.0, None)
            return (X + self._interpolate(X, u, None), *f)
        state = (self.X.clone().requires_grad_(), *self.f)
        for _ in range(self.case['steps']):
            state = checkpoint(one, state[0], s, g, *k, *state[1:], use_reentrant=False)
        X = state[0]
        loss = 0.0
        for (_, idx), c in zip(self.groups, c0):
            loss = loss + (_gyration_index(X[idx]) + (X[idx].mean(1) - c).square().sum(1)).sum()
        loss = loss / len(self.cfg.centers)
        got = torch.autograd.grad(loss, [X, *k, s, g])
        return {'loss': loss.detach().reshape(1), 'dX': got[0], 'grad': torch.cat([x.reshape(-1) for x in got[1:]])}


def exact(case, seed):
    r = _Reference(case, seed)
    res = r.gradient() if case['grad'] else {}
    with torch.no_grad():
        for _ in range(case['steps']):
            r.step()
        return {**res, **r.fields()}
