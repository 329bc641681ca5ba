"""Measured cases of the particle step, the downshifted step and the gradients.

A case is one pass of a user's program through the public entry points: a
window of particle steps with their deposits (and the re-sort by tet that
ends it on a large load), a window of downshifted steps, or one gradient.
Loads, meshes and fields follow the package's own workloads: Kuhn cubes of
n^3 x 6 tets (plain or with jittered interior nodes), thermal electrons in the
TE101 cavity mode, a 10 keV beam in plasma or electrons with heavy ions in
windowed random envelopes, dt = 0.5 ns.

A large window starts from a kept state, copied in at its beginning (as a
resumed or differentiated run does): every pass then does the same work, on
an order that has drifted by the window's own steps only, as in a run that
re-sorts on that cadence.

`exact` is the same pass in 64-bit torch arithmetic, independent of the
package: Whitney sums from their definition, the Boris step, the face walk
with the path-integral deposit, the downshifted rule with Gauss-Legendre
weights, and gradients by differentiating those step by step.
"""
import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2208_12795_gb300 import adjoint
from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState

Q_E, M_E, C_0 = 1.602176634e-19, 9.1093837015e-31, 299792458.0
OMEGA0 = C_0 * math.pi * math.sqrt(2.0)   # TE101 mode of the unit cube
DT = 0.5e-9
T0 = 60e-9                                # past the rise of the envelope: a(t) = 1
PRECISION = {"fp64": 0, "mixed": 1, "q24": 2}
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    def case(name, kind, form, cells, particles, steps, load="thermal", jitter=False, walls="reflect", sort=True):
        return dict(name=name, kind=kind, form=form, cells=cells, particles=particles, steps=steps, load=load,
                    jitter=jitter, walls=walls, sort=sort)

    return [
        # the smallest run: 384 tets, 2000 electrons, one step in full precision; launches and latency are all there is
        case("tiny_fp64", "step", "fp64", 4, 2000, 1, sort=False),
        # a small ragged load under the three-level envelope of a coarse field step, on a distorted mesh
        case("ragged_levels3", "levels3", "mixed", 16, 100003, 1, jitter=True, sort=False),
        # the cavity benchmark: 10M electrons, four steps of the contract form and the re-sort that follows them
        case("cavity_mixed", "step", "mixed", 48, 10000000, 4),
        # the same loop in the fast 24-bit variant
        case("cavity_q24", "step", "q24", 40, 6000001, 4),
        # the same loop in full precision (reference runs, convergence studies)
        case("cavity_fp64", "step", "fp64", 40, 6000000, 4),
        # a fast beam through plasma on a distorted mesh, walls that collect: many face crossings per step
        case("beam_mixed", "step", "mixed", 48, 24000000, 4, load="beam", jitter=True, walls="absorb"),
        # the largest: electrons and heavy ions, 72 per tet, the density of the 400M-particle production load
        case("species_mixed", "step", "mixed", 48, 48000000, 4, load="species"),
        # the downshifted integrator with its velocity and sample history, in full precision
        case("downshift_fp64", "downshift", "fp64", 32, 2000001, 8),
        # the same on the contract form, history re-sorted with its particles
        case("downshift_mixed", "downshift", "mixed", 48, 10000000, 8),
        # the differentiation workload: kinetic energy after 50 steps of 4M electrons, checkpoints every 10
        case("energy_grad_mixed", "energy_grad", "mixed", 48, 4000000, 50),
        # the same gradient in full precision (checks of a design study)
        case("energy_grad_fp64", "energy_grad", "fp64", 24, 500000, 20),
        # gradient of the deposited current (the coupling to a field or circuit) on a distorted mesh
        case("current_grad_mixed", "current_grad", "mixed", 24, 300007, 10, jitter=True),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "levels3", "downshift", "energy_grad", "current_grad"])
    form = rng.choice(["mixed", "mixed", "q24", "fp64"])
    most = {"step": 16e6, "levels3": 16e6, "downshift": 4e6, "energy_grad": 1e6, "current_grad": 4e5}[kind]
    cells = int(round(math.exp(rng.uniform(math.log(4), math.log(40)))))
    density = math.exp(rng.uniform(math.log(3), math.log(80)))
    particles = int(min(max(6 * cells ** 3 * density, 1000), most)) - rng.randrange(300)
    sort = particles >= 200000 and kind in ("step", "levels3", "downshift")
    load = rng.choice(["thermal", "thermal", "beam", "species"]) if kind != "downshift" else "thermal"
    walls = "absorb" if sort and kind in ("step", "levels3") and rng.random() < 0.3 else "reflect"
    steps = rng.randrange(5, 21) if kind.endswith("grad") else rng.randrange(2, 7) if sort else rng.randrange(1, 4)
    return dict(kind=kind, form=form, cells=cells, particles=particles, steps=steps, load=load,
                jitter=rng.random() < 0.5, walls=walls, sort=sort)


# ---------------------------------------------------------------- inputs
def mesh_of(case, seed):
    """Unit cube of cells^3 hexes in six Kuhn tets each; interior nodes jittered by up to 20 % of the spacing."""
    n, m = case["cells"], case["cells"] + 1
    i = torch.arange(m, device=DEVICE, dtype=torch.float64) / n
    nodes = torch.stack(torch.meshgrid(i, i, i, indexing="ij"), -1).permute(2, 1, 0, 3).reshape(-1, 3).contiguous()
    if case["jitter"]:
        g = torch.Generator(device=DEVICE).manual_seed(seed * 8 + 1)
        inside = ((nodes > 0.5 / n) & (nodes < 1 - 0.5 / n)).all(1)
        shift = (torch.rand(nodes.shape, generator=g, device=DEVICE, dtype=torch.float64) - 0.5) * (0.4 / n)
        nodes = nodes + shift * inside[:, None]
    c = torch.arange(n, device=DEVICE)
    corner = (c[None, None, :] + m * (c[None, :, None] + m * c[:, None, None])).reshape(-1)
    stride = (1, m, m * m)
    tets = []
    for p in itertools.permutations(range(3)):
        path = [corner]
        for axis in p:
            path.append(path[-1] + stride[axis])
        tets.append(torch.stack(path, 1))
    return nodes, torch.stack(tets, 1).reshape(-1, 4)


def numbering(nodes, tets):
    """Sorted tet nodes; edges and faces numbered by their sorted node tuples, and each tet's edge and face ids."""
    ts, nn = tets.sort(1).values, nodes.shape[0]
    e = torch.stack([ts[:, i] * nn + ts[:, j] for i, j in itertools.combinations(range(4), 2)], 1)
    f = torch.stack([(ts[:, i] * nn + ts[:, j]) * nn + ts[:, k] for i, j, k in ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))], 1)
    edges, te = torch.unique(e, return_inverse=True)
    faces, tf = torch.unique(f, return_inverse=True)
    edges = torch.stack([edges // nn, edges % nn], 1)
    faces = torch.stack([faces // nn // nn, faces // nn % nn, faces % nn], 1)
    return ts, edges, te, faces, tf


def fields_of(case, seed, nodes, edges, faces):
    """Envelope DoFs: the TE101 mode (edge circulations and face fluxes by
    midpoint quadrature of the mode at 10 kV/m), or complex normal DoFs in a
    Gaussian window about the centre (10 kV/m, 10 mT)."""
    g = torch.Generator(device=DEVICE).manual_seed(seed * 8 + 2)
    normal = lambda n: torch.complex(*(torch.randn(n, generator=g, device=DEVICE, dtype=torch.float64) for _ in range(2))) / math.sqrt(2)
    em, fm = nodes[edges].mean(1), nodes[faces].mean(1)
    if case["load"] == "thermal":
        s, c = (lambda x: torch.sin(math.pi * x)), (lambda x: torch.cos(math.pi * x))
        phase = complex(math.cos(seed % 7), math.sin(seed % 7))
        e = 1e4 * (nodes[edges[:, 1]] - nodes[edges[:, 0]])[:, 1] * s(em[:, 0]) * s(em[:, 2]) * phase
        area = 0.5 * torch.linalg.cross(nodes[faces[:, 1]] - nodes[faces[:, 0]], nodes[faces[:, 2]] - nodes[faces[:, 0]])
        flux = 1e4 * math.pi * (area[:, 2] * c(fm[:, 0]) * s(fm[:, 2]) - area[:, 0] * s(fm[:, 0]) * c(fm[:, 2]))
        return e, flux * (1j / OMEGA0) * phase
    h = 1.0 / case["cells"]
    window = lambda x: torch.exp(-((x - 0.5) ** 2).sum(1) / (2 * 0.25 ** 2))
    return 1e4 * h * normal(len(edges)) * window(em), 1e-2 * h * h * normal(len(faces)) * window(fm)


def levels_of(case, e, b):
    """Three slowly varying field levels about the middle of a field step of 21 particle steps, and their weights by time."""
    scale = (0.98 + 0.01j, 1.0, 1.02 - 0.01j)
    tau = [T0 + k * 21 * DT for k in (-1, 0, 1)]

    def weights(t):
        return [math.prod((t - tau[j]) / (tau[k] - tau[j]) for j in range(3) if j != k) for k in range(3)]

    return [e * s for s in scale], [b * s for s in scale], weights


def load_of(case, seed, nodes, ts):
    """Particles ordered by (species, tet): positions uniform in tets drawn by
    volume times the density profile, velocities, and the species table."""
    g = torch.Generator(device=DEVICE).manual_seed(seed * 8 + 3)
    f64 = dict(device=DEVICE, dtype=torch.float64)
    n = case["particles"]
    corners = nodes[ts]
    volume = torch.linalg.det(corners[:, 1:] - corners[:, :1]).abs()
    mid = corners.mean(1)

    def place(count, weight):
        total = weight.cumsum(0)
        u = torch.rand(count, generator=g, **f64).mul_(total[-1])
        tet = torch.searchsorted(total, u).clamp_(max=len(ts) - 1).sort().values
        lam = torch.rand((count, 4), generator=g, **f64).clamp_(min=1e-12).log_().neg_()
        lam /= lam.sum(1, keepdim=True)
        return tet, [(lam * corners[:, :, a][tet]).sum(1) for a in range(3)]

    def thermal(count, ev, mass):
        return [torch.randn(count, generator=g, **f64) * math.sqrt(Q_E * ev / mass) for _ in range(3)]

    if case["load"] == "thermal":
        ev = 1.0 if case["cells"] < 10 else 5.0
        parts = [(n, volume, thermal(n, ev, M_E), -Q_E, M_E)]
    elif case["load"] == "beam":   # a tenth of the load is a 10 keV beam along z, the rest plasma with a cosine profile
        nb = n // 10
        energy = 1e4 * (1 + 0.005 * torch.randn(nb, generator=g, **f64))
        zero = torch.zeros(nb, **f64)
        parts = [(nb, volume * torch.exp(-((mid[:, :2] - 0.5) ** 2).sum(1) / (2 * 0.1 ** 2)),
                  [zero, zero, torch.sqrt(2 * energy.clamp(min=0) * Q_E / M_E)], -Q_E, M_E),
                 (n - nb, volume * (1 + 0.5 * torch.cos(2 * math.pi * mid[:, 0])), thermal(n - nb, 5.0, M_E), -Q_E, M_E)]
    else:                          # electrons and heavy ions at 2 eV
        parts = [(n // 2, volume, thermal(n // 2, 2.0, M_E), -Q_E, M_E),
                 (n - n // 2, volume, thermal(n - n // 2, 2.0, 1836 * M_E), Q_E, 1836 * M_E)]
    placed = [place(count, weight) for count, weight, _, _, _ in parts]
    begin = np.cumsum([0] + [p[0] for p in parts])
    join = lambda lists: [torch.cat([x[a] for x in lists]) for a in range(3)]
    return SimpleNamespace(n=n, tet=torch.cat([t for t, _ in placed]), x=join([x for _, x in placed]),
                           v=join([p[2] for p in parts]), begin=begin.astype(np.int64),
                           q=np.array([p[3] for p in parts]), m=np.array([p[4] for p in parts]),
                           w=np.full(len(parts), 1e3))


def inputs_of(case, seed):
    nodes, tets = mesh_of(case, seed)
    ts, edges, te, faces, tf = numbering(nodes, tets)
    e, b = fields_of(case, seed, nodes, edges, faces)
    load = load_of(case, seed, nodes, ts)
    if case["form"] != "fp64":     # the mixed forms take complex64 DoFs and float32 velocities
        e, b = e.to(torch.complex64), b.to(torch.complex64)
        load.v = [v.float() for v in load.v]
    g = torch.Generator(device=DEVICE).manual_seed(seed * 8 + 4)
    u = torch.randn(len(edges), generator=g, device=DEVICE, dtype=torch.float64) if case["kind"] == "current_grad" else None
    return SimpleNamespace(nodes=nodes, tets=tets, ts=ts, edges=edges, te=te, faces=faces, tf=tf, e=e, b=b, load=load, u=u)


ARRAYS = ("x", "y", "z", "vx", "vy", "vz", "tet", "status", "n_cross")


def packed(n, vdtype, load, count):
    """A particle set in one allocation (each array on a 256-byte boundary)."""
    types = [torch.float64] * 3 + [vdtype] * 3 + [torch.int32, torch.uint8] + ([torch.int32] if count else [])
    sizes = [-(-n * t.itemsize // 256) * 256 for t in types]
    flat = torch.zeros(sum(sizes), dtype=torch.uint8, device=DEVICE)
    views = [flat[at:at + n * t.itemsize].view(t) for at, t in zip(np.cumsum([0] + sizes[:-1]), types)]
    st = ParticleState(*views[:6], load.begin, load.q, load.m, load.w, tet=views[6], track_crossings=False)
    st.status = views[7]
    st.n_cross = views[8] if count else None
    return flat, st


def prepare(case, seed):
    i = inputs_of(case, seed)
    s = SimpleNamespace(case=case, e=i.e, b=i.b, u=i.u, passes=0)
    s.env = FempicEnv(i.nodes.cpu().numpy(), i.tets.to(torch.int32).cpu().numpy(), precision=PRECISION[case["form"]],
                      wall_mode=int(case["walls"] == "absorb"))
    grad = case["kind"].endswith("grad")
    # small runs keep the crossing counter, the large loads and the gradients go without, as the benchmark does
    s.flat, s.st = packed(i.load.n, i.load.v[0].dtype, i.load, not case["sort"] and not grad)
    for name, values in zip(ARRAYS, i.load.x + i.load.v):
        getattr(s.st, name).copy_(values)
    s.env.locate(s.st)
    if case["sort"] and not grad:
        s.kept = s.flat.clone()
        s.spare_flat, s.spare = packed(i.load.n, i.load.v[0].dtype, i.load, False)
    if case["kind"] == "levels3":
        s.e, s.b, s.weights = levels_of(case, i.e, i.b)
    elif case["kind"] == "downshift":
        s.ds = Downshift(s.env, i.load.n)
    elif grad:
        s.schedule = adjoint.Schedule(lambda t: 1.0, OMEGA0, DT, case["steps"], 10 if case["steps"] > 20 else 5, T0)
    if not grad:
        s.dG = torch.empty(s.env.n_edges, dtype=torch.float64, device=DEVICE)
        s.G = torch.empty(s.env.n_edges, dtype=torch.complex128, device=DEVICE)
    return s


def run(s):
    case, env, st, kind = s.case, s.env, s.st, s.case["kind"]
    if kind == "energy_grad":
        L, eg, bg, a = adjoint.kinetic_energy_and_grad(env, st, s.e, s.b, s.schedule)
        return [L, eg, bg, a.rx, a.ry, a.rz, a.vx, a.vy, a.vz]
    if kind == "current_grad":
        L, eg, bg, a = adjoint.current_loss_and_grad(env, st, s.e, s.b, s.schedule, s.u)
        return [L, eg, bg, a.rx, a.ry, a.rz, a.vx, a.vy, a.vz]
    first = 0
    if case["sort"]:
        s.flat.copy_(s.kept)
    else:                          # a small run goes on from where the last pass left it
        first, s.passes = s.passes * case["steps"], s.passes + 1
    if kind == "downshift" and case["sort"]:
        s.ds.started = False       # the kept state starts a run: the first step fills the history
    for k in range(first, first + case["steps"]):
        t = T0 + k * DT
        if kind == "downshift":
            s.ds.step(st, s.e, s.b, 1.0, OMEGA0, t, DT)
        elif kind == "levels3":
            env.push_step3(st, s.e, s.b, s.weights(t), 1.0, OMEGA0, t, DT)
        else:
            env.push_step(st, s.e, s.b, 1.0, OMEGA0, t, DT)
        env.deposit(OMEGA0, t + DT, dG_out=s.dG, G_env_out=s.G)
    out = [st.x, st.y, st.z, st.vx, st.vy, st.vz, s.dG, s.G, st.tet, st.status]
    if kind == "downshift":
        out.append(s.ds.planes[:33])
    if case["sort"]:               # the state as stepped is left in the buffers sorted from
        s.ds.sort(st, s.spare) if kind == "downshift" else env.sort(st, s.spare)
        s.flat, s.spare_flat = s.spare_flat, s.flat
        # the sorted order shows in the tets; collected particles come last, in no stated order
        out.append(st.status if case["walls"] == "absorb" else st.tet)
    elif st.n_cross is not None:
        out.append(st.n_cross)
    return out


def work(case):
    """Bytes by call, each array of a call read or written once: the particle
    state in and out (positions, velocities, tet), the mesh's nodes and tets,
    the DoFs and the edge outputs; a sort and a restart move the whole state."""
    n, c, f64 = case["particles"], case["cells"], case["form"] == "fp64"
    nn, nt = (c + 1) ** 3, 6 * c ** 3
    ne = 3 * c * (c + 1) ** 2 + 3 * c * c * (c + 1) + c ** 3
    nf = 1 - nn + ne + nt
    vel = 24 if f64 else 12
    dof = (16 if f64 else 8) * (ne + nf)
    state = 24 + vel + 4
    step = 2 * state * n + 72 * nt + 24 * nn + dof + 40 * ne
    kind, steps = case["kind"], case["steps"]
    if kind.endswith("grad"):
        back = n * (state + 1 + vel + 2 * (24 + vel)) + 72 * nt + 24 * nn + 2 * dof
        sorts = -(-steps // (10 if steps > 20 else 5))
        return dict(bytes=steps * (2 * step + back) + sorts * n * 2 * (2 * state + vel), flops=steps * n * 700)
    if kind == "levels3":
        step += 2 * dof
    if kind == "downshift":
        step += 2 * 33 * (vel // 3) * n
    moved = 4 * (state + 1) * n if case["sort"] else 0
    if kind == "downshift" and case["sort"]:
        moved += 2 * 33 * (vel // 3) * n
    return dict(bytes=steps * step + moved, flops=steps * n * (450 if kind == "downshift" else 250))


# ---------------------------------------------------------------- 64-bit values
LOCAL_EDGES = list(itertools.combinations(range(4), 2))
LOCAL_FACES = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))
CHUNK = 1 << 20


class Exact:
    """The mesh in 64 bits: barycentric gradients, neighbours, walls, and the particle physics on it."""

    def __init__(self, i, absorb):
        self.i, self.absorb, self.ts, self.te = i, absorb, i.ts, i.te
        p = i.nodes[i.ts]
        inv = torch.linalg.inv((p[:, 1:] - p[:, :1]).transpose(1, 2))   # rows: gradients of lambda_1..3
        self.grad = torch.cat([-inv.sum(1, keepdim=True), inv], 1)
        self.x0, self.corner = p[:, 0].contiguous(), p
        nt = len(i.ts)
        flat = i.tf.reshape(-1)
        order = flat.sort(stable=True).indices
        same = flat[order][1:] == flat[order][:-1]
        a, b = order[:-1][same], order[1:][same]
        nb = torch.full((4 * nt,), -7, device=DEVICE)
        nb[a], nb[b] = b // 4, a // 4
        wall = i.nodes[i.faces][i.tf]                                   # [nt, 4, 3, 3]
        for axis in range(3):
            for side in range(2):
                on = (wall[..., axis] == float(side)).all(2).reshape(-1) & (nb == -7)
                nb[on] = -1 - (2 * axis + side)
        self.nb = nb.reshape(nt, 4)

    def vertex_fields(self, e, b):
        """E and B of real DoFs e, b at each tet's corners (both are affine inside a tet): [nt, 4, 6]."""
        g, ee, bb = self.grad, e[self.te], b[self.i.tf]
        E = [0.0] * 4
        for k, (i, j) in enumerate(LOCAL_EDGES):
            E[i] = E[i] + ee[:, k, None] * g[:, j]
            E[j] = E[j] - ee[:, k, None] * g[:, i]
        B = [0.0] * 4
        for k, f in enumerate(LOCAL_FACES):
            for r in range(3):
                i, j, l = f[r], f[(r + 1) % 3], f[(r + 2) % 3]
                B[i] = B[i] + 2 * bb[:, k, None] * torch.linalg.cross(g[:, j], g[:, l])
        return torch.cat([torch.stack(E, 1), torch.stack(B, 1)], 2)

    def bary(self, tet, r):
        l = (self.grad[tet, 1:] * (r - self.x0[tet])[:, None]).sum(2)
        return torch.cat([1 - l.sum(1, keepdim=True), l], 1)

    def gather(self, F, tet, r):
        return (self.bary(tet, r)[:, :, None] * F[tet]).sum(1)

    def boris(self, EB, v, kq, dt):
        E, B = EB[:, :3], EB[:, 3:]
        vm, t = v + kq * E, kq * B
        s = 2 * t / (1 + (t * t).sum(1, keepdim=True))
        return vm + torch.linalg.cross(vm + torch.linalg.cross(vm, t), s) + kq * E

    def walk(self, tet, a, b, piece):
        """Follow the segments a -> b from tet to tet, mirrored (or stopped) at
        walls; piece(tet, la, lb, particle) sees each in-tet piece.  Returns
        tets, end points, velocity signs and crossings; a stopped particle's
        tet comes back as -2 - tet."""
        n = len(tet)
        ids, T, la, sign = torch.arange(n, device=DEVICE), tet, self.bary(tet, a), torch.ones_like(a)
        entry = torch.full((n,), -1, device=DEVICE)
        crossings = torch.zeros(n, dtype=torch.int64, device=DEVICE)
        done = []
        while len(ids):
            lb = self.bary(T, b)
            out = (lb < 0) & (torch.arange(4, device=DEVICE) != entry[:, None])
            s = torch.where(out, la / torch.where(out, la - lb, torch.ones_like(lb)), torch.full_like(lb, math.inf))
            s, face = torch.where(out, s.clamp(min=0), s).min(1)
            stays = ~out.any(1)
            s = torch.where(stays, torch.ones_like(s), s)
            lp = la + s[:, None] * (lb - la)
            at = torch.arange(4, device=DEVICE) == face[:, None]
            lp = torch.where(stays[:, None], lb, torch.where(at, torch.zeros_like(lp), lp))
            piece(T, la, lp, ids)
            done.append((ids[stays], T[stays], b[stays], sign[stays]))
            ids, T, b, sign, face, lp = (x[~stays] for x in (ids, T, b, sign, face, lp))
            crossings[ids] += 1
            nbt = self.nb[T, face]
            hit = nbt < 0
            if self.absorb and bool(hit.any()):
                stop = (lp[hit][:, :, None] * self.corner[T[hit]]).sum(1)
                done.append((ids[hit], -2 - T[hit], stop, sign[hit]))
                ids, T, b, sign, face, lp, nbt = (x[~hit] for x in (ids, T, b, sign, face, lp, nbt))
                hit = nbt < 0
            axis, side = (-1 - nbt) // 2, (-1 - nbt) % 2
            flip = hit[:, None] & (torch.arange(3, device=DEVICE) == axis[:, None])
            b = torch.where(flip, 2.0 * side[:, None] - b, b)
            sign = torch.where(flip, -sign, sign)
            new = torch.where(hit, T, nbt)
            match = self.ts[T][:, None, :] == self.ts[new][:, :, None]   # [m, node of the new tet, node of the old]
            la = (match * lp[:, None, :]).sum(2)
            entry = torch.where(hit, face, (~match.any(2)).to(torch.int64).argmax(1))
            T = new
        back = torch.cat([d[0] for d in done]).argsort()
        return tuple(torch.cat([d[k] for d in done])[back] for k in (1, 2, 3)) + (crossings,)


def pieces(te, la, lb):
    """Path integrals of the six edge functions over a straight piece of each tet."""
    return te, torch.stack([la[:, i] * lb[:, j] - la[:, j] * lb[:, i] for i, j in LOCAL_EDGES], 1)


def real_dofs(case, i, t):
    """Re{c N_k(t) DoFs} summed over the levels, in 64 bits (one level: N = 1)."""
    c = complex(math.cos(OMEGA0 * t), math.sin(OMEGA0 * t))
    if case["kind"] != "levels3":
        return [(c * d.to(torch.complex128)).real for d in (i.e, i.b)]
    e3, b3, weights = levels_of(case, i.e, i.b)
    return [sum((c * w * d.to(torch.complex128)).real for w, d in zip(weights(t), d3)) for d3 in (e3, b3)]


def chunks(load):
    """(slice, q/m, q w, m w) of runs of one species, a million particles at most each."""
    for s in range(len(load.q)):
        for at in range(int(load.begin[s]), int(load.begin[s + 1]), CHUNK):
            yield (slice(at, min(at + CHUNK, int(load.begin[s + 1]))), load.q[s] / load.m[s], load.q[s] * load.w[s],
                   load.m[s] * load.w[s])


def exact(case, seed):
    i = inputs_of(case, seed)
    M = Exact(i, case["walls"] == "absorb")
    x, v = torch.stack(i.load.x, 1), torch.stack([w.double() for w in i.load.v], 1)
    if case["kind"].endswith("grad"):
        return exact_gradient(case, i, M, x, v)
    steps = range(case["steps"])
    times = [T0 + k * DT for k in steps]
    dG = torch.zeros((case["steps"], len(i.edges)), dtype=torch.float64, device=DEVICE)
    xo, vo = torch.empty_like(x), torch.empty_like(v)
    planes = None
    if case["kind"] == "downshift":
        parts = [[d.to(torch.complex128).real, d.to(torch.complex128).imag] for d in (i.e, i.b)]
        F = torch.cat([M.vertex_fields(parts[0][r], parts[1][r]) for r in range(2)], 2)   # Re E, Re B, Im E, Im B
        planes = torch.empty((33, len(x)), dtype=torch.float64, device=DEVICE)
    else:
        F = [M.vertex_fields(*real_dofs(case, i, t)) for t in times]
    for at, qm, qw, _ in chunks(i.load):
        tet, r, u = i.load.tet[at].clone(), x[at], v[at]
        history = None
        for k, t in zip(steps, times):
            live = (tet >= 0).nonzero()[:, 0]

            def piece(T, la, lb, ids):
                e, g = pieces(M.te[T], la, lb)
                dG[k].index_add_(0, e.reshape(-1), (qw * g).reshape(-1))

            if planes is None:
                new = M.boris(M.gather(F[k], tet[live], r[live]), u[live], qm * DT / 2, DT)
                T, end, sign, _ = M.walk(tet[live], r[live], r[live] + DT * new, piece)
                new = new * sign
            else:
                new, drift, history = downshifted(M, F, tet, r, u, qm, t, history)
                T, end, sign, _ = M.walk(tet, r, r + DT * drift, piece)
                new, history = new * sign, ([h * sign for h in history[0]], history[1])
            tet, r, u = tet.index_copy(0, live, T), r.index_copy(0, live, end), u.index_copy(0, live, new)
        xo[at], vo[at] = r, u
        if planes is not None:
            planes[:, at] = torch.cat([torch.cat(history[0], 1), torch.cat(history[1], 1)], 1).T
    t = times[-1] + DT
    G = dG.sum(0) * complex(math.cos(OMEGA0 * t), -math.sin(OMEGA0 * t))
    out = [xo[:, 0], xo[:, 1], xo[:, 2], vo[:, 0], vo[:, 1], vo[:, 2], dG[-1], G, None, None]
    return out + ([planes] if planes is not None else []) + [None]


def downshift_weights(t):
    """Integrals over [t, t + dt] of N_k and N_j N_k against cos and -sin of the carrier (40-point Gauss-Legendre)."""
    y, w = np.polynomial.legendre.leggauss(40)
    y, w = (y + 1) / 2, w * DT / 2
    N = [np.prod([(y + j) / (j - k) for j in range(3) if j != k], 0) for k in range(3)]
    c, s = np.cos(OMEGA0 * (t + DT * y)), -np.sin(OMEGA0 * (t + DT * y))
    return ([[float((w * N[k] * f).sum()) for k in range(3)] for f in (c, s)],
            [[[float((w * N[j] * N[k] * f).sum()) for k in range(3)] for j in range(3)] for f in (c, s)])


def downshifted(M, F, tet, r, v, qm, t, history):
    """Velocity rule on the newest three samples, Adams-Bashforth drift, and the history with this step's values in front."""
    f = M.gather(F, tet, r)
    now = torch.cat([f[:, 0:3], f[:, 6:9], f[:, 3:6], f[:, 9:12]], 1)   # Re E, Im E, Re B, Im B
    vh, fh = history or ([v] * 3, [now] * 2)
    S, V = [now] + fh, [v] + vh[:2]
    Mw, L = downshift_weights(t)
    dv = sum(S[k][:, 0:3] * Mw[0][k] + S[k][:, 3:6] * Mw[1][k] for k in range(3))
    for j in range(3):
        dv = dv + torch.linalg.cross(V[j], sum(S[k][:, 6:9] * L[0][j][k] + S[k][:, 9:12] * L[1][j][k] for k in range(3)))
    drift = (55 * v - 59 * vh[0] + 37 * vh[1] - 9 * vh[2]) / 24
    return v + qm * dv, drift, ([v] + vh[:2], [now, fh[0]])


def exact_gradient(case, i, M, x, v):
    """The loss and its gradients: the steps forward, then each differentiated alone from the last to the first."""
    energy = case["kind"] == "energy_grad"
    times = [T0 + k * DT for k in range(case["steps"])]
    L = torch.zeros((), dtype=torch.float64, device=DEVICE)
    gF = [None] * len(times)
    F = []
    for k, t in enumerate(times):
        F.append(M.vertex_fields(*real_dofs(case, i, t)))
        gF[k] = torch.zeros_like(F[k])
    rx, rv = torch.empty_like(x), torch.empty_like(v)

    def step(k, tet, r, u, qm, qw):
        loss = torch.zeros((), dtype=torch.float64, device=DEVICE)

        def piece(T, la, lb, ids):
            nonlocal loss
            if not energy:
                e, g = pieces(M.te[T], la, lb)
                loss = loss + qw * (i.u[e] * g).sum()

        new = M.boris(M.gather(F[k], tet, r), u, qm * DT / 2, DT)
        T, end, sign, _ = M.walk(tet, r, r + DT * new, piece)
        return T, end, new * sign, loss

    for at, qm, qw, mw in chunks(i.load):
        states = [(i.load.tet[at], x[at], v[at])]
        with torch.no_grad():
            for k in range(len(times)):
                T, r, u, loss = step(k, *states[-1], qm, qw)
                states.append((T, r, u))
                L += loss
        T, r, u = states.pop()
        if energy:
            L += 0.5 * mw * (u * u).sum()
        gr, gu = torch.zeros_like(r), mw * u if energy else torch.zeros_like(u)
        for k in reversed(range(len(times))):
            T, r, u = states.pop()
            leaf = [F[k], r.detach(), u.detach()]
            for w in leaf:
                w.requires_grad_(True)
            _, end, new, loss = step(k, T, leaf[1], leaf[2], qm, qw)
            total = (end * gr).sum() + (new * gu).sum() + loss
            d, gr, gu = torch.autograd.grad(total, leaf)
            gF[k] += d
            F[k] = F[k].detach()
        rx[at], rv[at] = gr, gu
    grads = [torch.zeros(len(d), dtype=torch.complex128, device=DEVICE) for d in (i.e, i.b)]
    for k, t in enumerate(times):
        dofs = [d.detach().requires_grad_(True) for d in real_dofs(case, i, t)]
        d = torch.autograd.grad((M.vertex_fields(*dofs) * gF[k]).sum(), dofs)
        c = complex(math.cos(OMEGA0 * t), -math.sin(OMEGA0 * t))   # Re{c z}: d/dRe + j d/dIm = conj(c)
        for g, one in zip(grads, d):
            g += c * one
    return [L] + grads + [rx[:, 0], rx[:, 1], rx[:, 2], rv[:, 0], rv[:, 1], rv[:, 2]]
