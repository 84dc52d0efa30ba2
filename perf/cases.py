"""Performance cases: the work a user of this package has it do, through its public calls.

A case is one mesh (triangles k = 2..5 or tetrahedra k = 2, 3), a batch of shots on it and one
call sequence over a window of a record:

  forward    Batch.forward: records (and the checkpoints that an adjoint would need)
  segment    Batch.forward_segment twice, as a shot server drives it: all lanes start a shot,
             then every other lane starts another while the rest continue
  gradient   Batch.forward, Batch.adjoint_misfit, Batch.gradient: one gradient of the misfit
  lanes      the same with each shot's own gradient (Batch.gradient_lanes)
  iteration  autograd.misfit and backward: velocity in, misfit and its derivative out, with the
             velocity set anew as in every iteration of an inversion

Meshes are structured grids with their inner vertices moved at random, so that no two elements
are alike; the velocity has water on top, a gradient below it and a fast lens. A mesh stays
resident while cases of other seeds run on it, as in a program that shoots many sources.
Per-DoF results come back as float32, the precision of a model and of the arithmetic behind
them, ordered by position (depth first).

`exact` is the same discretisation in 64 bits in plain torch: mass-lumped elements on their own
nodes, central differences, the damping layer's staggered auxiliaries, the transposed
recurrence, the gradient at every time level.
"""
import math

import numpy as np
import torch

import paper_2108_10946_gb300 as fwi
from paper_2108_10946_gb300 import autograd

DEV = "cuda" if torch.cuda.is_available() else "cpu"
WATER = 1.51          # km/s: no gradient where the velocity is below
H = 0.05              # km, grid spacing
# time step, in units of spacing / largest velocity: about 0.7 of the stability bound
STEP = {(2, 2): 0.090, (2, 3): 0.052, (2, 4): 0.026, (2, 5): 0.0081, (3, 2): 0.058, (3, 3): 0.030}
# multiply-adds of one derivative contraction per element: the node sets do not change under
# permutations of the vertices, so the derivative matrices fall apart into blocks
BLOCKS = {(2, 2): 26, (2, 3): 80, (2, 4): 180, (2, 5): 500, (3, 2): 162, (3, 3): 768}
NODES = {(2, 2): 7, (2, 3): 12, (2, 4): 18, (2, 5): 30, (3, 2): 15, (3, 3): 32}
# barycentric generators and weights (relative to a reference volume 1/dim!) of the node orbits
ORBITS = {
    (2, 2): [((1, 0, 0), 1 / 40), ((.5, .5, 0), 1 / 15), ((1 / 3, 1 / 3, 1 / 3), 9 / 40)],
    (2, 3): [((1, 0, 0), 0.007436456512410179), ((0.7065304440909599, 0.2934695559090401, 0), 0.024420840617025534),
             ((0.5853096486728182, 0.2073451756635909, 0.2073451756635909), 0.1103885289202053)],
    (2, 4): [((1, 0, 0), 0.003174603174602458), ((.5, .5, 0), 0.012698412698415549),
             ((0.7886751345948506, 0.2113248654051494, 0), 0.010714285714285694),
             ((0.7384168123404931, 0.1307915938297535, 0.13079159382975347), 0.05058386489568794),
             ((0.42476396172581077, 0.4247639617258107, 0.15047207654837857), 0.07878121446938935)],
    (2, 5): [((1, 0, 0), 0.0007094239707018946), ((0.6367019258439652, 0.36329807415603477, 0), 0.006190565003665707),
             ((0.8677354183629605, 0.13226458163703947, 0), 0.003480578640561698),
             ((0.8849446311766823, 0.05752768441165886, 0.057527684411658786), 0.01162613545992862),
             ((0.4578368380788056, 0.45783683807880554, 0.08432632384238892), 0.034530430377090596),
             ((0.4862817854748608, 0.25685910726256966, 0.2568591072625696), 0.04590123763022437),
             ((0.700806197612463, 0.2210012187612298, 0.07819258362630721), 0.027278575970133227)],
    (3, 2): [((1, 0, 0, 0), 17 / 5040), ((.5, .5, 0, 0), 32 / 5040), ((1 / 3, 1 / 3, 1 / 3, 0), 81 / 5040),
             ((.25, .25, .25, .25), 256 / 5040)],
    (3, 3): [((1, 0, 0, 0), 0.0006868823600253272), ((0.6857896575819671, 0.3142103424180329, 0, 0), 0.001510781491352611),
             ((0.5690355937288492, 0.21548220313557542, 0.21548220313557542, 0), 0.0050062894680040215),
             ((.5, 1 / 6, 1 / 6, 1 / 6), 0.02142857142857145)],
}


# ---- the cases -------------------------------------------------------------------------------
def _case(name, op, k, grid, shots, steps, rec, layer=False, ckpt=50, store=False):
    nx, ny, nz = (tuple(grid) + (0,))[:3]
    c = dict(op=op, k=k, nx=nx, ny=ny, nz=nz, shots=shots, steps=steps, rec=rec, layer=layer, ckpt=ckpt, store=store)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest gradient anyone asks for: a smoke test's mesh, launches and gaps alone
        _case("tri3_smoke_gradient", "gradient", 3, (10, 10), 4, 100, 5, ckpt=25, store=True),
        # the homogeneous-square validation run: 8,192 triangles, one shot
        _case("tri2_square_forward", "forward", 2, (64, 64), 1, 400, 100),
        # one iteration of a small inversion: its shots as one batch, velocity set anew
        _case("tri3_iteration", "iteration", 3, (151, 97), 8, 120, 51, layer=True),
        # the shot server: a rolling batch advanced by two segments, a gradient batch
        _case("tri4_serve_segment", "segment", 4, (353, 354), 4, 50, 50),
        _case("tri3_serve_lanes", "lanes", 3, (245, 245), 4, 75, 50),
        # one shot per launch: a high-order gradient, and the largest mesh a server keeps
        _case("tri5_one_shot_gradient", "gradient", 5, (157, 159), 1, 75, 50),
        _case("tri2_large_forward", "forward", 2, (1000, 1000), 1, 50, 50),
        # the marine section (a sixth-order element, a damping layer on three sides, 500 receivers)
        _case("tri5_marine_forward", "forward", 5, (790, 220), 4, 50, 500, layer=True),
        _case("tri5_marine_gradient", "gradient", 5, (790, 220), 4, 75, 500, layer=True, store=True),
        # the 3D thrust section with its damping layer
        _case("tet2_thrust_gradient", "gradient", 2, (41, 40, 25), 4, 40, 400, layer=True),
        _case("tet3_thrust_forward", "forward", 3, (41, 40, 25), 4, 25, 400, layer=True),
        _case("tet3_one_shot_gradient", "gradient", 3, (26, 25, 17), 1, 40, 100, layer=True),
    ]


def draw(rng):
    """One more case of the same ranges; a pass costs no more than the largest listed one."""
    most = 0.6 * max(_cost(c) for c in listed())
    while True:
        dim, k = rng.choice([(2, 2), (2, 3), (2, 4), (2, 5), (2, 5), (3, 2), (3, 3)])
        op = rng.choice(["forward", "forward", "gradient", "gradient", "lanes", "segment", "iteration"])
        shots = rng.choice([1, 1, 2, 4, 4, 4, 8, 16])
        cells = math.exp(rng.uniform(math.log(200), math.log(1.2e6 if dim == 2 else 250e3)))
        if dim == 2:
            r = math.exp(rng.uniform(math.log(0.4), math.log(3)))
            nx = max(7, round(math.sqrt(cells / 2 * r)))
            grid = (nx, max(7, round(cells / 2 / nx)))
        else:
            n = (cells / 6) ** (1 / 3)
            grid = tuple(max(4, round(n * f)) for f in (rng.uniform(0.9, 1.3), rng.uniform(0.9, 1.3), rng.uniform(0.6, 1.0)))
        c = _case(None, op, k, grid, shots, rng.randint(20, 130), rng.choice([1, 7, 50, 101, 333]), layer=rng.random() < 0.5,
                  ckpt=rng.choice([10, 25, 50, 50]), store=op == "gradient" and rng.random() < 0.4)
        if _cost(c) <= most:
            return c


def _dim(c):
    return 3 if c["nz"] else 2


def _elements(c):
    return 6 * c["nx"] * c["ny"] * c["nz"] if c["nz"] else 2 * c["nx"] * c["ny"]


def _dofs(c):
    nx, ny, nz, k = c["nx"], c["ny"], c["nz"], c["k"]
    if nz:
        e, v = 6 * nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1)
        f = (4 * e + 4 * (nx * ny + ny * nz + nx * nz)) // 2
        edges = v + f - e - 1  # Euler's formula for a ball
        return v + edges + f + e if k == 2 else v + 2 * edges + 3 * f + 4 * e
    e, v = 2 * nx * ny, (nx + 1) * (ny + 1)
    return v + (v + e - 1) * (k - 1) + e * (NODES[2, k] - 3 * k)


def _cost(c):
    passes = {"forward": 1, "segment": 2, "gradient": 4, "lanes": 4, "iteration": 4}[c["op"]]
    return passes * c["steps"] * c["shots"] * _dofs(c) * (1 if _dim(c) == 2 else 3)


def work(case):
    """Bytes and operations of one pass. A time step reads and writes the wavefield and its
    increment of every shot and reads two coefficients per DoF (state larger than the chip keeps;
    the smallest cases' state could stay on it, and only signals would move). A gradient takes one
    forward and one adjoint sweep, and the forward field once more at every level."""
    c, d, S, n = case, _dim(case), case["shots"], _dofs(case)
    steps = c["steps"] * (2 if c["op"] in ("gradient", "lanes", "iteration", "segment") else 1)
    signals = 4 * S * c["steps"] * (1 + c["rec"]) * (2 if c["op"] != "forward" else 1)
    state = n * (16 * S + 8)
    byts = signals + (state if state < 64e6 else state * steps)
    fl = 2 * BLOCKS[d, c["k"]] * 2 * _elements(c) * S * steps
    if c["op"] in ("gradient", "lanes", "iteration"):
        byts += 0 if state < 64e6 else 4 * n * S * c["steps"]
        byts += 8 * n * (S if c["op"] == "lanes" else 1)
        fl += 2 * BLOCKS[d, c["k"]] * _elements(c) * S * c["steps"]
    return {"bytes": byts, "flops": fl}


# ---- inputs ----------------------------------------------------------------------------------
def _mesh_arrays(c):
    """Vertices and cells: a grid of squares (two triangles each) or boxes (six tetrahedra)."""
    n = [c["nx"], c["ny"]] + ([c["nz"]] if c["nz"] else [])
    d = len(n)
    ax = [np.arange(m + 1) * H for m in n]
    V = np.stack([g.ravel() for g in np.meshgrid(*ax, indexing="ij")], 1)
    move = np.random.RandomState(sum(n)).uniform(-0.1 * H, 0.1 * H, V.shape)
    for a in range(d):
        inner = (V[:, a] > H / 2) & (V[:, a] < n[a] * H - H / 2)
        move[~inner] = 0.0
    V = V + move
    vid = np.arange(V.shape[0]).reshape([m + 1 for m in n])
    if d == 2:
        a, b, e, f = vid[:-1, :-1].ravel(), vid[1:, :-1].ravel(), vid[1:, 1:].ravel(), vid[:-1, 1:].ravel()
        cells = np.concatenate([np.stack([a, b, e], 1), np.stack([a, e, f], 1)])
    else:
        corner = lambda s: vid[s[0]:n[0] + s[0], s[1]:n[1] + s[1], s[2]:n[2] + s[2]].ravel()  # noqa: E731
        cells = []
        for p in ((0, 1, 2), (1, 2, 0), (2, 0, 1), (0, 2, 1), (2, 1, 0), (1, 0, 2)):
            at, path = [0, 0, 0], [corner((0, 0, 0))]
            for axis in p:
                at[axis] = 1
                path.append(corner(at))
            if p in ((0, 2, 1), (2, 1, 0), (1, 0, 2)):  # odd permutation: the other orientation
                path[1], path[2] = path[2], path[1]
            cells.append(np.stack(path, 1))
        cells = np.concatenate(cells)
    return V, cells.astype(np.int32), [m * H for m in n]


def _velocity(x, L, mod=np):
    """km/s at points x: water in the top tenth, a gradient below, a fast lens."""
    z = x[:, -1] / L[-1]
    c = 1.8 + 2.0 * z + 0.1 * mod.sin(5.0 * x[:, 0] / L[0] + 2.0 * z)
    r = ((x[:, 0] / L[0] - 0.55) / 0.2) ** 2 + ((z - 0.6) / 0.12) ** 2
    c = mod.where(r < 1, 4.4 + 0 * c, c)
    return mod.where(z < 0.1, 1.5 + 0 * c, c)


CMAX = 4.5


def _setup(c):
    """Everything about the mesh and the scheme that both sides need."""
    V, cells, L = _mesh_arrays(c)
    d = len(L)
    dt = STEP[d, c["k"]] * H / CMAX
    box, faces, width, smax = None, 0, 0.0, 0.0
    if c["layer"]:  # all sides but the top (the last axis is the depth, positive downward)
        width = H * max(1, round((0.08 if d == 2 else 0.1) * max(c["nx"], c["nz"] or c["ny"])))
        box = [(width, l - width) for l in L[:-1]] + [(-1.0, L[-1] - width)]
        faces = sum(3 << (2 * a) for a in range(d - 1)) | 2 << (2 * d - 2)
        smax = 1.5 * CMAX / width * math.log(1000.0)
    return dict(V=V, cells=cells, L=L, d=d, dt=dt, box=box, faces=faces, width=width, smax=smax)


def _by_depth(x):
    """Order of points x [N][d] by position (last axis first), rounded to a fine lattice."""
    n, d = x.shape
    scale = float(x.abs().max())
    bits = 24 if d == 2 else 20
    q = torch.round(x / scale * 2 ** bits + 0.137).to(torch.int64)
    key = q[:, -1]
    for a in range(d - 1):
        key = key * 2 ** (bits + 1) + q[:, a]
    return torch.argsort(key)


_resident = {}


def _resident_mesh(c):
    key = tuple(sorted((k, c[k]) for k in ("k", "nx", "ny", "nz", "steps", "layer", "ckpt")))
    if key not in _resident:
        _resident.clear()
        s = _setup(c)
        m = fwi.Mesh(s["V"], s["cells"], c["k"], c["steps"], dt=s["dt"], box=s["box"], layer_faces=s["faces"],
                     layer_width=s["width"], sigma_max=s["smax"], absorbing=True, ckpt_stride=c["ckpt"], water_speed=WATER)
        x = m.dof_coords()
        vel = _velocity(x, s["L"])
        m.set_velocity(vel)
        xt = torch.from_numpy(x).to(DEV)
        _resident[key] = dict(mesh=m, L=s["L"], dt=s["dt"], order=_by_depth(xt), x=xt, vel=torch.from_numpy(vel).to(DEV))
    return _resident[key]


def _signals(c, seed, L, dt):
    """Acquisition and signals of a seed: source positions near the top, receivers on a line (3D:
    scattered at one depth), Ricker sources whose two periods fill the window, observed traces."""
    rs = np.random.RandomState(seed % (1 << 31))
    S, R, nt, d = c["shots"], c["rec"], c["steps"], len(L)
    src = np.stack([rs.uniform(0.25, 0.75, S) * L[a] for a in range(d - 1)] + [rs.uniform(0.1, 0.4, S) * L[-1]], 1)
    rec = np.stack([rs.uniform(0.05, 0.95, R) * L[a] for a in range(d - 1)] + [np.full(R, rs.uniform(0.1, 0.4) * L[-1])], 1)
    near = (rs.rand(R) < 0.3) | (np.arange(R) == 0)  # some receivers close to a source, where a window's records are not yet quiet
    rec[near] = np.clip(src[rs.randint(0, S, R)] + rs.uniform(-1.5 * H, 1.5 * H, (R, d)), 0.02 * H, np.array(L) - 0.02 * H)[near]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def ricker(f, t0, n, shape):
        t = torch.arange(n, device=DEV, dtype=torch.float64).reshape(shape) * dt
        a = (math.pi * f * (t - t0)) ** 2
        return (1 - 2 * a) * torch.exp(-a)

    def uniform(lo, hi, *size):
        return lo + (hi - lo) * torch.rand(*size, generator=g, device=DEV, dtype=torch.float64)

    T = nt * dt
    wav = uniform(0.5, 2, S, 1) * ricker(uniform(1.5 / T, 2.5 / T, S, 1), uniform(0.2 * T, 0.5 * T, S, 1), nt, (1, nt))
    obs = uniform(-1, 1, S, 1, R) * ricker(uniform(1.5 / T, 2.5 / T, S, 1, R), uniform(0.2 * T, 0.8 * T, S, 1, R), nt + 1, (1, nt + 1, 1))
    return src, rec, wav.float().contiguous(), obs.float().contiguous()


def _model(vel, x, L, seed):
    """The velocity of one iteration, float32: the mesh's own with a smooth change of a few per cent
    below the water."""
    rs = np.random.RandomState(seed % (1 << 31))
    a, b = rs.uniform(2, 6, 2)
    change = 0.02 * torch.sin(a * x[:, 0] / L[0] + 1.0) * torch.cos(b * x[:, -1] / L[-1])
    return torch.where(vel < WATER, vel, vel * (1 + change)).float()


def prepare(case, seed):
    c = case
    r = _resident_mesh(c)
    mesh = r["mesh"]
    src, rec, wav, obs = _signals(c, seed, r["L"], r["dt"])
    b = fwi.Batch(mesh, src, rec)
    S, R, nt = c["shots"], c["rec"], c["steps"]
    st = dict(op=c["op"], mesh=mesh, batch=b, wav=wav, obs=obs, order=r["order"], nt=nt,
              rec=torch.zeros((S, nt + 1, R), device=DEV))
    if c["store"]:
        b.set_gradient_store(True)
    if c["op"] == "segment":
        st["rec2"] = torch.zeros_like(st["rec"])
        st["all"], st["some"] = (1 << S) - 1, sum(1 << s for s in range(0, S, 2))
    elif c["op"] == "gradient":
        st["grad"] = torch.zeros(mesh.N, dtype=torch.float64, device=DEV)
    elif c["op"] == "lanes":
        b.set_gradient_lanes(True)
        st["grad"] = torch.zeros((S, mesh.N), dtype=torch.float64, device=DEV)
    elif c["op"] == "iteration":
        st["c"] = _model(r["vel"], r["x"], r["L"], seed)
    return st


def run(st):
    b, op = st["batch"], st["op"]
    if op == "segment":
        b.forward_segment(st["nt"], st["all"], st["wav"], st["rec"])
        b.forward_segment(st["nt"], st["some"], st["wav"], st["rec2"])
        return {"records": st["rec"], "records2": st["rec2"]}
    if op == "iteration":
        c = st["c"].clone().requires_grad_(True)
        J = autograd.misfit(c, st["mesh"], b, st["wav"], st["obs"])
        J.backward()
        return {"misfit": J.detach().float(), "gradient": c.grad[st["order"]]}
    b.forward(st["wav"], st["rec"])
    out = {"records": st["rec"]}
    if op != "forward":
        b.adjoint_misfit(st["obs"])
        if op == "gradient":
            out["misfit"] = torch.tensor(b.gradient(st["grad"]), dtype=torch.float32)
            out["gradient"] = st["grad"].float()[st["order"]]
        else:
            out["misfit"] = torch.from_numpy(b.gradient_lanes(st["grad"])).float()
            out["gradient"] = st["grad"].float()[:, st["order"]]
    return out


# ---- the same in 64 bits ---------------------------------------------------------------------
def _monomials(x, e):
    """Values and derivatives [m][M](, [d]) of the monomials with exponents e [M][d] at x [m][d]."""
    p = np.prod(x[:, None, :] ** e[None], axis=2)
    g = []
    for a in range(x.shape[1]):
        ea = e.copy()
        ea[:, a] = np.maximum(ea[:, a] - 1, 0)
        g.append(e[None, :, a] * np.prod(x[:, None, :] ** ea[None], axis=2))
    return p, np.stack(g, 2)


def _space(x, k):
    """Spanning functions of the element's space at reference points x [m][d]: P_k and bubbles
    times polynomials; values [m][M] and derivatives [m][M][d]."""
    m, d = x.shape
    lam = np.concatenate([1 - x.sum(1, keepdims=True), x], 1)
    dlam = np.concatenate([-np.ones((1, d)), np.eye(d)])
    exps = lambda deg: np.array([e for e in np.ndindex(*([deg + 1] * d)) if sum(e) <= deg], dtype=float)  # noqa: E731
    groups = [((), k)]
    if d == 2:
        groups.append(((0, 1, 2), {2: 0, 3: 1, 4: 2, 5: 4}[k]))
    else:
        groups += [(f, k - 2) for f in ((0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3))] + [((0, 1, 2, 3), k - 2)]
    vals, ders = [], []
    for bubble, deg in groups:
        b, db = np.ones(m), np.zeros((m, d))
        for i in bubble:
            db = db * lam[:, i:i + 1] + b[:, None] * dlam[i][None]
            b = b * lam[:, i]
        p, g = _monomials(x, exps(deg))
        vals.append(b[:, None] * p)
        ders.append(db[:, None, :] * p[:, :, None] + b[:, None, None] * g)
    return np.concatenate(vals, 1), np.concatenate(ders, 1)


class _Element:
    def __init__(self, d, k):
        bary, w = [], []
        for gen, wt in ORBITS[d, k]:
            pts = {tuple(gen[i] for i in p) for p in _permutations(d + 1)}
            pts = sorted({tuple(round(v, 14) for v in p): p for p in pts}.values())
            bary += pts
            w += [wt] * len(pts)
        self.bary, self.w = np.array(bary, dtype=float), np.array(w)
        self.n, self.d, self.k = len(w), d, k
        vals, ders = _space(self.bary[:, 1:], k)
        self.coef = np.linalg.pinv(vals, rcond=1e-11)                    # [M][n]
        self.dhat = np.einsum("qmd,mj->dqj", ders, self.coef)
        # facet rules: one weight per orbit of the facet's nodes, exact for the symmetric polynomials
        self.facets = []
        for i in range(d + 1):
            on = np.where(np.abs(self.bary[:, i]) < 1e-12)[0]
            fb = np.delete(self.bary[on], i, axis=1)
            kinds = [tuple(v) for v in np.round(np.sort(fb, 1), 9)]
            keys = sorted(set(kinds))
            rows, rhs = [], []
            for j in range(len(keys)):  # 2D: powers of l0 l1; 3D: 1, e2, e3
                f = (lambda b: (b[:, 0] * b[:, 1]) ** j) if d == 2 else [
                    lambda b: np.ones(len(b)), lambda b: b[:, 0] * b[:, 1] + b[:, 1] * b[:, 2] + b[:, 0] * b[:, 2],
                    lambda b: b[:, 0] * b[:, 1] * b[:, 2]][j]
                rhs.append(math.factorial(j) ** 2 / math.factorial(2 * j + 1) if d == 2 else [1 / 2, 3 / 24, 1 / 120][j])
                v = f(fb)
                rows.append([sum(v[t] for t in range(len(on)) if kinds[t] == q) for q in keys])
            wk = np.linalg.solve(np.array(rows), np.array(rhs))
            self.facets.append((on, np.array([wk[keys.index(q)] for q in kinds])))

    def basis(self, x):
        return _space(x, self.k)[0] @ self.coef


def _permutations(n):
    if n == 1:
        return [(0,)]
    return [p[:i] + (n - 1,) + p[i:] for p in _permutations(n - 1) for i in range(n)]


class _Exact:
    """The scheme in 64 bits on one mesh, DoFs ordered by position."""

    def __init__(self, c):
        s = _setup(c)
        self.c, self.s = c, s
        d, k = s["d"], c["k"]
        el = self.el = _Element(d, k)
        T = lambda a, t=torch.float64: torch.as_tensor(a, dtype=t, device=DEV)  # noqa: E731
        V, cells = T(s["V"]), T(s["cells"], torch.int64)
        E, n = cells.shape[0], el.n
        X = V[cells]
        J = (X[:, 1:] - X[:, :1]).transpose(1, 2)
        self.det, self.Ji = torch.linalg.det(J), torch.linalg.inv(J)
        # DoFs: a node is its vertices (those with a nonzero coordinate) and their coordinates
        vals = sorted(set(np.round(el.bary, 9).ravel()))
        which = np.array([[vals.index(round(float(v), 9)) for v in row] for row in el.bary])
        base = V.shape[0] * 16 + 16
        keys = torch.empty((E, n), dtype=torch.int64, device=DEV)
        inner = 0
        for q in range(n):
            nz = [i for i in range(d + 1) if el.bary[q, i] > 1e-12]
            if len(nz) == d + 1:
                keys[:, q] = -1 - (torch.arange(E, device=DEV) * n + inner)
                inner += 1
                continue
            pairs = torch.stack([cells[:, i] * 16 + int(which[q, i]) + 1 for i in nz], 1).sort(1).values
            key = torch.zeros(E, dtype=torch.int64, device=DEV)
            for i in range(len(nz)):
                key = key * base + pairs[:, i]
            keys[:, q] = key
        uniq, conn = torch.unique(keys, return_inverse=True)
        N = self.N = uniq.numel()
        x = torch.empty((N, d), dtype=torch.float64, device=DEV)
        x[conn.reshape(-1)] = torch.einsum("qv,evd->eqd", T(el.bary), X).reshape(-1, d)
        order = _by_depth(x)
        rank = torch.empty_like(order)
        rank[order] = torch.arange(N, device=DEV)
        self.conn, self.x = rank[conn], x[order]
        self.w, self.dhat = T(el.w), T(el.dhat)
        self.M = self._sum((self.w[None] * self.det[:, None])[:, :, None])[:, 0]
        # damping profile, boundary mass
        sig = torch.zeros_like(self.x)
        if c["layer"]:
            for a, (lo, hi) in enumerate(s["box"]):
                if s["faces"] >> (2 * a) & 1:
                    sig[:, a] += ((lo - self.x[:, a]).clamp(min=0) / s["width"]) ** 2
                if s["faces"] >> (2 * a + 1) & 1:
                    sig[:, a] += ((self.x[:, a] - hi).clamp(min=0) / s["width"]) ** 2
            sig *= s["smax"]
        self.sig = sig
        self.Mb = torch.zeros(N, dtype=torch.float64, device=DEV)
        fk = torch.stack([cells[:, [v for v in range(d + 1) if v != i]].sort(1).values for i in range(d + 1)], 1)
        key = fk[:, :, 0]
        for i in range(1, d):
            key = key * V.shape[0] + fk[:, :, i]
        _, inv, cnt = torch.unique(key, return_inverse=True, return_counts=True)
        for i, (on, fw) in enumerate(el.facets):
            e = torch.where(cnt[inv[:, i]] == 1)[0]
            P = V[fk[e, i]]
            size = (P[:, 1] - P[:, 0]).norm(dim=1) if d == 2 else torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]).norm(dim=1)
            self.Mb.index_add_(0, self.conn[e][:, on].reshape(-1), (size[:, None] * T(fw)[None]).reshape(-1))

    def _sum(self, y):
        out = torch.zeros((self.N, y.shape[2]), dtype=torch.float64, device=DEV)
        return out.index_add_(0, self.conn.reshape(-1), y.reshape(-1, y.shape[2]))

    def grad(self, u):
        """Physical gradient [d] of [E][n][S] at every element's nodes."""
        g = [torch.matmul(self.dhat[r], u[self.conn]) for r in range(self.s["d"])]
        return [sum(self.Ji[:, r, a, None, None] * g[r] for r in range(len(g))) for a in range(len(g))]

    def div(self, f):
        """The transpose: DoF sums of the element vectors f [d] of [E][n][S]."""
        d = len(f)
        return self._sum(sum(torch.matmul(self.dhat[r].T, sum(self.Ji[:, r, a, None, None] * f[a] for a in range(d))) for r in range(d)))

    def set_velocity(self, vel):
        s, dt, d = self.sig, self.s["dt"], self.s["d"]
        self.vel = vel
        tr = s.sum(1)
        m3 = s[:, 0] * s[:, 1] if d == 2 else s[:, 0] * s[:, 1] + s[:, 0] * s[:, 2] + s[:, 1] * s[:, 2]
        a = tr + vel * self.Mb / self.M
        self.den, self.num, self.m3 = (1 + a * dt / 2)[:, None], (1 - a * dt / 2)[:, None], m3[:, None]
        self.det3 = s.prod(1)[:, None] if d == 3 else torch.zeros_like(tr)[:, None]
        self.psi2 = [(2 * s[:, k] - tr)[:, None] for k in range(d)]
        self.psi3 = [torch.stack([s[:, l] for l in range(d) if l != k]).prod(0)[:, None] for k in range(d)]
        self.pd = [(1 + dt * s[:, k] / 2)[:, None] for k in range(d)]
        self.pn = [(1 - dt * s[:, k] / 2)[:, None] for k in range(d)]
        self.wdet = (self.w[None] * self.det[:, None])[:, :, None]
        self.wc2 = self.wdet * (vel * vel)[self.conn][:, :, None]
        self.mask = (tr <= 0) & (vel >= WATER)

    def points(self, p):
        """Element and basis values of points [m][d]."""
        es, phis = [], []
        for q in torch.as_tensor(p, dtype=torch.float64, device=DEV):
            X0 = torch.as_tensor(self.s["V"], device=DEV)[torch.as_tensor(self.s["cells"], dtype=torch.int64, device=DEV)[:, 0]] if not hasattr(self, "X0") else self.X0
            self.X0 = X0
            near = torch.where((X0 - q).abs().max(1).values < 3 * H)[0]
            xh = torch.einsum("erc,ec->er", self.Ji[near], q - X0[near])
            ok = torch.minimum(xh.min(1).values, 1 - xh.sum(1)) >= -1e-12
            j = int(torch.where(ok)[0][0])
            es.append(int(near[j]))
            phis.append(self.el.basis(xh[j].cpu().numpy()[None])[0])
        return self.conn[es], torch.as_tensor(np.array(phis), device=DEV)

    def start(self, S):
        d = self.s["d"]
        z = lambda: torch.zeros((self.N, S), dtype=torch.float64, device=DEV)  # noqa: E731
        return [z(), z(), [z() for _ in range(d)] if self.c["layer"] else None, z() if self.c["layer"] and d == 3 else None]

    def step(self, st, src, w):
        """u, v, P, Y one step on; src: (conn [S][n], phi [S][n]) of the sources, w their samples."""
        u, v, P, Y = st
        d, dt = self.s["d"], self.s["dt"]
        g = self.grad(u)
        f = [self.wc2 * x for x in g]
        if P is not None:
            f = [f[a] + self.wdet * P[a][self.conn] for a in range(d)]
        y = self.div(f)
        for s in range(u.shape[1]):
            y[:, s].index_add_(0, src[0][s], -w[s] * src[1][s])
        vn = (self.num * v - dt * dt * (y / self.M[:, None] + self.m3 * u)) / self.den
        if P is not None:
            c2M = (self.vel ** 2 / self.M)[:, None]
            Pn = [self.pn[k] * P[k] - dt * self.psi2[k] * c2M * self._sum(self.wdet * g[k]) for k in range(d)]
            if d == 3:
                gy = self.grad(Y)
                Pn = [Pn[k] + dt * self.psi3[k] * c2M * self._sum(self.wdet * gy[k]) for k in range(d)]
                vn = vn - dt * dt * self.det3 * Y / self.den
                Y = Y + dt * u
            P = [Pn[k] / self.pd[k] for k in range(d)]
        return [u + vn, vn, P, Y]

    def back(self, st, rec, res):
        """One step of the transposed recurrence, driven by the residual res [S][R]."""
        u, v, P, Y = st
        d, dt = self.s["d"], self.s["dt"]
        g = self.grad(u)
        f = [self.wc2 * x for x in g]
        c2 = (self.vel ** 2)[:, None]
        if P is not None:
            f = [f[a] + self.wdet * (self.psi2[a] * c2 * P[a])[self.conn] for a in range(d)]
        y = self.div(f)
        y.index_add_(0, rec[0].reshape(-1), (rec[1][:, :, None] * res.T[:, None, :]).reshape(-1, u.shape[1]))
        vn = (self.num * v - dt * dt * (y / self.M[:, None] + self.m3 * u)) / self.den
        if P is not None:
            if d == 3:
                vn = vn + dt * dt * Y / self.den
                Y = Y - dt * self.det3 * u + dt / self.M[:, None] * self.div([self.wdet * (self.psi3[a] * c2 * P[a])[self.conn] for a in range(d)])
            P = [(self.pn[k] * P[k] - dt / self.M[:, None] * self._sum(self.wdet * g[k])) / self.pd[k] for k in range(d)]
        return [u + vn, vn, P, Y]

    def sample(self, rec, u):
        return torch.einsum("rn,rns->sr", rec[1], u[rec[0]])

    def forward(self, st, src, rec, wav, keep=False):
        out, fields = [self.sample(rec, st[0])], [st[0]]
        for n in range(wav.shape[1]):
            st = self.step(st, src, wav[:, n].tolist())
            out.append(self.sample(rec, st[0]))
            if keep:
                fields.append(st[0])
        return torch.stack(out, 1), st, fields

    def gradient(self, fields, rec, res):
        """dJ/dc [S][N] before the mass solve."""
        nt, S = res.shape[1] - 1, res.shape[0]
        st = self.start(S)
        g = torch.zeros((self.N, S), dtype=torch.float64, device=DEV)
        wt = 2 * self.wdet * self.vel[self.conn][:, :, None]
        for m in range(nt, 0, -1):
            if m < nt:
                a, b = self.grad(st[0]), self.grad(fields[m])
                g += self._sum(wt * sum(x * y for x, y in zip(a, b)))
            st = self.back(st, rec, res[:, m])
        return torch.where(self.mask[:, None], g, 0 * g).T


def exact(case, seed):
    c = case
    S, nt, d = c["shots"], c["steps"], _dim(c)
    sweeps = {"forward": 1, "segment": 2}.get(c["op"], 3)
    # about 2e11 multiply-adds a second with their memory; the sweeps' fields have to fit, too
    if sweeps * nt * _elements(c) * S * 2 * d * NODES[d, c["k"]] ** 2 > 3e12 or sweeps == 3 and 8.0 * nt * _dofs(c) * S > 60e9:
        return None
    x = _Exact(c)
    src, rec, wav, obs = _signals(c, seed, x.s["L"], x.s["dt"])
    vel = _velocity(x.x, x.s["L"], torch)
    if c["op"] == "iteration":
        vel = _model(vel, x.x, x.s["L"], seed).double()
    x.set_velocity(vel)
    ps, pr = x.points(src), x.points(rec)
    w = wav.double()
    d0, st, fields = x.forward(x.start(S), ps, pr, w, keep=sweeps == 3)
    if c["op"] == "forward":
        return {"records": d0}
    if c["op"] == "segment":
        keep = torch.tensor([0.0 if s % 2 == 0 else 1.0 for s in range(S)], dtype=torch.float64, device=DEV)
        st = [None if t is None else [p * keep for p in t] if isinstance(t, list) else t * keep for t in st]
        return {"records": d0, "records2": x.forward(st, ps, pr, w)[0]}
    res = d0 - obs.double()
    g = x.gradient(fields, pr, res)
    J = 0.5 * (res ** 2).sum((1, 2))
    if c["op"] == "iteration":
        return {"misfit": J.sum(), "gradient": g.sum(0)}
    g = g / x.M
    if c["op"] == "lanes":
        return {"records": d0, "misfit": J, "gradient": g}
    return {"records": d0, "misfit": J.sum(), "gradient": g.sum(0)}
