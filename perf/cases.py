"""What a user of this package has it do, as calls through its public entry points.

Most cases are a short run of the method from a given particle state: the
state is set, its statistics are taken, a number of time steps with their
statistics follow and the state is read back.  The others are the single
stages that such a run adds (statistics of a foreign state, velocity-
conditioned scalar means, the elliptic relaxation, the pressure projection)
and the training gradient of the network that proposes the relaxation's
initial guess.

`exact` restates the same mathematics in 64-bit torch operations (random
numbers, model, particle tracking, statistics, the finite-element systems),
without the package.
"""
import functools
import math

import numpy as np
import torch

import inputs
import paper_1006_0720_gb300 as pg

DT, NU, PI = 1e-3, 1e-3, 2e-3            # the channel runs' time step, viscosity and pressure gradient
STEPS = 7                                # steps of a run: with the first statistics two reorderings of the state
BIG = dict(nx=200, ny=400)               # the benchmark's channel mesh, 158,802 triangles


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the small channel of the method's own runs (1,482 triangles): one step is a
        # row of tiny launches, as in every debugging run and every training-data run
        dict(name="channel_small", kind="run", mesh="channel", nx=20, ny=40, ppe=50, precision="fp64"),
        # an ordinary channel of odd size with uneven particle counts
        dict(name="channel_ragged", kind="run", mesh="channel", nx=61, ny=93, ppe=37, ragged=True, precision="fp64"),
        # the benchmark: 15.9 million particles in FP64-accurate form
        dict(name="channel_big", kind="run", mesh="channel", ppe=100, precision="fp64", **BIG),
        # the FP32-state form on a middle-sized channel
        dict(name="channel_fp32", kind="run", mesh="channel", nx=141, ny=283, ppe=64, precision="fp32"),
        # the complex geometry at full size: 535,720 graded triangles, 68.6 million
        # particles, point source, re-injection
        dict(name="obstacles_fp32", kind="run", mesh="obstacles", h_min=0.0025, ratio=37.0, growth=1.04, ppe=128,
             precision="fp32"),
        # particles that live in the caller's host memory, stepped through the GPU
        dict(name="channel_host", kind="host", nx=100, ny=200, ppe=100),
        # statistics of a state from elsewhere: particles in no order
        dict(name="statistics_foreign", kind="stats", ppe=20, **BIG),
        # velocity-conditioned scalar means (IECM) at the benchmark's density
        dict(name="iecm", kind="iecm", nx=100, ny=200, ppe=100, bins=5),
        # the relaxation solve of the training-data runs, and of the benchmark mesh
        dict(name="relax_small", kind="relax", nx=20, ny=40),
        dict(name="relax_big", kind="relax", **BIG),
        # the pressure projection after a step's statistics
        dict(name="projection", kind="projection", ppe=20, **BIG),
        # one training batch of the relaxation's network
        dict(name="mlp_grad", kind="mlp", batch=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "obstacles", "host", "stats", "iecm", "relax", "projection", "mlp"])
    if kind == "mlp":
        return dict(kind="mlp", batch=_log_int(rng, 256, 65536))
    if kind == "obstacles":
        return dict(kind="run", mesh="obstacles", h_min=math.exp(rng.uniform(math.log(0.004), math.log(0.05))),
                    ratio=rng.uniform(6.0, 30.0), growth=rng.uniform(1.05, 1.3), ppe=_log_int(rng, 20, 128),
                    precision=rng.choice(["fp32", "fp64"]))
    nx = _log_int(rng, 20, 200)
    ny = max(20, min(400, int(nx * rng.uniform(1.4, 2.1))))
    if kind == "relax":
        return dict(kind="relax", nx=nx, ny=ny)
    if kind == "projection":
        return dict(kind="projection", nx=nx, ny=ny, ppe=_log_int(rng, 15, 60))
    if kind == "host":
        return dict(kind="host", nx=min(nx, 120), ny=min(ny, 240), ppe=_log_int(rng, 20, 100))
    if kind == "stats":
        return dict(kind="stats", nx=nx, ny=ny, ppe=_log_int(rng, 10, 100))
    if kind == "iecm":
        return dict(kind="iecm", nx=min(nx, 140), ny=min(ny, 280), ppe=_log_int(rng, 15, 120), bins=rng.choice([3, 4, 5]))
    return dict(kind="run", mesh="channel", nx=nx, ny=ny, ppe=_log_int(rng, 15, 100), ragged=rng.random() < 0.5,
                precision=rng.choice(["fp64", "fp64", "fp32"]))


@functools.lru_cache(maxsize=4)
def _mesh(kind, *sizes):
    if kind == "channel":
        return inputs.channel_mesh(sizes[0], sizes[1])
    return inputs.obstacle_mesh(h_min=sizes[0], ratio=sizes[1], growth=sizes[2])


def _mesh_of(case):
    if case.get("mesh") == "obstacles":
        return _mesh("obstacles", case["h_min"], case["ratio"], case["growth"])
    return _mesh("channel", case["nx"], case["ny"])


def _counts(case):
    """Particles per element; the smallest elements of the graded mesh and the
    sparse ones of an uneven channel keep a least number (as redistribution
    keeps it in long runs), below which the model's turbulent energy vanishes."""
    m = _mesh_of(case)
    if case.get("mesh") == "obstacles":
        return np.maximum(16, inputs.counts_by_area(m, case["ppe"]))
    n_tri = len(m["tri"])
    if case.get("ragged"):
        rng = np.random.default_rng(n_tri)
        return np.maximum(8, rng.poisson(case["ppe"] * rng.uniform(0.3, 1.7, n_tri))).astype(np.int32)
    return np.full(n_tri, case["ppe"], dtype=np.int32)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _state(case, seed, counts):
    """Particles uniform in their elements, Gaussian velocity fluctuations about
    the mean profile, Gamma(4, 1/4) frequencies, a slab of scalar."""
    m, dev = _mesh_of(case), _device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    n = int(counts.sum())

    def rand():
        return torch.rand(n, generator=g, device=dev, dtype=torch.float64)

    def randn():
        return torch.randn(n, generator=g, device=dev, dtype=torch.float64)

    elem = torch.repeat_interleave(torch.arange(len(counts), device=dev), torch.as_tensor(counts, device=dev).long())
    xy = torch.as_tensor(m["xy"], device=dev)
    tri = torch.as_tensor(m["tri"], device=dev).long()
    r1, r2 = (1e-6 + (1.0 - 4e-6) * rand() for _ in range(2))
    over = r1 + r2 > 1.0 - 1e-6
    r1, r2 = torch.where(over, 1.0 - r1, r1), torch.where(over, 1.0 - r2, r2)
    t = tri[elem]
    a = xy[t[:, 0]]
    p = a + r1[:, None] * (xy[t[:, 1]] - a) + r2[:, None] * (xy[t[:, 2]] - a)
    st = dict(x=p[:, 0].contiguous(), y=p[:, 1].contiguous())
    del t, a, p, over, r1, r2
    obstacles = case.get("mesh") == "obstacles"
    st["u"] = (1.0 if obstacles else 1.0 - st["y"] * st["y"]) + 0.1 * randn()
    st["v"], st["w"] = 0.1 * randn(), 0.1 * randn()
    om = torch.log(rand().clamp_min(1e-15))
    for _ in range(3):
        om += torch.log(rand().clamp_min(1e-15))
    st["om"] = om.mul_(-0.25)
    psi = np.zeros(len(counts)) if obstacles else inputs.scalar_slab(m)
    st["ps"] = torch.as_tensor(psi, device=dev)[elem]
    if case["kind"] in ("iecm", "stats"):  # a scalar field that varies inside the elements
        st["ps"] = (0.8 * st["ps"] + 0.2 * rand())
    st["elem"] = elem.int()
    if case["kind"] == "stats":
        order = torch.randperm(n, generator=g, device=dev)
        st = {k: v[order].contiguous() for k, v in st.items()}
    return st


def _node_stats(case, seed):
    """Node statistics [n_nodes, 12] of a channel run: smooth profiles and the
    sampling noise of some hundred particles per node; twins agree."""
    m = _mesh_of(case)
    rng = np.random.default_rng(seed)
    n, y = len(m["xy"]), m["xy"][:, 1]
    S = np.zeros((n, 12))
    noise = rng.normal(size=(n, 12))
    S[:, 0] = 1.0 - y * y + 0.004 * noise[:, 0]
    S[:, 1:3] = 0.004 * noise[:, 1:3]
    S[:, 3] = 1.0 + 0.02 * noise[:, 3]
    S[:, 5:8] = 0.01 * (0.4 + 0.6 * (1.0 - y * y))[:, None] * (1.0 + 0.06 * noise[:, 5:8])
    S[:, 8:11] = 4e-4 * noise[:, 8:11]
    twin = np.asarray(m["twin"])
    later = (twin >= 0) & (twin < np.arange(n))
    S[later] = S[twin[later]]
    return S


def _params(case, **kw):
    if case.get("mesh") == "obstacles":
        return pg.model_params(dt=DT, nu=NU, Pi=2e-2, closure="slm", tm_mode="source", src_x=2.0, src_y=0.5, src_r=0.05)
    return pg.model_params(dt=DT, nu=NU, Pi=PI, closure="glm", **kw)


def _outs(gm):
    def empty(*shape):
        return torch.empty(shape, dtype=torch.float64, device="cuda")
    return dict(elem_stats=empty(gm.n_tri, 13), node_stats=empty(gm.n_nodes, 12), node_derivs=empty(gm.n_nodes, 10))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        X, Y, flat = _mlp_inputs(case, seed)
        net = pg.Mlp(seed)
        net.set_params(flat)
        net.fit_norm(X, Y)
        return dict(kind=kind, net=net, X=X, Y=Y)
    gm = pg.Mesh(_mesh_of(case))
    s = dict(kind=kind, gm=gm, p=_params(case))
    if kind == "relax":
        s["ns"] = torch.as_tensor(_node_stats(case, seed), device="cuda")
        s["wp"] = torch.zeros((9, gm.n_nodes), dtype=torch.float64, device="cuda")
        return s
    counts = _counts(case)
    precision = pg.capi.PDF_FP32_STATE if case.get("precision") == "fp32" else pg.capi.PDF_FP64
    s["gp"] = pg.Particles(gm, seed, count=counts, precision=precision)
    s["init"] = _state(case, seed, counts)
    s["outs"] = _outs(gm)
    if kind == "iecm":
        s["gp"].set_iecm((case["bins"],) * 3, 2)
    if kind == "projection":
        s["p"] = _params(case, pressure="projection")
        s["zero"] = torch.zeros(gm.n_nodes, dtype=torch.float64, device="cuda")
    if kind == "host":
        s["gp"].set_state(s["init"])
        pg.pdf_estimate_stats(s["gp"], gm)
        s["host"] = {k: v.cpu().pin_memory() for k, v in s.pop("init").items()}
        s["step"] = 0
    return s


def run(s):
    kind = s["kind"]
    if kind == "mlp":
        loss, grad = s["net"].grad(s["X"], s["Y"])
        return dict(loss=np.float32(loss), grad=grad)
    gm, p = s["gm"], s["p"]
    if kind == "relax":
        s["wp"].zero_()
        pg.pdf_relax_solve(gm, p, s["ns"], s["wp"], rtol=1e-12, max_it=5000)
        return dict(wp=s["wp"])
    gp, outs = s["gp"], s["outs"]
    if kind == "host":
        # the caller's arrays are stepped in place
        pg.pdf_step_host_stats(gp, gm, p, s["host"], step=s["step"], **outs)
        s["step"] += 1
        return dict(s["host"], **outs)
    gp.set_state(s["init"])
    if kind == "run":
        pg.pdf_estimate_stats(gp, gm)
        for step in range(STEPS):
            pg.pdf_step(gp, gm, p, step=step)
            if step < STEPS - 1:
                pg.pdf_estimate_stats(gp, gm)
        pg.pdf_estimate_stats(gp, gm, **outs)
        return dict(gp.get_state(), **outs)
    pg.pdf_estimate_stats(gp, gm, **outs)
    if kind == "stats":
        return outs
    if kind == "iecm":
        return dict(outs, cond=gp.iecm_cond())
    pg.pdf_pressure_field(gp, gm, set=s["zero"])
    pg.pdf_pressure_project(gp, gm, p, rtol=1e-10, max_it=2000)
    return dict(pressure=pg.pdf_pressure_field(gp, gm), **gp.get_state())


def work(case):
    """Bytes: every particle's state (x, y and elem; u, v, w, omega and psi in the
    form they are stored in) read and written once a step, element and node
    tables once a call, a solve's unknowns once an iteration would need them at
    the least (matrix, vectors).  Flops: the model's arithmetic per particle."""
    kind = case["kind"]
    if kind == "mlp":
        pairs = 11 * 64 + 64 * 64 * 2 + 64 * 9
        return dict(bytes=case["batch"] * 20 * 4 + 9673 * 8, flops=6.0 * pairs * case["batch"])
    m = _mesh_of(case)
    nt, nn = len(m["tri"]), len(m["xy"])
    if kind == "relax":  # statistics in, solution out, one read of the matrices
        return dict(bytes=nn * (12 + 18) * 8 + 7 * nn * 3 * 8, flops=9 * 7 * 2.0 * nn)
    n = int(_counts(case).sum()) if case.get("mesh") == "obstacles" else nt * case["ppe"]
    value = 4 if case.get("precision") == "fp32" else 8
    state, tables = 16 + 4 + 5 * value, nt * 13 * 8 + nn * 22 * 8
    boundary = 60  # the interface's FP64 form
    if kind == "run":
        return dict(bytes=n * (2 * boundary + STEPS * 2 * state + state) + (STEPS + 1) * tables,
                    flops=STEPS * 250.0 * n)
    if kind == "host":
        return dict(bytes=n * 2 * boundary + tables, flops=250.0 * n)
    if kind == "stats":
        return dict(bytes=n * boundary + tables, flops=40.0 * n)
    if kind == "iecm":
        return dict(bytes=n * (boundary + 8) + tables, flops=60.0 * n)
    return dict(bytes=n * (2 * boundary) + tables + nn * 8 * 8, flops=50.0 * n)


def _mlp_inputs(case, seed):
    """Feature and target pairs like those of channel solves (local right-hand
    sides, logarithms of length ratios, smooth corrections) and He weights."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    n = case["batch"]
    X = torch.randn((n, 11), generator=g, device=dev)
    X = X * torch.tensor([0.01] * 9 + [0.8, 0.5], device=dev) + torch.tensor([-0.005] * 9 + [1.5, 2.0], device=dev)
    mix = torch.randn((11, 9), generator=g, device=dev)
    Y = 0.004 * torch.tanh(((X - X.mean(0)) / X.std(0)) @ mix / 3.0) + 0.001 * torch.randn((n, 9), generator=g, device=dev)
    rng = np.random.default_rng(seed)
    sizes = (11, 64, 64, 64, 9)
    flat = np.concatenate([np.concatenate([(rng.normal(size=o * i) * math.sqrt(2.0 / i)).astype(np.float32),
                                           (0.1 * rng.normal(size=o)).astype(np.float32)])
                           for i, o in zip(sizes[:-1], sizes[1:])])
    return X.contiguous(), Y.contiguous(), flat


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "mlp":
        return _mlp_exact(case, seed)
    M = _Mesh64(_mesh_of(case), dev)
    if kind == "relax":
        return dict(wp=_relax_exact(M, torch.as_tensor(_node_stats(case, seed), device=dev)))
    counts = _counts(case)
    st = _state(case, seed, counts)
    es, ns, nd = M.statistics(st)

    def outs():
        return dict(elem_stats=es, node_stats=ns, node_derivs=nd)

    if kind == "stats":
        return outs()
    if kind == "iecm":
        return dict(outs(), cond=_iecm_exact(M, st, case["bins"], 2))
    if kind == "projection":
        P, gx, gy = _projection_exact(M, ns, nd)
        e = st["elem"].long()
        st["u"], st["v"] = st["u"] - DT * gx[e], st["v"] - DT * gy[e]
        return dict(st, pressure=P, elem=None)
    slm = case.get("mesh") == "obstacles"
    for step in range(1 if kind == "host" else STEPS):
        M.step(st, M.rows(ns, nd, slm), seed, step, slm)
        es, ns, nd = M.statistics(st, ns)
    return dict(st, elem=None, **outs())


def _fma(a, b, c):
    """FP32 fused multiply-add (the product is exact in 64 bits)."""
    return (a.double() * (b.double() if torch.is_tensor(b) else b) + (c.double() if torch.is_tensor(c) else c)).float()


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    c = [torch.full_like(c0, v) if not torch.is_tensor(v) else v for v in (c0, c1, c2, c3)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _gauss(w1, w2):
    """Box-Muller in FP32 as the method specifies it: the logarithm by the atanh
    series, sine and cosine by their Taylor series, every operation rounded."""
    f = torch.float32

    def uniform(w):
        return ((w >> 9).to(f) + 0.5) * 2.0 ** -23

    def c32(v):
        return float(np.float32(v))

    m, e = torch.frexp(uniform(w1))
    low = m < c32(0.70710678)
    m, e = torch.where(low, m * 2.0, m), torch.where(low, e - 1, e).to(f)
    s = (m - 1.0) / (m + 1.0)
    z = s * s
    p = _fma(z, c32(1 / 9), c32(1 / 7))
    for c in (1 / 5, 1 / 3, 1.0):
        p = _fma(p, z, c32(c))
    ln = _fma(e, 1420.0 / 2048.0, _fma(e, c32(-2.12194440054690582e-4), (2.0 * s) * p))
    rad = torch.sqrt((-2.0 * ln).double()).float()
    t = 4.0 * uniform(w2)
    q = torch.round(t)
    th = (t - q) * c32(math.pi / 2)
    z = th * th
    ps = _fma(z, c32(1 / 362880), c32(-1 / 5040))
    for c in (1 / 120, -1 / 6, 1.0):
        ps = _fma(ps, z, c32(c))
    s = th * ps
    pc = _fma(z, c32(-1 / 3628800), c32(1 / 40320))
    for c in (-1 / 720, 1 / 24, -0.5, 1.0):
        pc = _fma(pc, z, c32(c))
    q = q.long() & 3
    sn = torch.where(q == 0, s, torch.where(q == 1, pc, torch.where(q == 2, -s, -pc)))
    cs = torch.where(q == 0, pc, torch.where(q == 1, -s, torch.where(q == 2, -pc, s)))
    return (rad * cs).double(), (rad * sn).double()


class _Mesh64:
    """Connectivity, statistics, coefficients and the particle step of a mesh."""

    def __init__(self, m, dev):
        xy, tri, n = m["xy"], m["tri"].astype(np.int64), len(m["xy"])
        twin = np.asarray(m["twin"], dtype=np.int64)
        self.period, self.n, self.nt, self.dev = float(m["period"]), n, len(tri), dev
        # neighbours across the edge opposite local vertex k, by matching edge keys
        a, b = tri[:, [1, 2, 0]], tri[:, [2, 0, 1]]
        key = (np.minimum(a, b) * n + np.maximum(a, b)).ravel()
        order = np.argsort(key, kind="stable")
        same = np.nonzero(key[order][:-1] == key[order][1:])[0]
        nbr = np.full(3 * self.nt, -1, dtype=np.int64)
        i, j = order[same], order[same + 1]
        nbr[i], nbr[j] = j // 3, i // 3
        # boundary edges: walls stay -1, the others join their twins
        tags = {int(min(p, q)) * n + int(max(p, q)): int(t) for p, q, t in m["bnd"]}
        shift, reinj = np.zeros(3 * self.nt), np.zeros(3 * self.nt, dtype=bool)
        open_edges = [f for f in np.nonzero(nbr < 0)[0]]
        at = {int(key[f]): int(f) for f in open_edges}
        walls = []
        for f in open_edges:
            p, q = int(a.ravel()[f]), int(b.ravel()[f])
            tag = tags[int(key[f])]
            if tag == 1:
                walls.append((p, q, f // 3))
                continue
            tp, tq = int(twin[p]), int(twin[q])
            nbr[f] = at[min(tp, tq) * n + max(tp, tq)] // 3
            shift[f] = round((xy[tp, 0] - xy[p, 0]) / self.period)
            reinj[f] = tag == 4
        # elements around each node, ascending, padded with -1
        deg = np.bincount(tri.ravel(), minlength=n)
        esup = np.full((n, deg.max()), -1, dtype=np.int64)
        byn = np.argsort(tri.ravel(), kind="stable")
        first = np.cumsum(deg) - deg
        nodes = tri.ravel()[byn]
        esup[nodes, np.arange(len(byn)) - first[nodes]] = byn // 3
        rep = np.arange(n)
        rep[twin >= 0] = np.minimum(rep[twin >= 0], twin[twin >= 0])

        def put(v):
            return torch.as_tensor(v, device=dev)

        self.xy, self.tri, self.nbr = put(xy), put(tri), put(nbr.reshape(-1, 3))
        self.shift, self.reinj, self.esup, self.rep = put(shift.reshape(-1, 3)), put(reinj.reshape(-1, 3)), put(esup), put(rep)
        P = self.xy[self.tri]
        self.px, self.py = P[:, :, 0].contiguous(), P[:, :, 1].contiguous()
        bx, by = self.px[:, [1, 2, 0]], self.py[:, [1, 2, 0]]
        cx, cy = self.px[:, [2, 0, 1]], self.py[:, [2, 0, 1]]
        self.area = 0.5 * ((self.px[:, 1] - self.px[:, 0]) * (self.py[:, 2] - self.py[:, 0])
                           - (self.py[:, 1] - self.py[:, 0]) * (self.px[:, 2] - self.px[:, 0]))
        self.gx, self.gy = (by - cy) / (2 * self.area)[:, None], (cx - bx) / (2 * self.area)[:, None]
        self.walls = walls

    # ---- statistics and derivatives
    def at_nodes(self, q, w=None, before=None):
        """Mean over the surrounding elements (with w > 0) of element values [nt, k],
        twins merged; a node with none keeps its value from before."""
        w = torch.ones(self.nt, dtype=torch.float64, device=self.dev) if w is None else (w > 0).double()
        s = torch.zeros((self.n, q.shape[1]), dtype=torch.float64, device=self.dev)
        c = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        for k in range(3):
            s.index_add_(0, self.rep[self.tri[:, k]], q * w[:, None])
            c.index_add_(0, self.rep[self.tri[:, k]], w)
        out = (s / c.clamp_min(1.0)[:, None])[self.rep]
        return out if before is None else torch.where((c[self.rep] > 0)[:, None], out, before)

    def gradient(self, q):
        """Element gradients of nodal fields [n, k]: two tensors [nt, k]."""
        v = q[self.tri]
        return (self.gx[:, :, None] * v).sum(1), (self.gy[:, :, None] * v).sum(1)

    def statistics(self, st, before=None):
        e = st["elem"].long()
        N = torch.bincount(e, minlength=self.nt).double()
        D = N.clamp_min(1.0)

        def mean(q):
            return torch.zeros(self.nt, dtype=torch.float64, device=self.dev).index_add_(0, e, q) / D

        names = ("u", "v", "w", "om", "ps")
        mu = [mean(st[k]) for k in names]
        d = {k: st[k] - c[e] for k, c in zip(names, mu)}
        pairs = (("u", "u"), ("v", "v"), ("w", "w"), ("u", "v"), ("u", "w"), ("v", "w"), ("ps", "ps"))
        es = torch.stack([N] + mu + [mean(d[a] * d[b]) for a, b in pairs], 1)
        ns = self.at_nodes(es[:, 1:], N, before)
        return es, ns, self.derivatives(ns)

    def derivatives(self, ns):
        gx, gy = self.gradient(ns[:, [0, 1, 2, 6]])
        g = self.at_nodes(torch.cat([gx, gy], 1))
        hx, hy = self.gradient(g)
        lap = self.at_nodes(hx[:, 0:3] + hy[:, 4:7])
        return torch.stack([g[:, 0], g[:, 4], g[:, 1], g[:, 5], g[:, 2], g[:, 6], lap[:, 0], lap[:, 1], lap[:, 2], g[:, 7]], 1)

    # ---- the model's coefficients, averaged over each element's nodes
    def rows(self, S, D, slm):
        k = (0.5 * (S[:, 5] + S[:, 6] + S[:, 7])).clamp_min(1e-12)
        om = S[:, 3]
        eps = k * om if slm else om * (k + NU * 36.0 * om)
        eg = eps.clamp_min(1e-12)
        zero = torch.zeros_like(k)
        c = [S[:, 0], S[:, 1], S[:, 2]] + [D[:, i] for i in range(6)]
        Pi = 2e-2 if slm else PI
        if slm:
            g = -(0.5 + 0.75 * 3.5) * om
            c += [Pi + zero, D[:, 9], zero] + [g if i % 4 == 0 else zero for i in range(9)]
            c.append(torch.sqrt(3.5 * eps.clamp_min(0.0)))
        else:
            c += [Pi + 2 * NU * D[:, 6], D[:, 9] + 2 * NU * D[:, 7], 2 * NU * D[:, 8]]
            wp = _relax_rhs(S, D, k)
            R = _stresses(S)
            wr = sum(wp[i][j] * R[i][j] for i in range(3) for j in range(3))
            c += [(wp[i][j] - (0.5 * eg if i == j else 0.0)) / k for i in range(3) for j in range(3)]
            c.append(torch.sqrt((-2.0 * wr / (3.0 * k * eg)).clamp_min(0.0) * eg))
        prod = -(S[:, 5] * D[:, 0] + S[:, 8] * D[:, 1] + S[:, 8] * D[:, 2] + S[:, 6] * D[:, 3] + S[:, 9] * D[:, 4]
                 + S[:, 10] * D[:, 5])
        tm = torch.maximum(k / eg, 6.0 * torch.sqrt(NU / eg))
        if slm:
            d = torch.hypot(self.xy[:, 0] - 2.0, self.xy[:, 1] - 0.5)
            uc = torch.sqrt(S[:, 0] ** 2 + S[:, 1] ** 2 + S[:, 2] ** 2).clamp_min(1e-12)
            tm = torch.minimum(tm, 0.02 * (0.05 ** 2 / eg) ** (1.0 / 3.0) + 0.7 * d / uc)
        c += [om, 0.73 - 0.5 * prod / eg, S[:, 4], 1.0 / tm]
        return torch.stack(c, 1)[self.tri].mean(1)

    # ---- one time step in place
    def step(self, st, rows, seed, step, slm):
        e = st["elem"].long()
        pid = torch.arange(len(e), device=self.dev)
        w = _philox(pid, step, 0, 0, seed)
        g = [*_gauss(w[0], w[1]), *_gauss(w[2], w[3])]
        w = _philox(pid, step, 1, 0, seed)
        g += [*_gauss(w[0], w[1])] + [_gauss(w[2], w[3])[0]]
        del w
        sdt, s2nu = math.sqrt(DT), 0.0 if slm else math.sqrt(2 * NU)
        dW = [sdt * v for v in g[:6]]
        U = [st["u"], st["v"], st["w"]]
        x, y = st["x"] + U[0] * DT + s2nu * dW[0], st["y"] + U[1] * DT + s2nu * dW[1]
        c = lambda q: rows[:, q][e]  # noqa: E731
        dU = [U[j] - c(j) for j in range(3)]
        new = []
        for i in range(3):
            drift = sum(c(12 + 3 * i + j) * dU[j] for j in range(3))
            new.append(U[i] + c(9 + i) * DT + s2nu * (c(3 + 2 * i) * dW[0] + c(4 + 2 * i) * dW[1]) + drift * DT
                       + c(21) * dW[2 + i])
        o, mo = st["om"], c(22)
        on = o - 5.0 * mo * (o - mo) * DT - c(23) * mo * o * DT + torch.sqrt(2.5 * mo * mo * o.clamp_min(0.0)) * dW[5]
        ps = st["ps"] - (st["ps"] - c(24)) * DT * c(25)
        x, y, new[0], new[1], e, reinj = self.track(x, y, new[0], new[1], e)
        if slm:
            ps = torch.where(reinj, torch.zeros_like(ps), ps)
            ps = torch.where((x - 2.0) ** 2 + (y - 0.5) ** 2 <= 0.05 ** 2, torch.ones_like(ps), ps)
        st.update(x=x, y=y, u=new[0], v=new[1], w=new[2], om=on.abs(), ps=ps, elem=e.int())

    def subareas(self, e, x, y):
        px, py = self.px[e], self.py[e]
        na = 0.5 * ((px[:, 2] - px[:, 1]) * (y - py[:, 1]) - (py[:, 2] - py[:, 1]) * (x - px[:, 1]))
        nc = 0.5 * ((x - px[:, 1]) * (py[:, 0] - py[:, 1]) - (y - py[:, 1]) * (px[:, 0] - px[:, 1]))
        return torch.stack([na, self.area[e] - na - nc, nc], 1)

    def track(self, x, y, u, v, e):
        """Neighbour walk to the new host element, periodic shifts and wall reflections."""
        reinj = torch.zeros(len(e), dtype=torch.bool, device=self.dev)
        act = torch.arange(len(e), device=self.dev)
        for _ in range(80):
            N = self.subareas(e[act], x[act], y[act])
            out = (N < 0.0).any(1)
            act, N = act[out], N[out]
            if not len(act):
                break
            k = torch.where(N[:, 1] < N[:, 0], 1, 0)
            k = torch.where(N[:, 2] < N.gather(1, k[:, None])[:, 0], 2, k)
            ea = e[act]
            to = self.nbr[ea, k]
            go = to >= 0
            at, ka = act[go], k[go]
            x[at] += self.shift[ea[go], ka] * self.period
            reinj[at] |= self.reinj[ea[go], ka]
            e[at] = to[go]
            at, ka, ea = act[~go], k[~go], ea[~go]
            if not len(at):
                continue
            hit = torch.full_like(at, -1)  # behind a concave corner: the elements around the nodes first
            for j in range(3):
                for i in range(self.esup.shape[1]):
                    f = self.esup[self.tri[ea, j], i]
                    ok = (hit < 0) & (f >= 0) & (self.subareas(f.clamp_min(0), x[at], y[at]) >= 0.0).all(1)
                    hit = torch.where(ok, f, hit)
            e[at] = torch.where(hit >= 0, hit, ea)
            at, ka, ea = at[hit < 0], ka[hit < 0], ea[hit < 0]
            i = torch.arange(len(at), device=self.dev)
            a, b = (ka + 1) % 3, (ka + 2) % 3
            xa, ya = self.px[ea, a], self.py[ea, a]
            tx, ty = self.px[ea, b] - xa, self.py[ea, b] - ya
            ln = torch.sqrt(tx * tx + ty * ty)
            nx, ny = ty / ln, -tx / ln
            d, un = (x[at] - xa) * nx + (y[at] - ya) * ny, u[at] * nx + v[at] * ny
            x[at], y[at] = x[at] - 2 * d * nx, y[at] - 2 * d * ny
            u[at], v[at] = u[at] - 2 * un * nx, v[at] - 2 * un * ny
        return x, y, u, v, e, reinj

    # ---- finite elements over the unknowns (twins merged)
    def wall_frame(self):
        """Per node: the unit outward normal of the nearest wall edge."""
        dist = torch.full((self.n,), math.inf, dtype=torch.float64, device=self.dev)
        nx, ny = torch.zeros_like(dist), torch.zeros_like(dist)
        for side in (-1.0, 1.0):  # the channel's walls y = -1 and y = 1
            d = (self.xy[:, 1] - side).abs()
            near = d < dist
            dist, ny = torch.where(near, d, dist), torch.where(near, torch.full_like(ny, side), ny)
        return dist, nx, ny

    def matrix(self, element):
        """Sparse matrix of the element matrices [nt, 3, 3]."""
        t = self.rep[self.tri]
        i = t[:, :, None].expand(-1, 3, 3).reshape(-1)
        j = t[:, None, :].expand(-1, 3, 3).reshape(-1)
        A = torch.sparse_coo_tensor(torch.stack([i, j]), element.reshape(-1), (self.n, self.n)).coalesce()
        return A.to_sparse_csr()

    def stiffness(self):
        return self.area[:, None, None] * (self.gx[:, :, None] * self.gx[:, None, :] + self.gy[:, :, None] * self.gy[:, None, :])


def _stresses(S):
    return [[S[:, 5], S[:, 8], S[:, 9]], [S[:, 8], S[:, 6], S[:, 10]], [S[:, 9], S[:, 10], S[:, 7]]]


def _relax_rhs(S, D, k):
    R = _stresses(S)
    det = (R[0][0] * (R[1][1] * R[2][2] - R[1][2] * R[2][1]) - R[0][1] * (R[1][0] * R[2][2] - R[1][2] * R[2][0])
           + R[0][2] * (R[1][0] * R[2][1] - R[1][1] * R[2][0]))
    Av = (1.4 * det / (2.0 * k / 3.0) ** 3).clamp_max(1.0)
    b = [[R[i][j] / (2.0 * k) - (1.0 / 3.0 if i == j else 0.0) for j in range(3)] for i in range(3)]
    zero = torch.zeros_like(k)
    G = [[D[:, 2 * i], D[:, 2 * i + 1], zero] for i in range(3)]
    g5 = 0.1
    out = [[None] * 3 for _ in range(3)]
    for i in range(3):
        for j in range(3):
            h = (0.63 * Av + g5 / 3.0) * G[i][j] - g5 / 3.0 * G[j][i]
            h = h + g5 * sum(b[i][q] * (G[q][j] - G[j][q]) for q in range(3))
            out[i][j] = (0.5 * (1.0 - 1.85) * k * S[:, 3] if i == j else 0.0) + k * h
    return out


def _solve(A, b, free, tol=1e-14, limit=6000):
    """Jacobi-preconditioned conjugate gradients in 64 bits; rows outside `free` stay 0."""
    f = free.double()
    crow, col, val = A.crow_indices(), A.col_indices(), A.values()
    rows = torch.repeat_interleave(torch.arange(len(b), device=b.device), crow[1:] - crow[:-1])
    diag = torch.ones_like(b)
    diag[rows[rows == col]] = val[rows == col]
    x, r = torch.zeros_like(b), b * f
    z = r / diag
    p, rz, stop = z.clone(), torch.dot(r, z), tol * torch.linalg.vector_norm(b * f)
    for it in range(limit):
        q = (A @ p) * f
        alpha = rz / torch.dot(p, q)
        x += alpha * p
        r -= alpha * q
        if it % 25 == 0 and not torch.linalg.vector_norm(r) > stop:
            break
        z = r / diag
        rz, old = torch.dot(r, z), rz
        p = z + (rz / old) * p
    return x


def _relax_exact(M, S):
    D = M.derivatives(S)
    k = (0.5 * (S[:, 5] + S[:, 6] + S[:, 7])).clamp_min(1e-12)
    eps = (S[:, 3] * (k + NU * 36.0 * S[:, 3])).clamp_min(1e-12)
    rhs = _relax_rhs(S, D, k)
    dist, nx, ny = M.wall_frame()
    is_rep = M.rep == torch.arange(M.n, device=M.dev)
    mass = M.area[:, None, None] * (1.0 + torch.eye(3, dtype=torch.float64, device=M.dev)) / 12.0
    Mm, K = M.matrix(mass), M.stiffness()
    out = []
    for i in range(3):
        for j in range(3):
            cxi = 1.0 + 1.3 * (nx if i == 0 else ny) ** 2 if i == j and i < 2 else torch.ones_like(k)
            L = 0.134 * torch.maximum(cxi * k ** 1.5 / eps, 72.0 * (NU ** 3 / eps) ** 0.25)
            A = M.matrix(mass + (L * L)[M.tri].mean(1)[:, None, None] * K)
            free = is_rep if i == j else is_rep & (dist > 0.0)
            out.append(_solve(A, Mm @ torch.where(is_rep, rhs[i][j], torch.zeros_like(k)), free)[M.rep])
    return torch.stack(out)


def _projection_exact(M, S, D):
    """The first projection from a zero field: K dP = -d / dt + G."""
    gx, gy = M.gradient(S[:, [0, 1, 5, 6, 8]])
    load = (-(gx[:, 0] + gy[:, 1]) * M.area / 3.0 / DT)
    b = torch.zeros(M.n, dtype=torch.float64, device=M.dev)
    for q in range(3):
        b.index_add_(0, M.rep[M.tri[:, q]], load)
    ends = torch.tensor([(p, q) for p, q, _ in M.walls], device=M.dev)
    e = torch.tensor([int(f) for _, _, f in M.walls], device=M.dev)
    t = M.xy[ends[:, 1]] - M.xy[ends[:, 0]]  # the edge runs counter-clockwise: (t_y, -t_x) points out
    hx = NU * D[ends, 6].mean(1) - (gx[e, 2] + gy[e, 4])
    hy = NU * D[ends, 7].mean(1) - (gx[e, 4] + gy[e, 3])
    h = 0.5 * (hx * t[:, 1] - hy * t[:, 0])
    for q in range(2):
        b.index_add_(0, M.rep[ends[:, q]], h)
    is_rep = M.rep == torch.arange(M.n, device=M.dev)
    b = torch.where(is_rep, b - b.sum() / is_rep.sum(), torch.zeros_like(b))
    x = _solve(M.matrix(M.stiffness()), b, is_rep)
    x = (x - x.sum() / is_rep.sum())[M.rep]
    px, py = M.gradient(x[:, None])
    return x, px[:, 0], py[:, 0]


def _iecm_exact(M, st, nb, m_min):
    """Sort-and-divide binning: by U, then V, then W inside each element."""
    n = len(st["u"])
    group = st["elem"].long()
    order = torch.arange(n, device=M.dev)
    for key in ("u", "v", "w"):
        order = torch.argsort(st[key], stable=True)
        order = order[torch.argsort(group[order], stable=True)]
        g = group[order]
        first = torch.ones(n, dtype=torch.bool, device=M.dev)
        first[1:] = g[1:] != g[:-1]
        run = torch.cumsum(first, 0) - 1
        start = torch.nonzero(first)[:, 0]
        size = torch.diff(start, append=torch.tensor([n], device=M.dev))
        parts = (size // m_min).clamp(1, nb)
        pos = torch.arange(n, device=M.dev) - start[run]
        group = torch.empty_like(group)
        group[order] = run * nb + parts[run] * pos // size[run]
    _, group = torch.unique(group, return_inverse=True)
    cnt = torch.bincount(group).double()
    return (torch.zeros_like(cnt).index_add_(0, group, st["ps"]) / cnt)[group]


def _mlp_exact(case, seed):
    X, Y, flat = _mlp_inputs(case, seed)
    X, Y = X.double(), Y.double()
    X, Y = ((v - v.mean(0)) / v.std(0, unbiased=False) for v in (X, Y))
    p = torch.as_tensor(flat, device=X.device).double().requires_grad_()
    sizes, at, a = (11, 64, 64, 64, 9), 0, X
    for i, o in zip(sizes[:-1], sizes[1:]):
        W, b = p[at:at + o * i].view(o, i), p[at + o * i:at + o * i + o]
        at += o * i + o
        a = a @ W.T + b
        if o != 9:
            a = torch.nn.functional.gelu(a)
    loss = (a - Y).square().mean()
    loss.backward()
    return dict(loss=loss.detach(), grad=p.grad)
