"""The work a user has this library do, through its Python binding and C ABI.

Every case is one control period: measured state and reference in, actuated
control and updated plan out.  Four kinds of caller:

* ``step``: a program that owns one controller and steps it from host arrays
  (``Controller.step`` and ``Controller.get_control``), with the launch shape
  the library chooses;
* ``static``: a program whose state lives in device memory and that may not
  allocate once it runs (``mppi_step_static``);
* ``batch``: a simulator or fleet planner that steps many controllers of mixed
  size together (``Batch.step`` and ``Batch.controls``);
* ``serve``: a server that takes one request from each of its robots and
  waits for all the answers (``Server.submit`` and ``Server.poll``).

The library computes in 32 bits and hands its results over in 64-bit
containers; outputs are returned here in the type they are computed in.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_2504_06437_gb300 import binding
from paper_2504_06437_gb300 import workloads as W

MODELS = {"unicycle": W.UNICYCLE, "quad2d": W.QUAD2D, "ackermann": W.ACKERMANN, "quad5": W.QUAD5}


# --------------------------------------------------------------------- cases
def listed() -> list[dict]:
    def step(name, model, K, T, J, **more):
        return dict(name=name, kind="step", model=model, K=K, T=T, J=J, sgf=0, order=0, res=0.0, **more)

    return [
        # the smallest controller: a small robot that replans at a high rate,
        # where latency is all there is
        step("unicycle_small", "unicycle", 256, 30, 10),
        # the paper's two missions at the sizes it prints (1024 samples, 20
        # steps); the quadrotor smooths its update as Algorithm 1 does
        step("ackermann_mission", "ackermann", 1024, 20, 5),
        dict(step("quad5_smoothed", "quad5", 1024, 20, 3), sgf=11, order=3),
        # the vehicle planning on a grid map made from its point cloud
        dict(step("ackermann_grid", "ackermann", 1024, 20, 0), res=0.1),
        # an ordinary planar quadrotor among 40 obstacles
        step("quad2d", "quad2d", 4096, 50, 40),
        # odd sizes, as a user types them in: nothing divides anything
        step("ackermann_ragged", "ackermann", 9973, 73, 117),
        # a long look ahead with few samples
        step("unicycle_long", "unicycle", 2048, 250, 64),
        # the large single controller: a fast vehicle in a crowded field
        step("unicycle_stress", "unicycle", 65536, 100, 200),
        # the largest robot of the serving mix
        step("quad2d_crowded", "quad2d", 32768, 100, 500),
        # the allocation-free step of a real-time loop on device memory
        dict(name="quad2d_static", kind="static", model="quad2d", K=8192, T=40, J=60, sgf=0, order=0, res=0.0),
        # a fleet stepped together, half unicycles and half quadrotors
        dict(name="batch_mix", kind="batch", n=512),
        # one request from each robot of a served fleet
        dict(name="serving_mix", kind="serve", n=96),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    what = rng.random()
    if what < 0.12:
        return dict(kind="batch", n=_log_uniform(rng, 2, 256))
    if what < 0.2:
        return dict(kind="serve", n=_log_uniform(rng, 4, 96))
    kind = "static" if what < 0.35 else "step"
    model = rng.choice(sorted(MODELS))
    K = _log_uniform(rng, 64, 32768 if kind == "static" else 65536)
    T = _log_uniform(rng, 10, 200 if kind == "step" else 100)
    J = _log_uniform(rng, 3, 500)
    sgf = order = 0
    if rng.random() < 0.25:
        sgf, order = rng.choice([(5, 2), (7, 2), (9, 3)])
    res = 0.0
    if kind == "step" and model == "ackermann" and rng.random() < 0.4:
        J, res = 0, rng.choice([0.1, 0.2])
    return dict(kind=kind, model=model, K=K, T=T, J=J, sgf=sgf, order=order, res=res)


# -------------------------------------------------------------------- inputs
def _world(case, seed) -> W.World:
    """Parameters, obstacles, start, goal and reference speed of one
    controller, in the density and proportions of the presets."""
    m, K, T, J = case["model"], case["K"], case["T"], case["J"]
    if m == "ackermann":
        w = W.ackermann_grid(seed, K=K, T=T, res=case["res"]) if case["res"] else W.ackermann(seed, K=K, T=T, J=J)
    elif m == "quad5":
        w = W.quad5(seed, K=K, T=T, J=J)
    else:
        g = W.rng(seed)
        if m == "unicycle":
            side = 10.0 * math.sqrt(max(J, 10) / 10.0)
            p = W.base_params(W.UNICYCLE, K=K, T=T, dt=0.05, seed=seed)
            start, goal = np.array([1.0, 1.0, math.pi / 4]), np.array([side - 1.0, side - 1.0, math.pi / 4])
            obs = W.obstacle_field(g, J, (0, 0), (side, side), 0.3, 0.8, keep_clear=(start, goal))
        else:
            length = 20.0 * max(1.0, J / 40.0)
            p = W.base_params(W.QUAD2D, K=K, T=T, dt=0.02, seed=seed)
            start, goal = np.zeros(6), np.zeros(6)
            start[:2], goal[:2] = (1.0, 5.0), (length - 1.0, 5.0)
            obs = W.obstacle_field(g, J, (0, 0), (length, 10), 0.2, 0.6, keep_clear=(start, goal))
        p["x_goal"] = goal
        w = W.World(p, obs, start, goal, v_ref=1.0, name=m)
    if case["sgf"]:
        w.params.update(sgf_window=case["sgf"], sgf_order=case["order"])
    return w


def _underway(w: W.World, seed):
    """Measured state, reference and warm-start sequence of a controller in
    mid-run: a little off the start, with a plan from the period before."""
    g = W.rng(seed + 7)
    p, T = w.params, int(w.params["T"])
    x0 = w.x_start + 0.1 * g.uniform(-1.0, 1.0, w.n)
    amp = {W.UNICYCLE: (0.3, 0.3), W.QUAD2D: (0.05, 0.05), W.ACKERMANN: (0.05, 0.3), W.QUAD5: (0.1, 0.05)}[p["model"]]
    t = np.arange(T)[:, None]
    U = np.array(amp) * np.sin(2.0 * math.pi * (t / 40.0 + g.random(2)))
    if p["model"] == W.UNICYCLE:
        U[:, 0] += 0.7
    U = np.clip(U, p["u_min"], p["u_max"])
    return x0, w.reference(x0), U


def _fleet(case, seed):
    worlds = (W.batch_mix if case["kind"] == "batch" else W.serving_mix)(case["n"], seed=seed)
    return worlds, [_underway(w, seed + 13 * i) for i, w in enumerate(worlds)]


class _Static:
    """A real-time program's device memory: inputs, state and outputs."""

    def __init__(self, w, x0, xref, U):
        p, dev = w.params, torch.device("cuda")
        f64 = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.params = binding.make_params(p)
        self.K, self.T, self.J = int(p["K"]), int(p["T"]), len(w.obstacles)
        self.inputs = [f64(w.obstacles), f64(x0), f64(xref)]
        ctl = np.array([p["mu_coarse"], 0.0, 1.0, 0.0, 0.0])
        # the sequence, the controller's state, the control and the costs
        # in one block that the program takes over as a whole
        self.sizes = [2 * self.T, 5, 2, self.K]
        self.block = f64(np.concatenate([U.ravel(), ctl, np.zeros(2), np.zeros(self.K)]))
        U_, ctl_, u0_, costs_ = torch.split(self.block, self.sizes)
        ptr = lambda a: C.c_void_p(a.data_ptr())  # noqa: E731
        ob, x, xr = self.inputs
        self.args = (C.byref(self.params), ptr(ob), C.c_int32(self.J), ptr(x), ptr(xr), ptr(U_), ptr(ctl_), ptr(u0_),
                     ptr(costs_))
        self.step = binding.load().mppi_step_static

    def run(self):
        rc = self.step(*self.args, C.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != binding.MPPI_OK:
            raise binding.MppiError(rc, binding.load().mppi_last_error().decode())
        return torch.split(self.block.float(), self.sizes)


def prepare(case, seed):
    if case["kind"] == "batch":
        worlds, now = _fleet(case, seed)
        b = binding.Batch(len(worlds), (64 << 20) + len(worlds) * (1 << 20))
        slots = [b.add(w.params, w.obstacles, u_init=U) for w, (_, _, U) in zip(worlds, now)]
        return dict(kind="batch", b=b, slots=slots, x0s=[x for x, _, _ in now], xrefs=[r for _, r, _ in now])
    if case["kind"] == "serve":
        worlds, now = _fleet(case, seed)
        s = binding.Server(len(worlds), (64 << 20) + len(worlds) * (2 << 20), lanes=4)
        # small requests apart from the large, least work first, served by
        # the resident kernel
        s.set_policy(small_ops_max=2e9, small_lanes=3, large_share=0.75, batch_ops_small=4e9, batch_ops_large=5e10,
                     shortest_first=True, max_wait_s=0.05, device_queue=True)
        robots = [s.join(w.params, w.obstacles, u_init=U) for w, (_, _, U) in zip(worlds, now)]
        return dict(kind="serve", s=s, robots=robots, x0s=[x for x, _, _ in now], xrefs=[r for _, r, _ in now])
    w = _world(case, seed)
    x0, xref, U = _underway(w, seed)
    if case["kind"] == "static":
        return dict(kind="static", s=_Static(w, x0, xref, U))
    c = binding.Controller(w.params, u_init=U)
    c.set_obstacles(w.obstacles)
    if case["res"]:
        p = w.params
        c.set_grid(p["grid"], p["grid_ox"], p["grid_oy"], p["grid_res"])
    return dict(kind="step", c=c, x0=x0, xref=xref)


# ---------------------------------------------------------------------- pass
def run(state):
    kind = state["kind"]
    if kind == "step":
        c = state["c"]
        c.step(state["x0"], state["xref"])
        u0, U = c.get_control(want_U=True)
        return dict(u0=u0.astype(np.float32), U=U.astype(np.float32))
    if kind == "static":
        U, ctl, u0, costs = state["s"].run()
        return dict(u0=u0, U=U, ctl=ctl, costs=costs)
    if kind == "batch":
        b = state["b"]
        b.step(state["slots"], state["x0s"], state["xrefs"])
        return dict(u0=b.controls().astype(np.float32))
    s, robots = state["s"], state["robots"]
    for r, x0, xref in zip(robots, state["x0s"], state["xrefs"]):
        s.submit(r, x0, xref)
    got = {}
    while len(got) < len(robots):
        for r, u0, x1, _, status in s.poll():
            if status != binding.MPPI_OK:
                raise RuntimeError(f"robot {r}: request failed ({status})")
            got[r] = (u0, x1)
    return dict(u0=np.array([got[r][0] for r in robots], dtype=np.float32),
                x1=np.array([got[r][1] for r in robots], dtype=np.float32))


def _work_one(K, T, J, P, n, grid_points, costs):
    """Bytes in and out and FP32 operations of one step: 7 for a pair of
    shape point and obstacle, 24 for a grid lookup, 135 for a step of a sample
    (draws, dynamics, costs), as the benchmark counts them."""
    flops = K * T * (7.0 * P * J + (24.0 * P if grid_points else 0.0) + 135.0)
    data = 8.0 * n * (T + 2) + 24.0 * J + 2 * 16.0 * T + 16.0 + (8.0 * K if costs else 0.0)
    return data + min(4.0 * grid_points, 16.0 * K * T * P), flops


def work(case) -> dict:
    if case["kind"] in ("batch", "serve"):
        # the mix's mean robot: K log-uniform, T and J uniform, half
        # unicycles (P 1, n 3) and half quadrotors (P 7, n 6)
        K0, K1, T, J = (1024, 16384, 50, 152.5) if case["kind"] == "batch" else (512, 32768, 60, 252.5)
        K = (K1 - K0) / math.log(K1 / K0)
        each = [_work_one(K, T, J, P, n, 0, False) for P, n in ((1, 3), (7, 6))]
        return dict(bytes=case["n"] * sum(e[0] for e in each) / 2, flops=case["n"] * sum(e[1] for e in each) / 2)
    m = MODELS[case["model"]]
    P = {W.UNICYCLE: 1, W.ACKERMANN: 8}.get(m, 7)
    grid = round(100.0 / case["res"] + 1) * round(30.0 / case["res"] + 1) if case["res"] else 0
    b, f = _work_one(case["K"], case["T"], case["J"], P, W.state_dim(m), grid, case["kind"] == "static")
    return dict(bytes=b, flops=f)


# ---------------------------------------------- the same step in 64 bits
def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    mask = 0xFFFFFFFF
    k0, k1 = key & mask, key >> 32

    def mul(a, b):  # high and low words of a 32 x 32 bit product
        p, q = (a >> 16) * b, (a & 0xFFFF) * b
        return (p + (q >> 16)) >> 16, ((p << 16) + q) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _draws(p, S_e, ks, T, dev):
    """Perturbations of samples ks, first iteration: len(ks) x T x 2."""
    k = ks.view(-1, 1).expand(-1, T)
    t = torch.arange(T, device=dev).view(1, -1).expand(len(ks), -1)
    zero = torch.zeros_like(k)
    u = [((r >> 8) | 1).double() * 2.0 ** -24 for r in _philox(k, t, zero, zero, int(p["seed"]))]
    ra, rb = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    za = [ra * torch.cos(2 * math.pi * u[1]), ra * torch.sin(2 * math.pi * u[1])]
    zb = [rb * torch.cos(2 * math.pi * u[3]), rb * torch.sin(2 * math.pi * u[3])]
    L = np.linalg.cholesky(S_e * np.asarray(p["sigma"]).reshape(2, 2))
    n = [L[0, 0] * za[0], L[1, 0] * za[0] + L[1, 1] * za[1]]
    return torch.stack([n[d] * torch.exp(p["ln_mu"] + p["ln_sigma"] * zb[d]) for d in (0, 1)], dim=-1)


def _rollout(p, x0, V):
    """States x_1..x_T of each sequence in V (k x T x 2): k x T x n."""
    m, dt, g = p["model"], p["dt"], p["gravity"]
    x = [torch.full_like(V[:, 0, 0], float(a)) for a in x0]
    out = []
    for t in range(V.shape[1]):
        a, b = V[:, t, 0], V[:, t, 1]
        c, s = torch.cos(x[2]), torch.sin(x[2])
        if m == W.UNICYCLE:
            d = [a * c, a * s, b]
        elif m == W.ACKERMANN:
            d = [x[3] * c, x[3] * s, x[3] * torch.tan(a) / p["wheelbase"], b]
        elif m == W.QUAD5:
            acc = g + b / p["mass"]
            d = [x[3], x[4], a, -acc * s, acc * c - g]
        else:
            acc = g + (a + b) / p["mass"]
            d = [x[3], x[4], x[5], -acc * s, acc * c - g, (b - a) * p["arm"] / p["inertia"]]
        x = [xi + di * dt for xi, di in zip(x, d)]
        out.append(torch.stack(x, dim=-1))
    return torch.stack(out, dim=1)


def _grid_h(p, grid, X, Y):
    ny, nx = grid.shape
    u = ((X - p["grid_ox"]) / p["grid_res"]).clamp(0, nx - 1)
    v = ((Y - p["grid_oy"]) / p["grid_res"]).clamp(0, ny - 1)
    i, j = u.floor().long().clamp(max=nx - 2), v.floor().long().clamp(max=ny - 2)
    fx, fy = u - i, v - j
    a = (1 - fx) * grid[j, i] + fx * grid[j, i + 1]
    b = (1 - fx) * grid[j + 1, i] + fx * grid[j + 1, i + 1]
    return (1 - fy) * a + fy * b


def _barrier(p, obs, grid, states):
    """Fused barrier and smallest h at each pose of states (... x n)."""
    sh = torch.as_tensor(np.asarray(p["shape"], dtype=np.float64).reshape(-1, 2), device=states.device)
    flat = states.reshape(-1, states.shape[-1])
    B, mn = [], []
    step = max(1, 40_000_000 // max(1, len(sh) * max(1, len(obs))))
    for part in flat.split(step):
        c, s = torch.cos(part[:, 2:3]), torch.sin(part[:, 2:3])
        X = part[:, 0:1] + c * sh[:, 0] - s * sh[:, 1]
        Y = part[:, 1:2] + s * sh[:, 0] + c * sh[:, 1]
        h = X.new_full((len(part), 0), 0.0)
        if len(obs):
            h = ((X[..., None] - obs[:, 0]) ** 2 + (Y[..., None] - obs[:, 1]) ** 2 - obs[:, 2] ** 2).flatten(1)
        if grid is not None:
            h = torch.cat([h, _grid_h(p, grid, X, Y)], dim=1)
        if h.shape[1] == 0:
            h = torch.full((len(part), 1), math.inf, dtype=torch.float64, device=X.device)
        B.append((1.0 / h.clamp(min=p["h_eps"])).sum(1))
        mn.append(h.amin(1))
    return torch.cat(B).view(states.shape[:-1]), torch.cat(mn).view(states.shape[:-1])


def _smooth(y, Wn, order):
    """Least-squares polynomial smoothing of the columns of y (T x 2)."""
    T = len(y)
    A = np.vander(np.linspace(-1.0, 1.0, Wn), order + 1)
    H = A @ np.linalg.pinv(A)
    out = np.empty_like(y)
    for t in range(T):
        s = min(max(t - Wn // 2, 0), T - Wn)
        out[t] = H[t - s] @ y[s:s + Wn]
    return out


def _step64(w, x0, xref, U):
    """First step of a controller: u0, shifted sequence, costs, and the
    state (S_e, beta) it goes on with; and the state after u0."""
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    p = w.params
    f64 = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=dev)  # noqa: E731
    K, T, gam, S_e = int(p["K"]), int(p["T"]), p["gamma_bas"], p["mu_coarse"]
    obs = f64(w.obstacles).view(-1, 3)
    grid = f64(p["grid"]) if "grid" in p else None
    Ut, ref = f64(U), f64(xref)
    lo, hi, Q, Qf = f64(p["u_min"]), f64(p["u_max"]), f64(p["Q"])[:w.n], f64(p["Qf"])[:w.n]
    A = p["gamma_ctrl"] * torch.linalg.inv(S_e * f64(p["sigma"]).view(2, 2))
    beta = float(_barrier(p, obs, grid, f64(x0).view(1, -1))[0][0])
    beta_d = float(_barrier(p, obs, grid, f64(p["x_goal"]).view(1, -1))[0][0])

    def bas(B):  # sum over t of the barrier state along each rollout
        s, total = torch.full_like(B[:, 0], beta), torch.zeros_like(B[:, 0])
        for t in range(T):
            s = B[:, t] + gam * (s - beta_d)
            total = total + s
        return p["R_B"] * total

    costs, V = [], []
    for ks in torch.arange(K, device=dev).split(max(1, 4_000_000 // T)):
        v = torch.minimum(torch.maximum(Ut + _draws(p, S_e, ks, T, dev), lo), hi)
        X = _rollout(p, x0, v)
        B, mn = _barrier(p, obs, grid, X)
        S = (Q * (X - ref[1:]) ** 2).sum((1, 2)) + (Qf * (X[:, -1] - ref[-1]) ** 2).sum(1)
        S = S + ((v @ A.T) * Ut).sum((1, 2)) + bas(B) + p["C_coll"] * (mn <= 0).sum(1)
        costs.append(S)
        V.append(v)
    S, V = torch.cat(costs), torch.cat(V)
    e = torch.exp(-(S - S.min()) / p["lambda"])
    dU = (torch.einsum("k,ktd->td", e, V - Ut) / e.sum()).cpu().numpy()
    if p.get("sgf_window", 0):
        dU = _smooth(dU, p["sgf_window"], p["sgf_order"])
    Us = np.clip(U + dU, p["u_min"], p["u_max"])
    X = _rollout(p, x0, f64(Us)[None])
    CB = float(bas(_barrier(p, obs, grid, X)[0])[0])
    x1 = np.zeros(6)
    x1[:w.n] = X[0, 0].cpu().numpy()
    return dict(u0=Us[0], U=np.concatenate([Us[1:], Us[-1:]]), costs=S.cpu().numpy(), x1=x1,
                S_e=p["mu_coarse"] * math.log(math.e + max(CB, 0.0)), beta=beta)


def exact(case, seed):
    if case["kind"] in ("batch", "serve"):
        got = [_step64(w, *now) for w, now in zip(*_fleet(case, seed))]
        out = dict(u0=np.array([g["u0"] for g in got]))
        if case["kind"] == "serve":
            out["x1"] = np.array([g["x1"] for g in got])
        return out
    w = _world(case, seed)
    g = _step64(w, *_underway(w, seed))
    if case["kind"] == "static":
        return dict(u0=g["u0"], U=g["U"].ravel(), ctl=np.array([g["S_e"], g["beta"], 0.0, 1.0, 0.0]), costs=g["costs"])
    return dict(u0=g["u0"], U=g["U"])
