"""The work a user has this library do, as cases that can be timed and compared.

A gas solver calls the collision step every time step, on gases from a few
thousand particles (a one-dimensional Couette gas) to nine million (the
hypersonic flow), through the direct call, a captured step graph or the
host-memory call; the scattering integral is evaluated in batches (data for
training, tables); the chi-MLP synthesises look-up tables; the neural operator
trains on mini-batches or on the whole harvested set.  Sizes are those of
`paper_2602_21244_gb300.workloads`, `bench.py` and the tests.

`exact` is a plain torch evaluation in 64 bits of the same definitions.
"""
import math

import numpy as np
import torch

from paper_2602_21244_gb300 import dsmc as D
from paper_2602_21244_gb300 import workloads as W

DEV = "cuda"
F64 = torch.float64
CHI_T_LO, CHI_T_HI = math.log(5.0), math.log(6.0e4)
TABLE_NODES = 512
CHI_NODES = 32
SIGMA_V = math.sqrt(2.0 * W.KB * 273.0 / W.M_AR)
PATHS = {"vhs": D.PATH_VHS, "jager": D.PATH_JAGER, "neural": D.PATH_NEURAL, "table": D.PATH_TABLE}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest gas: one-dimensional Couette flow, a step per call
        dict(name="couette_vhs", kind="step", call="step", path="vhs", flow="couette", nx=100, ny=1, mean=50.0,
             order="shuffled"),
        # a small cavity on an odd grid, fed back from its last step (nearly in cell order)
        dict(name="cavity_small_table", kind="step", call="step", path="table", flow="cavity", nx=61, ny=47, mean=20.0,
             order="moved"),
        # the lid-driven cavity's full grid, neural operator, as a captured step graph
        dict(name="cavity_neural_graph", kind="step", call="graph", path="neural", flow="cavity", nx=200, ny=200,
             mean=20.0, order="shuffled"),
        # the hypersonic flow: the neural step that the benchmark quotes (step graph)
        dict(name="hyper_neural_graph", kind="step", call="graph", path="neural", flow="hypersonic", nx=500, ny=300,
             mean=40.0, order="shuffled"),
        # the same flow on the look-up path, the gas as the solver's last step left it
        dict(name="hyper_table", kind="step", call="step", path="table", flow="hypersonic", nx=500, ny=300, mean=40.0,
             order="moved"),
        # the phenomenological kernel on the same flow
        dict(name="hyper_vhs", kind="step", call="step", path="vhs", flow="hypersonic", nx=500, ny=300, mean=40.0,
             order="moved"),
        # the exact scattering integral in the step, a quarter of the flow's area
        dict(name="hyper_half_jager", kind="step", call="step", path="jager", flow="hypersonic", nx=250, ny=150,
             mean=40.0, order="shuffled"),
        # a host solver's arrays in and out (page-locked), neural operator
        dict(name="hyper_half_host", kind="step", call="host", path="neural", flow="hypersonic", nx=250, ny=150,
             mean=40.0, order="moved"),
        # deflection angles for a batch of pairs (harvesting, checks)
        dict(name="chi_batch_4m", kind="chi", n=1 << 22),
        # the chi-MLP's 512 x 512 look-up table
        dict(name="chi_mlp_table_512", kind="chi_mlp", nb=512, nE=512),
        # a training step (forward, backward, Adam) on a mini-batch ...
        dict(name="train_16k", kind="train", n=1 << 14),
        # ... and on the whole harvested set
        dict(name="train_1m", kind="train", n=1 << 20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["chi", "chi_mlp", "train", "train"])
    if kind == "chi":
        return dict(kind="chi", n=_log_int(rng, 1 << 16, 1 << 22))
    if kind == "chi_mlp":
        return dict(kind="chi_mlp", nb=_log_int(rng, 40, 512), nE=_log_int(rng, 40, 512))
    if kind == "train":
        return dict(kind="train", n=16 * _log_int(rng, 1 << 10, 1 << 16))
    path = rng.choice(["vhs", "table", "neural", "jager"])
    call = rng.choice(["step", "graph", "graph", "host"])
    order = rng.choice(["shuffled", "moved"])
    flow = rng.choice(["couette", "cavity", "hypersonic", "hypersonic"])
    if flow == "couette":
        nx, ny, mean = _log_int(rng, 40, 400), 1, float(rng.randint(11, 100))
    elif flow == "cavity":
        nx, ny, mean = _log_int(rng, 23, 240), _log_int(rng, 23, 240), rng.uniform(8.0, 40.0)
    else:
        # the exact integral costs most per pair and the host call moves every array: smaller gases
        s = math.exp(rng.uniform(math.log(0.08), math.log(0.55 if path == "jager" or call == "host" else 1.0)))
        nx, ny, mean = int(round(500 * s)), int(round(300 * s)), 40.0
    return dict(kind="step", call=call, path=path, flow=flow, nx=nx, ny=ny, mean=mean, order=order)


# ------------------------------------------------------------------ inputs
def _rand(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _profile(case):
    """Mean particles, temperature and mean velocity (x, y) of each cell, and the gas of the flow."""
    nx, ny, mean = int(case["nx"]), int(case["ny"]), float(case["mean"])
    nc = nx * ny
    ones = torch.ones(nc, dtype=F64, device=DEV)
    ix = torch.arange(nx, dtype=F64, device=DEV).repeat_interleave(ny)
    iy = torch.arange(ny, dtype=F64, device=DEV).repeat(nx)
    if case["flow"] == "couette":
        lam, T, ux, uy = mean * ones, 273.0 * ones, -100.0 + 200.0 * (ix + 0.5) / nx, 0.0 * ones
        gas = dict(fn_over_vc=1e20 / mean, dt=1e-7)
    elif case["flow"] == "cavity":
        x, y, rmax = ix + 0.5 - 0.5 * nx, iy + 0.5 - 0.5 * ny, math.hypot(0.5 * nx, 0.5 * ny)
        lam, T, ux, uy = mean * ones, 273.0 * ones, -100.0 * y / rmax, 100.0 * x / rmax
        gas = dict(fn_over_vc=1.294e22 / mean, dt=5.3e-8)
    else:
        s = nx / 500.0
        d = torch.hypot(ix + 0.5 - 350.0 * s, iy + 0.5 - 150.0 * s) - 60.0 * s
        shock = 0.5 * (1.0 - torch.tanh((d - 35.0 * s) / (6.0 * s)))
        lam = torch.where(d < 0.0, 0.0 * shock, mean * (1.0 + 5.25 * shock))
        T, ux, uy = 200.0 + 7800.0 * shock, 2634.1 * (1.0 - 0.9 * shock), 0.0 * shock
        gas = dict(fn_over_vc=4.247e20 / mean, dt=1e-7)
    gas.update(mass=W.M_AR, d_ref=4.17e-10, omega=0.81, T_ref=273.0, model=0 if case["path"] == "vhs" else 1,
               b_max=1.2e-9)
    return nc, lam, T, ux, uy, gas


def _particles(case, seed):
    """Maxwellian particles of every cell: in random order, or as a solver feeds them back: in cell
    order with one in ten moved to a neighbouring cell."""
    gen = _rand(seed)
    nc, lam, T, ux, uy, gas = _profile(case)
    # the same number of particles for every seed, so that buffers of one size serve all of them
    counts = lam.round() if case["flow"] == "couette" else torch.poisson(lam, generator=_rand(11))
    cell = torch.arange(nc, device=DEV).repeat_interleave(counts.long())
    n = cell.numel()
    v = torch.randn((3, n), dtype=F64, device=DEV, generator=gen) * torch.sqrt(W.KB * T / W.M_AR)[cell]
    v[0] += ux[cell]
    v[1] += uy[cell]
    if case["order"] == "shuffled":
        p = torch.randperm(n, device=DEV, generator=gen)
        cell, v = cell[p], v[:, p]
    else:
        u = torch.rand(n, device=DEV, generator=gen)
        cell = (cell + (u < 0.05).long() - (u > 0.95).long()).clamp_(0, nc - 1)
    return dict(nc=nc, n=n, T=T, gas=dict(gas, seed=int(seed)), cell=cell.int(), v=v.contiguous())


def _mlp_weights(seed):
    w = W.mlp_weights(seed=int(seed) % 1000003)
    return (torch.from_numpy(w["W_bits"].view(np.int16)).to(DEV),
            torch.randn(3 * 128 + 3, device=DEV, generator=_rand(seed + 7)) * 0.05)


def _mlp():
    return D.make_mlp(8, 128, 3, 3, 0, SIGMA_V, 273.0, 1e-12)


def _capacity(case):
    """Room for the accepted pairs of a step: twice the expected number."""
    return int(2.0 * _pairs_expected(case)) + 4096


def _pairs_expected(case):
    nc, lam, T, _, _, g = _profile(case)
    power = 1.0 if g["model"] == 1 else 2.0 - 2.0 * g["omega"]        # sigma g = scale g^power
    scale = math.pi * g["b_max"] ** 2
    if g["model"] == 0:
        scale = (math.pi * g["d_ref"] ** 2 / math.gamma(2.5 - g["omega"])
                 * (2.0 * W.KB * g["T_ref"] / (0.5 * g["mass"])) ** (g["omega"] - 0.5))
    mean = scale * (4.0 * W.KB * T / g["mass"]) ** (0.5 * power) * math.gamma(1.5 + 0.5 * power) / math.gamma(1.5)
    return float((0.5 * lam * lam * g["fn_over_vc"] * mean * g["dt"]).sum())


def _pair_batch(n, seed):
    """Relative speeds log-uniform in [300, 15000] m/s, impact parameters uniform in b^2 up to 12 A."""
    gen = _rand(seed)
    u = torch.rand((2, n), dtype=F64, device=DEV, generator=gen)
    return (12.0 * torch.sqrt(u[0])).float(), (300.0 * 50.0 ** u[1]).float()


def _harvest(n, seed):
    """Pre-collision pairs to harvest: relative speed log-uniform, isotropic; centre of mass Maxwellian."""
    gen = _rand(seed)
    u = torch.rand((6, n), dtype=F64, device=DEV, generator=gen)
    g, mu, ph, T = 300.0 * 50.0 ** u[0], 2.0 * u[1] - 1.0, 2.0 * math.pi * u[2], 200.0 * 40.0 ** u[3]
    st = torch.sqrt(1.0 - mu * mu)
    vr = g[:, None] * torch.stack([mu, st * torch.cos(ph), st * torch.sin(ph)], 1)
    cm = torch.randn((n, 3), dtype=F64, device=DEV, generator=gen) * torch.sqrt(W.KB * T / (2.0 * W.M_AR))[:, None]
    return dict(vi=cm + 0.5 * vr, vj=cm - 0.5 * vr, T=T, b=12.0 * torch.sqrt(u[4]), eps=2.0 * math.pi * u[5])


def _theta(seed):
    gen = _rand(seed)
    dims = [8, 128, 128, 128, 3]
    parts = []
    for i, o in zip(dims[:-1], dims[1:]):
        a = math.sqrt(6.0 / (i + o))
        parts.append((2.0 * torch.rand(o * i, device=DEV, generator=gen) - 1.0) * a)
    parts += [0.02 * torch.randn(o, device=DEV, generator=gen) for o in dims[1:]]
    return torch.cat(parts)


def _chi_gas():
    return dict(mass=W.M_AR, d_ref=4.17e-10, omega=0.81, T_ref=273.0, fn_over_vc=1.0, dt=1.0, seed=3, model=1,
                b_max=1.2e-9)


# ------------------------------------------------------------------ the calls
_ctx = None


def _context():
    """The program's library context (a captured graph or reserved host buffers have one of their own)."""
    global _ctx
    if _ctx is None:
        _ctx = D.Context(torch.cuda.current_device())
    return _ctx


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, t=0)
    if kind == "chi":
        b, g = _pair_batch(case["n"], seed)
        return dict(s, ctx=_context(), b=b, g=g, gas=D.make_gas(_chi_gas()),
                    pot=D.make_potential(W.JAGER_SYNTHETIC_AR))
    if kind == "chi_mlp":
        ctx, w = _context(), W.chi_mlp_weights(seed=int(seed) % 1000003)
        packed = ctx.chi_mlp_pack(torch.from_numpy(w["W_bits"].view(np.int16)).to(DEV))
        return dict(s, ctx=ctx, packed=packed, bias=torch.from_numpy(w["bias"].astype(np.float32)).to(DEV))
    if kind == "train":
        ctx, h, theta = _context(), _harvest(case["n"], seed), _theta(seed + 5)
        ti, tj = ctx.harvest_jager(D.make_gas(_chi_gas()), D.make_potential(W.JAGER_SYNTHETIC_AR), h["vi"], h["vj"],
                                   h["b"], h["eps"], n_nodes=CHI_NODES)
        nw = 128 * 8 + 2 * 128 * 128 + 3 * 128
        return dict(s, ctx=ctx, mlp=_mlp(), theta=theta, m=torch.zeros_like(theta), v=torch.zeros_like(theta),
                    grad=torch.empty_like(theta), loss=torch.zeros(1, dtype=F64, device=DEV), vi=h["vi"], vj=h["vj"],
                    T=h["T"], ti=ti, tj=tj, ws=ctx.train_workspace(), seed=int(seed),
                    w_bits=torch.empty(nw, dtype=torch.int16, device=DEV),
                    bias=torch.empty(theta.numel() - nw, dtype=torch.float32, device=DEV))
    p = _particles(case, seed)
    gas, call = D.make_gas(p["gas"]), case["call"]
    ctx = _context() if call == "step" else D.Context(torch.cuda.current_device())
    w_bits, bias = _mlp_weights(seed)
    pot = D.make_potential(W.JAGER_SYNTHETIC_AR)
    table = None
    if case["path"] == "table":
        table = ctx.chi_table_build(gas, pot, TABLE_NODES, TABLE_NODES, CHI_T_LO, CHI_T_HI, CHI_NODES)
    path = D.make_path(PATHS[case["path"]], pot=pot, n_nodes=CHI_NODES, mlp=_mlp(), w_bits=w_bits, bias=bias,
                       table=table)
    s.update(ctx=ctx, gas=gas, path=path)
    if call == "host":
        ctx.reserve(p["n"], p["nc"], _capacity(case))
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        s.update(cell=pin(p["cell"]), v=[pin(c) for c in p["v"]], T=pin(p["T"]), perm=pin(p["cell"]),
                 sv=[pin(c) for c in p["v"]])
        return s
    st = D.StepState(ctx, p["n"], p["nc"], _capacity(case))
    st.cell_id.copy_(p["cell"])
    for dst, src in zip((st.vx, st.vy, st.vz), p["v"]):
        dst.copy_(src)
    ctx.sigma_g_max_init(gas, p["T"], 5.0, out=st.sigma_g_max)
    s.update(st=st)
    if call == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        ctx.step_graph_capture(gas, path, st, side)
        torch.cuda.current_stream().wait_stream(side)
    return s


def run(s):
    kind, ctx, t = s["case"]["kind"], s["ctx"], s["t"]
    s["t"] = t + 1
    if kind == "chi":
        return ctx.jager_chi(s["gas"], s["pot"], s["b"], s["g"], n_nodes=CHI_NODES)
    if kind == "chi_mlp":
        return ctx.chi_mlp_table(s["packed"], s["bias"], s["case"]["nb"], s["case"]["nE"])
    if kind == "train":
        ctx.train_step(s["mlp"], s["theta"], s["m"], s["v"], t + 1, 1e-3, s["seed"], s["vi"], s["vj"], s["T"], s["ti"],
                       s["tj"], s["grad"], s["loss"], s["ws"], s["w_bits"], s["bias"])
        return dict(theta=s["theta"], grad=s["grad"], loss=s["loss"], m=s["m"], v=s["v"],
                    w=s["w_bits"].view(torch.bfloat16), bias=s["bias"])
    call = s["case"]["call"]
    if call == "host":
        pairs = ctx.step_host(s["gas"], s["path"], s["cell"], *s["v"], s["T"], t, s["perm"], *s["sv"])
        return dict(perm=s["perm"], vx=s["sv"][0], vy=s["sv"][1], vz=s["sv"][2], pairs=pairs)
    if call == "graph":
        ctx.step_graph_launch(t)
    else:
        ctx.step(s["gas"], s["path"], s["st"], t)
    st = s["st"]
    return dict(perm=st.perm, cell_start=st.cell_start, vx=st.svx, vy=st.svy, vz=st.svz, mom=st.mom,
                sigma_g_max=st.sigma_g_max, info=st.info)


# ------------------------------------------------------------------ what a pass cannot do without
CHI_FLOP = 3000.0           # a root of the radicand and 32 nodes of the integrand
MLP_FLOP = 2.0 * (8 * 128 + 2 * 128 * 128 + 128 * 3)
CHI_MLP_FLOP = 2.0 * (2 * 512 + 2 * 512 * 512 + 512 * 256 + 256 * 128 + 128)


def work(case):
    kind = case["kind"]
    if kind == "chi":
        return dict(bytes=12.0 * case["n"], flops=CHI_FLOP * case["n"])
    if kind == "chi_mlp":
        return dict(bytes=4.0 * case["nb"] * case["nE"] + CHI_MLP_FLOP, flops=CHI_MLP_FLOP * case["nb"] * case["nE"])
    if kind == "train":
        # forward, and the backward's two products per layer; a pair reads two states and two targets
        return dict(bytes=104.0 * case["n"] + 7 * 4 * 34563, flops=3.0 * MLP_FLOP * case["n"])
    nc, lam, _, _, _, _ = _profile(case)
    n, pairs = float(lam.sum()), _pairs_expected(case)
    # cell id and velocity in; permutation and velocity out; per cell its start, moments and (sigma g)_max;
    # every pair reads the four nearest entries of a table that stays on the chip
    per_pair = {"vhs": 100.0, "table": 220.0, "neural": MLP_FLOP + 300.0, "jager": CHI_FLOP + 300.0}[case["path"]]
    return dict(bytes=56.0 * n + 60.0 * nc, flops=pairs * per_pair + 40.0 * n)


# ------------------------------------------------------------------ the same in 64 bits
M32 = 0xFFFFFFFF


def _philox(idx, cell, step, tag, sub, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    c = [idx, cell, torch.full_like(idx, step & M32), torch.full_like(idx, tag | (sub << 8) | ((step >> 32) << 16))]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & M32) ^ c[1] ^ k0, b & M32, ((a >> 32) & M32) ^ c[3] ^ k1, a & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _u53(a, b):
    # bits of (a << 32 | b) >> 11
    return ((a << 21) | (b >> 11)).to(F64) * 2.0 ** -53


def _below(w, n):
    return ((w * n) >> 32) & M32


def _potential(r):
    """V/k_B (K) of the Jager form with Tang-Toennies damping; screened Coulomb core."""
    P = W.JAGER_SYNTHETIC_AR
    x, total, term, damped = P["beta"] * r, torch.ones_like(r), torch.ones_like(r), torch.zeros_like(r)
    e = torch.exp(-x)
    for k in range(1, 17):
        term = term * x / k
        total = total + term
        if k >= 6 and k % 2 == 0:
            damped = damped + P["C"][(k - 6) // 2] / r ** k * (1.0 - e * total)
    rep = P["A"] * torch.exp(P["a1"] * r + P["a2"] * r * r + P["am1"] / r + P["am2"] / (r * r))
    core = P["At"] * torch.exp(-P["at"] * r) / r
    return torch.where(r < 0.4 * P["R_eps"], core, rep - damped)


def _chi(b, E):
    """chi(b, E): the outermost root of the radicand by scanning inwards and bisection, then Gauss-Legendre in
    s, r = r_min / (1 - s^2), on the difference from the free-particle integrand; the panels shrink towards
    s = 0, where the integrand of a nearly orbiting pair is steep."""
    if b.numel() > 1 << 21:
        return torch.cat([_chi(x, e) for x, e in zip(b.split(1 << 21), E.split(1 << 21))])
    F = lambda r: 1.0 - (b / r) ** 2 - _potential(r) / E  # noqa: E731
    hi = torch.clamp(b, min=3.6) * 1.000001
    lo, found = hi.clone(), torch.zeros_like(b, dtype=torch.bool)
    for step in range(900):
        nxt = torch.where(found, lo, lo * 0.995)
        neg = F(nxt) < 0.0
        hi = torch.where(found | neg, hi, nxt)
        lo = nxt
        found = found | neg
        if step % 50 == 49 and bool(found.all()):
            break
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        neg = F(mid) < 0.0
        lo, hi = torch.where(neg, mid, lo), torch.where(neg, hi, mid)
    r0 = hi
    bt, F0 = b / r0, F(r0)
    x, w = np.polynomial.legendre.leggauss(48)
    ends = [0.0, 0.004, 0.02, 0.08, 0.3, 1.0]
    rule = [(a + 0.5 * (e - a) * (xs + 1.0), 0.5 * (e - a) * ws) for a, e in zip(ends[:-1], ends[1:]) for xs, ws in zip(x, w)]
    total = torch.zeros_like(b)
    V0 = _potential(r0)
    for xs, ws in rule:
        s2 = float(xs * xs)
        u = 1.0 - s2
        G0 = bt * bt * s2 * (1.0 + u)
        dG = (_potential(r0 / u) - V0) / E - F0
        G = torch.clamp(G0 - dG, min=1e-30)
        total += float(ws) * 2.0 * float(xs) * dG / (torch.sqrt(G * G0) * (torch.sqrt(G) + torch.sqrt(G0)))
    return torch.where(b > 0.0, -2.0 * bt * total, torch.full_like(b, math.pi))


def _rotate(vr, chi, eps):
    """v_r deflected by chi at azimuth eps (Bird 1994, Eq. 2.22)."""
    x, y, z = vr
    q2, g2 = y * y + z * z, x * x + y * y + z * z
    g, q = torch.sqrt(g2), torch.sqrt(q2)
    flat = ~(q2 > 1e-24 * g2)
    qs, gs = torch.where(flat, torch.ones_like(q), q), torch.where(g2 > 0, g, torch.ones_like(g))
    zero = torch.zeros_like(q)
    c = [zero, torch.where(flat, zero + 1, z / qs), torch.where(flat, zero, -y / qs)]
    a = [torch.where(flat, zero, q / gs), torch.where(flat, zero, -x * y / (gs * qs)),
         torch.where(flat, torch.where(x >= 0, zero - 1, zero + 1), -x * z / (gs * qs))]
    cc, sc, ce, se = torch.cos(chi), torch.sin(chi), torch.cos(eps), torch.sin(eps)
    return [cc * v + g * sc * (ce * ci + se * ai) for v, ci, ai in zip(vr, c, a)]


def _mlp64(x, weights, bias):
    for l, (w, b) in enumerate(zip(weights, bias)):
        x = x @ w.T + b
        if l < len(weights) - 1:
            x = x * torch.sigmoid(x)
    return x


def _layers(flat, bias, dims):
    ws, bs, o, q = [], [], 0, 0
    for i, n in zip(dims[:-1], dims[1:]):
        ws.append(flat[o:o + n * i].reshape(n, i))
        bs.append(bias[q:q + n])
        o, q = o + n * i, q + n
    return ws, bs


def _box_muller(w):
    rho, th = torch.sqrt(-2.0 * torch.log(1.0 - _u53(w[0], w[1]))), 2.0 * math.pi * _u53(w[2], w[3])
    return rho * torch.cos(th), rho * torch.sin(th)


def _cell_moments(cell, v, nc):
    N = torch.zeros(nc, dtype=F64, device=DEV).index_add_(0, cell, torch.ones_like(v[0]))
    S = [torch.zeros(nc, dtype=F64, device=DEV).index_add_(0, cell, c) for c in v]
    u = [s / N.clamp(min=1.0) for s in S]
    theta = torch.zeros(nc, dtype=F64, device=DEV).index_add_(0, cell, sum((c - m[cell]) ** 2 for c, m in zip(v, u)))
    return N, S, u, theta


def _exact_step(case, seed):
    p = _particles(case, seed)
    g, nc, step = p["gas"], p["nc"], 0
    perm = torch.sort(p["cell"], stable=True).indices
    cell = p["cell"][perm].long()
    v = [c[perm].clone() for c in p["v"]]
    counts = torch.bincount(cell, minlength=nc)
    start = torch.zeros(nc + 1, dtype=torch.int64, device=DEV)
    start[1:] = counts.cumsum(0)
    N, S, u_pre, theta = _cell_moments(cell, v, nc)
    mom = torch.stack([N] + S + [theta], 1)

    def sigma_g(gr):
        if g["model"] == 1:
            return math.pi * g["b_max"] ** 2 * gr
        x = 2.0 * W.KB * g["T_ref"] / (0.5 * g["mass"] * gr * gr)
        return math.pi * g["d_ref"] ** 2 * x ** (g["omega"] - 0.5) / math.gamma(2.5 - g["omega"]) * gr

    sg_max = sigma_g(5.0 * torch.sqrt(2.0 * W.KB * p["T"] / g["mass"]))
    # No-Time-Counter candidates
    k = torch.arange(nc, device=DEV)
    w = _philox(torch.zeros_like(k), k, step, 1, 0, g["seed"])
    M = torch.floor(0.5 * N * (N - 1.0) * g["fn_over_vc"] * sg_max * g["dt"] + _u53(w[0], w[1])).long()
    M = torch.where(counts >= 2, M, torch.zeros_like(M))
    ck = k.repeat_interleave(M)
    m = torch.arange(ck.numel(), device=DEV) - (M.cumsum(0) - M)[ck]
    w = _philox(m, ck, step, 2, 0, g["seed"])
    i = _below(w[0], counts[ck])
    j = _below(w[1], counts[ck] - 1)
    j = j + (j >= i).long() + start[ck]
    i = i + start[ck]
    sg = sigma_g(torch.sqrt((v[0][i] - v[0][j]) ** 2 + (v[1][i] - v[1][j]) ** 2 + (v[2][i] - v[2][j]) ** 2))
    acc = _u53(w[2], w[3]) < sg / sg_max[ck]
    sg_max = sg_max.scatter_reduce(0, ck, sg, "amax")
    n_cand = ck.numel()
    i, j, ck, m = i[acc], j[acc], ck[acc], m[acc]
    n_pairs, rounds = i.numel(), 0
    path = case["path"]
    if path == "neural":
        bits, bias = _mlp_weights(seed)
        weights = _layers(bits.view(torch.bfloat16).to(F64), bias.to(F64), [8, 128, 128, 128, 3])
    if path == "table":
        lnE = torch.linspace(CHI_T_LO, CHI_T_HI, TABLE_NODES, dtype=F64, device=DEV)
        bt = torch.linspace(0.0, 1.0, TABLE_NODES, dtype=F64, device=DEV)
        nodes = _chi((12.0 * bt).repeat(TABLE_NODES), torch.exp(lnE).repeat_interleave(TABLE_NODES))
    left = torch.arange(n_pairs, device=DEV)
    while left.numel():
        # the pairs whose particles no earlier pair still needs
        first = torch.full((p["n"],), n_pairs, dtype=torch.int64, device=DEV)
        first.scatter_reduce_(0, i[left], left, "amin").scatter_reduce_(0, j[left], left, "amin")
        ready = (first[i[left]] == left) & (first[j[left]] == left)
        now, left, rounds = left[ready], left[~ready], rounds + 1
        a, b, kk, mm = i[now], j[now], ck[now], m[now]
        vr = [c[a] - c[b] for c in v]
        g2 = vr[0] ** 2 + vr[1] ** 2 + vr[2] ** 2
        gr = torch.sqrt(g2)
        if path == "vhs":
            w = _philox(mm, kk, step, 3, 0, g["seed"])
            c, e = 2.0 * _u53(w[0], w[1]) - 1.0, 2.0 * math.pi * _u53(w[2], w[3])
            sn = torch.sqrt(1.0 - c * c)
            out = [gr * c, gr * sn * torch.cos(e), gr * sn * torch.sin(e)]
        elif path == "neural":
            z = _box_muller(_philox(mm, kk, step, 5, 0, g["seed"])) + _box_muller(_philox(mm, kk, step, 5, 1, g["seed"]))
            T = g["mass"] * theta[kk] / (3.0 * W.KB * N[kk])
            y = _mlp64(torch.stack([c / SIGMA_V for c in vr] + [T / 273.0] + list(z), 1), *weights)
            y = y / torch.sqrt((y * y).sum(1, keepdim=True)) * gr[:, None]
            out = [y[:, 0], y[:, 1], y[:, 2]]
        else:
            w = _philox(mm, kk, step, 4, 0, g["seed"])
            bt, eps, E = torch.sqrt(_u53(w[0], w[1])), 2.0 * math.pi * _u53(w[2], w[3]), g["mass"] * g2 / (4.0 * W.KB)
            if path == "jager":
                chi = _chi(12.0 * bt, E)
            else:
                x = bt * (TABLE_NODES - 1)
                y = ((torch.log(E) - CHI_T_LO) * (TABLE_NODES - 1) / (CHI_T_HI - CHI_T_LO)).clamp(0, TABLE_NODES - 1)
                x0, y0 = x.floor().clamp(max=TABLE_NODES - 2), y.floor().clamp(max=TABLE_NODES - 2)
                at, fx, fy = (y0 * TABLE_NODES + x0).long(), x - x0, y - y0
                chi = ((1 - fy) * ((1 - fx) * nodes[at] + fx * nodes[at + 1])
                       + fy * ((1 - fx) * nodes[at + TABLE_NODES] + fx * nodes[at + TABLE_NODES + 1]))
            out = _rotate(vr, chi, eps)
        for c, o in zip(v, out):
            cm = 0.5 * (c[a] + c[b])
            c[a] = cm + 0.5 * o
            c[b] = cm - 0.5 * o
    _, _, u_post, theta_post = _cell_moments(cell, v, nc)
    alpha = torch.where((N >= 2) & (theta_post > 0), torch.sqrt(theta / theta_post.clamp(min=1e-300)), torch.ones_like(N))
    v = [up[cell] + alpha[cell] * (c - uq[cell]) for c, up, uq in zip(v, u_pre, u_post)]
    out = dict(perm=perm.int(), cell_start=start.int(), vx=v[0], vy=v[1], vz=v[2], mom=mom, sigma_g_max=sg_max,
               info=torch.tensor([n_pairs, n_cand, rounds]))
    if case["call"] == "host":
        return dict(perm=out["perm"], vx=v[0], vy=v[1], vz=v[2], pairs=n_pairs)
    return out


def _exact_train(case, seed):
    h, theta = _harvest(case["n"], seed), _theta(seed + 5)
    n, sv, noise_step = case["n"], SIGMA_V, 1
    target = {}
    vr = h["vi"] - h["vj"]
    E = W.M_AR * (vr * vr).sum(1) / (4.0 * W.KB)
    rot = torch.stack(_rotate([vr[:, 0], vr[:, 1], vr[:, 2]], _chi(h["b"], E), h["eps"]), 1)
    cm = 0.5 * (h["vi"] + h["vj"])
    target["i"], target["j"] = cm + 0.5 * rot, cm - 0.5 * rot
    idx = torch.arange(n, device=DEV)
    zero = torch.zeros_like(idx)
    z = _box_muller(_philox(idx, zero, noise_step, 5, 0, seed)) + _box_muller(_philox(idx, zero, noise_step, 5, 1, seed))
    x = torch.cat([vr / sv, (h["T"] / 273.0)[:, None], torch.stack(z, 1)], 1)
    nw = 128 * 8 + 2 * 128 * 128 + 3 * 128
    # the network runs on the weights rounded to bf16; the gradient is with respect to those
    used = torch.cat([theta[:nw].bfloat16().to(F64), theta[nw:].to(F64)]).requires_grad_(True)
    loss, grad = 0.0, torch.zeros_like(used)
    for part in torch.arange(n // 16, device=DEV).split(1 << 13):
        rows = (part[:, None] * 16 + torch.arange(16, device=DEV)).reshape(-1)
        y = _mlp64(x[rows], *_layers(used[:nw], used[nw:], [8, 128, 128, 128, 3]))
        gr = torch.sqrt((vr[rows] ** 2).sum(1, keepdim=True))
        o = 0.5 * gr * y / torch.sqrt((y * y).sum(1, keepdim=True))
        new = torch.stack([cm[rows] + o, cm[rows] - o], 1).reshape(-1, 32, 3)
        pre = torch.stack([h["vi"][rows], h["vj"][rows]], 1).reshape(-1, 32, 3)
        want = torch.stack([target["i"][rows], target["j"][rows]], 1).reshape(-1, 32, 3)
        u0, u1 = pre.mean(1, keepdim=True), new.mean(1, keepdim=True)
        alpha = torch.sqrt(((pre - u0) ** 2).sum((1, 2), keepdim=True) / ((new - u1) ** 2).sum((1, 2), keepdim=True))
        part_loss = ((u0 + alpha * (new - u1) - want) ** 2).sum() / (2.0 * n * sv * sv)
        grad += torch.autograd.grad(part_loss, used)[0]
        loss = loss + float(part_loss.detach())
    m, v = 0.1 * grad, 0.001 * grad * grad
    new = theta.to(F64) - 1e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return dict(theta=new, grad=grad, loss=torch.tensor([loss], dtype=F64), m=m, v=v, w=new[:nw], bias=new[nw:])


def exact(case, seed):
    kind = case["kind"]
    if kind == "chi":
        b, g = _pair_batch(case["n"], seed)
        return _chi(b.to(F64), W.M_AR * g.to(F64) ** 2 / (4.0 * W.KB))
    if kind == "chi_mlp":
        w = W.chi_mlp_weights(seed=int(seed) % 1000003)
        ws, bs = _layers(torch.from_numpy(w["W"]).to(DEV), torch.from_numpy(w["bias"]).to(DEV), W.CHI_MLP_DIMS)
        nb, nE = case["nb"], case["nE"]
        x = torch.stack([torch.linspace(0, 1, nE, dtype=F64, device=DEV).repeat_interleave(nb),
                         torch.linspace(0, 1, nb, dtype=F64, device=DEV).repeat(nE)], 1)
        y = torch.nn.functional.softplus(_mlp64(x, ws, bs), threshold=1e9)
        return torch.expm1(y).reshape(nE, nb)
    if kind == "train":
        return _exact_train(case, seed)
    return _exact_step(case, seed)
