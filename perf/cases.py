"""Timed cases of the CRKSPH neighbor-sum path.

Each case is one call chain a program makes through the public entry points of
``paper_2511_21921_gb300.solver``, on seeded gas generated on the device.  The
shapes follow the workloads of ``synth.py`` (jittered lattice, lognormal boxes
of variance 1.5 and 3, many boxes of uneven size; about 100 neighbors within
h), the sizes go from 16^3 to 256^3 particles.
"""
import math

import torch

from paper_2511_21921_gb300.solver import Solver, rates

N_H = (300.0 / (4.0 * math.pi)) ** (1.0 / 3.0)  # h of about 100 neighbors: N_H V^(1/3)
LAMBDA = 0.2                                    # relaxation of h per step
KDK_DT = 1e-8                                   # short: thousands of steps keep this gas what it is
COOL = dict(nodes=1251, log10_min=-2.5, dex=0.004, A=0.6, dt=0.05)

# The tuned cases time every launch variant once per size and process and
# replay the choice on later plans, as a program with a stored choice does.
_tuned = {}


def listed():
    return [
        # a differentiable small box: one gradient step of a fit, dominated by launches
        dict(name="grad_lattice_4k", kind="grad", n=4096, shape="lattice", L=1.0),
        # forward rates of a modest box of odd size, with the density asked for as well
        dict(name="forward_30k", kind="forward", n=30011, shape="lognormal", var=1.5, L=1.0),
        # rates and their gradient in one call, cotangents known in advance
        dict(name="fused_50k", kind="fused", n=50021, shape="lognormal", var=1.5, L=1.0),
        # the FP64 form: a reference gradient on a small box
        dict(name="grad_fp64_14k", kind="grad", n=13824, shape="lognormal", var=1.5, L=1.0,
             fp64=True),
        # gradient of an ordinary box: unequal masses, a side that is no power of two
        dict(name="grad_masses_100k", kind="grad", n=100003, shape="lognormal", var=1.5, L=2.5,
             masses=True),
        # the benchmark's small box: whole step, tuned, replayed from a CUDA graph
        dict(name="step_graph_262k", kind="step", n=262144, shape="lognormal", var=1.5, L=1.0,
             tuned=True, graph=True),
        # one kick-drift-kick hydro step, as a simulation loop calls it
        dict(name="kdk_262k", kind="kdk", n=262144, shape="lognormal", var=1.5, L=1.0),
        # a sub-step of a time-bin hierarchy: a quarter of the particles active
        dict(name="active_262k", kind="active", n=262144, shape="lognormal", var=1.5, L=1.0,
             fraction=0.25),
        # stars and black holes over the gas, and radiative cooling of the gas
        dict(name="subgrid_cool_262k", kind="subgrid", n=262144, shape="lognormal", var=1.5,
             L=1.0, n_s=13107),
        # many independent boxes of uneven size in one call, with gradients
        dict(name="grad_boxes_24", kind="grad", n=0, shape="boxes", boxes=24, side_max=72,
             var=1.5, L=1.0),
        # forward rates of a large, strongly clustered box
        dict(name="forward_clustered_2m", kind="forward", n=2097152, shape="lognormal", var=3.0,
             L=1.0),
        # the largest box: whole step, tuned
        dict(name="step_17m", kind="step", n=16777216, shape="lognormal", var=1.5, L=1.0,
             tuned=True),
    ]


def draw(rng):
    kind = rng.choice(["grad", "grad", "forward", "forward", "fused", "step", "kdk", "active",
                       "subgrid"])
    top = {"grad": 2.0e6, "forward": 4.0e6, "fused": 2.0e6, "step": 4.0e6, "kdk": 1.0e6,
           "active": 1.0e6, "subgrid": 5.0e5}[kind]
    c = dict(kind=kind, shape="lognormal", var=rng.choice([0.5, 1.5, 3.0]),
             L=rng.choice([1.0, 1.0, 2.5, 0.7]))
    if kind in ("grad", "forward") and rng.random() < 0.2:
        c.update(shape="boxes", boxes=rng.randint(2, 32), side_max=rng.randint(16, 64), n=0)
        return c
    if kind in ("grad", "fused") and rng.random() < 0.2:
        c["fp64"] = True
        top = 2.0e4
    low = 2500.0
    if kind == "kdk":  # its h follows the volume: below half a side in the emptiest region
        low, c["var"] = 40000.0, min(c["var"], 1.5)
    c["n"] = int(math.exp(rng.uniform(math.log(low), math.log(top)))) | 1
    c["masses"] = rng.random() < 0.3 and kind != "kdk"
    if kind == "step":
        c["graph"] = rng.random() < 0.5
        c["tuned"] = rng.random() < 0.5
    if kind == "active":
        c["fraction"] = round(rng.uniform(0.05, 0.6), 3)
    if kind == "subgrid":
        c["n_s"] = max(64, int(c["n"] * rng.uniform(0.01, 0.1)))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sides(case):
    """Side of every box: uneven, log-uniform from 8 up, fixed by the case."""
    import random
    r = random.Random(99 + case["boxes"])
    return [int(round(math.exp(r.uniform(math.log(8), math.log(case["side_max"])))))
            for _ in range(case["boxes"])]


def _field(g, ng, var):
    """Lognormal density on an ng^3 grid, P(k) ~ k^-2."""
    k = torch.fft.fftfreq(ng, device="cuda") * ng
    kz = torch.fft.rfftfreq(ng, device="cuda") * ng
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2.clamp_min(1.0) ** -0.5, torch.zeros_like(k2))
    d = torch.fft.irfftn(torch.fft.rfftn(torch.randn((ng,) * 3, generator=g, device="cuda")) * amp,
                         s=(ng,) * 3)
    d = d * (math.sqrt(var) / d.std())
    return torch.exp(d - 0.5 * var)


def _reach(g, x, L, lo, hi):
    """h with about U(lo, hi) particles within it: where the count in spheres
    (the particle counts on a grid, smoothed with top hats of growing radius)
    crosses the target."""
    n = x.shape[1]
    ng = min(512, 2 * max(8, round(n ** (1 / 3))))
    cell = L / ng
    q = (x / cell).long().clamp_(0, ng - 1)
    at = (q[0] * ng + q[1]) * ng + q[2]
    fk = torch.fft.rfftn(torch.bincount(at, minlength=ng ** 3).reshape(ng, ng, ng).float())
    k = torch.fft.fftfreq(ng, device="cuda") * (2 * math.pi / cell)
    kz = torch.fft.rfftfreq(ng, device="cuda") * (2 * math.pi / cell)
    kk = torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2)
    want = lo + (hi - lo) * torch.rand(n, generator=g, device="cuda")
    h = 0.45 * L * (1 - 0.02 * torch.rand(n, generator=g, device="cuda"))  # no more than this
    most = h
    found = torch.zeros(n, dtype=torch.bool, device="cuda")
    prev_R, prev_N = None, None
    R = 0.62 * cell
    while R < 0.45 * L:
        y = (kk * R).clamp_min(0.05)
        win = 3 * (torch.sin(y) - y * torch.cos(y)) / y ** 3
        N = torch.fft.irfftn(fk * win, s=(ng,) * 3).reshape(-1)[at] * (4 / 3 * math.pi * (R / cell) ** 3)
        N = N.clamp_min(1e-3)
        if prev_N is None:
            r = R * (want / N) ** (1 / 3)
        else:
            N = torch.maximum(N, prev_N * 1.0001)
            r = prev_R * torch.exp(torch.log(want / prev_N) / torch.log(N / prev_N)
                                   * math.log(R / prev_R))
        now = ~found & (N >= want)
        h = torch.where(now, r, h)
        found |= now
        if bool(found.all()):
            break
        prev_R, prev_N = R, N
        R *= 1.15
    return torch.minimum(h.clamp_min(1e-4 * L), most).double()


def _box(g, n, case, var):
    """x (3, n), h (n) of one box in double."""
    L = case["L"]
    if case["shape"] == "lattice":
        side = round(n ** (1 / 3))
        a = torch.arange(side, device="cuda").double()
        grid = torch.stack(torch.meshgrid(a, a, a, indexing="ij")).reshape(3, -1)
        jit = (torch.rand((3, n), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.4
        x = (grid + 0.5 + jit) * (L / side)
        near = 57 + 14 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        return x, L * (3 * near / (4 * math.pi * n)) ** (1 / 3)
    ng = min(256, max(8, round(n ** (1 / 3))))
    rho = _field(g, ng, var).reshape(-1)
    edge = torch.cumsum((rho.double() * (2.0 ** 40 / float(rho.double().sum()))).long() + 1, 0)
    pick = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * float(edge[-1])).long()
    c = torch.searchsorted(edge, pick, right=True).clamp_(max=ng ** 3 - 1)
    q = torch.stack([c // (ng * ng), (c // ng) % ng, c % ng]).double()
    x = (q + torch.rand((3, n), generator=g, device="cuda", dtype=torch.float64)) * (L / ng)
    x = torch.where(x >= L, torch.zeros_like(x), x)
    return x, _reach(g, x, L, 90, 110)


def _gas(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float64 if case.get("fp64") else torch.float32
    d = {}
    if case["shape"] == "boxes":
        parts = [_box(g, s ** 3, case, case["var"]) for s in _sides(case)]
        d["x"] = torch.cat([p[0] for p in parts], 1).contiguous()
        h = torch.cat([p[1] for p in parts])
        counts = torch.tensor([0] + [s ** 3 for s in _sides(case)])
        d["box_off"] = torch.cumsum(counts, 0).cuda()
        d["box_L"] = torch.full((case["boxes"],), case["L"], dtype=torch.float64, device="cuda")
    else:
        x, h = _box(g, case["n"], case, case.get("var"))
        d["x"] = x.contiguous()
    n = h.shape[0]

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    m = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    if case.get("masses"):
        m = m * torch.exp(0.7 * normal(n).clamp(-2.5, 2.5))
    d.update(h=h.to(real), m=m.to(real), v=(0.1 * normal(3, n)).to(real),
             u=torch.exp(1.151 * normal(n).clamp(-3, 3)).to(real),
             ga=normal(3, n).to(real), gu=normal(n).to(real))
    if case["kind"] == "active":
        d["flags"] = (torch.rand(n, generator=g, device="cuda") < case["fraction"]).to(torch.uint8)
    if case["kind"] == "subgrid":
        # subgrid particles sit where the gas is dense
        at = torch.randint(0, n, (case["n_s"],), generator=g, device="cuda")
        jit = normal(3, case["n_s"]) * 0.1 * h[at]
        xs = torch.remainder(d["x"][:, at] + jit, case["L"])
        d["x_s"] = torch.where(xs >= case["L"], torch.zeros_like(xs), xs).contiguous()
        d["h_s"] = h[at].float()
        d["q_s"] = torch.rand((3, case["n_s"]), generator=g, device="cuda")
        d["rho"] = torch.exp(0.5 * normal(n)).float()
        k = torch.arange(COOL["nodes"], dtype=torch.float64, device="cuda")
        d["lam"] = COOL["A"] * (10.0 ** (COOL["log10_min"] + COOL["dex"] * k)) ** 1.5
    return d


def prepare(case, seed):
    d = _gas(case, seed)
    n = d["h"].shape[0]
    nb = case.get("boxes", 1)
    s = Solver(n, nb, "fp64" if case.get("fp64") else "mixed")
    st = dict(case=case, d=d, s=s)
    st["boxes"] = dict(L_box=case["L"])
    if nb > 1:
        st["boxes"].update(box_off=d["box_off"], box_L=d["box_L"])
    s.cell_build(d["x"], d["h"], **st["boxes"])  # grows the neighbor lists to what this gas needs
    kind = case["kind"]
    real = d["h"].dtype

    def like(*shape):
        return torch.empty(shape, dtype=real, device="cuda")

    if case.get("tuned"):
        if n in _tuned:
            s.tune_set(_tuned[n])
        else:
            _tuned[n] = s.autotune(d["m"], d["v"], d["u"], d["ga"], d["gu"],
                                   repeats=3 if n < 10 ** 6 else 1)
    if kind == "step":
        st["rates"] = (like(3, n), like(n))
        st["grads"] = (like(3, n), like(3, n), like(n), like(n))
        if case.get("graph"):
            st["graph"] = s.capture(lambda: _step(st))
    elif kind == "kdk":
        st["der"] = s.kdk_init(d["x"], d["v"], d["u"], d["h"], d["m"], KDK_DT, LAMBDA, N_H,
                               **st["boxes"])
        st["scratch"] = (like(3, n), like(n))
    elif kind == "active":
        V, coef = s.moments(d["m"], want_V=True, want_coef=True)
        _, _, rho, gradv = s.rates(d["v"], d["u"], want_rho=True, want_gradv=True)
        st["stored"] = (V, coef, rho, gradv)
    elif kind == "subgrid":
        s.moments(d["m"])
    elif kind == "grad":
        st["leaves"] = [d[k].requires_grad_() for k in ("x", "v", "u", "h")]
    return st


def _step(st):
    d, s = st["d"], st["s"]
    s.cell_build(d["x"], d["h"], check=False, **st["boxes"])
    s.moments(d["m"])
    s.rates(d["v"], d["u"], out=st["rates"])
    s.adjoint(d["v"], d["u"], d["ga"], d["gu"], recompute=False, out=st["grads"])


def run(st):
    case, d, s, boxes = st["case"], st["d"], st["s"], st["boxes"]
    kind = case["kind"]
    if kind == "grad":
        x, v, u, h = st["leaves"]
        dv, du = rates(x, v, u, h, d["m"], s, **boxes)
        gx, gv, gu, gh = torch.autograd.grad((dv, du), (x, v, u, h), (d["ga"], d["gu"]))
        # the mixed form's position gradient has single precision in a double tensor
        return dict(dvdt=dv, dudt=du, gx=gx.to(v.dtype), gv=gv, gu=gu, gh=gh)
    if kind == "forward":
        out = s.forward(d["x"], d["h"], d["m"], d["v"], d["u"], want_rho=True, **boxes)
        return dict(dvdt=out["dvdt"], dudt=out["dudt"], rho=out["rho"])
    if kind == "fused":
        s.cell_build(d["x"], d["h"], **boxes)
        s.moments(d["m"])
        return list(s.rates_adjoint(d["v"], d["u"], d["ga"], d["gu"]))
    if kind == "step":
        if "graph" in st:
            st["graph"].replay()
        else:
            _step(st)
        return list(st["rates"]) + list(st["grads"])
    if kind == "kdk":
        der = s.kdk_step(d["x"], d["v"], d["u"], d["h"], d["m"], st["der"], KDK_DT, LAMBDA, N_H,
                         scratch=st["scratch"], **boxes)
        return dict(x=d["x"], v=d["v"], u=d["u"], h=d["h"], a=der["a"], du=der["du"],
                    hrate=der["hrate"], div=der["div"])
    if kind == "active":
        s.cell_build(d["x"], d["h"], check=False, **boxes)
        V, coef, rho, gradv = st["stored"]
        s.moments_active(d["m"], d["flags"], V, coef)
        dv, du = s.rates_active(d["v"], d["u"], rho, gradv)
        return dict(dvdt=dv, dudt=du, V=V, coef=coef, rho=rho, gradv=gradv)
    V, h = s.subgrid_volume(d["x_s"], d["h_s"], n_h=N_H)
    dq, A = s.subgrid_deposit(d["x_s"], d["h_s"], d["q_s"])
    u1 = s.cool(COOL["dt"], d["rho"], d["u"], d["lam"], COOL["log10_min"], COOL["dex"])
    return dict(V=V, h=h, dq=dq, A=A, u1=u1)


def work(case):
    """Bytes: every input and output once.  Operations: the pairs (100 within
    h, 116 in the union of both directions) times what one pair takes."""
    n = sum(s ** 3 for s in _sides(case)) if case["shape"] == "boxes" else case["n"]
    R = 8 if case.get("fp64") else 4
    near = 64 if case["shape"] == "lattice" else 100
    forward = near * (31 + 114 + 117) + 1.16 * near * 253
    adjoint = 1.16 * near * 654 + near * (511 + 458 + 93)
    state = 24 + 6 * R  # x; h, m, u, v
    kind = case["kind"]
    if kind == "forward":
        return dict(bytes=n * (state + 5 * R), flops=n * forward)
    if kind in ("grad", "fused", "step"):
        return dict(bytes=n * (state + 4 * R + 4 * R + 8 * R), flops=n * (forward + adjoint))
    if kind == "kdk":
        return dict(bytes=n * (2 * state + 2 * 6 * R), flops=n * forward)
    if kind == "active":
        f = case["fraction"]
        return dict(bytes=n * (state + 1 + 27 * R + f * 31 * R), flops=n * f * forward)
    n_s = case["n_s"]
    return dict(bytes=n * (24 + 3 * 4 + 4 * R + 4 * R) + n_s * (24 + 16 + 12),
                flops=n_s * near * 3 * 40 + n * 400)


# ---------------------------------------------------------------------------
# the same results in 64 bits, with plain torch
# ---------------------------------------------------------------------------
def _image(t, L):
    t = torch.where(t > 0.5 * L, t - L, t)
    return torch.where(t < -0.5 * L, t + L, t)


def _pairs(x, h, L):
    """Ordered pairs i != j with r < max(h_i, h_j)."""
    n = h.shape[0]
    rows = max(1, (1 << 27) // n)
    I, J = [], []
    for a in range(0, n, rows):
        b = min(n, a + rows)
        r2 = torch.zeros((b - a, n), dtype=torch.float64, device="cuda")
        for c in range(3):
            r2 += _image(x[c, a:b, None] - x[c, None, :], L) ** 2
        hit = r2 < torch.maximum(h[a:b, None], h[None, :]) ** 2
        i, j = torch.nonzero(hit, as_tuple=True)
        i = i + a
        keep = i != j
        I.append(i[keep])
        J.append(j[keep])
    return torch.cat(I), torch.cat(J)


def _kernel(r, h):
    q = r / h
    om = (1 - q).clamp_min(0)
    cw = 495 / (32 * math.pi)
    W = cw / h ** 3 * om ** 6 * (1 + 6 * q + 35 / 3 * q * q)
    g = -(56 / 3) * cw / h ** 5 * om ** 5 * (1 + 5 * q)  # W'(r) / r
    return W, g


def _sum(i, n, v):
    return torch.zeros((n,) + v.shape[1:], dtype=v.dtype, device=v.device).index_add(0, i, v)


def _parts(i, n, limit):
    """Slices of the pairs (sorted by i) of at most about `limit` pairs, on row borders."""
    if i.numel() <= limit:
        return [slice(0, i.numel())]
    edge = torch.searchsorted(i, torch.arange(0, n + 1, device=i.device)).tolist()
    out, a = [], 0
    for k in range(1, n + 1):
        if k == n or edge[k + 1] - edge[a] > limit:
            out.append(slice(edge[a], edge[k]))
            a = k
    return out


def _evaluate(x, v, u, h, m, L, limit=1 << 62):
    """V, A, B, grad A, grad B, rho, grad v and the rates; x, v (n, 3)."""
    n = h.shape[0]
    with torch.no_grad():
        I, J = _pairs(x.t().contiguous(), h, L)
        near = ((_image(x[I] - x[J], L) ** 2).sum(1) < h[I] ** 2)
    i, j = I[near], J[near]
    eye = torch.eye(3, dtype=x.dtype, device=x.device)

    def separation(i, j):
        d = _image(x[i] - x[j], L)
        return d, torch.sqrt((d * d).sum(1).clamp_min(1e-300))

    W0 = 495 / (32 * math.pi) / h ** 3
    s = m * W0
    for p in _parts(i, n, limit):
        d, r = separation(i[p], j[p])
        s = s + _sum(i[p], n, m[j[p]] * _kernel(r, h[i[p]])[0])
    V = m / s
    m0 = V * W0
    z = lambda *k: torch.zeros((n,) + k, dtype=x.dtype, device=x.device)  # noqa: E731
    m1, m2, S0, S2, S3 = z(3), z(3, 3), z(3), z(3, 3), z(3, 3, 3)
    for p in _parts(i, n, limit):
        a, b = i[p], j[p]
        d, r = separation(a, b)
        W, g = _kernel(r, h[a])
        w, gv = V[b] * W, V[b] * g
        dd = d[:, :, None] * d[:, None, :]
        m0 = m0 + _sum(a, n, w)
        m1 = m1 + _sum(a, n, w[:, None] * d)
        m2 = m2 + _sum(a, n, w[:, None, None] * dd)
        S0 = S0 + _sum(a, n, gv[:, None] * d)
        S2 = S2 + _sum(a, n, gv[:, None, None] * dd)
        S3 = S3 + _sum(a, n, gv[:, None, None, None] * dd[:, :, :, None] * d[:, None, None, :])
    # grad m0 = S0, d_g m1_a = S2_ag + delta_ag m0, d_g m2_ab = S3_abg + delta_ag m1_b + delta_bg m1_a
    dm1 = S2 + eye * m0[:, None, None]
    dm2 = S3 + eye[None, :, None, :] * m1[:, None, :, None] + eye[None, None, :, :] * m1[:, :, None, None]
    M = torch.linalg.inv(m2)
    B = -torch.einsum("nab,nb->na", M, m1)
    A = 1 / (m0 + (B * m1).sum(1))
    dM = -torch.einsum("nab,nbcg,ncd->nadg", M, dm2, M)
    dB = -torch.einsum("nabg,nb->nag", dM, m1) - torch.einsum("nab,nbg->nag", M, dm1)
    dA = -(A * A)[:, None] * (S0 + torch.einsum("nag,na->ng", dB, m1) + torch.einsum("na,nag->ng", B, dm1))

    def corrected(k, d, r):  # W^R and its gradient at particle k, d = x_k - x_other
        W, g = _kernel(r, h[k])
        lin = 1 + (B[k] * d).sum(1)
        G = (dA[k] * (lin * W)[:, None]
             + (A[k] * W)[:, None] * (torch.einsum("pag,pa->pg", dB[k], d) + B[k])
             + (A[k] * lin * g)[:, None] * d)
        return A[k] * lin * W, G

    num, den, gradv = m * V * A * W0, V * V * A * W0, z(3, 3)
    for p in _parts(i, n, limit):
        a, b = i[p], j[p]
        d, r = separation(a, b)
        WR, G = corrected(a, d, r)
        num = num + _sum(a, n, m[b] * V[b] * WR)
        den = den + _sum(a, n, V[b] ** 2 * WR)
        gradv = gradv - _sum(a, n, V[b][:, None, None] * (v[a] - v[b])[:, :, None] * G[:, None, :])
    rho = num / den
    gamma = 5 / 3
    P, cs = (gamma - 1) * rho * u, torch.sqrt(gamma * (gamma - 1) * u)
    acc, du = z(3), z()
    crit, fold = 1 / N_H, 0.2
    for p in _parts(I, n, limit):
        a, b = I[p], J[p]
        d, r = separation(a, b)
        Gi, Gj = corrected(a, d, r)[1], corrected(b, -d, r)[1]
        gd = torch.einsum("pab,pb->pa", gradv[a], d), torch.einsum("pab,pb->pa", gradv[b], d)
        pa, pb = (d * gd[0]).sum(1), (d * gd[1]).sum(1)
        same = pa * pb > 0
        phi = torch.where(same, 4 * pa * pb / torch.where(same, pa + pb, torch.ones_like(pa)) ** 2,
                          torch.zeros_like(pa))
        eta = r / torch.maximum(h[a], h[b])
        phi = torch.where(eta < crit, phi * torch.exp(-((eta - crit) / fold) ** 2), phi)
        vij = v[a] - v[b]
        vx = ((vij - 0.5 * phi[:, None] * (gd[0] + gd[1])) * d).sum(1)

        def Q(k):
            mu = (vx / h[k] / ((r / h[k]) ** 2 + 0.01)).clamp_max(0)
            return rho[k] * (-2 * cs[k] * mu + mu * mu)

        F = (-0.5 * V[a] * V[b] * (P[a] + P[b] + Q(a) + Q(b)))[:, None] * (Gi - Gj)
        acc = acc + _sum(a, n, F)
        du = du - _sum(a, n, 0.5 * (F * vij).sum(1))
    coef = torch.cat([A[:, None], B, dA, dB.transpose(1, 2).reshape(n, 9)], 1)
    return dict(V=V, coef=coef, rho=rho, gradv=gradv, dvdt=acc / m[:, None], dudt=du / m)


def _exact_box(d, L, sel, adjoint):
    """Rates (and gradients) of one box; the box's particles are `sel`."""
    x, v = d["x"].detach()[:, sel].t().contiguous(), d["v"].detach()[:, sel].t().double().contiguous()
    u, h, m = (d[k].detach()[sel].double() for k in ("u", "h", "m"))
    if not adjoint:
        with torch.no_grad():
            return _evaluate(x, v, u, h, m, L, limit=1 << 22), None
    for t in (x, v, u, h):
        t.requires_grad_()
    o = _evaluate(x, v, u, h, m, L)
    ga, gu = d["ga"][:, sel].t().double(), d["gu"][sel].double()
    gx, gv, gu_, gh = torch.autograd.grad((o["dvdt"], o["dudt"]), (x, v, u, h), (ga, gu))
    return {k: t.detach() for k, t in o.items()}, (gx.t(), gv.t(), gu_, gh)


def exact(case, seed):
    kind = case["kind"]
    n = sum(s ** 3 for s in _sides(case)) if case["shape"] == "boxes" else case["n"]
    biggest = max(_sides(case)) ** 3 if case["shape"] == "boxes" else n
    if biggest > 300000 or n > 2000000:
        return None
    d, L = _gas(case, seed), case["L"]
    if kind == "subgrid":
        return _exact_subgrid(case, d)
    if kind == "kdk":
        return _exact_kdk(d, L)
    adjoint = kind in ("grad", "fused", "step") and biggest <= 60000
    if case["shape"] == "boxes":
        e = d["box_off"].tolist()
        spans = [slice(a, b) for a, b in zip(e[:-1], e[1:])]
    else:
        spans = [slice(0, n)]
    got, grads = [], []
    for p in spans:
        o, g = _exact_box(d, L, p, adjoint)
        got.append(o)
        grads.append(g)
        torch.cuda.empty_cache()
    o = {k: torch.cat([b[k] for b in got]) for k in got[0]}
    dv, du = o["dvdt"].t().contiguous(), o["dudt"]
    if kind == "forward":
        return dict(dvdt=dv, dudt=du, rho=o["rho"])
    if kind == "active":
        on = d["flags"].bool()
        return dict(dvdt=dv * on, dudt=du * on, V=o["V"], coef=o["coef"].t().contiguous(),
                    rho=o["rho"], gradv=o["gradv"].reshape(n, 9).t().contiguous())
    if adjoint:
        gx, gv, gu, gh = (torch.cat([g[k] for g in grads], -1) for k in range(4))
    else:
        gx = gv = gu = gh = None
    if kind == "grad":
        return dict(dvdt=dv, dudt=du, gx=gx, gv=gv, gu=gu, gh=gh)
    return [dv, du, gx, gv, gu, gh]


def _exact_kdk(d, L):
    x, v = d["x"].t().contiguous(), d["v"].t().double()
    u, h, m = (d[k].double() for k in ("u", "h", "m"))
    dt = KDK_DT

    def evaluate(x, v, u, h):
        with torch.no_grad():
            o = _evaluate(x, v, u, h, m, L, limit=1 << 22)
        div = torch.einsum("naa->n", o["gradv"])
        ht = h * (1 - LAMBDA) + LAMBDA * N_H * o["V"] ** (1 / 3)
        return o["dvdt"], o["dudt"], ((ht - h) / dt + h * div / 3) / h, div

    a, du, hr, _ = evaluate(x, v, u, h)
    v, u = v + 0.5 * dt * a, u + 0.5 * dt * du
    x = torch.remainder(x + v * dt, L)
    # the library keeps h in single precision, which decides who is a neighbor
    h = (h * torch.exp(hr * dt)).to(d["h"].dtype).double()
    a, du, hr, div = evaluate(x, v + 0.5 * dt * a, u + 0.5 * dt * du, h)
    v, u = v + 0.5 * dt * a, u + 0.5 * dt * du
    return dict(x=x.t().contiguous(), v=v.t().contiguous(), u=u, h=h, a=a.t().contiguous(), du=du,
                hrate=hr, div=div)


def _exact_subgrid(case, d):
    L, n = case["L"], case["n"]
    x, h, m = d["x"], d["h"].double(), d["m"].double()
    with torch.no_grad():
        i, j = _pairs(x, h, L)
        r = torch.sqrt((_image(x[:, i] - x[:, j], L) ** 2).sum(0))
        s = m * 495 / (32 * math.pi) / h ** 3 + _sum(i, n, m[j] * _kernel(r, h[i])[0])
        Vg = m / s
        xs, hs, q = d["x_s"], d["h_s"].double(), d["q_s"].double()
        n_s = hs.shape[0]
        vol, A = torch.zeros(n_s, dtype=torch.float64, device="cuda"), None
        dq = torch.zeros((3, n), dtype=torch.float64, device="cuda")
        A = torch.zeros(n_s, dtype=torch.float64, device="cuda")
        rows = max(1, (1 << 27) // n)
        for a in range(0, n_s, rows):
            b = min(n_s, a + rows)
            r2 = torch.zeros((b - a, n), dtype=torch.float64, device="cuda")
            for c in range(3):
                r2 += _image(xs[c, a:b, None] - x[c, None, :], L) ** 2
            r = torch.sqrt(r2)
            vol[a:b] = (_kernel(r, h[None, :])[0]).sum(1)
            w = Vg * _kernel(r, hs[a:b, None])[0]
            tot = w.sum(1)
            A[a:b] = torch.where(tot > 0, 1 / tot.clamp_min(1e-300), torch.zeros_like(tot))
            dq += q[:, a:b] @ (w * A[a:b, None])
        V = 1 / (vol + 495 / (32 * math.pi) / hs ** 3)
        # lambda(u) = A u^1.5: du/dt = -rho lambda, down to the lowest node
        u, rho = d["u"].double(), d["rho"].double()
        lo, hi = (10.0 ** (COOL["log10_min"] + COOL["dex"] * k) for k in (0, COOL["nodes"] - 1))
        u1 = (u ** -0.5 + 0.5 * COOL["A"] * rho * COOL["dt"]) ** -2
        u1 = torch.where((u >= lo) & (u <= hi), u1.clamp_min(lo), u)
    return dict(V=V, h=N_H * V ** (1 / 3), dq=dq, A=A, u1=u1)
