"""The work that a user of this library has it do, as measurable cases.

Every case goes through the public Python binding (paper_0901_3512_gb300.seedcg), which
is a thin layer over the C ABI.  Inputs are drawn on the GPU from the seed alone, by the
recipe of paper_0901_3512_gb300.workloads: links exp(i eps A) with eps = 0.5 and Gaussian
traceless Hermitian A, point or Z2 sources, b = D^dag eta.

kinds:
  apply      one operator application on n fields (D, D^dag or M; FP64 or FP32)
  apply_eo   the even-odd operator of Section 3 on odd-site half vectors
  solve      Improved Seed-CG for all right-hand sides of one gauge field
  solve_eo   the same on the even-odd preconditioned system
  batch      three gauge fields of uneven sizes in one batched solve
  predict    the learned initial guess, inference on n right-hand sides
  grad       the learned guess's loss and weight gradient over a mini-batch

The solves run to ||b - M x|| <= 1e-12 ||b||, so that the solutions are defined to about
ten digits whatever path the iteration took; kappa lies below the near-critical values
of the workload table so that every random field is safely solvable (cond(M) about 1e3).
"""
import math

import torch

from paper_0901_3512_gb300 import seedcg, workloads

TOL = 1e-12
EPS = 0.5
LISTED = [
    # the smallest call: one field on a 4^4 lattice, for a caller that cannot allocate;
    # launches and latency are all it costs
    {"name": "apply_noalloc_tiny", "kind": "apply", "dims": "4x4x4x4", "n": 1, "op": 0, "prec": 0, "multi": 0,
     "noalloc": True, "kappa": 0.2},
    # M on twelve fields in single precision on the 8^3x16 lattice (residuals and smoothing steps
    # of a caller's own iteration)
    {"name": "apply_m_f32_mid", "kind": "apply", "dims": "8x8x8x16", "n": 12, "op": 2, "prec": 1, "multi": 1,
     "noalloc": False, "kappa": 0.2},
    # forming b = D^dag eta for twelve sources on the 16^3x32 lattice, before every solve there
    {"name": "apply_ddag_f64_large", "kind": "apply", "dims": "16x16x16x32", "n": 12, "op": 1, "prec": 0, "multi": 1,
     "noalloc": False, "kappa": 0.2},
    # A^dag A of Section 3 in single precision on six half vectors of the 12^3x24 lattice
    {"name": "apply_eo_f32_mid", "kind": "apply_eo", "dims": "12x12x12x24", "n": 6, "op": 2, "prec": 1, "kappa": 0.2},
    # plain FP64 seed-CG on 4^4 with four Z2 sources: every launch is tiny
    {"name": "solve_f64_tiny", "kind": "solve", "dims": "4x4x4x4", "nrhs": 4, "precision": "fp64", "source": "z2",
     "past": 1.5, "period": 10, "seed_mode": 1, "m_max": 1000, "kappa": 0.2},
    # plain FP64 seed-CG on 8^3x16 with twelve point sources
    {"name": "solve_f64_small", "kind": "solve", "dims": "8x8x8x16", "nrhs": 12, "precision": "fp64",
     "source": "point", "past": 2.0, "period": 10, "seed_mode": 1, "m_max": 1000, "kappa": 0.2},
    # a lattice of unequal extents with an odd number of sources, complex64 basis
    {"name": "solve_v32_ragged", "kind": "solve", "dims": "10x6x14x12", "nrhs": 5, "precision": "mixed_v32",
     "source": "z2", "past": 1.5, "period": 10, "seed_mode": 1, "m_max": 1000, "kappa": 0.2},
    # the headline shape: 16^3x32, twelve point sources, bf16 basis, tensor-core seeds
    {"name": "solve_bf16_large", "kind": "solve", "dims": "16x16x16x32", "nrhs": 12, "precision": "mixed_vbf16",
     "source": "point", "past": 2.0, "period": 10, "seed_mode": 1, "m_max": 1000, "kappa": 0.2},
    # the paper's own setting: the even-odd preconditioned system on the same lattice and sources
    {"name": "solve_eo_bf16_large", "kind": "solve_eo", "dims": "16x16x16x32", "nrhs": 12,
     "precision": "mixed_vbf16", "source": "point", "past": 2.0, "period": 10, "seed_mode": 1, "m_max": 1000,
     "kappa": 0.2},
    # three uneven fields (24, 12 and 6 Z2 sources) sharing one batched CG
    {"name": "batch3_v32", "kind": "batch", "dims": "8x8x8x16 12x12x12x24 16x16x16x32", "nrhs": "24 12 6",
     "precision": "mixed_v32", "source": "z2", "past": 1.5, "period": 10, "seed_mode": 1, "m_max": 1000,
     "kappa": 0.2},
    # the learned guess: inference for twelve right-hand sides of the 16^3x32 field
    {"name": "predict_large", "kind": "predict", "dims": "16x16x16x32", "n": 12, "kappa": 0.2},
    # the learned guess: loss and weight gradient of a mini-batch of eight pairs (forward and backward)
    {"name": "grad_large", "kind": "grad", "dims": "16x16x16x32", "n": 8, "kappa": 0.2},
]


def listed():
    return [dict(c) for c in LISTED]


# ---------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------
def _dims(case_dims):
    return [tuple(int(v) for v in d.split("x")) for d in case_dims.split()]


def _vol(dims):
    return math.prod(dims)


def _rand_dims(rng, vmax=16 * 16 * 16 * 32):
    """Even extents, the volume spread over its logarithm between 4^4 and 16^3 x 32."""
    v = math.exp(rng.uniform(math.log(256), math.log(vmax)))
    while True:
        e = v ** 0.25
        d = [2 * max(2, round(0.5 * e * math.exp(rng.uniform(-0.45, 0.45)))) for _ in range(3)]
        d.append(2 * max(2, round(0.5 * v / math.prod(d))))
        if d[3] <= 64 and _vol(d) <= vmax:
            return "x".join(str(x) for x in d)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply_eo", "solve", "solve", "solve", "solve_eo", "batch", "predict", "grad"])
    kappa = round(rng.uniform(0.18, 0.2), 4)
    c = {"kind": kind, "dims": _rand_dims(rng), "kappa": kappa}
    if kind in ("apply", "apply_eo"):
        c.update(n=max(1, round(math.exp(rng.uniform(0, math.log(12))))), op=rng.randrange(3), prec=rng.randrange(2))
        if kind == "apply":
            c.update(multi=1 if rng.random() < 0.7 else 0)
            fits = 3 * c["n"] * _vol(_dims(c["dims"])[0]) * 12 * (8 if c["prec"] else 16) <= seedcg.NOALLOC_SCRATCH_BYTES
            c.update(noalloc=fits and rng.random() < 0.5)
    elif kind in ("predict", "grad"):
        c.update(n=rng.randint(1, 12 if kind == "predict" else 8))
    else:
        c.update(precision=rng.choice(["fp64", "mixed_v32", "mixed_vbf16"]), source="z2", past=rng.choice([1.0, 1.5, 2.0]),
                 period=rng.choice([10, 20]), seed_mode=3 if kind != "batch" and rng.random() < 0.2 else 1, m_max=1000)
        if c["precision"] == "fp64":
            c["dims"] = _rand_dims(rng, 8 * 8 * 8 * 16)
        if kind == "batch":
            nf = rng.randint(2, 3)
            vmax = 8 * 8 * 8 * 16 if c["precision"] == "fp64" else 12 * 12 * 12 * 24
            c["dims"] = " ".join(_rand_dims(rng, vmax) for _ in range(nf))
            c["nrhs"] = " ".join(str(rng.randint(1, 12)) for _ in range(nf))
        else:
            c["nrhs"] = rng.randint(1, 12)
            if rng.random() < 0.3:
                c["source"] = "point"
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gauge(dims, g):
    """Links exp(i eps A), complex128 [V][4][3][3], on the GPU."""
    lam = torch.from_numpy(workloads.gell_mann()).cuda()
    coef = torch.randn(_vol(dims) * 4, 8, dtype=torch.float64, device="cuda", generator=g)
    a = torch.matmul(coef.to(torch.complex128), lam.reshape(8, 9)).reshape(-1, 3, 3) * (1j * EPS / 16)
    u = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(a).clone()
    term = u.clone()
    for k in range(1, 13):   # ||eps A / 16|| < 0.4: the series ends below 1e-15
        term = torch.matmul(term, a) / k
        u += term
    for _ in range(4):
        u = torch.matmul(u, u)
    return u.reshape(_vol(dims), 4, 3, 3).contiguous()


def _sources(dims, n, source, g):
    v = _vol(dims)
    if source == "point":
        eta = torch.zeros(n, v, 4, 3, dtype=torch.complex128, device="cuda")
        at = int(torch.randint(v, (1,), device="cuda", generator=g))
        for j in range(n):
            eta[j, at, j // 3, j % 3] = 1.0
        return eta
    bits = torch.randint(0, 2, (n, v, 4, 3), device="cuda", generator=g)
    return (2.0 * bits - 1.0).to(torch.complex128)


def _spinors(n, v, g):
    z = torch.randn(n, v, 4, 3, 2, dtype=torch.float64, device="cuda", generator=g)
    return torch.view_as_complex(z)


def _weights(g):
    """Starting weights of the network, as workloads.guess_weights draws them."""
    parts = []
    for ci, co in ((1, 8), (8, 8), (8, 1)):
        sd = 0.1 / math.sqrt(9 * ci * 4)
        z = torch.randn(9 * co * ci * 16, 2, dtype=torch.float64, device="cuda", generator=g)
        parts.append(torch.view_as_complex(sd * z))
    return torch.cat(parts)


def _inputs(case, seed):
    """Everything that is drawn for a case, the same for prepare() and exact()."""
    g = _gen(seed)
    kind = case["kind"]
    d = {"dims": _dims(case["dims"])}
    d["gauge"] = [_gauge(x, g) for x in d["dims"]]
    v = _vol(d["dims"][0])
    if kind == "apply":
        d["in"] = _spinors(case["n"], v, g)
    elif kind == "apply_eo":
        d["in"] = _spinors(case["n"], v // 2, g)
    elif kind in ("predict", "grad"):
        d["eta"] = [_sources(d["dims"][0], case["n"], "z2", g)]
        d["w"] = _weights(g)
    else:
        ns = [int(x) for x in str(case["nrhs"]).split()]
        d["eta"] = [_sources(x, n, case["source"], g) for x, n in zip(d["dims"], ns)]
    return d


class State:
    pass


def prepare(case, seed):
    d = _inputs(case, seed)
    s = State()
    s.case, s.kind = case, case["kind"]
    opts = {}
    if s.kind in ("solve", "solve_eo", "batch"):
        opts = {"precision": case["precision"], "past_factor": case["past"], "m_max": case["m_max"],
                "seed_mode": case["seed_mode"]}
    elif s.kind == "grad":
        opts = {"precision": "mixed_v32", "seed_mode": 3}
    s.solvers = [seedcg.Solver(x, u, case["kappa"], **opts) for x, u in zip(d["dims"], d["gauge"])]
    first = s.solvers[0]
    if s.kind in ("apply", "apply_eo"):
        s.inp = d["in"]
        s.out = torch.empty_like(s.inp)
    elif s.kind == "solve_eo":
        s.B = d["eta"]
        s.X = [torch.empty_like(b) for b in s.B]
    else:
        s.B = [torch.empty_like(e) for e in d["eta"]]
        for sv, e, b in zip(s.solvers, d["eta"], s.B):
            sv.apply(seedcg.OP_DDAG, e, b, prec=0, multi=1)
        s.X = [torch.empty_like(b) for b in s.B]
        if s.kind in ("predict", "grad"):
            if s.kind == "grad":   # the pairs that the network learns from: b and its solution
                first.solve(s.B[0], s.X[0], tol=TOL)
            seedcg.seedcg_guess_set_weights(first.h, d["w"].cpu().numpy())
    torch.cuda.synchronize()
    return s


def run(s):
    c, first = s.case, s.solvers[0]
    if s.kind == "apply":
        f = seedcg.seedcg_apply_noalloc if c["noalloc"] else seedcg.seedcg_apply
        f(first.h, c["op"], c["prec"], c["multi"], c["n"], s.inp, s.out)
        return s.out
    if s.kind == "apply_eo":
        seedcg.seedcg_apply_eo(first.h, c["op"], c["prec"], s.inp, s.out)
        return s.out
    if s.kind == "solve":
        first.solve(s.B[0], s.X[0], tol=TOL, extra_iters=0, reorth_period=c["period"])
        return s.X[0]
    if s.kind == "solve_eo":
        seedcg.seedcg_solve_eo(first.h, s.B[0], s.X[0], TOL, 0, c["period"])
        return s.X[0]
    if s.kind == "batch":
        seedcg.seedcg_batch_solve([x.h for x in s.solvers], s.B, s.X, TOL, 0, c["period"])
        return list(s.X)
    if s.kind == "predict":
        seedcg.seedcg_guess_predict(first.h, s.B[0], s.X[0])
        return s.X[0]
    # the gradient feeds an FP32 Adam step: it is held in complex64, the loss in a default float
    loss, grad = seedcg.seedcg_guess_loss_grad(first.h, s.B[0], s.X[0])
    return {"loss": loss, "grad": torch.from_numpy(grad).to(torch.complex64)}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
_HOP_FLOPS = 1344.0     # one Wilson D at one site for one field


def _iterations(case):
    """CG iterations to the tolerance on random fields: 175 at kappa = 0.18 and 312 at 0.2 (measured; half
    of that for the even-odd system), and about geometric in between."""
    it = 175.0 * (312.0 / 175.0) ** ((case["kappa"] - 0.18) / 0.02)
    return it * (0.5 if case["kind"] == "solve_eo" else 1.0)


def work(case):
    kind, dims = case["kind"], _dims(case["dims"])
    v = [_vol(d) for d in dims]
    if kind in ("apply", "apply_eo"):
        sites = v[0] // (2 if kind == "apply_eo" else 1)
        apps = (2 if case["op"] == 2 else 1)
        link = 36.0 * (8 if case["prec"] else 16) * v[0]
        return {"bytes": 2.0 * case["n"] * sites * 192 + link, "flops": apps * case["n"] * v[0] * _HOP_FLOPS}
    if kind in ("predict", "grad"):
        # per field: the input and output fields, the links, and the hidden activations (8 channels,
        # bf16) written and read once; the gradient reads them again and writes their gradients
        n = case["n"]
        acts = 8 * 48.0 * v[0]
        net = 2.0 * 4 * 9 * 16 * 3 * (8 + 64 + 8) * v[0]
        if kind == "predict":
            return {"bytes": n * (2 * 192.0 * v[0] + 4 * acts) + 288.0 * v[0], "flops": n * net}
        return {"bytes": n * (2 * 192.0 * v[0] + 12 * acts) + 288.0 * v[0], "flops": 3.0 * n * net}
    # a solve: read b, write x; Lanczos on the first system (skipped with seed_mode 3), two passes over the
    # stored rows per re-orthogonalisation, the seeds, and CG on every system
    ns = [int(x) for x in str(case["nrhs"]).split()]
    half = 0.5 if kind == "solve_eo" else 1.0
    el = 16.0 if case["precision"] == "fp64" else 8.0
    row = {"fp64": 16.0, "mixed_v32": 8.0, "mixed_vbf16": 4.0}[case["precision"]]
    it = _iterations(case)
    by = fl = 0.0
    for vol, n in zip(v, ns):
        vec = 12.0 * vol * half
        by += 2.0 * n * vol * 192 + it * (n * vec * 11 * el + 36 * el * vol)
        fl += 2.0 * it * n * vol * _HOP_FLOPS
        if case["seed_mode"] != 3:
            m = min(case["past"] * it, case["m_max"])
            by += m * (vec * 9 * el + 72 * el * vol) + m * vec * row * (m / case["period"] + 2)
            fl += 2.0 * m * vol * _HOP_FLOPS + 16.0 * m * vec * (m / case["period"] + n)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# 64-bit values, in plain torch
# ---------------------------------------------------------------------------
_EXACT_SITES = 1600000   # sites times fields that a solution in plain torch takes seconds for
_PERM = ((3, 2, 1, 0), (3, 2, 1, 0), (2, 3, 0, 1), (2, 3, 0, 1))
_PHASE = ((-1j, -1j, 1j, 1j), (-1, 1, 1, -1), (-1j, 1j, 1j, -1j), (1, 1, 1, 1))


class _Lattice:
    """Hops on fields [V][3][spins x anything] (colour second), antiperiodic in t."""

    def __init__(self, dims, u):
        self.dims = dims
        self.u = [u[:, mu].contiguous() for mu in range(4)]
        self.ph = [torch.tensor(p, dtype=torch.complex128, device="cuda") for p in _PHASE]

    def shift(self, f, mu, back):
        """f(x + mu) or f(x - mu) with the sign of a hop across t."""
        lx, ly, lz, lt = self.dims
        z = torch.roll(f.reshape(lt, lz, ly, lx, *f.shape[1:]), 1 if back else -1, dims=3 - mu)
        if mu == 3:
            z[0 if back else lt - 1] *= -1
        return z.reshape(f.shape)

    def transport(self, f, mu, back):
        """U_mu(x) f(x + mu) or U_mu(x - mu)^dag f(x - mu); f [V][3][k]."""
        if not back:
            return torch.matmul(self.u[mu], self.shift(f, mu, False))
        return self.shift(torch.matmul(self.u[mu].mH, f), mu, True)

    def hop(self, psi, dag):
        """H psi (dag: the hopping term of D^dag); psi [n][V][4][3]."""
        n, v = psi.shape[:2]
        f = psi.permute(1, 3, 2, 0).reshape(v, 3, 4 * n)
        out = torch.zeros_like(f).reshape(v, 3, 4, n)
        for mu in range(4):
            for back in (False, True):
                h = self.transport(f, mu, back).reshape(v, 3, 4, n)
                s = (1.0 if back else -1.0) * (-1.0 if dag else 1.0)
                out += h
                out += s * self.ph[mu][:, None] * h[:, :, _PERM[mu]]
        return out.permute(3, 0, 2, 1).contiguous()


def _solve_d(lat, kappa, eta):
    """D x = eta by CG on D^dag D in 64 bits, to about 1e-15."""
    def d(x, dag):
        return x - kappa * lat.hop(x, dag)

    def dot(a, b):
        return (a.conj() * b).real.sum(dim=(1, 2, 3))

    b = d(eta, True)
    x = torch.zeros_like(b)
    stop = 1e-30 * dot(b, b)
    for _ in range(2):   # the second round starts from the true residual
        r = b - d(d(x, False), True)
        p, rr = r.clone(), dot(r, r)
        for it in range(2000):
            t = d(p, False)
            a = (rr / dot(t, t))[:, None, None, None]
            x += a * p
            r -= a * d(t, True)
            new = dot(r, r)
            p = r + (new / rr)[:, None, None, None] * p
            rr = new
            if it % 10 == 9 and bool((rr <= stop).all()):
                break
    return x


def _net(lat, w, b):
    """The network on b [V][4][3]; w: three complex tensors [9][co][ci][4][4]."""
    def layer(f, wl):   # f [V][3][ci][4]
        v, _, ci, _ = f.shape
        flat = f.reshape(v, 3, ci * 4)
        out = 0
        for d in range(9):
            g = flat if d == 0 else lat.transport(flat, (d - 1) // 2, bool((d - 1) % 2))
            out = out + torch.matmul(g, wl[d].permute(1, 3, 0, 2).reshape(ci * 4, -1))
        return out.reshape(v, 3, -1, 4)

    def relu(z):
        return torch.complex(torch.relu(z.real), torch.relu(z.imag))

    nb = torch.linalg.vector_norm(b)
    f = (b / nb).permute(0, 2, 1)[:, :, None, :]
    h = relu(layer(f, w[0]))
    h = relu(layer(h, w[1]))
    return nb * layer(h, w[2])[:, :, 0, :].permute(0, 2, 1)


def _layers(w):
    a, b = 9 * 8 * 16, 9 * 64 * 16
    return [w[:a].reshape(9, 8, 1, 4, 4), w[a:a + b].reshape(9, 8, 8, 4, 4), w[a + b:].reshape(9, 1, 8, 4, 4)]


def exact(case, seed):
    d = _inputs(case, seed)
    lats = [_Lattice(x, u) for x, u in zip(d["dims"], d["gauge"])]
    lat, kappa, kind = lats[0], case["kappa"], case["kind"]
    if kind == "apply":
        x = d["in"]
        if case["op"] != 1:
            x = x - kappa * lat.hop(x, False)
        if case["op"] != 0:
            x = x - kappa * lat.hop(x, True)
        return x
    if kind == "apply_eo":
        x = d["in"]
        v = _vol(d["dims"][0])
        site = torch.arange(v, device="cuda")
        par, left = torch.zeros_like(site), site
        for ext in d["dims"][0]:
            par, left = par + left % ext, left // ext
        odd, even = site[par % 2 == 1], site[par % 2 == 0]

        def half(f, to, frm, dag):
            full = torch.zeros(f.shape[0], v, 4, 3, dtype=f.dtype, device=f.device)
            full[:, frm] = f
            return lat.hop(full, dag)[:, to]

        for dag in ((False,), (True,), (False, True))[case["op"]]:
            x = x - kappa * kappa * half(half(x, even, odd, dag), odd, even, dag)
        return x
    if kind in ("solve", "solve_eo", "batch"):
        if sum(e.shape[0] * e.shape[1] for e in d["eta"]) > _EXACT_SITES:
            return None   # too long in plain torch
        sol = [_solve_d(lt, kappa, e) for lt, e in zip(lats, d["eta"])]
        return sol if kind == "batch" else sol[0]
    eta = d["eta"][0]
    b = eta - kappa * lat.hop(eta, True)
    if kind == "predict":
        w = _layers(d["w"])
        return torch.stack([_net(lat, w, b[k]) for k in range(case["n"])])
    if eta.shape[0] * eta.shape[1] > _EXACT_SITES:
        return None
    x = _solve_d(lat, kappa, eta)
    w = d["w"].clone().requires_grad_()
    total = 0.0
    for k in range(case["n"]):
        y = _net(lat, _layers(w), b[k])
        loss = ((y - x[k]).abs() ** 2).sum() / (x[k].abs() ** 2).sum() / case["n"]
        loss.backward()
        total += float(loss.detach())
    return {"loss": torch.tensor(total, dtype=torch.float64), "grad": w.grad}
