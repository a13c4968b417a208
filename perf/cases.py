"""The work that users of this library have it do, as measurable cases.

Every case goes through the public entry points (``stag.Context`` and
``autograd.fermion_action``) on device-resident FP64 buffers:

* ``op``      one application of M^dag M or of a half operator in FP64: what a
              program calls to check a residual or to build its own solver;
* ``solve``   the mixed-precision CG for some sources and masses on one lattice
              (propagators; the even-site equation), or, with ``full``, the
              full-lattice equation M x = b;
* ``ragged``  one batch of solves on lattices of different sizes;
* ``step``    the fermion part of a molecular-dynamics step: the action by an
              FP64 CG on a freshly uploaded gauge field, and its gradients;
* ``hyp``     HYP smearing of a gauge field;
* ``npr``     the four-fermion contraction of the NPR workload.

Gauge fields are the repository's synthetic ones, reunitarise(exp(i c H)) with c
= 0.3 or 0.4, and sources complex Gaussian.  Solves run to a true residual of
1e-11, the differentiable action's to its default of 1e-12: the output is the
solution itself, and its own error can be some ten times the residual.
"""
import math

import torch

from paper_1511_00088_gb300 import stag
from paper_1511_00088_gb300.autograd import fermion_action

TOL, STEP_TOL = 1e-11, 1e-12
MAXITER = 100000
FULL, R12 = "fp32", "fp32_r12"  # FP32 links in the inner iteration: all rows, or two with the third rebuilt


def listed():
    return [
        # the smallest call: M^dag M on a test-sized lattice, all latency
        {"name": "op_mdagm_8x8", "kind": "op", "op": "mdagm", "lat": "8,8,8,8", "c": 0.3},
        # the residual check on the production lattice
        {"name": "op_mdagm_20x64", "kind": "op", "op": "mdagm", "lat": "20,20,20,64", "c": 0.4},
        # the smallest solve: a 2048-site CG, bound by the latency of an iteration
        {"name": "solve_8x8", "kind": "solve", "lat": "8,8,8,8", "c": 0.3, "links": FULL, "nrhs": 1, "masses": "0.05",
         "full": False},
        # a mid-sized lattice with plain FP32 links
        {"name": "solve_16x32", "kind": "solve", "lat": "16,16,16,32", "c": 0.4, "links": FULL, "nrhs": 1,
         "masses": "0.02", "full": False},
        # the benchmark: one source at the light mass of the 20^3 x 64 ensembles
        {"name": "solve_20x64", "kind": "solve", "lat": "20,20,20,64", "c": 0.4, "links": R12, "nrhs": 1,
         "masses": "0.01", "full": False},
        # a lattice whose links are many times the L2 cache, at a heavy mass
        {"name": "solve_48x96", "kind": "solve", "lat": "48,48,48,96", "c": 0.4, "links": R12, "nrhs": 1,
         "masses": "0.1", "full": False},
        # a propagator's 12 sources at 4 masses in one call
        {"name": "solve_20x64_12x4", "kind": "solve", "lat": "20,20,20,64", "c": 0.4, "links": R12, "nrhs": 12,
         "masses": "0.01,0.02,0.03,0.05", "full": False},
        # the full-lattice equation for a few sources on an uneven lattice
        {"name": "full_12x6x10x14", "kind": "solve", "lat": "12,6,10,14", "c": 0.4, "links": R12, "nrhs": 3,
         "masses": "0.05", "full": True},
        # lattices of four sizes in one batch
        {"name": "ragged_4", "kind": "ragged", "lat": "8,8,8,8;12,12,12,24;16,16,16,32;20,20,20,64", "c": 0.4,
         "links": R12, "masses": "0.02"},
        # an HMC trajectory's fermion step: upload, FP64 CG, action, gradients of links and pseudofermion
        {"name": "step_16x32", "kind": "step", "lat": "16,16,16,32", "c": 0.4, "mass": 0.05},
        # smearing the production gauge field
        {"name": "hyp_20x64", "kind": "hyp", "lat": "20,20,20,64", "c": 0.4},
        # one operator's contraction on the production lattice
        {"name": "npr_20x64", "kind": "npr", "lat": "20,20,20,64", "c": 0.4, "spin_taste": "1,2,4,7"},
    ]


def _dims(text):
    return tuple(int(v) for v in text.split(","))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _masses(case):
    return [float(v) for v in case["masses"].split(",")]


def _draw_dims(rng, lo, hi):
    """Even extents, time the longest as a rule, with about exp(uniform) sites in [lo, hi]."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = v ** 0.25
        d = [max(2, 2 * round(side * math.exp(rng.uniform(-0.35, 0.25)) / 2)) for _ in range(3)]
        d.append(max(2, 2 * round(v / (2 * d[0] * d[1] * d[2]))))
        if lo <= _volume(d) <= hi and d[3] <= 128:
            return d


def draw(rng):
    kind = rng.choice(["op", "solve", "solve", "solve", "ragged", "step", "hyp", "npr"])
    c = rng.choice([0.3, 0.4])

    def lat(lo, hi):
        return ",".join(str(v) for v in _draw_dims(rng, lo, hi))

    if kind == "op":
        return {"kind": kind, "op": rng.choice(["mdagm", "dslash_oe", "dslash_eo"]), "lat": lat(256, 1000000), "c": c}
    if kind == "solve":
        nrhs = rng.choice([1, 1, 1, 2, 3, 5, 12])
        nmass = rng.choice([1, 1, 1, 2, 3])
        full = rng.random() < 0.25
        masses = [round(math.exp(rng.uniform(math.log(0.02 if nrhs * nmass < 4 else 0.04), math.log(0.3))), 4)
                  for _ in range(nmass)]
        return {"kind": kind, "lat": lat(256, 1500000 if nrhs * nmass == 1 else 300000), "c": c,
                "links": rng.choice([FULL, R12]), "nrhs": nrhs, "masses": ",".join(str(m) for m in masses),
                "full": full}
    if kind == "ragged":
        return {"kind": kind, "lat": ";".join(lat(256, 200000) for _ in range(rng.randint(2, 4))), "c": c,
                "links": rng.choice([FULL, R12]), "masses": str(round(rng.uniform(0.02, 0.1), 4))}
    if kind == "step":
        return {"kind": kind, "lat": lat(256, 150000), "c": c, "mass": round(rng.uniform(0.03, 0.2), 4)}
    if kind == "hyp":
        return {"kind": kind, "lat": lat(256, 600000), "c": c}
    return {"kind": "npr", "lat": lat(256, 600000), "c": c,
            "spin_taste": ",".join(str(rng.randrange(16)) for _ in range(4))}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _links(dims, c, gen):
    """(4, V, 3, 3) complex128: Gram-Schmidt of exp(i c H), H traceless Hermitian Gaussian."""
    n = 4 * _volume(dims)
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    step = 1 << 22
    for s in range(0, n, step):
        m = min(step, n - s)
        z = torch.randn((m, 9), dtype=torch.float64, device="cuda", generator=gen)
        h = torch.zeros((m, 3, 3), dtype=torch.complex128, device="cuda")
        tr = (z[:, 0] + z[:, 1] + z[:, 2]) / 3.0
        for i in range(3):
            h[:, i, i] = z[:, i] - tr
        for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
            w = torch.complex(z[:, 3 + 2 * k], z[:, 4 + 2 * k])
            h[:, i, j] = w
            h[:, j, i] = w.conj()
        # exp(i c H) = (Taylor of i c H / 8)^8
        a = h * (1j * c / 8.0)
        e = torch.eye(3, dtype=torch.complex128, device="cuda") + a / 8.0
        for k in range(7, 0, -1):
            e = torch.eye(3, dtype=torch.complex128, device="cuda") + _mm(a, e) / k
        for _ in range(3):
            e = _mm(e, e)
        r0 = e[:, 0] / torch.linalg.vector_norm(e[:, 0], dim=-1, keepdim=True)
        r1 = e[:, 1] - (r0.conj() * e[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        out[s:s + m, 0] = r0
        out[s:s + m, 1] = r1
        out[s:s + m, 2] = torch.linalg.cross(r0, r1, dim=-1).conj()
    return out.reshape(4, -1, 3, 3)


def _gauss(n, gen):
    return torch.complex(torch.randn((n, 3), dtype=torch.float64, device="cuda", generator=gen),
                         torch.randn((n, 3), dtype=torch.float64, device="cuda", generator=gen))


def _inputs(case, seed):
    """The arrays of a case, from its seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    got = []
    for text in case["lat"].split(";"):
        dims = _dims(text)
        V = _volume(dims)
        links = _links(dims, case["c"], gen)
        kind = case["kind"]
        if kind == "solve":
            vecs = [_gauss(V if case["full"] else V // 2, gen) for _ in range(case["nrhs"])]
        elif kind == "npr":
            vecs = [_gauss(V, gen) for _ in range(4)]
        elif kind == "hyp":
            vecs = []
        else:
            vecs = [_gauss(V // 2, gen)]
        got.append((dims, links, vecs))
    return got


def prepare(case, seed):
    kind = case["kind"]
    ins = _inputs(case, seed)
    state = {"case": case, "vecs": [v for _, _, v in ins]}
    recon = case.get("links") == R12
    state["ctx"] = [stag.Context(dims, recon12=recon) for dims, _, _ in ins]
    if kind == "step":  # the field is uploaded in the step
        state["links"] = ins[0][1].requires_grad_()
        state["vecs"][0][0].requires_grad_()
    elif kind == "hyp":  # smeared before it is uploaded
        state["links"] = ins[0][1]
    else:
        for ctx, (_, links, _) in zip(state["ctx"], ins):
            ctx.links_upload(links)
    return state


def run(state):
    case, ctx, vecs = state["case"], state["ctx"], state["vecs"]
    kind = case["kind"]
    if kind == "op":
        x = vecs[0][0]
        if case["op"] == "mdagm":
            return ctx[0].mdagm(x, 0.05)
        return ctx[0].dslash_oe(x) if case["op"] == "dslash_oe" else ctx[0].dslash_eo(x)
    if kind == "solve":
        solve = ctx[0].solve_full if case["full"] else ctx[0].cg_solve
        return solve(vecs[0], _masses(case), tol=TOL, maxiter=MAXITER, precision=stag.STAG_FP32)[0]
    if kind == "ragged":
        batch = [(c, v, _masses(case)) for c, v in zip(ctx, vecs)]
        return stag.cg_solve_ragged(batch, tol=TOL, maxiter=MAXITER, precision=stag.STAG_FP32)[0]
    if kind == "step":
        links, phi = state["links"], vecs[0][0]
        s = fermion_action(links, phi, ctx[0], case["mass"], tol=STEP_TOL, precision=stag.STAG_FP64, maxiter=MAXITER)
        g_links, g_phi = torch.autograd.grad(s, (links, phi))
        return {"action": s.detach(), "grad_links": g_links, "grad_phi": g_phi}
    if kind == "hyp":
        return ctx[0].hyp_smear(state["links"])
    o, total = ctx[0].npr_contract([int(v) for v in case["spin_taste"].split(",")], *vecs[0])
    return {"hypercubes": o, "sum_re": total.real, "sum_im": total.imag}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _iterations(mass, tol=TOL):
    """CG iterations on these fields: 29.6 / m to 1e-10, in proportion to log(2 / tol)."""
    return 29.6 / mass * math.log(2 / tol) / math.log(2 / 1e-10)


def work(case):
    kind = case["kind"]
    nbytes = flops = 0.0
    for text in case["lat"].split(";"):
        V = _volume(_dims(text))
        Ve = V // 2
        link, vec = 4 * V * 144, Ve * 48  # all links, one checkerboard vector (FP64)
        if kind == "op":
            halves = 2 if case["op"] == "mdagm" else 1
            nbytes += link + 2 * vec
            flops += halves * 570 * Ve
        elif kind in ("solve", "ragged"):
            nrhs, masses = case.get("nrhs", 1), _masses(case)
            nbytes += link + (nrhs + nrhs * len(masses)) * vec * (2 if case.get("full") else 1)
            flops += nrhs * sum(_iterations(m) for m in masses) * 1212 * Ve
        elif kind == "step":
            nbytes += 2 * link + 2 * vec
            flops += (_iterations(case["mass"], STEP_TOL) * 1212 + 2 * 570) * Ve + 4 * V * 72
        elif kind == "hyp":
            # staples: 2 products of 198 flops each and a sum, per +-direction; 28 projections a site, of about
            # 5 Newton steps of 250 flops
            nbytes += 2 * link
            flops += V * ((12 * 2 + 12 * 4 + 4 * 6) * 2 * 216 + 28 * 5 * 250)
        else:
            nbytes += link / 2 + 4 * V * 48 + V  # the links inside hypercubes, four fields, O(z)
            flops += V / 16 * 99072
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _mm(a, b):
    """Products of 3 x 3 matrices, any leading shape."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _dag(a):
    return a.transpose(-1, -2).conj()


class _Op:
    """D_oe and D_eo on one lattice: neighbour tables and, per site, its 8 signed links."""

    def __init__(self, dims, links):
        Lx, Ly, Lz, Lt = dims
        V = _volume(dims)
        lex = torch.arange(V, device="cuda")
        x = [lex % Lx, lex // Lx % Ly, lex // (Lx * Ly) % Lz, lex // (Lx * Ly * Lz)]
        parity = (x[0] + x[1] + x[2] + x[3]) % 2
        strides = (1, Lx, Lx * Ly, Lx * Ly * Lz)
        self.cb = [lex[parity == 0], lex[parity == 1]]  # lexicographic sites of a parity, in checkerboard order
        self.nb, self.u = [], []
        for par in (0, 1):
            s = self.cb[par]
            nb, us = [], []
            for mu in range(4):
                xm = x[mu][s]
                eta = 1.0 - 2.0 * (sum((x[nu][s] for nu in range(mu)), torch.zeros_like(s)) % 2)
                fwd = s + torch.where(xm == dims[mu] - 1, 1 - dims[mu], 1) * strides[mu]
                bwd = s + torch.where(xm == 0, dims[mu] - 1, -1) * strides[mu]
                sf = sb = eta
                if mu == 3:
                    sf = torch.where(xm == Lt - 1, -eta, eta)
                    sb = torch.where(xm == 0, -eta, eta)
                nb += [fwd // 2, bwd // 2]
                us += [sf[:, None, None] * links[mu][s], -sb[:, None, None] * _dag(links[mu][bwd])]
            self.nb.append(torch.stack(nb, 1))
            self.u.append(torch.stack(us, 1))  # (sites, 8, 3, 3)

    def half(self, par_out, v):
        out = torch.empty_like(v)
        nb, u = self.nb[par_out], self.u[par_out]
        for s in range(0, v.shape[0], 1 << 20):
            e = s + (1 << 20)
            out[s:e] = (u[s:e] * v[nb[s:e]].unsqueeze(2)).sum((1, 3))
        return out

    def a(self, v, mass):
        return 4 * mass * mass * v - self.half(0, self.half(1, v))

    def solve(self, b, mass, tol=1e-15):
        """CG with restarts from the recomputed residual."""
        x = torch.zeros_like(b)
        norm = torch.linalg.vector_norm(b)
        for _ in range(4):
            r = b - self.a(x, mass)
            rho = torch.linalg.vector_norm(r) ** 2
            stop = max(float(tol * norm) ** 2, 1e-18 * float(rho))
            if float(rho) <= stop:
                break
            p, d = r.clone(), torch.zeros_like(b)
            for k in range(20000):
                ap = self.a(p, mass)
                alpha = rho / (p.conj() * ap).sum().real
                d += alpha * p
                r -= alpha * ap
                new = torch.linalg.vector_norm(r) ** 2
                if k % 16 == 15 and float(new) <= stop:
                    break
                p = r + (new / rho) * p
                rho = new
            x += d
        return x


def _exact_solve(case, dims, links, srcs):
    op = _Op(dims, links)
    masses = _masses(case)
    V = _volume(dims)
    out = []
    for r, b in enumerate(srcs):
        for m in masses:
            # of a large batch only some systems: the others would take too long
            if len(srcs) * len(masses) * V > 2e6 and (r > 0 or m < 0.025):
                out.append(None)
                continue
            if case.get("full"):
                be, bo = b[op.cb[0]], b[op.cb[1]]
                xe = op.solve(2 * m * be - op.half(0, bo), m)
                x = torch.empty_like(b)
                x[op.cb[0]] = xe
                x[op.cb[1]] = (bo - op.half(1, xe)) / (2 * m)
            else:
                x = op.solve(b, m)
            out.append(x)
    return out


def _exact_step(case, dims, links, phi):
    mass = case["mass"]
    op = _Op(dims, links)
    x = op.solve(phi, mass)
    y = op.half(1, x)
    action = (phi.conj() * x).sum().real
    V = _volume(dims)
    psi = torch.empty((V, 3), dtype=torch.complex128, device="cuda")
    psi[op.cb[0]], psi[op.cb[1]] = x, y
    grad = torch.empty_like(links)
    for par in (0, 1):
        s = op.cb[par]
        for mu in range(4):
            # the forward neighbour and sign s of each link: dS = Re Tr(K dU), K = +-2 s psi(x+mu) psi(x)^dag
            a = psi[op.cb[1 - par][op.nb[par][:, 2 * mu]]]
            sign = (op.u[par][:, 2 * mu] * links[mu][s].conj()).sum((1, 2)).real / 3.0
            k = (2.0 if par == 0 else -2.0) * sign.round()
            grad[mu][s] = k[:, None, None] * psi[s].unsqueeze(2) * a.conj().unsqueeze(1)
    return {"action": action, "grad_links": grad, "grad_phi": 2 * x}


def _project(x):
    """Unitary polar factor without the phase of its determinant: Newton's iteration, inverses by cofactors."""
    y = x
    for k in range(9):
        r = [y[..., i, :] for i in range(3)]
        cof = torch.stack([torch.linalg.cross(r[1], r[2], dim=-1), torch.linalg.cross(r[2], r[0], dim=-1),
                           torch.linalg.cross(r[0], r[1], dim=-1)], -2)
        det = (r[0] * cof[..., 0, :]).sum(-1)[..., None, None]
        g = det.abs() ** (-1.0 / 3.0) if k < 4 else 1.0
        y = 0.5 * (g * y + (cof / det).conj() / g)
    det = (y[..., 0, :] * torch.linalg.cross(y[..., 1, :], y[..., 2, :], dim=-1)).sum(-1)
    return y * torch.exp(-1j * det.angle() / 3.0)[..., None, None]


def _exact_hyp(dims, links):
    a1, a2, a3 = 0.75, 0.6, 0.3
    grid = tuple(reversed(dims))  # (t, z, y, x)
    u = links.reshape((4,) + grid + (3, 3))

    def shift(f, mu, n):  # f(x + n mu)
        return torch.roll(f, -n, dims=3 - mu)

    def staples(side, mid, mu, d):
        up = _mm(_mm(side, shift(mid, d, 1)), _dag(shift(side, mu, 1)))
        down = _mm(_mm(_dag(side), mid), shift(side, mu, 1))
        return up + shift(down, d, -1)

    vb = {(mu, e): _project((1 - a3) * u[mu] + a3 / 2 * staples(u[e], u[mu], mu, e))
          for mu in range(4) for e in range(4) if e != mu}
    vt = {}
    for mu in range(4):
        for nu in range(4):
            if nu != mu:
                acc = 0
                for r in range(4):
                    if r not in (mu, nu):
                        s = 6 - mu - nu - r
                        acc = acc + staples(vb[r, s], vb[mu, s], mu, r)
                vt[mu, nu] = _project((1 - a2) * u[mu] + a2 / 4 * acc)
    out = torch.empty_like(links)
    for mu in range(4):
        acc = 0
        for nu in range(4):
            if nu != mu:
                acc = acc + staples(vt[nu, mu], vt[mu, nu], mu, nu)
        out[mu] = _project((1 - a1) * u[mu] + a1 / 6 * acc).reshape(-1, 3, 3)
    return out


def _gammas():
    """g_A = g_1^A1 g_2^A2 g_3^A3 g_4^A4 of Euclidean Hermitian gamma matrices, A = 0 .. 15."""
    s = [torch.tensor(m, dtype=torch.complex128) for m in
         ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
    one = torch.eye(2, dtype=torch.complex128)
    g = [torch.kron(s[1], m) for m in s] + [torch.kron(s[0], one)]
    out = []
    for a in range(16):
        m = torch.eye(4, dtype=torch.complex128)
        for mu in range(4):
            if a >> mu & 1:
                m = m @ g[mu]
        out.append(m)
    return out


def _exact_npr(case, dims, links, fields):
    S1, F1, S2, F2 = (int(v) for v in case["spin_taste"].split(","))
    hyp = [d // 2 for d in dims]
    n = hyp[0] * hyp[1] * hyp[2] * hyp[3]
    z = torch.arange(n, device="cuda")
    zc = [z % hyp[0], z // hyp[0] % hyp[1], z // (hyp[0] * hyp[1]) % hyp[2], z // (hyp[0] * hyp[1] * hyp[2])]

    def site(a):
        x = [2 * zc[mu] + (a >> mu & 1) for mu in range(4)]
        return x[0] + dims[0] * (x[1] + dims[1] * (x[2] + dims[2] * x[3]))

    sites = [site(a) for a in range(16)]
    w = {(a, a): torch.eye(3, dtype=torch.complex128, device="cuda").expand(n, 3, 3) for a in range(16)}
    for level in range(1, 5):  # the average over the shortest paths, by the direction of the last step
        for a in range(16):
            for d in range(16):
                if bin(a ^ d).count("1") != level:
                    continue
                acc = 0
                for mu in range(4):
                    if (a ^ d) >> mu & 1:
                        q = d ^ (1 << mu)
                        link = links[mu][sites[min(q, d)]]
                        acc = acc + _mm(w[a, q], link if d > q else _dag(link))
                w[a, d] = acc / level
    g = _gammas()

    def weight(s, f, a, b):
        return float((torch.trace(g[a].conj().T @ g[s] @ g[b] @ g[f].conj().T) / 4).real)

    f = [[v[sites[a]] for a in range(16)] for v in fields]
    o = torch.zeros(n, dtype=torch.complex128, device="cuda")
    for a in range(16):
        b = a ^ S1 ^ F1
        for c in range(16):
            d = c ^ S2 ^ F2
            t1 = (f[0][a].unsqueeze(2) * w[a, d] * f[3][d].unsqueeze(1)).sum((1, 2))
            t2 = (f[2][c].unsqueeze(2) * w[c, b] * f[1][b].unsqueeze(1)).sum((1, 2))
            o += weight(S1, F1, a, b) * weight(S2, F2, c, d) * t1 * t2
    total = complex(o.sum())
    return {"hypercubes": o, "sum_re": total.real, "sum_im": total.imag}


def exact(case, seed):
    kind = case["kind"]
    if max(_volume(_dims(text)) for text in case["lat"].split(";")) > 2e6:
        return None  # the plain solve would take minutes
    ins = _inputs(case, seed)
    dims, links, vecs = ins[0]
    if kind == "op":
        op = _Op(dims, links)
        if case["op"] == "mdagm":
            return op.a(vecs[0], 0.05)
        return op.half(1 if case["op"] == "dslash_oe" else 0, vecs[0])
    if kind == "solve":
        return _exact_solve(case, dims, links, vecs)
    if kind == "ragged":
        return [_exact_solve(case, d, u, v) for d, u, v in ins]
    if kind == "step":
        return _exact_step(case, dims, links, vecs[0])
    if kind == "hyp":
        return _exact_hyp(dims, links)
    return _exact_npr(case, dims, links, vecs)
