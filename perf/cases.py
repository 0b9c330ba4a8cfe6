"""What this library is measured on: one pass of each routine, as a program that uses it calls it.

Sizes come from the repository's own configurations, tests and benchmark: the 8^4 solve (m = 0.1),
the four 32^4 sources (m = 0.01), the nine-shift multi-shift solve, the 1-16-16-16-1 network, the
24^4 and 32^4 volumes of the link construction and the two forces, and ragged lattices such as
those of the tests.  Inputs are synthetic, made on the GPU from the seed alone: SU(3) thin links
near exp(0.3 i H), Gaussian sources and residuals.  Solves run to 1e-12, the accuracy to which the
library's training targets (and an action evaluation) are computed, so that what is compared is
the solution and not where the iteration stopped.
"""

import math

import torch

import paper_1712_00143_gb300 as stag

EPS = 0.3  # thin links exp(i EPS H), reunitarised
C1, C_STAPLE, C3 = 1.0, 0.125, -1.0 / 24.0  # fat and Naik coefficients of the workloads
CHANNELS = (1, 16, 16, 16, 1)
TOL = 1e-12
# tadpole-improved one-loop gauge action at u0 = 0.87 (beta = 6)
BETA, U0 = 6.0, 0.87
_ALPHA_S = -4.0 * math.log(U0) / 3.0684
C_PL, C_RT, C_PG = 1.0, -(1.0 + 0.4805 * _ALPHA_S) / (20.0 * U0**2), -0.03325 * _ALPHA_S / U0**2


def listed():
    return [
        # The smallest call: M on the 8^4 test lattice in FP64, where launches are all there is
        # (a caller's own residual check, or its own Krylov loop on a small lattice).
        {"name": "apply_small", "kind": "apply", "dims": "8x8x8x8", "prec": "fp64", "recon": 18, "mass": 0.1},
        # The single-vector FP32 Dslash on the paper's 24^4 per-node volume (its single-GPU L^4 sweep).
        {"name": "dslash_fp32", "kind": "dslash", "dims": "24x24x24x24", "prec": "fp32", "recon": 12, "nrhs": 1,
         "parity": 1},
        # Eight vectors on one gauge field at the headline volume: the operator of the batched groups.
        {"name": "dslash_multi", "kind": "dslash", "dims": "32x32x32x32", "prec": "fp32", "recon": 12, "nrhs": 8,
         "parity": 0},
        # Fixed-point links with FP32 vectors, a ragged lattice, and a vector count that is no power of two.
        {"name": "dslash_fx16", "kind": "dslash", "dims": "28x20x18x36", "prec": "fx16l", "recon": 12, "nrhs": 6,
         "parity": 1},
        # One mixed-precision solve on the small lattice: some 180 short iterations, launch-bound.
        {"name": "cg_small", "kind": "cg", "dims": "8x8x8x8", "mode": "mixed32", "recon": 18, "mass": 0.1},
        # The headline: four sources on one 32^4 lattice solved together.
        {"name": "batch_sources", "kind": "batch", "dims": "32x32x32x32", "mode": "mixed32", "recon": 12, "nrhs": 4,
         "mass": 0.01},
        # The production solver of the paper: multi-shift CG in double precision.
        {"name": "multishift_fp64", "kind": "multishift", "dims": "16x16x16x32", "mode": "plain64", "recon": 18,
         "shifts": 9, "mass": 0.02},
        # One application of the learned preconditioner (each flexible-CG iteration has one).
        {"name": "net_apply", "kind": "net", "dims": "24x24x24x24", "recon": 12},
        # One training pair: loss and weight gradient, forward and backward, on a ragged lattice.
        {"name": "net_grad", "kind": "grad", "dims": "16x20x12x24", "recon": 12, "mass": 0.01},
        # Fat and Naik links from thin links, once per trajectory step, at the headline volume.
        {"name": "links", "kind": "links", "dims": "32x32x32x32"},
        # The gauge force at the paper's per-node volume.
        {"name": "gauge_force", "kind": "gauge", "dims": "24x24x24x24"},
        # The fermion force of an eight-term rational approximation, a ragged lattice.
        {"name": "fermion_force", "kind": "fermion", "dims": "20x24x16x28", "terms": 8},
    ]


def _draw_dims(rng, lo, hi):
    """Even extents >= 4 (odd multiples of two among them) with lo <= volume <= hi, spread over the logarithm."""
    while True:
        side = math.exp(rng.uniform(math.log(lo), math.log(hi))) ** 0.25
        d = [max(4, 2 * int(round(side * math.exp(rng.uniform(-0.35, 0.35)) / 2))) for _ in range(4)]
        if lo <= d[0] * d[1] * d[2] * d[3] <= hi:
            return "x".join(map(str, d))


def draw(rng):
    kind = rng.choice(["apply", "dslash", "dslash", "cg", "batch", "multishift", "net", "grad", "links", "gauge",
                       "fermion"])
    recon = rng.choice([12, 18])
    if kind == "apply":
        return {"kind": kind, "dims": _draw_dims(rng, 4**4, 32**4), "recon": recon,
                "prec": rng.choice(["fp64", "fp32", "fx16", "fx16l", "df64"]), "mass": rng.choice([0.01, 0.05, 0.1])}
    if kind == "dslash":
        return {"kind": kind, "dims": _draw_dims(rng, 4**4, 32**4), "recon": recon,
                "prec": rng.choice(["fp64", "fp32", "fp16", "fx16", "fx16l"]), "nrhs": rng.randint(1, 8),
                "parity": rng.randint(0, 1)}
    if kind == "cg":
        return {"kind": kind, "dims": _draw_dims(rng, 8**4, 20**4), "recon": recon,
                "mode": rng.choice(["plain64", "mixed32", "mixedfx16", "mixed16l"]),
                "mass": rng.choice([0.02, 0.05, 0.1])}
    if kind == "batch":
        return {"kind": kind, "dims": _draw_dims(rng, 8**4, 24**4), "recon": recon,
                "mode": rng.choice(["mixed32", "mixed32", "mixed16l"]), "nrhs": rng.randint(2, 8),
                "mass": rng.choice([0.01, 0.02, 0.05])}
    if kind == "multishift":
        return {"kind": kind, "dims": _draw_dims(rng, 8**4, 18**4), "recon": recon,
                "mode": rng.choice(["plain64", "plain64", "mixed32"]), "shifts": rng.randint(4, 12),
                "mass": rng.choice([0.02, 0.05])}
    if kind in ("net", "grad"):
        c = {"kind": kind, "dims": _draw_dims(rng, 8**4, 28**4 if kind == "net" else 20**4), "recon": recon}
        return dict(c, mass=0.01) if kind == "grad" else c
    c = {"kind": kind, "dims": _draw_dims(rng, 6**4, 28**4)}
    return dict(c, terms=rng.randint(1, 12)) if kind == "fermion" else c


# ------------------------------------------------------------------ inputs
def _dims(case):
    return tuple(int(v) for v in case["dims"].split("x"))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _normals(gen, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=gen)


def _complex(gen, *shape):
    return torch.complex(_normals(gen, *shape), _normals(gen, *shape))


def _thin(dims, gen):
    """SU(3) links near exp(i EPS H), H traceless Hermitian: the exponential to second order, reunitarised."""
    n = 4 * _volume(dims)
    a = _complex(gen, 3, 3, n)
    h = 0.5 * (a + a.transpose(0, 1).conj())
    tr = (h[0, 0] + h[1, 1] + h[2, 2]) / 3.0
    for i in range(3):
        h[i, i] -= tr
    rows = []
    for i in range(2):
        u = [1j * EPS * h[i, j] - 0.5 * EPS**2 * sum(h[i, k] * h[k, j] for k in range(3)) for j in range(3)]
        u[i] = u[i] + 1.0
        for q in rows:
            s = sum(q[j].conj() * u[j] for j in range(3))
            u = [u[j] - s * q[j] for j in range(3)]
        norm = torch.sqrt(sum(v.real**2 + v.imag**2 for v in u))
        rows.append([v / norm for v in u])
    p, q = rows
    rows.append([(p[1] * q[2] - p[2] * q[1]).conj(), (p[2] * q[0] - p[0] * q[2]).conj(),
                 (p[0] * q[1] - p[1] * q[0]).conj()])
    return torch.stack([torch.stack(r, -1) for r in rows], -2).reshape(_volume(dims), 4, 3, 3).contiguous()


def _net_params(gen):
    """A flat parameter array like a trained network's: per layer W[9][Cout][Cin], then b[Cout] of a hidden layer."""
    out = []
    for l in range(len(CHANNELS) - 1):
        ci, co = CHANNELS[l], CHANNELS[l + 1]
        w = 0.3 / math.sqrt(9 * ci) * _normals(gen, 9, co, ci)
        w[0] += torch.eye(co, ci, dtype=torch.float64, device="cuda")
        out.append(w.reshape(-1))
        if l + 2 < len(CHANNELS):
            out.append(-1.0 + 0.5 * _normals(gen, co))
    return torch.cat(out).float()


def _shifts(case):
    """10^(-4 + k/2), k = 0, 1, ..."""
    return [10.0 ** (-4.0 + 0.5 * k) for k in range(case["shifts"])]


def _inputs(case, seed):
    """Every input of a case, from the seed alone."""
    dims = _dims(case)
    vh = _volume(dims) // 2
    gen = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)
    kind = case["kind"]
    d = {"thin": _thin(dims, gen)}
    if kind in ("apply", "cg", "multishift", "net"):
        d["b"] = _complex(gen, vh, 3)
    elif kind in ("dslash", "batch"):
        d["b"] = _complex(gen, *([vh, 3] if case["nrhs"] == 1 else [case["nrhs"], vh, 3]))
    elif kind == "grad":
        d["b"], d["e"] = _complex(gen, vh, 3), _complex(gen, vh, 3)
    elif kind == "fermion":
        d["x"], d["y"] = _complex(gen, case["terms"], vh, 3), _complex(gen, case["terms"], vh, 3)
        d["alphas"] = [0.05 + 0.35 * i / max(1, case["terms"] - 1) for i in range(case["terms"])]
    if kind in ("net", "grad"):
        d["params"] = _net_params(gen)
    return d


_COPIES = {"plain64": ("fp64",), "mixed32": ("fp64", "fp32", "df64"), "mixedfx16": ("fp64", "fx16", "df64"),
           "mixed16l": ("fp64", "fx16", "df64")}


def prepare(case, seed):
    d, dims, kind = _inputs(case, seed), _dims(case), case["kind"]
    state = {"case": case, "dims": dims}
    if kind in ("links", "gauge", "fermion"):
        state.update(d)
        state["out"] = torch.empty_like(d["thin"])
        if kind == "links":
            state["out2"] = torch.empty_like(d["thin"])
        return state
    fat, lng = stag.stag_build_links(dims, d.pop("thin"), c1=C1, c_staple=C_STAPLE, c3=C3)
    if kind in ("apply", "dslash"):
        copies = ({"fx16l": "fx16"}.get(case["prec"], case["prec"]),)
    elif kind in ("net", "grad"):
        copies = ("fp32",)
    else:
        copies = _COPIES[case["mode"]]
    mask = 0
    for c in copies:
        mask |= 1 << stag.PREC[c]
    state["h"] = stag.stag_load_links(dims, fat, lng, recon_long=case["recon"], long_coeff=C3, prec_mask=mask)
    state.update(d)
    if kind == "multishift":
        state["x"] = [torch.zeros_like(d["b"]) for _ in range(case["shifts"])]
    elif kind != "grad":
        state["x"] = torch.zeros_like(d["b"])
    if kind in ("net", "grad"):
        state["net"] = stag.stag_net_create(CHANNELS, seed=1)
        stag.stag_net_set_params(state["net"], d["params"].cpu().numpy())
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "apply":
        return stag.stag_apply_m(state["h"], state["x"], state["b"], case["mass"], prec=case["prec"])
    if kind == "dslash":
        return stag.stag_dslash(state["h"], state["x"], state["b"], case["parity"], prec=case["prec"],
                                nrhs=case["nrhs"])
    if kind == "cg":
        stag.stag_cg(state["h"], state["x"], state["b"], case["mass"], mode=case["mode"], tol=TOL)
        return state["x"]
    if kind == "batch":
        stag.stag_batch_solve([(state["h"], state["x"], state["b"], case["nrhs"], case["mass"])], mode=case["mode"],
                              tol=TOL)
        return state["x"]
    if kind == "multishift":
        stag.stag_multishift_cg(state["h"], state["x"], state["b"], case["mass"], _shifts(case), mode=case["mode"],
                                tol=TOL)
        return state["x"]
    if kind == "net":
        return stag.stag_net_apply(state["net"], state["h"], state["x"], state["b"])
    if kind == "grad":
        loss, grad = stag.stag_net_loss_grad(state["net"], state["h"], state["b"], state["e"], loss="residual",
                                             mass=case["mass"])
        return {"loss": loss, "grad": grad}
    if kind == "links":
        fat, lng = stag.stag_build_links(state["dims"], state["thin"], state["out"], state["out2"], c1=C1,
                                         c_staple=C_STAPLE, c3=C3)
        return {"fat": fat, "lng": lng}
    if kind == "gauge":
        return stag.stag_gauge_force(state["dims"], state["thin"], BETA, C_PL, C_RT, C_PG, force=state["out"])
    return stag.stag_fermion_force(state["dims"], state["thin"], state["x"], state["y"], state["alphas"], c1=C1,
                                   c_staple=C_STAPLE, c3=C3, force=state["out"])


# ------------------------------------------------------------------ what a pass cannot do without
_CPLX = {"fp64": 16, "fp32": 8, "fp16": 4, "fx16": 4, "fx16l": 4, "df64": 16}  # bytes of one stored link entry
_SLOPPY = {"plain64": "fp64", "mixed32": "fp32", "mixedfx16": "fx16", "mixed16l": "fx16l"}


def _link_bytes(prec, recon):
    """The sixteen hop matrices of one output site (two Naik rows of three with 12 reals)."""
    return 8 * (9 + (6 if recon == 12 and prec not in ("fp64", "df64") else 9)) * _CPLX[prec]


def _iterations(case):
    """CG iterations to TOL: half log(2/tol) times the root of the condition number, whose lower end is the
    mass and the lattice's lowest momentum (about 2.2/L on these smooth fields; upper end about 9.9)."""
    low = (2.2 / max(_dims(case))) ** 2 + case["mass"] ** 2
    return 0.5 * math.log(2.0 / TOL) * math.sqrt(9.9 / low)


def work(case):
    dims, kind = _dims(case), case["kind"]
    v = _volume(dims)
    vh = v // 2
    vec = 48 * vh  # one canonical field
    if kind == "apply":
        return {"bytes": 2 * vec + 2 * vh * _link_bytes(case["prec"], case["recon"]), "flops": vh * (2 * 1146 + 12)}
    if kind == "dslash":
        n = case["nrhs"]
        return {"bytes": 2 * n * vec + vh * _link_bytes(case["prec"], case["recon"]), "flops": n * vh * 1146}
    if kind in ("cg", "batch", "multishift"):
        prec = _SLOPPY[case["mode"]]
        n, ns = case.get("nrhs", 1), case.get("shifts", 1)
        per = {"fp64": 48, "fx16": 16}.get(prec, 24) * vh
        it = _iterations(case)
        # per iteration: the links once, and per system p, t, Ap, x and r through the operator and the updates
        one = 2 * vh * _link_bytes(prec, case["recon"]) + n * 11 * per + (ns - 1) * 4 * per
        return {"bytes": it * one + (n + ns) * vec, "flops": it * n * vh * (2 * 1146 + 72 + 24 * (ns - 1))}
    if kind in ("net", "grad"):
        # activations could stay on chip: the field in and out, and the fat links of both parities
        fwd = v * sum(2 * 9 * 6 * ci * co + 8 * 66 * min(ci, co) for ci, co in zip(CHANNELS, CHANNELS[1:]))
        links = v * 8 * 9 * 8
        if kind == "net":
            return {"bytes": 2 * vec + links, "flops": fwd}
        return {"bytes": 2 * vec + links + 2 * vh * _link_bytes("fp32", case["recon"]), "flops": 3 * fwd + 4 * vh * 1146}
    if kind == "links":
        return {"bytes": 3 * v * 576, "flops": v * 44 * 216}
    if kind == "gauge":
        return {"bytes": 2 * v * 576, "flops": v * 196 * 216}
    n = case["terms"]
    return {"bytes": 2 * v * 576 + 2 * n * vec, "flops": v * (112 * 216 + 4 * 144 * n)}


# ------------------------------------------------------------------ the same results in plain torch, 64 bits
_AXIS = {0: 3, 1: 2, 2: 1, 3: 0}


def _grid(dims):
    return (dims[3], dims[2], dims[1], dims[0])


def _shift(a, mu, k):
    return torch.roll(a, -k, _AXIS[mu])


def _dag(a):
    return a.conj().transpose(-1, -2)


def _mm(a, b):
    return torch.matmul(a, b)


def _coords(dims):
    lt, lz, ly, lx = _grid(dims)
    ar = lambda n: torch.arange(n, device="cuda")  # noqa: E731
    return torch.meshgrid(ar(lt), ar(lz), ar(ly), ar(lx), indexing="ij")[::-1]  # x, y, z, t


def _eta(dims, mu):
    c = _coords(dims)
    s = sum(c[:mu]) if mu else torch.zeros_like(c[0])
    return 1.0 - 2.0 * (s % 2).double()


def _fat_naik(dims, u):
    """u: list of four grids of 3x3 matrices."""
    fat, lng = [], []
    for mu in range(4):
        s = C1 * u[mu]
        for nu in range(4):
            if nu == mu:
                continue
            up = _mm(_mm(u[nu], _shift(u[mu], nu, 1)), _dag(_shift(u[nu], mu, 1)))
            dn = _mm(_mm(_dag(u[nu]), u[mu]), _shift(u[nu], mu, 1))
            s = s + C_STAPLE * (up + _shift(dn, nu, -1))
        fat.append(s)
        lng.append(C3 * _mm(_mm(u[mu], _shift(u[mu], mu, 1)), _shift(u[mu], mu, 2)))
    return fat, lng


def _split(dims, links):
    return [links[:, mu].reshape(*_grid(dims), 3, 3) for mu in range(4)]


def _join(links):
    return torch.stack([f.reshape(-1, 3, 3) for f in links], 1)


class _Operator:
    """The hops of one gauge field as sixteen matrices and neighbour indices per site of each parity."""

    def __init__(self, dims, thin):
        fat, lng = _fat_naik(dims, _split(dims, thin))
        x, y, z, t = _coords(dims)
        lex = torch.arange(_volume(dims), device="cuda").reshape(_grid(dims))
        par = ((x + y + z + t) % 2).reshape(-1)
        self.sites = [torch.nonzero(par == p).reshape(-1) for p in (0, 1)]
        self.w, self.nb = [[], []], [[], []]
        for mu in range(4):
            eta = _eta(dims, mu)[..., None, None]
            for f, k in ((fat[mu], 1), (lng[mu], 3)):
                for m, s in ((0.5 * eta * f, k), (-0.5 * eta * _dag(_shift(f, mu, -k)), -k)):
                    n = (_shift(lex, mu, s) // 2).reshape(-1)
                    m = m.reshape(-1, 3, 3)
                    for p in (0, 1):
                        self.w[p].append(m[self.sites[p]].contiguous())
                        self.nb[p].append(n[self.sites[p]])

    def hop(self, v, p):
        """D v on parity p; v: [..., V/2, 3] of the other parity."""
        out = 0
        for w, n in zip(self.w[p], self.nb[p]):
            out = out + (w * v[..., n, :].unsqueeze(-2)).sum(-1)
        return out

    def apply(self, v, c):
        return c * v - self.hop(self.hop(v, 1), 0)


def _solve(op, b, c, tol=2e-14, most=4000):
    """(c - D D) x = b for a block of systems ([n, V/2, 3], c: [n, 1, 1]), conjugate gradients with restarts."""
    dot = lambda p, q: (p.conj() * q).real.sum((-1, -2), keepdim=True)  # noqa: E731
    x, bb = torch.zeros_like(b), dot(b, b)
    for _ in range(4):
        r = b - op.apply(x, c)
        p, rr = r.clone(), dot(r, r)
        if float((rr / bb).max()) <= tol**2:
            break
        goal = torch.maximum(bb * tol**2, rr * 1e-20)
        for i in range(most):
            ap = op.apply(p, c)
            live = (rr > 0.25 * goal).double()
            a = live * rr / dot(p, ap)
            x, r = x + a * p, r - a * ap
            new = dot(r, r)
            p, rr = r + live * (new / rr) * p, new
            if i % 16 == 15 and bool((rr <= goal).all()):
                break
    return x


def _layers(params):
    """[(W, b or None)] in 64 bits; weights as the network holds them, rounded to bfloat16."""
    at, out = 0, []
    for l in range(len(CHANNELS) - 1):
        ci, co = CHANNELS[l], CHANNELS[l + 1]
        w = params[at:at + 9 * co * ci].bfloat16().double().reshape(9, co, ci)
        at += 9 * co * ci
        b = None
        if l + 2 < len(CHANNELS):
            b = params[at:at + co].double()
            at += co
        out.append((w, b))
    return out


def _network(dims, thin, layers, r):
    """(prediction on even sites for the scaled residual, scale)"""
    fat = _fat_naik(dims, _split(dims, thin))[0]
    hops = []
    for mu in range(4):
        eta = 0.5 * _eta(dims, mu)[..., None, None]
        hops.append((eta * fat[mu], mu, 1))
        hops.append((-eta * _dag(_shift(fat[mu], mu, -1)), mu, -1))
    x, y, z, t = _coords(dims)
    even = ((x + y + z + t) % 2 == 0).reshape(-1)
    scale = math.sqrt(r.shape[0]) / torch.linalg.vector_norm(r)
    h = torch.zeros(_volume(dims), 3, 1, dtype=torch.complex128, device="cuda")
    h[even, :, 0] = r * scale
    for w, b in layers:
        h = h.reshape(*_grid(dims), 3, h.shape[-1])
        pre = torch.matmul(h, w[0].T.to(h.dtype))
        for d, (m, mu, s) in enumerate(hops):
            pre = pre + torch.matmul(_mm(m, _shift(h, mu, s)), w[d + 1].T.to(h.dtype))
        if b is not None:
            n2 = (pre.real**2 + pre.imag**2).sum(-2, keepdim=True)
            pre = pre * torch.sigmoid(n2 - b)
        h = pre
    return h.reshape(-1, 3)[even], scale


def _ta(m):
    a = 0.5 * (m - _dag(m))
    tr = torch.diagonal(a, dim1=-2, dim2=-1).sum(-1) / 3.0
    return a - tr[..., None, None] * torch.eye(3, dtype=m.dtype, device=m.device)


def _force(dims, thin, action, sign):
    """sign * TA[U Z] with dS = Re Tr[dU Z], by differentiating the action."""
    u = [f.clone().requires_grad_(True) for f in _split(dims, thin)]
    g = torch.autograd.grad(action(u), u)
    return _join([sign * _ta(_mm(f.detach(), _dag(d))) for f, d in zip(u, g)])


def _retr(a, b):
    """sum Re Tr(a b)"""
    return (a * b.transpose(-1, -2)).real.sum()


def _gauge_action(u):
    """-beta/3 sum c Re Tr W over plaquettes, rectangles and parallelograms."""
    def path(steps):
        """Product along signed steps from every site."""
        m, at = None, [0, 0, 0, 0]
        for d, s in steps:
            if s < 0:
                at[d] -= 1
            link = u[d]
            for k in range(4):
                if at[k]:
                    link = _shift(link, k, at[k])
            link = link if s > 0 else _dag(link)
            if s > 0:
                at[d] += 1
            m = link if m is None else _mm(m, link)
        return m

    def loop(steps):
        n = len(steps) // 2
        back = [(d, -s) for d, s in reversed(steps[n:])]
        return _retr(path(steps[:n]), _dag(path(back)))

    total = 0.0
    for a in range(4):
        for b in range(4):
            if a < b:
                total = total + C_PL * loop([(a, 1), (b, 1), (a, -1), (b, -1)])
            if a != b:
                total = total + C_RT * loop([(a, 1), (a, 1), (b, 1), (a, -1), (a, -1), (b, -1)])
            for c in range(b + 1, 4):
                if a < b:
                    for sb in (1, -1):
                        for sc in (1, -1):
                            total = total + C_PG * loop([(a, 1), (b, sb), (c, sc), (a, -1), (b, -sb), (c, -sc)])
    return -BETA / 3.0 * total


def _fermion_action(dims, d):
    """The action's link dependence at fixed outer products: sum Re Tr[F G^F + L G^L]."""
    x, y, z, t = _coords(dims)
    par = ((x + y + z + t) % 2).reshape(-1)
    n = len(d["alphas"])
    full = torch.zeros(n, _volume(dims), 3, dtype=torch.complex128, device="cuda")
    full[:, par == 0], full[:, par == 1] = d["x"], d["y"]
    full = full.reshape(n, *_grid(dims), 3)
    sign = (1.0 - 2.0 * par.double()).reshape(*_grid(dims), 1, 1)
    gf, gl = [], []
    for mu in range(4):
        w = sign * _eta(dims, mu)[..., None, None]
        for g, k in ((gf, 1), (gl, 3)):
            g.append(w * sum(a * _shift(f, mu, k).unsqueeze(-1) * f.conj().unsqueeze(-2)
                             for a, f in zip(d["alphas"], full)))

    def action(u):
        fat, lng = _fat_naik(dims, u)
        return sum(_retr(fat[mu], gf[mu]) + _retr(lng[mu], gl[mu]) for mu in range(4))

    return action


def exact(case, seed):
    d, dims, kind = _inputs(case, seed), _dims(case), case["kind"]
    vh = _volume(dims) // 2
    if kind == "links":
        fat, lng = _fat_naik(dims, _split(dims, d["thin"]))
        return {"fat": _join(fat), "lng": _join(lng)}
    if kind == "gauge":
        return _force(dims, d["thin"], _gauge_action, -1.0)
    if kind == "fermion":
        return _force(dims, d["thin"], _fermion_action(dims, d), -1.0)
    if kind == "net":
        z, scale = _network(dims, d["thin"], _layers(d["params"]), d["b"])
        return z / scale
    if kind == "grad":
        layers = _layers(d["params"])
        leaves = [t.requires_grad_(True) for w, b in layers for t in ((w, b) if b is not None else (w,))]
        op = _Operator(dims, d["thin"])
        z, scale = _network(dims, d["thin"], layers, d["b"])
        diff = op.apply(z, case["mass"] ** 2) - d["b"] * scale
        loss = (diff.real**2 + diff.imag**2).sum() / vh
        g = torch.autograd.grad(loss, leaves)
        return {"loss": float(loss.detach()), "grad": torch.cat([t.reshape(-1) for t in g])}
    op = _Operator(dims, d["thin"])
    if kind == "apply":
        return op.apply(d["b"], case["mass"] ** 2)
    if kind == "dslash":
        return op.hop(d["b"], case["parity"])
    m2 = case["mass"] ** 2
    if kind == "cg":
        return _solve(op, d["b"][None], torch.full((1, 1, 1), m2, dtype=torch.float64, device="cuda"))[0]
    if kind == "batch":
        if case["nrhs"] * vh > 700_000:
            return None  # too long in plain torch
        return _solve(op, d["b"], torch.full((case["nrhs"], 1, 1), m2, dtype=torch.float64, device="cuda"))
    if case["shifts"] * vh > 700_000:
        return None
    c = torch.tensor([m2 + s for s in _shifts(case)], dtype=torch.float64, device="cuda").reshape(-1, 1, 1)
    return list(_solve(op, d["b"].expand(case["shifts"], vh, 3).contiguous(), c))
