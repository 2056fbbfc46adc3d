"""What the performance of this framework is measured on.

A case is one call of the public Python binding on one lattice: the Dslash and the normal operator, the
solvers (single mass in both modes, multi-shift, batched, flexible with the learned preconditioner), the
preconditioner network forward and backward, the HISQ link construction and the loading of a
configuration. `kind` names the call; the other entries are its sizes and options.

Solvers run at a relative residual of 1e-11, as the action of an accept/reject step and the pseudofermion
heat bath need it (molecular-dynamics forces take less). Their number of iterations is a property of the
gauge field: work() counts the nominal number that fields of this distribution take.
"""

import math
import os

import numpy as np
import torch

import paper_1611_00728_gb300 as sq

TOL = 1e-11
PARAMS = os.path.join(os.path.dirname(os.path.abspath(sq.__file__)), "trained", "fcg_network_16x16x16x16.npy")


def listed():
    return [
        # the smallest call: one FP32 Dslash on a small lattice (latency of a call and of one launch)
        {"name": "dslash f32 8^4", "kind": "dslash", "prec": "f32", "lx": 8, "ly": 8, "lz": 8, "lt": 8, "recon": False},
        # the operator of the mixed solvers on a production lattice, 12-real long links
        {"name": "normal op f32 32^4", "kind": "normal", "prec": "f32", "lx": 32, "ly": 32, "lz": 32, "lt": 32,
         "recon": True},
        # a propagator on a small ragged lattice: the solver's latency per iteration
        {"name": "cg mixed 10x12x14x16", "kind": "cg", "mode": "mixed", "lx": 10, "ly": 12, "lz": 14, "lt": 16,
         "recon": True, "mass": 0.01},
        # the headline solve
        {"name": "cg mixed 32^4", "kind": "cg", "mode": "mixed", "lx": 32, "ly": 32, "lz": 32, "lt": 32,
         "recon": True, "mass": 0.01},
        # the paper's arithmetic: everything in double precision
        {"name": "cg f64 16^3x32", "kind": "cg", "mode": "f64", "lx": 16, "ly": 16, "lz": 16, "lt": 32, "recon": False,
         "mass": 0.02},
        # the multi-mass solve of RHMC
        {"name": "multishift 11 mixed 32^4", "kind": "multishift", "mode": "mixed", "lx": 32, "ly": 32, "lz": 32,
         "lt": 32, "recon": True, "shifts": 11},
        # many sources on ensembles of two volumes in one solve
        {"name": "batched 8 rhs 16^4 24^4", "kind": "batched", "lx": 16, "ly": 16, "lz": 16, "lt": 16, "nrhs": 8,
         "lx2": 24, "ly2": 24, "lz2": 24, "lt2": 24, "recon": True, "mass": 0.02},
        # the preconditioner alone, in its default arithmetic
        {"name": "network 24^4", "kind": "network", "lx": 24, "ly": 24, "lz": 24, "lt": 24},
        # the preconditioned solve, channel mixing on the tensor cores
        {"name": "fcg bf16 16^4", "kind": "fcg", "mixing": "bf16", "lx": 16, "ly": 16, "lz": 16, "lt": 16,
         "recon": True, "mass": 0.005},
        # the backward direction: loss and gradient of one training pair on the training lattice
        {"name": "network gradient 16^4", "kind": "gradient", "lx": 16, "ly": 16, "lz": 16, "lt": 16, "norm": 2},
        # fat and long links of a new configuration, on the device
        {"name": "hisq 24^3x32", "kind": "hisq", "lx": 24, "ly": 24, "lz": 24, "lt": 32},
        # a configuration from host memory, installed and used once
        {"name": "load links 16^4", "kind": "load", "lx": 16, "ly": 16, "lz": 16, "lt": 16, "recon": True,
         "eight": False},
    ]


# kind: (share of draws, largest volume): no drawn case costs more than the largest listed one
_DRAWS = {"dslash": (2, 1 << 20), "normal": (2, 1 << 20), "cg": (4, 1 << 19), "multishift": (2, 1 << 18),
          "batched": (1, 1 << 17), "network": (2, 1 << 19), "fcg": (1, 1 << 17), "gradient": (2, 1 << 17),
          "hisq": (2, 440000), "load": (1, 1 << 17)}


def _draw_dims(rng, vmax):
    """Even extents from 4 to 40, ragged, with the volume spread over its logarithm up to vmax."""
    want = math.exp(rng.uniform(math.log(4 * 4 * 4 * 6), math.log(vmax)))
    d = [max(4, min(40, 2 * round(want ** 0.25 * rng.uniform(0.7, 1.4) / 2))) for _ in range(4)]
    while d[0] * d[1] * d[2] * d[3] > vmax:
        k = max(range(4), key=lambda j: d[j])
        d[k] -= 2
    return dict(zip(("lx", "ly", "lz", "lt"), d))


def draw(rng):
    kind = rng.choice([k for k, (n, _) in _DRAWS.items() for _ in range(n)])
    c = {"kind": kind, **_draw_dims(rng, _DRAWS[kind][1])}
    if kind in ("dslash", "normal", "cg", "multishift", "batched", "fcg", "load"):
        c["recon"] = rng.random() < 0.5
    if kind in ("dslash", "normal", "load"):
        c["eight"] = rng.random() < 0.2
    if kind == "dslash":
        c["prec"] = rng.choice(["f32", "f32", "f64", "ff"])
    if kind == "normal":
        c["prec"] = rng.choice(["f32", "f64"])
    if kind in ("cg", "multishift"):
        c["mode"] = rng.choice(["mixed", "mixed", "f64"])
    if kind in ("cg", "batched", "fcg"):
        c["mass"] = round(math.exp(rng.uniform(math.log(0.005), math.log(0.1))), 4)
    if kind == "multishift":
        c["shifts"] = rng.randint(1, 14)
    if kind == "batched":
        c["nrhs"] = rng.randint(1, 12)
        c.update({k + "2": v for k, v in _draw_dims(rng, _DRAWS[kind][1]).items()})
    if kind == "fcg":
        c["mixing"] = rng.choice(["fp32", "bf16"])
    if kind == "gradient":
        c["norm"] = rng.choice([1, 2])
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dims(c, suffix=""):
    return tuple(c[k + suffix] for k in ("lx", "ly", "lz", "lt"))


def _volume(L):
    return L[0] * L[1] * L[2] * L[3]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _mm(a, b):
    """3x3 complex products over the leading dimensions."""
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _thin(L, seed, width=0.3):
    """Random SU(3) links exp(i width H) near the identity, complex128 [V][4][3][3] on the device."""
    n = _volume(L) * 4
    g = torch.randn(n, 8, dtype=torch.float64, device="cuda", generator=_gen(seed)) * (0.5 * width)
    h = torch.zeros(n, 3, 3, dtype=torch.complex128, device="cuda")
    g8 = g[:, 7] / math.sqrt(3.0)
    h[:, 0, 0], h[:, 1, 1], h[:, 2, 2] = g[:, 2] + g8, g8 - g[:, 2], -2 * g8
    for (i, j), (a, b) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
        h[:, i, j] = torch.complex(g[:, a], -g[:, b])
        h[:, j, i] = torch.complex(g[:, a], g[:, b])
    h = 1j * h
    u = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(h).clone()
    for k in range(10, 0, -1):  # Horner form of the exponential series
        u = _mm(h, u) / k
        u.diagonal(dim1=-2, dim2=-1).add_(1.0)
    r0 = u[:, 0] / u[:, 0].norm(dim=-1, keepdim=True)
    r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.norm(dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], dim=-2).reshape(_volume(L), 4, 3, 3)


def _roll(a, L, mu, k):
    """a(n + k mu) for a field [V, ...] in lexicographic order."""
    v = a.reshape((L[3], L[2], L[1], L[0]) + tuple(a.shape[1:]))
    return torch.roll(v, -k, dims=3 - mu).reshape(a.shape)


def _fat_long(L, seed):
    """Fat links 0.9 W and long links -1/24 W W W of one thin field, complex128 [V][4][3][3] on the device."""
    w = _thin(L, seed)
    lng = torch.empty_like(w)
    for mu in range(4):
        wm = w[:, mu]
        lng[:, mu] = _mm(_mm(wm, _roll(wm, L, mu, 1)), _roll(wm, L, mu, 2)) * (-1.0 / 24.0)
    return 0.9 * w, lng


def _lattice(c, seed, suffix=""):
    L = _dims(c, suffix)
    lat = sq.Lattice(L)
    fat, lng = (t.cpu().numpy() for t in _fat_long(L, seed))
    lat.load_links(fat, lng, recon12=c.get("recon", False), eight_way=c.get("eight", False))
    return lat


_PREC = {"f32": sq.F32, "f64": sq.F64, "ff": sq.FF}


def _vector(L, seed, prec="f64", count=None):
    """Gaussian colour vector(s) of one parity in the device layout."""
    shape = (() if count is None else (count,)) + (3, _volume(L) // 2, 2)
    v = torch.randn(shape, dtype=torch.float64, device="cuda", generator=_gen(seed))
    if prec == "f32":
        return v.float()
    if prec == "ff":
        hi = v.float()
        return torch.stack([hi, (v - hi.double()).float()], dim=-1).reshape(shape[:-1] + (4,))
    return v


def _shifts(c):
    return np.logspace(-4, 0, c["shifts"]).tolist()


def _network(lat, c):
    net = sq.Network(lat)
    net.set_params(np.load(PARAMS))
    if c.get("mixing") == "bf16":
        net.set_mixing(sq.NN_MIX_BF16)
    return net


def _pair(c, seed):
    """A training pair on the device: an error e and its residual r = A e, in FP64 before rounding."""
    L = _dims(c)
    lat = _lattice(c, seed)
    e = _vector(L, seed + 1)
    r = lat.normal_op(_GRAD_SIGMA, e, lat.new_spinor())
    return lat, r.float(), e.float()


_GRAD_SIGMA = 4 * 0.005 ** 2


def prepare(case, seed):
    c, seed, k = case, 1000003 * (seed % (1 << 30)) + 17, case["kind"]
    L = _dims(c)
    if k in ("dslash", "normal"):
        lat = _lattice(c, seed)
        return {"case": c, "lat": lat, "psi": _vector(L, seed + 1, c["prec"]), "out": lat.new_spinor(_PREC[c["prec"]])}
    if k in ("cg", "fcg"):
        lat = _lattice(c, seed)
        s = {"case": c, "lat": lat, "b": _vector(L, seed + 1), "x": lat.new_spinor()}
        if k == "fcg":
            s["net"] = _network(lat, c)
        return s
    if k == "multishift":
        lat = _lattice(c, seed)
        return {"case": c, "lat": lat, "b": _vector(L, seed + 1), "xs": [lat.new_spinor() for _ in _shifts(c)]}
    if k == "batched":
        lats = [_lattice(c, seed), _lattice(c, seed + 1, "2")]
        bs = [_vector(_dims(c), seed + 2, count=c["nrhs"]), _vector(_dims(c, "2"), seed + 3, count=c["nrhs"])]
        return {"case": c, "lats": lats, "bs": bs, "xs": [torch.zeros_like(b) for b in bs]}
    if k == "network":
        lat = _lattice(c, seed)
        return {"case": c, "lat": lat, "net": _network(lat, c), "r": _vector(L, seed + 1, "f32"),
                "z": lat.new_spinor(sq.F32)}
    if k == "gradient":
        lat, r, e = _pair(c, seed)
        net = _network(lat, c)
        net.set_loss(c["norm"])
        return {"case": c, "lat": lat, "net": net, "r": r, "e": e}
    if k == "hisq":
        thin = torch.view_as_real(_thin(L, seed)).contiguous()
        ws = torch.empty(sq.hisq_workspace_bytes(L), dtype=torch.uint8, device="cuda")
        return {"case": c, "thin": thin, "fat": torch.empty_like(thin), "lng": torch.empty_like(thin), "ws": ws}
    if k == "load":
        fat, lng = (t.cpu().numpy() for t in _fat_long(L, seed))
        lat = sq.Lattice(L)
        return {"case": c, "lat": lat, "fat": fat, "lng": lng, "psi": _vector(L, seed + 1),
                "psi32": _vector(L, seed + 1, "f32"), "out": lat.new_spinor(), "out32": lat.new_spinor(sq.F32)}
    raise ValueError(k)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    s, c = state, state["case"]
    k = c["kind"]
    if k == "dslash":
        return s["lat"].dslash(0, s["psi"], s["out"], _PREC[c["prec"]])
    if k == "normal":
        return s["lat"].normal_op(0.01, s["psi"], s["out"], _PREC[c["prec"]])
    if k == "cg":
        s["x"].zero_()
        s["lat"].cg_solve(c["mass"], s["b"], s["x"], tol=TOL, mode=sq.MODE_MIXED if c["mode"] == "mixed" else sq.MODE_F64)
        return s["x"]
    if k == "multishift":
        s["lat"].multishift_cg_solve(_shifts(c), s["b"], s["xs"], tol=TOL,
                                     mode=sq.MODE_MIXED if c["mode"] == "mixed" else sq.MODE_F64)
        return s["xs"]
    if k == "batched":
        for x in s["xs"]:
            x.zero_()
        sq.cg_solve_batched(s["lats"], [c["mass"]] * 2, s["bs"], s["xs"], tol=TOL)
        return s["xs"]
    if k == "network":
        return s["net"].apply(s["r"], s["z"])
    if k == "fcg":
        s["x"].zero_()
        s["net"].fcg_solve(c["mass"], s["b"], s["x"], tol=TOL)
        return s["x"]
    if k == "gradient":
        loss, grad = s["net"].loss_grad(_GRAD_SIGMA, s["r"], s["e"])
        return {"loss": loss, "gradient": grad}
    if k == "hisq":
        sq.hisq_smear(_dims(c), s["thin"], s["fat"], s["lng"], s["ws"])
        return {"fat": s["fat"], "long": s["lng"]}
    if k == "load":
        s["lat"].load_links(s["fat"], s["lng"], recon12=c["recon"], eight_way=c["eight"])
        return {"f64": s["lat"].dslash(0, s["psi"], s["out"]),
                "f32": s["lat"].dslash(0, s["psi32"], s["out32"], sq.F32)}
    raise ValueError(k)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _iterations(V, mass=0.0):
    """Nominal CG iterations to TOL on fields of this distribution: the smallest mode falls with the extent."""
    root = (34 + 5.5 * V ** 0.25) / 9.6  # square root of the condition number at small masses
    return 0.5 * math.log(2 / TOL) * min(root, math.sqrt(1 + 18.0 / (4 * mass * mass))) if mass else \
        0.5 * math.log(2 / TOL) * root


def work(case):
    c, k = case, case["kind"]
    L = _dims(c)
    V = _volume(L)
    Vh = V // 2
    wide = 2 if c.get("prec") in ("f64", "ff") or c.get("mode") == "f64" else 1
    links = 8 * (72 + (72 if wide == 2 or not c.get("recon") else 48)) * wide  # bytes of a site's 16 links
    vec = 24 * wide
    if k == "dslash":
        return {"bytes": Vh * (links + 2 * vec), "flops": 1146 * Vh}
    if k == "normal":
        return {"bytes": Vh * (2 * links + 3 * vec), "flops": 2 * 1146 * Vh}
    if k in ("cg", "fcg"):
        it = _iterations(V, c["mass"])
        if k == "fcg":  # about 0.57 of the iterations, each with the network's three layers
            it *= 0.57
            return {"bytes": it * Vh * (2 * links + 12 * vec + 3344), "flops": it * Vh * (2 * 1146 + 42000)}
        return {"bytes": it * Vh * (2 * links + 12 * vec), "flops": it * Vh * (2 * 1146 + 60)}
    if k == "multishift":
        it = _iterations(V)
        return {"bytes": it * Vh * (2 * links + 8 * vec + 48 * c["shifts"]), "flops": it * Vh * (2 * 1146 + 24 * c["shifts"])}
    if k == "batched":
        n, b, f = c["nrhs"], 0.0, 0.0
        for s in ("", "2"):
            v = _volume(_dims(c, s))
            it = _iterations(v, c["mass"])
            b += it * v / 2 * (2 * links + 12 * vec * n)
            f += it * v / 2 * n * (2 * 1146 + 60)
        return {"bytes": b, "flops": f}
    if k == "network":  # links once a layer, the hidden activations once each way
        return {"bytes": V * (3 * 288 + 2 * 2 * 192) + 48 * Vh, "flops": V * (18432 + 2 * 960 + 960)}
    if k == "gradient":
        return {"bytes": V * (6 * 288 + 8 * 192) + 96 * Vh, "flops": 3 * V * (18432 + 3 * 960)}
    if k == "hisq":  # thin in, fat and long out, and W once each way between the two levels
        return {"bytes": V * 4 * 144 * 5, "flops": V * 4 * 98 * 198}
    if k == "load":  # both fields read once and written once in each precision
        return {"bytes": V * 4 * (2 * 144 + 2 * 144 + 72 + (48 if c["recon"] else 72)), "flops": 2 * 1146 * Vh}
    raise ValueError(k)


# ---------------------------------------------------------------------------
# the same in 64 bits, by plain tensor operations on lexicographic full-lattice fields
# ---------------------------------------------------------------------------
def _coords(L):
    t, z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda") for n in (L[3], L[2], L[1], L[0])], indexing="ij")
    return [a.reshape(-1) for a in (x, y, z, t)]


def _fold(L, u, hop):
    """Links with the staggered phases and the antiperiodic time boundary of their forward hop."""
    x, y, z, t = _coords(L)
    out = u.clone()
    for mu, e in enumerate((torch.zeros_like(x), x, x + y, x + y + z)):
        s = (1 - 2 * (e & 1)).double()
        if mu == 3:
            s = s * torch.where(t + hop >= L[3], -1.0, 1.0)
        out[:, mu] *= s[:, None, None]
    return out


def _parity(L):
    x, y, z, t = _coords(L)
    return [torch.nonzero(((x + y + z + t) & 1) == p)[:, 0] for p in (0, 1)]


def _full(L, v, par):
    """Device vector (3, Vh, 2) or (3, Vh, 4) of one parity -> complex128 [V][3], zero elsewhere."""
    v = v.double()
    if v.shape[-1] == 4:
        v = torch.stack([v[..., 0] + v[..., 1], v[..., 2] + v[..., 3]], dim=-1)
    out = torch.zeros(_volume(L), 3, dtype=torch.complex128, device="cuda")
    out[_parity(L)[par]] = torch.view_as_complex(v.contiguous()).T
    return out


def _half(L, f, par):
    """complex128 [V][3] -> (3, Vh, 2) float64 of one parity."""
    return torch.view_as_real(f[_parity(L)[par]].T.contiguous())


def _mv(u, v):
    return (u * v[:, None, :]).sum(-1)


def _mdv(u, v):
    return (u.conj() * v[:, :, None]).sum(-2)


class _Operator:
    def __init__(self, L, fat, lng):
        self.L, self.links = L, ((1, _fold(L, fat, 1)), (3, _fold(L, lng, 3)))

    def d(self, v):
        out = torch.zeros_like(v)
        for hop, u in self.links:
            for mu in range(4):
                out += _mv(u[:, mu], _roll(v, self.L, mu, hop))
                out -= _roll(_mdv(u[:, mu], v), self.L, mu, -hop)
        return out

    def normal(self, sigma, v):
        return sigma * v - self.d(self.d(v))


def _solve(op, sigmas, b):
    """(sigma_s - D D)^-1 b for all sigmas (the smallest first): multi-shift CG in 64 bits, then each solution
    corrected from its own residual."""
    xs = _krylov(op, sigmas, b)
    if len(sigmas) == 1:
        return [xs[0] + _krylov(op, sigmas, b - op.normal(sigmas[0], xs[0]), 1e-5)[0]]
    return xs


def _krylov(op, sigmas, b, eps=1e-14):
    n = len(sigmas)
    x = [torch.zeros_like(b) for _ in range(n)]
    p = [b.clone() for _ in range(n)]
    r = b.clone()
    rr = bb = float((r.abs() ** 2).sum())
    z, zp, alpha_p, beta_p = [1.0] * n, [1.0] * n, 1.0, 0.0
    for _ in range(4000):
        ap = op.normal(sigmas[0], p[0])
        a = rr / float((p[0].conj() * ap).sum().real)
        r -= a * ap
        new = float((r.abs() ** 2).sum())
        beta = new / rr
        for s in range(n):
            if z[s] == 0.0:
                continue
            zn = z[s] * zp[s] * alpha_p / (a * beta_p * (zp[s] - z[s]) + zp[s] * alpha_p * (1 + (sigmas[s] - sigmas[0]) * a))
            x[s] += (a * zn / z[s]) * p[s]
            p[s].mul_(beta * (zn / z[s]) ** 2).add_(r, alpha=zn)
            zp[s], z[s] = z[s], (zn if abs(zn) * math.sqrt(new / bb) > eps or s == 0 else 0.0)
        alpha_p, beta_p, rr = a, beta, new
        if math.sqrt(rr / bb) < eps:
            break
    return x


def _taps(op_links, L, h):
    """The nine tap fields of h [C][V][3]: self, then for each direction forward and backward."""
    out = [h]
    for mu in range(4):
        u = op_links[:, mu]
        out.append(torch.stack([_mv(u, _roll(v, L, mu, 1)) for v in h]))
        out.append(torch.stack([_roll(_mdv(u, v), L, mu, -1) for v in h]))
    return out


def _net_weights():
    p = torch.from_numpy(np.load(PARAMS)).cuda()
    nw = sq.NN_LAYERS[-1][0].stop
    return torch.cat([p[:nw].bfloat16().double(), p[nw:].double()])


def _net(L, fat, w, r):
    """The network on a full-lattice field r [V][3] that is zero on odd sites; w: the 1472 weights in 64 bits."""
    W = [torch.view_as_complex(w[sl].reshape(shape + (2,))) for sl, shape in sq.NN_LAYERS]
    gates = [(w[a], w[b]) for a, b in sq.NN_GATES]
    links = _fold(L, fat, 1)
    scale = torch.sqrt(3.0 * _volume(L) / 2 / (r.abs() ** 2).sum())
    h = (r * scale)[None]
    for k in range(3):
        taps = _taps(links, L, h)
        h = sum(torch.einsum("oc,cva->ova", W[k][t], taps[t]) for t in range(9))
        if k < 2:
            a, b = gates[k]
            n2 = (h.real ** 2 + h.imag ** 2).sum(-1, keepdim=True)
            h = h * torch.sigmoid(a[:, None, None] * n2 + b[:, None, None])
    even = _parity(L)[0]
    z = torch.zeros_like(r)
    z[even] = h[0][even] / scale
    return z


def _wrap(L, U, X, mu, d):
    """Both signs of direction d around a direction-mu field X: U_d(n) X(n+d) U_d(n+mu)^+ and its backward mate."""
    ud = U[:, d]
    um = _roll(ud, L, mu, 1)
    fwd = _mm(_mm(ud, _roll(X, L, d, 1)), um.mH)
    return fwd, _roll(_mm(_mm(ud.mH, X), um), L, d, -1)


def _smear(L, U, c1, c3, c5, c7, cl):
    out = torch.empty_like(U)
    for mu in range(4):
        dirs = [d for d in range(4) if d != mu]
        S = {d: _wrap(L, U, U[:, mu], mu, d) for d in dirs}
        S3 = {d: S[d][0] + S[d][1] for d in dirs}
        f = c1 * U[:, mu] + c3 * sum(S3.values())
        for nu in dirs:
            rho, sig = [d for d in dirs if d != nu]
            z = c5 * (S3[rho] + S3[sig]) + c7 * (sum(_wrap(L, U, S3[sig], mu, rho)) + sum(_wrap(L, U, S3[rho], mu, sig)))
            f = f + sum(_wrap(L, U, z, mu, nu))
            if cl:  # twice the same direction and sign
                f = f + cl * (_wrap(L, U, S[nu][0], mu, nu)[0] + _wrap(L, U, S[nu][1], mu, nu)[1])
        out[:, mu] = f
    return out


def _unitary(V):
    """The unitary polar factor by Newton's iteration."""
    X = V
    for _ in range(60):
        r0, r1, r2 = X[..., 0, :], X[..., 1, :], X[..., 2, :]
        cof = torch.stack([torch.linalg.cross(r1, r2, dim=-1), torch.linalg.cross(r2, r0, dim=-1),
                           torch.linalg.cross(r0, r1, dim=-1)], dim=-2)
        inv_t = cof / (r0 * cof[..., 0, :]).sum(-1)[..., None, None]
        new = 0.5 * (X + inv_t.conj())
        step = float((new - X).abs().max())
        X = new
        if step < 1e-15:
            break
    return X


def exact(case, seed):
    c, seed, k = case, 1000003 * (seed % (1 << 30)) + 17, case["kind"]
    L = _dims(c)
    if k == "hisq":
        if _volume(L) > 1 << 19:
            return None
        W = _unitary(_smear(L, _thin(L, seed), 1 / 8, 1 / 16, 1 / 64, 1 / 384, 0.0))
        lng = torch.empty_like(W)
        for mu in range(4):
            w = W[:, mu]
            lng[:, mu] = _mm(_mm(w, _roll(w, L, mu, 1)), _roll(w, L, mu, 2)) * (-1.0 / 24.0)
        fat = _smear(L, W, 1.0, 1 / 16, 1 / 64, 1 / 384, -1 / 8)
        return {"fat": torch.view_as_real(fat), "long": torch.view_as_real(lng)}
    if k == "batched":
        out = []
        for j, s in enumerate(("", "2")):
            Lj = _dims(c, s)
            op = _Operator(Lj, *_fat_long(Lj, seed + j))
            bs = _vector(Lj, seed + 2 + j, count=c["nrhs"])
            out.append(torch.stack([_half(Lj, _solve(op, [4 * c["mass"] ** 2], _full(Lj, b, 0))[0], 0) for b in bs]))
        return out
    fat, lng = _fat_long(L, seed)
    if k in ("network", "gradient"):
        w = _net_weights()
        if k == "network":
            return _half(L, _net(L, fat, w, _full(L, _vector(L, seed + 1, "f32"), 0)), 0)
        op = _Operator(L, fat, lng)
        e64 = _full(L, _vector(L, seed + 1), 0)
        r = _full(L, _half(L, op.normal(_GRAD_SIGMA, e64), 0).float(), 0)
        e = _full(L, _half(L, e64, 0).float(), 0)
        w = w.requires_grad_(True)
        d = _net(L, fat, w, r) - e
        Ad = op.normal(_GRAD_SIGMA, d)
        if c["norm"] == 2:
            loss = (Ad.abs() ** 2).sum() / (r.abs() ** 2).sum()
        else:
            loss = (d.conj() * Ad).sum().real / (e.conj() * r).sum().real
        loss.backward()
        return {"loss": float(loss.detach()), "gradient": w.grad.detach()}
    op = _Operator(L, fat, lng)
    if k in ("dslash", "normal"):
        v = _full(L, _vector(L, seed + 1, c["prec"]), 1 if k == "dslash" else 0)
        y = _half(L, op.d(v) if k == "dslash" else op.normal(0.01, v), 0)
        if c["prec"] != "ff":
            return y
        hi = y.float()  # laid out as the pair it is returned as
        return torch.stack([hi.double(), y - hi.double()], dim=-1).reshape(y.shape[:-1] + (4,))
    if k == "load":
        return {"f64": _half(L, op.d(_full(L, _vector(L, seed + 1), 1)), 0),
                "f32": _half(L, op.d(_full(L, _vector(L, seed + 1, "f32"), 1)), 0)}
    b = _full(L, _vector(L, seed + 1), 0)
    sigmas = _shifts(c) if k == "multishift" else [4 * c["mass"] ** 2]
    xs = [_half(L, x, 0) for x in _solve(op, sigmas, b)]
    return xs if k == "multishift" else xs[0]
