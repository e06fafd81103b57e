"""Performance cases of the Clover-Wilson SAP-BiCGStab solver.

A case is one call (or one short sequence of calls) that a user's program
makes through the public entry points, on inputs of the kind it meets: a
seeded SU(3) gauge field U = exp(i eps H) per lattice and Gaussian or point
sources.  ``listed()`` holds the standing cases, ``draw()`` gives more of the
same ranges; ``exact()`` repeats a case in float64 with plain torch.

Kinds
-----
apply     D or D^dag on device-resident fields (internal layout), 1 to 12
          right-hand sides: what an iterative solver, an eigensolver or a
          molecular-dynamics step of the user's own calls in a loop.
canonical Lattice.apply_D on a canonical complex128 field: import, float64
          operator, export; the checking and analysis path.
sap       the SAP preconditioner (M_SAP or A M_SAP) on device-resident fields.
config    a new gauge configuration arrives: set_gauge, set_params,
          build_clover, then the first applications of D and C_inv to a field.
solve     D x = b for one or several right-hand sides (a propagator is the
          twelve spin-colour point sources together).
train     one differentiable step: the solve as a torch function, its loss
          Re(eta^dag x), and the gradients with respect to b and U.
ragged    many lattices of different sizes solved together.
"""

import math

import torch

from paper_2109_10687_gb300 import binding as B
from paper_2109_10687_gb300.autograd import solve as dirac_solve
from paper_2109_10687_gb300.lattice import Lattice

PREC = {"double": B.PREC_DOUBLE, "single": B.PREC_SINGLE, "half": B.PREC_HALF, "half_gauge": B.PREC_HALF_GAUGE}


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _case(kind, dims, **kw):
    c = {"kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "domain": "4x4x4x4",
         "bc_t": -1, "basis": "chiral", "eps": 0.3, "kappa": 0.125, "csw": 1.0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one D on an 8^4 test lattice, bound by latency
        _case("apply", (8, 8, 8, 8), name="d_f32_8x8x8x8", prec="single", dagger=False, nrhs=1),
        # the operator at the size of a production sub-lattice, bound by memory
        _case("apply", (32, 32, 32, 32), name="d_f32_32x32x32x32", prec="single", dagger=False, nrhs=1),
        # D^dag on a block of twelve vectors (the spin-colour components of a
        # propagator, or a block eigensolver's basis)
        _case("apply", (24, 24, 24, 32), name="ddag_f32_24x24x24x32_rhs12", prec="single", dagger=True, nrhs=12),
        # the preconditioner in its production storage at production size
        _case("sap", (32, 32, 32, 32), name="sap_half_32x32x32x32", prec="half", n_sap=4, n_jac=4, with_A=False,
              nrhs=1, sdom=""),
        # A M_SAP with the published algorithm parameters on 16x6x4x3 domains
        _case("sap", (32, 24, 16, 24), name="sap_16x6x4x3_domains_32x24x16x24", prec="half_gauge", n_sap=4, n_jac=2,
              with_A=True, nrhs=1, sdom="16x6x4x3"),
        # the next configuration of an ensemble
        _case("config", (24, 24, 24, 48), name="config_24x24x24x48"),
        # the smallest solve, with the default parameters
        _case("solve", (8, 8, 8, 8), name="solve_single_8x8x8x8", kappa=0.12, source="gauss", nrhs=1, prec="single",
              inner_tol=1e-6, graph=0, n_sap=4, n_jac=4),
        # extents that only 2^4 domains fit, in the printed gamma basis with periodic time
        _case("solve", (12, 20, 12, 28), name="solve_single_12x20x12x28_domains_2x2x2x2", domain="2x2x2x2",
              basis="paper", bc_t=1, kappa=0.12, source="gauss", nrhs=1, prec="single", inner_tol=1e-6, graph=0,
              n_sap=4, n_jac=4),
        # the flagship solve: float16 storage, device-side inner loop
        _case("solve", (32, 32, 32, 32), name="solve_half_32x32x32x32", source="gauss", nrhs=1, prec="half",
              inner_tol=1e-5, graph=2, n_sap=4, n_jac=4),
        # a point-to-all propagator: twelve right-hand sides at once
        _case("solve", (16, 16, 16, 32), name="propagator_16x16x16x32", eps=0.25, csw=1.1, source="point", nrhs=12,
              prec="half", inner_tol=1e-5, graph=2, n_sap=4, n_jac=4),
        # one step of training through the solve: a configuration, x, and both gradients
        _case("train", (16, 16, 16, 16), name="train_16x16x16x16", kappa=0.12, prec="half", inner_tol=1e-5, graph=2),
        # an ensemble of small lattices of different sizes in one call
        _case("ragged", (8, 8, 8, 8), name="ragged_32_lattices", nlat=32, big=16, prec="half", inner_tol=1e-5,
              graph=2),
    ]


_DOMAINS = {"4x4x4x4": (4, 4, 4, 4), "2x2x2x2": (2, 2, 2, 2), "8x4x4x2": (8, 4, 4, 2), "2x4x2x4": (2, 4, 2, 4)}


def _draw_dims(rng, domain, lo, hi):
    """Extents that fit the domain, the volume spread over [lo, hi] logarithmically."""
    d = [int(v) for v in domain.split("x")]
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    for _ in range(1000):
        dims = [2 * m * rng.randint(1, max(1, 64 // (2 * m))) for m in d]
        v = math.prod(dims)
        if target / 1.5 <= v <= min(target * 1.5, hi):
            return dims
    return [2 * m for m in d]


def draw(rng):
    kind = rng.choice(["apply", "apply", "canonical", "sap", "sap", "config", "solve", "solve", "train", "ragged"])
    dom = rng.choice(["4x4x4x4", "4x4x4x4", "4x4x4x4", "2x2x2x2", "8x4x4x2", "2x4x2x4"])
    common = {"domain": dom, "bc_t": rng.choice([-1, -1, 1]), "basis": rng.choice(["chiral", "chiral", "paper"]),
              "eps": round(rng.uniform(0.2, 0.3), 3), "kappa": round(rng.uniform(0.115, 0.125), 4),
              "csw": rng.choice([1.0, 1.1])}
    if kind == "apply":
        nrhs = rng.choice([1, 1, 2, 3, 5, 12])
        dims = _draw_dims(rng, dom, 4096, 1 << 20 if nrhs == 1 else (1 << 22) // nrhs)
        return _case(kind, dims, prec=rng.choice(["single", "single", "double"]), dagger=rng.random() < 0.5,
                     nrhs=nrhs, **{**common, "basis": "chiral"})
    if kind == "canonical":
        return _case(kind, _draw_dims(rng, dom, 4096, 1 << 19), dagger=rng.random() < 0.5, nrhs=rng.choice([1, 2]),
                     **common)
    if kind == "sap":
        sdom = ""
        prec = rng.choice(["half", "half", "half_gauge", "single"])
        nrhs = rng.choice([1, 1, 2, 3])
        dims = _draw_dims(rng, dom, 4096, (1 << 19) // nrhs)
        if rng.random() < 0.3:
            sd = rng.choice([(16, 6, 4, 3), (8, 6, 4, 3), (16, 6, 4, 6), (8, 4, 4, 4), (6, 6, 6, 4)])
            # stored in 2^4 blocks, which all of these extents allow
            dims = [2 * m * rng.randint(1, 2) for m in sd]
            dims = [2 * v if v % 4 else v for v in dims]
            sdom, prec, nrhs, common["domain"] = "x".join(map(str, sd)), "half_gauge", 1, "2x2x2x2"
        return _case(kind, dims, prec=prec, n_sap=rng.randint(1, 4), n_jac=rng.randint(1, 4),
                     with_A=rng.random() < 0.5, nrhs=nrhs, sdom=sdom, **{**common, "basis": "chiral"})
    if kind == "config":
        return _case(kind, _draw_dims(rng, dom, 4096, 1 << 19), **{**common, "basis": "chiral"})
    if kind == "solve":
        nrhs = rng.choice([1, 1, 2, 12])
        dims = _draw_dims(rng, dom, 4096, (1 << 18) // nrhs if nrhs > 1 else 1 << 18)
        prec = rng.choice(["half", "half_gauge", "single"])
        return _case(kind, dims, source="point" if nrhs > 2 else "gauss", nrhs=nrhs, prec=prec,
                     inner_tol=rng.choice([1e-5, 1e-6]), graph=rng.choice([0, 2]), n_sap=4, n_jac=4, **common)
    if kind == "train":
        return _case(kind, _draw_dims(rng, dom, 4096, 1 << 16), prec=rng.choice(["half", "half_gauge"]),
                     inner_tol=1e-5, graph=2, **common)
    return _case(kind, (8, 8, 8, 8), nlat=rng.choice([3, 7, 16, 24]), big=rng.choice([8, 16]),
                 prec=rng.choice(["half", "half_gauge", "single"]), inner_tol=1e-5, graph=2,
                 **{**common, "domain": "4x4x4x4"})


def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _domain(case):
    return _DOMAINS[case["domain"]]


def _vol(case):
    return math.prod(_dims(case))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _mul3(a, b):
    """Products of stacks of small matrices, elementwise (exact float64 sums)."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _gauge(dims, eps, seed, salt, device):
    """Links exp(i eps H), H = sum_a h_a lambda_a / 2 with h_a ~ N(0, 1):
    [t][z][y][x][mu][3][3] complex128, SU(3) to rounding."""
    lx, ly, lz, lt = dims
    h = torch.randn((lt, lz, ly, lx, 4, 8), generator=_gen(seed, salt, device), device=device, dtype=torch.float64)
    m = torch.zeros((lt, lz, ly, lx, 4, 3, 3), dtype=torch.complex128, device=device)
    off = ((0, 1, 0), (0, 2, 3), (1, 2, 5))
    for i, j, a in off:
        m[..., i, j] = torch.complex(h[..., a], -h[..., a + 1])
        m[..., j, i] = torch.complex(h[..., a], h[..., a + 1])
    r3 = 1.0 / math.sqrt(3.0)
    m[..., 0, 0] = (h[..., 2] + r3 * h[..., 7]).to(torch.complex128)
    m[..., 1, 1] = (-h[..., 2] + r3 * h[..., 7]).to(torch.complex128)
    m[..., 2, 2] = (-2.0 * r3 * h[..., 7]).to(torch.complex128)
    m *= 0.5j * eps / 8.0
    eye = torch.eye(3, dtype=torch.complex128, device=device)
    u = eye + m / 14.0
    for k in range(13, 0, -1):  # Taylor series of exp(i eps H / 8), then three squarings
        u = eye + _mul3(m, u) / k
    for _ in range(3):
        u = _mul3(u, u)
    return u.contiguous()


def _spinor(dims, nrhs, seed, salt, device):
    lx, ly, lz, lt = dims
    shape = ((nrhs,) if nrhs > 1 else ()) + (lt, lz, ly, lx, 3, 4)
    g = _gen(seed, salt, device)
    return torch.complex(torch.randn(shape, generator=g, device=device, dtype=torch.float64),
                         torch.randn(shape, generator=g, device=device, dtype=torch.float64))


def _point_sources(dims, nrhs, seed, device):
    """Unit spin-colour sources at one seeded site."""
    lx, ly, lz, lt = dims
    b = torch.zeros((nrhs, lt, lz, ly, lx, 3, 4), dtype=torch.complex128, device=device)
    g = _gen(seed, 5, "cpu")
    t, z, y, x = (int(torch.randint(0, n, (1,), generator=g)) for n in (lt, lz, ly, lx))
    for r in range(nrhs):
        b[r, t, z, y, x, r // 4, r % 4] = 1.0
    return b


def _source(case, seed, device):
    if case["source"] == "point":
        return _point_sources(_dims(case), case["nrhs"], seed, device)
    return _spinor(_dims(case), case["nrhs"], seed, 2, device)


def _ragged_inputs(case, seed, device):
    """Per lattice: extents in {8, big}, its own links, source and kappa."""
    g = _gen(seed, 7, "cpu")
    lats = []
    for i in range(case["nlat"]):
        # the sizes belong to the case (lattice i of every seed has the same
        # extents), the fields to the seed
        dims = tuple(case["big"] if (i * 5 + mu * 3 + i // 3) % 2 else 8 for mu in range(4))
        kappa = 0.115 + 0.01 * float(torch.rand((1,), generator=g, dtype=torch.float64))
        lats.append((dims, kappa, _gauge(dims, case["eps"], seed, 100 + 2 * i, device),
                     _spinor(dims, 1, seed, 101 + 2 * i, device)))
    return lats


def _params(case, n_sap=4, n_jac=4):
    p = B.qcd_solve_params_default()
    p.tol, p.inner_tol, p.sap_prec, p.use_graph = 1e-10, case["inner_tol"], PREC[case["prec"]], case["graph"]
    p.n_sap, p.n_jac = n_sap, n_jac
    return p


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    kind, dims = case["kind"], _dims(case)
    st = {"case": case}
    if kind == "ragged":
        st["lats"], st["bs"], st["xs"] = [], [], []
        for dims_i, kappa, u, b in _ragged_inputs(case, seed, dev):
            st["lats"].append(Lattice(dims_i, (4, 4, 4, 4), case["bc_t"], case["basis"], dev)
                              .setup(u, kappa, case["csw"]))
            st["bs"].append(torch.view_as_real(b).contiguous())
            st["xs"].append(torch.zeros_like(st["bs"][-1]))
        st["batch"] = _Batch(st["lats"])
        st["params"] = _params(case)
        return st
    lat = Lattice(dims, _domain(case), case["bc_t"], case["basis"], dev)
    u = _gauge(dims, case["eps"], seed, 1, dev)
    st["lat"] = lat
    if kind == "config":
        st["u"] = u
        st["in"] = lat.to_internal(_spinor(dims, 1, seed, 2, dev), "double")
        st["d"], st["c"] = lat.field("double"), lat.field("double")
        return st
    if kind == "train":
        st["u"] = u.requires_grad_(True)
        st["b"] = _spinor(dims, 1, seed, 2, dev).requires_grad_(True)
        st["eta"] = _spinor(dims, 1, seed, 3, dev)
        st["params"] = _params(case)
        return st
    lat.setup(u, case["kappa"], case["csw"])
    if kind == "solve":
        st["b"] = _source(case, seed, dev)
        st["params"] = _params(case, case["n_sap"], case["n_jac"])
        return st
    psi = _spinor(dims, case["nrhs"], seed, 2, dev)
    if kind == "canonical":
        st["psi"] = psi
        return st
    prec = case["prec"] if kind == "apply" else "single"
    st["in"] = lat.to_internal(psi, prec, case["nrhs"])
    st["out"] = lat.field(prec, case["nrhs"])
    if kind == "sap" and case["sdom"]:
        B.qcd_set_sap_domain(lat.ctx, [int(v) for v in case["sdom"].split("x")])
    return st


class _Batch:
    """The handle of a ragged batch, destroyed before its lattices."""

    def __init__(self, lats):
        self.lats = lats
        self.handle = B.qcd_batch_create([lat.ctx for lat in lats])

    def __del__(self):
        try:
            B.qcd_batch_destroy(self.handle)
        except Exception:
            pass


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        B.qcd_apply_D(st["lat"].ctx, st["out"], st["in"], PREC[case["prec"]], int(case["dagger"]), case["nrhs"])
        return st["out"].view(torch.float64 if case["prec"] == "double" else torch.float32)
    if kind == "canonical":
        return torch.view_as_real(st["lat"].apply_D(st["psi"], "double", case["dagger"], case["nrhs"]))
    if kind == "sap":
        ctx, prec = st["lat"].ctx, PREC[case["prec"]]
        if case["nrhs"] == 1:
            B.qcd_sap_apply(ctx, st["out"], st["in"], case["n_sap"], case["n_jac"], prec, int(case["with_A"]))
        else:
            B.qcd_sap_apply_nrhs(ctx, st["out"], st["in"], case["nrhs"], case["n_sap"], case["n_jac"], prec,
                                 int(case["with_A"]))
        return st["out"].view(torch.float32)
    if kind == "config":
        lat = st["lat"]
        lat.setup(st["u"], case["kappa"], case["csw"])
        B.qcd_apply_D(lat.ctx, st["d"], st["in"], B.PREC_DOUBLE)
        B.qcd_apply_clover(lat.ctx, st["c"], st["in"], B.PREC_DOUBLE, 1)
        return [st["d"].view(torch.float64), st["c"].view(torch.float64)]
    if kind == "solve":
        x, _, _ = st["lat"].solve(st["b"], nrhs=case["nrhs"], params=st["params"])
        return torch.view_as_real(x)
    if kind == "train":
        st["b"].grad = st["u"].grad = None
        x = dirac_solve(st["b"], st["u"], st["lat"], case["kappa"], case["csw"], st["params"])
        loss = (st["eta"].conj() * x).sum().real
        loss.backward()
        return [torch.view_as_real(t) for t in (x.detach(), st["b"].grad, st["u"].grad)]
    B.qcd_batch_solve(st["batch"].handle, st["xs"], st["bs"], st["params"])
    return list(st["xs"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _sap_flops(case, n_sap, n_jac, d):
    """Per site, in the constants of the published accounting: 168 per hop,
    600 per C_inv multiply and update; the hops inside and between domains
    counted apart."""
    inside = sum((m - 1) / m for m in d)  # per direction pair: share of hops that stay
    f_in = 600 + 2 * 168 * inside
    face = 1 - math.prod(max(m - 2, 0) / m for m in d)
    f_out = 2 * 168 * (4 - inside) + 600 * face
    tot = 0.0
    for sweep in range(n_sap + 1):
        for colour in (0, 1):
            tot += 0.5 * ((f_out if sweep or colour else 0) + n_jac * f_in + (f_in + 48 if sweep < n_sap else 0))
    return tot


def _solve_work(case, vol, nrhs, n_sap, n_jac, d):
    # about eight iterations of two A M_SAP each at these kappas, two residuals
    per = 8 * 2 * (_sap_flops(case, n_sap, n_jac, d) + 1824) + 2 * 1824
    return {"bytes": vol * (4 * 18 * 8 + 72 * 8 + nrhs * 2 * 192), "flops": vol * nrhs * per}


def work(case):
    kind, v = case["kind"], _vol(case)
    nrhs = case.get("nrhs", 1)
    if kind == "apply":
        if case["prec"] == "double":
            return {"bytes": v * (576 + 576 + nrhs * 384), "flops": v * nrhs * 1824}
        # SU(3) links need two rows (48 B), the clover term two Hermitian blocks
        return {"bytes": v * (192 + 288 + nrhs * 192), "flops": v * nrhs * 1824}
    if kind == "canonical":
        return {"bytes": v * (576 + 576 + nrhs * 384), "flops": v * nrhs * 1824}
    if kind == "sap":
        d = [int(k) for k in (case["sdom"] or case["domain"]).split("x")]
        e = 4 if case["prec"] == "single" else 2
        return {"bytes": v * (72 * e + 72 * e + nrhs * 192),
                "flops": v * nrhs * (_sap_flops(case, case["n_sap"], case["n_jac"], d)
                                     + (1824 if case["with_A"] else 0))}
    if kind == "config":
        # U in, a field in, two fields out; eight 3x3 products per plaquette
        # and plane, two 6x6 Hermitian inversions, D and C_inv
        return {"bytes": v * (576 + 3 * 192), "flops": v * (6 * 8 * 216 + 2 * 1000 + 1824 + 552)}
    if kind == "solve":
        return _solve_work(case, v, nrhs, case["n_sap"], case["n_jac"], _domain(case))
    if kind == "train":
        w = _solve_work(case, v, 2, 4, 4, _domain(case))
        # the clover term and its force on top
        return {"bytes": w["bytes"] + v * 576 * 2, "flops": w["flops"] + v * (6 * 8 * 216 + 2000 + 4 * 48 * 216)}
    out = {"bytes": 0, "flops": 0}
    for i in range(case["nlat"]):
        dims = [case["big"] if (i * 5 + mu * 3 + i // 3) % 2 else 8 for mu in range(4)]
        w = _solve_work(case, math.prod(dims), 1, 4, 4, (4, 4, 4, 4))
        out = {k: out[k] + w[k] for k in out}
    return out


def tolerance(case):
    """About four times the difference seen between the library's result and
    the same call in plain float64 torch: float64 sums 2.7e-16 (in another
    order up to 5e-16), float32 operators 9.5e-8, the SAP 1.5e-7 in float32,
    1.9e-4 with float16 links and C_inv, 2.6e-4 with float16 vectors as well;
    solves up to 6.4e-10, which is what the stopping test at a residual of 1e-10
    leaves; the float32 force of a training step 1.5e-7."""
    kind = case["kind"]
    if kind in ("canonical", "config") or (kind == "apply" and case["prec"] == "double"):
        return {"rel": 2e-15}
    if kind == "apply":
        return {"rel": 4e-7}
    if kind == "sap":
        return {"rel": {"single": 6e-7, "half_gauge": 8e-4, "half": 1e-3}[case["prec"]]}
    if kind == "train":
        return {"rel": 6e-7}
    return {"rel": 3e-9}


# ---------------------------------------------------------------------------
# the same in float64 with plain torch
# ---------------------------------------------------------------------------
_AXIS = (3, 2, 1, 0)  # site axis of mu = x, y, z, t in [t][z][y][x]
# gamma_mu in the printed basis: entry (row, column) -> value
_GAMMA = [
    [[0, 0, 0, 1j], [0, 0, 1j, 0], [0, -1j, 0, 0], [-1j, 0, 0, 0]],
    [[0, 0, 0, 1], [0, 0, -1, 0], [0, -1, 0, 0], [1, 0, 0, 0]],
    [[0, 0, 1j, 0], [0, 0, 0, -1j], [-1j, 0, 0, 0], [0, 1j, 0, 0]],
    [[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, -1, 0], [0, 0, 0, -1]],
]


def _dag(m):
    return m.transpose(-1, -2).conj()


class _Plain:
    """D = 1 + C - kappa H on a canonical complex128 field [t][z][y][x][3][4]."""

    def __init__(self, u, kappa, csw, bc_t, basis):
        self.u, self.kappa, self.csw, self.bc_t = u, kappa, csw, bc_t
        g = torch.tensor(_GAMMA, dtype=torch.complex128, device=u.device)
        if basis == "chiral":
            i2 = torch.eye(2, dtype=torch.complex128, device=u.device)
            s = torch.cat([torch.cat([i2, i2], 1), torch.cat([i2, -i2], 1)], 0) / math.sqrt(2.0)
            g = torch.stack([s @ m @ s.conj().T for m in g])
            g = torch.view_as_complex(torch.view_as_real(g).round())  # entries are 0, +-1, +-i
        self.g = g
        self.perm, self.phase = [], []
        for mu in range(4):
            p = g[mu].abs().argmax(1)
            self.perm.append(p)
            self.phase.append(g[mu][torch.arange(4, device=u.device), p])
        self.g5 = g[0] @ g[1] @ g[2] @ g[3]
        self.m = self._clover()

    def _at(self, d, **off):
        m = self.u[..., d, :, :]
        for k, s in off.items():
            m = torch.roll(m, -s, _AXIS[int(k[1:])])
        return m

    def _clover(self):
        """1 + C as a 12x12 matrix per site, index (colour, spin)."""
        u, g = self.u, self.g
        c = torch.zeros(u.shape[:4] + (3, 4, 3, 4), dtype=torch.complex128, device=u.device)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a, b = f"d{mu}", f"d{nu}"
                at = self._at
                q = _mul3(_mul3(at(mu), at(nu, **{a: 1})), _mul3(_dag(at(mu, **{b: 1})), _dag(at(nu))))
                q = q + _mul3(_mul3(at(nu), _dag(at(mu, **{a: -1, b: 1}))),
                              _mul3(_dag(at(nu, **{a: -1})), at(mu, **{a: -1})))
                q = q + _mul3(_mul3(_dag(at(mu, **{a: -1})), _dag(at(nu, **{a: -1, b: -1}))),
                              _mul3(at(mu, **{a: -1, b: -1}), at(nu, **{b: -1})))
                q = q + _mul3(_mul3(_dag(at(nu, **{b: -1})), at(mu, **{b: -1})),
                              _mul3(at(nu, **{a: 1, b: -1}), _dag(at(mu))))
                f = (q - _dag(q)) / 8.0
                sig = 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])
                c = c + f[..., :, None, :, None] * sig[:, None, :]
        m = (1j * self.kappa * self.csw * c).reshape(u.shape[:4] + (12, 12))
        return m + torch.eye(12, dtype=torch.complex128, device=u.device)

    def _site(self, m, x):
        return (m * x.reshape(x.shape[:-2] + (1, 12))).sum(-1).reshape(x.shape)

    def inverse(self):
        """(1 + C)^-1 per site."""
        if not hasattr(self, "minv"):
            flat = self.m.reshape(-1, 12, 12)
            self.minv = torch.cat([torch.linalg.inv(c) for c in flat.split(1 << 17)]).reshape(self.m.shape)
        return self.minv

    def clover_inv(self, x):
        return self._site(self.inverse(), x)

    def _gm(self, mu, x):
        return self.phase[mu] * x[..., self.perm[mu]]

    def _shift(self, x, mu, n):
        y = torch.roll(x, -n, _AXIS[mu])
        if mu == 3 and self.bc_t != 1:
            sg = torch.ones(x.shape[0], dtype=torch.float64, device=x.device)
            sg[-1 if n > 0 else 0] = self.bc_t
            y = y * sg.reshape((-1,) + (1,) * (x.dim() - 1))
        return y

    def hop(self, x, fmask=None, bmask=None):
        out = None
        for mu in range(4):
            um = self.u[..., mu, :, :]
            f = _mul3(um, self._shift(x, mu, 1))
            f = f - self._gm(mu, f)
            b = self._shift(_mul3(_dag(um), x), mu, -1)
            b = b + self._gm(mu, b)
            if fmask is not None:
                f, b = f * fmask[mu], b * bmask[mu]
            out = f + b if out is None else out + f + b
        return out

    def D(self, x):
        return self._site(self.m, x) - self.kappa * self.hop(x)

    def Ddag(self, x):
        g5 = self.g5.diagonal() if torch.count_nonzero(self.g5 - torch.diag(self.g5.diagonal())) == 0 else None
        if g5 is not None:
            return g5 * self.D(g5 * x)
        return self.D(x @ self.g5.T) @ self.g5.T

    # red/black Schwarz (Algorithms 1 and 2) on domains d
    def set_domain(self, d):
        lt, lz, ly, lx = self.u.shape[:4]
        dev = self.u.device
        ax = [torch.arange(n, device=dev) for n in (lx, ly, lz, lt)]
        shape = [(1, 1, 1, -1), (1, 1, -1, 1), (1, -1, 1, 1), (-1, 1, 1, 1)]
        co = [a.reshape(s) for a, s in zip(ax, shape)]
        col = sum(c // m for c, m in zip(co, d)) % 2
        self.cmask = [(col == k).double()[..., None, None] for k in (0, 1)]
        one = torch.ones((lt, lz, ly, lx), dtype=torch.float64, device=dev)
        self.fin = [(one * (c % m != m - 1))[..., None, None] for c, m in zip(co, d)]
        self.bin = [(one * (c % m != 0))[..., None, None] for c, m in zip(co, d)]
        self.fout, self.bout = [1 - m for m in self.fin], [1 - m for m in self.bin]

    def _block(self, x, row, col):
        xc = self.cmask[col] * x
        if row == col:
            h = self.hop(xc, self.fin, self.bin)
            return self.cmask[row] * (xc - self.kappa * self.clover_inv(h))
        return self.cmask[row] * (-self.kappa * self.clover_inv(self.hop(xc, self.fout, self.bout)))

    def _jacobi(self, b, c, n_jac):
        b = self.cmask[c] * b
        x = 2 * b - self._block(b, c, c)
        for _ in range(1, n_jac):
            x = x + b - self._block(x, c, c)
        return x

    def msap(self, b, n_sap, n_jac):
        s = b.clone()
        for _ in range(n_sap):
            for c in (0, 1):
                x = self._jacobi(s, c, n_jac)
                s = s + self.cmask[c] * (b - self._block(x, c, c))
                s = s - self._block(x, 1 - c, c)
        xe = self._jacobi(s, 0, n_jac)
        s = s - self._block(xe, 1, 0)
        return xe + self._jacobi(s, 1, n_jac)

    def A(self, x):
        return x - self.kappa * self.clover_inv(self.hop(x))

    def solve(self, b, op=None, tol=1e-14):
        """BiCGStab on C_inv D x = C_inv b, restarted until |b - D x| stops falling."""
        op = op or self.D
        x = torch.zeros_like(b)
        r = b.clone()
        bn = b.norm().item()
        best = 1.0
        for _ in range(8):
            r0, p, rr, y = r, r, r, torch.zeros_like(b)
            rho = torch.vdot(r0.flatten(), rr.flatten())
            target = 1e-8 * rr.norm().item()
            for _ in range(400):
                q = op(p)
                alpha = rho / torch.vdot(r0.flatten(), q.flatten())
                s = rr - alpha * q
                t = op(s)
                om = torch.vdot(t.flatten(), s.flatten()) / torch.vdot(t.flatten(), t.flatten())
                y = y + alpha * p + om * s
                rr = s - om * t
                if rr.norm().item() < target:
                    break
                rho1 = torch.vdot(r0.flatten(), rr.flatten())
                p = rr + (rho1 / rho) * (alpha / om) * (p - om * q)
                rho = rho1
            x = x + y
            r = b - op(x)
            rel = r.norm().item() / bn
            if rel < tol or rel > 0.5 * best:
                break
            best = rel
        return x


def _internal(x, dims, d, double):
    """Canonical complex128 [rhs][t][z][y][x][3][4] -> the library's device
    layout, as reals: domains of extents d, all of even colour first, each
    colour in lexicographic order; inside a domain one block per pair of
    components (float32) or per component (float64), the sites innermost;
    components ordered (spin, colour)."""
    lx, ly, lz, lt = dims
    n = [L // m for L, m in zip(dims, d)]
    x = x.reshape((-1, n[3], d[3], n[2], d[2], n[1], d[1], n[0], d[0], 3, 4))
    # [rhs][domain t z y x][spin colour][site t z y x]
    x = x.permute(0, 1, 3, 5, 7, 10, 9, 2, 4, 6, 8).reshape(x.shape[0], math.prod(n), 12, math.prod(d))
    ax = torch.meshgrid(*[torch.arange(k, device=x.device) for k in (n[3], n[2], n[1], n[0])], indexing="ij")
    colour = (sum(ax) % 2).flatten()
    order = torch.cat([torch.nonzero(colour == 0).flatten(), torch.nonzero(colour == 1).flatten()])
    x = torch.view_as_real(x[:, order].contiguous())
    if not double:
        x = x.reshape(x.shape[0], x.shape[1], 6, 2, math.prod(d), 2).permute(0, 1, 2, 4, 3, 5)
    return x.contiguous().flatten()


def _each(f, x, nrhs):
    return torch.stack([f(x[r]) for r in range(nrhs)]) if nrhs > 1 else f(x)


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    kind, dims, d = case["kind"], _dims(case), _domain(case)
    if kind == "ragged":
        return [torch.view_as_real(_Plain(u, kappa, case["csw"], case["bc_t"], case["basis"]).solve(b))
                for _, kappa, u, b in _ragged_inputs(case, seed, dev)]
    u = _gauge(dims, case["eps"], seed, 1, dev)
    if kind == "train":
        return _exact_train(case, seed, u, dev)
    op = _Plain(u, case["kappa"], case["csw"], case["bc_t"], case["basis"])
    nrhs = case.get("nrhs", 1)
    if kind == "solve":
        return torch.view_as_real(_each(op.solve, _source(case, seed, dev), nrhs))
    psi = _spinor(dims, nrhs, seed, 2, dev)
    if kind == "canonical":
        return torch.view_as_real(_each(op.Ddag if case["dagger"] else op.D, psi, nrhs))
    if kind == "apply":
        return _internal(_each(op.Ddag if case["dagger"] else op.D, psi, nrhs), dims, d, case["prec"] == "double")
    if kind == "config":
        return [_internal(op.D(psi), dims, d, True), _internal(op.clover_inv(psi), dims, d, True)]
    op.set_domain([int(v) for v in case["sdom"].split("x")] if case["sdom"] else d)

    def m(v):
        z = op.msap(v, case["n_sap"], case["n_jac"])
        return op.A(z) if case["with_A"] else z

    return _internal(_each(m, psi, nrhs), dims, d, False)


def _exact_train(case, seed, u, dev):
    """x = D^-1 b, grad_b = D^-dag eta, and grad_U of -Re(lambda^dag D[U] x)."""
    b, eta = _spinor(_dims(case), 1, seed, 2, dev), _spinor(_dims(case), 1, seed, 3, dev)
    with torch.no_grad():
        op = _Plain(u, case["kappa"], case["csw"], case["bc_t"], case["basis"])
        x = op.solve(b)
        lam = op.solve(eta, op.Ddag)
    v = u.clone().requires_grad_(True)
    op = _Plain(v, case["kappa"], case["csw"], case["bc_t"], case["basis"])
    loss = -(lam.conj() * op.D(x)).sum().real
    loss.backward()
    return [torch.view_as_real(t) for t in (x, lam, v.grad)]
