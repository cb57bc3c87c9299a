"""Performance cases: the calls a user of this solver makes, over the sizes they make them at.

A case is a dict of plain values; ``kind`` says which public entry points it calls:

  dirac      amg_apply_D on nrhs canonical vectors (AMG_F32, AMG_F16 or AMG_F64)
  sap        amg_sap, the smoother, on nrhs vectors
  transfer   amg_restrict and amg_prolong on nrhs vectors
  coarse     amg_apply_coarse on nrhs coarse vectors (FP32, or bfloat16 on the tensor cores)
  solve      amg_solve of nrhs right-hand sides on a hierarchy that is set up already
  ragged     amg_solve_ragged of independent problems of several lattice sizes
  config     a new gauge field: operator, adaptive setup and the solves of nrhs sources
  train      amg_nn_train_step, one Adam step of the learned preconditioner

Fields are synthetic: links exp(i eps H) with Gaussian Hermitian traceless H, Gaussian
vectors or point sources, drawn from the seed.  Lattice extents are (Lx, Ly, Lz, Lt).

``exact`` restates each operation in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_2111_05012_gb300 import capi

TOL = 1e-10


# ------------------------------------------------------------------ the cases
def _dirac(name, dims, prec, nrhs, kappa=0.130):
    return dict(name=name, kind="dirac", lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], prec=prec, nrhs=nrhs,
                eps=0.6, kappa=kappa)


def _grid(name, kind, dims, block, nvec, nrhs, **kw):
    c = dict(name=name, kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], bx=block[0], by=block[1],
             bz=block[2], bt=block[3], nvec=nvec, nrhs=nrhs, eps=0.6, kappa=0.130)
    c.update(kw)
    return c


def listed():
    return [
        # the operator inside somebody else's Krylov solver on a test lattice: a call is all latency
        _dirac("dirac_f32_4", (4, 4, 4, 4), "f32", 1, kappa=0.124),
        # the operator alone at a production local volume, one vector
        _dirac("dirac_f32_32", (32, 32, 32, 64), "f32", 1),
        # half-precision storage, several vectors at a time
        _dirac("dirac_f16_24", (24, 24, 24, 48), "f16", 4),
        # residual checks in double precision
        _dirac("dirac_f64_16", (16, 16, 16, 32), "f64", 1),
        # the smoother as a preconditioner of its own, a batch of vectors
        _grid("sap_24", "sap", (24, 24, 24, 48), (4, 4, 4, 4), 8, 4, vec="f32"),
        # deflation-style use of the test vectors: restrict and prolong a few vectors
        _grid("transfer_24", "transfer", (24, 24, 24, 48), (4, 4, 4, 4), 24, 4, vec="f32"),
        # the coarse operator on 16 vectors on the tensor cores (8192 coarse sites, Nc 48)
        _grid("coarse_bf16_16", "coarse", (16, 16, 16, 32), (2, 2, 2, 2), 24, 16, vec="f32", prec="bf16"),
        # one Gaussian right-hand side: latency of an ordinary solve
        _grid("solve_16", "solve", (16, 16, 16, 32), (4, 4, 4, 4), 24, 1, vec="f16", coarse="f32", source="normal",
              outer_m=16),
        # a propagator: the 12 spin-colour point sources in lockstep, coarse solves on the tensor cores
        _grid("propagator_24", "solve", (24, 24, 24, 48), (4, 4, 4, 4), 24, 12, vec="f16", coarse="bf16",
              source="point", outer_m=8, eps=0.5, kappa=0.129),
        # many small configurations of three lattice sizes at once
        dict(name="ragged_12", kind="ragged", nprob=12, nvec=24, eps=0.6, kappa=0.130),
        # a new configuration of an ensemble: operator, adaptive setup and its propagator
        _grid("config_16", "config", (16, 16, 16, 32), (4, 4, 4, 4), 24, 12, vec="f16", coarse="bf16",
              source="point", outer_m=8),
        # one training step of the learned preconditioner, a batch of 16 pairs
        dict(name="train_24", kind="train", lx=24, ly=24, lz=24, lt=48, channels=4, npairs=16, eps=0.6, kappa=0.130),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: every extent is drawn by itself, so lattices are rarely cubic."""
    kind = rng.choice(["dirac", "dirac", "dirac", "sap", "sap", "transfer", "coarse", "solve", "solve", "ragged",
                       "config", "train"])
    eps = round(rng.uniform(0.3, 0.6), 3)
    kappa = round(rng.uniform(0.122, 0.130), 4)
    if kind == "dirac":
        while True:
            dims = tuple(_log_int(rng, 3, 32) for _ in range(3)) + (_log_int(rng, 3, 64),)
            if math.prod(dims) <= 32 ** 3 * 64:
                break
        prec = rng.choice(["f32", "f32", "f16", "f64"])
        nrhs = min(_log_int(rng, 1, 12), max(1, 4 * 24 ** 3 * 48 // math.prod(dims)))
        if prec == "f16" and math.prod(dims) % 4:
            nrhs = 1   # a half-precision field of such a volume does not end on a 16-byte boundary
        if prec == "f64":
            nrhs = min(nrhs, max(1, 16 ** 3 * 32 * 4 // math.prod(dims)))
        return dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], prec=prec, nrhs=nrhs, eps=eps,
                    kappa=kappa)
    if kind == "ragged":
        return dict(kind=kind, nprob=rng.randint(2, 12), nvec=rng.choice([8, 12, 16, 20, 24]), eps=eps, kappa=kappa)
    if kind == "train":
        dims = tuple(rng.randint(6, 20) for _ in range(3)) + (rng.randint(6, 32),)
        return dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], channels=rng.randint(1, 4),
                    npairs=rng.randint(1, 16), eps=eps, kappa=kappa)
    # domains of 2, 3 or 4 sites and an even number of them in each direction; a domain has at
    # least 36 sites so that its test vectors stay independent
    most = 16 ** 3 * 32 if kind in ("solve", "config", "coarse") else 24 ** 3 * 48
    while True:
        block = tuple(rng.choice([2, 3, 4, 4]) for _ in range(4))
        nblk = tuple(2 * rng.randint(1, 4) for _ in range(4))
        dims = tuple(b * n for b, n in zip(block, nblk))
        if math.prod(block) >= 36 and 2048 <= math.prod(dims) <= most:
            break
    V = math.prod(dims)
    nvec = rng.choice([8, 16, 24])
    c = dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], bx=block[0], by=block[1], bz=block[2],
             bt=block[3], nvec=nvec, nrhs=_log_int(rng, 1, 12), eps=eps, kappa=kappa, vec="f32")
    if kind in ("sap", "transfer"):
        c["nrhs"] = min(c["nrhs"], max(1, 4 * 24 ** 3 * 48 // V))
        if kind == "sap":
            c["nvec"] = 8
    elif kind == "coarse":
        c["prec"] = rng.choice(["f32", "bf16"])
        c["nrhs"] = _log_int(rng, 1, 16)
    else:
        c["vec"] = rng.choice(["f32", "f16"])
        c["coarse"] = rng.choice(["f32", "bf16"])
        c["source"] = rng.choice(["normal", "point"])
        c["outer_m"] = rng.choice([8, 16])
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, k=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + 7919 * k) % (1 << 62))
    return g


def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _volume(c):
    return math.prod(_dims(c))


def _block(c):
    return (c["bx"], c["by"], c["bz"], c["bt"])


def _cmul(a, b):
    """Product of small matrices over the last two indices."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _links(dims, eps, seed):
    """Links [Lt][Lz][Ly][Lx][mu][3][3], complex128: exp(i eps H) by scaling and squaring."""
    n = (dims[3], dims[2], dims[1], dims[0], 4, 3, 3)
    g = _gen(seed)
    out = torch.empty(n, dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for t in range(dims[3]):
        a = torch.randn(n[1:] + (2,), generator=g, dtype=torch.float64, device="cuda")
        a = torch.view_as_complex(a)
        h = 0.5 * (a + a.mH)
        h = h - eye * (h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3)[..., None, None]
        x = (1j * eps / 16) * h
        u = eye + x / 12
        for k in range(11, 0, -1):
            u = eye + _cmul(x, u) / k
        for _ in range(4):
            u = _cmul(u, u)
        out[t] = u
    return out


def _normal(dims, n, seed, k):
    """n canonical Gaussian fields, float64 [n][V * 24]."""
    return torch.randn((n, math.prod(dims) * 24), generator=_gen(seed, k), dtype=torch.float64, device="cuda")


def _points(dims, n, seed):
    """n spin-colour point sources at one site drawn from the seed."""
    V = math.prod(dims)
    site = int(torch.randint(V, (1,), generator=torch.Generator().manual_seed(int(seed))).item())
    b = torch.zeros((n, V * 24), dtype=torch.float64, device="cuda")
    for k in range(n):
        b[k, site * 24 + 2 * (k % 12)] = 1.0
    return b


class _Field:
    """Lattice, links and operator handles, freed with the object."""

    def __init__(self, dims, links, kappa):
        self.lat = capi.amg_lattice_create(dims, True)
        self.gauge = self.d = None
        self.gauge = capi.amg_gauge_create(self.lat, torch.view_as_real(links).cpu().numpy())
        self.d = capi.amg_dirac_create(self.gauge, kappa, 1.0)
        self.below = []

    def hierarchy(self, h):
        self.below.append((capi.amg_hierarchy_destroy, h))
        return h

    def network(self, nn):
        self.below.append((capi.amg_nn_destroy, nn))
        return nn

    def close(self):
        for free, h in self.below:
            free(h)
        self.below = []
        if self.d is not None:
            capi.amg_dirac_destroy(self.d)
        if self.gauge is not None:
            capi.amg_gauge_destroy(self.gauge)
        if self.lat is not None:
            capi.amg_lattice_destroy(self.lat)
        self.d = self.gauge = self.lat = None

    def __del__(self):
        self.close()


def _params(c, block, variant=-1):
    p = capi.amg_params_default()
    p.nlevels = 2
    for mu in range(4):
        p.block[0][mu] = block[mu]
    p.nvec[0] = c["nvec"]
    p.sap_variant = variant
    if c.get("vec") == "f16":
        p.prec_vectors = capi.AMG_F16
    if c.get("coarse") == "bf16" or c.get("prec") == "bf16":
        p.prec_coarsest = capi.AMG_BF16
        p.coarse_tc = 1
    if "outer_m" in c:
        p.outer_m = c["outer_m"]
    return p


_PREC = {"f64": capi.AMG_F64, "f32": capi.AMG_F32, "f16": capi.AMG_F16, "bf16": capi.AMG_BF16}
_RAGGED = [((8, 8, 8, 8), (4, 4, 4, 4)), ((12, 12, 12, 12), (3, 3, 3, 3)), ((16, 16, 16, 32), (4, 4, 4, 4))]


def _sources(c, seed):
    if c["source"] == "point":
        return _points(_dims(c), c["nrhs"], seed)
    return _normal(_dims(c), c["nrhs"], seed, 1)


def _coarse_sites(c):
    return _volume(c) // math.prod(_block(c))


def _weights(c, seed):
    """Weights of the 1-n-1 network: small complex Gaussians around a split identity."""
    n = c["channels"]
    g = _gen(seed, 5)
    w1 = 0.02 * torch.randn((n, 1, 9, 4, 4, 2), generator=g, dtype=torch.float64, device="cuda")
    w2 = 0.02 * torch.randn((1, n, 9, 4, 4, 2), generator=g, dtype=torch.float64, device="cuda")
    for s in range(4):
        w1[:, 0, 0, s, s, 0] += n ** -0.5
        w2[0, :, 0, s, s, 0] += n ** -0.5
    return w1.float(), w2.float()


def _pairs(c, op, seed):
    """(r, e) pairs: Gaussian errors e and their residuals r = D e, float32 [npairs][V * 24]."""
    dims = _dims(c)
    e = torch.randn((c["npairs"], math.prod(dims) * 24), generator=_gen(seed, 6), dtype=torch.float32, device="cuda")
    r = torch.empty_like(e)
    for k in range(c["npairs"]):
        r[k] = _flat(op.apply(_field(e[k].double(), dims))).float()
    return r, e


def prepare(c, seed):
    kind = c["kind"]
    if kind == "ragged":
        fields, hs, bs, xs = [], [], [], []
        for k in range(c["nprob"]):
            dims, block = _RAGGED[k % 3]
            f = _Field(dims, _links(dims, c["eps"], seed * 64 + k), c["kappa"])
            v = _normal(dims, c["nvec"], seed * 64 + k, 2)
            hs.append(f.hierarchy(capi.amg_setup(f.d, _params(c, block), [v])))
            fields.append(f)
            bs.append(_normal(dims, 1, seed * 64 + k, 1)[0])
            xs.append(torch.zeros_like(bs[-1]))
        return dict(kind=kind, fields=fields, hs=hs, bs=bs, xs=xs)
    dims, V = _dims(c), _volume(c)
    U = _links(dims, c["eps"], seed)
    if kind == "config":
        return dict(kind=kind, dims=dims, kappa=c["kappa"], U=torch.view_as_real(U).cpu().numpy(),
                    params=_params(c, _block(c)), init=_normal(dims, c["nvec"], seed, 2), b=_sources(c, seed),
                    x=torch.zeros((c["nrhs"], V * 24), dtype=torch.float64, device="cuda"), nrhs=c["nrhs"])
    f = _Field(dims, U, c["kappa"])
    if kind == "dirac":
        dt = torch.float64 if c["prec"] == "f64" else torch.float32
        x = _normal(dims, c["nrhs"], seed, 1).to(dt)
        return dict(kind=kind, f=f, x=x, y=torch.empty_like(x), nrhs=c["nrhs"], prec=_PREC[c["prec"]])
    if kind == "train":
        r, e = _pairs(c, _Dirac(U, c["kappa"]), seed)
        ch = [1, c["channels"], 1]
        w = np.concatenate([t.cpu().numpy().reshape(-1) for t in _weights(c, seed)])
        nn = f.network(capi.amg_nn_create(f.d, ch, w))
        return dict(kind=kind, f=f, nn=nn, ch=ch, r=r, e=e, npairs=c["npairs"])
    del U
    v = _normal(dims, c["nvec"], seed, 2)
    s = dict(kind=kind, f=f, nrhs=c["nrhs"])
    if kind == "solve":
        s["h"] = f.hierarchy(capi.amg_setup(f.d, _params(c, _block(c)), [v]))
        s["b"] = _sources(c, seed)
        s["x"] = torch.zeros_like(s["b"])
        return s
    # the FP32 smoother with its FP32 operator throughout (variant -1 may take a half-precision copy of it)
    s["h"] = f.hierarchy(capi.amg_setup_from_vectors(f.d, _params(c, _block(c), 0), [v]))
    if kind == "coarse":
        n = _coarse_sites(c) * 2 * c["nvec"] * 2
        s["x"] = torch.randn((c["nrhs"], n), generator=_gen(seed, 3), dtype=torch.float32, device="cuda")
        s["y"] = torch.empty_like(s["x"])
        s["prec"] = _PREC[c["prec"]]
        return s
    s["b"] = _normal(dims, c["nrhs"], seed, 1).float()
    s["x"] = torch.empty_like(s["b"])
    if kind == "transfer":
        n = _coarse_sites(c) * 2 * c["nvec"] * 2
        s["c"] = torch.randn((c["nrhs"], n), generator=_gen(seed, 3), dtype=torch.float32, device="cuda")
        s["bc"] = torch.empty_like(s["c"])
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    kind = s["kind"]
    if kind == "dirac":
        capi.amg_apply_D(s["f"].d, s["x"], s["y"], s["nrhs"], s["prec"])
        return s["y"]
    if kind == "sap":
        capi.amg_sap(s["h"], s["b"], s["x"], capi.AMG_F32, nrhs=s["nrhs"])
        return s["x"]
    if kind == "transfer":
        capi.amg_restrict(s["h"], 0, s["b"], s["bc"], s["nrhs"], capi.AMG_F32)
        capi.amg_prolong(s["h"], 0, s["c"], s["x"], s["nrhs"], capi.AMG_F32)
        return s["bc"], s["x"]
    if kind == "coarse":
        capi.amg_apply_coarse(s["h"], 1, s["x"], s["y"], s["nrhs"], s["prec"])
        return s["y"]
    if kind == "solve":
        capi.amg_solve(s["h"], s["b"], s["x"], s["nrhs"], TOL, 200)
        return s["x"]
    if kind == "ragged":
        capi.amg_solve_ragged(s["hs"], s["bs"], s["xs"], TOL, 200)
        return s["xs"]
    if kind == "config":
        lat = capi.amg_lattice_create(s["dims"], True)
        gauge = capi.amg_gauge_create(lat, s["U"])
        d = capi.amg_dirac_create(gauge, s["kappa"], 1.0)
        h = capi.amg_setup(d, s["params"], [s["init"]])
        capi.amg_solve(h, s["b"], s["x"], s["nrhs"], TOL, 200)
        capi.amg_hierarchy_destroy(h)
        capi.amg_dirac_destroy(d)
        capi.amg_gauge_destroy(gauge)
        capi.amg_lattice_destroy(lat)
        return s["x"]
    loss = capi.amg_nn_train_step(s["nn"], s["r"], s["e"], s["npairs"], 1e-3)
    # the network computes in single precision, and so does what a user plots of it
    return np.float32(loss), capi.amg_nn_get_weights(s["nn"], s["ch"], effective=False)


# ------------------------------------------------------------------ what a pass cannot do without
_SAP_STEPS, _MR_STEPS = 4, 6
_D_FLOP = 1872.0                                        # one application of D, per site
_SAP_FLOP = _SAP_STEPS * (1896.0 + _MR_STEPS * 1830.0)   # per site: residuals and MR steps on D_SAP


def _sap_flop(V, nrhs):
    return nrhs * V * (_SAP_FLOP - 1896.0)               # the first sweep starts from x = 0


def _vec_bytes(c):
    return 52.0 if c.get("vec") == "f16" else 96.0       # one test vector, per site


def _solve_work(V, c, nrhs, nc, vc, steps):
    # links, clover and test vectors once, the coarse operator once, b and x; per step a cycle and D
    per = _SAP_FLOP + _D_FLOP + 2 * 96.0 * c["nvec"]
    cop = 9.0 * nc * nc * vc * (4 if c.get("coarse") == "bf16" else 8)
    return dict(bytes=V * (480.0 + _vec_bytes(c) * c["nvec"] + nrhs * 384.0) + cop,
                flops=nrhs * (steps * V * per + steps * 4 * 8.0 * 9 * nc * nc * vc))


def work(c):
    kind = c["kind"]
    if kind == "ragged":
        out = dict(bytes=0.0, flops=0.0)
        for k in range(c["nprob"]):
            dims, block = _RAGGED[k % 3]
            V = math.prod(dims)
            w = _solve_work(V, c, 1, 2 * c["nvec"], V // math.prod(block), 3)
            out = {q: out[q] + w[q] for q in out}
        return out
    V = _volume(c)
    nrhs = c.get("nrhs", 1)
    if kind == "dirac":
        # links as two rows, packed clover; the caller's vectors are doubles for f64, else floats
        op = {"f32": 480.0, "f16": 240.0, "f64": 960.0}[c["prec"]]
        return dict(bytes=V * (op + nrhs * (384.0 if c["prec"] == "f64" else 192.0)), flops=V * nrhs * _D_FLOP)
    if kind == "train":
        n = c["channels"]
        # transports of the input, of each hidden channel and of the output gradient; the spin
        # matrices of two layers forwards, one backwards and of both weight gradients
        per = 8 * 288.0 * (2 + n) + 5 * 9 * n * 384.0
        return dict(bytes=V * (192.0 + c["npairs"] * 192.0), flops=c["npairs"] * V * per)
    nc, vc = 2 * c["nvec"], _coarse_sites(c)
    if kind == "sap":
        return dict(bytes=V * (480.0 + nrhs * 192.0), flops=_sap_flop(V, nrhs))
    if kind == "transfer":
        return dict(bytes=2.0 * V * (_vec_bytes(c) * c["nvec"] + nrhs * 96.0) + 2.0 * nrhs * nc * vc * 8,
                    flops=2 * 96.0 * V * nrhs * c["nvec"])
    if kind == "coarse":
        return dict(bytes=9.0 * nc * nc * vc * (4 if c["prec"] == "bf16" else 8) + 2.0 * nrhs * nc * vc * 8,
                    flops=8.0 * 9 * nc * nc * vc * nrhs)
    w = _solve_work(V, c, nrhs, nc, vc, 3)
    if kind == "config":
        # three smoothing passes and two cycles on every test vector, the coarse operator thrice
        w["flops"] += V * c["nvec"] * (5 * _SAP_FLOP + 3 * 2 * (9 * 200.0 + 9 * 96.0 * c["nvec"]))
        w["bytes"] += V * (576.0 + 192.0 * c["nvec"])
    return w


# ------------------------------------------------------------------ the same in 64 bits
def _shift(x, mu, step):
    """x(s + step * mu_hat); the four leading indices of x are t, z, y, x."""
    return torch.roll(x, -step, dims=3 - mu)


def _gamma():
    s = torch.zeros((3, 2, 2), dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:] = 1j * s[k]
        g[k, 2:, :2] = -1j * s[k]
    g[3, :2, 2:] = torch.eye(2)
    g[3, 2:, :2] = torch.eye(2)
    return g


def _field(v, dims):
    """Canonical reals of one vector as [Lt][Lz][Ly][Lx][spin][colour]."""
    return torch.view_as_complex(v.reshape(dims[3], dims[2], dims[1], dims[0], 4, 3, 2).contiguous())


def _flat(f):
    return torch.view_as_real(f.contiguous()).reshape(-1)


class _Dirac:
    """D = 1 + F - kappa sum_mu [(1 - g_mu) U_mu(x) T_mu + (1 + g_mu) U_mu(x - mu)^dag T_-mu],
    antiperiodic in t, F the clover term with c_sw = 1."""

    def __init__(self, U, kappa):
        self.U, self.kappa = U, kappa
        g = _gamma()
        self.proj = [[(torch.eye(4) - s * g[mu]).to(U.device) for s in (1, -1)] for mu in range(4)]
        self.clover = self._clover(g)

    def _clover(self, g):
        A = torch.zeros(self.U.shape[:4] + (4, 3, 4, 3), dtype=torch.complex128, device=self.U.device)
        for s in range(4):
            for a in range(3):
                A[..., s, a, s, a] = 1
        for mu in range(4):
            for nu in range(mu + 1, 4):
                um, un = self.U[..., mu, :, :], self.U[..., nu, :, :]
                # the plaquette from the corner x, and its three shifted leaves based at x
                a, b = um, _shift(un, mu, 1)
                c, d = _shift(um, nu, 1).mH, un.mH
                Q = _cmul(_cmul(a, b), _cmul(c, d))
                Q = Q + _shift(_cmul(_cmul(b, c), _cmul(d, a)), mu, -1)
                Q = Q + _shift(_shift(_cmul(_cmul(c, d), _cmul(a, b)), mu, -1), nu, -1)
                Q = Q + _shift(_cmul(_cmul(d, a), _cmul(b, c)), nu, -1)
                F = (Q - Q.mH) / 8j
                tr = F.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
                F = F - tr[..., None, None] * torch.eye(3, dtype=F.dtype, device=F.device)
                sig = ((g[mu] @ g[nu] - g[nu] @ g[mu]) / 2j).to(F.device)
                for s in range(4):
                    for t in range(4):
                        if sig[s, t] != 0:
                            A[..., s, :, t, :] -= self.kappa * sig[s, t] * F
        return A.reshape(A.shape[:4] + (12, 12))

    def hop(self, psi, mu, step):
        """The covariantly shifted field U_mu(x) psi(x + mu) or U_mu(x - mu)^dag psi(x - mu)."""
        if step > 0:
            v = _shift(psi, mu, 1)
            if mu == 3:
                v = torch.cat([v[:-1], -v[-1:]])
            u = self.U[..., mu, :, :]
        else:
            v = _shift(psi, mu, -1)
            if mu == 3:
                v = torch.cat([-v[:1], v[1:]])
            u = _shift(self.U[..., mu, :, :], mu, -1).mH
        return (u.unsqueeze(-3) * v.unsqueeze(-2)).sum(-1)

    def apply(self, psi, block=None):
        """D psi, or with block the part of D inside the domains."""
        out = (self.clover @ psi.reshape(psi.shape[:4] + (12, 1))).reshape(psi.shape)
        for mu in range(4):
            for k, step in enumerate((1, -1)):
                w = torch.einsum("st,abcdtk->abcdsk", self.proj[mu][k], self.hop(psi, mu, step))
                if block is not None:
                    at = torch.arange(psi.shape[3 - mu], device=psi.device) % block[mu]
                    keep = (at != block[mu] - 1) if step > 0 else (at != 0)
                    shape = [1] * 6
                    shape[3 - mu] = -1
                    w = w * keep.reshape(shape)
                out = out - self.kappa * w
        return out


def _to_blocks(f, dims, b):
    """[Lt][Lz][Ly][Lx][...] -> [block][site of the block][...], both with x fastest."""
    n = [dims[3] // b[3], b[3], dims[2] // b[2], b[2], dims[1] // b[1], b[1], dims[0] // b[0], b[0]]
    f = f.reshape(n + list(f.shape[4:]))
    rest = list(range(8, f.dim()))
    return f.permute([0, 2, 4, 6, 1, 3, 5, 7] + rest).reshape([_nblocks(dims, b), math.prod(b)] + list(f.shape[8:]))


def _nblocks(dims, b):
    return math.prod(d // k for d, k in zip(dims, b))


def _from_blocks(f, dims, b):
    n = [dims[3] // b[3], dims[2] // b[2], dims[1] // b[1], dims[0] // b[0], b[3], b[2], b[1], b[0]]
    f = f.reshape(n + list(f.shape[2:]))
    rest = list(range(8, f.dim()))
    return f.permute([0, 4, 1, 5, 2, 6, 3, 7] + rest).reshape([dims[3], dims[2], dims[1], dims[0]] + list(f.shape[8:]))


def _sap_exact(op, b, dims, block):
    cdim = [d // k for d, k in zip(dims, block)]
    X = [torch.arange(n, device=b.device) for n in cdim]
    colour = (X[3][:, None, None, None] + X[2][:, None, None] + X[1][:, None] + X[0]).reshape(-1) % 2
    x = torch.zeros_like(b)

    def dots(u, v):
        return (u.conj() * v).sum((1, 2, 3))

    for _ in range(_SAP_STEPS):
        for col in range(2):
            keep = (colour == col).double()[:, None, None, None]
            r = _to_blocks(b - op.apply(x), dims, block) * keep
            z = torch.zeros_like(r)
            for _ in range(_MR_STEPS):
                Ar = _to_blocks(op.apply(_from_blocks(r, dims, block), block), dims, block)
                n = dots(Ar, Ar).real
                a = torch.where(n > 0, dots(Ar, r) / torch.where(n > 0, n, torch.ones_like(n)), 0)
                a = a[:, None, None, None]
                z = z + a * r
                r = r - a * Ar
            x = x + _from_blocks(z, dims, block)
    return x


def _basis(c, seed):
    """Orthonormal columns per (block, chirality) of the test vectors: [block][chi][6 Vb][nvec]."""
    dims, block, n = _dims(c), _block(c), c["nvec"]
    v = _normal(dims, n, seed, 2)
    Q = torch.stack([_to_blocks(_field(v[i], dims), dims, block) for i in range(n)], -1)
    Q = Q.reshape(Q.shape[0], Q.shape[1], 2, 6, n).transpose(1, 2).reshape(Q.shape[0], 2, -1, n)
    for i in range(n):
        w = Q[..., i]
        for _ in range(2):
            if i:
                w = w - (Q[..., :i] @ (Q[..., :i].mH @ w[..., None]))[..., 0]
        Q[..., i] = w / torch.linalg.vector_norm(w, dim=-1, keepdim=True)
    return Q


def _restrict(Q, f, dims, block):
    """<X, chi, i | f> as [block][chi * nvec]."""
    w = _to_blocks(f, dims, block)
    w = w.reshape(w.shape[0], w.shape[1], 2, 6).transpose(1, 2).reshape(w.shape[0], 2, -1, 1)
    return (Q.mH @ w).reshape(w.shape[0], -1)


def _prolong(Q, y, dims, block):
    w = Q @ y.reshape(y.shape[0], 2, -1, 1)
    w = w.reshape(w.shape[0], 2, -1, 6).transpose(1, 2).reshape(w.shape[0], -1, 4, 3)
    return _from_blocks(w, dims, block)


def _cview(v):
    return torch.view_as_complex(v.double().reshape(-1, 2).contiguous())


def _bicgstab(op, b, tol=1e-13):
    """D x = b by BiCGStab from x = 0."""
    x = torch.zeros_like(b)
    r = b.clone()
    rt, p = r.clone(), r.clone()
    bn = float(torch.linalg.vector_norm(b))

    def dot(u, v):
        return complex((u.conj() * v).sum())

    rho = dot(rt, r)
    for _ in range(1000):
        q = op.apply(p)
        alpha = rho / dot(rt, q)
        s = r - alpha * q
        t = op.apply(s)
        omega = dot(t, s) / dot(t, t).real
        x = x + alpha * p + omega * s
        r = s - omega * t
        if float(torch.linalg.vector_norm(r)) <= tol * bn:
            break
        new = dot(rt, r)
        p = r + (alpha / omega) * (new / rho) * (p - omega * q)
        rho = new
    return x


def _bf16(w):
    return w.to(torch.bfloat16).double()


def _train_exact(c, seed):
    """Loss and weights after the first Adam step, layer by layer (Wirtinger gradients)."""
    dims = _dims(c)
    op = _Dirac(_links(dims, c["eps"], seed), c["kappa"])
    r, e = _pairs(c, op, seed)
    masters = _weights(c, seed)
    W1, W2 = (torch.view_as_complex(_bf16(w).contiguous()) for w in masters)
    n = c["channels"]
    G1, G2 = torch.zeros_like(W1), torch.zeros_like(W2)
    steps = [(None, 0)] + [(mu, 1) for mu in range(4)] + [(mu, -1) for mu in range(4)]
    back = [0, 5, 6, 7, 8, 1, 2, 3, 4]

    def moved(f, k):
        return f if k == 0 else op.hop(f, steps[k][0], steps[k][1])

    def spin(w, f):
        return torch.einsum("st,abcdtk->abcdsk", w, f)

    def corr(g, f):
        return g.reshape(-1, 4, 3).transpose(1, 2).reshape(-1, 4).T @ f.reshape(-1, 4, 3).transpose(1, 2).reshape(-1, 4).conj()

    loss = 0.0
    for k in range(c["npairs"]):
        f0, target = _field(r[k].double(), dims), _field(e[k].double(), dims)
        phi1 = [moved(f0, d) for d in range(9)]
        h = [sum(spin(W1[a, 0, d], phi1[d]) for d in range(9)) for a in range(n)]
        y = sum(spin(W2[0, a, d], moved(h[a], d)) for a in range(n) for d in range(9))
        ne = float((target.conj() * target).sum().real)
        loss += float(((y - target).conj() * (y - target)).sum().real) / ne
        g = (y - target) / ne
        for a in range(n):
            for d in range(9):
                G2[0, a, d] += corr(g, moved(h[a], d))
        gm = [moved(g, back[d]) for d in range(9)]
        for a in range(n):
            ga = sum(spin(W2[0, a, d].mH, gm[d]) for d in range(9))
            for d in range(9):
                G1[a, 0, d] += corr(ga, phi1[d])
    out = []
    for w, G in zip(masters, (G1, G2)):
        gr = 2 * torch.view_as_real(G) / c["npairs"]
        out.append((w.double() - 1e-3 * gr / (gr.abs() + 1e-8)).reshape(-1))
    return loss / c["npairs"], torch.cat(out)


def exact(c, seed):
    kind = c["kind"]
    if kind == "train":
        return _train_exact(c, seed)
    if kind == "ragged":
        out = []
        for k in range(c["nprob"]):
            dims = _RAGGED[k % 3][0]
            op = _Dirac(_links(dims, c["eps"], seed * 64 + k), c["kappa"])
            out.append(_flat(_bicgstab(op, _field(_normal(dims, 1, seed * 64 + k, 1)[0], dims))))
        return out
    dims, nrhs = _dims(c), c["nrhs"]
    if kind in ("solve", "config") and _volume(c) * nrhs > 16 ** 3 * 32 * 12:
        return None
    op = _Dirac(_links(dims, c["eps"], seed), c["kappa"])
    if kind in ("solve", "config"):
        b = _sources(c, seed)
        return torch.stack([_flat(_bicgstab(op, _field(b[q], dims))) for q in range(nrhs)])
    if kind == "dirac":
        x = _normal(dims, nrhs, seed, 1)
        if c["prec"] != "f64":
            x = x.float().double()
        return torch.stack([_flat(op.apply(_field(x[q], dims))) for q in range(nrhs)])
    block = _block(c)
    if kind == "sap":
        b = _normal(dims, nrhs, seed, 1).float().double()
        return torch.stack([_flat(_sap_exact(op, _field(b[q], dims), dims, block)) for q in range(nrhs)])
    Q = _basis(c, seed)
    n = _coarse_sites(c) * 2 * c["nvec"] * 2
    xc = torch.randn((nrhs, n), generator=_gen(seed, 3), dtype=torch.float32, device="cuda")
    nb = _coarse_sites(c)
    if kind == "coarse":
        return torch.stack([_flat(_restrict(Q, op.apply(_prolong(Q, _cview(xc[q]).reshape(nb, -1), dims, block)),
                                            dims, block)) for q in range(nrhs)])
    b = _normal(dims, nrhs, seed, 1).float().double()
    return (torch.stack([_flat(_restrict(Q, _field(b[q], dims), dims, block)) for q in range(nrhs)]),
            torch.stack([_flat(_prolong(Q, _cview(xc[q]).reshape(nb, -1), dims, block)) for q in range(nrhs)]))
