"""What this framework is measured on: the calls that a lattice program makes, each through a public entry point.

  dslash   one application of D_eo / D_oe (or of A) to device vectors: the smallest call (8^4, where the launch
           is what counts), the benchmark's 48^3x12 with one and with eight right-hand sides, and a large
           lattice in the most compact storage (16-bit, compressed long links)
  cg       whole solves to a true residual of 1e-10 from x = 0: the plain FP64 method on 8^4 (bound by
           latency), the benchmark's mixed-precision solve, several sources in 16-bit storage on a lattice
           whose extents divide by nothing convenient
  shifts   multi-shift CG with RHMC's 14 shifts
  batch    many lattices of uneven sizes in one solve
  fcg      flexible CG with the learned preconditioner
  train    one training step of that preconditioner: loss and both layers' weight gradients
  gauge    a new gauge field: the two HISQ smearing levels, the link load, and one Dslash with the new links

Links are drawn as the repository's other workloads draw them: thin U = exp(i eps H) with Gaussian H, fat = U
plus complex Gaussian noise, long = -1/24 of the product of three thin links; sources are complex Gaussian.
Everything is made on the GPU from the seed. The launches' tuning, which a program keeps in a saved report, is
kept from one state to the next in the same way; everything else belongs to its state.
"""
import math

import numpy as np
import torch

import paper_2111_10354_gb300 as h

PRECS = {"f64": h.HISQ_F64, "f32": h.HISQ_F32, "f16": h.HISQ_F16, "bf16": h.HISQ_BF16, "df64": h.HISQ_DF64}
REAL_BYTES = {"f64": 8, "df64": 8, "f32": 4, "f16": 2, "bf16": 2}
NAIK = -1.0 / 24.0
NOISE = 0.1
CHANNELS = 8
LEVEL1 = dict(c1=1 / 8, c3=1 / 16, c5=1 / 64, c7=1 / 384)
LEVEL2 = dict(c1=5 / 8, c3=1 / 16, c5=1 / 64, c7=1 / 384, cL=-1 / 16, cN=NAIK)
SHIFTS = (1e-5, 1.0)  # the range of a shift set, spaced by its logarithm
SHIFT_MASS = 0.0025
FCG_MASS = 0.001
MAXITER = 20000
# CG iterations to 1e-10 on these links (eps 0.3, 48^3x12), as work() counts them; they barely move with the lattice
ITERATIONS = {"cg": 145, "shifts": 127, "batch": 200, "fcg": 100}


# ---------------------------------------------------------------- the cases

def listed():
    return [
        dict(name="dslash-8c8-f64", kind="dslash", Lx=8, Ly=8, Lz=8, Lt=8, prec="f64", nrhs=1, op="D_eo", layout="blocked",
             comp=False),
        dict(name="dslash-48c12-f32", kind="dslash", Lx=48, Ly=48, Lz=48, Lt=12, prec="f32", nrhs=1, op="D_oe",
             layout="blocked", comp=False),
        dict(name="dslash-48c12-f32-n8", kind="dslash", Lx=48, Ly=48, Lz=48, Lt=12, prec="f32", nrhs=8, op="D_eo",
             layout="blocked", comp=False),
        dict(name="dslash-64c16-f16-comp", kind="dslash", Lx=64, Ly=64, Lz=64, Lt=16, prec="f16", nrhs=1, op="A",
             layout="blocked", comp=True),
        dict(name="cg-8c8-f64", kind="cg", Lx=8, Ly=8, Lz=8, Lt=8, prec="f64", spinor="f32", nrhs=1, mass=0.1),
        dict(name="cg-48c12-f32", kind="cg", Lx=48, Ly=48, Lz=48, Lt=12, prec="f32", spinor="f32", nrhs=1, mass=0.01),
        dict(name="cg-ragged-f16-n5", kind="cg", Lx=20, Ly=12, Lz=28, Lt=10, prec="f16", spinor="f16", nrhs=5, mass=0.02),
        dict(name="shifts-48c12", kind="shifts", Lx=48, Ly=48, Lz=48, Lt=12, prec="f32", nshift=14, tol=1e-9),
        dict(name="batch-16", kind="batch", n16=8, n24=5, n32=3, prec="f32"),
        dict(name="fcg-32c8", kind="fcg", Lx=32, Ly=32, Lz=32, Lt=8),
        dict(name="train-32c8-n16", kind="train", Lx=32, Ly=32, Lz=32, Lt=8, npairs=16),
        dict(name="gauge-32c8-f64", kind="gauge", Lx=32, Ly=32, Lz=32, Lt=8, prec="f64"),
    ]


def _draw_dims(rng, low, high):
    """Four even extents, 4 or more, whose volume lies near a value drawn over the logarithm of [low, high]."""
    while True:
        volume = math.exp(rng.uniform(math.log(low), math.log(high)))
        side = volume ** 0.25
        ext = [max(4, 2 * round(side * math.exp(rng.uniform(-0.5, 0.5)) / 2)) for _ in range(3)]
        ext.append(max(4, 2 * round(volume / (ext[0] * ext[1] * ext[2]) / 2)))
        if low <= math.prod(ext) <= high and max(ext) <= 96:
            return dict(zip(("Lx", "Ly", "Lz", "Lt"), ext))


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "dslash", "cg", "cg", "shifts", "batch", "fcg", "train", "gauge"])
    c = {"kind": kind}
    if kind == "dslash":
        prec = rng.choice(sorted(PRECS))
        c.update(_draw_dims(rng, 256, 64 ** 3 * 16 if prec in ("f32", "f16", "bf16") else 48 ** 3 * 12))
        layout = rng.choice(["blocked", "blocked", "interleaved"])
        nrhs = min(16, int(math.exp(rng.uniform(0, math.log(17)))))
        if layout == "interleaved":  # whole 16-byte words of vectors
            word = {"f32": 2, "f16": 4, "bf16": 4}.get(prec, 1)
            nrhs = -(-nrhs // word) * word
        c.update(prec=prec, nrhs=nrhs, op=rng.choice(["D_eo", "D_oe", "A"]), layout=layout,
                 comp=prec in ("f32", "f16", "bf16") and rng.random() < 0.25)
    elif kind == "cg":
        prec = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        nrhs = rng.choice([1, 1, 2, 3, 5, 8])
        c.update(_draw_dims(rng, 4096, min(48 ** 3 * 12, 48 ** 3 * 12 * 2 // (nrhs * (4 if prec == "f64" else 1)))))
        c.update(prec=prec, spinor=rng.choice(["f32", prec]) if prec in ("f16", "bf16") else "f32", nrhs=nrhs,
                 mass=round(math.exp(rng.uniform(math.log(0.002), math.log(0.1))), 4))
    elif kind == "shifts":
        c.update(_draw_dims(rng, 16 ** 4, 40 ** 3 * 12))
        c.update(prec="f32", nshift=rng.randint(4, 14), tol=rng.choice([1e-8, 1e-9]))
    elif kind == "batch":
        c.update(n16=rng.randint(1, 8), n24=rng.randint(0, 5), n32=rng.randint(0, 3), prec=rng.choice(["f32", "f32", "f64"]))
        if c["prec"] == "f64":
            c.update(n24=c["n24"] // 2, n32=c["n32"] // 2)
    elif kind == "fcg":
        c.update(_draw_dims(rng, 8 ** 4, 32 ** 3 * 12))
    elif kind == "train":
        c.update(_draw_dims(rng, 8 ** 4, 32 ** 3 * 8))
        c.update(npairs=rng.randint(2, 16))
    else:
        prec = rng.choice(["f64", "df64"])
        c.update(_draw_dims(rng, 4096, 32 ** 3 * 8 if prec == "f64" else 48 ** 3 * 8))
        c.update(prec=prec)
    return c


def _dims(case):
    return case["Lx"], case["Ly"], case["Lz"], case["Lt"]


def _lattices(case):
    """Extents of a batch's lattices."""
    return [(16, 16, 16, 16)] * case["n16"] + [(24, 24, 24, 8)] * case["n24"] + [(32, 32, 32, 8)] * case["n32"]


# ---------------------------------------------------------------- inputs (no code of the framework)

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _mul(a, b):
    """Products of 3x3 matrices (..., 3, 3), entry by entry."""
    return torch.stack([sum(a[..., :, k] * b[..., k, j, None] for k in range(3)) for j in range(3)], -1)


def _dag(a):
    return a.mH


def _thin_links(L, eps, g):
    """U = exp(i eps H), H = sum_a h_a lambda_a / 2, h_a ~ N(0, 1): (Lt, Lz, Ly, Lx, 4, 3, 3) complex128."""
    n = math.prod(L) * 4
    a = torch.randn(8, n, generator=g, device="cuda", dtype=torch.float64) * (0.5 * eps / 4)
    H = torch.zeros(n, 3, 3, dtype=torch.complex128, device="cuda")
    for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        H[:, i, j] = torch.complex(a[2 * k], -a[2 * k + 1])
        H[:, j, i] = torch.complex(a[2 * k], a[2 * k + 1])
    r3 = 1 / math.sqrt(3.0)
    H[:, 0, 0], H[:, 1, 1], H[:, 2, 2] = a[6] + r3 * a[7], r3 * a[7] - a[6], -2 * r3 * a[7]
    one = torch.eye(3, dtype=torch.complex128, device="cuda")
    X, U = 1j * H, one.expand_as(H)
    for k in range(12, 0, -1):  # exp(X) by Horner's rule, |X| below 1/2; then squared twice
        U = one + _mul(X, U) / k
    U = _mul(U, U)
    U = _mul(U, U)
    return U.reshape(*L[::-1], 4, 3, 3)


def _shift(a, mu, k):
    """a(x + k mu) for a field with its site axes (t, z, y, x) first."""
    return torch.roll(a, -k, 3 - mu)


def _cgauss(shape, g):
    z = torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(0.5)
    return torch.view_as_complex(z)


def _links(L, eps, g):
    """(fat, long) links."""
    U = _thin_links(L, eps, g)
    lng = torch.empty_like(U)
    for mu in range(4):
        u = U[..., mu, :, :]
        lng[..., mu, :, :] = NAIK * _mul(_mul(u, _shift(u, mu, 1)), _shift(u, mu, 2))
    U += NOISE * _cgauss(U.shape, g)
    return U, lng


def _source(L, nrhs, g):
    return _cgauss((nrhs, math.prod(L) // 2, 3), g)


def _to_storage(v, prec):
    """complex128 vectors in the storage of a precision (16-bit types have a last axis (re, im))."""
    if prec in ("f64", "df64"):
        return v
    if prec == "f32":
        return v.to(torch.complex64)
    return torch.view_as_real(v).to(torch.float16 if prec == "f16" else torch.bfloat16)


def _from_storage(v):
    return v.to(torch.complex128) if v.is_complex() else torch.view_as_complex(v.to(torch.float64).contiguous())


def _dslash_inputs(case, seed):
    g = _generator(seed)
    L = _dims(case)
    fat, lng = _links(L, 0.3, g)
    v = _source(L, case["nrhs"], g)
    if case["layout"] == "interleaved":
        v = v.permute(1, 2, 0).contiguous()
    return fat, lng, _to_storage(v, case["prec"])


def _solve_inputs(case, seed, eps, nrhs):
    g = _generator(seed)
    fat, lng = _links(_dims(case), eps, g)
    return fat, lng, _source(_dims(case), nrhs, g)


def _batch_inputs(case, seed):
    """Per lattice: links drawn with their own eps in [0.2, 0.4], a mass log-uniform in [0.005, 0.1], a source."""
    g, r = _generator(seed), np.random.RandomState(seed % (1 << 32))
    for L in _lattices(case):
        fat, lng = _links(L, r.uniform(0.2, 0.4), g)
        yield L, fat, lng, _source(L, 1, g)[0], math.exp(r.uniform(math.log(0.005), math.log(0.1)))


def _bf16_exact(w):
    return torch.view_as_complex(torch.view_as_real(w).to(torch.bfloat16).to(torch.float32))


def _trained_weights(g):
    """Tied first-layer weights (8, 1, 9) like those that training arrives at: the identity hop, and for each direction a
    channel that adds its two transports with one sign, so that B^dag B falls where -D_eo D_oe grows; some noise."""
    w = torch.complex(*(0.004 * torch.randn(2, CHANNELS, 1, 9, generator=g, device="cuda", dtype=torch.float32)))
    for mu in range(4):
        w[mu, 0, 1 + mu] += 0.125
        w[mu, 0, 5 + mu] += 0.125
        w[4 + mu, 0, 0] += 0.145
    return _bf16_exact(w)


def _tie(w1):
    """Layer 2 as the adjoint of layer 1: W2[0, a, h] = conj(W1[a, 0, h']), h' the opposite hop."""
    return w1[:, 0, [0, 5, 6, 7, 8, 1, 2, 3, 4]].conj()[None]


def _train_inputs(case, seed):
    """Links, weights, and pairs (b, x) with x close to A^-1 b (30 iterations of CG, plain torch)."""
    g = _generator(seed)
    L = _dims(case)
    fat, lng = _links(L, 0.35, g)
    w1, w2 = (_bf16_exact(torch.complex(*(0.05 * torch.randn(2, *s, generator=g, device="cuda", dtype=torch.float32))))
              for s in ((CHANNELS, 1, 9), (1, CHANNELS, 9)))
    w1[0, 0, 0] += 1
    w1 = _bf16_exact(w1)
    b = _source(L, case["npairs"], g).to(torch.complex64)
    op = _Operator(L, fat.to(torch.complex64), lng.to(torch.complex64))
    x = _cg(lambda v: op.A(v, FCG_MASS), b, 1e-3, 30)
    return fat, lng, w1, w2, b, x


# ---------------------------------------------------------------- states

_tuned = {}  # lattice and kind of work -> the launches' tuning, as a program saves it


def _tune(ctx, case, once):
    """Takes over a saved tuning, or, the first time, makes it by one call."""
    key = (_dims(case), case["kind"], case.get("prec"), case.get("comp"), case.get("nrhs"), case.get("op"))
    if key in _tuned:
        h.hisq_tune_load(ctx, _tuned[key])
    else:
        once()
        _tuned[key] = h.hisq_tune_report(ctx)


def _lattice(case, precs, fat, lng):
    lat = h.Lattice(_dims(case), precs=precs)
    if case.get("comp"):
        lat.compress_long(NAIK)
    return lat.load(fat, lng)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "dslash":
        fat, lng, v = _dslash_inputs(case, seed)
        s.update(lat=_lattice(case, (PRECS[case["prec"]],), fat, lng), v=v, out=torch.empty_like(v), op=case["op"],
                 prec=PRECS[case["prec"]], nrhs=case["nrhs"], il=case["layout"] == "interleaved")
    elif kind in ("cg", "shifts"):
        nrhs = case.get("nrhs", 1)
        fat, lng, b = _solve_inputs(case, seed, 0.3, nrhs)
        s.update(lat=_lattice(case, (PRECS[case["prec"]],), fat, lng), b=b)
        if kind == "cg":
            s.update(x=torch.zeros_like(b), mass=case["mass"],
                     opts=dict(nrhs=nrhs, inner_prec=PRECS[case["prec"]], spinor_prec=PRECS[case["spinor"]]))
        else:
            s.update(x=torch.zeros((case["nshift"],) + b.shape[1:], dtype=b.dtype, device="cuda"), tol=case["tol"],
                     shifts=np.geomspace(*SHIFTS, case["nshift"]), opts=dict(inner_prec=PRECS[case["prec"]]))
    elif kind == "batch":
        s["batch"] = h.Batch(_lattices(case))
        b, s["masses"] = [], []
        for k, (_, fat, lng, src, mass) in enumerate(_batch_inputs(case, seed)):
            s["batch"].load(k, fat.cpu().numpy(), lng.cpu().numpy())
            b.append(src)
            s["masses"].append(mass)
        s["b"] = torch.cat(b)
        s.update(x=torch.zeros_like(s["b"]), opts=dict(inner_prec=PRECS[case["prec"]]))
    elif kind == "fcg":
        fat, lng, b = _solve_inputs(case, seed, 0.35, 1)
        w1 = _trained_weights(_generator(seed + 1))
        s.update(lat=_lattice(case, (h.HISQ_F64, h.HISQ_F32), fat, lng), b=b, x=torch.zeros_like(b))
        s["net"] = h.Ptc(s["lat"], CHANNELS)
        s["net"].set_tied(True)
        s["net"].set_weights(w1.cpu().numpy(), _tie(w1).cpu().numpy())
    elif kind == "train":
        fat, lng, w1, w2, b, x = _train_inputs(case, seed)
        s.update(lat=_lattice(case, (h.HISQ_F64, h.HISQ_F32), fat, lng), b=b, x=x, npairs=case["npairs"])
        s["net"] = h.Ptc(s["lat"], CHANNELS)
        s["net"].set_weights(w1.cpu().numpy(), w2.cpu().numpy())
    else:
        g = _generator(seed)
        L = _dims(case)
        s.update(thin=_thin_links(L, 0.3, g), v=_source(L, 1, g),
                 lat=h.Lattice(L, precs=(h.HISQ_F64, h.HISQ_F32)), prec=PRECS[case["prec"]])
        s.update(fat=torch.empty_like(s["thin"]), lng=torch.empty_like(s["thin"]), out=torch.empty_like(s["v"]))
    if "lat" in s:
        _tune(s["lat"].ctx, case, lambda: run(s))
    torch.cuda.synchronize()
    return s


def run(s):
    kind = s["kind"]
    if kind == "dslash":
        lat = s["lat"]
        if s["op"] == "A":
            (lat.apply_A_interleaved if s["il"] else lat.apply_A)(s["out"], s["v"], 0.01, s["prec"], s["nrhs"])
        else:
            (lat.dslash_interleaved if s["il"] else lat.dslash)(0 if s["op"] == "D_eo" else 1, s["out"], s["v"], s["prec"],
                                                               s["nrhs"])
        return s["out"]
    if kind == "cg":
        s["x"].zero_()
        s["lat"].cg(s["x"], s["b"], s["mass"], 1e-10, MAXITER, **s["opts"])
        return s["x"]
    if kind == "shifts":
        s["lat"].multishift_cg(s["x"], s["b"], s["shifts"], SHIFT_MASS, s["tol"], MAXITER, **s["opts"])
        return s["x"]
    if kind == "batch":
        s["x"].zero_()
        s["batch"].cg(s["x"], s["b"], s["masses"], 1e-10, MAXITER, **s["opts"])
        return s["x"]
    if kind == "fcg":
        s["x"].zero_()
        s["net"].fcg(s["x"], s["b"], FCG_MASS, 1e-10, MAXITER)
        return s["x"]
    if kind == "train":
        return s["net"].train_step(s["b"], s["x"], s["npairs"], 0.0)
    s["lat"].hisq_links(s["fat"], s["lng"], s["thin"], LEVEL1, LEVEL2, s["prec"])
    s["lat"].load(s["fat"], s["lng"])
    s["lat"].dslash(0, s["out"], s["v"], h.HISQ_F64)
    return s["fat"], s["lng"], s["out"]


# ---------------------------------------------------------------- work and tolerances

def _dslash_bytes(half, prec, nrhs, comp=False):
    link = (8 * 18 + 8 * (12 if comp else 18)) * REAL_BYTES[prec]
    return half * (link + nrhs * 12 * REAL_BYTES[prec])


def work(case):
    """Bytes and operations of one pass. A solve counts its iterations' two Dslash (every link once, every vector in and
    out once) and nothing else; smearing counts its 50 products of 3x3 matrices per link and level."""
    kind = case["kind"]
    if kind == "batch":
        half = sum(math.prod(L) for L in _lattices(case)) // 2
        it = ITERATIONS["batch"]
        return {"bytes": 2.0 * it * _dslash_bytes(half, case["prec"], 1), "flops": 2.0 * it * half * 1146}
    V = math.prod(_dims(case))
    half = V // 2
    if kind == "dslash":
        n = 2 if case["op"] == "A" else 1
        return {"bytes": float(n * _dslash_bytes(half, case["prec"], case["nrhs"], case["comp"])),
                "flops": 1146.0 * n * half * case["nrhs"]}
    if kind == "cg":
        it = ITERATIONS["cg"]
        return {"bytes": 2.0 * it * _dslash_bytes(half, case["prec"], case["nrhs"]), "flops": 2292.0 * it * half * case["nrhs"]}
    if kind == "shifts":  # the shared Krylov space, and each shift's two vectors updated in every iteration
        it = ITERATIONS["shifts"]
        return {"bytes": it * (2.0 * _dslash_bytes(half, case["prec"], 1) + case["nshift"] * half * 96.0),
                "flops": 2292.0 * it * half}
    if kind == "fcg":  # two FP32 Dslash and two passes over the fat links
        it = ITERATIONS["fcg"]
        return {"bytes": it * half * (2.0 * 1200 + 2 * 8 * 72), "flops": it * half * 3600.0}
    if kind == "train":  # per pair: b and x, the 8-channel activation of the odd sites written and read in both directions
        per_site = 2 * 24 + 4 * CHANNELS * 24 + 3 * 8 * 72
        return {"bytes": float(case["npairs"]) * half * per_site, "flops": case["npairs"] * half * 3 * (8 * 66.0 * (1 + CHANNELS)
                                                                                                       + 9 * CHANNELS * 24.0)}
    return {"bytes": V * 4 * 144.0 * (3 + 3) + V * 4 * 2 * (144 + 72), "flops": 2.0 * 4 * 50 * 216 * V}


def tolerance(case):
    """About four times what another order of the sums, or another correct rounding of the storage, was seen to give."""
    kind = case["kind"]
    if kind == "dslash":
        return {"rel": {"f64": 2e-15, "df64": 5e-14, "f32": 1e-6, "f16": 1.5e-3, "bf16": 1.2e-2}[case["prec"]]}
    if kind in ("cg", "batch", "fcg"):  # residuals of 1e-10 leave x within some 1e-10 to 1e-9
        return {"rel": 5e-9}
    if kind == "shifts":
        return {"rel": 30 * case["tol"]}
    if kind == "train":  # activations and gradients enter the products in bf16, and average over the sites
        return {"rel": 1e-3}
    return {"rel": 1e-14 if case["prec"] == "f64" else 1e-13}


# ---------------------------------------------------------------- the same in 64 bits, plain torch

class _Operator:
    """D with phases and the antiperiodic time boundary, on vectors (n, V/2, 3) of one parity."""

    def __init__(self, L, fat, lng):
        self.L = L
        t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in L[::-1]), indexing="ij")
        sites = (x + y + z + t).reshape(-1) % 2
        self.sites = [torch.nonzero(sites == p).reshape(-1) for p in (0, 1)]
        ones = torch.ones_like(x)
        eta = [ones, 1 - 2 * (x % 2), 1 - 2 * ((x + y) % 2), 1 - 2 * ((x + y + z) % 2)]
        self.hops = []
        for mu in range(4):
            for k, links in ((1, fat), (3, lng)):
                sign = eta[mu] * (1 - 2 * (t >= L[3] - k).long() if mu == 3 else ones)
                self.hops.append((mu, k, links[..., mu, :, :] * sign[..., None, None]))

    def full(self, v, parity):
        f = torch.zeros((math.prod(self.L), 3, v.shape[0]), dtype=v.dtype, device=v.device)
        f[self.sites[parity]] = v.permute(1, 2, 0)
        return f.reshape(*self.L[::-1], 3, v.shape[0])

    def take(self, f, parity):
        return f.reshape(-1, 3, f.shape[-1])[self.sites[parity]].permute(2, 0, 1).contiguous()

    @staticmethod
    def times(U, f):
        return torch.stack([sum(U[..., i, j, None] * f[..., j, :] for j in range(3)) for i in range(3)], -2)

    def D(self, v, out_parity):
        f = self.full(v, 1 - out_parity)
        out = torch.zeros_like(f)
        for mu, k, U in self.hops:
            out += self.times(U, _shift(f, mu, k))
            out -= _shift(self.times(U.mH, f), mu, -k)
        return self.take(out, out_parity)

    def A(self, v, mass, sigma=0.0):
        return (4 * mass * mass + sigma) * v - self.D(self.D(v, 1), 0)


def _dot(a, b):
    """Real parts of the inner products of n vectors (n, V/2, 3), shaped to scale them."""
    return (torch.view_as_real(a) * torch.view_as_real(b)).sum((1, 2, 3), dtype=torch.float64)[:, None, None]


def _cg(A, b, tol, maxiter):
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rr = bb = _dot(b, b)
    for _ in range(maxiter):
        q = A(p)
        a = rr / _dot(p, q)
        x += a.to(b.real.dtype) * p
        r -= a.to(b.real.dtype) * q
        rr, old = _dot(r, r), rr
        if bool((rr <= tol * tol * bb).all()):
            break
        p = r + (rr / old).to(b.real.dtype) * p
    return x


def _cg_refined(A, b):
    """CG restarted once from its true residual: good to about 1e-14 of b."""
    x = _cg(A, b, 1e-12, 5000)
    return x + _cg(A, b - A(x), 1e-3, 5000)


def _staple(Ub, X, b, mu, sign):
    """Ub(x) X(x+b) Ub(x+mu)^dag, or Ub(x-b)^dag X(x-b) Ub(x-b+mu)."""
    if sign > 0:
        return _mul(_mul(Ub, _shift(X, b, 1)), _dag(_shift(Ub, mu, 1)))
    return _shift(_mul(_mul(_dag(Ub), X), _shift(Ub, mu, 1)), b, -1)


def _smear(U, c1=0.0, c3=0.0, c5=0.0, c7=0.0, cL=0.0, cN=0.0):
    """One level on links [mu] of (t, z, y, x, 3, 3): (fat, long)."""
    fat, lng = [], []
    for mu in range(4):
        nus = [n for n in range(4) if n != mu]
        S = {(n, s): _staple(U[n], U[mu], n, mu, s) for n in nus for s in (1, -1)}
        f = c1 * U[mu]
        for a in nus:
            Y = c3 * U[mu]
            for b in nus:
                if b != a:
                    c = [n for n in nus if n not in (a, b)][0]
                    X = c5 * U[mu] + c7 * (S[c, 1] + S[c, -1])
                    Y = Y + _staple(U[b], X, b, mu, 1) + _staple(U[b], X, b, mu, -1)
            for s in (1, -1):
                f = f + _staple(U[a], Y + cL * S[a, s], a, mu, s)
        fat.append(f)
        lng.append(cN * _mul(_mul(U[mu], _shift(U[mu], mu, 1)), _shift(U[mu], mu, 2)))
    return fat, lng


def _project(W):
    """W (W^dag W)^(-1/2), by Newton's iteration X <- (X + X^(-dag)) / 2, which doubles its digits each time."""
    X = W
    for _ in range(8):
        a, b, c = X[..., 0, :], X[..., 1, :], X[..., 2, :]
        cof = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], -2)
        det = (a * cof[..., 0, :]).sum(-1)[..., None, None]
        X = 0.5 * (X + (cof / det).conj())
    return X


def _transports(op, psi):
    """The nine hops of the network's layer on fields (t, z, y, x, 3, n): identity, +mu, -mu through the fat links."""
    fats = {mu: U for mu, k, U in op.hops if k == 1}
    return [psi] + [op.times(fats[mu], _shift(psi, mu, 1)) for mu in range(4)] + \
        [_shift(op.times(fats[mu].mH, psi), mu, -1) for mu in range(4)]


def _exact_train(case, seed):
    fat, lng, w1, w2, b, x = _train_inputs(case, seed)
    op = _Operator(_dims(case), fat, lng)
    w1, w2 = (w.to(torch.complex128).requires_grad_() for w in (w1, w2))
    total = 0.0
    for q in range(case["npairs"]):
        r, target = b[q:q + 1].to(torch.complex128), x[q:q + 1].to(torch.complex128)
        first = torch.stack(_transports(op, op.full(r, 0)), -1)[..., 0, :]
        psi = torch.einsum("ah,...ch->...ca", w1[:, 0], first)
        second = torch.stack(_transports(op, psi), -1)
        z = op.take(torch.einsum("ah,...cah->...c", w2[0], second)[..., None], 0)
        loss = (z - target).abs().square().sum() / target.abs().square().sum() / case["npairs"]
        loss.backward()
        total += float(loss.detach())
    # torch's gradient of a real loss is twice the derivative with respect to conj(w)
    return total, (w1.grad / 2).cpu().numpy(), (w2.grad / 2).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    L = None if kind == "batch" else _dims(case)
    if kind == "dslash":
        fat, lng, v = _dslash_inputs(case, seed)
        op, v = _Operator(L, fat, lng), _from_storage(v)
        il = case["layout"] == "interleaved"
        v = v.permute(2, 0, 1) if il else v
        out = []
        for k in range(case["nrhs"]):
            u = v[k:k + 1]
            out.append(op.A(u, 0.01) if case["op"] == "A" else op.D(u, 0 if case["op"] == "D_eo" else 1))
        out = torch.cat(out)
        out = out.permute(1, 2, 0).contiguous() if il else out
        return out if case["prec"] in ("f64", "f32", "df64") else torch.view_as_real(out)
    if kind == "cg":
        fat, lng, b = _solve_inputs(case, seed, 0.3, case["nrhs"])
        op = _Operator(L, fat, lng)
        return _cg_refined(lambda v: op.A(v, case["mass"]), b)
    if kind == "shifts":
        if case["nshift"] * math.prod(L) > 14 * 24 ** 3 * 8:
            return None  # a CG for each shift takes too long
        fat, lng, b = _solve_inputs(case, seed, 0.3, 1)
        op = _Operator(L, fat, lng)
        return torch.cat([_cg_refined(lambda v: op.A(v, SHIFT_MASS, float(s)), b)
                          for s in np.geomspace(*SHIFTS, case["nshift"])])
    if kind == "batch":
        out = []
        for dims, fat, lng, src, mass in _batch_inputs(case, seed):
            op = _Operator(dims, fat, lng)
            out.append(_cg_refined(lambda v: op.A(v, mass), src[None])[0])
        return torch.cat(out)
    if kind == "fcg":
        fat, lng, b = _solve_inputs(case, seed, 0.35, 1)
        op = _Operator(L, fat, lng)
        return _cg_refined(lambda v: op.A(v, FCG_MASS), b)
    if kind == "train":
        return _exact_train(case, seed)
    g = _generator(seed)
    U = _thin_links(L, 0.3, g)
    v = _source(L, 1, g)
    level1, _ = _smear([U[..., mu, :, :] for mu in range(4)], **LEVEL1)
    fat, lng = (torch.stack(f, -3) for f in _smear([_project(W) for W in level1], **LEVEL2))
    return fat, lng, _Operator(L, fat, lng).D(v, 0)
