"""What a user of the Wilson-Dirac library runs, as measurable cases.

Four kinds of call, each through the public binding (``paper_1810_04201_gb300.wd``):

* ``apply``  one application of D, D^dag or D^dag D to device fields, in every precision, with
  whole and compressed links, one or many right-hand sides;
* ``solve``  D x = b on device fields: plain FP64 CG, mixed precision, even-odd, many right-hand sides;
* ``config`` a new gauge configuration: its links are loaded, then one system given in pinned host
  memory is solved end to end (upload, solve, download);
* ``batch``  many small uneven lattices in one call.

The launch shapes are the library's defaults: no case autotunes, as a program that meets a new
lattice size for the first time does not either.
"""
import math

import numpy as np
import torch

from paper_1810_04201_gb300 import wd

PREC = {"f64": wd.WD_F64, "f32": wd.WD_F32, "f16": wd.WD_F16, "df32": wd.WD_DF32}
SPINOR_BYTES = {"f64": 192, "f32": 96, "f16": 52, "df32": 192}  # one site, 12 components (FP16: and its scale)
LINK_BYTES = {("f64", 18): 144, ("f64", 12): 96, ("f32", 18): 72, ("f32", 12): 48, ("f16", 18): 36, ("f16", 12): 24,
              ("df32", 18): 144, ("df32", 12): 96}
FLOPS = 1320  # of one Dslash per site
# kappa and the CG iterations of a 1e-10 solve (plain, even-odd) per kind of links
LINKS = {"haar": (0.12, 45, 23), "smooth": (0.124, 180, 67)}
BATCH_SHAPES = ((8, 8, 8, 8), (8, 8, 8, 16), (12, 12, 12, 12), (12, 12, 12, 24), (16, 16, 16, 16))


def _apply(name, dims, op="D", prec="f64", recon=18, nrhs=1):
    c = {"kind": "apply", "x": dims[0], "y": dims[1], "z": dims[2], "t": dims[3], "op": op, "prec": prec,
         "recon": recon, "nrhs": nrhs, "links": "haar"}
    return dict(c, name=name) if name else c


def _solve(name, dims, inner="f64", eo=False, nrhs=1, links="haar", recon_in=18, source="gauss"):
    c = {"kind": "solve", "x": dims[0], "y": dims[1], "z": dims[2], "t": dims[3], "inner": inner, "eo": eo,
         "nrhs": nrhs, "links": links, "recon_in": recon_in, "source": source}
    return dict(c, name=name) if name else c


def _config(name, dims, inner="f32", eo=False):
    c = {"kind": "config", "x": dims[0], "y": dims[1], "z": dims[2], "t": dims[3], "inner": inner, "eo": eo,
         "links": "haar"}
    return dict(c, name=name) if name else c


def _batch(name, n, inner="f32", shapes=99, recon_in=18):
    c = {"kind": "batch", "n": n, "inner": inner, "shapes": shapes, "recon_in": recon_in}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's own small lattice: one operator call, bound by latency
        _apply("apply f64 8^3x12", (8, 8, 8, 12)),
        # D^dag D at double precision, the building block of a user's own Krylov method
        _apply("normal f64 16^4", (16, 16, 16, 16), "DdagD"),
        # D^dag in double-FP32 on an odd, ragged lattice
        _apply("dagger df32 15x13x17x21", (15, 13, 17, 21), "Ddag", "df32"),
        # the single-precision operator on the largest lattice
        _apply("apply f32 32^3x64", (32, 32, 32, 64), "D", "f32"),
        # half-precision storage with compressed links: the inner operator of a user's multigrid or mixed solver
        _apply("apply f16 r12 24^3x48", (24, 24, 24, 48), "D", "f16", 12),
        # the 12 spin-colour columns of a propagator at once
        _apply("apply f32 x12 24^3x48", (24, 24, 24, 48), "D", "f32", 18, 12),
        # a short mixed-precision solve on a small lattice: launches and host work count
        _solve("solve f32 eo 8^3x16", (8, 8, 8, 16), "f32", True),
        # the default solve: plain FP64 CG
        _solve("solve f64 24^4", (24, 24, 24, 24), "f64"),
        # a propagator: 12 point sources in one solve
        _solve("solve f32 x12 24^3x48", (24, 24, 24, 48), "f32", False, 12, source="point"),
        # the production solve on the largest lattice: even-odd, FP16 inner iteration, compressed inner links
        _solve("solve f16 eo 32^3x64", (32, 32, 32, 64), "f16", True, 1, "smooth", 12),
        # a new configuration end to end: links in, source from the host, solution back
        _config("config f32 16^3x32", (16, 16, 16, 32)),
        # an ensemble of 64 small uneven lattices in one call
        _batch("batch f32 64 lattices", 64),
    ]


def _dims(rng, lo, hi, even):
    """Four extents, volume spread over [lo, hi] on a log scale."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        d = [max(2, round(v ** 0.25 * math.exp(rng.uniform(-0.35, 0.35)))) for _ in range(3)]
        d.append(max(2, round(v / (d[0] * d[1] * d[2]))))
        if even:
            d = [max(2, e + e % 2) for e in d]
        if lo / 2 <= d[0] * d[1] * d[2] * d[3] <= hi and d[3] <= 96:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "solve", "config", "batch"])
    if kind == "apply":
        nrhs = rng.choice([1, 1, 1, 2, 3, 4, 7, 12])
        prec = rng.choice(["f64", "f32", "f16", "df32"])
        dims = _dims(rng, 256, 32 ** 3 * 64 // (1 if nrhs == 1 else nrhs), False)
        return _apply(None, dims, rng.choice(["D", "Ddag", "DdagD"]), prec, rng.choice([18, 12]), nrhs)
    if kind == "solve":
        inner = rng.choice(["f64", "f32", "f32", "f16", "df32"])
        nrhs = rng.choice([1, 1, 1, 2, 5, 12])
        eo = rng.random() < 0.5
        # a plain FP64 or double-FP32 solve costs several times a mixed one
        hi = 32 ** 3 * 64 // (1 if inner in ("f32", "f16") else 12)
        dims = _dims(rng, 256, max(512, hi // (1 if nrhs == 1 else 2 * nrhs)), eo)
        recon_in = 18 if inner == "f64" else rng.choice([18, 12])
        return _solve(None, dims, inner, eo, nrhs, "haar", recon_in, rng.choice(["gauss", "point"]))
    if kind == "config":
        eo = rng.random() < 0.5
        return _config(None, _dims(rng, 256, 16 ** 3 * 64, eo), rng.choice(["f64", "f32", "f16"]), eo)
    return _batch(None, rng.randint(3, 64), rng.choice(["f32", "f16"]), rng.randint(1, 10000), rng.choice([18, 12]))


# ------------------------------------------------------------------ inputs (torch, from the seed alone)
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _normal(g, *shape):
    re = torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)
    im = torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.complex(re, im) * math.sqrt(0.5)


def _haar(g, n):
    """n Haar-random SU(3) matrices: Gram-Schmidt on the rows of a complex Gaussian matrix, then the third row
    conj(row0 x row1), which makes the determinant one."""
    z = _normal(g, n, 2, 3)
    a = z[:, 0] / z[:, 0].abs().square().sum(1, keepdim=True).sqrt()
    b = z[:, 1]
    for _ in range(2):
        b = b - (a.conj() * b).sum(1, keepdim=True) * a
    b = b / b.abs().square().sum(1, keepdim=True).sqrt()
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], 1)


def _matmul3(a, b):
    return (a[:, :, :, None] * b[:, None, :, :]).sum(2)


def _smooth(g, n, eps=0.4):
    """n matrices exp(i eps H), H = sum_a w_a lambda_a / 2 with w_a ~ N(0, 1): Taylor series and squarings."""
    w = torch.randn(n, 8, generator=g, device="cuda", dtype=torch.float64) * (0.5 * eps / 16)
    z = torch.zeros(n, 3, 3, device="cuda", dtype=torch.complex128)
    i = 1j
    s3 = 1 / math.sqrt(3)
    z[:, 0, 1], z[:, 1, 0] = i * w[:, 0] + w[:, 1], i * w[:, 0] - w[:, 1]
    z[:, 0, 2], z[:, 2, 0] = i * w[:, 3] + w[:, 4], i * w[:, 3] - w[:, 4]
    z[:, 1, 2], z[:, 2, 1] = i * w[:, 5] + w[:, 6], i * w[:, 5] - w[:, 6]
    z[:, 0, 0], z[:, 1, 1], z[:, 2, 2] = i * (w[:, 2] + s3 * w[:, 7]), i * (s3 * w[:, 7] - w[:, 2]), -2 * s3 * i * w[:, 7]
    eye = torch.eye(3, device="cuda", dtype=torch.complex128)
    u = eye + z / 9
    for k in range(8, 0, -1):
        u = eye + _matmul3(z, u) / k
    for _ in range(4):
        u = _matmul3(u, u)
    return u


def _links(kind, dims, seed):
    v = math.prod(dims)
    u = torch.empty(4, v, 3, 3, device="cuda", dtype=torch.complex128)
    for mu in range(4):
        g = _gen(seed, 10 + mu)
        u[mu] = _haar(g, v) if kind == "haar" else _smooth(g, v)
    return u


def _sources(case, dims, nrhs, seed):
    v = math.prod(dims)
    if case.get("source") == "point":
        b = torch.zeros(nrhs, v, 4, 3, device="cuda", dtype=torch.complex128)
        site = int(np.random.RandomState(seed % 2 ** 31).randint(v))
        for r in range(nrhs):
            b[r, site, (r % 12) // 3, r % 3] = 1.0
        return b
    return _normal(_gen(seed, 1), nrhs, v, 4, 3)


def _case_dims(case):
    return case["x"], case["y"], case["z"], case["t"]


def _batch_members(case):
    rng = np.random.RandomState(case["shapes"])
    return [(BATCH_SHAPES[rng.randint(len(BATCH_SHAPES))], 0.10 + 0.025 * rng.random_sample()) for _ in range(case["n"])]


def prepare(case, seed):
    if case["kind"] == "batch":
        lats, kappas, bs, xs = [], [], [], []
        for i, (dims, kappa) in enumerate(_batch_members(case)):
            lat = wd.Lattice(dims)
            lat.set_gauge(_links("haar", dims, seed + 7919 * i))
            if case["recon_in"] != 18:
                lat.set_link_compression(PREC[case["inner"]], case["recon_in"])
            lats.append(lat)
            kappas.append(kappa)
            bs.append(lat.pack(_sources(case, dims, 1, seed + 7919 * i)[0]))
            xs.append(lat.new_field())
        return {"case": case, "lats": lats, "kappas": kappas, "bs": bs, "xs": xs}
    dims = _case_dims(case)
    lat = wd.Lattice(dims)
    state = {"case": case, "lat": lat}
    u = _links(case["links"], dims, seed)
    if case["kind"] == "config":
        b = _sources(case, dims, 1, seed)
        state.update(u=u, b=b.cpu().pin_memory(), x=torch.zeros(b.shape, dtype=torch.complex128).pin_memory())
        return state
    if case["kind"] == "apply":
        prec, n = PREC[case["prec"]], case["nrhs"]
        lat.set_gauge(u, recon=case["recon"])
        state.update(src=lat.pack(_sources(case, dims, n, seed), prec), dst=lat.new_field(prec, n))
        return state
    lat.set_gauge(u)
    if case["recon_in"] != 18:
        lat.set_link_compression(PREC[case["inner"]], case["recon_in"])
    n = case["nrhs"]
    state.update(b=lat.pack(_sources(case, dims, n, seed)), x=lat.new_field(nrhs=n))
    return state


# ------------------------------------------------------------------ one pass
def _columns(field, prec, nrhs):
    """The values of a device field, right-hand side by right-hand side."""
    out = []
    for f in field.view(nrhs, -1):
        if prec == "f16":  # 3 arrays of 16 bytes a site, then one float a site
            half = f.numel() // 52 * 48
            out.append([f[:half].view(torch.float16), f[half:].view(torch.float32)])
        else:
            out.append(f.view(torch.float64 if prec == "f64" else torch.float32))
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        for x in state["xs"]:
            x.zero_()
        wd.cg_batched(state["lats"], state["kappas"], state["bs"], state["xs"], tol=1e-10, inner=PREC[case["inner"]])
        return [x.view(torch.float64) for x in state["xs"][:60]]
    lat = state["lat"]
    kappa = LINKS[case["links"]][0]
    if case["kind"] == "apply":
        prec, n = PREC[case["prec"]], case["nrhs"]
        if case["op"] == "DdagD":
            lat.normal_apply(kappa, state["src"], state["dst"], prec, n)
        else:
            lat.apply(kappa, state["src"], state["dst"], prec, n, dagger=case["op"] == "Ddag")
        return _columns(state["dst"], case["prec"], n)
    if case["kind"] == "config":
        lat.set_gauge(state["u"])
        state["x"].zero_()
        lat.cg_canonical(kappa, state["b"], state["x"], tol=1e-10, inner=PREC[case["inner"]],
                         precondition=int(case["eo"]))
        return state["x"]
    state["x"].zero_()
    lat.cg(kappa, state["b"], state["x"], tol=1e-10, inner=PREC[case["inner"]], nrhs=case["nrhs"],
           precondition=int(case["eo"]))
    return _columns(state["x"], "f64", case["nrhs"])


# ------------------------------------------------------------------ what a pass cannot do without
def _dslash_bytes(v, prec, recon, nrhs):
    return v * (4 * LINK_BYTES[prec, recon] + 2 * nrhs * SPINOR_BYTES[prec])


def _solve_work(v, inner, recon_in, nrhs, iters, eo):
    """A 1e-10 solve: per iteration the operator and its adjoint in the inner precision (even-odd: each link once
    per hop onto a parity, half the sites per field), the vectors x, r, p read and written once."""
    per_op = _dslash_bytes(v, inner, recon_in, nrhs) if not eo else \
        v * (2 * 4 * LINK_BYTES[inner, recon_in] + 2 * nrhs * SPINOR_BYTES[inner])
    vec = nrhs * v * SPINOR_BYTES[inner] * 5 // (2 if eo else 1)
    return {"bytes": iters * (2 * per_op + vec), "flops": iters * nrhs * 2 * FLOPS * v}


def work(case):
    if case["kind"] == "batch":
        total = {"bytes": 0, "flops": 0}
        for dims, _ in _batch_members(case):
            w = _solve_work(math.prod(dims), case["inner"], case["recon_in"], 1, 42, False)
            total = {k: total[k] + w[k] for k in total}
        return total
    v = math.prod(_case_dims(case))
    if case["kind"] == "apply":
        k = 2 if case["op"] == "DdagD" else 1
        return {"bytes": k * _dslash_bytes(v, case["prec"], case["recon"], case["nrhs"]),
                "flops": k * FLOPS * v * case["nrhs"]}
    iters = LINKS[case["links"]][2 if case["eo"] else 1]
    if case["kind"] == "config":
        w = _solve_work(v, case["inner"], 18, 1, iters, case["eo"])
        return {"bytes": w["bytes"] + v * (2 * 4 * 144 + 2 * 192), "flops": w["flops"]}
    return _solve_work(v, case["inner"], case["recon_in"], case["nrhs"], iters, case["eo"])


def tolerance(case):
    if case["kind"] == "apply":
        # about four times the measured distance from 64 bits: rounding of the inputs, links and sums of each type
        # (the two floats of a DF32 number are compared as they stand: the high one is rounded to 24 bits)
        rel = {"f64": 1e-15, "f32": 8e-7, "f16": 3e-3, "df32": 2e-7}[case["prec"]]
        return {"rel": rel, "max": 40 * rel}
    # a solve stops at a normal residual of 1e-10; the solution is off by that times the condition number
    rel = 4e-9 if case.get("links") == "smooth" else 1e-9
    return {"rel": rel, "max": 1e-6}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _gammas():
    i = 1j
    a = [np.array(m, dtype=np.complex128) for m in
         ([[0, i], [i, 0]], [[0, -1], [1, 0]], [[i, 0], [0, -i]], [[1, 0], [0, 1]])]
    g = []
    for m in a:  # gamma = [[0, A], [A^dag, 0]]
        x = np.zeros((4, 4), dtype=np.complex128)
        x[:2, 2:], x[2:, :2] = m, m.conj().T
        g.append(torch.from_numpy(x).cuda())
    return g


def _exact_d(u, psi, kappa, dims, dagger, gammas):
    """D psi (D^dag psi): psi (V, 4, 3), antiperiodic in t."""
    lx, ly, lz, lt = dims
    f = psi.view(lt, lz, ly, lx, 4, 3)
    s = 1.0 if dagger else -1.0
    out = psi.clone().view(f.shape)
    for mu in range(4):
        ax = 3 - mu
        um = u[mu].view(lt, lz, ly, lx, 3, 3)
        fwd = torch.roll(f, -1, ax)
        if mu == 3:
            fwd[-1] = -fwd[-1]
        h = fwd + s * torch.einsum("ij,tzyxja->tzyxia", gammas[mu], fwd)
        out -= kappa * torch.einsum("tzyxab,tzyxib->tzyxia", um, h)
        h = f - s * torch.einsum("ij,tzyxja->tzyxia", gammas[mu], f)
        h = torch.roll(torch.einsum("tzyxba,tzyxib->tzyxia", um.conj(), h), 1, ax)
        if mu == 3:
            h[0] = -h[0]
        out -= kappa * h
    return out.view(psi.shape)


def _exact_solve(u, b, kappa, dims, gammas, tol=1e-14, most=400):
    """x with D x = b, by conjugate gradients on D^dag D x = D^dag b far below the library's tolerance."""
    d = lambda v, dag: _exact_d(u, v, kappa, dims, dag, gammas)  # noqa: E731
    x = torch.zeros_like(b)
    r = d(b, True)
    p, rr = r.clone(), r.abs().square().sum()
    stop = rr * tol ** 2
    for k in range(most):
        t = d(p, False)
        alpha = rr / t.abs().square().sum()
        x += alpha * p
        r -= alpha * d(t, True)
        new = r.abs().square().sum()
        p = r + (new / rr) * p
        rr = new
        if k % 8 == 7 and bool(rr <= stop):
            break
    return x


def _layout(psi, prec):
    """A canonical spinor (V, 4, 3) in the library's field layout of a precision, as _columns() shows it."""
    v = psi.shape[0]
    vs = (v + 63) // 64 * 64
    a = torch.zeros(12, vs, 2, device="cuda", dtype=torch.float64)
    a[:, :v] = torch.view_as_real(psi.reshape(v, 12).t().contiguous())
    if prec == "f64":
        return a.reshape(-1)
    if prec == "f32":
        return a.view(6, 2, vs, 2).permute(0, 2, 1, 3).reshape(-1)
    if prec == "df32":
        hi = a.float()
        return torch.cat([hi.double(), a - hi.double()], 2).reshape(-1)
    scale = a.abs().amax((0, 2))
    a = a / torch.where(scale > 0, scale, torch.ones_like(scale))[None, :, None]
    return [a.view(3, 4, vs, 2).permute(0, 2, 1, 3).reshape(-1), scale]


def exact(case, seed):
    gammas = _gammas()
    if case["kind"] == "batch":  # the first lattices speak for all
        out = []
        for i, (dims, kappa) in enumerate(_batch_members(case)[:60]):
            if i >= 8:
                out.append(None)
                continue
            u = _links("haar", dims, seed + 7919 * i)
            out.append(_layout(_exact_solve(u, _sources(case, dims, 1, seed + 7919 * i)[0], kappa, dims, gammas), "f64"))
        return out
    dims = _case_dims(case)
    kappa = LINKS[case["links"]][0]
    n = case.get("nrhs", 1)
    if case["kind"] != "apply" and case["links"] == "smooth" and math.prod(dims) > 500000:
        return None
    u = _links(case["links"], dims, seed)
    src = _sources(case, dims, n, seed)
    if case["kind"] == "apply":
        out = []
        for r in range(n):
            y = src[r]
            for dag in {"D": [False], "Ddag": [True], "DdagD": [False, True]}[case["op"]]:
                y = _exact_d(u, y, kappa, dims, dag, gammas)
            out.append(_layout(y, case["prec"]))
        return out
    if case["kind"] == "config":
        return _exact_solve(u, src[0], kappa, dims, gammas)[None]
    # the first columns speak for all
    return [_layout(_exact_solve(u, src[r], kappa, dims, gammas), "f64") if r < 2 else None for r in range(n)]
