"""The work that programs give this library, as measurable cases.

A case is a dict of plain values.  ``prepare`` makes what a program holds before
the call (gauge field loaded, two-link field built, source vectors on the GPU),
``run`` is one pass through the public entry points, ``work`` the bytes and
operations that pass cannot do without, and ``exact`` the same result in 64-bit
torch arithmetic.  Every program keeps its unsmeared sources, so a smearing pass
copies them into the buffer that is smeared in place.

Four kinds:
  smear    one tls_smear call on a resident two-link field
  config   a new configuration: load the links, optionally APE-smear them, build
           the two-link field, smear its first sources, release the field
  onelink  one tls_smear_onelink call on a resident link field
  serve    a burst of jobs through the serving loop on two resident fields
"""

import math
import random

import torch

from paper_2301_05518_gb300 import tls

# storage, two-link precision, reals kept per matrix: the combinations in use
FORMATS = (("F64", "F64", 18), ("F32", "F32", 18), ("F32", "F32", 12), ("F32", "F32", 8),
           ("F16", "F32", 18), ("F16", "F16", 18), ("F16", "F16", 12), ("BF16", "F32", 18), ("BF16", "BF16", 12))


def _case(name=None, kind="smear", dims=(8, 8, 8, 8), links="haar", nvec=1, N=10, sigma_per_N=0.2, storage="F32",
          wprec="F32", recon=18, t0=-1, source="gauss", tuned=False, ape=0, host=False, norms=False, jobs=0,
          jobs_seed=0):
    c = dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], links=links, nvec=nvec, N=N,
             sigma_per_N=sigma_per_N, storage=storage, wprec=wprec, recon=recon, t0=t0, source=source, tuned=tuned,
             ape=ape, host=host, norms=norms, jobs=jobs, jobs_seed=jobs_seed)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one point source smeared on its own slice in double precision: the smallest call,
        # all latency (the 8^3 x 16 point-source workload)
        _case("point_8x16_f64", dims=(8, 8, 8, 16), links="near", N=10, storage="F64", wprec="F64", t0=0,
              source="point"),
        # three colour-wall sources smeared on the source slice alone, n = 50: the usual call
        # before a solve; everything fits in L2
        _case("walls_48_slice_f32", dims=(48, 48, 48, 8), links="near", nvec=3, N=50, t0=0, source="wall",
              norms=True),
        # the 32^3 x 64 mixed workload in double precision, the reference-quality run
        _case("mixed_32x64_f64", dims=(32, 32, 32, 64), links="near", nvec=6, N=40, storage="F64", wprec="F64"),
        # one vector on every slice: the single right-hand-side stencil
        _case("single_48x64_f32", dims=(48, 48, 48, 64), links="near", N=30),
        # batches of 24 dense vectors on Haar links, FP32 and 16-bit storage
        _case("gauss_48x32_f32_24", dims=(48, 48, 48, 32), nvec=24, N=40),
        _case("gauss_48x32_f16_24", dims=(48, 48, 48, 32), nvec=24, N=40, storage="F16"),
        # the large lattice, 24 vectors, n = 80, by a program that autotunes first (fewer
        # slices than 64^3 x 96; slices are independent)
        _case("tuned_64x24_f32_24", dims=(64, 64, 64, 24), links="near", nvec=24, N=80, tuned=True),
        # sink smearing: 72 propagator columns with one two-link field, n = 30
        _case("sinks_48x24_f32_72", dims=(48, 48, 48, 24), links="near", nvec=72, N=30),
        # a new configuration: load, build, smear its three first colour-wall sources, n = 50
        _case("first_source_48x64", kind="config", dims=(48, 48, 48, 64), links="near", nvec=3, N=50, source="wall"),
        # gauge-smeared links: load, three APE steps, build, smear one point source on its slice
        _case("ape_32x32", kind="config", dims=(32, 32, 32, 32), links="near", nvec=1, N=20, source="point", t0=0,
              ape=3),
        # one-link Gaussian smearing of 12 propagator columns
        _case("onelink_32x64_f32_12", kind="onelink", dims=(32, 32, 32, 64), links="near", nvec=12, N=40),
        # serving: twelve jobs in flight on resident 16^3 x 32 and 32^3 x 32 fields, 1-24
        # vectors each, FP32 and FP16 storage, n = 10-80
        _case("serve_12_jobs", kind="serve", dims=(32, 32, 32, 32), nvec=24, N=80, jobs=12, jobs_seed=5),
    ]


def _flops(c):
    """Algorithmic operations of one pass."""
    V = c["lx"] * c["ly"] * c["lz"]
    sites = V * (1 if c["t0"] >= 0 else c["lt"])
    if c["kind"] == "serve":
        return sum(450.0 * j["N"] * j["nvec"] * math.prod(j["dims"]) for j in _jobs(c))
    f = (438.0 if c["kind"] == "onelink" else 450.0) * c["N"] * c["nvec"] * sites
    if c["kind"] == "config":
        # the product, and per APE step and link eight 3x3 products and about four inverses
        f += 648.0 * V * c["lt"] + c["ape"] * 3 * V * c["lt"] * (8 * 198.0 + 4 * 250.0)
    return f


def _cost(c):
    """Rough relative cost: FP64 work counts more on this hardware."""
    f = _flops(c)
    if c["storage"] == "F64":
        return 30.0 * f
    return f + (60.0 * c["ape"] * 3 * 2600.0 * c["lx"] * c["ly"] * c["lz"] * c["lt"] if c["ape"] else 0.0)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(rng, lo, hi):
    return max(lo, 2 * (_log_int(rng, lo, hi) // 2))


def draw(rng):
    kind = rng.choice(("smear", "smear", "smear", "smear", "smear", "config", "onelink", "serve"))
    top = 4.0e12
    while True:
        if rng.random() < 0.7:
            n = _even(rng, 8, 64)
            dims = [n, n, n]
        else:
            dims = [_even(rng, 6, 64) for _ in range(3)]
        dims.append(_log_int(rng, 4, 96))
        N = rng.randint(10, 80)
        s = round(rng.uniform(0.05, 0.3), 3)
        links = rng.choice(("near", "haar"))
        if kind == "smear":
            storage, wprec, recon = rng.choice(FORMATS[:2] + FORMATS[1:])
            nvec = _log_int(rng, 1, 96)
            t0 = rng.randrange(dims[3]) if rng.random() < 0.25 else -1
            c = _case(dims=dims, links=links if recon != 8 else "haar", nvec=nvec, N=N, sigma_per_N=s,
                      storage=storage, wprec=wprec, recon=recon, t0=t0, source=rng.choice(("gauss", "wall", "point")),
                      tuned=rng.random() < 0.2, norms=rng.random() < 0.3)
        elif kind == "config":
            c = _case(kind="config", dims=dims, links=links, nvec=rng.randint(1, 6), N=N, sigma_per_N=s,
                      recon=rng.choice((18, 18, 12)), source=rng.choice(("wall", "point")),
                      ape=rng.choice((0, 0, 1, 2, 3)), host=rng.random() < 0.3)
        elif kind == "onelink":
            storage = rng.choice(("F32", "F32", "F16", "BF16", "F64"))
            c = _case(kind="onelink", dims=dims, links=links, nvec=_log_int(rng, 1, 72), N=N, storage=storage,
                      wprec="F64" if storage == "F64" else "F32")
        else:
            n = _even(rng, 12, 48)
            dims = [n, n, n, _log_int(rng, 4, 64)]
            c = _case(kind="serve", dims=dims, nvec=24, N=80, jobs=rng.randint(2, 16), jobs_seed=rng.randrange(1000))
        V = math.prod(dims)
        if 2e3 <= V <= 8e6 and V * c["nvec"] <= 2e8 and 1e6 <= _cost(c) <= top:
            return c


def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _links(c, dims, seed):
    """SU(3) links [t, z, y, x, 4, 3, 3]: Gram-Schmidt of two rows of complex Gaussians (Haar), or of
    1 + 0.2 i H with H a Gaussian Hermitian matrix (near the unit), and the third row from them."""
    Lx, Ly, Lz, Lt = dims
    g = torch.Generator(device="cuda").manual_seed(seed)
    U = torch.empty((Lt, Lz, Ly, Lx, 4, 3, 3), dtype=torch.complex128, device="cuda")
    for t in range(Lt):
        h = torch.randn((Lz, Ly, Lx, 4, 2, 3, 2), generator=g, device="cuda")
        m = torch.view_as_complex(h).to(torch.complex128)
        if c["links"] == "near":
            d = 0.1 * torch.complex(-m.imag, m.real)  # i H / 5 above the diagonal
            r0 = torch.stack([1 + 0.2j * m[..., 0, 0].real, d[..., 0, 1], d[..., 0, 2]], dim=-1)
            r1 = torch.stack([-d[..., 0, 1].conj(), 1 + 0.2j * m[..., 1, 1].real, d[..., 1, 2]], dim=-1)
        else:
            r0, r1 = m[..., 0, :], m[..., 1, :]
        r0 = r0 * ((r0.real ** 2 + r0.imag ** 2).sum(-1, keepdim=True) ** -0.5)
        r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
        r1 = r1 * ((r1.real ** 2 + r1.imag ** 2).sum(-1, keepdim=True) ** -0.5)
        U[t, ..., 0, :], U[t, ..., 1, :] = r0, r1
        U[t, ..., 2, :] = torch.linalg.cross(r0, r1).conj()
    return U


def _sources(c, dims, nvec, seed, dtype):
    Lx, Ly, Lz, Lt = dims
    g = torch.Generator(device="cuda").manual_seed(seed)
    if c["source"] == "gauss":
        x = torch.empty((nvec, Lt, Lz, Ly, Lx, 3), dtype=dtype, device="cuda")
        torch.view_as_real(x).normal_(generator=g)
        return x
    t = max(c["t0"], 0)
    x = torch.zeros((nvec, Lt, Lz, Ly, Lx, 3), dtype=dtype, device="cuda")
    pos = torch.randint(0, 1 << 20, (nvec, 3), generator=g, device="cuda").tolist()
    for v in range(nvec):
        if c["source"] == "wall":  # a colour wall with the random phases of a stochastic source
            ph = torch.rand((Lz, Ly, Lx), generator=g, device="cuda", dtype=torch.float64) * (2 * math.pi)
            x[v, t, ..., v % 3] = torch.polar(torch.ones_like(ph), ph).to(dtype)
        else:
            px, py, pz = pos[v]
            x[v, t, pz % Lz, py % Ly, px % Lx, v % 3] = 1
    return x


def _dtype(c):
    return torch.complex128 if c["storage"] == "F64" else torch.complex64


def _io(c):
    return tls.TLS_F64 if c["storage"] == "F64" else tls.TLS_F32


def _prec(name):
    return getattr(tls, "TLS_" + name)


def _jobs(c):
    """The burst of a serve case: dims, vectors, steps, width and storage of each job."""
    r = random.Random(c["jobs_seed"])
    small = (16, 16, 16, 32)
    out = []
    for _ in range(c["jobs"]):
        N = r.randint(10, c["N"])
        out.append(dict(dims=r.choice((small, _dims(c))), nvec=r.randint(1, c["nvec"]), N=N,
                        sigma=N * r.uniform(0.05, 0.3), storage=r.choice(("F32", "F16"))))
    return out


def prepare(case, seed):
    c, dims = case, _dims(case)
    st = {"case": c, "ctx": tls.Context(0)}
    ctx = st["ctx"]
    if c["kind"] == "serve":
        gid = {}
        for k, d in enumerate(((16, 16, 16, 32), dims)):
            U = _links(c, d, seed + 7 * k)
            gid[d] = ctx.load_gauge(U, 4, d)
            ctx.build_twolink(gid[d], tls.TLS_F32, 18, keep_U=0)
            del U
        st["jobs"] = []
        for k, j in enumerate(_jobs(c)):
            src = _sources(c, j["dims"], j["nvec"], seed + 100 + k, torch.complex64)
            st["jobs"].append((gid[j["dims"]], src, torch.empty_like(src), j))
        ctx.serve_start(max_slots=48, steps_per_launch=4, use_graphs=1)
        return st
    U = _links(c, dims, seed)
    st["src"] = _sources(c, dims, c["nvec"], seed + 1, _dtype(c))
    st["out"] = torch.empty_like(st["src"])
    if c["kind"] == "config":
        st["U"] = U.cpu().pin_memory() if c["host"] else U
        return st
    st["gid"] = ctx.load_gauge(U, 4, dims)
    del U
    if c["kind"] == "onelink":
        ctx.build_links(st["gid"], _prec(c["wprec"]), keep_U=0)
        return st
    ctx.build_twolink(st["gid"], _prec(c["wprec"]), c["recon"], keep_U=0)
    if c["tuned"]:
        ctx.autotune(st["gid"], c["nvec"], _prec(c["storage"]), c["t0"], steps=4)
    return st


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "serve":
        for _, src, x, _ in state["jobs"]:
            x.copy_(src)
        torch.cuda.current_stream().synchronize()  # the scheduler reads the vectors on its own streams
        ids = [ctx.serve_submit(gid, x, tls.TLS_F32, j["nvec"], j["N"], j["sigma"], storage=_prec(j["storage"]))
               for gid, _, x, j in state["jobs"]]
        for i in ids:
            ctx.serve_wait(i, 120)
        return [x for _, _, x, _ in state["jobs"]]
    x = state["out"]
    x.copy_(state["src"])
    if c["kind"] == "onelink":
        ctx.smear_onelink(state["gid"], x, _io(c), c["nvec"], c["N"], 0.05, storage=_prec(c["storage"]))
        return x
    if c["kind"] == "config":
        gid = ctx.load_gauge(state["U"], 4, _dims(c))
        if c["ape"]:
            ctx.ape_smear(gid, 0.5, c["ape"])
        ctx.build_twolink(gid, _prec(c["wprec"]), c["recon"], keep_U=0)
    else:
        gid = state["gid"]
    norms = ctx.smear(gid, x, _io(c), c["nvec"], c["N"], c["sigma_per_N"] * c["N"], timeslice=c["t0"],
                      storage=_prec(c["storage"]), norms=c["norms"])
    if c["kind"] == "config":
        ctx.free_gauge(gid)
    return [x, norms] if c["norms"] else x


def _wbytes(wprec, recon):
    return {"F64": 8, "F32": 4, "F16": 2, "BF16": 2}[wprec] * recon


def work(case):
    """Links or two-link field and vectors read once, vectors written once."""
    c = case
    if c["kind"] == "serve":
        b = 0.0
        for d in ((16, 16, 16, 32), _dims(c)):
            js = [j for j in _jobs(c) if j["dims"] == d]
            b += math.prod(d) * ((216.0 if js else 0.0) + sum(2 * 24.0 * j["nvec"] for j in js))
        return {"bytes": b, "flops": _flops(c)}
    V = c["lx"] * c["ly"] * c["lz"]
    sites = V * (1 if c["t0"] >= 0 else c["lt"])
    vec = 2.0 * c["nvec"] * sites * (48 if c["storage"] == "F64" else 24)
    if c["kind"] == "config":
        w = V * c["lt"] * 3 * 144.0
    elif c["kind"] == "onelink":
        w = sites * 3.0 * _wbytes(c["wprec"], 18)
    else:
        w = sites * 3.0 * _wbytes(c["wprec"], c["recon"])
    return {"bytes": vec + w, "flops": _flops(c)}


# ---- 64-bit values in plain torch --------------------------------------------------
_AXIS = (3, 2, 1)  # x, y, z of [t, z, y, x, ...]


def _ape_exact(U, a, n):
    def sh(m, mu, d):  # m(x + d mu)
        return torch.roll(m, -d, dims=_AXIS[mu])
    U = U[..., :3, :, :]
    for _ in range(n):
        new = torch.empty_like(U)
        for mu in range(3):
            u = U[..., mu, :, :]
            s = torch.zeros_like(u)
            for nu in range(3):
                if nu == mu:
                    continue
                v = U[..., nu, :, :]
                s += v @ sh(u, nu, 1) @ sh(v, mu, 1).mH
                s += sh(v.mH @ u @ sh(v, mu, 1), nu, -1)
            x = (1 - a) * u + (a / 4) * s
            for _ in range(40):  # Newton's iteration to the unitary polar factor
                r = torch.linalg.cross(x[..., 1, :], x[..., 2, :]), torch.linalg.cross(x[..., 2, :], x[..., 0, :]), \
                    torch.linalg.cross(x[..., 0, :], x[..., 1, :])
                cof = torch.stack(r, dim=-2)
                det = (x[..., 0, :] * cof[..., 0, :]).sum(-1)
                y = 0.5 * (x + (cof / det[..., None, None]).conj())
                small = float((y - x).abs().max()) < 1e-14
                x = y
                if small:
                    break
            det = (x[..., 0, :] * torch.linalg.cross(x[..., 1, :], x[..., 2, :])).sum(-1)
            phi = torch.angle(det) / 3
            new[..., mu, :, :] = x * torch.polar(torch.ones_like(phi), -phi)[..., None, None]
        U = new
    return U


def _steps(A, x, hop, N, alpha, diag):
    """N steps of x <- x + alpha (sum of hops + diag x) on [t, z, y, x, 3, nvec]; A holds the six
    matrices of each site side by side, [t, z, y, x, 3, 18]."""
    for _ in range(N):
        b = torch.cat([torch.roll(x, s * hop, dims=_AXIS[mu]) for mu in range(3) for s in (-1, 1)], dim=-2)
        x = x + alpha * (A @ b + diag * x)
    return x


def _smear_exact(links, src, N, alpha, hop, diag, t0):
    """links(t): one slice [1, z, y, x, 3, 3, 3] of the matrices of the forward hops."""
    out = src.to(torch.complex128).clone()
    for t in ([t0] if t0 >= 0 else range(src.shape[1])):
        if not bool(torch.count_nonzero(src[:, t])):
            continue
        M = links(t)
        A = torch.cat([m for mu in range(3)
                       for m in (M[..., mu, :, :], torch.roll(M[..., mu, :, :], hop, dims=_AXIS[mu]).mH)], dim=-1)
        x = out[:, t].permute(1, 2, 3, 4, 0)[None].contiguous()
        out[:, t] = _steps(A, x, hop, N, alpha, diag)[0].permute(4, 0, 1, 2, 3)
    return out


def _twolink(U):
    return torch.stack([U[..., mu, :, :] @ torch.roll(U[..., mu, :, :], -1, dims=_AXIS[mu]) for mu in range(3)],
                       dim=-3)


def exact(case, seed):
    c, dims = case, _dims(case)
    active = _flops(c)
    if c["source"] != "gauss" and c["t0"] < 0:
        active /= c["lt"]  # one slice holds the source, the others stay zero
    if active > 2e12:
        return None
    if c["kind"] == "serve":
        fields = {d: _links(c, d, seed + 7 * k) for k, d in enumerate(((16, 16, 16, 32), dims))}
        out = []
        for k, j in enumerate(_jobs(c)):
            src = _sources(c, j["dims"], j["nvec"], seed + 100 + k, torch.complex64)
            U = fields[j["dims"]]
            out.append(_smear_exact(lambda t: _twolink(U[t:t + 1]), src, j["N"], j["sigma"] / (4 * j["N"]), 2, -6.0,
                                    -1))
        return out
    U = _links(c, dims, seed)
    src = _sources(c, dims, c["nvec"], seed + 1, _dtype(c))
    if c["kind"] == "onelink":
        return _smear_exact(lambda t: U[t:t + 1, ..., :3, :, :], src, c["N"], 0.05, 1, 0.0, -1)
    def twolink(t):
        u = U[t:t + 1]
        return _twolink(_ape_exact(u, 0.5, c["ape"]) if c["ape"] else u)
    x = _smear_exact(twolink, src, c["N"], c["sigma_per_N"] / 4, 2, -6.0, c["t0"])
    if not c["norms"]:
        return x
    part = x if c["t0"] < 0 else x[:, c["t0"]:c["t0"] + 1]
    return [x, (part.abs() ** 2).reshape(c["nvec"], -1).sum(1)]
