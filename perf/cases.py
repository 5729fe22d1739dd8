"""The work that users of this framework have it do, as cases to time and to compare.

A case is a chain of heatbath sweeps (one lattice, an ensemble, a served mix
of jobs, or a pipeline step with host input) of the kind the verification
runs, the benchmark and the tests use.  `prepare` builds what a program holds
before the call, `run` makes one pass through the public Python API, `exact`
states the result in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_0904_0642_gb300 as su3

STORAGE = {"fp64_18": su3.SU3_FP64_18, "fp32_12": su3.SU3_FP32_12, "fp32_18": su3.SU3_FP32_18}
BYTES_PER_LINK = {"fp64_18": 144, "fp32_12": 48, "fp32_18": 72}

BASE = {
    "kind": "chain",      # chain, ensemble, served, input
    "dims": "4x4x4x4",    # even extents; served: one shape per job, separated by spaces
    "layers": 1,          # 2: the double-layered torus
    "glue": 0,            # its glued directions (0: all)
    "storage": "fp64_18",
    "beta": 6.0,
    "hits": 2,
    "sweeps": 1,          # sweeps of one pass
    "reunit": 10,         # re-unitarise every so many sweeps
    "measure": 0,         # record plaquette and Polyakov loop every so many sweeps
    "read": "",           # what the program reads after the sweeps: "", "latest", "plaquette"
    "ndiv": "",           # sublattices per direction
    "chains": 1,          # ensemble: chains of the same shape
    "tuned": False,       # launch shape from the autotuner, as the benchmark does
}


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # The plain double-precision sweep of the smallest lattice, one sweep
        # at a time: a first program, and the parity workload.
        _case("f64_4^4", dims="4x4x4x4", beta=6.0, hits=2, sweeps=1),
        # The paper's Table 1 run (one hit, a measurement every second sweep)
        # in the default storage: measured between short runs of sweeps.
        _case("f64_8^3x4", dims="8x8x8x4", beta=5.65, hits=1, sweeps=10, measure=2, read="latest"),
        # The double-layered torus of Table 3, all directions glued.
        _case("f64_dlt_8^3x4", dims="8x8x8x4", layers=2, beta=5.55, hits=1, sweeps=4),
        # A large double-precision lattice whose extents are no power of two;
        # the program asks for the plaquette after every sweep.
        _case("f64_24^4", dims="24x24x24x24", beta=6.0, hits=2, sweeps=1, read="plaquette"),
        # The paper's small lattice in float: long runs of sweeps with
        # measurements, as the verification campaign makes them.
        _case("f32_8^3x4", dims="8x8x8x4", storage="fp32_12", beta=5.65, hits=1, sweeps=40, measure=2, read="latest"),
        # The same cut into the paper's sublattices with halo exchange.
        _case("f32_8^3x4_cut", dims="8x8x8x4", storage="fp32_12", beta=5.65, hits=1, sweeps=40, measure=2,
              read="latest", ndiv="2x2x2x1"),
        # Finite temperature on the double-layered torus, glued in time.
        _case("f32_dlt_16^3x4", dims="16x16x16x4", layers=2, glue=8, storage="fp32_12", beta=5.7, sweeps=10),
        # Three dimensions.
        _case("f32_64^3", dims="64x64x64", storage="fp32_12", beta=10.0, sweeps=10),
        # The 18-real float form, a mid-sized ragged lattice.
        _case("f32_18_18^3x12", dims="18x18x18x12", storage="fp32_18", beta=5.9, hits=2, sweeps=10, measure=10,
              read="latest"),
        # The benchmark's chain: larger than L2, tuned, a re-unitarisation
        # and a measurement every ten sweeps.
        _case("f32_32^4", dims="32x32x32x32", storage="fp32_12", beta=6.0, sweeps=10, measure=10, tuned=True),
        # Many chains in one fused launch per phase.
        _case("f32_256x8^4", kind="ensemble", dims="8x8x8x8", chains=256, storage="fp32_12", beta=6.0, sweeps=10),
        # Jobs of different shapes through the server.
        _case("served_8_jobs", kind="served", storage="fp32_12", beta=6.0, sweeps=20,
              dims="8x8x8x8 12x12x12x12 16x16x16x4 8x8x8x8 24x24x24 12x12x12x12 8x8x8x4 16x16x16x4"),
    ]


def _dims(text):
    return [int(n) for n in text.split("x")]


def _even(rng, lo, hi):
    """An even extent, spread over the logarithm of its range."""
    return 2 * int(round(math.exp(rng.uniform(math.log(lo / 2), math.log(hi / 2)))))


def _volume(dims):
    v = 1
    for n in dims:
        v *= n
    return v


def _updates(case):
    """Link updates of one pass."""
    shapes = [_dims(t) for t in case["dims"].split(" ")]
    return case["sweeps"] * case["layers"] * case["chains"] * sum(_volume(d) * len(d) for d in shapes)


#: Link updates of one pass at most, by storage: those of the largest listed case of each.
MOST = {"fp64_18": 1_400_000, "fp32_12": 42_000_000, "fp32_18": 20_000_000}


def draw(rng):
    while True:
        kind = rng.choice(["chain"] * 8 + ["ensemble", "input", "served"])
        storage = rng.choice(["fp64_18", "fp64_18", "fp32_12", "fp32_12", "fp32_18"]) if kind != "served" else "fp32_12"
        D = rng.choice([4, 4, 4, 3, 2])
        c = dict(BASE, kind=kind, storage=storage, beta=round(rng.uniform(5.5, 6.5) if D == 4 else rng.uniform(5.5, 12.0), 3),
                 hits=rng.choice([1, 2, 2, 3]))
        hi = {4: 32, 3: 64, 2: 256}[D]
        dims = [_even(rng, 4, hi) for _ in range(D)]
        if kind == "ensemble":
            dims = [_even(rng, 4, 12) for _ in range(D)]
            c["chains"] = _even(rng, 2, 256)
        c["dims"] = "x".join(map(str, dims))
        if kind == "served":
            c["dims"] = " ".join("x".join(str(_even(rng, 4, 16)) for _ in range(rng.choice([3, 4, 4])))
                                 for _ in range(rng.randint(2, 8)))
        if kind == "chain":
            if rng.random() < 0.3:
                c["layers"], c["glue"] = 2, rng.choice([0, 1 << (D - 1), (1 << (D - 1)) - 1])
            elif storage != "fp64_18" and rng.random() < 0.15:
                c["ndiv"] = "x".join("2" if n % 4 == 0 and n < 16 else "1" for n in dims)
            c["read"] = rng.choice(["", "latest", "plaquette"])
            c["measure"] = 2 if c["read"] == "latest" else 0
        if kind == "input":
            c["read"], c["measure"] = "latest", 2
        c["sweeps"] = _even(rng, 2, 20 if storage != "fp64_18" else 10 if D == 4 else 2)
        if 1000 <= _updates(c) <= MOST[storage] and ("2" in c["ndiv"] or not c["ndiv"]):
            return c


# ---------------------------------------------------------------- inputs


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _gram_schmidt(m):
    a = m[..., 0, :]
    a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
    b = m[..., 1, :]
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2)


def _shift(t, axis, step, layers, glued):
    """Field at x + step e on [layer, x^D .. x^1, ...]; a step across a glued boundary changes the layer."""
    r = torch.roll(t, -step, axis)
    if layers == 2 and glued:
        at = [slice(None)] * r.ndim
        at[axis] = r.shape[axis] - 1 if step > 0 else 0
        r[tuple(at)] = r[tuple(at)].flip(0)
    return r


def _glued(case, D):
    return [case["layers"] == 2 and bool(((case["glue"] or (1 << D) - 1) >> mu) & 1) for mu in range(D)]


def _start(case, dims, seed):
    """Links of a chain in equilibrium, as far as one link update can tell:
    Haar-random links whose plaquette average is about 0.58 (a random gauge
    transformation of links near one).  complex128 [layer, x^D .. x^1, mu, 3, 3]."""
    D, L = len(dims), case["layers"]
    g = torch.Generator(device=_device()).manual_seed(int(seed) & 0x7FFFFFFF)

    def gauss(*shape):
        return torch.complex(*[torch.randn(*shape, generator=g, device=_device(), dtype=torch.float64) for _ in range(2)])

    grid = [L] + dims[::-1]
    one = torch.eye(3, device=_device(), dtype=torch.complex128)
    U = _gram_schmidt(one + 0.22 * gauss(*grid, D, 3, 3))
    G = _gram_schmidt(gauss(*grid, 3, 3))
    glued = _glued(case, D)
    for mu in range(D):
        far = _shift(G, D - mu, 1, L, glued[mu])
        U[..., mu, :, :] = G @ U[..., mu, :, :] @ far.mH
    return U


_stream = None


def _one_stream():
    """The stream of all of a program's lattices: their passes follow one another."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _canonical(U):
    """[layer][site][mu][row][col][re, im] doubles."""
    return torch.view_as_real(U.contiguous()).reshape(U.shape[0], -1, U.shape[-3], 3, 3, 2)


def _boundary(case):
    return su3.SU3_DLT if case["layers"] == 2 else su3.SU3_PBC


def _config(case, dims, seed, **kw):
    return su3.make_config(dims, boundary=_boundary(case), glue_mask=case["glue"], beta=case["beta"], seed=seed,
                           storage=STORAGE[case["storage"]], hits=case["hits"], reunit_every=case["reunit"],
                           measure_every=case["measure"], measure_capacity=64, **kw)


def _chain_seed(seed):
    return 20090406 + int(seed)


def _buffer(case, dims):
    n = case["layers"] * _volume(dims) * len(dims) * BYTES_PER_LINK[case["storage"]]
    f64 = case["storage"] == "fp64_18"
    return torch.zeros(n // (8 if f64 else 4), device="cuda", dtype=torch.float64 if f64 else torch.float32)


def prepare(case, seed):
    dims = _dims(case["dims"].split(" ")[0])
    s = {"case": case}
    if case["kind"] == "ensemble":
        betas = np.random.default_rng(2009 + int(seed)).uniform(case["beta"] - 0.3, case["beta"] + 0.3, case["chains"])
        s["buf"] = torch.stack([_buffer(case, dims) for _ in betas])  # one row of links per chain
        torch.cuda.synchronize()
        s["ens"] = su3.Ensemble([_config(dict(case, beta=float(b)), dims, _chain_seed(seed) + 5000 * (i + 1),
                                         start=su3.SU3_START_HOT, buffer=s["buf"][i]) for i, b in enumerate(betas)],
                              stream=_one_stream())
        return s
    if case["kind"] == "served":
        s["jobs"] = []
        for i, text in enumerate(case["dims"].split(" ")):
            d = _dims(text)
            s["jobs"].append((_config(case, d, _chain_seed(seed) + i, start=su3.SU3_START_HOT),
                              np.zeros((case["layers"], _volume(d), len(d), 3, 3, 2))))
        s["server"] = su3.Server(max_slots=64)
        return s
    kw = {}
    if case["ndiv"]:
        kw["ndiv"] = _dims(case["ndiv"])
    else:
        s["buf"] = _buffer(case, dims)
        torch.cuda.synchronize()
    links = _canonical(_start(case, dims, seed)).cpu()
    s["lat"] = su3.Lattice(dims, boundary=_boundary(case), glue_mask=case["glue"], beta=case["beta"],
                           seed=_chain_seed(seed), storage=STORAGE[case["storage"]], hits=case["hits"],
                           reunit_every=case["reunit"], measure_every=case["measure"], measure_capacity=64,
                           buffer=s.get("buf"), stream=_one_stream(), **kw)
    if case["kind"] == "input":
        rows = links[..., :2, :, :].to(torch.float32).contiguous().pin_memory()
        s["pinned"], s["rows"] = rows, rows.numpy()
    else:
        s["lat"].set_links(links.numpy())
    if case["tuned"]:
        s["lat"].autotune()
    return s


# ---------------------------------------------------------------- one pass


def run(s):
    case = s["case"]
    if case["kind"] == "ensemble":
        s["ens"].sweep(case["sweeps"])
        return s["buf"]
    if case["kind"] == "served":
        ids = [s["server"].submit(cfg, case["sweeps"], links_out=out) for cfg, out in s["jobs"]]
        done = [s["server"].wait(i, 60.0) for i in ids]
        return [[np.array(list(r.plaquette) + list(r.polyakov)) for r in done], [out for _, out in s["jobs"]]]
    lat = s["lat"]
    if case["kind"] == "input":
        lat.stage_links(s["rows"], su3.SU3_LINKS_FP32_12)
        lat.apply_links()
    lat.sweep(case["sweeps"])
    out = []
    if case["read"] == "latest":
        out.append(lat.latest_measurement())
    elif case["read"] == "plaquette":
        out.append(np.array(lat.plaquette()))
    out.append(s["buf"] if "buf" in s else lat.get_links())
    return out


def work(case):
    """Links read once and written once per pass (and what the host hands in
    or takes out), and the arithmetic of every link update of the pass."""
    shapes = [_dims(t) for t in case["dims"].split(" ")]
    nbytes = flops = 0.0
    for d in shapes:
        links = case["layers"] * case["chains"] * _volume(d) * len(d)
        nbytes += 2 * links * BYTES_PER_LINK[case["storage"]]
        if case["kind"] == "served" or case["ndiv"]:
            nbytes += links * 144  # the links go to the host
        if case["kind"] == "input":
            nbytes += links * 48
        # per staple two two-row products, their third rows and the sum; then
        # three projections, draws and rotations
        flops += case["sweeps"] * links * (2 * (len(d) - 1) * 2 * 204 + 3 * 2 * 200)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits

_M32 = 0xFFFFFFFF


def _mulhilo(m, c):
    """High and low words of m c for 32-bit words held in int64."""
    p = c * (m >> 16) + ((c * (m & 0xFFFF)) >> 16)
    return p >> 16, (c * m) & _M32


def _philox(c, key):
    """Philox4x32-10 (Salmon, Moraes, Dror, Shaw)."""
    c, (k0, k1) = list(c), key
    for r in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _uniform(w):
    return (w.double() + 0.5) * 2.0 ** -32


def _su2_draw(alpha, hits, site, sweep, tag, key):
    """Kennedy-Pendleton: x0..x3 from exp(alpha x0) and which sites accepted."""
    zero = torch.zeros_like(site)
    X, acc = torch.zeros_like(alpha), torch.zeros_like(alpha, dtype=torch.bool)
    for h in range(hits):
        w = _philox((site, zero + sweep, zero + (tag | h), zero), key)
        cs = torch.cos(2 * math.pi * _uniform(w[1]))
        new = -(torch.log(_uniform(w[0])) + cs * cs * torch.log(_uniform(w[2]))) / alpha
        X = torch.where(acc, X, new)
        acc = acc | (_uniform(w[3]).square() <= 1 - 0.5 * new)
    sg = (tag >> 8) & 3
    w = _philox((site, zero + sweep, zero + ((tag & ~(3 << 8)) | ((sg & 2) << 8) | 255), zero), key)
    u, v = (w[2], w[3]) if sg == 1 else (w[0], w[1])
    ct, phi = 2 * _uniform(u) - 1, 2 * math.pi * _uniform(v)
    st, rho = torch.sqrt(1 - ct * ct), torch.sqrt((X * (2 - X)).clamp_min(0))
    return (1 - X, rho * st * torch.cos(phi), rho * st * torch.sin(phi), rho * ct), acc


def _sweep(U, case, dims, sweep, seed, site, parity):
    D, L = len(dims), case["layers"]
    glued = _glued(case, D)
    key = (seed & _M32, seed >> 32)

    def sh(t, mu, step):
        return _shift(t, D - mu, step, L, glued[mu])

    for colour in range(2):
        on = parity == colour
        for mu in range(D):
            A = torch.zeros_like(U[..., 0, :, :])
            for nu in range(D):
                if nu != mu:
                    um, un = U[..., mu, :, :], U[..., nu, :, :]
                    far = sh(un, mu, 1)
                    A += far @ sh(um, nu, 1).mH @ un.mH
                    A += sh(far.mH @ um.mH @ un, nu, -1)
            u = U[..., mu, :, :].clone()
            for sg, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
                wi = u[..., (i, j), :] @ A[..., :, (i, j)]
                a = ((wi[..., 0, 0] + wi[..., 1, 1]).real / 2, (wi[..., 0, 1] + wi[..., 1, 0]).imag / 2,
                     (wi[..., 0, 1] - wi[..., 1, 0]).real / 2, (wi[..., 0, 0] - wi[..., 1, 1]).imag / 2)
                k = torch.sqrt(sum(t * t for t in a))
                tag = (sg << 8) | (mu << 10) | (colour << 14)
                x, ok = _su2_draw(2 * case["beta"] * k / 3, case["hits"], site, sweep, tag, key)
                v = [t / k for t in a]
                # r = x v^+
                r0 = x[0] * v[0] + x[1] * v[1] + x[2] * v[2] + x[3] * v[3]
                r1 = -x[0] * v[1] + v[0] * x[1] + (x[2] * v[3] - x[3] * v[2])
                r2 = -x[0] * v[2] + v[0] * x[2] + (x[3] * v[1] - x[1] * v[3])
                r3 = -x[0] * v[3] + v[0] * x[3] + (x[1] * v[2] - x[2] * v[1])
                R = torch.stack([torch.stack([torch.complex(r0, r3), torch.complex(r2, r1)], -1),
                                 torch.stack([torch.complex(-r2, r1), torch.complex(r0, -r3)], -1)], -2)
                rows = torch.matmul(R, u[..., (i, j), :])
                go = (ok & on)[..., None, None]
                u[..., (i, j), :] = torch.where(go, rows, u[..., (i, j), :])
            U[..., mu, :, :] = u


def _measured(U, case, dims):
    """[total, space, time, Re, Im of the Polyakov loop] per layer, then for all."""
    D, L = len(dims), case["layers"]
    glued = _glued(case, D)

    def sh(t, mu, step=1):
        return _shift(t, D - mu, step, L, glued[mu])

    space, time = torch.zeros(L, device=U.device, dtype=torch.float64), torch.zeros(L, device=U.device, dtype=torch.float64)
    for mu in range(D):
        for nu in range(mu + 1, D):
            um, un = U[..., mu, :, :], U[..., nu, :, :]
            p = (um @ sh(un, mu) @ (un @ sh(um, nu)).mH).diagonal(dim1=-2, dim2=-1).sum(-1).real
            t = p.reshape(L, -1).mean(1) / 3
            if nu == D - 1:
                time += t / (D - 1)
            else:
                space += t / ((D - 1) * (D - 2) / 2)
    P = step = U[..., D - 1, :, :]
    for _ in range(dims[D - 1] * (2 if glued[D - 1] else 1) - 1):
        step = sh(step, D - 1)
        P = P @ step
    loop = P[:, 0].diagonal(dim1=-2, dim2=-1).sum(-1).reshape(L, -1).mean(1) / 3
    ns, nt = (D - 1) * (D - 2) / 2, D - 1
    per = torch.stack([(space * ns + time * nt) / (ns + nt), space, time, loop.real, loop.imag], 1)
    return torch.cat([per, per.mean(0, keepdim=True)])


def _stored(U, case):
    """The links in the layout of the caller's buffer: planes [layer][colour][mu][vector][jj]."""
    L, D = case["layers"], U.shape[-3]
    dims = list(U.shape[1:1 + D])[::-1]
    c = _canonical(U).reshape(L, _volume(dims), D, 18)
    c = c[..., :12] if case["storage"] == "fp32_12" else c
    planes = []
    colour = _parity(dims, U.device).reshape(-1)
    for l in range(L):
        for col in range(2):
            for mu in range(D):
                v = c[l, colour == col, mu]  # [jj][values]
                if case["storage"] == "fp64_18":
                    planes.append(v.reshape(-1, 9, 2).permute(1, 0, 2).reshape(-1))
                else:
                    planes.append(v[:, :12].reshape(-1, 3, 4).permute(1, 0, 2).reshape(-1))
                    if case["storage"] == "fp32_18":
                        planes += [v[:, 12:16].reshape(-1), v[:, 16:].reshape(-1)]
    return torch.cat(planes)


def _parity(dims, device):
    p = torch.zeros([1] * len(dims), device=device, dtype=torch.int64)
    for i, n in enumerate(dims):
        shape = [1] * len(dims)
        shape[len(dims) - 1 - i] = n
        p = p + torch.arange(n, device=device).reshape(shape)
    return p & 1


def _rounded(U, storage):
    """The links as the storage keeps them."""
    if storage == "fp64_18":
        return U
    U = torch.view_as_complex(torch.view_as_real(U).float().double())
    if storage == "fp32_12":
        U = torch.stack([U[..., 0, :], U[..., 1, :], torch.linalg.cross(U[..., 0, :], U[..., 1, :]).conj()], -2)
    return U


def exact(case, seed):
    # Float chains long enough for a decision to fall the other way in
    # float say nothing; an ensemble's and a job's start is the library's own.
    if case["kind"] in ("ensemble", "served") or _updates(case) > (1_500_000 if case["storage"] == "fp64_18" else 200_000):
        return None
    dims = _dims(case["dims"])
    U = _start(case, dims, seed)
    U = _rounded(U, "fp32_12" if case["kind"] == "input" else case["storage"])
    D, L = len(dims), case["layers"]
    site = torch.arange(L * _volume(dims), device=U.device).reshape([L] + dims[::-1])
    parity = _parity(dims, U.device).expand(site.shape)
    last = None
    for n in range(1, case["sweeps"] + 1):
        _sweep(U, case, dims, n - 1, _chain_seed(seed), site, parity)
        if case["reunit"] and n % case["reunit"] == 0:
            U = _gram_schmidt(U)
        if case["measure"] and n % case["measure"] == 0:
            last = _measured(U, case, dims) if n + case["measure"] > case["sweeps"] else None
    out = []
    if case["read"] == "latest":
        out.append(last)
    elif case["read"] == "plaquette":
        out.append(_measured(U, case, dims)[-1, :3])
    out.append(_canonical(U) if case["ndiv"] else _stored(U, case))
    return out
