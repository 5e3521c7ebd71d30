"""Workloads for timing the library through its public calls, and their results in plain 64-bit torch.

A case is a dict: "call" names the entry point, the rest are its sizes and options.

    matvec    vie_matvec on device vectors, as a Krylov solver of the caller's applies it
    jm        vie_jm_matvec: the coupled electric and magnetic system
    pwc       vie_matvec of a piecewise-constant handle
    hfields   vie_hfields: magnetic field, b1+ and magnetic energy of a solution (the K operator, FP64)
    solve     vie_solve and vie_fields on a handle that is kept
    request   a new subject from the material map to the maps: vie_setup, vie_rhs_dipoles, vie_solve, vie_fields
"""

import math

import numpy as np
import torch

import paper_1902_02196_gb300 as vie

PRECISION = {"f32": vie.VIE_FP32, "f64": vie.VIE_FP64, "bf16x3": vie.VIE_BF16X3}
OPERATOR = {"A": vie.VIE_OP_A, "PA": vie.VIE_OP_PA, "NSCAT": vie.VIE_OP_NSCAT}

# The 60 distinct tensors of the PWL system: vector pairs p <= q, scalar pairs l <= l'
VECTOR_PAIRS = [(p, q) for p in range(3) for q in range(p, 3)]
SCALAR_PAIRS = [(l, m) for l in range(4) for m in range(l, 4)]


def _case(name, call, nx, ny, nz, voxel, nrhs, precision="f32", op="PA", freq=298e6, **more):
    return {"name": name, "call": call, "nx": nx, "ny": ny, "nz": nz, "voxel": voxel, "nrhs": nrhs,
            "precision": precision, "op": op, "freq": freq, **more}


def listed():
    return [
        # The smallest call: one current on the 16^3 sphere grid, where launches and latency count.
        _case("matvec_sphere16", "matvec", 16, 16, 16, 0.0125, 1),
        # Three sources on an odd box whose x and y transforms differ in length (64 and 128 points).
        _case("matvec_ragged", "matvec", 30, 61, 41, 0.0035, 3, op="A"),
        # One Arnoldi step of the head benchmark: 64^3 voxels of 3 mm, sixteen coil elements.
        _case("matvec_head64", "matvec", 64, 64, 64, 0.003, 16),
        # One Arnoldi step of the body grid at 128 MHz, the largest grid of the configurations.
        _case("matvec_body128", "matvec", 128, 128, 256, 0.005, 8, freq=128e6),
        # The residual of a refinement sweep, and every step of a plain FP64 solve, on the head grid.
        _case("matvec_head64_f64", "matvec", 64, 64, 64, 0.003, 16, precision="f64"),
        # FP64 on the 31^3 grid of the sphere comparison, one plane wave.
        _case("matvec_sphere31_f64", "matvec", 31, 31, 31, 0.005, 1, precision="f64", op="A"),
        # The tensor-core precision on the inclusions grid with its 32 sources.
        _case("matvec_incl64_bf16x3", "matvec", 64, 64, 64, 0.002, 32, precision="bf16x3", freq=447e6),
        # Transmit fields of eight coil elements after a head solve.
        _case("hfields_head64", "hfields", 64, 64, 64, 0.003, 8, precision="f64"),
        # One step of the magnetodielectric solve's inner iteration at 32^3.
        _case("jm_matvec32", "jm", 32, 32, 32, 0.00625, 1),
        # The comparison solver with constant basis functions on the 61^3 sphere grid.
        _case("pwc_sphere61_f64", "pwc", 61, 61, 61, 0.0025, 1, precision="f64", op="A"),
        # One request of a serving stream: a 32^3 head with eight sources, everything from the material map on.
        _case("request_head32", "request", 32, 32, 32, 0.006, 8),
        # The head benchmark's whole solve and its maps on a kept handle.
        _case("solve_head64", "solve", 64, 64, 64, 0.003, 16),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    # operator applications are most of what the library does, FP32 ones above all
    call, precision = rng.choice([("matvec", "f32")] * 4 + [("matvec", "f64")] * 2 + [("matvec", "bf16x3")] +
                                 [("hfields", "f64"), ("jm", "f32"), ("jm", "f64"), ("pwc", "f32"), ("pwc", "f64"),
                                  ("solve", "f32"), ("request", "f32")])
    whole = call in ("solve", "request")
    top = {"solve": 40, "request": 32, "pwc": 64}.get(call, 96)
    nx = log_int(12, top)
    if rng.random() < 0.5:  # a cube-like box, or one with sides of its own
        ny, nz = nx, max(8, min(top, nx + rng.randint(-4, 4)))
    else:
        ny, nz = log_int(12, top), log_int(8, top)
    most = max(1, min(32, (16 if precision != "f64" else 8) * 64 ** 3 // (nx * ny * nz)))
    nrhs = log_int(1, min(8, most) if whole else most)
    op = "PA" if whole or call == "hfields" else rng.choice(["PA", "PA", "A"] + (["NSCAT"] if call != "jm" else []))
    return {"call": call, "nx": nx, "ny": ny, "nz": nz, "voxel": round(0.192 / max(nx, ny, nz), 6), "nrhs": nrhs,
            "precision": precision, "op": op, "freq": rng.choice([64e6, 128e6, 298e6])}


def _grid(case):
    return (case["nx"], case["ny"], case["nz"], case["voxel"], case["voxel"], case["voxel"])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _materials(case, g):
    """eps_r and sigma of an ellipsoid of four tissue shells with 15% noise, air around it."""
    n = (case["nz"], case["ny"], case["nx"])
    axes = [(torch.arange(k, device="cuda", dtype=torch.float64) + 0.5 - k / 2) / (0.48 * k) for k in n]
    rho = (axes[0][:, None, None] ** 2 + axes[1][None, :, None] ** 2 + axes[2][None, None, :] ** 2).sqrt()
    eps, sig = torch.ones(n, device="cuda", dtype=torch.float64), torch.zeros(n, device="cuda", dtype=torch.float64)
    noise = 1 + 0.15 * torch.randn(n, device="cuda", dtype=torch.float64, generator=g).clamp(-3, 3)
    for scale, e, s in ((1.0, 40.0, 0.6), (0.92, 15.0, 0.1), (0.85, 75.0, 2.0), (0.6, 52.0, 0.55)):
        eps = torch.where(rho <= scale, (e * noise).clamp(5, 80), eps)
        sig = torch.where(rho <= scale, (s * noise).clamp(0.05, 2), sig)
    return eps, sig


def _vector(shape, dtype, g):
    """Current coefficients: complex normal, as a Krylov vector has them."""
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(*shape, 2, device="cuda", dtype=real, generator=g))


def _derivative(n, d, f):
    """The derivative of order n = (n_x, n_y, n_z) of a function of the distance; f[k] = (1/rho d/drho)^k of it."""
    out = 0
    for m in ((a, b, c) for a in range(n[0] // 2 + 1) for b in range(n[1] // 2 + 1) for c in range(n[2] // 2 + 1)):
        w, term = 1.0, f[sum(n) - sum(m)]
        for i in range(3):
            w *= math.factorial(n[i]) / (math.factorial(m[i]) * math.factorial(n[i] - 2 * m[i]) * 2 ** m[i])
            if n[i] > 2 * m[i]:
                term = term * d[i] ** (n[i] - 2 * m[i])
        out = out + w * term
    return out


def _toeplitz(case):
    """The 60 tensors of N - G at offsets >= 0, [nz][ny][nx] complex128 each: the free-space dyadic Green function
    between voxel centres, softened inside a voxel's own sphere, and its derivatives for the linear functions."""
    k0, h = 2 * math.pi * case["freq"] / 299792458.0, case["voxel"]
    z, y, x = (torch.arange(case[k], device="cuda", dtype=torch.float64) * h for k in ("nz", "ny", "nx"))
    d = (x[None, None, :], y[None, :, None], z[:, None, None])
    r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2 + h * h * (3 / (4 * math.pi)) ** (2 / 3)
    rho = r2.sqrt()
    e = torch.polar(torch.ones_like(rho) / (4 * math.pi), -k0 * rho)
    below, f = e * (1j / k0), [e / rho]
    for k in range(4):
        below, nxt = f[-1], -((2 * k + 1) * f[-1] + k0 * k0 * below) / r2
        f.append(nxt)
    for p, q in VECTOR_PAIRS:
        for l, m in SCALAR_PAIRS:
            n = [0, 0, 0]
            for a in (l, m):
                if a:
                    n[a - 1] += 1
            full = list(n)
            full[p] += 1
            full[q] += 1
            t = _derivative(full, d, f)
            if p == q:
                t = t + k0 * k0 * _derivative(n, d, f)
            yield (4 * p + l, 4 * q + m), (-1 if m else 1) * h ** 6 * (h / 12) ** sum(n) * t


def _gram(case, alpha):
    return case["voxel"] ** 3 * (1.0 if alpha % 4 == 0 else 1 / 12)


def _kept_handle(case, eps, sig):
    """A handle on the tensors of _toeplitz, which a caller hands in and which are quick to make."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    # the call takes all 144 entries at all offsets and reads these
    table = torch.zeros(144, 2 * nz - 1, 2 * ny - 1, 2 * nx - 1, device="cuda", dtype=torch.complex128)
    for (a, b), t in _toeplitz(case):
        part = table[12 * a + b, nz - 1:, ny - 1:, nx - 1:]
        part.copy_(t)
        if a == b:
            part[0, 0, 0] += _gram(case, a)
    torch.cuda.synchronize()
    handle = vie.vie_setup_green_external(_grid(case), case["freq"], eps, sig, table)
    del table, part
    torch.cuda.empty_cache()
    return handle


def _dipoles(case, seed):
    """One z-directed source per right-hand side on a ring outside the box."""
    rng = np.random.default_rng(seed)
    phi = 2 * np.pi * (np.arange(case["nrhs"]) + rng.uniform()) / case["nrhs"]
    radius = 0.78 * case["voxel"] * max(case["nx"], case["ny"])
    pos = np.stack([radius * np.cos(phi), radius * np.sin(phi), np.zeros(case["nrhs"])], axis=1)
    return pos, np.tile([0.0, 0.0, 1.0], (case["nrhs"], 1))


def prepare(case, seed):
    g = _generator(seed)
    call, R, n = case["call"], case["nrhs"], (case["nz"], case["ny"], case["nx"])
    eps, sig = _materials(case, g)
    s = {"case": case}
    c128 = dict(device="cuda", dtype=torch.complex128)
    if call in ("matvec", "pwc", "jm"):
        dtype = torch.complex128 if case["precision"] == "f64" else torch.complex64
        if call == "pwc":
            s["h"] = vie.vie_setup(_grid(case), case["freq"], eps, sig, vie.VIE_SETUP_PWC)
        else:
            s["h"] = _kept_handle(case, eps, sig)
        if call == "jm":  # a magnetodielectric body: the same shells with a permeability
            vie.vie_set_permeability(s["h"], torch.where(eps > 1, 2.0, 1.0).double(),
                                     torch.where(eps > 1, 0.5, 0.0).double())
        s["x"] = _vector((R, {"matvec": 12, "pwc": 3, "jm": 24}[call], *n), dtype, g)
        s["y"] = torch.empty_like(s["x"])
    elif call == "hfields":
        s["h"] = _kept_handle(case, eps, sig)
        s["x"] = _vector((R, 12, *n), torch.complex128, g) * (eps > 1)
        s["h_inc"] = _vector((R, 12, *n), torch.complex128, g) * case["voxel"] ** 3
        s["out"] = torch.empty(R, 12, *n, **c128)
        s["b1"] = torch.empty(R, *n, **c128)
    else:
        s["dipoles"] = _dipoles(case, seed)
        for k in ("e_inc", "b", "x", "e"):
            s[k] = torch.empty(R, 12, *n, **c128)
        s["p_abs"] = torch.empty(R, *n, device="cuda", dtype=torch.float64)
        if call == "solve":
            s["h"] = vie.vie_setup(_grid(case), case["freq"], eps, sig)
            vie.vie_rhs_dipoles(s["h"], *s["dipoles"], s["e_inc"], s["b"])
        else:  # a new subject's maps arrive on the host
            s["maps"] = (eps.cpu().numpy(), sig.cpu().numpy())
    torch.cuda.synchronize()
    return s


def run(s):
    case, call = s["case"], s["case"]["call"]
    stream = torch.cuda.current_stream()
    precision, op = PRECISION[case["precision"]], OPERATOR[case["op"]]
    if call in ("matvec", "pwc"):
        vie.vie_matvec(s["h"], s["x"], s["y"], precision, op, stream)
        return s["y"]
    if call == "jm":
        vie.vie_jm_matvec(s["h"], s["x"], s["y"], op, precision, stream)
        return s["y"]
    if call == "hfields":
        energy = vie.vie_hfields(s["h"], s["x"], s["h_inc"], s["out"], s["b1"], stream)
        return {"h": s["out"], "b1_plus": s["b1"], "W_m": np.array(energy)}
    h = s["h"] if call == "solve" else vie.vie_setup(_grid(case), case["freq"], *s["maps"])
    if call == "request":
        vie.vie_rhs_dipoles(h, *s["dipoles"], s["e_inc"], s["b"])
    vie.vie_solve(h, s["b"], s["x"], tol=1e-6, restart=50, maxit=30, mode=vie.VIE_SOLVE_FP32_REFINE)
    power = vie.vie_fields(h, s["x"], s["e_inc"], s["e"], s["p_abs"])
    if call == "request":
        h.close()
    # solved to a residual of 1e-6, which is a few 1e-6 in the maps: they are kept in single precision
    return {"x": s["x"].to(torch.complex64), "e": s["e"].to(torch.complex64), "p_abs": s["p_abs"].float(),
            "P_abs": np.array(power, dtype=np.float32)}


def exact(case, seed):
    """The matvec of the tensors of _toeplitz by zero-padded 64-bit FFTs; the calls whose tensors come from the
    singular integrals (or which iterate) have no such value here."""
    if case["call"] != "matvec":
        return None
    g = _generator(seed)
    R, n = case["nrhs"], (case["nz"], case["ny"], case["nx"])
    eps, sig = _materials(case, g)
    x = _vector((R, 12, *n), torch.complex128 if case["precision"] == "f64" else torch.complex64, g).to(torch.complex128)
    full = tuple(2 * k for k in n)
    spectra, entries = [], {}
    for t, ((a, b), tensor) in enumerate(_toeplitz(case)):
        circ = torch.zeros(full, device="cuda", dtype=torch.complex128)
        circ[:n[0], :n[1], :n[2]] = tensor
        for i in range(3):  # mirror axis by axis: an entry is odd along the axes that an odd number of its factors is
            axis = 2 - i
            odd = sum((c // 4 == i) + (c % 4 == i + 1) for c in (a, b)) % 2
            part = circ.narrow(axis, 1, n[axis] - 1).flip(axis)
            circ.narrow(axis, n[axis] + 1, n[axis] - 1).copy_(-part if odd else part)
        spectra.append(torch.fft.fftn(circ))
        (p, l), (q, m) = divmod(a, 4), divmod(b, 4)
        sign = -1.0 if (l > 0) != (m > 0) else 1.0
        for u, v in {(p, q), (q, p)}:
            entries[4 * u + l, 4 * v + m] = (t, 1.0)
            if l != m:
                entries[4 * u + m, 4 * v + l] = (t, sign)
    e = torch.complex(eps, -sig / (2 * math.pi * case["freq"] * 8.8541878128e-12))
    y = torch.empty_like(x)
    for r in range(R):
        hat = [torch.fft.fftn(x[r, b], s=full) for b in range(12)]
        for a in range(12):
            acc = torch.zeros(full, device="cuda", dtype=torch.complex128)
            for b in range(12):
                t, sign = entries[a, b]
                acc.addcmul_(spectra[t], hat[b], value=sign)
            v = torch.fft.ifftn(acc)[:n[0], :n[1], :n[2]]  # (N - G) x
            gram = _gram(case, a)
            y[r, a] = {"NSCAT": lambda: v, "A": lambda: gram * x[r, a] - (e - 1) * v,
                       "PA": lambda: x[r, a] / e - (e - 1) / e * v / gram}[case["op"]]()
    return y


def _product_work(case, nrhs, ncomp, ntensors, entries, size):
    """Bytes and operations of one operator: vectors and octant spectra once, pruned transforms, block products."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nv, lines = nx * ny * nz, nrhs * ncomp

    def fft(k):
        return 5 * 2 * k * math.log2(2 * k)

    transforms = 2 * lines * (ny * nz * fft(nx) + 2 * nx * nz * fft(ny) + 4 * nx * ny * fft(nz))
    return (2 * lines * nv * size + ntensors * (nx + 1) * (ny + 1) * (nz + 1) * size + 2 * nv * size,
            transforms + 8 * entries * 8 * nv * nrhs)


def work(case):
    R, call = case["nrhs"], case["call"]
    size = 16 if case["precision"] == "f64" else 8
    nv = case["nx"] * case["ny"] * case["nz"]
    if call == "pwc":
        b, f = _product_work(case, R, 3, 6, 9, size)
    elif call == "jm":  # N and K of both currents
        (b, f), (b2, f2) = _product_work(case, 2 * R, 12, 60, 144, size), _product_work(case, 2 * R, 12, 30, 96, size)
        b, f = 2 * b - b2, f + f2  # one set of vectors; K's 30 tensors are half of N's 60
    elif call == "hfields":
        b, f = _product_work(case, R, 12, 30, 96, size)
        b += R * 13 * nv * size
    else:
        b, f = _product_work(case, R, 12, 60, 144, size)
        if call in ("solve", "request"):  # about 230 operator applications at this contrast and tolerance
            b, f = 230 * b, 230 * f
    return {"bytes": float(b), "flops": float(f)}
