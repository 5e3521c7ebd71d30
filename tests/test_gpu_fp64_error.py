"""Error of the FP64 products against direct sums in twice the precision, for the constant and the linear
components apart, on inputs whose spectra are flat, peaked, or far larger in some places than in others.

Tolerance per class of components (2-norm over the sampled voxels, relative to the class's norm): 1.2e-15.  Three
transforms each way of at most 9 stages round about 2 * 27 times by 2^-53 / 2 of the values at hand, at random: 4e-16 of
the norm where input, tensors and result have it in the same places, and three times that for linear components,
which are results of cancellation on smooth inputs.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 1.2e-15


@pytest.fixture(scope="module")
def vie():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_02196_gb300 as v

    v.build()
    return v


def parity(a, i):
    return (-1 if a // 4 == i else 1) * (-1 if a % 4 == i + 1 else 1)


def entry_n(a, b):
    """(pair p <= q, pair l <= l', sign) of the tensor of entry (a, b) of N."""
    (p, l), (q, m) = divmod(a, 4), divmod(b, 4)
    sign = -1.0 if l > m and (l > 0) != (m > 0) else 1.0
    return (min(p, q), max(p, q)), (min(l, m), max(l, m)), sign


def far_table(shape):
    """Tensors of the right parities that a smooth function of the distance and its derivatives make: the linear
    functions couple through differences, so they are weak where the spectrum is large."""
    nx, ny, nz = shape
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    d = [v.astype(float) for v in (x, y, z)]
    rho = np.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2 + 0.4)
    tensors = {}
    for p in range(3):
        for q in range(p, 3):
            for l in range(4):
                for m in range(l, 4):
                    t = np.exp(-0.05j * rho) / rho * 12.0 ** -((l > 0) + (m > 0))
                    for i in range(3):
                        if parity(4 * p + l, i) * parity(4 * q + m, i) < 0:
                            t = t * d[i] / rho ** 2
                    tensors[(p, q), (l, m)] = t
    return tensors


def handle_of(vie, shape, tensors):
    nx, ny, nz = shape
    table = np.zeros((144, 2 * nz - 1, 2 * ny - 1, 2 * nx - 1), dtype=np.complex128)
    for (p, q), (l, m) in tensors:
        table[12 * (4 * p + l) + 4 * q + m, nz - 1:, ny - 1:, nx - 1:] = tensors[(p, q), (l, m)]
    eps = np.full((nz, ny, nx), 3.0)
    # a Gram entry so small that taking it off changes no tensor
    return vie.vie_setup_green_external((nx, ny, nz, 1e-9, 1e-9, 1e-9), 3e6, eps, 0 * eps, table)


def field(kind, nc, shape, seed=4):
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    v = rng.standard_normal((nc, nz, ny, nx)) + 1j * rng.standard_normal((nc, nz, ny, nx))
    if kind == "mean":
        v = (1 + 0.5j) + 0.01 * v
    if kind == "decay":
        v = v * np.exp(-0.35 * (x + y + z))
    if kind == "peak":  # one value a million times the others
        v *= 1e-6
        v[nc // 2, nz // 2, ny // 2, nx // 3] = 1 - 2j
    if kind == "wave":  # a wave that fades towards the sides, the linear functions a small part of it
        w = np.exp(-0.1j * (0.6 * x + 0.5 * y + 0.62 * z))
        w = w * np.exp(-((x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2) / (0.3 * max(shape)) ** 2)
        weak = np.where(np.arange(nc) % 4 == 0, 1.0, 0.03) if nc == 12 else np.ones(nc)
        v = weak[:, None, None, None] * w * (1 + 0.001 * v)
    return v


def split(a):  # two halves of 26 bits, whose products are exact
    c = 134217729.0 * a
    hi = c - (c - a)
    return hi, a - hi


def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def exact_sum(terms):
    """Sum of a row, and the rounding errors of the pairwise sum added up."""
    err = torch.zeros(terms.shape[0], dtype=torch.float64, device=terms.device)
    while terms.shape[1] > 1:
        if terms.shape[1] % 2:
            terms = torch.nn.functional.pad(terms, (0, 1))
        terms, e = two_sum(terms[:, 0::2].contiguous(), terms[:, 1::2].contiguous())
        err += e.sum(1)
    return terms[0, 0], err[0]


def products(u, v):
    (uh, ul), (vh, vl) = split(u), split(v)
    return torch.stack([uh * vh, uh * vl, ul * vh, ul * vl], 1).flatten(1)


def direct(tensor_of, x, voxel):
    """((re, its error), (im, its error)) of the nc outputs at a voxel; tensor_of(a, b): (tensor at offsets >= 0, sign,
    parities per axis) or None."""
    nc, nz, ny, nx = x.shape
    off = [voxel[2] - torch.arange(nx, device="cuda"), voxel[1] - torch.arange(ny, device="cuda"),
           voxel[0] - torch.arange(nz, device="cuda")]
    idx = [o.abs() for o in off]
    re, im = [], []
    for a in range(nc):
        tr = []
        for b in range(nc):
            entry = tensor_of(a, b)
            if entry is None:
                tr.append(torch.zeros_like(x[0]))
                continue
            t, sign, par = entry
            v = t[idx[2]][:, idx[1]][:, :, idx[0]] * sign
            for i, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
                if par[i] < 0:
                    v = v * torch.where(off[i] < 0, -1.0, 1.0).reshape(shape)
            tr.append(v)
        t = torch.stack(tr).reshape(1, -1)
        f = x.reshape(1, -1)
        re.append(exact_sum(torch.cat([products(t.real, f.real), products(-t.imag, f.imag)], 1)))
        im.append(exact_sum(torch.cat([products(t.real, f.imag), products(t.imag, f.real)], 1)))
    return re, im


def errors(y, x, tensor_of, nvox, seed=1):
    """Relative error of the constant components and, with twelve components, of the linear ones."""
    nc, nz, ny, nx = x.shape
    rng = np.random.default_rng(seed)
    sums = torch.zeros(nc, dtype=torch.float64, device="cuda")
    for _ in range(nvox):
        v = [int(rng.integers(n)) for n in (nz, ny, nx)]
        re, im = direct(tensor_of, x, v)
        for a in range(nc):
            got = y[a, v[0], v[1], v[2]]
            sums[a] += ((got.real - re[a][0]) - re[a][1]) ** 2 + ((got.imag - im[a][0]) - im[a][1]) ** 2
    classes = [[a for a in range(nc) if nc == 3 or a % 4 == 0]] + ([[a for a in range(12) if a % 4]] if nc == 12 else [])
    return [(sums[c].sum() * (nx * ny * nz / nvox)).sqrt().item() / torch.linalg.vector_norm(y[c]).item() for c in classes]


def matvec(vie, h, x, op="NSCAT"):
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    vie.vie_matvec(h, x[None].contiguous(), y[None], vie.VIE_FP64, getattr(vie, "VIE_OP_" + op))
    torch.cuda.synchronize()
    return y


def check_n(vie, shape, kinds, nvox=12):
    tensors = far_table(shape)
    h = handle_of(vie, shape, tensors)
    dev = {k: torch.from_numpy(t).cuda() for k, t in tensors.items()}

    def tensor_of(a, b):
        pq, lm, sign = entry_n(a, b)
        return dev[pq, lm], sign, [parity(a, i) * parity(b, i) for i in range(3)]

    for kind in kinds:
        x = torch.from_numpy(field(kind, 12, shape)).cuda()
        for e, name in zip(errors(matvec(vie, h, x), x, tensor_of, nvox), ("constant", "linear")):
            assert e <= TOL, (kind, name, e)
    h.close()


# FFT lengths along z 8 to 512, on the line transforms and on the small plane ones
@pytest.mark.parametrize("shape", [(6, 9, 4), (5, 6, 8), (4, 7, 13), (5, 5, 30), (6, 11, 60), (12, 16, 100), (8, 7, 200)])
def test_z_transforms_and_product(vie, shape):
    check_n(vie, shape, ["random", "mean", "wave", "decay"])


# the square xy kernels at every length (8 to 128), even and odd sides, at a short z
@pytest.mark.parametrize("shape", [(4, 3, 4), (7, 8, 5), (16, 13, 4), (32, 29, 6), (64, 61, 3), (64, 64, 3), (33, 60, 4)])
@pytest.mark.parametrize("kind", ["random", "mean", "decay", "peak", "wave"])
def test_plane_transforms(vie, shape, kind):
    """A table that is the identity leaves the transforms' error alone: relative 2-norm at most 2^-52.  The two spectra in
    memory and the result are FP64 numbers (2^-53 / sqrt(6) of their norm each, 8e-17 together), and the six
    passes round at 2^-56 of a line's largest value, at most some eight times its root mean square (2^-53 each)."""
    nx, ny, nz = shape
    one = np.zeros((nz, ny, nx), dtype=np.complex128)
    one[0, 0, 0] = 1.0
    h = handle_of(vie, shape, {((p, p), (l, l)): one for p in range(3) for l in range(4)})
    # the same field in every component: the product's scale is common to them
    x = torch.from_numpy(np.tile(field(kind, 3, shape)[1:2], (12, 1, 1, 1))).cuda()
    y = matvec(vie, h, x)
    h.close()
    for a in range(12):
        e = (torch.linalg.vector_norm(y[a] - x[a]) / torch.linalg.vector_norm(x[a])).item()
        assert e <= 2.0 ** -52, (a, e)


# FFT lengths along z 8 to 512
@pytest.mark.parametrize("shape", [(6, 9, 4), (4, 7, 8), (5, 5, 13), (6, 11, 30), (9, 9, 60), (20, 13, 70), (5, 6, 240)])
@pytest.mark.parametrize("kind", ["random", "mean", "decay", "wave"])
def test_pwc(vie, shape, kind):
    """The 3 x 3 block's z pass against the 12 x 12 one, whose constant components have the same tensors and the same
    transforms along x and y: within 4e-16 of each other.  The 3 x 3 product has nine FP64 multiply-adds a value
    (1.1e-16) and its spectrum is rounded to FP64 before and after it, as both results are (4.5e-17 each): 1.5e-16
    together, with a margin for what the integers of the two add."""
    nx, ny, nz = shape
    eps = np.full((nz, ny, nx), 3.0)
    grid = (nx, ny, nz, 0.004, 0.005, 0.0045)
    h3 = vie.vie_setup(grid, 298e6, eps, 0 * eps, vie.VIE_SETUP_PWC)
    h12 = vie.vie_setup(grid, 298e6, eps, 0 * eps)
    x = torch.from_numpy(field(kind, 3, shape)).cuda()
    x12 = torch.zeros((12, nz, ny, nx), dtype=torch.complex128, device="cuda")
    x12[0::4] = x
    y, want = matvec(vie, h3, x), matvec(vie, h12, x12)[0::4]
    h3.close()
    h12.close()
    e = (torch.linalg.vector_norm(y - want) / torch.linalg.vector_norm(want)).item()
    assert e <= 4e-16, e


# the square xy kernels, the line ones, and an FFT length along z of 512
@pytest.mark.parametrize("shape", [(4, 4, 4), (9, 20, 5), (4, 3, 140)])
@pytest.mark.parametrize("kind", ["N", "PWC"])
def test_subnormal_results(vie, shape, kind):
    """Inputs so small that the results are subnormal numbers give those of ordinary ones times the power of two, within
    the spacing of the subnormal numbers, 2^-1074, for each of the values of a plane that are summed (a quarter of
    its points, half a spacing each)."""
    nx, ny, nz = shape
    eps = np.full((nz, ny, nx), 3.0)
    h = vie.vie_setup((nx, ny, nz, 0.5, 0.4, 0.45), 3e6, eps, 0 * eps, vie.VIE_SETUP_PWC if kind == "PWC" else 0)
    x = torch.from_numpy(field("random", 3 if kind == "PWC" else 12, shape)).cuda()
    want = matvec(vie, h, x)
    top = want.abs().max().item()
    scale = 2.0 ** -(1030 + int(np.ceil(np.log2(top))))  # the largest result 2^-1030
    got = matvec(vie, h, x * scale)
    h.close()
    planes = 4 * nx * ny * 4  # points of a plane at most
    err = torch.linalg.vector_norm((torch.view_as_real(got) - torch.view_as_real(want) * scale).reshape(-1) * 2.0 ** 1000,
                                   ord=float("inf")).item() * 2.0 ** -1000
    assert err <= planes / 8 * 2.0 ** -1074, err / 2.0 ** -1074


# the square xy kernels and the line ones, FFT lengths along z of 16, 64 and 512
@pytest.mark.parametrize("shape", [(5, 6, 7), (3, 7, 20), (4, 3, 130)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_not_finite_table(vie, shape, value):
    """A NaN or an Inf in one tensor makes the outputs that it couples to any input not finite, for every input, zero
    among them, and leaves the others as the table without it gives them (to 1e-14)."""
    nx, ny, nz = shape
    clean = far_table(shape)
    for (p, q), (l, m) in [((0, 0), (0, 0)), ((0, 2), (0, 1)), ((1, 1), (2, 3))]:
        bad = {k: t.copy() for k, t in clean.items()}
        bad[(p, q), (l, m)][1, 2, 1] = value
        reached = {4 * u + v for u in (p, q) for v in (l, m)}
        x = torch.from_numpy(field("random", 12, shape)).cuda()
        h = handle_of(vie, shape, clean)
        want = matvec(vie, h, x)
        h.close()
        h = handle_of(vie, shape, bad)
        for v in (x, 0 * x, 1e-300 * x):
            y = matvec(vie, h, v)
            for a in range(12):
                if a in reached:
                    assert not torch.isfinite(torch.view_as_real(y[a])).all(-1).any(), (a, v[0, 0, 0, 0])
                else:
                    assert torch.isfinite(torch.view_as_real(y[a])).all()
            if v is x:
                for a in set(range(12)) - reached:
                    assert torch.linalg.vector_norm(y[a] - want[a]) <= 1e-14 * torch.linalg.vector_norm(want[a])
        h.close()


# the square xy kernels and the line ones, FFT lengths along z of 16, 64 and 512
@pytest.mark.parametrize("shape", [(5, 6, 7), (3, 7, 20), (4, 3, 130)])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_k_not_finite(vie, shape, value):
    """K does not couple a direction's components to themselves: a NaN or an Inf leaves them as they were (to 1e-13, a
    hundred times the error of the product) and no finite value in the other two directions'; the other right-hand
    side stays as it is."""
    nx, ny, nz = shape
    eps = np.full((nz, ny, nx), 3.0)
    h = vie.vie_setup((nx, ny, nz, 0.01, 0.012, 0.011), 298e6, eps, 0 * eps)
    x = torch.from_numpy(np.stack([field("random", 12, shape, seed) for seed in (4, 5)])).cuda()

    def apply(v):
        y = torch.empty_like(v)
        torch.cuda.synchronize()
        vie.vie_matvec(h, v, y, vie.VIE_FP64, vie.VIE_OP_K)
        torch.cuda.synchronize()
        return y

    want = apply(x)
    for comp in (1, 4, 11):
        v = x.clone()
        v[0, comp, nz // 2, 1, 1] = value
        y = apply(v)
        own = list(range(4 * (comp // 4), 4 * (comp // 4) + 4))
        other = [a for a in range(12) if a not in own]
        assert torch.linalg.vector_norm(y[0, own] - want[0, own]) <= 1e-13 * torch.linalg.vector_norm(want[0, own])
        assert not torch.isfinite(torch.view_as_real(y[0, other])).all(-1).any()
        assert torch.equal(y[1], want[1])
    h.close()


# FFT lengths along z of 128 and 512 (two right-hand sides to a group, and one), on the line and on the plane transforms
@pytest.mark.parametrize("shape", [(5, 9, 40), (9, 12, 50), (4, 7, 140)])
@pytest.mark.parametrize("op", ["NSCAT", "K"])
def test_groups_of_right_hand_sides(vie, shape, op):
    """Five right-hand sides of very different sizes: each has the bits that it has alone, and the K product's error
    against direct sums is below 1e-12 (its linear entries are small differences of large integrals, good to 1e-14)."""
    nx, ny, nz = shape
    eps = np.full((nz, ny, nx), 3.0)
    h = vie.vie_setup((nx, ny, nz, 0.004, 0.005, 0.0045), 298e6, eps, 0 * eps)
    sizes = [1.0, 1e-200, 1e100, 1e-9, 0.0]
    x = torch.from_numpy(np.stack([s * field("random", 12, shape, seed) for seed, s in enumerate(sizes)])).cuda()

    def apply(v):
        y = torch.empty_like(v)
        torch.cuda.synchronize()
        vie.vie_matvec(h, v, y, vie.VIE_FP64, getattr(vie, "VIE_OP_" + op))
        torch.cuda.synchronize()
        return y

    y = apply(x)
    for r in range(5):
        assert torch.equal(apply(x[r:r + 1].contiguous())[0], y[r]), r
    if op == "K":
        tensors = torch.zeros((30, nz, ny, nx), dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        vie.vie_green_toeplitz_k(h, tensors)
        torch.cuda.synchronize()

        def tensor_of(a, b):
            (p, l), (q, m) = divmod(a, 4), divmod(b, 4)
            if p == q:
                return None
            j = 3 - p - q
            lo, hi = min(l, m), max(l, m)
            pair = {0: hi, 1: 3 + hi, 2: 5 + hi, 3: 9}[lo]
            sign = (-1.0 if (j - p) % 3 == 1 else 1.0) * (-1.0 if l > m and (l > 0) != (m > 0) else 1.0)
            return tensors[10 * j + pair], sign, [-parity(a, i) * parity(b, i) for i in range(3)]

        for e in errors(y[0], x[0], tensor_of, 8):
            assert e <= 1e-12, e
    h.close()
