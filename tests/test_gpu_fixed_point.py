"""The FP64 matvec's scaled-integer transforms and split block product at every compiled FFT length, on inputs of
very different sizes, against NumPy's FP64 FFTs with a random Toeplitz table of the right parities.

Tolerance per right-hand side (relative 2-norm): 5e-15.  NumPy's three transforms each way and the 24-term sums
are good for about 1e-15 at these lengths; the kernels round at 2^-56 of the largest value, with the spectrum
stored in FP64 twice.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 5e-15


@pytest.fixture(scope="module")
def vie():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_02196_gb300 as v

    v.build()
    return v


def parity(a, i):
    return (-1 if a // 4 == i else 1) * (-1 if a % 4 == i + 1 else 1)


def make(vie, shape, seed):
    """(handle on random tensors, the 144 circulant spectra by entry and sign) of an nx x ny x nz grid."""
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    table = np.zeros((144, 2 * nz - 1, 2 * ny - 1, 2 * nx - 1), dtype=np.complex128)
    spectra = {}
    dec = 1.0 / (1 + np.add.outer(np.add.outer(np.arange(nz), np.arange(ny)), np.arange(nx)))  # decays as the entries do
    for p in range(3):
        for q in range(p, 3):
            for l in range(4):
                for m in range(l, 4):
                    a, b = 4 * p + l, 4 * q + m
                    size = 12.0 ** (-0.5 * ((l > 0) + (m > 0)))  # of the Gram entries' square roots
                    t = size * dec * (rng.standard_normal((nz, ny, nx)) + 1j * rng.standard_normal((nz, ny, nx)))
                    circ = np.zeros((2 * nz, 2 * ny, 2 * nx), dtype=np.complex128)
                    for axis, i in ((2, 0), (1, 1), (0, 2)):  # an odd tensor vanishes at offset 0 of its axis
                        if parity(a, i) * parity(b, i) < 0:
                            t[(slice(None),) * axis + (0,)] = 0
                    circ[:nz, :ny, :nx] = t
                    for axis, i, n in ((2, 0, nx), (1, 1, ny), (0, 2, nz)):
                        s = parity(a, i) * parity(b, i)
                        src = np.moveaxis(circ, axis, 0)
                        for d in range(1, n):
                            src[2 * n - d] = s * src[d]
                    table[12 * a + b, nz - 1:, ny - 1:, nx - 1:] = t
                    if a == b:  # the library keeps N - G
                        table[12 * a + b, nz - 1, ny - 1, nx - 1] += 1.0 if l == 0 else 1 / 12
                    hat = np.fft.fftn(circ)
                    swap = -1.0 if (l > 0) != (m > 0) else 1.0
                    for u, v in {(p, q), (q, p)}:
                        spectra[4 * u + l, 4 * v + m] = (hat, 1.0)
                        if l != m:
                            spectra[4 * u + m, 4 * v + l] = (hat, swap)
    eps = np.full((nz, ny, nx), 3.0)
    h = vie.vie_setup_green_external((nx, ny, nz, 1.0, 1.0, 1.0), 3e6, eps, 0 * eps, table)
    return h, spectra


def reference(spectra, shape, x):
    nx, ny, nz = shape
    hat = [np.fft.fftn(x[b], s=(2 * nz, 2 * ny, 2 * nx), axes=(0, 1, 2)) for b in range(12)]
    out = np.empty_like(x)
    for a in range(12):
        acc = sum(spectra[a, b][1] * spectra[a, b][0] * hat[b] for b in range(12))
        out[a] = np.fft.ifftn(acc)[:nz, :ny, :nx]
    return out


def apply(vie, h, x):
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    vie.vie_matvec(h, xd, yd, vie.VIE_FP64, vie.VIE_OP_NSCAT)
    torch.cuda.synchronize()
    return yd.cpu().numpy()


# FFT lengths (x, y, z): (8, 8, 8), (16, 16, 16), (32, 32, 32), (64, 64, 64), (128, 128, 8), (8, 8, 128), (8, 8, 256),
# (8, 8, 512), and the line transforms with (8, 16, 64) and (256, 8, 16)
@pytest.mark.parametrize("shape", [(4, 3, 4), (8, 7, 5), (13, 16, 9), (20, 17, 32), (33, 40, 3), (4, 4, 40), (3, 4, 100),
                                   (4, 3, 200), (3, 7, 20), (70, 3, 5)])
def test_sizes_and_scales(vie, shape):
    nx, ny, nz = shape
    h, spectra = make(vie, shape, seed=nx + 10 * ny + 100 * nz)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((6, 12, nz, ny, nx)) + 1j * rng.standard_normal((6, 12, nz, ny, nx))
    x[1] *= 1e-295  # close to the smallest normal numbers
    x[2] = 0
    x[2, 7, nz // 2, ny - 1, 0] = 3e200 - 1e200j  # one large value
    x[3] *= 1e-9 ** rng.random((12, 1, 1, 1))  # components of different sizes
    x[4, :, :, :, 1:] *= 1e-12  # one column above the rest
    x[5] = x[5].astype(np.complex64)  # short mantissas: low words of the fixed-point values at their ends
    y = apply(vie, h, x)
    for r in range(6):
        s = 10.0 ** -np.round(np.log10(np.max(np.abs(x[r]))))  # the reference at ordinary sizes
        ref = reference(spectra, shape, x[r] * s)
        err = np.linalg.norm(y[r] * s - ref) / np.linalg.norm(ref)
        assert err <= TOL, (r, err)
    # a right-hand side does not depend on its neighbours, of any size
    assert np.array_equal(apply(vie, h, x[3:4])[0], y[3])
    h.close()


# line transforms of every length (x, y): 32 x 64, 64 x 32, 128 x 256, 512 x 16, 16 x 512; a last CTA with lines to spare
@pytest.mark.parametrize("shape", [(9, 20, 3), (32, 11, 2), (50, 128, 1), (200, 5, 3), (6, 256, 2)])
def test_line_lengths(vie, shape):
    test_sizes_and_scales(vie, shape)


@pytest.mark.parametrize("shape", [(5, 6, 7), (3, 7, 20)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_not_finite(vie, shape, value):
    """A NaN or an Inf leaves no finite value in its right-hand side, as every output depends on every input, and
    the others as they are; zero stays zero."""
    nx, ny, nz = shape
    h, _ = make(vie, shape, seed=3)
    rng = np.random.default_rng(6)
    x = rng.standard_normal((3, 12, nz, ny, nx)) + 1j * rng.standard_normal((3, 12, nz, ny, nx))
    x[1] = 0
    clean = apply(vie, h, x)
    assert np.all(clean[1] == 0)
    x[0, 4, 1, 2, 1] = value
    y = apply(vie, h, x)
    assert not np.any(np.isfinite(y[0]))
    assert np.array_equal(y[1:], clean[1:])
    h.close()


# FFT lengths (x, y, z) of the PWC z pass: tiles of 8 columns up to 256 points, of 4 at 512, and Lx = 8 with one tile
@pytest.mark.parametrize("shape", [(4, 4, 4), (8, 7, 7), (5, 5, 13), (9, 16, 31), (33, 35, 50), (4, 3, 70), (7, 2, 150)])
def test_pwc_sizes_and_scales(vie, shape):
    """The 3 x 3 block's z pass against the constant components of the 12 x 12 one on the same grid and materials, on
    the same inputs (5e-15: both are within about 1e-15 of the exact product), and FP32 against FP64 (2e-6, some
    tens of FP32 roundings)."""
    nx, ny, nz = shape
    rng = np.random.default_rng(11)
    grid = (nx, ny, nz, 0.004, 0.005, 0.0045)
    eps = rng.uniform(1, 80, (nz, ny, nx))
    h12 = vie.vie_setup(grid, 298e6, eps, 0 * eps)
    h3 = vie.vie_setup(grid, 298e6, eps, 0 * eps, vie.VIE_SETUP_PWC)
    x3 = rng.standard_normal((4, 3, nz, ny, nx)) + 1j * rng.standard_normal((4, 3, nz, ny, nx))
    x3[1] *= 1e-280
    x3[2, :, nz // 2:] *= 1e-10
    x3[3] = 0
    x12 = np.zeros((4, 12, nz, ny, nx), dtype=np.complex128)
    x12[:, [0, 4, 8]] = x3
    want = apply(vie, h12, x12)[:, [0, 4, 8]]
    got = apply(vie, h3, x3)
    assert np.all(got[3] == 0)
    for r in range(3):
        s = 10.0 ** -np.round(np.log10(np.max(np.abs(x3[r]))))
        assert np.linalg.norm((got[r] - want[r]) * s) <= TOL * np.linalg.norm(want[r] * s), r
    xd = torch.from_numpy(x3[[0, 2]]).to("cuda", torch.complex64)
    yd = torch.empty_like(xd)
    vie.vie_matvec(h3, xd, yd, vie.VIE_FP32, vie.VIE_OP_NSCAT)
    torch.cuda.synchronize()
    assert np.linalg.norm(yd.cpu().numpy() - want[[0, 2]]) <= 2e-6 * np.linalg.norm(want[[0, 2]])
    x3[0, 1, 0, 0, 0] = np.nan
    bad = apply(vie, h3, x3)
    assert not np.any(np.isfinite(bad[0])) and np.array_equal(bad[1:], got[1:])
    h12.close()
    h3.close()


# FFT lengths along z 8, 16, 32, 64 and 64: the FP32 z pass deals the right-hand sides of small spectra to several
# CTAs and an item's points to idle threads
@pytest.mark.parametrize("shape", [(4, 4, 4), (5, 4, 8), (10, 9, 12), (16, 13, 20), (6, 30, 32)])
@pytest.mark.parametrize("op", ["NSCAT", "K"])
def test_fp32_small_spectra(vie, shape, op):
    """Each of 9 right-hand sides bitwise as alone, and within 2e-6 (some tens of FP32 roundings) of FP64."""
    nx, ny, nz = shape
    h = vie.vie_setup((nx, ny, nz, 0.01, 0.01, 0.01), 3e8, np.full((nz, ny, nx), 4.0), np.zeros((nz, ny, nx)))
    rng = np.random.default_rng(8)
    x = torch.from_numpy(rng.standard_normal((9, 12, nz, ny, nx)) + 1j * rng.standard_normal((9, 12, nz, ny, nx))).cuda()
    x = x.to(torch.complex64).to(torch.complex128)
    torch.cuda.synchronize()
    opc = getattr(vie, "VIE_OP_" + op)
    y64 = torch.empty_like(x)
    vie.vie_matvec(h, x, y64, vie.VIE_FP64, opc)
    x32 = x.to(torch.complex64)
    torch.cuda.synchronize()
    y32 = torch.empty_like(x32)
    vie.vie_matvec(h, x32, y32, vie.VIE_FP32, opc)
    for r in range(9):
        alone = torch.empty_like(x32[:1])
        vie.vie_matvec(h, x32[r:r + 1], alone, vie.VIE_FP32, opc)
        torch.cuda.synchronize()  # the calls return before the device is done
        assert torch.equal(alone[0], y32[r])
        assert torch.linalg.vector_norm(y32[r] - y64[r]) <= 2e-6 * torch.linalg.vector_norm(y64[r])
    h.close()


@pytest.mark.parametrize("restart", [1, 2, 31, 33, 128])
def test_restart_lengths(vie, restart):
    """The triangular solve and the rotations at their smallest and largest sizes, and around a warp's: the residual
    of the returned x, formed here with the FP64 operator, is the one asked for (1e-10, with 1 % for its own rounding)."""
    n = 6
    rng = np.random.default_rng(9)
    h = vie.vie_setup((n, n, n, 0.01, 0.01, 0.01), 3e8, 1.0 + rng.random((n, n, n)), np.zeros((n, n, n)))
    b = torch.from_numpy(rng.standard_normal((3, 12, n, n, n)) + 1j * rng.standard_normal((3, 12, n, n, n))).cuda()
    x = torch.zeros_like(b)
    rc, info = vie.vie_solve(h, b, x, tol=1e-10, restart=restart, maxit=400, mode=vie.VIE_SOLVE_FP64, true_resid=True)
    assert rc == vie.VIE_OK, info
    ax = torch.empty_like(b)
    vie.vie_matvec(h, x, ax, vie.VIE_FP64, vie.VIE_OP_A)
    torch.cuda.synchronize()
    for r in range(3):
        true = (torch.linalg.vector_norm(b[r] - ax[r]) / torch.linalg.vector_norm(b[r])).item()
        assert info[r]["resid"] <= 1e-10
        assert abs(true - info[r]["true_resid"]) <= 0.01 * true
    h.close()
