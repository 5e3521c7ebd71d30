"""Device memory of a handle: what vie_info counts, what the device gives, and what the server reserves for it."""

import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vie():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_02196_gb300 as v

    v.build()
    return v


def pow2(n):
    return 1 << max(n - 1, 1).bit_length()


# the fused z passes; FFT lengths along z of 4 and 1024, which take the generic one
@pytest.mark.parametrize("shape", [(40, 36, 33), (20, 24, 2), (4, 3, 300)])
def test_handle_memory(vie, shape):
    nx, ny, nz = shape
    nv, octant = nx * ny * nz, int(np.prod([pow2(2 * n - 1) // 2 + 1 for n in shape]))
    eps = np.full((nz, ny, nx), 3.0)
    grid = (nx, ny, nz, 0.004, 0.005, 0.0045)
    vie.vie_setup(grid, 298e6, eps, 0 * eps).close()  # what the first call loads
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    h = vie.vie_setup(grid, 298e6, eps, 0 * eps)
    held, used = vie.vie_info(h)[1], free0 - torch.cuda.mem_get_info()[0]
    # 48 bytes per octant value of the 60 tensors, the table, seven material arrays, twiddles and maps
    most = 60 * octant * 48 + 60 * nv * 16 + nv * 88 + (1 << 20)
    assert held <= most
    assert used <= held + 20 * (2 << 20)  # allocations come in blocks of 2 MiB
    x = torch.randn((1, 12, nz, ny, nx), dtype=torch.complex128, device="cuda")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    vie.vie_matvec(h, x, y, vie.VIE_FP64, vie.VIE_OP_NSCAT)
    before = vie.vie_info(h)[1]
    vie.vie_matvec(h, x, y, vie.VIE_FP64, vie.VIE_OP_K)
    torch.cuda.synchronize()
    assert vie.vie_info(h)[1] - before <= 30 * octant * 40
    h.close()


def test_server_reserves_what_a_handle_holds(vie):
    """The device bytes that a request needs, read from the refusal of a budget of one byte, cover the Green part of a
    handle (its working set comes on top)."""
    n = 48
    eps = np.full((n, n, n), 3.0)
    sig = 0 * eps
    h = vie.vie_setup((n, n, n, 0.004, 0.004, 0.004), 298e6, eps, sig)
    held = vie.vie_info(h)[1]
    h.close()
    s = vie.Server(hbm_budget_bytes=1, max_concurrent=1)
    with pytest.raises(vie.VieError) as e:
        s.submit((n, n, n, 0.004, 0.004, 0.004), 298e6, eps, sig, np.array([[0.3, 0.0, 0.0]]), np.array([[0.0, 0.0, 1.0]]), restart=1)
    s.close()
    need = int(re.search(r"needs (\d+) device bytes", str(e.value)).group(1))
    # of that, the working set: solver basis and vectors, spectra, maps (a lower bound of the server's sum)
    work = 8 * 2 * 12 * n ** 3 + 16 * 12 * n ** 3 * 9 + 16 * 12 * n * (n * 128 + 128 * 128) + (64 << 20)
    assert need - work >= held
