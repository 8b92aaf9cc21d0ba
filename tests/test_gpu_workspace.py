"""Device memory that the first prepared evaluation allocates: only what its kernels read. Lengths
with the warp-specialized kernels (512 along y) take two scaled copies of a tensor component and the
segment partials, the others the partials of the z chunks."""

import pytest
import torch

from paper_1707_09898_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
TB, SLACK = 16, 6 << 20  # columns of a tile; each allocation is rounded up to 2 MiB


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__

    __graft_entry__.build()


def growth(n):
    from paper_1707_09898_gb300 import Magnet

    m = Magnet((n, n, n), n, (1e-3,) * 3, M0=(0.0, 0.0, W.MS), p=3.0, device=0)
    mask = torch.zeros((n, n, n), dtype=torch.uint8, device=DEV)
    mask[n - 1, 2:-2, 2:-2] = 1
    m.set_target(mask, Ht_const=(0.0, 0.0, 0.1 * W.MS))
    rho, G = torch.full((n, n, n), 0.5, device=DEV), torch.empty((n, n, n), device=DEV)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info(DEV)[0]
    m.evaluate(rho, G=G)
    return before - torch.cuda.mem_get_info(DEV)[0]


@pytest.mark.parametrize("n", [128, 256])
def test_first_evaluation_allocates_what_it_reads(n):
    growth(n)  # the modules of the kernels are loaded at their first launch
    L = 2 * n
    P = (L // 2 + 1 + TB - 1) // TB * TB
    nsm = torch.cuda.get_device_properties(DEV).multi_processor_count
    if L == 512:
        most = 2 * 4 * n * (L // 2 + 1) * P + 2 * nsm * L * TB * 8
    else:
        most = min(n, max(1, nsm // (P // TB))) * L * P * 8
    assert growth(n) <= most + SLACK
