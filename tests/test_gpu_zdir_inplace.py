"""The direct z sums with target planes inside the design, where the adjoint reads its source
planes and writes its outputs in the same slots: every warp of a block reads the source planes,
and one of them owns the range of z that overwrites them. Repeated evaluations give the same
bits, and the values agree with the float64 oracle.

The target lies on the first plane of a warp's share of the design (the plane that is
overwritten first), on the design's only planes, and on more planes than the design has (the
forward sum is then the one with few inputs). Tolerances as in test_gpu_zpass.py."""

import functools

import numpy as np
import pytest
import torch

from oracle import convolution as C
from oracle import objective as O
from paper_1707_09898_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
REPEATS = 24
ALONG_Z = np.array([0.0, 0.0, W.MS])
TILTED = np.array([0.48, -0.6, 0.64]) * W.MS


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__

    __graft_entry__.build()


@functools.lru_cache(maxsize=1)
def operator(n, nzd):
    return C.FFTOperator(C.Geometry(n, nzd, (1e-3,) * 3))


def up(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


GRIDS = [((60, 44, 40), 40, 10),  # a share of 5 planes: the target starts a share
         ((60, 44, 40), 33, 25),
         ((44, 60, 12), 7, 0)]    # at most one plane to a warp


@pytest.mark.parametrize("n,nzd,z0", GRIDS)
@pytest.mark.parametrize("planes", [1, 2, 4, 8])
def test_target_inside_design(n, nzd, z0, planes):
    from paper_1707_09898_gb300 import Magnet

    nx, ny, nz = n
    op = operator(n, nzd)
    rng = np.random.default_rng(100 * nzd + planes)
    rho = rng.random((nzd, ny, nx)).astype(np.float32)
    M0v = (W.MS * rng.normal(size=(3, nzd, ny, nx))).astype(np.float32)
    Ht = (0.05 * W.MS * rng.normal(size=(3, nz, ny, nx))).astype(np.float32)
    mask = np.zeros((nz, ny, nx), np.uint8)
    mask[z0:z0 + planes, 1:ny - 1, 2:nx - 1] = 1
    m = Magnet(n, nzd, (1e-3,) * 3, M0=tuple(TILTED), p=3.0, device=0)
    m.set_fused(False)
    rhod = up(rho)
    for M0 in (ALONG_Z, TILTED, M0v):
        m.set_M0(up(M0) if M0.ndim == 4 else tuple(M0))
        for w in ((0.0, 0.0, 1.0), (1.0, 0.5, 2.0)):
            m.set_target(up(mask), Ht=up(Ht), w=w)
            J0, G = m.evaluate(rhod)
            G0 = G.clone()
            Jr, Gr, _ = O.objective_and_gradient(op, rho, M0, 3.0, mask, Ht, w)
            assert abs(J0 - Jr) <= 1e-5 * abs(Jr)
            g = G0.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(g - Gr) <= 1e-5 * np.linalg.norm(Gr)
            for _ in range(REPEATS):
                J, G = m.evaluate(rhod)
                assert J == J0 and torch.equal(G, G0)
