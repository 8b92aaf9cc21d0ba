"""The z passes at the edges of their plans, against the float64 oracle: every supported z
length with full and odd grids, with the input and output counts of a constant and of a
varying magnetization, and the direct z sums on one to eight planes.

Tolerance: float32 transforms of N points carry a relative L2 error of about 0.6 log2(N)
roundings of 6e-8 each way, below 1e-6 for the lengths here; tensor and products add a few
roundings. 3e-6 for the field; 3e-6 for the gradient with a random cotangent, whose field
sums without cancellation in L2. J is compared with the sum of its terms at 1e-5.
"""

import numpy as np
import pytest
import torch

from oracle import convolution as C
from oracle import objective as O
from paper_1707_09898_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
TILTED = np.array([0.48, -0.6, 0.64]) * W.MS


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__

    __graft_entry__.build()


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def case(nx, ny, nz, nzd, seed):
    rng = np.random.default_rng(seed)
    rho = rng.random((nzd, ny, nx)).astype(np.float32)
    gH = rng.normal(size=(3, nz, ny, nx)).astype(np.float32)
    M0v = (W.MS * rng.normal(size=(3, nzd, ny, nx))).astype(np.float32)
    return rho, gH, M0v


def up(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("Lz,nz", [(8, 4), (12, 6), (16, 7), (18, 9), (24, 12), (32, 16), (36, 17), (48, 24), (64, 32),
                                   (72, 35), (96, 48), (128, 63), (144, 72), (192, 96), (256, 127), (256, 30), (288, 144),
                                   (384, 190), (512, 256), (512, 40), (576, 288)])
def test_every_length(Lz, nz):
    from paper_1707_09898_gb300 import Magnet

    nx, ny = 9, 6
    nzd = max(1, nz - nz // 5)
    rho, gH, M0v = case(nx, ny, nz, nzd, Lz)
    d = (1e-3, 0.9e-3, 1.2e-3)
    op = C.FFTOperator(C.Geometry((nx, ny, nz), nzd, d))
    m = Magnet((nx, ny, nz), nzd, d, M0=tuple(TILTED), p=3.0, device=0, fft_lengths=(0, 0, Lz))
    assert m.fft_lengths()[2] == Lz
    for M0 in (TILTED, M0v):
        m.set_M0(up(M0) if M0.ndim == 4 else tuple(M0))
        Hr = op.forward(O.magnetization(rho, M0, 3.0))
        assert rel(m.stray_field(up(rho)).cpu().numpy(), Hr) <= 3e-6   # one to three, three to three
        Gr = O.chain_rule(rho, M0, 3.0, op.adjoint(gH))
        assert rel(m.stray_field_adjoint(up(rho), up(gH)).cpu().numpy(), Gr) <= 3e-6  # three to one, three to three
    # a target on the whole grid in two components: two inputs to one output in the adjoint
    m.set_M0(tuple(TILTED))
    mask = np.ones((nz, ny, nx), np.uint8)
    Ht = (0.05 * W.MS * gH).astype(np.float32)
    for w in ((1.0, 0.0, 0.5), (0.0, 0.7, 0.0)):
        Jr, Gr, _ = O.objective_and_gradient(op, rho, TILTED, 3.0, mask, Ht, w)
        J, G = m.objective_and_gradient(up(rho), up(mask), Ht=up(Ht), w=w)
        assert abs(J - Jr) <= 1e-5 * abs(Jr)
        assert rel(G.cpu().numpy(), Gr) <= 1e-5


@pytest.mark.parametrize("Lz,nz,z0,z1", [(48, 24, 23, 24), (144, 72, 3, 6), (512, 256, 250, 256)])
def test_one_shot_planes(Lz, nz, z0, z1):
    """Targets on a few planes: the planes come from the device in the unprepared call."""
    from paper_1707_09898_gb300 import Magnet

    nx, ny, nzd = 9, 6, nz - 2
    rho, gH, M0v = case(nx, ny, nz, nzd, Lz + 1)
    op = C.FFTOperator(C.Geometry((nx, ny, nz), nzd, (1e-3,) * 3))
    m = Magnet((nx, ny, nz), nzd, (1e-3,) * 3, M0=tuple(TILTED), p=3.0, device=0, fft_lengths=(0, 0, Lz))
    mask = np.zeros((nz, ny, nx), np.uint8)
    mask[z0:z1, 1:5, 2:7] = 1
    Ht = (0.05 * W.MS * gH).astype(np.float32)
    for M0, w in ((TILTED, (1.0, 0.5, 2.0)), (TILTED, (0.0, 0.0, 1.0)), (M0v, (1.0, 0.5, 2.0))):
        m.set_M0(up(M0) if M0.ndim == 4 else tuple(M0))
        Jr, Gr, _ = O.objective_and_gradient(op, rho, M0, 3.0, mask, Ht, w)
        J, G = m.objective_and_gradient(up(rho), up(mask), Ht=up(Ht), w=w)
        assert abs(J - Jr) <= 1e-5 * abs(Jr)
        assert rel(G.cpu().numpy(), Gr) <= 1e-5


@pytest.mark.parametrize("n,nzd,z0,np_", [((9, 6, 13), 10, 12, 1), ((9, 6, 13), 13, 4, 2), ((30, 7, 9), 9, 0, 3),
                                          ((20, 16, 11), 8, 6, 5), ((8, 8, 40), 33, 32, 8), ((36, 5, 4), 4, 0, 4)])
def test_direct_planes(n, nzd, z0, np_):
    """Prepared targets on one to eight planes (above, inside and below the design), one and
    three components, constant and varying M0, fused with the y pass and not."""
    from paper_1707_09898_gb300 import Magnet

    nx, ny, nz = n
    rho, gH, M0v = case(nx, ny, nz, nzd, nx + np_)
    op = C.FFTOperator(C.Geometry(n, nzd, (1e-3,) * 3))
    m = Magnet(n, nzd, (1e-3,) * 3, M0=tuple(TILTED), p=3.0, device=0)
    mask = np.zeros((nz, ny, nx), np.uint8)
    mask[z0:z0 + np_, 1:ny - 1, 1:nx - 2] = 1
    Ht = (0.05 * W.MS * gH).astype(np.float32)
    for M0 in (np.array([0.0, 0.0, W.MS]), TILTED, M0v):
        m.set_M0(up(M0) if M0.ndim == 4 else tuple(M0))
        for w in ((0.0, 0.0, 1.0), (1.0, 0.0, 0.5), (1.0, 0.5, 2.0)):
            Jr, Gr, _ = O.objective_and_gradient(op, rho, M0, 3.0, mask, Ht, w)
            m.set_target(up(mask), Ht=up(Ht), w=w)
            for fused in (True, False):
                m.set_fused(fused)
                J, G = m.evaluate(up(rho))
                assert abs(J - Jr) <= 1e-5 * abs(Jr)
                assert rel(G.cpu().numpy(), Gr) <= 1e-5


@pytest.mark.parametrize("L", [8, 12, 16, 18, 24, 32, 36, 48, 64, 72, 96, 128, 144, 192, 256, 288, 384, 512, 576])
def test_single_product_every_length(L):
    """One target plane and one tensor component with a full and an odd grid at every length of
    x and y: the y transforms fused with the z sums, the plane's finish and the objective."""
    from paper_1707_09898_gb300 import Magnet

    for n, lengths in (((L // 2, 5, 5), (L, 0, 0)), ((5, L // 2, 5), (0, L, 0)), ((7, max(4, L // 2 - 3), 4), (0, L, 0))):
        nx, ny, nz = n
        rho, gH, _ = case(nx, ny, nz, nz - 1, L)
        op = C.FFTOperator(C.Geometry(n, nz - 1, (1e-3,) * 3))
        m = Magnet(n, nz - 1, (1e-3,) * 3, M0=(0.0, 0.0, W.MS), p=3.0, device=0, fft_lengths=lengths)
        mask = (gH[0] > -0.5).astype(np.uint8)
        mask[:nz - 1] = 0
        Ht = (0.05 * W.MS * gH).astype(np.float32)
        for M0, w in (((0.0, 0.0, W.MS), (0.0, 0.0, 1.0)), ((0.0, 0.0, W.MS), (0.0, 1.0, 0.0)),
                      ((W.MS, 0.0, 0.0), (0.0, 0.5, 0.0)), ((W.MS, 0.0, 0.0), (0.0, 0.0, 2.0))):
            m.set_M0(M0)
            Jr, Gr, _ = O.objective_and_gradient(op, rho, np.array(M0), 3.0, mask, Ht, w)
            m.set_target(up(mask), Ht=up(Ht), w=w)
            J, G = m.evaluate(up(rho))
            assert abs(J - Jr) <= 1e-5 * abs(Jr)
            assert rel(G.cpu().numpy(), Gr) <= 1e-5


@pytest.mark.parametrize("n,nzd", [((128, 12, 83), 82), ((144, 9, 75), 75), ((200, 24, 61), 37)])
def test_single_product_many_planes(n, nzd):
    """Many design planes on a wide grid, the target plane inside the design."""
    from paper_1707_09898_gb300 import Magnet

    nx, ny, nz = n
    rho, gH, _ = case(nx, ny, nz, nzd, nx)
    op = C.FFTOperator(C.Geometry(n, nzd, (1e-3,) * 3))
    m = Magnet(n, nzd, (1e-3,) * 3, M0=(0.0, 0.0, W.MS), p=3.0, device=0)
    mask = np.zeros((nz, ny, nx), np.uint8)
    mask[nz // 2, 1:ny - 1, 1:nx - 2] = 1
    Ht = (0.05 * W.MS * gH).astype(np.float32)
    Jr, Gr, _ = O.objective_and_gradient(op, rho, np.array([0.0, 0.0, W.MS]), 3.0, mask, Ht, (0.0, 1.0, 0.0))
    m.set_target(up(mask), Ht=up(Ht), w=(0.0, 1.0, 0.0))
    J, G = m.evaluate(up(rho))
    assert abs(J - Jr) <= 1e-5 * abs(Jr)
    assert rel(G.cpu().numpy(), Gr) <= 1e-5
