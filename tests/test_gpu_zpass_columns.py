"""The z pass with one input and several outputs on both sides of the line between an output on
blocks of its own (few column tiles) and all outputs in one block, at every length, against the
float64 oracle. Tolerances as in test_gpu_zpass.py."""

import numpy as np
import pytest

from oracle import convolution as C
from oracle import objective as O
from paper_1707_09898_gb300 import workloads as W
from test_gpu_zpass import TILTED, _build, rel, up  # noqa: F401

pytestmark = pytest.mark.gpu
LENGTHS = [8, 12, 16, 18, 24, 32, 36, 48, 64, 72, 96, 128, 144, 192, 256, 288, 384, 576]


@pytest.mark.parametrize("few", [True, False])
@pytest.mark.parametrize("L", LENGTHS)
def test_outputs_apart_and_together(L, few):
    from paper_1707_09898_gb300 import Magnet

    nz = max(4, L // 2 - L % 7)
    nx, ny = (9, 6) if few else (40, 80) if L == 576 else (9, 80)
    nzd = nz - nz // 6
    rng = np.random.default_rng(L + few)
    rho = rng.random((nzd, ny, nx)).astype(np.float32)
    op = C.FFTOperator(C.Geometry((nx, ny, nz), nzd, (1e-3,) * 3))
    m = Magnet((nx, ny, nz), nzd, (1e-3,) * 3, M0=tuple(TILTED), p=3.0, device=0,
               fft_lengths=(0, 0 if few else 192, L))
    mask = np.ones((nz, ny, nx), np.uint8)
    Ht = (0.05 * W.MS * rng.normal(size=(3, nz, ny, nx))).astype(np.float32)
    for M0 in (np.array([0.0, 0.0, W.MS]), TILTED):
        m.set_M0(tuple(M0))
        assert rel(m.stray_field(up(rho)).cpu().numpy(), op.forward(O.magnetization(rho, M0, 3.0))) <= 3e-6
        Jr, Gr, _ = O.objective_and_gradient(op, rho, M0, 3.0, mask, Ht, (0.5, 0.0, 1.0))  # two outputs
        J, G = m.objective_and_gradient(up(rho), up(mask), Ht=up(Ht), w=(0.5, 0.0, 1.0))
        assert abs(J - Jr) <= 1e-5 * abs(Jr)
        assert rel(G.cpu().numpy(), Gr) <= 1e-5
