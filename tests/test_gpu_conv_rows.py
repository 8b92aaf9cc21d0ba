"""The row kernels of the warm-start convolutions (forward, data gradient, weight gradient) at
the edges of their tiles, against the float64 oracle: one plane and two per tile, planes and
rows that do not fill a tile, more tiles than blocks, one to six channel chunks, weights that
stay in shared memory and weights that do not, windows of output channels, and repeated
calls, which give the same bits.

Bounds as for the other tests of these kernels: inputs hold bfloat16 values, so a float32 sum
of K products carries at most K 2^-24 sum|terms| (1e-5 covers K = 27 * 96 and a few hundred
voxels a channel; the sums are added pairwise over blocks) and a bfloat16 output one rounding.
"""

import numpy as np
import pytest
import torch

from oracle import unet as U
from test_gpu_warmstart import DEV, S, bf16_round, f32, net_status, p, to_bf16_dev, wf_wb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    from paper_1707_09898_gb300 import _lib

    __graft_entry__.build()
    return _lib.lib()


CASES = [((1, 1, 1, 64), 16, 16), ((2, 3, 5, 64), 48, 16), ((1, 4, 9, 64), 64, 32), ((1, 3, 2, 64), 32, 64),
         ((1, 2, 3, 32), 16, 16), ((3, 5, 6, 32), 96, 32), ((1, 7, 4, 32), 32, 64), ((2, 5, 11, 16), 64, 64),
         ((1, 1, 1, 16), 16, 64), ((4, 21, 41, 16), 16, 16), ((2, 3, 17, 8), 32, 32), ((1, 9, 40, 8), 96, 32)]


@pytest.mark.parametrize("dims,cin,cout", CASES)
def test_rows(L, dims, cin, cout):
    rng = np.random.default_rng(dims[1] * 1000 + cin + cout)
    x = bf16_round(rng.normal(size=dims + (cin,)))
    W = bf16_round(rng.normal(0, 0.1, size=(27, cin, cout)))
    b = rng.normal(0, 0.1, size=cout).astype(np.float32).astype(np.float64)
    g = bf16_round(rng.normal(size=dims + (cout,)))
    Wf, Wb = wf_wb(L, W)
    xd, gd = to_bf16_dev(x), f32(g)
    out = torch.empty(dims + (cout,), dtype=torch.bfloat16, device=DEV)
    din = torch.empty(dims + (cin,), device=DEV)
    dW, db = torch.empty(27, cin, cout, device=DEV), torch.empty(cout, device=DEV)
    base = L.tmn_conv3d_backward_weight_work(int(np.prod(dims)), cin, cout)
    first = None
    for extra in (0, 0, 64 * 27 * cin * cout):  # the smallest scratch twice, then room for more blocks
        work = torch.empty(base + extra, device=DEV)
        assert L.tmn_conv3d_forward(p(xd), p(Wf), p(f32(b)), p(out), *dims, cin, cout, 0, S()) == 0
        assert L.tmn_conv3d_backward_data(p(gd), p(Wb), p(din), *dims, cin, cout, 0, S()) == 0
        assert L.tmn_conv3d_backward_weight(p(xd), p(gd), p(dW), p(db), p(work), work.numel(), *dims, cin, cout, S()) == 0
        now = [t.clone() for t in (out, din, dW, db)]
        if first is not None and extra == 0:
            assert all(torch.equal(a, c) for a, c in zip(first, now))
        first = now
        ref, bound = U.conv(x, W, b), U.conv(np.abs(x), np.abs(W), np.abs(b))
        assert np.all(np.abs(out.float().cpu().numpy() - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5 * bound)
        refs, bounds = U.conv_backward(x, W, g), U.conv_backward(np.abs(x), np.abs(W), np.abs(g))
        for got, r, e in zip((din, dW, db), refs, bounds):
            assert np.all(np.abs(got.cpu().numpy() - r) <= 1e-5 * e + 1e-30)
    assert L.tmn_conv3d_backward_data(p(gd), p(Wb), p(din), *dims, cin, cout, 1, S()) == 0  # accumulate
    assert np.all(np.abs(din.cpu().numpy() - 2 * refs[0]) <= 2e-5 * bounds[0] + 1e-30)
    assert net_status(L) == 0
