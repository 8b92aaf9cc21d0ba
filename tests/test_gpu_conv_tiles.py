"""The row kernels of the convolutions with several tiles per block: the accumulator ring, the
staged rows and weights, the exchange between the two warps of a 64-voxel row and the data
gradient's output buffer are all reused from tile to tile, two planes to a tile and one, with
weights that stay in shared memory and weights that do not, planes and rows that do not fill
the last tiles. Every case has at least twice as many tiles as SMs.

Reference: products of the same bfloat16 values in 64 bits, one matrix product per tap. Bounds as
in test_gpu_conv_rows.py: one bfloat16 rounding of the output, 1e-5 of the sum of the terms'
magnitudes for the float32 sums."""

import pytest
import torch

from test_gpu_warmstart import DEV, S, net_status, p

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    from paper_1707_09898_gb300 import _lib

    __graft_entry__.build()
    return _lib.lib()


def shifted(x):
    """x of every tap's voxel, zero outside the grid: [tap] -> [voxels][channels]"""
    n, d, h, w, c = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    return lambda t: xp[:, t // 9:t // 9 + d, t // 3 % 3:t // 3 % 3 + h, t % 3:t % 3 + w].reshape(-1, c)


def conv(x, W):
    s = shifted(x)
    return sum(s(t) @ W[t] for t in range(27)).reshape(x.shape[:-1] + (W.shape[2],))


def check(got, ref, bound, rounding=0.0, factor=1e-5):
    assert bool(((got.double() - ref).abs() <= rounding * ref.abs() + factor * bound + 1e-30).all())


CASES = [((2, 18, 40, 64), 48, 16), ((2, 35, 23, 64), 16, 16), ((1, 36, 40, 64), 64, 32), ((1, 24, 26, 64), 32, 64),
         ((2, 33, 41, 32), 96, 32), ((2, 32, 37, 32), 32, 64), ((4, 40, 45, 16), 64, 64), ((3, 37, 59, 16), 96, 16),
         ((4, 41, 70, 8), 32, 32), ((3, 52, 80, 8), 96, 32), ((4, 40, 64, 8), 16, 64)]


@pytest.mark.parametrize("dims,cin,cout", CASES)
def test_many_tiles(L, dims, cin, cout):
    gen = torch.Generator(device=DEV).manual_seed(dims[1] + cin + cout)
    x = torch.randn(dims + (cin,), generator=gen, device=DEV).to(torch.bfloat16)
    W = (0.1 * torch.randn((27, cin, cout), generator=gen, device=DEV)).to(torch.bfloat16).float()
    b = 0.1 * torch.randn(cout, generator=gen, device=DEV)
    g = torch.randn(dims + (cout,), generator=gen, device=DEV).to(torch.bfloat16).float()
    wf = torch.empty(27 * cin * cout, dtype=torch.bfloat16, device=DEV)
    wb = torch.empty_like(wf)
    assert L.tmn_pack_conv_weights(p(W), p(wf), p(wb), cin, cout, S()) == 0
    out = torch.empty(dims + (cout,), dtype=torch.bfloat16, device=DEV)
    din = torch.empty(dims + (cin,), device=DEV)
    dW, db = torch.empty_like(W), torch.empty_like(b)
    nvox = x.numel() // cin
    work = torch.empty(L.tmn_conv3d_backward_weight_work(nvox, cin, cout) + 160 * 28 * cin * cout, device=DEV)
    first = None
    for _ in range(4):
        for t in (out, din, dW, db):
            t.fill_(float("nan"))
        assert L.tmn_conv3d_forward(p(x), p(wf), p(b), p(out), *dims, cin, cout, 0, S()) == 0
        assert L.tmn_conv3d_backward_data(p(g), p(wb), p(din), *dims, cin, cout, 0, S()) == 0
        assert L.tmn_conv3d_backward_weight(p(x), p(g), p(dW), p(db), p(work), work.numel(), *dims, cin, cout, S()) == 0
        now = [t.clone() for t in (out, din, dW, db)]
        if first is None:
            first = now
        assert all(torch.equal(a, c) for a, c in zip(first, now))
    xd, Wd, gd = x.double(), W.double(), g.double()
    check(out, conv(xd, Wd) + b.double(), conv(xd.abs(), Wd.abs()) + b.double().abs(), 2.0 ** -8)
    back = Wd.flip(0).transpose(1, 2)
    ref, bound = conv(gd, back), conv(gd.abs(), back.abs())
    check(din, ref, bound)
    s, sa, gv = shifted(xd), shifted(xd.abs()), gd.reshape(-1, cout)
    for t in range(27):
        check(dW[t], s(t).T @ gv, sa(t).T @ gv.abs())
    check(db, gv.sum(0), gv.abs().sum(0))
    assert L.tmn_conv3d_backward_data(p(g), p(wb), p(din), *dims, cin, cout, 1, S()) == 0  # accumulate
    check(din, 2 * ref, bound, factor=2e-5)
    assert net_status(L) == 0
