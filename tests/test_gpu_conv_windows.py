"""The data gradient for 96 channels, two windows of 48, with two planes to a tile: the sizes at
which that form is taken (weights that do not stay in shared memory, or no more rounds of tiles
than with one plane), planes and rows that do not fill the last tile, against the same products
in 64 bits. Bounds as in test_gpu_conv_tiles.py."""

import pytest
import torch

from test_gpu_conv_tiles import DEV, L, S, check, conv, net_status, p  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [((1, 26, 13, 64), 64), ((1, 31, 16, 64), 32), ((3, 27, 30, 32), 64), ((1, 31, 32, 32), 32),
         ((4, 19, 37, 16), 64), ((2, 76, 16, 16), 32), ((4, 19, 40, 8), 64), ((4, 76, 16, 8), 32), ((2, 25, 17, 64), 48)]


@pytest.mark.parametrize("dims,cout", CASES)
def test_two_planes(L, dims, cout):  # noqa: F811
    cin = 96
    gen = torch.Generator(device=DEV).manual_seed(dims[1] + cout)
    W = (0.1 * torch.randn((27, cin, cout), generator=gen, device=DEV)).to(torch.bfloat16).float()
    g = torch.randn(dims + (cout,), generator=gen, device=DEV).to(torch.bfloat16).float()
    wf = torch.empty(27 * cin * cout, dtype=torch.bfloat16, device=DEV)
    wb = torch.empty_like(wf)
    assert L.tmn_pack_conv_weights(p(W), p(wf), p(wb), cin, cout, S()) == 0
    back = W.double().flip(0).transpose(1, 2)
    ref, bound = conv(g.double(), back), conv(g.double().abs(), back.abs())
    first = None
    for _ in range(4):
        din = torch.full(dims + (cin,), float("nan"), device=DEV)
        assert L.tmn_conv3d_backward_data(p(g), p(wb), p(din), *dims, cin, cout, 0, S()) == 0
        first = din if first is None else first
        assert torch.equal(first, din)
    check(din, ref, bound)
    assert L.tmn_conv3d_backward_data(p(g), p(wb), p(din), *dims, cin, cout, 1, S()) == 0
    check(din, 2 * ref, bound, factor=2e-5)
    assert net_status(L) == 0
