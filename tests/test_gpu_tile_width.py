"""The SM-pair product through rift_linear at sizes where it takes 192-wide tiles (as many waves as with
256-wide ones, more than one): a last tile of 64 columns, of 8, two and three waves, a K tail, against fp64
products of the same operands."""
import pytest
import torch

from synth import rng

pytestmark = pytest.mark.gpu

# fp16 outputs: one rounding, 2^-11 of the element, plus fp32 sums of K products of size ~0.05: K 2^-24
# of the sum of their magnitudes at worst, sqrt(K) 2^-24 of it for random signs.  Relative to the
# largest output both stay under these.
F16_TOL = 6e-4
F32_TOL = 2e-5

# (rows, weight rows, K); with 76 SM pairs the tiles are 96 : 132 (256 wide : 192 wide), 85 : 110, 160 : 220,
# 86 : 115
SHAPES = [(1300, 4096, 1032), (1100, 4104, 64), (2400, 4096, 200), (256, 22016, 520)]


def _rand(shape, stream, scale=1.0):
    n = shape[0] * shape[1]
    return (rng.normal_f32(6, rng.stream_id("tile-width", stream), n).view(*shape) * scale).to(torch.float16)


def _rel(g, o):
    return float((g.double().cpu() - o).abs().max() / o.abs().max())


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_narrow_tiles_all_epilogues(M, N, K, cuda, riftlib):
    A, W = _rand((M, K), 1), _rand((N, K), 2, 0.05)
    y = A.double() @ W.double().T
    a, w = A.to(cuda), W.to(cuda)
    out = torch.full((M, N), float("nan"), dtype=torch.float16, device=cuda)
    riftlib.linear(a, w, M, N, K, riftlib.RIFT_EPI_STORE_F16, out)
    R0 = rng.normal_f32(6, 79, M * N).view(M, N)
    R = R0.to(cuda)
    riftlib.linear(a, w, M, N, K, riftlib.RIFT_EPI_RESID_F32, R)
    riftlib.sync_status()
    assert _rel(out, y) < F16_TOL
    assert _rel(R, R0.double() + y) < F32_TOL
    if N % 32 == 0:
        act = torch.full((M, N // 2), float("nan"), dtype=torch.float16, device=cuda)
        riftlib.linear(a, w, M, N, K, riftlib.RIFT_EPI_SWIGLU, act)
        riftlib.sync_status()
        g, u = y.view(M, N // 32, 2, 16).unbind(2)
        assert _rel(act, (g / (1 + torch.exp(-g)) * u).reshape(M, N // 2)) < F16_TOL
