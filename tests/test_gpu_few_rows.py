"""The cluster split-K product (few rows: weights as the 128-row operand, K split over a
thread-block cluster) through rift_linear, at the edges of its row tiles (16 to 160 rows; at most 48
where K is too short to split), weight tiles (128 rows), K-blocks (64) and cluster sizes, and of the rows it
takes before the SM pairs' kernel does, against fp64 products of the same operands."""
import pytest
import torch

from synth import rng

pytestmark = pytest.mark.gpu

# fp16 outputs: one rounding, 2^-11 of the element, plus fp32 sums of K products of size ~0.05: K 2^-24
# of the sum of their magnitudes at worst, sqrt(K) 2^-24 of it for random signs.  Relative to the
# largest output both stay under these.
F16_TOL = 6e-4
F32_TOL = 2e-5

# (rows, weight rows, K): one K-block; 1, 2, 3 and 8 slices of K (8 K-blocks each at least), uneven
# ones, a K tail; rows around 16, 128, 160 and in two and three row tiles; a partial weight tile
SHAPES = [(1, 128, 64), (1, 160, 520), (2, 136, 1032), (15, 264, 1600), (16, 4096, 4096), (17, 1024, 4104),
          (127, 288, 2816), (160, 1024, 11008), (161, 1024, 4096), (203, 672, 4104), (333, 288, 11008)]
# short K: 48 and 49 rows, a K tail, the last K-block count that is short and the first that is not
SHAPES += [(48, 128, 200), (49, 136, 64), (300, 256, 256), (1000, 264, 72), (1023, 768, 960), (161, 96, 1016), (161, 96, 1024)]
# as many short tiles as fit on 152 SMs at once (16 x 19), one row more (SM pairs, K tail), and SM pairs with tails in
# rows, weight rows and K
SHAPES += [(768, 2432, 200), (769, 2432, 200), (4400, 2056, 1032)]
# tiles whose count times the cluster size fits while the clusters do not (40 tiles: 38 clusters of 7 fit, 46 of 6)
SHAPES += [(100, 5120, 4096), (777, 1024, 4104)]
# 128 x 256 tiles of one SM (fewer waves than the pairs'): one and several tiles a CTA, tails in rows, weight rows and K
SHAPES += [(257, 12288, 1032), (300, 12296, 1096), (384, 22016, 1032), (777, 5128, 1032)]


def _rand(shape, stream, scale=1.0):
    n = shape[0] * shape[1]
    return (rng.normal_f32(6, rng.stream_id("few-rows", stream), n).view(*shape) * scale).to(torch.float16)


def _rel(g, o):
    return float((g.double().cpu() - o).abs().max() / o.abs().max())


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_few_rows_all_epilogues(M, N, K, cuda, riftlib):
    A, W = _rand((M, K), 1), _rand((N, K), 2, 0.05)
    y = A.double() @ W.double().T
    a, w = A.to(cuda), W.to(cuda)
    out = torch.full((M, N), float("nan"), dtype=torch.float16, device=cuda)
    riftlib.linear(a, w, M, N, K, riftlib.RIFT_EPI_STORE_F16, out)
    R0 = rng.normal_f32(6, 78, M * N).view(M, N)
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


def test_one_sm_tiles_with_rope_and_cache(cuda, riftlib):
    """The QKV product of 300 rows at d = 4096 runs on tiles of one SM, that of 600 rows on SM pairs: the same keys,
    values and hidden states for the rows the two batches share."""
    from paper_2609_29029_gb300 import DeviceModel
    from synth import workloads as W
    dec = W.DecoderShape(n_layers=1, d=4096, n_heads=32, head_dim=128, ffn=64, vocab=504)
    dm = DeviceModel(dec, [W.make_layer(dec, 0, "cpu")], W.make_final_norm(dec, "cpu"), cuda)
    rows = torch.randn(600, dec.d, device=cuda).to(torch.bfloat16)

    def prefill(lens):
        T, n = sum(lens), len(lens)
        cu = torch.tensor([sum(lens[:i]) for i in range(n + 1)], dtype=torch.int32, device=cuda)
        pos = torch.cat([torch.arange(L, dtype=torch.int32, device=cuda) for L in lens])
        hid = rows[:T].clone()
        kv = torch.full((1, 2, T, dec.d), float("nan"), dtype=torch.float16, device=cuda)
        need = riftlib.prefill_workspace_bytes(dm.struct, T, n, max(lens))
        ws = torch.empty(need, dtype=torch.uint8, device=cuda)
        riftlib.prefill_layers(dm.struct, hid, T, cu, n, max(lens), pos, ws, need, kv_out=kv)
        riftlib.sync_status()
        return hid.float(), kv.float()

    h1, kv1 = prefill([100, 31, 169])
    h2, kv2 = prefill([100, 31, 169, 300])
    assert float((kv1 - kv2[:, :, :300]).abs().max()) <= 2.0 ** -10 * float(kv1.abs().max())
    assert float((h1 - h2[:300]).abs().max()) <= 2.0 ** -7 * float(h1.abs().max())
